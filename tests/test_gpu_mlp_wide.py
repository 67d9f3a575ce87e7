"""Networks with more inputs than one chunk of the first product (128): the input is converted by a launch of its
own. Widths around its groups (8 and 32 columns, padding to 16), batches around 8, 16 and 128 rows, an input that
starts off a 16-byte boundary, a batch smaller than the one before; outputs and gradients against the oracle with
the tolerances of BF16 operands (2e-2, 3e-2), and the same bits wherever the input lies."""
import ctypes as C

import numpy as np
import pytest

from oracle import mlp_oracle as M

pytestmark = pytest.mark.gpu


def _rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("sizes", [[129, 16], [137, 33, 9], [144, 64], [255, 40, 20], [1025, 48], [4096, 17, 16]], ids=str)
def test_wide_inputs(sizes):
    import torch
    import __graft_entry__ as g
    g.build()
    from paper_1608_04601_gb300 import mlp
    rng = np.random.default_rng(sizes[0])
    net = mlp.MLP(sizes, max_batch=131, seed=2)
    p = M.weights_bf16(net.get_params(), sizes)
    for b in (131, 128, 17, 8, 1):
        x = rng.standard_normal((b, sizes[0])).astype(np.float32)
        t = rng.standard_normal((b, sizes[-1])).astype(np.float32)
        y = net.forward(x).cpu().numpy()
        assert _rel(y, M.forward(p, sizes, x)[-1]) < 2e-2, b
        buf = torch.zeros(x.size + 1, dtype=torch.float32, device="cuda")
        buf[1:] = torch.from_numpy(x.ravel()).cuda()
        y1 = torch.zeros(b, sizes[-1], device="cuda")
        torch.cuda.synchronize()
        net._ck(net.L.mlp_forward(net.h, b, C.c_void_p(buf.data_ptr() + 4), C.c_void_p(y1.data_ptr())))
        net._ck(net.L.mlp_sync(net.h))
        assert np.array_equal(y1.cpu().numpy(), y), b
        loss = net.loss_grad(x, t)
        ref_loss, ref_g = M.loss_grad(p, sizes, x, t)
        assert abs(loss - ref_loss) <= 1e-2 * ref_loss
        got = net.grads()
        for w, o, i, n in M.layout(sizes)[0]:
            assert _rel(got[w:w + i * n], ref_g[w:w + i * n]) < 3e-2, b
            assert _rel(got[o:o + n], ref_g[o:o + n]) < 3e-2, b
    net.close()

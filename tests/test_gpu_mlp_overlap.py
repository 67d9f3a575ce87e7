"""mlp_forward with outputs that overlap its inputs gives the outputs of separate arrays, bit for bit: in place and
shifted, one layer (whose product reads x in one tile while it writes y from another) and two."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[64, 64], [33, 200], [300, 40], [64, 48, 64]], ids=str)
@pytest.mark.parametrize("batch", [1, 40, 300])
def test_forward_over_its_own_input(sizes, batch):
    import torch
    import __graft_entry__ as g
    g.build()
    from paper_1608_04601_gb300 import mlp
    net = mlp.MLP(sizes, max_batch=300, seed=5)
    x = torch.from_numpy(np.random.default_rng(batch).standard_normal((batch, sizes[0])).astype(np.float32)).cuda()
    want = net.forward(x).cpu().numpy().ravel()
    nx, ny = x.numel(), want.size
    for at in (0, 7, max(0, nx - 1)):  # y starts in place, inside x, at its last value
        buf = torch.zeros(nx + ny + 8, dtype=torch.float32, device="cuda")
        buf[:nx] = x.reshape(-1)
        torch.cuda.synchronize()
        net._ck(net.L.mlp_forward(net.h, batch, C.c_void_p(buf.data_ptr()), C.c_void_p(buf.data_ptr() + 4 * at)))
        net._ck(net.L.mlp_sync(net.h))
        assert np.array_equal(buf[at:at + ny].cpu().numpy(), want), at
        o = max(0, ny - 1 - at)  # x starts inside y
        buf = torch.zeros(nx + ny + 8, dtype=torch.float32, device="cuda")
        buf[o:o + nx] = x.reshape(-1)
        torch.cuda.synchronize()
        net._ck(net.L.mlp_forward(net.h, batch, C.c_void_p(buf.data_ptr() + 4 * o), C.c_void_p(buf.data_ptr())))
        net._ck(net.L.mlp_sync(net.h))
        assert np.array_equal(buf[:ny].cpu().numpy(), want), o
    net.close()

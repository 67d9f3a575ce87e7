// pic_kernels.cu -- CUDA kernels (sm_103a) of the 1d3v PIC/MCC time step of
// arXiv:1608.04601, section "PIC/MCC simulation procedure".
//
// One time step is two launches (and the sort every K steps):
//   k_sweep     persistent, one CTA per SM; every warp takes a contiguous run
//               of chunks (32 PPT slots) of each store and per chunk draws the
//               candidates, collides them, then pushes all its particles in one
//               pass (CIC gather of E_n from shared memory, half kicks, drift,
//               walls) and writes the survivors in slot order into the chunk's
//               own output region, newborns into the chunk's newborn regions.
//               CIC deposits and energy go to shared-memory histograms of exact
//               32-bit pieces, flushed with global atomics. Chunk counts are
//               summed per slice.
//   k_post      per slice of chunks: the region starts of the new layout and
//               the newborn copies; per discharge, concurrently: the store
//               totals (new counts) and Poisson (Eq. poisson, rf Dirichlet
//               boundary) from exact integer prefix sums of the deposits, node
//               field, cycle-average accumulators, J(t).
//   sort        every K steps: stable counting sort of each store by cell
//               into a dense store (else an order-preserving repack).
//   k_diag      at the steps the diagnostics schedule names, before the sweep:
//               the electrons' node moments and energy histogram.
#include "pic_internal.h"
#include "pic_device.cuh"
#include "pic_sort.cuh"

namespace pic {

#define E_CHARGE 1.602176634e-19
#define M_ELEC 9.1093837015e-31
#define EPS0 8.8541878128e-12
#define PI_D 3.14159265358979323846
#define TWO32_D 4294967296.0

template <typename T> __device__ __forceinline__ const Consts<T>& consts_of(const Disc& d);
template <> __device__ __forceinline__ const Consts<float>& consts_of<float>(const Disc& d) { return d.cf; }
template <> __device__ __forceinline__ const Consts<double>& consts_of<double>(const Disc& d) { return d.cd; }

template <typename T> struct T4;
template <> struct T4<float> { using type = float4; using two = float2; };
template <> struct T4<double> { using type = d4; using two = double2; };

template <int V>
struct IC { static constexpr int value = V; };
template <typename T>
struct Part {
    int c;
    T f, vx, vy, vz;
};

template <typename T> __device__ __forceinline__ const Seg<T>* segs_of(const Disc& d);
template <> __device__ __forceinline__ const Seg<float>* segs_of<float>(const Disc& d) { return d.sf; }
template <> __device__ __forceinline__ const Seg<double>* segs_of<double>(const Disc& d) { return d.sd; }

// Programmatic dependent launch (the kernels of a step, launched by launch_pdl): wait until the
// previous kernel in the stream has completed and its writes are visible. Every such kernel calls this
// before its first access to memory that kernels write (a no-op for a kernel launched without the
// attribute); what needs no results (shared memory cleared, constants fetched) may come before. Memory that
// the kernel before may still be writing when this one starts is not read-only over its lifetime, so it is
// never read through the non-coherent path (__ldg, or a plain load from a const __restrict__ pointer), but
// with __ldcg or from unrestricted pointers. No kernel
// triggers its dependents early: they launch as its CTAs exit (with early triggers in the sweep and k_post
// the smallest runs gained 0.6 us of 26 a step and the larger ones lost 1-2 %).
__device__ __forceinline__ void grid_dep_sync() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename T>
__device__ __forceinline__ int drift(int N, T dtdx, int c, T f, T vz, int& cn, T& fn, int& err) {
    const T s = fma_(vz, dtdx, f);
    if (!(s == s)) err |= ERR_NONFINITE;
    if (!(s >= (T)(-c))) return 0;
    if (s >= (T)(N - c)) return 1;
    const T fl = floor_(s);
    T fr = sub_(s, fl);
    if (fr >= (T)1) fr = one_minus_ulp<T>();
    cn = c + (int)fl;
    fn = fr;
    return -1;
}

// The drift of the sweep's main pass, the same values as drift() with fewer operations: floor(s) by
// adding 1.5 2^23 (2^52 in double) rounded towards minus infinity, which leaves the integer in the low
// mantissa bits; exact for |s| < 8192, and a particle further out (or not a number) is not alive: a
// discharge has at most 4096 cells. Returns whether the particle stays; s >= 0 then tells the electrode.
__device__ __forceinline__ bool drift_fast(int N, float dtdx, int c, float f, float vz, int& cn, float& fn, float& s) {
    s = __fmaf_rn(vz, dtdx, f);
    const float t = __fadd_rd(s, 12582912.0f);
    cn = c + (__float_as_int(t) - 0x4B400000);
    fn = fminf(__fsub_rn(s, __fsub_rn(t, 12582912.0f)), one_minus_ulp<float>());
    return fabsf(s) < 8192.0f && (unsigned)cn < (unsigned)N;
}
__device__ __forceinline__ bool drift_fast(int N, double dtdx, int c, double f, double vz, int& cn, double& fn,
                                           double& s) {
    s = __fma_rn(vz, dtdx, f);
    const double t = __dadd_rd(s, 6755399441055744.0);
    cn = c + __double2loint(t);
    fn = __dsub_rn(s, __dsub_rn(t, 6755399441055744.0));
    if (__double2hiint(fn) >= 0x3FF00000) fn = one_minus_ulp<double>();  // rounded to 1
    return (__double2hiint(s) & 0x7FFFFFFF) < 0x40C00000 && (unsigned)cn < (unsigned)N;  // |s| < 8192
}

// Exact 64-bit add into a shared-memory word with native 32-bit atomics: the low
// word's returned old value tells whether this add carried into the high word.
__device__ __forceinline__ void sadd64(unsigned long long* p, unsigned long long v) {
    unsigned* w = reinterpret_cast<unsigned*>(p);
    const unsigned lo = (unsigned)v, hi = (unsigned)(v >> 32);
    const unsigned old = atomicAdd(&w[0], lo);
    const unsigned up = hi + ((unsigned)(old + lo) < old ? 1u : 0u);
    if (up) atomicAdd(&w[1], up);
}

__device__ __forceinline__ void hist_add(unsigned long long* h, int c, unsigned long long F) {
    atomicAdd(&h[c], (1ull << 32) - F);
    if (F) atomicAdd(&h[c + 1], F);
}

// Same, into a shared-memory histogram.
__device__ __forceinline__ void shist_add(unsigned long long* h, int c, unsigned long long F) {
    sadd64(&h[c], (1ull << 32) - F);
    if (F) sadd64(&h[c + 1], F);
}

// Round-to-nearest-even conversion of a value in [0, 2^32) to an unsigned integer.
__device__ __forceinline__ unsigned rint_u32(float a) { return __float2uint_rn(a); }
__device__ __forceinline__ unsigned rint_u32(double a) {
    return (unsigned)__double2loint(__dadd_rn(a, 6755399441055744.0));  // 1.5 2^52: the integer in the low bits
}

__device__ __forceinline__ unsigned long long cic_F(float f) {
    return (unsigned long long)__float2uint_rn(__fmul_rn(f, 4294967296.0f));  // f < 1: below 2^32
}
// May round to 2^32. Adding 1.5 2^20 rounds f to a multiple of 2^-32 (ties to even) and leaves the
// multiple in the low mantissa bits: one FP64 addition (the FP64 pipe is the slow one here).
__device__ __forceinline__ unsigned long long cic_F(double f) {
    return (unsigned long long)(__double_as_longlong(__dadd_rn(f, 1572864.0)) - 0x4138000000000000ll);
}

// The sweep's shared-memory histograms hold exact sums in 32-bit pieces, added with atomics whose
// result is not read (no return trip, no carry logic); arrays of one word per cell c, `hs` words apart:
//   0 particles n_c; 1, 2 the sum of F = rn(f 2^32) as low and high 16-bit parts; node j then receives
//     2^32 n_j - F_j + F_{j-1} (the charge split (2^32 - F, F) of every particle);
//   3, 4 (electrons) the sums of the low 17 bits of the energy E and of its share H = rn(E f); node j
//     receives E_j - H_j + H_{j-1}. The bits above (an electron of more than 32 eV) go to one more array, of
//     one word per node (below 2^25), where shared memory holds it beside the rest (one electron in five is
//     above 32 eV while the sheaths of a he_family discharge form, one in thirty later: global adds took
//     26.1 us a step then, the array takes 24.4; 64 such discharges 84.2 -> 82.8), else straight to the
//     global sums (above about 1970 cells of FP32: the array would cost a warp, 4 % of the sweep).
// The 64-bit node values are formed when the CTA flushes. A piece sum stays below 2^32 while the CTA has
// added at most FLUSH_PARTICLES particles of a species (plus as many newborns) since its last flush.
template <typename T>
__host__ __device__ constexpr int flush_particles() { return sizeof(T) == 4 ? 32768 : 16384; }  // F = 2^32 occurs in double
//
// On a cell-sorted store the lanes of a warp add to the same few cells, and adds to one word run one
// after another. So each species also has a window of WIN cells around the CTA's chunks with WCOP copies
// of every word, lane l adding to copy l % WCOP: at most 32 / WCOP adds meet. A flush folds the window
// into the full arrays. (The sweep of a freshly sorted store of 1.2e7 + 1.2e7 particles in 2048 cells
// spent a third of its time in these conflicts.)
// A CTA with fewer than WIN_CHUNKS chunks of a store goes without: it has few adds, and the extra pass of
// its flush costs more (2e4 + 2e4 particles: 22.4 us a step with windows everywhere, 21.5 with this rule).
constexpr int WIN = 64, WCOP = 8, WWORDS = WIN * WCOP, WIN_CHUNKS = 16, NO_WIN = -(1 << 30);
struct Hist {
    unsigned* full;  // arrays of hs words
    unsigned* win;   // arrays of WWORDS words: cell w0 + j, copy k at j WCOP + k
    int hs, w0;
    // the words of cell c for this lane: first array and distance between arrays
    __device__ __forceinline__ unsigned* at(int c, int lane, int& st) const {
        const unsigned j = (unsigned)(c - w0);
        const bool in = j < (unsigned)WIN;
        st = in ? WWORDS : hs;
        return in ? win + (j * WCOP + (lane & (WCOP - 1))) : full + c;
    }
};
__device__ __forceinline__ void dep_add(const Hist& h, int c, unsigned long long F, int lane) {
    int st;
    unsigned* a = h.at(c, lane, st);
    atomicAdd(a, 1u);
    atomicAdd(a + st, (unsigned)(F & 0xFFFFu));
    atomicAdd(a + 2 * st, (unsigned)(F >> 16));
}
// Deposit of one particle per lane (key = cell, < 0: none). UNIFORM (ions: slow, so a row of a sorted
// store mostly shares a cell): such a row is reduced across the warp and added by one lane.
template <bool UNIFORM>
__device__ __forceinline__ void warp_dep(const Hist& h, int key, unsigned long long F, int lane) {
    if (UNIFORM) {
        const int k0 = __shfl_sync(FULL, key, 0);
        if (__all_sync(FULL, key == k0)) {
            const unsigned lo = __reduce_add_sync(FULL, (unsigned)(F & 0xFFFFu));
            const unsigned hi = __reduce_add_sync(FULL, (unsigned)(F >> 16));
            if (lane == 0 && key >= 0) {
                int st;
                unsigned* a = h.at(key, lane, st);
                atomicAdd(a, 32u);
                atomicAdd(a + st, lo);
                atomicAdd(a + 2 * st, hi);
            }
            return;
        }
    }
    if (key >= 0) dep_add(h, key, F, lane);
}
// Energy moment of the lanes' electrons (`on`; every lane of the warp calls) of energy speed^2 kappa_E
// (2^-12 eV, clamped at 2^26) at (c, f).
template <typename T>
__device__ __forceinline__ void energy_add(const Hist& h, unsigned* hi, unsigned long long* Qg, bool on, int c, T f,
                                           T e2, T kappa_E, int lane) {
    T eq = mul_(e2, kappa_E);
    if (!(eq <= (T)0x1p26)) eq = (T)0x1p26;
    const unsigned Et = rint_u32(eq), Eh = rint_u32(mul_(eq, f));
    if (on) {
        int st;
        unsigned* a = h.at(c, lane, st);
        atomicAdd(a + 3 * st, Et & 0x1FFFFu);
        atomicAdd(a + 4 * st, Eh & 0x1FFFFu);
    }
    const bool high = on && (Et >> 17);
    if (__any_sync(FULL, high)) {
        if (high) {
            const unsigned ht = Et >> 17, hh = Eh >> 17;
            if (hi) {
                if (ht != hh) atomicAdd(hi + c, ht - hh);
                if (hh) atomicAdd(hi + c + 1, hh);
            } else {
                atomicAdd(&Qg[c], (unsigned long long)(ht - hh) << 17);
                if (hh) atomicAdd(&Qg[c + 1], (unsigned long long)hh << 17);
            }
        }
        __syncwarp();  // keeps this a branch: as predicated instructions the rare part costs every row 17 of them
    }
}

template <typename T>
__device__ __forceinline__ void store_rec(int32_t* c, void* p, unsigned i, const Part<T>& q);
template <>
__device__ __forceinline__ void store_rec<float>(int32_t* c, void* p, unsigned i, const Part<float>& q) {
    c[i] = q.c;
    reinterpret_cast<float4*>(p)[i] = make_float4(q.f, q.vx, q.vy, q.vz);
}
template <>
__device__ __forceinline__ void store_rec<double>(int32_t* c, void* p, unsigned i, const Part<double>& q) {
    c[i] = q.c;
    double2* pp = reinterpret_cast<double2*>(p) + 2 * i;
    pp[0] = make_double2(q.f, q.vx);
    pp[1] = make_double2(q.vy, q.vz);
}

template <typename T>
__device__ __forceinline__ void load_rec(const void* p, unsigned i, T& f, T& vx, T& vy, T& vz);
template <>
__device__ __forceinline__ void load_rec<float>(const void* p, unsigned i, float& f, float& vx, float& vy,
                                                float& vz) {
    const float4 a = __ldcs(reinterpret_cast<const float4*>(p) + i);
    f = a.x; vx = a.y; vy = a.z; vz = a.w;
}
template <>
__device__ __forceinline__ void load_rec<double>(const void* p, unsigned i, double& f, double& vx, double& vy,
                                                 double& vz) {
    const double2* pp = reinterpret_cast<const double2*>(p) + 2 * i;
    const double2 a = __ldcs(pp), b = __ldcs(pp + 1);
    f = a.x; vx = a.y; vy = b.x; vz = b.y;
}

// A whole record, coherent (see grid_dep_sync).
__device__ __forceinline__ float4 ldcg_rec(const float4* p) { return __ldcg(p); }
__device__ __forceinline__ d4 ldcg_rec(const d4* p) {
    const double2 a = __ldcg(reinterpret_cast<const double2*>(p)), b = __ldcg(reinterpret_cast<const double2*>(p) + 1);
    return d4{a.x, a.y, b.x, b.y};
}

// draw() of pic_device.cuh with the counter's second and third words prepared once.
struct Stream {
    unsigned long long seed;
    uint32_t w1, w2, did;  // step bits 0..31; step bits 32..47 << 16 | species << 8; discharge
    __device__ __forceinline__ U4 draw(uint32_t slot, int call) const {
        return philox4x32_10(slot, w1, w2 | (uint32_t)call, did, (uint32_t)seed, (uint32_t)(seed >> 32));
    }
};

// The collision candidates of a chunk are queued by their warp in shared memory as their indices
// in the chunk; the lane that processes one reads the particle from the staged records, collides
// it, writes the new velocity back into the staged record and flags the newborns it left after
// their first drift, which it stores at the candidate's rank in the chunk's newborn regions (the
// warp then compacts them into parent-slot order).
// A collision candidate of a chunk: its velocity v_n and gathered field on entry; the velocity after
// the collision on return; newborns flagged in `out` (bit 1: same species, bit 2: other species).
template <typename T>
struct Cand {
    T ef;
    T vx, vy, vz;
};

// The collision of a queued candidate (null-collision method: process
// selection against the cumulative rate tables, then the kinematics).
template <typename T>
__device__ __forceinline__ uint32_t collide(const Seg<T>& S, int SP, unsigned long long* Dother, Cand<T>& q, int qc, T qf, uint32_t slot, uint32_t ridx,
                                         const Stream& rs, const Hist& sH, unsigned* sC,
                                         int& err) {
    using Row4 = typename T4<T>::type;
    using Row2 = typename T4<T>::two;
    const Consts<T>& K = S.k;
    const int N = S.N;
    T vx = q.vx, vy = q.vy, vz = q.vz;
    uint32_t out = 0;
    if (SP == 0) {
        const T e2 = fma_(vx, vx, fma_(vy, vy, mul_(vz, vz)));
        bool child = false;
        T cvx = 0, cvy = 0, cvz = 0, ivx = 0, ivy = 0, ivz = 0;
        // the two table rows are requested first, so that their latency runs under the draw
        const T xi = mul_(e2, K.kappa_e);
        const bool above = !(xi < (T)(S.n_pts - 1));  // beyond the last row: its values
        const int it = above ? S.n_pts - 2 : (int)xi;
        const Row4* Te = reinterpret_cast<const Row4*>(S.Te) + it;
        const Row4 ta = Te[0], tb = Te[1];
        const U4 r = rs.draw(slot, 0);
        const T fr = sub_(xi, (T)it);
        T C0 = fma_(fr, sub_(tb.x, ta.x), ta.x), C1 = fma_(fr, sub_(tb.y, ta.y), ta.y);
        T C2 = fma_(fr, sub_(tb.z, ta.z), ta.z), C3 = fma_(fr, sub_(tb.w, ta.w), ta.w);
        if (above) {
            C0 = tb.x; C1 = tb.y; C2 = tb.z; C3 = tb.w;
            atomicAdd(&sC[CNT_CLAMP + 0], 1u);
        }
        const T R = mul_((T)u01(r.y), K.kmax_e);
        const int j = (R < C0) ? 0 : (R < C1) ? 1 : (R < C2) ? 2 : (R < C3) ? 3 : 4;
        if (j < 4) {
            // the scattered electron's direction: the same draw for every process, so it is
            // formed once, outside the per-process branches
            T nx, ny, nz;
            iso_dir(u01(r.z), u01(r.w), nx, ny, nz);
            if (j == 0) {  // elastic, target at rest: v' = beta v + (1-beta)|v| n
                const T g = sqrt_(e2);
                const T og = mul_(K.omb, g);
                vx = fma_(K.beta, vx, mul_(og, nx));
                vy = fma_(K.beta, vy, mul_(og, ny));
                vz = fma_(K.beta, vz, mul_(og, nz));
                atomicAdd(&sC[CNT_COLL_E + 0], 1u);
            } else if (j <= S.n_exc) {  // excitation of level j
                const T e2n = sub_(e2, K.de2_exc[j - 1]);
                if (e2n > (T)0) {
                    const T sp = sqrt_(e2n);
                    vx = mul_(sp, nx);
                    vy = mul_(sp, ny);
                    vz = mul_(sp, nz);
                    atomicAdd(&sC[CNT_COLL_E + j], 1u);
                } else {
                    atomicAdd(&sC[CNT_NULL_INEL], 1u);
                }
            } else {  // ionization: remaining energy shared equally
                const T e2r = sub_(e2, K.de2_iz);
                if (e2r > (T)0) {
                    const T sp = sqrt_(mul_((T)0.5, e2r));
                    vx = mul_(sp, nx);
                    vy = mul_(sp, ny);
                    vz = mul_(sp, nz);
                    const U4 q1 = rs.draw(slot, 1);
                    const U4 w = rs.draw(slot, 2);
                    iso_dir(u01(q1.x), u01(q1.y), nx, ny, nz);
                    cvx = mul_(sp, nx);
                    cvy = mul_(sp, ny);
                    cvz = mul_(sp, nz);
                    float b0, b1, b2, b3;
                    box_muller(u01(q1.z), u01(q1.w), b0, b1);
                    box_muller(u01(w.x), u01(w.y), b2, b3);
                    ivx = mul_(K.sig_n, (T)b0);
                    ivy = mul_(K.sig_n, (T)b1);
                    ivz = mul_(K.sig_n, (T)b2);
                    child = true;
                    atomicAdd(&sC[CNT_COLL_E + 3], 1u);
                } else {
                    atomicAdd(&sC[CNT_NULL_INEL], 1u);
                }
            }
        }
        if (child) {  // newborns: second half kick and drift from the parent's position
            int cn;
            T fn;
            if (!S.leapfrog) cvz = fma_(K.K[0], q.ef, cvz);  // born at t_n (Verlet): the second half kick
            int side = drift(N, K.dtdx, qc, qf, cvz, cn, fn, err);
            if (side < 0) {
                store_rec<T>(S.sc, S.sp_, ridx, Part<T>{cn, fn, cvx, cvy, cvz});
                dep_add(sH, cn, cic_F(fn), threadIdx.x & 31);
                out |= 2u;
            } else {
                atomicAdd(&sC[CNT_ABS + side], 1u);
            }
            if (!S.leapfrog) ivz = fma_(K.K[1], q.ef, ivz);
            side = drift(N, K.dtdx, qc, qf, ivz, cn, fn, err);
            if (side < 0) {
                store_rec<T>(S.bc, S.bp, ridx, Part<T>{cn, fn, ivx, ivy, ivz});
                hist_add(Dother, cn, cic_F(fn));
                out |= 4u;
            } else {
                atomicAdd(&sC[CNT_ABS + 2 + side], 1u);
            }
        }
    } else {
        const U4 r = rs.draw(slot, 0);
        const U4 q1 = rs.draw(slot, 1);
        float a0, a1, a2, a3;
        box_muller(u01(q1.x), u01(q1.y), a0, a1);
        box_muller(u01(q1.z), u01(q1.w), a2, a3);
        const T vnx = mul_(K.sig_n, (T)a0), vny = mul_(K.sig_n, (T)a1), vnz = mul_(K.sig_n, (T)a2);
        const T gx = sub_(vx, vnx), gy = sub_(vy, vny), gz = sub_(vz, vnz);
        const T g2 = fma_(gx, gx, fma_(gy, gy, mul_(gz, gz)));
        const T xi = mul_(g2, K.kappa_i);
        const Row2* Ti = reinterpret_cast<const Row2*>(S.Ti);
        T C0, C1;
        if (!(xi < (T)(S.n_pts - 1))) {
            const Row2 a = Ti[S.n_pts - 1];
            C0 = a.x; C1 = a.y;
            atomicAdd(&sC[CNT_CLAMP + 1], 1u);
        } else {
            const int i = (int)xi;
            const T fr = sub_(xi, (T)i);
            const Row2 a = Ti[i], b = Ti[i + 1];
            C0 = fma_(fr, sub_(b.x, a.x), a.x);
            C1 = fma_(fr, sub_(b.y, a.y), a.y);
        }
        const T R = mul_((T)u01(r.y), K.kmax_i);
        if (R < C0) {  // isotropic in the centre-of-mass frame, equal masses
            const T hg = mul_((T)0.5, sqrt_(g2));
            T nx, ny, nz;
            iso_dir(u01(r.z), u01(r.w), nx, ny, nz);
            vx = fma_(hg, nx, mul_(add_(vx, vnx), (T)0.5));
            vy = fma_(hg, ny, mul_(add_(vy, vny), (T)0.5));
            vz = fma_(hg, nz, mul_(add_(vz, vnz), (T)0.5));
            atomicAdd(&sC[CNT_COLL_I + 0], 1u);
        } else if (R < C1) {  // backward: the ion takes the atom's velocity
            vx = vnx;
            vy = vny;
            vz = vnz;
            atomicAdd(&sC[CNT_COLL_I + 1], 1u);
        }
    }
    q.vx = vx;
    q.vy = vy;
    q.vz = vz;
    return out;
}

// Secondary electron of an ion absorbed at electrode `side` (added option).
template <typename T>
__device__ __forceinline__ bool emit_see(const Seg<T>& S, unsigned long long* Dother, uint32_t slot, const Stream& rs,
                                      int side, Part<T>& p, unsigned* sC) {
    const Consts<T>& K = S.k;
    const U4 w = rs.draw(slot, 3);
    if (!((T)u01(w.x) < K.gamma)) return false;
    const T vn = mul_(K.sig_see_n, (T)__fsqrt_rn(-own_logf(u01(w.y))));
    float t0, t1;
    box_muller(u01(w.z), u01(w.w), t0, t1);
    const int ce = side == 0 ? 0 : S.N - 1;
    const T fe = side == 0 ? (T)0 : one_minus_ulp<T>();
    p = Part<T>{ce, fe, mul_(K.sig_see, (T)t0), mul_(K.sig_see, (T)t1), side == 0 ? vn : -vn};
    hist_add(Dother, ce, cic_F(fe));
    atomicAdd(&sC[CNT_SEE], 1u);
    atomicAdd(&sC[CNT_SEE_SIDE + side], 1u);
    return true;
}

// Newborn compaction of a round: every lane's record src (where `on`) to dst <= src of the same buffer. All
// lanes of the warp call. One lane's destination may be another's source, so all of them load before any
// stores.
template <typename T>
__device__ __forceinline__ void compact_recs(int32_t* c, void* p, bool on, unsigned src, unsigned dst) {
    using R = typename Rec<T>::type;
    R* pp = reinterpret_cast<R*>(p);
    const bool move = on && src != dst;
    int cv = 0;
    R rv{};
    if (move) {
        cv = c[src];
        rv = pp[src];
    }
    __syncwarp();
    if (move) {
        c[dst] = cv;
        pp[dst] = rv;
    }
}

// n mod m and n / m for step numbers (32-bit operations below 2^31, the slow 64-bit ones out of line).
__device__ __noinline__ int mod_slow(long long n, int m) { return (int)(n % m); }
__device__ __noinline__ long long div_slow(long long n, int m) { return n / m; }
__device__ __forceinline__ int step_mod(long long n, int m) { return n >> 31 ? mod_slow(n, m) : (int)((unsigned)n % (unsigned)m); }
__device__ __forceinline__ long long step_div(long long n, int m) { return n >> 31 ? div_slow(n, m) : (unsigned)n / (unsigned)m; }

// Store totals after a sweep, for discharge d, by one warp of k_post: from the slice sums of parity
// par, the new counts and the layout of the output buffer (the sweep's chunks become its regions,
// the newborns its dense part at R0); on a full step the per-period mean counts; then the slice
// sums of the other parity cleared for the next sweep.
__device__ __forceinline__ void store_totals(const Disc& D, int d, Ctl* ctl, int lane, int par, bool full_step,
                                             int out_buf, int& err) {
    long long chunks[2], slices[2];
    for (int sp = 0; sp < 2; ++sp) {
        chunks[sp] = ctl->chunks_in[d][sp];
        slices[sp] = (chunks[sp] + SLICE - 1) / SLICE;
    }
    const unsigned* T0 = D.slice_tot[0] + (size_t)par * 3 * D.slice_n[0];
    const unsigned* T1 = D.slice_tot[1] + (size_t)par * 3 * D.slice_n[1];
    // survivors of both sweeps, ionization electrons and ions of the electron sweep, SEE electrons
    long long main0 = 0, main1 = 0, same0 = 0, see = 0, ions = 0;
    for (long long k = lane; k < max(slices[0], slices[1]); k += 32) {
        if (k < slices[0]) {
            main0 += __ldcg(T0 + 3 * k + 0);
            ions += __ldcg(T0 + 3 * k + 1);
            same0 += __ldcg(T0 + 3 * k + 2);
        }
        if (k < slices[1]) {
            main1 += __ldcg(T1 + 3 * k + 0);
            see += __ldcg(T1 + 3 * k + 1);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        main0 += __shfl_xor_sync(FULL, main0, o);
        main1 += __shfl_xor_sync(FULL, main1, o);
        same0 += __shfl_xor_sync(FULL, same0, o);
        see += __shfl_xor_sync(FULL, see, o);
        ions += __shfl_xor_sync(FULL, ions, o);
    }
    for (int sp = 0; sp < 2; ++sp) {
        const long long main_total = sp == 0 ? main0 : main1;
        const long long nb = sp == 0 ? same0 + see : ions;
        const long long bcap = D.bcap;
        const long long nbk = nb < bcap ? nb : bcap;
        const long long ch = chunks[sp];
        long long n_new = main_total + nbk;
        if (lane == 0) {
            if (nb > bcap) err |= ERR_CAPACITY;
            // more regions than the next sweep has output regions for: a sort or a repack is overdue
            if (ch > D.rmax[sp]) err |= ERR_CAPACITY;
            D.start[sp][ch] = (int)main_total;
            if (n_new > D.cap[sp]) {
                err |= ERR_CAPACITY;
                n_new = D.cap[sp];
            }
            ctl->count[d][sp] = n_new;
            Lay& L = ctl->lay[d][sp][out_buf];
            L.K = (int)ch;
            L.M = main_total;
            L.D0 = D.R0[sp];
            if (full_step) {  // per-period mean counts (steady-state criterion)
                const long long n_step = ctl->step;  // this step is n; the counts belong to n+1
                ctl->period_acc[d][sp] += (double)n_new;
                if (D.steps_per_period > 0 && step_mod(n_step + 1, D.steps_per_period) == 0) {
                    const long long per = step_div(n_step + 1, D.steps_per_period) - 1;
                    D.period_mean[(per % PERIOD_HIST) * 2 + sp] = ctl->period_acc[d][sp] / D.steps_per_period;
                    ctl->period_acc[d][sp] = 0.0;
                }
            }
        }
        // the next sweep adds into the other parity
        unsigned* Tn = D.slice_tot[sp] + (size_t)(par ^ 1) * 3 * D.slice_n[sp];
        for (int k = lane; k < 3 * D.slice_n[sp]; k += 32) Tn[k] = 0;
    }
}

// Bulk copies into shared memory (the asynchronous copy engine) with an mbarrier per buffer.
__device__ __forceinline__ unsigned smem_u32(const void* p) { return static_cast<unsigned>(__cvta_generic_to_shared(p)); }
__device__ __forceinline__ void mbar_init(unsigned long long* mb) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(mb)) : "memory");
}
__device__ __forceinline__ void mbar_expect(unsigned long long* mb, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(mb)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, unsigned bytes, unsigned long long* mb) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(mb))
                 : "memory");
}
// Waits for phase `parity` of the barrier to complete, at most `tries` polls (each poll may block
// for a hardware-defined time); false if it gave up.
constexpr int MBAR_TRIES = 1 << 20;
__device__ __forceinline__ bool mbar_wait(unsigned long long* mb, unsigned parity, int tries = MBAR_TRIES) {
    const unsigned a = smem_u32(mb);
    for (int it = 0; it < tries; ++it) {
        unsigned done;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(a), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}
// The same by a whole warp, with one answer for all its lanes: true only if none gave up (what follows is full
// of warp-wide operations, so no lane may take another way than the rest).
__device__ __forceinline__ bool warp_wait(unsigned long long* mb, unsigned parity, int tries = MBAR_TRIES) {
    return __all_sync(FULL, mbar_wait(mb, parity, tries));
}

// Dynamic shared memory of the sweep: per cell the field and its difference to the next node (E_c,
// E_{c+1} - E_c), the histograms (`sets` 2: both species at once, 5 + 3 arrays; 1: one species at a
// time, 5 arrays) and their windows, per warp two staging buffers of one chunk (records, then cells) and its candidate
// queue, per store its layout, per species the chunk prefix over the discharges.
struct alignas(16) StoreSnap {
    int K, M, D0, n;
    const int* start;  // of the input buffer
    const void* rec;
    const int32_t* cell;
    long long pad_;
};
template <typename T, int PPT>
__host__ __device__ constexpr unsigned sweep_stage_bytes() {  // one buffer of one warp
    return 32u * PPT * (sizeof(typename Rec<T>::type) + 4);
}
__host__ __device__ constexpr int sweep_hist_words(int sets) { return sets == 2 ? 8 : 5; }
template <typename T>
__host__ __device__ constexpr unsigned sweep_hist_offset(int max_N) { return (2u * sizeof(T) * max_N + 15) / 16 * 16; }
template <typename T>
__host__ __device__ constexpr unsigned sweep_stage_offset(int max_N, int sets) {
    return (sweep_hist_offset<T>(max_N) + 4u * sweep_hist_words(sets) * (max_N + WWORDS) + 127) / 128 * 128;
}
template <typename T, int PPT>
__host__ __device__ constexpr unsigned sweep_smem(int max_N, int sets, int warps, int n_disc) {
    return sweep_stage_offset<T>(max_N, sets) + (unsigned)warps * (2 * sweep_stage_bytes<T, PPT>() + 32 * PPT) +
           (unsigned)sizeof(StoreSnap) * 2 * n_disc + 4u * 2 * (n_disc + 1);
}

constexpr unsigned SWEEP_SMEM_LIMIT = 227 * 1024 - 4096;  // dynamic shared memory; the static part is below 4 KB

// Threads of a sweep CTA at most (one CTA per SM): the FP32 chunk code takes 80 registers (24 warps), the
// FP64 code 128 (16 warps).
template <typename T>
__host__ __device__ constexpr int sweep_max_threads() { return sizeof(T) == 4 ? 768 : 512; }

// ---------------------------------------------------------------------------
// The sweep. One persistent CTA per SM. The chunks of all electron stores and those of all ion stores
// are split evenly over the CTAs (CTA b takes the contiguous chunks [total b / G, total (b+1) / G) of
// each list), and each CTA's part of a store over its warps, again contiguous. So a CTA meets few
// stores, its deposits few cells, and consecutive chunks of a warp share a candidate call.
// A chunk's records and cells arrive in the warp's staging buffer by a bulk copy issued while the warp
// worked on its previous chunk; the warp draws the chunk's candidate words and queues the candidates in
// slot order; collides them (32 at a time, the final velocity written back into the staged record, the
// staged cell marked COLLIDED); then takes all particles in one pass: gather, half kicks, energy moment,
// drift, walls, deposit, survivors in slot order to the chunk's own output region [CHUNK cs, ...), cs the
// chunk index. Newborns go in parent-slot order to the chunk's regions of the newborn buffers (same
// species: ionization electrons; other species: ionization ions, or SEE electrons of the ion sweep), and
// the chunk records the three counts. The CTA synchronises only between discharges (with one histogram
// set, between stores) and for a flush of its histograms.
//
// What bounds it: instruction issue, then the shared-memory atomics; for a store of a few chunks per SM
// the latency of one chunk (cold instructions, table look-ups, 40 % of it the collisions). Measured, with
// the FP32 chunk of 128 slots at 80 registers and 24 warps (32 warps at 64 registers spill: 40.5 against
// 35.7 us a step at 1e6 + 1e6 and 392 against 320 at 1.2e7 + 1.2e7): 31 us a launch at 1e6 + 1e6
// particles, 512 cells (before: one CTA of 8 warps per 1024 slots, three passes over a chunk and a gather
// in each, 40 us), 262 at 1.2e7 + 1.2e7, 2048 cells (372), 58 for 64 discharges of 2e4 + 2e4 in one launch
// (109), FP64 at 1e6 + 1e6 90 (150).
template <typename T, int PPT>
__global__ void __launch_bounds__(sweep_max_threads<T>(), 1)
    k_sweep(const Disc* __restrict__ discs, int n_disc, Ctl* __restrict__ ctl, int in_buf, unsigned long long seed,
            int max_N, int sets, unsigned hi) {
    using R = typename Rec<T>::type;
    using T2 = typename T4<T>::two;
    constexpr int CHUNK = 32 * PPT;
    constexpr unsigned REC_BYTES = CHUNK * sizeof(R), CELL_BYTES = CHUNK * 4;
    constexpr int COLLIDED = 1 << 30;  // mark in a staged cell: the record holds the particle's final velocity
    constexpr int MAXW = sweep_max_threads<T>() / 32;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nthr = blockDim.x, NW = nthr >> 5;
    T2* s_E = reinterpret_cast<T2*>(smem_raw);
    unsigned* s_win = reinterpret_cast<unsigned*>(smem_raw + sweep_hist_offset<T>(max_N));  // 16-byte aligned
    unsigned* s_h = s_win + sweep_hist_words(sets) * WWORDS;
    unsigned char* s_stage = smem_raw + sweep_stage_offset<T>(max_N, sets);
    unsigned char* stage = s_stage + (unsigned)warp * 2 * sweep_stage_bytes<T, PPT>();
    unsigned char* s_queue = s_stage + (unsigned)NW * 2 * sweep_stage_bytes<T, PPT>();
    uint8_t* Q = s_queue + warp * CHUNK;  // the chunk indices of the candidates, in slot order (CHUNK <= 256)
    StoreSnap* s_store = reinterpret_cast<StoreSnap*>(s_queue + NW * CHUNK);
    int* s_pre = reinterpret_cast<int*>(s_store + 2 * n_disc);  // [species][n_disc + 1]
    // [node], behind everything else (0: none)
    unsigned* const s_hi = hi ? reinterpret_cast<unsigned*>(smem_raw + hi) : nullptr;

    __shared__ Seg<T> s_seg[2];
    __shared__ long long s_step;
    __shared__ int s_par, s_dpar;  // parities of the slice sums and of the deposits
    __shared__ unsigned s_cnt[NCNT];
    __shared__ int s_err;
    __shared__ unsigned long long s_mbar[MAXW][2];
    __shared__ int2 s_range[2 * MAXD];
    __shared__ unsigned s_mask[4];
    __shared__ int s_w0[2];  // first cell of each species' window

    if (lane == 0) {
        mbar_init(&s_mbar[warp][0]);
        mbar_init(&s_mbar[warp][1]);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // the two stores' constants of discharge d
    auto load_seg = [&](int d) {
        const unsigned* src = reinterpret_cast<const unsigned*>(segs_of<T>(discs[d]));
        unsigned* dst = reinterpret_cast<unsigned*>(s_seg);
        for (int j = tid; j < (int)(sizeof(s_seg) / 4); j += nthr) dst[j] = __ldg(src + j);
    };
    if (tid == 0) s_err = 0;
    if (tid < NCNT) s_cnt[tid] = 0;
    load_seg(0);  // of a context with one discharge: nothing more to fetch after the wait
    for (int j = tid; j < sweep_hist_words(sets) * (max_N + WWORDS); j += nthr) s_win[j] = 0;
    for (int j = tid; hi && j <= max_N; j += nthr) s_hi[j] = 0;
    __syncthreads();
    grid_dep_sync();
    auto load_field = [&]() {
        const T* E = reinterpret_cast<const T*>(s_seg[0].E);
        const int N = s_seg[0].N;
        for (int j = tid; j < N; j += nthr) {
            const T e0 = __ldcg(E + j), e1 = __ldcg(E + j + 1);
            T2 v;
            v.x = e0;
            v.y = sub_(e1, e0);
            s_E[j] = v;
        }
    };
    // every store's layout; 31 bits hold slots, chunks and record offsets (the host caps the buffers)
    const int n_store = 2 * n_disc;
    for (int s = tid; s < n_store; s += nthr) {
        const int d = s >> 1, sp = s & 1;
        const Lay L = ctl->lay[d][sp][in_buf];
        const long long n = ctl->count[d][sp];
        long long ch = chunks_of(L, n, CHUNK);
        if (ch > discs[d].ralloc[sp]) {  // more chunks than output regions: reported, the rest dropped
            ch = discs[d].ralloc[sp];
            if (blockIdx.x == 0) atomicOr(&s_err, ERR_CAPACITY);
        }
        const Seg<T>& G = segs_of<T>(discs[d])[sp];
        s_store[s] = StoreSnap{L.K, (int)L.M, (int)L.D0, (int)n, G.start, G.p[in_buf], G.c[in_buf], 0};
        if (blockIdx.x == 0) ctl->chunks_in[d][sp] = (int)ch;  // read by the post-sweep grid
        s_pre[sp * (n_disc + 1) + d + 1] = (int)ch;
        if (d == 0) s_pre[sp * (n_disc + 1)] = 0;
    }
    if (tid == 0) {
        s_step = ctl->step;
        s_par = ctl->slice_par;
        s_dpar = ctl->dep_par;
    }
    if (n_disc == 1) load_field();
    if (n_disc > 1) {  // inclusive prefix over at most 64 discharges: warp sp takes its species, two per lane
        __syncthreads();
        if (warp < 2) {
            int* p = s_pre + warp * (n_disc + 1) + 1;
            const int v0 = 2 * lane < n_disc ? p[2 * lane] : 0, v1 = 2 * lane + 1 < n_disc ? p[2 * lane + 1] : 0;
            int x = v0 + v1;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(FULL, x, o);
                if (lane >= o) x += y;
            }
            if (2 * lane < n_disc) p[2 * lane] = x - v1;
            if (2 * lane + 1 < n_disc) p[2 * lane + 1] = x;
        }
        __syncthreads();
    }
    // this CTA's chunks [lo, hi) of every store (electrons and ions of a discharge in turn) and the bits
    // of the stores it has any of
    auto take = [&](int t) {  // warp-uniform trip counts: every lane calls
        int lo = 0, hi = 0;
        if (t < n_store) {
            const int* p = s_pre + (t & 1) * (n_disc + 1);
            const unsigned tot = (unsigned)p[n_disc], G = gridDim.x, b = blockIdx.x;
            const unsigned w = tot / G, x = tot - w * G;  // the first x CTAs take w + 1 chunks
            const int r0 = (int)(b * w + min(b, x)), r1 = r0 + (int)(w + (b < x ? 1 : 0));
            const int p0 = p[t >> 1], p1 = p[(t >> 1) + 1];
            lo = min(max(r0, p0), p1) - p0;
            hi = min(max(r1, p0), p1) - p0;
            s_range[t] = make_int2(lo, hi);
        }
        const unsigned m = __ballot_sync(FULL, hi > lo);
        if (lane == 0) s_mask[t >> 5] = m;
    };
    if (n_disc == 1) {
        if (warp == 0) {
            __syncwarp();
            take(lane);
        }
    } else {
        for (int t = tid; t < 2 * MAXD; t += nthr) take(t);
    }
    __syncthreads();
    const long long step = s_step;
    // the next store after s (-1: the first) that this CTA has chunks of, n_store if none
    auto next_store = [&](int s) {
        ++s;
        unsigned m = s < n_store ? s_mask[s >> 5] >> (s & 31) : 0u;
        if (m) return s + __ffs(m) - 1;
        for (int w = (s >> 5) + 1; 32 * w < n_store; ++w)
            if (s_mask[w]) return 32 * w + __ffs(s_mask[w]) - 1;
        return n_store;
    };
    // this warp's part of them; the ions in the opposite warp order, so that a warp with one chunk more
    // of one species tends to have one less of the other
    auto warp_range = [&](int s, int& lo, int& hi) {
        const int2 r = s_range[s];
        const unsigned w = (s & 1) ? NW - 1 - warp : warp, m = r.y - r.x, q = m / NW, x = m % NW;
        lo = r.x + (int)(w * q + min(w, x));
        hi = lo + (int)(q + (w < x ? 1 : 0));
    };

    // the chunk whose copy is in flight (or landed) in buffer pf_b: its store (n_store: none), index,
    // the warp's last chunk of that store, first and end slot
    int pf_s = -1, pf_k = 0, pf_end = 0, pf_base = 0, pf_stop = 0, pf_b = 1;
    unsigned phases = 0;  // bit b: phase of buffer b's barrier the next wait expects
    auto prefetch_next = [&]() {
        ++pf_k;
        while (pf_k >= pf_end) {
            pf_s = next_store(pf_s);
            if (pf_s >= n_store) return;
            warp_range(pf_s, pf_k, pf_end);
        }
        pf_b ^= 1;
        const StoreSnap& ss = s_store[pf_s];
        unsigned src;
        if (pf_k < ss.K) {
            src = (unsigned)pf_k * CHUNK;
            const int* st = ss.start + pf_k;
            pf_base = __ldcg(st);
            pf_stop = __ldcg(st + 1);
        } else {
            const int j = (pf_k - ss.K) * CHUNK;
            src = (unsigned)(ss.D0 + j);
            pf_base = ss.M + j;
            pf_stop = min(ss.n, pf_base + CHUNK);
        }
        if (lane == 0) {
            unsigned char* buf = stage + (unsigned)pf_b * sweep_stage_bytes<T, PPT>();
            unsigned long long* mb = &s_mbar[warp][pf_b];
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // earlier reads and writes of the buffer
            mbar_expect(mb, REC_BYTES + CELL_BYTES);
            bulk_g2s(buf, static_cast<const R*>(ss.rec) + src, REC_BYTES, mb);
            bulk_g2s(buf + REC_BYTES, ss.cell + src, CELL_BYTES, mb);
        }
    };
    prefetch_next();

    const unsigned lt = (1u << lane) - 1u;
    int err = 0, cur_d = -1;
    unsigned sumA = 0, sumB = 0, sumS = 0;  // survivors and newborns since the last add to the slice sums
    unsigned carry = 0, carry_q = 0xFFFFFFFFu;  // candidate bits of the last call of the warp's previous chunk

    // One warp's chunk of the store of species SP (see above).
    auto chunk = [&](unsigned cs, int base, int cnt, R* srec, int32_t* scell, auto spc) { constexpr int SP = decltype(spc)::value;
        const Seg<T>& S = s_seg[SP];
        const int h0 = SP == 1 && sets == 2 ? 5 : 0;
        const Hist h{s_h + h0 * max_N, s_win + h0 * WWORDS, max_N, s_w0[SP]};
        const unsigned obase = cs * CHUNK;
        unsigned offA = obase, offB = obase, offS = obase;  // output cursors of the chunk's regions
        const int N = S.N;
        const T Ksp = S.k.K[SP];
        const Stream rs{seed, (uint32_t)step, ((uint32_t)((unsigned long long)step >> 32) & 0xFFFFu) << 16 | (uint32_t)SP << 8,
                        S.did};
        if (cnt > 0) {
            // ---- candidates. Slots 4q..4q+3 take the four words of one Philox call (call 4, counter
            // word 0 = q) and are candidates where a word is below the threshold. The chunk needs the
            // calls q0 .. (base + cnt - 1) / 4; the first is the previous chunk's last one when that
            // chunk's slots run into this one's, so its bits are carried over and 32 calls cover 128
            // slots at any alignment.
            constexpr int NG = (CHUNK / 4 + 1 + 31) / 32;
            const unsigned q0 = (unsigned)base >> 2;
            const int al = base & 3;
            const int ncalls = (int)(((unsigned)base + cnt - 1) >> 2) - (int)q0 + 1;
            const int sh = carry_q == q0 ? 1 : 0;
            int qn = 0;
            if (sh) {  // words al.. of the carried call: chunk indices 0..3 - al
                const unsigned cm = (carry >> al) & ((1u << min(cnt, 4 - al)) - 1u);
                if (cm) {
                    if (lane < 4 && ((cm >> lane) & 1u)) Q[__popc(cm & lt)] = (uint8_t)lane;
                    qn = __popc(cm);
                }
            }
            const int li = ncalls - 1 - sh;  // the last call is drawn by lane li % 32 of group li / 32
            unsigned next = carry;
#pragma unroll
            for (int m = 0; m < NG; ++m)
                if (32 * m <= li) {
                    const U4 w = rs.draw(q0 + sh + lane + 32 * m, 4);
                    const uint32_t thr = S.thr;
                    unsigned nib = (w.x < thr ? 1u : 0u) | (w.y < thr ? 2u : 0u) | (w.z < thr ? 4u : 0u) |
                                   (w.w < thr ? 8u : 0u);
                    if ((li >> 5) == m) next = __shfl_sync(FULL, nib, li & 31);
                    // word k is chunk index i0 + k; only those in [0, cnt) count
                    const int i0 = 4 * (lane + sh + 32 * m) - al;
                    if (i0 < 0) nib &= 0xFu << -i0;
                    const int left = cnt - i0;
                    if (left < 4) nib = left > 0 ? nib & ((1u << left) - 1u) : 0u;
                    if (__any_sync(FULL, nib != 0)) {
                        const unsigned b0 = __ballot_sync(FULL, nib & 1u), b1 = __ballot_sync(FULL, nib & 2u),
                                       b2 = __ballot_sync(FULL, nib & 4u), b3 = __ballot_sync(FULL, nib & 8u);
                        int pos = qn + __popc(b0 & lt) + __popc(b1 & lt) + __popc(b2 & lt) + __popc(b3 & lt);
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            if ((nib >> k) & 1u) Q[pos++] = (uint8_t)(i0 + k);
                        qn += __popc(b0) + __popc(b1) + __popc(b2) + __popc(b3);
                    }
                }
            carry = next;
            carry_q = q0 + ncalls - 1;
            // ---- the candidates' collisions, 32 at a time; newborns in queue (= slot) order
            if (qn) __syncwarp();
            for (int r0 = 0; r0 < qn; r0 += 32) {
                const int q = r0 + lane;
                uint32_t o = 0;
                const int i = Q[min(q, qn - 1)];
                const int c0 = scell[i];
                const bool cand = q < qn && (unsigned)c0 < (unsigned)N;  // a corrupt cell is dropped and reported below
                const int c = cand ? c0 : 0;
                R rec = srec[i];
                const T2 e = s_E[c];
                const T ef = fma_(rec.x, e.y, e.x);
                const T vzn = fma_(Ksp, ef, rec.w);  // v_n
                if (SP == 0)
                    energy_add<T>(h, s_hi, S.Qg, cand, c, rec.x, fma_(rec.y, rec.y, fma_(rec.z, rec.z, mul_(vzn, vzn))),
                                  S.k.kappa_E, lane);
                if (cand) {
                    Cand<T> v{ef, rec.y, rec.z, S.leapfrog ? fma_(Ksp, ef, vzn) : vzn};  // leapfrog: at v_{n+1/2}
                    o = collide<T>(S, SP, S.Dother + s_dpar * (N + 1), v, c, rec.x, (uint32_t)base + i, obase + q, rs, h, s_cnt, err);
                    rec.y = v.vx;
                    rec.z = v.vy;
                    rec.w = S.leapfrog ? v.vz : fma_(Ksp, ef, v.vz);  // the second half kick
                    srec[i] = rec;
                    scell[i] = c | COLLIDED;
                }
                __syncwarp();
                const unsigned mc = __ballot_sync(FULL, cand);
                if (lane == 0 && mc) atomicAdd(&s_cnt[CNT_CAND + SP], (unsigned)__popc(mc));
                if (SP == 0) {  // the round's newborns, from the candidates' ranks to parent-slot order (dst <= src)
                    const unsigned m1 = __ballot_sync(FULL, (o & 2u) != 0), m2 = __ballot_sync(FULL, (o & 4u) != 0);
                    if (m1 | m2) {
                        compact_recs<T>(S.sc, S.sp_, (o & 2u) != 0, obase + q, offS + __popc(m1 & lt));
                        compact_recs<T>(S.bc, S.bp, (o & 4u) != 0, obase + q, offB + __popc(m2 & lt));
                        offS += __popc(m1);
                        offB += __popc(m2);
                        __syncwarp();
                    }
                }
            }
            if (qn) __syncwarp();
            // ---- all particles: gather, half kicks, energy moment, drift, walls, deposit, survivors
            const T dtdx = S.k.dtdx, kE = S.k.kappa_E;
            int32_t* __restrict__ cout = S.c[1 - in_buf];
            void* pout = S.p[1 - in_buf];
            int c_next = scell[lane];
            R r_next = srec[lane];
#pragma unroll 1
            for (int k = 0; k < PPT; ++k) {
                if (32 * k >= cnt) break;
                const int i = 32 * k + lane, craw = c_next;
                const R r = r_next;
                if (k + 1 < PPT) {  // the next row's loads, before this row's atomics
                    c_next = scell[i + 32];
                    r_next = srec[i + 32];
                }
                // branch-free for the common case: a lane without a particle computes on cell 0 and
                // takes no part in the atomics and stores; rare cases behind warp votes
                const bool coll = (craw & COLLIDED) != 0, in = i < cnt;
                const int c0 = craw & ~COLLIDED;
                const bool valid = in && (unsigned)c0 < (unsigned)N;
                const int c = valid ? c0 : 0;
                const T2 e = s_E[c];
                const T ef = fma_(r.x, e.y, e.x);
                const T vzn = fma_(Ksp, ef, r.w);  // v_n
                if (SP == 0)
                    energy_add<T>(h, s_hi, S.Qg, valid && !coll, c, r.x, fma_(r.y, r.y, fma_(r.z, r.z, mul_(vzn, vzn))), kE,
                                  lane);
                const T vz = coll ? r.w : fma_(Ksp, ef, vzn);
                int cn;
                T fn, s;
                const bool alive = drift_fast(N, dtdx, c, r.x, vz, cn, fn, s) && valid;
                const unsigned mA = __ballot_sync(FULL, alive);
                if (mA != (cnt - 32 * k < 32 ? (1u << (cnt - 32 * k)) - 1u : FULL)) {  // some left the gap
                    bool see = false;
                    Part<T> Pse{};
                    if (in && !alive) {
                        if (!valid || !(s == s)) err |= ERR_NONFINITE;  // a corrupt cell index is dropped too
                        if (valid) {
                            const int side = s >= (T)0 ? 1 : 0;
                            atomicAdd(&s_cnt[CNT_ABS + 2 * SP + side], 1u);
                            if (SP == 1 && S.has_see)
                                see = emit_see<T>(S, S.Dother + s_dpar * (N + 1), (uint32_t)base + i, rs, side, Pse, s_cnt);
                        }
                    }
                    if (SP == 1) {
                        const unsigned mB = __ballot_sync(FULL, see);
                        if (see) store_rec<T>(S.bc, S.bp, offB + __popc(mB & lt), Pse);
                        offB += __popc(mB);
                    }
                    __syncwarp();
                }
                warp_dep<SP == 1>(h, alive ? cn : -1, cic_F(fn), lane);
                if (alive) store_rec<T>(cout, pout, offA + __popc(mA & lt), Part<T>{cn, fn, r.y, r.z, vz});
                offA += __popc(mA);
            }
        }
        sumA += offA - obase;
        sumB += offB - obase;
        sumS += offS - obase;
        if (lane == 0) {
            S.cnt_main[cs] = (int)(offA - obase);
            S.cnt_birth[cs] = (int)(offB - obase);
            if (SP == 0) S.cnt_same[cs] = (int)(offS - obase);
        }
        // the slice sums once per run of the warp's chunks in a slice
        if (pf_s != 2 * cur_d + SP || (cs + 1) % SLICE == 0) {
            if (lane == 0) {
                unsigned* sl = S.slice_tot + s_par * S.slice_stride + 3 * (cs / SLICE);
                if (sumA) atomicAdd(&sl[0], sumA);
                if (sumB) atomicAdd(&sl[1], sumB);
                if (sumS) atomicAdd(&sl[2], sumS);
            }
            sumA = sumB = sumS = 0;
        }
    };

    // Adds the CTA's histograms and counters to the global sums of the current discharge and clears them.
    auto flush = [&](int sp_cur) {
        __syncthreads();
        const int N = s_seg[0].N;
        const bool folds = s_w0[0] != NO_WIN || s_w0[1] != NO_WIN;
        for (int k = tid; folds && k < sweep_hist_words(sets) * WIN; k += nthr) {  // fold and clear the windows
            const int a = k / WIN, j = k % WIN, sp = sets == 2 ? a >= 5 : sp_cur;
            uint4* w = reinterpret_cast<uint4*>(s_win + a * WWORDS + j * WCOP);  // all zero without a window
            const uint4 x = w[0], y = w[1];
            const unsigned v = x.x + x.y + x.z + x.w + y.x + y.y + y.z + y.w;
            if (v) {
                s_h[a * max_N + s_w0[sp] + j] += v;
                w[0] = w[1] = make_uint4(0u, 0u, 0u, 0u);
            }
        }
        if (folds) __syncthreads();
        for (int sp = 0; sp < 2; ++sp) {
            if (sets == 1 && sp != sp_cur) continue;
            unsigned* h = s_h + (sp == 1 && sets == 2 ? 5 * max_N : 0);
            unsigned long long* Dg = s_seg[sp].Dg + s_dpar * (N + 1);
            for (int j = tid; j <= N; j += nthr) {
                unsigned long long v = 0, q = 0;
                if (j < N) {
                    v = ((unsigned long long)h[j] << 32) -
                        ((unsigned long long)h[j + max_N] + ((unsigned long long)h[j + 2 * max_N] << 16));
                    if (sp == 0) q = (unsigned long long)h[j + 3 * max_N] - h[j + 4 * max_N];
                }
                if (j > 0) {
                    v += (unsigned long long)h[j - 1 + max_N] + ((unsigned long long)h[j - 1 + 2 * max_N] << 16);
                    if (sp == 0) q += h[j - 1 + 4 * max_N];
                }
                if (sp == 0 && hi) q += (unsigned long long)s_hi[j] << 17;
                if (v) atomicAdd(&Dg[j], v);
                if (sp == 0 && q) atomicAdd(&s_seg[0].Qg[j], q);
            }
        }
        if (tid < NCNT && s_cnt[tid]) atomicAdd(&s_seg[0].cnt[tid], (unsigned long long)s_cnt[tid]);
    };
    auto clear = [&]() {
        __syncthreads();
        for (int j = tid; j < sweep_hist_words(sets) * max_N; j += nthr) s_h[j] = 0;  // the windows: in the flush
        for (int j = tid; hi && j <= max_N; j += nthr) s_hi[j] = 0;
        if (tid < NCNT) s_cnt[tid] = 0;
        __syncthreads();
    };

    const int flush_rounds = max(1, flush_particles<T>() / (NW * CHUNK));
    int cur_sp = 0;
    for (int s = next_store(-1); s < n_store; s = next_store(s)) {
        const int d = s >> 1, sp = s & 1;
        if (cur_d >= 0 && (d != cur_d || sets == 1)) {
            flush(cur_sp);
            clear();
        }
        if (d != cur_d) {
            if (n_disc > 1) {
                load_seg(d);
                __syncthreads();
            }
            const int N = s_seg[0].N;
            if (lane == 0 && warp < 2) {  // the species' window: around the first cells of the CTA's first and
                const int q = warp;       // last chunk (any value is right)
                const int2 g = s_range[2 * d + q];
                int w0 = NO_WIN;
                if (g.y - g.x >= WIN_CHUNKS) {
                    const StoreSnap& ss = s_store[2 * d + q];
                    auto first_cell = [&](int k) {
                        return __ldcg(ss.cell +
                                      (k < ss.K ? (unsigned)k * CHUNK : (unsigned)(ss.D0 + (k - ss.K) * CHUNK)));
                    };
                    const int a = first_cell(g.x), b = first_cell(g.y - 1);
                    w0 = max(0, min((min(max(a, 0), N) + min(max(b, 0), N)) / 2 - WIN / 2, N - WIN));
                }
                s_w0[q] = w0;
            }
            if (n_disc > 1) load_field();
            __syncthreads();
            cur_d = d;
        }
        cur_sp = sp;
        carry_q = 0xFFFFFFFFu;
        const int rounds = (s_range[s].y - s_range[s].x + NW - 1) / NW;  // chunks of this store a warp has at most
        for (int r = 0, f = flush_rounds; r < rounds; ++r) {
            if (f-- == 0) {
                flush(cur_sp);
                clear();
                f = flush_rounds - 1;
            }
            if (pf_s != s) continue;
            const unsigned cs = (unsigned)pf_k;
            const int base = pf_base, cnt = pf_stop - pf_base, b = pf_b;
            if (!warp_wait(&s_mbar[warp][b], (phases >> b) & 1u)) {  // given up: the warp takes no more chunks
                err |= ERR_TIMEOUT;
                pf_s = n_store;
                continue;
            }
            phases ^= 1u << b;
            __syncwarp();
            prefetch_next();  // the warp's next chunk, into the other buffer
            unsigned char* buf = stage + (unsigned)b * sweep_stage_bytes<T, PPT>();
            R* srec = reinterpret_cast<R*>(buf);
            int32_t* scell = reinterpret_cast<int32_t*>(buf + REC_BYTES);
            if (sp == 0) chunk(cs, base, cnt, srec, scell, IC<0>{}); else chunk(cs, base, cnt, srec, scell, IC<1>{});
            __syncwarp();
        }
    }
    // a copy is in flight past this point only if its wait was given up (each one issued is of a chunk this warp
    // takes, and the next is issued after the wait): the one of buffer pf_b, waited for once more, with a limit
    if (err & ERR_TIMEOUT) mbar_wait(&s_mbar[warp][pf_b], (phases >> pf_b) & 1u);
    if (cur_d >= 0) flush(cur_sp);
    if (err) atomicOr(&s_err, err);
    __syncthreads();
    if (tid == 0 && s_err) atomicOr(&ctl->error, s_err);
}


// ---------------------------------------------------------------------------
// Exact prefix terms of the Poisson solve over a run of nodes, per species: r = sum of the deposits
// D_k, and the sum of k D_k in two 64-bit halves, a of the low and b of the high 32 bits of D_k (so no
// sum needs a carry chain). With R_j = sum_{1<=k<=j} D_k and M_j = sum_{1<=k<=j} k D_k = b 2^32 + a the
// double sum S_{j+1} = sum_{i<=j} R_i equals (j + 1) R_j - M_j, so one scan of plain integer sums gives
// both R and S (integer, so any order gives the same).
struct PSum {
    unsigned long long v[6];  // r of electrons, ions; a; b
    __device__ __forceinline__ void add(int j, unsigned long long de, unsigned long long di) {
        v[0] += de;
        v[1] += di;
        v[2] += (unsigned long long)j * (unsigned)de;
        v[3] += (unsigned long long)j * (unsigned)di;
        v[4] += (unsigned long long)j * (unsigned)(de >> 32);
        v[5] += (unsigned long long)j * (unsigned)(di >> 32);
    }
};
// Nearest double of a 128-bit integer below 2^115 in magnitude (two roundings at most).
__device__ __forceinline__ double i128_to_double(__int128 x) {
    const long long hi = (long long)(x >> 64);
    const unsigned long long lo = (unsigned long long)x;
    return __fma_rn((double)hi, 0x1p64, __ull2double_rn(lo));
}
// S at node j1 from the sums through node j1 - 1, in charge units: pr1 S_ions - pr0 S_electrons. Out of
// line: the grid runs once per step from a cold instruction cache, where a second copy costs more than
// the call.
__device__ __noinline__ double poisson_S(unsigned long long r0, unsigned long long r1, unsigned long long a0,
                                         unsigned long long a1, unsigned long long b0, unsigned long long b1, int j1,
                                         double pr0, double pr1) {
    const __int128 S0 = (__int128)((unsigned __int128)(unsigned)j1 * r0 - (((unsigned __int128)b0 << 32) + a0));
    const __int128 S1 = (__int128)((unsigned __int128)(unsigned)j1 * r1 - (((unsigned __int128)b1 << 32) + a1));
    return __fma_rn(pr1, i128_to_double(S1), -pr0 * i128_to_double(S0));
}
// After a sweep (mode bit 1) and for every solve, one grid (x = slice or role, y = store):
//   x < nsl          the region starts of the chunks of slice x of store y (the first slot each chunk's
//                    survivors take in the new layout) and its newborns, copied into the newborn area;
//   y even, x >= nsl the field of discharge y / 2 at the FIELD_NODES nodes of part x - nsl (every part
//                    scans all deposits; the FP64 work per node, slow on this part, is what is split);
//   y odd, x == nsl  the slice sums of discharge y / 2 into the new counts and layouts, the sums of the
//                    other parity cleared for the next sweep;
//   y odd, x > nsl   the moments of the nodes of part x - nsl - 1, and the deposits of the previous
//                    solve (the other deposit parity) cleared for the next sweep.
// mode bits: 1 layouts after a sweep; 2 accumulate moments and advance the step; 4 initial solve at t =
// n dt (load); 8 segments only (no solve, deposits kept). The last CTA to finish advances the step (mode
// bit 2) and flips the slice parity (mode bit 1) and the deposit parity (a solve).
template <int BLOCK>
__device__ __forceinline__ void seg_apply(const Disc* __restrict__ discs, Ctl* __restrict__ ctl, int out_buf, int tid, int lane,
                          int warp) {
    constexpr int K = SLICE / BLOCK, NW = BLOCK / 32;
    static_assert(SLICE % BLOCK == 0 && NW <= 32 && NW >= 3, "seg_apply block shape");
    using R = float4;
    __shared__ int s_w[3][NW];
    // the slice's chunk counts (each at most one chunk of slots: 16 bits), loaded coalesced while
    // every thread scans K consecutive chunks
    __shared__ unsigned short s_cnt[3][SLICE];
    const int d = blockIdx.y >> 1, sp = blockIdx.y & 1;
    const Disc& D = discs[d];
    // every field is read before the first store (the stores could otherwise alias them)
    const int CHUNK = D.chunk;
    const int* __restrict__ cnt_m = D.cnt_main[sp];
    const int* __restrict__ cnt_b = D.cnt_birth[sp];
    const int* __restrict__ cnt_s = D.cnt_same;
    int* __restrict__ st = D.start[sp];
    const int q = 1 - sp;  // store of the other-species newborns
    const long long bcap = D.bcap;
    const int rw = D.rec_words;  // record size in 16-byte words
    int32_t* __restrict__ oc_q = D.c[out_buf][q] + D.R0[q];
    R* __restrict__ op_q = reinterpret_cast<R*>(D.p[out_buf][q]) + D.R0[q] * rw;
    int32_t* __restrict__ oc_0 = D.c[out_buf][0] + D.R0[0];
    R* __restrict__ op_0 = reinterpret_cast<R*>(D.p[out_buf][0]) + D.R0[0] * rw;
    const int32_t* __restrict__ bc = D.bc[sp];
    const R* __restrict__ bp = reinterpret_cast<const R*>(D.bp[sp]);
    const int32_t* __restrict__ sc = D.sc;
    const R* __restrict__ spr = reinterpret_cast<const R*>(D.sp_);
    const unsigned* __restrict__ slice0 = D.slice_tot[0];
    const unsigned* __restrict__ slice_s = D.slice_tot[sp];
    const int sn0 = D.slice_n[0], sn_s = D.slice_n[sp];
    const long long chunks = ctl->chunks_in[d][sp];
    const long long t0 = (long long)blockIdx.x * SLICE;
    if (t0 >= chunks) return;
    // output offsets of this slice: the sums of the slices before it (survivors, other-species
    // newborns, same-species newborns); the ion sweep's SEE electrons follow all ionization
    // electrons of the electron sweep
    __shared__ long long s_pre[3];
    if (warp == 0) {
        const int par = ctl->slice_par;
        const unsigned* Tp = slice_s + (size_t)par * 3 * sn_s;
        long long a = 0, b = 0, c = 0;
        for (int k = lane; k < (int)blockIdx.x; k += 32) {
            a += __ldcg(Tp + 3 * k + 0);
            b += __ldcg(Tp + 3 * k + 1);
            c += __ldcg(Tp + 3 * k + 2);
        }
        if (sp == 1) {
            const long long ch0 = ctl->chunks_in[d][0];
            const unsigned* T0 = slice0 + (size_t)par * 3 * sn0;
            for (long long k = lane; k < (ch0 + SLICE - 1) / SLICE; k += 32) b += __ldcg(T0 + 3 * k + 2);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            a += __shfl_xor_sync(FULL, a, o);
            b += __shfl_xor_sync(FULL, b, o);
            c += __shfl_xor_sync(FULL, c, o);
        }
        if (lane == 0) {
            s_pre[0] = a;
            s_pre[1] = b;
            s_pre[2] = c;
        }
    }
#pragma unroll
    for (int i = 0; i < K; ++i) {
        const int k = i * BLOCK + tid;
        const bool in = t0 + k < chunks;
        s_cnt[0][k] = (unsigned short)(in ? __ldcg(cnt_m + t0 + k) : 0);
        s_cnt[1][k] = (unsigned short)(in ? __ldcg(cnt_b + t0 + k) : 0);
        s_cnt[2][k] = (unsigned short)((in && sp == 0) ? __ldcg(cnt_s + t0 + k) : 0);
    }
    __syncthreads();
    const long long tb = t0 + (long long)tid * K;
    int rm = 0, rb = 0, rs = 0;
#pragma unroll
    for (int i = 0; i < K; ++i) {
        rm += s_cnt[0][tid * K + i];
        rb += s_cnt[1][tid * K + i];
        rs += s_cnt[2][tid * K + i];
    }
    int xm = rm, xb = rb, xs = rs;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int ym = __shfl_up_sync(FULL, xm, o), yb = __shfl_up_sync(FULL, xb, o), ys = __shfl_up_sync(FULL, xs, o);
        if (lane >= o) {
            xm += ym;
            xb += yb;
            xs += ys;
        }
    }
    if (lane == 31) {
        s_w[0][warp] = xm;
        s_w[1][warp] = xb;
        s_w[2][warp] = xs;
    }
    __syncthreads();
    if (warp < 3) {  // warp k scans the NW warp sums of count k (NW <= 32)
        const int v = lane < NW ? s_w[warp][lane] : 0;
        int x = v;
#pragma unroll
        for (int o = 1; o < NW; o <<= 1) {
            const int y = __shfl_up_sync(FULL, x, o);
            if (lane >= o) x += y;
        }
        if (lane < NW) s_w[warp][lane] = x - v;
    }
    __syncthreads();
    long long em = s_pre[0] + s_w[0][warp] + xm - rm;
    const long long eb0 = s_pre[1] + s_w[1][warp] + xb - rb;  // this thread's first newborn of each kind
    const long long es0 = s_pre[2] + s_w[2][warp] + xs - rs;
#pragma unroll 1
    for (int i = 0; i < K; ++i) {  // rolled: this code runs once per step, from a cold instruction cache
        const long long t = tb + i;
        if (t < chunks) st[t] = (int)em;  // the first slot of region t of the new layout
        em += s_cnt[0][tid * K + i];
    }
    // The newborns of the warp's chunks, copied by the whole warp: newborn j of a kind belongs to the
    // last lane u whose first newborn is at or before j (a search over the lanes' starts), and within
    // lane u's K chunks to the one whose running count passes j. All lanes load, then all store.
    int err = 0;
#pragma unroll 1
    for (int kind = 0; kind < 2; ++kind) {
        if (kind == 1 && sp != 0) break;  // same-species newborns: the electron sweep's only
        const int row = kind == 0 ? 1 : 2;
        const long long e0 = kind == 0 ? eb0 : es0;
        const int r = kind == 0 ? rb : rs;
        const int32_t* __restrict__ cin = kind == 0 ? bc : sc;
        const R* __restrict__ pin = kind == 0 ? bp : spr;
        int32_t* __restrict__ cdst = kind == 0 ? oc_q : oc_0;
        R* __restrict__ pdst = kind == 0 ? op_q : op_0;
        const long long w0 = __shfl_sync(FULL, e0, 0), w1 = __shfl_sync(FULL, e0 + r, 31);
        for (long long jb = w0; jb < w1; jb += 32) {
            const long long j = jb + lane;
            int u = 0;  // last lane with start <= j
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const long long su = __shfl_sync(FULL, e0, u + o);
                if (su <= j) u += o;
            }
            const long long su = __shfl_sync(FULL, e0, u);
            if (j >= w1) continue;
            long long rem = j - su;
            int ci = 0;
            const int tw = (warp * 32 + u) * K;  // lane u's first chunk in the slice
            while (ci < K - 1 && rem >= s_cnt[row][tw + ci]) rem -= s_cnt[row][tw + ci++];
            const long long srcr = (t0 + tw + ci) * CHUNK + rem;
            if (j < bcap) {  // records of one (FP32) or two (FP64) 16-byte words; no runtime-indexed array
                const int cv = __ldcg(cin + srcr);
                const R r0 = __ldcg(pin + srcr * rw);
                const R r1 = rw == 2 ? __ldcg(pin + srcr * rw + 1) : r0;
                cdst[j] = cv;
                pdst[j * rw] = r0;
                if (rw == 2) pdst[j * rw + 1] = r1;
            } else {
                err = ERR_CAPACITY;
            }
        }
    }
    if (err) atomicOr(&ctl->error, err);
}

constexpr int POST_BLOCK = 512;   // threads per k_post CTA
constexpr int FIELD_NODES = 128;  // nodes of a field or moments part
constexpr int FIELD_SUMS = 128;   // partial sums of the solve

// Discharge current density over step n (section "Boundary conditions", equation for J(t)):
// J = eps0 dE/dt + e0 (Gamma_i - Gamma_e), with the particle fluxes counted positive towards +z
// from the step's absorbed and emitted superparticles: at z = 0 an absorbed ion (moving towards
// -z) carries -e w_i, an absorbed electron +e w_e, an emitted secondary electron (towards +z)
// -e w_e; at z = d the absorbed particles' signs flip and emitted electrons move towards -z.
// FP64, by one thread of the first field part beside the node field: everything that does not need
// the new electrode fields is read and formed before they are known (before()). The initial solve of a
// load (mode bit 4) only records the fields and counters. On a full step the current at z = 0 is also
// projected onto the rf period's first harmonic (sin and cos at the step midpoint); at the end of a
// period the amplitude is stored.
struct Current {
    unsigned long long c[6];
    double cond0, condN, E0, EN, js0, js1, jt0, jt1, vs;
    int have, k, jslot, par;
    __device__ __forceinline__ void before(const Disc& D, int d, const Ctl* ctl, long long step) {
        unsigned long long o[6];
#pragma unroll
        for (int i = 0; i < 4; ++i) c[i] = __ldcg(D.cnt + CNT_ABS + i);  // [species][electrode]
        c[4] = __ldcg(D.cnt + CNT_SEE_SIDE);
        c[5] = __ldcg(D.cnt + CNT_SEE_SIDE + 1);
#pragma unroll
        for (int i = 0; i < 6; ++i) o[i] = ctl->cnt_solve[d][i];
        have = ctl->have_solve[d];
        E0 = ctl->E_wall[d][0];
        EN = ctl->E_wall[d][1];
        js0 = ctl->J_sum[d][0];
        js1 = ctl->J_sum[d][1];
        par = ctl->dep_par;
        vs = ctl->V_scale[d][par];
        jslot = step_mod(step, D.jh);
        k = 0;
        if (D.jtab) {
            k = step_mod(step, D.steps_per_period);
            jt0 = D.jtab[2 * k];
            jt1 = D.jtab[2 * k + 1];
        }
        const double we = D.w[0], wi = D.w[1], rdt = D.inv_dt;  // FP64 division is slow on this part
        cond0 = E_CHARGE * (we * (double)(c[0] - o[0]) - wi * (double)(c[2] - o[2]) - we * (double)(c[4] - o[4])) * rdt;
        condN = E_CHARGE * (wi * (double)(c[3] - o[3]) - we * (double)(c[1] - o[1]) + we * (double)(c[5] - o[5])) * rdt;
    }
    __device__ __forceinline__ void after(const Disc& D, int d, Ctl* ctl, int mode, long long step, double Ew0,
                                          double Ew1) {
        ctl->E0_last[d] = Ew0;
        if (!(mode & 4)) {  // a solve after a sweep (or a stand-alone solve): the current of step n
            const double rdt = D.inv_dt;
            double J0 = 0.0, JN = 0.0;  // no earlier solve: no current
            if (have) {
                J0 = EPS0 * (Ew0 - E0) * rdt + cond0;
                JN = EPS0 * (Ew1 - EN) * rdt + condN;
            }
            D.J_hist[2 * jslot] = J0;
            D.J_hist[2 * jslot + 1] = JN;
            const int spp = D.steps_per_period;
            if ((mode & 2) && D.jtab && spp > 0) {
                js0 += J0 * jt0;
                js1 += J0 * jt1;
                if (k == spp - 1) {
                    const double a = 2.0 * js0 / spp, b = 2.0 * js1 / spp;
                    const double amp = sqrt(a * a + b * b);
                    const long long per = step_div(step, spp) % PERIOD_HIST;
                    D.J_amp[per] = amp;
                    D.V_hist[per] = D.V_rf * vs;
                    const double Jd = ctl->J_drive[d];
                    if (Jd > 0.0 && amp > 0.0) vs = vs * (Jd / amp);  // Eq. (adaptivevoltage)
                    js0 = js1 = 0.0;
                }
                ctl->J_sum[d][0] = js0;
                ctl->J_sum[d][1] = js1;
            }
        }
        ctl->V_scale[d][par ^ 1] = vs;  // for the next solve (other parts may still read this one's)
        ctl->have_solve[d] = 1;
        ctl->E_wall[d][0] = Ew0;
        ctl->E_wall[d][1] = Ew1;
#pragma unroll
        for (int i = 0; i < 6; ++i) ctl->cnt_solve[d][i] = c[i];
    }
};

// Field of one discharge after its deposits are complete, nodes of part `part`. Poisson, Eq. (poisson):
// phi_{j-1} - 2 phi_j + phi_{j+1} = -r_j with r_j = rho_j dx^2 / eps0, phi_0 = V_rf sin(2 pi f t),
// phi_N = 0. With R_j = sum_{k<=j} r_k and S_j = sum_{i<j} R_i: phi_j = phi_0 + j g_1 - S_j, g_1 = (phi_N
// - phi_0 + S_N) / N. R and S are linear in the deposits: R_j = c_i IR_i,j - c_e IR_e,j, S_{j+1} = c_i
// IS_i,j - c_e IS_e,j with the exact integer sums IR_s,j = sum_{1<=k<=j} D_s,k (64 bits: a store holds
// below 2^30 particles of 2^32 each) and IS_s,j = sum_{i<=j} IR_s,i (128 bits), from one scan (PSum).
//
// What bounds it is latency, above all instruction fetches: the grid runs once per step after other
// code, so the code is short: one small scan run by six warps, one sum each (the earlier scan held
// 128-bit pairs in registers), J(t) in a warp of its own, loads requested together. FP64 (2 operations per
// clock and SM here) is used once per node, with no division (host reciprocals), 128 nodes to a CTA: at
// 2048 cells one CTA took 14 us for all of them. Measured, a launch: 13.1 -> 8.5 us at 128 cells, 18.9 ->
// 8.9 at 512, 30.1 -> 12.9 at 2048, 21.8 -> 13.1 for 16 discharges.
template <typename T>
__device__ __forceinline__ void field_solve(const Disc& D, int d, Ctl* __restrict__ ctl, int mode, int part, int tid,
                                            int lane, int warp, unsigned long long* s_f, int max_N,
                                            unsigned long long (*s_ps)[FIELD_SUMS], unsigned long long* s_tot,
                                            double* s_g1, Current& J) {
    const int N = D.N;
    if (part * FIELD_NODES > N) return;
    // everything that is read is requested first; the deposits of both parities, so that their loads need
    // not wait for the parity
    const int par = ctl->dep_par;
    const long long step = ctl->step;
    const double vs0 = ctl->V_scale[d][0], vs1 = ctl->V_scale[d][1];
    // the last warp (one thread of it) takes J(t) and g_1, so it does not wait for the other warps until the
    // sums are there: its loads and FP64 conversions run beside the scan (a step of 2.5e4 particles: 20.9 -> 20.4 us)
    constexpr int OTHERS = POST_BLOCK - 32;
    const bool last = warp == OTHERS / 32;
    auto others_sync = [&]() { asm volatile("bar.sync 1, %0;" ::"n"(OTHERS) : "memory"); };
    unsigned long long* sde = s_f;
    unsigned long long* sdi = sde + (max_N + 1);
    for (int j = last ? N + 1 : tid; j <= N; j += OTHERS) {
        const unsigned long long e0 = __ldcg(D.D[0] + j), e1 = __ldcg(D.D[0] + N + 1 + j);
        const unsigned long long i0 = __ldcg(D.D[1] + j), i1 = __ldcg(D.D[1] + N + 1 + j);
        sde[j] = par ? e1 : e0;
        sdi[j] = par ? i1 : i0;
    }
    const long long ns = (mode & 4) ? step : step + 1;  // time level of the solve
    const double* Vt = D.V0tab;
    const double Vk = Vt ? Vt[step_mod(ns, D.steps_per_period)] : 0.0;
    if (!last) others_sync();
    else if (part == 0 && lane == 0) J.before(D, d, ctl, step);
    // thread t < FIELD_SUMS sums the nodes [t per, (t + 1) per) (node 0 carries no deposit term), 1 <= j < N
    const int per = (N + FIELD_SUMS - 1) / FIELD_SUMS;
    if (tid < FIELD_SUMS) {
        PSum own{};
#pragma unroll 1
        for (int j = max(tid * per, 1); j < min(N, (tid + 1) * per); ++j) own.add(j, sde[j], sdi[j]);
        // lane l of the scan below takes threads 4 l .. 4 l + 3
#pragma unroll
        for (int q = 0; q < 6; ++q) s_ps[q][(tid & 3) * 32 + (tid >> 2)] = own.v[q];
    }
    if (!last) others_sync();
    if (warp < 6) {  // exclusive scan of sum `warp` over the partial sums
        unsigned long long* p = s_ps[warp] + lane;
        const unsigned long long x0 = p[0], x1 = p[32], x2 = p[64], x3 = p[96];
        const unsigned long long x = x0 + x1 + x2 + x3;
        unsigned long long y = x;
#pragma unroll 1
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long z = __shfl_up_sync(FULL, y, o);
            if (lane >= o) y += z;
        }
        if (lane == 31) s_tot[warp] = y;
        y -= x;
        p[0] = y;
        p[32] = y + x0;
        p[64] = y + x0 + x1;
        p[96] = y + x0 + x1 + x2;
    }
    __syncthreads();
    const double pr0 = D.pc_r[0], pr1 = D.pc_r[1];
    // R_j -> r_j sums in FP64, as c_i x_i - c_e x_e
    auto Rr_of = [&](unsigned long long r0, unsigned long long r1) {
        return __fma_rn(pr1, (double)(long long)r1, -pr0 * (double)(long long)r0);
    };
    const double V0 = (Vt ? Vk : D.V_rf * sin(2.0 * PI_D * D.f_rf * ((double)ns * D.dt))) * (par ? vs1 : vs0);
    // warps 0-3: R_{j-1}, R_j and S_j of node j; the last warp: g_1 (with S_N from the totals), while they
    // do not need it yet
    const int j = part * FIELD_NODES + tid;
    const bool node = tid < FIELD_NODES && j <= N, inside = node && j > 0 && j < N;
    double Rprev = 0.0, Rj = 0.0, Sj = 0.0;
    if (inside) {
        PSum run;
        const int t = j / per;
#pragma unroll
        for (int q = 0; q < 6; ++q) run.v[q] = s_ps[q][(t & 3) * 32 + (t >> 2)];
#pragma unroll 1
        for (int i = max(t * per, 1); i < j; ++i) run.add(i, sde[i], sdi[i]);
        Rprev = Rr_of(run.v[0], run.v[1]);
        Rj = Rr_of(run.v[0] + sde[j], run.v[1] + sdi[j]);
        Sj = poisson_S(run.v[0], run.v[1], run.v[2], run.v[3], run.v[4], run.v[5], j, pr0, pr1);
    } else if (tid == OTHERS) {
        *s_g1 = (poisson_S(s_tot[0], s_tot[1], s_tot[2], s_tot[3], s_tot[4], s_tot[5], N, pr0, pr1) - V0) * D.inv_N;
    }
    __syncthreads();
    const double g1 = *s_g1;
    // Gauss's law over the half cells at the electrodes
    auto wall = [&](int n) {
        const double rw = __fma_rn(D.pc_w[1], (double)sdi[n], -D.pc_w[0] * (double)sde[n]);
        return n == 0 ? -g1 * D.inv_dx - rw * D.hdx_eps
                      : -(g1 - Rr_of(s_tot[0], s_tot[1])) * D.inv_dx + rw * D.hdx_eps;
    };
    if (part == 0 && tid == OTHERS) J.after(D, d, ctl, mode, step, wall(0), wall(N));
    if (!node) return;
    // g_j = phi_j - phi_{j-1} = g_1 - R_{j-1}; node field E_j = -(g_j + g_{j+1}) / (2 dx) inside
    // (the central difference of phi, without the cancellation of large phi values)
    const double E = inside ? ((g1 - Rprev) + (g1 - Rj)) * D.m_inv_2dx : wall(j);
    reinterpret_cast<T*>(D.E)[j] = (T)E;
    D.E64[j] = E;
    D.phi[j] = inside ? V0 + (double)j * g1 - Sj : j == 0 ? V0 : 0.0;
}

// The moments of the nodes of a part (mode bit 2), and zeroed arrays for the next sweep: the energy
// moment and the deposits of the other parity, which are those at x_n (of the previous solve).
__device__ __forceinline__ void moments_part(const Disc& D, int d, Ctl* __restrict__ ctl, int mode, int part, int tid) {
    const int N = D.N, j = part * FIELD_NODES + tid;
    if (part == 0 && tid == 0 && (mode & 2)) ctl->acc_steps[d] += 1;
    if (tid >= FIELD_NODES || j > N) return;
    const int par = ctl->dep_par;
    const size_t po = (size_t)par * (N + 1) + j, pn = (size_t)(par ^ 1) * (N + 1) + j;
    unsigned long long* __restrict__ D0 = D.D[0];
    unsigned long long* __restrict__ D1 = D.D[1];
    unsigned long long* __restrict__ Qd = D.Q;
    if (mode & 2) {
        unsigned __int128* __restrict__ acc = D.acc_D[0] + j;  // n_e, n_i, energy, n_e at x_n, N + 1 apart
        const int n1 = N + 1;
        const unsigned long long de = __ldcg(D0 + po), di = __ldcg(D1 + po), q = __ldcg(Qd + j), dp = __ldcg(D0 + pn);
        auto ld128 = [](const unsigned __int128* a) {
            const ulonglong2 v = __ldcg(reinterpret_cast<const ulonglong2*>(a));
            return ((unsigned __int128)v.y << 64) | v.x;
        };
        const unsigned __int128 a0 = ld128(acc), a1 = ld128(acc + n1), a2 = ld128(acc + 2 * n1), a3 = ld128(acc + 3 * n1);
        acc[0] = a0 + de;
        acc[n1] = a1 + di;
        acc[2 * n1] = a2 + q;
        acc[3 * n1] = a3 + dp;
    }
    D0[pn] = 0;
    D1[pn] = 0;
    Qd[j] = 0;
}

template <typename T>
__global__ void __launch_bounds__(POST_BLOCK, 2) k_post(const Disc* __restrict__ discs, int n_disc, Ctl* __restrict__ ctl,
                                                     int out_buf, int mode, int nsl, int max_N) {
    constexpr int BLOCK = POST_BLOCK;
    extern __shared__ __align__(16) unsigned long long s_f[];
    __shared__ unsigned long long s_ps[6][FIELD_SUMS], s_tot[6];
    __shared__ double s_g1;
    __shared__ Current s_J;  // of one thread, kept out of its registers
    __shared__ int s_err;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int d = blockIdx.y >> 1, part = (int)blockIdx.x - nsl;
    if (tid == 0) s_err = 0;
    __syncthreads();
    grid_dep_sync();
    if (part < 0) {
        seg_apply<BLOCK>(discs, ctl, out_buf, tid, lane, warp);
    } else if ((blockIdx.y & 1) == 0) {
        if (!(mode & 8)) field_solve<T>(discs[d], d, ctl, mode, part, tid, lane, warp, s_f, max_N, s_ps, s_tot, &s_g1, s_J);
    } else if (part > 0) {
        if (!(mode & 8)) moments_part(discs[d], d, ctl, mode, part - 1, tid);
    } else if ((mode & 1) && warp == 0) {  // store totals
        int e2 = 0;
        store_totals(discs[d], d, ctl, lane, ctl->slice_par, (mode & 2) != 0, out_buf, e2);
        if (e2 && lane == 0) atomicOr(&s_err, e2);
    }
    __syncthreads();
    // the last CTA advances the step (bit 2) and the parities. Every CTA has consumed its reads of all
    // three before its count (data dependence), and the last CTA reads no other CTA's results, so no
    // fence: the kernel boundary publishes everything
    if (tid == 0) {
        if (s_err) atomicOr(&ctl->error, s_err);
        const unsigned prev = atomicAdd(&ctl->fin_done, 1u);
        if (prev == gridDim.x * gridDim.y - 1) {
            ctl->fin_done = 0;
            if (mode & 2) ctl->step = ctl->step + 1;
            if (mode & 1) ctl->slice_par = ctl->slice_par ^ 1;
            if (!(mode & 8)) ctl->dep_par = ctl->dep_par ^ 1;
        }
    }
}

// ---------------------------------------------------------------------------
// Initial load: uniform positions, Maxwellian velocities (Philox calls 0xF0,
// 0xF1 at step 0). grid.y = store (d, species).
template <typename T>
__global__ void k_load(const Disc* __restrict__ discs, Ctl* __restrict__ ctl, int buf, unsigned long long seed) {
    const int seg = blockIdx.y, d = seg >> 1, sp = seg & 1;
    const Disc& D = discs[d];
    const Consts<T>& K = consts_of<T>(D);
    const long long n = ctl->count[d][sp];
    const int N = D.N;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        const U4 r = draw(seed, (uint32_t)k, 0, sp, 0xF0, D.discharge_id);
        const U4 q = draw(seed, (uint32_t)k, 0, sp, 0xF1, D.discharge_id);
        const T x = mul_((T)u01(r.x), (T)N);
        int c = (int)x;
        T f;
        if (c >= N) {
            c = N - 1;
            f = one_minus_ulp<T>();
        } else {
            f = sub_(x, (T)c);
        }
        float n0, n1, n2, n3;
        box_muller(u01(r.y), u01(r.z), n0, n1);
        box_muller(u01(r.w), u01(q.x), n2, n3);
        const T sg = K.sig0[sp];
        store_rec<T>(D.c[buf][sp], D.p[buf][sp], k, Part<T>{c, f, mul_(sg, (T)n0), mul_(sg, (T)n1), mul_(sg, (T)n2)});
    }
}

// Warm start: particles sampled from profiles on a uniform grid of P points
// (calls 0xF2, 0xF3 at step 0): position by inverse of the piecewise-constant
// CDF, electrons Maxwellian at kT = 2/3 <eps>(z), ions at T_i0.
template <typename T>
struct WarmDev {
    const T* cdf[2];  // per species, P entries, cdf[0] = 0, cdf[P-1] = 1
    const T* eps;     // P entries, eV
    int P, pad_;
    T scale;          // N / (P - 1)
    T K23;            // 2 e / (3 m_e)
};

template <typename T>
__global__ void k_load_profile(const Disc* __restrict__ discs, Ctl* __restrict__ ctl, int buf,
                               unsigned long long seed, const WarmDev<T>* __restrict__ warm) {
    const int seg = blockIdx.y, d = seg >> 1, sp = seg & 1;
    const Disc& D = discs[d];
    const WarmDev<T>& W = warm[d];
    const long long n = ctl->count[d][sp];
    const int N = D.N, P = W.P;
    const T* cdf = W.cdf[sp];
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        const U4 r = draw(seed, (uint32_t)k, 0, sp, 0xF2, D.discharge_id);
        const U4 q = draw(seed, (uint32_t)k, 0, sp, 0xF3, D.discharge_id);
        const T u = (T)u01(r.x);
        int lo = 0, hi = P - 2;  // largest j in [0, P-2] with cdf[j] <= u
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (cdf[mid] <= u) lo = mid;
            else hi = mid - 1;
        }
        const int j = lo;
        const T den = sub_(cdf[j + 1], cdf[j]);
        T t = den > (T)0 ? div_(sub_(u, cdf[j]), den) : (T)0;
        if (t >= (T)1) t = one_minus_ulp<T>();
        const T x = mul_(add_((T)j, t), W.scale);
        int c = (int)x;
        T f;
        if (c >= N) {
            c = N - 1;
            f = one_minus_ulp<T>();
        } else {
            f = sub_(x, (T)c);
        }
        T sg;
        if (sp == 0) {
            T el = fma_(t, sub_(W.eps[j + 1], W.eps[j]), W.eps[j]);
            if (!(el > (T)0)) el = (T)0;
            sg = sqrt_(mul_(el, W.K23));
        } else {
            sg = consts_of<T>(D).sig0[1];
        }
        float n0, n1, n2, n3;
        box_muller(u01(r.y), u01(r.z), n0, n1);
        box_muller(u01(r.w), u01(q.x), n2, n3);
        store_rec<T>(D.c[buf][sp], D.p[buf][sp], k, Part<T>{c, f, mul_(sg, (T)n0), mul_(sg, (T)n1), mul_(sg, (T)n2)});
    }
}

// CIC deposit of whole stores (used after a load or a state upload).
template <typename T>
__global__ void k_deposit(const Disc* __restrict__ discs, const Ctl* __restrict__ ctl, int buf, int max_N) {
    extern __shared__ __align__(16) unsigned long long s_h[];
    const int seg = blockIdx.y, d = seg >> 1, sp = seg & 1;
    const Disc& D = discs[d];
    const int N = D.N;
    for (int j = threadIdx.x; j <= N; j += blockDim.x) s_h[j] = 0;
    __syncthreads();
    const long long n = ctl->count[d][sp];
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        T f, vx, vy, vz;
        load_rec<T>(D.p[buf][sp], k, f, vx, vy, vz);
        shist_add(s_h, D.c[buf][sp][k], cic_F(f));
    }
    __syncthreads();
    for (int j = threadIdx.x; j <= N; j += blockDim.x)
        if (s_h[j]) atomicAdd(&D.D[sp][(size_t)ctl->dep_par * (N + 1) + j], s_h[j]);
}

// Half back-kick after the initial solve: stored v_z = v_0 - (q/m) E_0 dt / 2.
template <typename T>
__global__ void k_backkick(const Disc* __restrict__ discs, const Ctl* __restrict__ ctl, int buf) {
    const int seg = blockIdx.y, d = seg >> 1, sp = seg & 1;
    const Disc& D = discs[d];
    const Consts<T>& K = consts_of<T>(D);
    const T* E = reinterpret_cast<const T*>(D.E);
    const long long n = ctl->count[d][sp];
    using R = typename Rec<T>::type;
    R* P = reinterpret_cast<R*>(D.p[buf][sp]);
    const T mK = -K.K[sp];
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        const int c = D.c[buf][sp][k];
        R r = P[k];
        const T e0 = E[c], e1 = E[c + 1];
        const T ef = fma_(r.x, sub_(e1, e0), e0);
        r.w = fma_(mK, ef, r.w);
        P[k] = r;
    }
}

// Rate-coefficient tables sigma_j * v, cumulative over processes, rounded to T.
// Electrons: v = sqrt(2 e eps / m_e). Ions: g = sqrt(4 e eps / M) (c.m. energy).
template <typename T>
__global__ void k_tables(int n_pts, int n_proc, double de, double M, const double* __restrict__ se,
                         const double* __restrict__ si, T* __restrict__ Te, T* __restrict__ Ti,
                         unsigned long long* __restrict__ kmax) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n_pts) return;
    const double eps = (double)k * de;
    const double v = sqrt(2.0 * E_CHARGE * eps / M_ELEC);
    double cum = 0.0;
    for (int j = 0; j < 4; ++j) {
        if (j < n_proc) cum = __dadd_rn(cum, __dmul_rn(se[(size_t)k * n_proc + j], v));
        Te[(size_t)k * 4 + j] = (T)cum;
    }
    const double gr = sqrt(4.0 * E_CHARGE * eps / M);
    cum = 0.0;
    for (int j = 0; j < 2; ++j) {
        cum = __dadd_rn(cum, __dmul_rn(si[(size_t)k * 2 + j], gr));
        Ti[(size_t)k * 2 + j] = (T)cum;
    }
    atomicMax(&kmax[0], (unsigned long long)__double_as_longlong((double)Te[(size_t)k * 4 + 3]));
    atomicMax(&kmax[1], (unsigned long long)__double_as_longlong((double)Ti[(size_t)k * 2 + 1]));
}

// ---------------------------------------------------------------------------
// Chunk k of a store with layout L (see Lay): first slot, slots and record offset. Regions take
// their first and end slots from the start table.
struct ChunkDesc {
    long long src;
    int base, cnt;
};
__device__ __forceinline__ ChunkDesc chunk_desc(const Lay& L, long long n, const int* st, long long k, int chunk) {
    ChunkDesc c;
    if (k < L.K) {
        c.src = k * chunk;
        c.base = __ldcg(st + k);
        c.cnt = __ldcg(st + k + 1) - c.base;
    } else {
        const long long j = k - L.K;
        c.src = L.D0 + j * chunk;
        c.base = (int)(L.M + j * chunk);
        c.cnt = (int)min((long long)chunk, n - c.base);
    }
    return c;
}

// ---------------------------------------------------------------------------
// Kinetic diagnostics of the electrons (section "Results": the EEDF, the fast-electron density and
// the profiles at a fixed rf phase), taken from the store at (x_n, v_n) before the sweep of step n.
// Per electron: the gathered field and the first half kick as in the sweep, the energy in 2^-12 eV
// clamped at 2^26, then per node array an integer value X rounded in the particle precision and
// split like the charge (X - rn(X f) to node c, rn(X f) to node c + 1). Units of X:
//   DG_D  2^32 per particle (the deposit's F split)     DG_U  energy, 2^-12 eV
//   DG_V  v_z, 2^-6 m/s                                  DG_W  energy x v_z, formed as (eq v_z) 2^-16
//   DG_K  ionization rate coefficient, 2^-72 m^3/s       DG_F  2^32 per electron above the threshold
//   DG_FA as DG_F, at the EEDF samples
// Sums are exact (int64, mod 2^64); warp groups of equal cells are reduced in three 22/22/20-bit
// parts, so no partial sum overflows 32 bits.
template <typename T> __device__ __forceinline__ long long rint_ll(T x);
template <> __device__ __forceinline__ long long rint_ll<float>(float x) { return __float2ll_rn(x); }
template <> __device__ __forceinline__ long long rint_ll<double>(double x) { return __double2ll_rn(x); }

__device__ __forceinline__ unsigned long long group_sum64(unsigned peers, unsigned long long v) {
    const unsigned a = __reduce_add_sync(peers, (unsigned)(v & 0x3FFFFFu));
    const unsigned b = __reduce_add_sync(peers, (unsigned)((v >> 22) & 0x3FFFFFu));
    const unsigned c = __reduce_add_sync(peers, (unsigned)(v >> 44));
    return (unsigned long long)a + ((unsigned long long)b << 22) + ((unsigned long long)c << 44);
}

// a to node key, b to node key + 1 of a shared histogram: reduced over the lanes of `peers` and
// added by the leader, or (lanewise) added lane by lane.
__device__ __forceinline__ void warp_add_pair(unsigned long long* h, int key, unsigned long long a,
                                              unsigned long long b, unsigned peers, bool leader, bool lanewise) {
    if (lanewise) {
        if (key >= 0) {
            if (a) sadd64(&h[key], a);
            if (b) sadd64(&h[key + 1], b);
        }
        return;
    }
    const unsigned long long sa = group_sum64(peers, a), sb = group_sum64(peers, b);
    if (leader && key >= 0) {
        if (sa) sadd64(&h[key], sa);
        if (sb) sadd64(&h[key + 1], sb);
    }
}

template <typename T>
__device__ __forceinline__ void split_rint(T x, T f, unsigned long long& a, unsigned long long& b) {
    const long long X = rint_ll<T>(x), Xh = rint_ll<T>(mul_(x, f));
    a = (unsigned long long)(X - Xh);
    b = (unsigned long long)Xh;
}

template <typename T4r, typename T>
__device__ __forceinline__ T col4(const T4r& r, int j) {
    return j == 0 ? r.x : j == 1 ? r.y : j == 2 ? r.z : r.w;
}

constexpr int DIAG_BLOCK = 256, DIAG_NW = DIAG_BLOCK / 32;

template <typename T>
__global__ void __launch_bounds__(DIAG_BLOCK) k_diag(const Disc* __restrict__ discs, const Ctl* ctl, int buf,
                                                     DiagArgs A) {
    grid_dep_sync();
    extern __shared__ __align__(16) unsigned long long s_dg[];  // [arrays of the mask][N + 1], EEDF [bins] u32
    using R = typename Rec<T>::type;
    using Row4 = typename T4<T>::type;
    const int d = blockIdx.y;
    const Disc& D = discs[d];
    const int N = D.N, N1 = N + 1, CHUNK = D.chunk, RPC = CHUNK / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool phase = A.mode & DIAG_PHASE, sample = A.mode & DIAG_SAMPLE;
    const int nar = __popc(A.mask), nb = sample ? A.bins : 0;
    unsigned* s_eedf = reinterpret_cast<unsigned*>(s_dg + (size_t)nar * N1);
    for (int j = tid; j < nar * N1; j += DIAG_BLOCK) s_dg[j] = 0;
    for (int j = tid; j < nb; j += DIAG_BLOCK) s_eedf[j] = 0;
    const T* E = reinterpret_cast<const T*>(D.E);
    if (blockIdx.x == 0 && (A.mode & DIAG_COUNT)) {  // field sum of the snapshot, snapshot and sample counts
        if (phase)
            for (int j = tid; j <= N; j += DIAG_BLOCK) D.dg_E[j] += (double)E[j];
        if (tid == 0) {
            if (phase) D.dg_n[0] += 1;
            if (sample) D.dg_n[1] += 1;
        }
    }
    __syncthreads();
    unsigned long long* h[DG_ARRAYS];
#pragma unroll
    for (int a = 0; a < DG_ARRAYS; ++a) h[a] = s_dg + (size_t)__popc(A.mask & ((1u << a) - 1u)) * N1;
    const bool mD = A.mask & (1u << DG_D), mU = A.mask & (1u << DG_U), mV = A.mask & (1u << DG_V),
               mW = A.mask & (1u << DG_W), mK = A.mask & (1u << DG_K), mF = A.mask & (1u << DG_F),
               mFa = A.mask & (1u << DG_FA);
    const Consts<T>& K = consts_of<T>(D);
    const T thr = (T)A.thr, inv_bin = (T)A.inv_bin, top = (T)(D.n_pts - 1), binsT = (T)A.bins;
    const int ciz = 1 + D.n_exc;  // ionization column of the cumulative electron table
    const Row4* Te = reinterpret_cast<const Row4*>(D.Te);
    const long long n = ctl->count[d][0];
    const Lay L = ctl->lay[d][0][buf];
    const long long chunks = chunks_of(L, n, CHUNK);
    const int32_t* cc = D.c[buf][0];
    const R* P = reinterpret_cast<const R*>(D.p[buf][0]);
    for (long long k = (long long)blockIdx.x * DIAG_NW + warp; k < chunks; k += (long long)gridDim.x * DIAG_NW) {
        const ChunkDesc cd = chunk_desc(L, n, D.start[0], k, CHUNK);
        for (int r = 0; r < RPC; ++r) {
            const int i = 32 * r + lane;
            int c = -1;
            T f = 0, vx = 0, vy = 0, vz = 0;
            if (i < cd.cnt) {
                c = __ldcg(cc + cd.src + i);
                const R q = ldcg_rec(P + cd.src + i);
                f = q.x;
                vx = q.y;
                vy = q.z;
                vz = q.w;
                if (!((unsigned)c < (unsigned)N)) c = -1;
            }
            unsigned long long F = 0, uA = 0, uB = 0, vA = 0, vB = 0, wA = 0, wB = 0, kA = 0, kB = 0;
            bool fast = false;
            int bin = 0;
            if (c >= 0) {
                const T E0 = E[c], E1 = E[c + 1];
                const T ef = fma_(f, sub_(E1, E0), E0);
                vz = fma_(K.K[0], ef, vz);  // v_n
                const T e2 = fma_(vx, vx, fma_(vy, vy, mul_(vz, vz)));
                T eq = mul_(e2, K.kappa_E);
                if (!(eq <= (T)0x1p26)) eq = (T)0x1p26;
                F = cic_F(f);
                fast = eq > thr;
                if (mU) split_rint<T>(eq, f, uA, uB);
                if (mV) split_rint<T>(mul_(vz, (T)64), f, vA, vB);
                if (mW) split_rint<T>(mul_(mul_(eq, vz), (T)0x1p-16), f, wA, wB);
                if (mK) {
                    const T xi = mul_(e2, K.kappa_e);
                    T Cz, Cy;
                    if (!(xi < top)) {
                        const Row4 a = Te[D.n_pts - 1];
                        Cz = col4<Row4, T>(a, ciz);
                        Cy = col4<Row4, T>(a, ciz - 1);
                    } else {
                        const int ii = (int)xi;
                        const T fr = sub_(xi, (T)ii);
                        const Row4 a = Te[ii], b = Te[ii + 1];
                        const T az = col4<Row4, T>(a, ciz), ay = col4<Row4, T>(a, ciz - 1);
                        Cz = fma_(fr, sub_(col4<Row4, T>(b, ciz), az), az);
                        Cy = fma_(fr, sub_(col4<Row4, T>(b, ciz - 1), ay), ay);
                    }
                    split_rint<T>(mul_(sub_(Cz, Cy), (T)0x1p72), f, kA, kB);
                }
                if (sample) {
                    const T xb = mul_(eq, inv_bin);
                    bin = xb < binsT ? (int)xb : A.bins - 1;
                }
            }
            // a row of one cell (common on a cell-sorted store) is reduced across the warp, any other
            // row added lane by lane (grouping by match_any cost more than it saved in the sweep)
            const int c0 = __shfl_sync(FULL, c, 0);
            const bool lanewise = !__all_sync(FULL, c == c0);
            const unsigned peers = FULL;
            const bool leader = lane == 0;
            const unsigned long long dA = c >= 0 ? (1ull << 32) - F : 0ull, dB = c >= 0 ? F : 0ull;
            if (mD) warp_add_pair(h[DG_D], c, dA, dB, peers, leader, lanewise);
            if (mU) warp_add_pair(h[DG_U], c, uA, uB, peers, leader, lanewise);
            if (mV) warp_add_pair(h[DG_V], c, vA, vB, peers, leader, lanewise);
            if (mW) warp_add_pair(h[DG_W], c, wA, wB, peers, leader, lanewise);
            if (mK) warp_add_pair(h[DG_K], c, kA, kB, peers, leader, lanewise);
            if (mF) warp_add_pair(h[DG_F], c, fast ? dA : 0ull, fast ? dB : 0ull, peers, leader, lanewise);
            if (mFa) warp_add_pair(h[DG_FA], c, fast ? dA : 0ull, fast ? dB : 0ull, peers, leader, lanewise);
            if (sample && c >= 0) atomicAdd(&s_eedf[bin], 1u);
        }
    }
    __syncthreads();
#pragma unroll
    for (int a = 0; a < DG_ARRAYS; ++a)
        if (A.mask & (1u << a)) {
            unsigned long long* g = D.dg + (size_t)a * N1;
            for (int j = tid; j < N1; j += DIAG_BLOCK)
                if (h[a][j]) atomicAdd(&g[j], h[a][j]);
        }
    for (int j = tid; j < nb; j += DIAG_BLOCK)
        if (s_eedf[j]) atomicAdd(&D.dg_eedf[j], (unsigned long long)s_eedf[j]);
}

// Stable counting sort of every store by cell into the other buffer (dense):
//   k_sort_count   tiles of 4096 slots: each slot's cell and its rank among the tile's slots of the same
//                  cell (in slot order), packed into kr, and the tile's cell counts into hist[t N + c];
//   k_sort_rows    per cell: exclusive scan of the counts over the tiles; the last CTA of a store scans the
//                  cell totals (first slot of every cell);
//   k_sort_scatter the same tiles: destination = first slot of its cell + the tile's offset in that cell +
//                  its rank.
// The first and last run over one list of the tiles of all stores: with a CTA per (store, possible tile), 64
// discharges of 2e4 + 2e4 launched 38912 CTAs, most of them empty, in 72 us each. A tile: warp w walks chunks
// t SORT_NW CPW + w CPW .. + CPW - 1 (CPW = SORT_R 32 / CHUNK) in slot order. What bounds them is latency (of
// the loads, and of the warp's serial ranks), so many warps with the loads of several rows in flight: 16-bit
// counters, offsets of 4 rows at a time. Measured on aged stores, the three kernels in a row: 33
// -> 20 us at 2e4 + 2e4 particles (128 cells), 154 -> 51 for 64 such discharges, 45 -> 35 at 1e6 + 1e6
// (512), 473 -> 298 at 1.2e7 + 1.2e7 (2048). Sorting a store of 2.5e4 whole by one CTA took 40 us.
__device__ __forceinline__ long long sort_tiles(long long chunks, int chunk) {
    const long long per = (long long)SORT_NW * (SORT_R * 32 / chunk);
    return (chunks + per - 1) / per;
}
// The list: per store the tiles before it. Called by all threads; s_pre has 2 n_disc + 1 entries.
__device__ __forceinline__ void sort_list(const Disc* __restrict__ discs, const Ctl* ctl, int n_disc, int buf, int* s_pre) {
    const int n_store = 2 * n_disc;
    for (int s = threadIdx.x; s < n_store; s += blockDim.x) {
        const int d = s >> 1, sp = s & 1;
        s_pre[s + 1] = (int)sort_tiles(chunks_of(ctl->lay[d][sp][buf], ctl->count[d][sp], discs[d].chunk), discs[d].chunk);
    }
    if (threadIdx.x == 0) s_pre[0] = 0;
    __syncthreads();
    if (threadIdx.x < 32) {  // inclusive prefix over at most 128 stores, four per lane
        const int lane = threadIdx.x, b = 4 * lane + 1;
        int v[4], x = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            v[i] = b + i <= n_store ? s_pre[b + i] : 0;
            x += v[i];
        }
        int y = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int z = __shfl_up_sync(FULL, y, o);
            if (lane >= o) y += z;
        }
        y -= x;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            y += v[i];
            if (b + i <= n_store) s_pre[b + i] = y;
        }
    }
    __syncthreads();
}
__device__ __forceinline__ int sort_store(const int* s_pre, int n_store, int item) {  // last store with s_pre <= item
    int lo = 0, hi = n_store - 1;
    while (lo < hi) {
        const int m = (lo + hi + 1) >> 1;
        if (s_pre[m] <= item) lo = m;
        else hi = m - 1;
    }
    return lo;
}

__global__ void __launch_bounds__(SORT_BLOCK, 3) k_sort_count(const Disc* __restrict__ discs, int n_disc,
                                                           Ctl* __restrict__ ctl, int src, int dst,
                                                           unsigned* __restrict__ hist,
                                                           const long long* __restrict__ hoff,
                                                           unsigned* __restrict__ kr_all,
                                                           const long long* __restrict__ eoff, int max_N) {
    extern __shared__ __align__(16) unsigned short s_w[];  // [SORT_NW][nw2] counts, then prefixes
    __shared__ int s_pre[2 * MAXD + 1];
    const int nw2 = (max_N + 1) / 2 * 2;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned lt = (1u << lane) - 1u;
    unsigned short* W = s_w + warp * nw2;
    grid_dep_sync();
    sort_list(discs, ctl, n_disc, src, s_pre);
    if (blockIdx.x == 0)  // every sorted store is dense
        for (int s = tid; s < 2 * n_disc; s += SORT_BLOCK) ctl->lay[s >> 1][s & 1][dst] = Lay{0, 0, 0, 0};
    const int items = s_pre[2 * n_disc];
    for (int item = blockIdx.x; item < items; item += gridDim.x) {
        const int seg = sort_store(s_pre, 2 * n_disc, item), d = seg >> 1, sp = seg & 1;
        const Disc& D = discs[d];
        const long long n = ctl->count[d][sp];
        const Lay L = ctl->lay[d][sp][src];
        const int N = D.N, CHUNK = D.chunk, rs = __ffs(CHUNK) - 6, rm = (1 << rs) - 1, CPW = SORT_R >> rs;
        const int t = item - s_pre[seg];
        const long long chunks = chunks_of(L, n, CHUNK);
        const int32_t* __restrict__ cc = D.c[src][sp];
        for (int j = tid; j < SORT_NW * nw2 / 2; j += SORT_BLOCK) reinterpret_cast<unsigned*>(s_w)[j] = 0;
        const long long k0 = ((long long)t * SORT_NW + warp) * CPW;
        // the warp's chunk descriptors by its first lanes, then all cell loads
        const ChunkDesc my = lane < CPW && k0 + lane < chunks ? chunk_desc(L, n, D.start[sp], k0 + lane, CHUNK)
                                                             : ChunkDesc{0, 0, 0};
        unsigned kr[SORT_R];
#pragma unroll
        for (int r = 0; r < SORT_R; ++r) {
            const int ci = r >> rs, i = 32 * (r & rm) + lane;
            const int s0 = __shfl_sync(FULL, (int)my.src, ci), cnt = __shfl_sync(FULL, my.cnt, ci);
            kr[r] = i < cnt ? (unsigned)__ldcs(cc + s0 + i) : 0xFFFFu;
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < SORT_R; ++r) {
            if (kr[r] >= (unsigned)N) kr[r] = 0xFFFFu;  // past the store, or a corrupt cell index: not placed
            kr[r] |= row_rank(W, kr[r], N, lane, lt) << 16;
        }
        __syncthreads();
        unsigned* H = hist + hoff[seg] + (size_t)t * N;
        for (int j = tid; j < (N + 1) / 2; j += SORT_BLOCK) {  // two cells per word: prefix over the warps, tile counts
            unsigned run = 0;
#pragma unroll
            for (int w = 0; w < SORT_NW; ++w) {
                unsigned* p = reinterpret_cast<unsigned*>(s_w + w * nw2) + j;
                const unsigned v = *p;
                *p = run;
                run += v;
            }
            H[2 * j] = run & 0xFFFFu;
            if (2 * j + 1 < N) H[2 * j + 1] = run >> 16;
        }
        __syncthreads();
        unsigned* KR = kr_all + eoff[seg] + (size_t)t * SORT_TILE + warp * (32 * SORT_R) + lane;
#pragma unroll
        for (int r = 0; r < SORT_R; ++r) {
            const unsigned k = kr[r] & 0xFFFFu;
            KR[32 * r] = k < (unsigned)N ? kr[r] + ((unsigned)W[k] << 16) : 0xFFFFu;
        }
        __syncthreads();
    }
}

// Per (store, group of 32 cells): sort_rows.
__global__ void __launch_bounds__(1024) k_sort_rows(const Disc* __restrict__ discs, Ctl* __restrict__ ctl, int buf,
                                                    unsigned* __restrict__ hist, const long long* __restrict__ hoff,
                                                    unsigned* __restrict__ tot) {
    grid_dep_sync();
    const int seg = blockIdx.y, d = seg >> 1, sp = seg & 1;
    const int N = discs[d].N;
    if (blockIdx.x * 32 >= N) return;
    const unsigned Ts = (unsigned)sort_tiles(chunks_of(ctl->lay[d][sp][buf], ctl->count[d][sp], discs[d].chunk),
                                             discs[d].chunk);
    sort_rows(hist + hoff[seg], Ts, N, tot + (long long)seg * MAXN, &ctl->sort_rows_done[d][sp]);
}

template <typename T>
__global__ void __launch_bounds__(SORT_BLOCK) k_sort_scatter(const Disc* __restrict__ discs, int n_disc,
                                                             const Ctl* ctl, int src, int dst, const unsigned* hist,
                                                             const long long* __restrict__ hoff, const unsigned* tot,
                                                             const unsigned* kr_all,
                                                             const long long* __restrict__ eoff) {
    __shared__ int s_pre[2 * MAXD + 1];
    grid_dep_sync();
    sort_list(discs, ctl, n_disc, src, s_pre);
    using R = typename Rec<T>::type;
    constexpr int B = sizeof(T) == 4 ? 4 : 2;  // rows whose loads go out together
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int items = s_pre[2 * n_disc];
    for (int item = blockIdx.x; item < items; item += gridDim.x) {
        const int seg = sort_store(s_pre, 2 * n_disc, item), d = seg >> 1, sp = seg & 1;
        const Disc& D = discs[d];
        const int N = D.N, CHUNK = D.chunk, rs = __ffs(CHUNK) - 6, rm = (1 << rs) - 1, CPW = SORT_R >> rs;
        const int t = item - s_pre[seg];
        const long long n = ctl->count[d][sp];
        const Lay L = ctl->lay[d][sp][src];
        const long long chunks = chunks_of(L, n, CHUNK), k0 = ((long long)t * SORT_NW + warp) * CPW;
        const R* __restrict__ ps = reinterpret_cast<const R*>(D.p[src][sp]);
        R* __restrict__ pd = reinterpret_cast<R*>(D.p[dst][sp]);
        int32_t* __restrict__ cd = D.c[dst][sp];
        const unsigned* H = hist + hoff[seg] + (size_t)t * N;
        const unsigned* cstart = tot + (long long)seg * MAXN;
        const unsigned* KR = kr_all + eoff[seg] + (size_t)t * SORT_TILE + warp * (32 * SORT_R) + lane;
        const ChunkDesc my = lane < CPW && k0 + lane < chunks ? chunk_desc(L, n, D.start[sp], k0 + lane, CHUNK)
                                                             : ChunkDesc{0, 0, 0};
#pragma unroll 1
        for (int r0 = 0; r0 < SORT_R; r0 += B) {
            unsigned kr[B], o[B];
            R rec[B];
#pragma unroll
            for (int q = 0; q < B; ++q) kr[q] = __ldcs(KR + 32 * (r0 + q));
#pragma unroll
            for (int q = 0; q < B; ++q) {
                const int r = r0 + q, i = 32 * (r & rm) + lane;
                const int s0 = __shfl_sync(FULL, (int)my.src, r >> rs), cnt = __shfl_sync(FULL, my.cnt, r >> rs);
                if (i < cnt) rec[q] = ps[s0 + i];
                else kr[q] = 0xFFFFu;
            }
#pragma unroll
            for (int q = 0; q < B; ++q) {
                // A corrupt cell index (reported by the sweep): dropped. Coherent loads by their unrestricted
                // pointers, through L1: a tile's slots meet in one row of H. With __ldcg, which asks L2 for
                // each slot: 1e6 + 1e6 in 64 cells 36 -> 47 us, unsorted in 512 cells 63 -> 117.
                const unsigned k = kr[q] & 0xFFFFu;
                o[q] = k < (unsigned)N ? cstart[k] + H[k] + (kr[q] >> 16) : 0xFFFFFFFFu;
            }
#pragma unroll
            for (int q = 0; q < B; ++q)
                if (o[q] < (unsigned long long)n) {
                    cd[o[q]] = (int)(kr[q] & 0xFFFFu);
                    pd[o[q]] = rec[q];
                }
        }
    }
}

// Order-preserving repack of every store into a dense buffer (the slots keep their order): bounds
// the number of regions when the sort runs rarely or never. One warp per chunk.
template <typename T>
__global__ void k_repack(const Disc* __restrict__ discs, Ctl* __restrict__ ctl, int src, int dst) {
    grid_dep_sync();
    const int seg = blockIdx.y, d = seg >> 1, sp = seg & 1;
    const Disc& D = discs[d];
    const int CHUNK = D.chunk;
    const long long n = ctl->count[d][sp];
    const Lay L = ctl->lay[d][sp][src];
    const long long chunks = chunks_of(L, n, CHUNK);
    using R = typename Rec<T>::type;
    const R* ps = reinterpret_cast<const R*>(D.p[src][sp]);
    const int32_t* cs_ = D.c[src][sp];
    R* __restrict__ pd = reinterpret_cast<R*>(D.p[dst][sp]);
    int32_t* __restrict__ cd = D.c[dst][sp];
    const int lane = threadIdx.x & 31;
    const long long w0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = ((long long)gridDim.x * blockDim.x) >> 5;
    if (blockIdx.x == 0 && threadIdx.x == 0) ctl->lay[d][sp][dst] = Lay{0, 0, 0, 0};
    for (long long k = w0; k < chunks; k += nw) {
        const ChunkDesc c = chunk_desc(L, n, D.start[sp], k, CHUNK);
        for (int i = lane; i < c.cnt; i += 32) {
            cd[c.base + i] = __ldcs(cs_ + c.src + i);
            pd[c.base + i] = ldcg_rec(ps + c.src + i);
        }
    }
}

// 16-byte groups of the SoA arrays of a state transfer: W consecutive particles, their cells in
// one W-wide integer vector and each real array in one 16-byte vector.
template <typename T>
struct XferVec;
template <>
struct XferVec<float> {
    typedef int4 CV;
    typedef float4 RV;
    static constexpr int W = 4;
};
template <>
struct XferVec<double> {
    typedef int2 CV;
    typedef double2 RV;
    static constexpr int W = 2;
};

__device__ __forceinline__ bool aligned16(const void* a, const void* b, const void* c, const void* d,
                                          const void* e) {
    return ((reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b) | reinterpret_cast<uintptr_t>(c) |
             reinterpret_cast<uintptr_t>(d) | reinterpret_cast<uintptr_t>(e)) & 15) == 0;
}

// State upload: SoA arrays (device staging, or the caller's mapped pinned host arrays) -> the
// store's records; cells outside [0, N) are counted. With 16-byte aligned arrays each
// thread reads whole 16-byte groups (over the host link, wide loads keep more bytes in flight
// per thread), the ragged tail one by one. The last CTA sets the store: n particles, or none if a cell was
// out of range, dense in buffer buf; the count of such cells goes to *bad_out (mapped host memory). Bounded by
// the host link (1e6 particles, 20 MB: 99 us, the copy engine takes 97); the layout, the check word and its way
// back in this launch, and no staging for mapped arrays: a call of 1e6 particles 134 (250 where the
// staging had grown) -> 121 us.
template <typename T>
__global__ void k_pack_state(const Disc* __restrict__ discs, Ctl* __restrict__ ctl, int d, int sp, int buf, long long n,
                             const int32_t* __restrict__ c, const T* __restrict__ f, const T* __restrict__ vx,
                             const T* __restrict__ vy, const T* __restrict__ vz, unsigned* __restrict__ bad_out) {
    typedef XferVec<T> X;
    const Disc& D = discs[d];
    const long long t0 = blockIdx.x * (long long)blockDim.x + threadIdx.x, nt = (long long)gridDim.x * blockDim.x;
    const long long groups = aligned16(c, f, vx, vy, vz) ? n / X::W : 0;
    unsigned nbad = 0;
    for (long long g = t0; g < groups; g += nt) {
        const typename X::CV cv = reinterpret_cast<const typename X::CV*>(c)[g];
        const typename X::RV a = reinterpret_cast<const typename X::RV*>(f)[g];
        const typename X::RV b = reinterpret_cast<const typename X::RV*>(vx)[g];
        const typename X::RV e = reinterpret_cast<const typename X::RV*>(vy)[g];
        const typename X::RV h = reinterpret_cast<const typename X::RV*>(vz)[g];
        const int* cs = reinterpret_cast<const int*>(&cv);
        const T *as = reinterpret_cast<const T*>(&a), *bs = reinterpret_cast<const T*>(&b);
        const T *es = reinterpret_cast<const T*>(&e), *hs = reinterpret_cast<const T*>(&h);
#pragma unroll
        for (int k = 0; k < X::W; ++k) {
            nbad += (unsigned)cs[k] >= (unsigned)D.N;
            store_rec<T>(D.c[buf][sp], D.p[buf][sp], (unsigned)(g * X::W + k), Part<T>{cs[k], as[k], bs[k], es[k], hs[k]});
        }
    }
    for (long long i = groups * X::W + t0; i < n; i += nt) {
        const int ci = c[i];
        nbad += (unsigned)ci >= (unsigned)D.N;
        store_rec<T>(D.c[buf][sp], D.p[buf][sp], (unsigned)i, Part<T>{ci, f[i], vx[i], vy[i], vz[i]});
    }
    if (nbad) atomicAdd(&ctl->up_bad, nbad);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0 && atomicAdd(&ctl->up_done, 1u) == gridDim.x - 1) {
        __threadfence();
        const unsigned all_bad = atomicExch(&ctl->up_bad, 0u);
        ctl->up_done = 0;
        ctl->count[d][sp] = all_bad ? 0 : n;
        ctl->lay[d][sp][buf] = Lay{0, 0, 0, 0};
        *bad_out = all_bad;
    }
}

// Position i of the state in the store: regions (binary search of the start table; empty regions
// share their start) and then the dense part by offset.
__device__ __forceinline__ long long state_slot(const Lay& L, const int* st, int chunk, long long i) {
    if (i >= L.M) return L.D0 + (i - L.M);
    int lo = 0, hi = L.K - 1;  // last region with start <= i
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if ((long long)st[mid] <= i) lo = mid;
        else hi = mid - 1;
    }
    return (long long)lo * chunk + (i - st[lo]);
}

// State download: the store, read through its layout -> SoA arrays (device staging, or the
// caller's mapped pinned host arrays; null outputs are skipped). The count comes from the control
// block and goes to *n_out if that is not null; above cap nothing else is written. With 16-byte aligned
// outputs each thread writes whole 16-byte groups.
template <typename T>
__global__ void k_unpack_state(const Disc* __restrict__ discs, const Ctl* __restrict__ ctl, int d, int sp, int buf,
                               long long cap, int32_t* __restrict__ c, T* __restrict__ f, T* __restrict__ vx,
                               T* __restrict__ vy, T* __restrict__ vz, long long* __restrict__ n_out) {
    typedef XferVec<T> X;
    const Disc& D = discs[d];
    const long long n = ctl->count[d][sp];
    if (n_out && blockIdx.x == 0 && threadIdx.x == 0) *n_out = n;
    if (n > cap) return;
    const Lay L = ctl->lay[d][sp][buf];
    const int* st = D.start[sp];
    const long long t0 = blockIdx.x * (long long)blockDim.x + threadIdx.x, nt = (long long)gridDim.x * blockDim.x;
    const long long groups = aligned16(c, f, vx, vy, vz) ? n / X::W : 0;  // null is aligned
    for (long long g = t0; g < groups; g += nt) {
        typename X::CV cv;
        typename X::RV a, b, e, h;
        int* cs = reinterpret_cast<int*>(&cv);
        T *as = reinterpret_cast<T*>(&a), *bs = reinterpret_cast<T*>(&b);
        T *es = reinterpret_cast<T*>(&e), *hs = reinterpret_cast<T*>(&h);
#pragma unroll
        for (int k = 0; k < X::W; ++k) {
            const long long o = state_slot(L, st, D.chunk, g * X::W + k);
            load_rec<T>(D.p[buf][sp], (unsigned)o, as[k], bs[k], es[k], hs[k]);
            cs[k] = D.c[buf][sp][o];
        }
        if (c) reinterpret_cast<typename X::CV*>(c)[g] = cv;
        if (f) reinterpret_cast<typename X::RV*>(f)[g] = a;
        if (vx) reinterpret_cast<typename X::RV*>(vx)[g] = b;
        if (vy) reinterpret_cast<typename X::RV*>(vy)[g] = e;
        if (vz) reinterpret_cast<typename X::RV*>(vz)[g] = h;
    }
    for (long long i = groups * X::W + t0; i < n; i += nt) {
        const long long o = state_slot(L, st, D.chunk, i);
        T a, b, e, g;
        load_rec<T>(D.p[buf][sp], (unsigned)o, a, b, e, g);
        if (c) c[i] = D.c[buf][sp][o];
        if (f) f[i] = a;
        if (vx) vx[i] = b;
        if (vy) vy[i] = e;
        if (vz) vz[i] = g;
    }
}

// Several device arrays into one block of mapped host memory. A read-back of a few 10 KB is bounded by its
// launches: one of these in place of three to five copies (each about 8 us of engine and queue) takes
// pic_moments from 90 to 74 us at 512 cells (16 us of launch and copy; the rest is the host's
// conversion of the exact sums), a batch of 64 discharges' by 1.5 ms.
__global__ void __launch_bounds__(256) k_gather(const Gather g, unsigned* __restrict__ out) {
    const unsigned words = g.end[g.n - 1];
    for (unsigned i = blockIdx.x * 256 + threadIdx.x; i < words; i += gridDim.x * 256) {
        int q = 0;
        while (i >= g.end[q]) ++q;
        const unsigned k = i - (q ? g.end[q - 1] : 0u);
        out[g.off[q] / 4 + k] = __ldcg(static_cast<const unsigned*>(g.src[q]) + k);
    }
}

// Every store dense in buffer buf (after a load).
__global__ void k_set_dense(const Disc* __restrict__ discs, int n_disc, Ctl* __restrict__ ctl, int buf) {
    grid_dep_sync();
    const int i = threadIdx.x;
    if (i >= 2 * n_disc) return;
    ctl->lay[i >> 1][i & 1][buf] = Lay{0, 0, 0, 0};
}

// ---------------------------------------------------------------------------
__global__ void k_debug_philox(long long n, const uint32_t* __restrict__ ctr, uint32_t k0, uint32_t k1,
                               uint32_t* __restrict__ out) {
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const U4 r = philox4x32_10(ctr[4 * i], ctr[4 * i + 1], ctr[4 * i + 2], ctr[4 * i + 3], k0, k1);
    out[4 * i] = r.x;
    out[4 * i + 1] = r.y;
    out[4 * i + 2] = r.z;
    out[4 * i + 3] = r.w;
}

__global__ void k_debug_math(long long n, const float* __restrict__ x, const float* __restrict__ y,
                             float* __restrict__ lg, float* __restrict__ sn, float* __restrict__ cs) {
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= n) return;
    lg[i] = own_logf(x[i]);
    float s, c;
    own_sincospif(y[i], s, c);
    sn[i] = s;
    cs[i] = c;
}

}  // namespace pic

// ---------------------------------------------------------------------------
// Launch wrappers used by the host runtime.
#include "pic_launch.h"
#include "pic_limits.h"

namespace pic {

// Bounded-wait check, one warp: one mbarrier expecting a single arrival. With arrive = 0 nothing arrives, so
// the wait gives up after `tries` polls and the kernel reports ERR_TIMEOUT in *out; nothing is in
// flight when it returns. With arrive = 1 a thread arrives first and the wait succeeds. With arrive = 2 a
// thread arrives but lane 0 gives up without a poll: every lane has to report the timeout (ERR_NONFINITE if
// they differ).
__global__ void k_debug_wait(int arrive, int tries, int* out) {
    __shared__ __align__(8) unsigned long long mb;
    if (threadIdx.x == 0) mbar_init(&mb);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    __syncthreads();
    if (threadIdx.x == 0 && arrive)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&mb)) : "memory");
    const bool got = warp_wait(&mb, 0u, arrive == 2 && threadIdx.x == 0 ? 0 : tries);
    const unsigned m = __ballot_sync(FULL, got);
    if (threadIdx.x == 0) *out = m == FULL ? 0 : m == 0 ? ERR_TIMEOUT : ERR_NONFINITE;
}

template <typename K>
static cudaError_t smem_attr(K kern, size_t smem) {
    return raise_smem_limit(reinterpret_cast<const void*>(kern), smem);
}

// Launch with programmatic stream serialization: the grid may be scheduled while the kernel before
// it in the stream is still finishing (it takes SMs as they free up). Every such kernel calls
// grid_dep_sync() before it touches memory that kernels write, which returns once the kernel before has
// completed and its writes are visible. So the kernel-to-kernel gap of a step shrinks while the ordering
// stays that of plain launches.
template <typename... KArgs, typename... Args>
static cudaError_t launch_pdl(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                             Args... args) {
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
}

template <typename T, int PPT>
static cudaError_t launch_sweep_t(const SweepLaunch& L) {
    const unsigned rest = sweep_smem<T, PPT>(L.max_N, L.sets, L.warps, L.n_disc);
    const unsigned with_hi = rest + 4u * (L.max_N + 1);  // the array of the energies above 32 eV behind it
    const unsigned hi = with_hi <= SWEEP_SMEM_LIMIT ? rest : 0u;
    const size_t smem = hi ? with_hi : rest;
    auto kern = k_sweep<T, PPT>;
    cudaError_t e = smem_attr(kern, smem);
    if (e != cudaSuccess) return e;
    e = launch_pdl(kern, dim3(L.grid), dim3(32 * L.warps), smem, L.stream, L.discs, L.n_disc, L.ctl, L.in_buf, L.seed,
                   L.max_N, L.sets, hi);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

template <typename T>
static cudaError_t launch_sweep_p(const SweepLaunch& L) {
    if (L.ppt == 2) return launch_sweep_t<T, 2>(L);
    if (L.ppt == 8) return launch_sweep_t<T, 8>(L);
    return launch_sweep_t<T, 4>(L);
}

cudaError_t launch_sweep(const SweepLaunch& L) {
    return L.fp64 ? launch_sweep_p<double>(L) : launch_sweep_p<float>(L);
}

// Warps of a sweep CTA and its histogram sets. As many warps as registers and shared memory hold, but
// no more than the CTA's share of the chunks (small stores: a smaller CTA starts faster) and at least 4;
// two sets (no barrier between a discharge's electrons and ions) unless the second set costs more than
// a quarter of the warps (above about 2900 cells).
template <typename T, int PPT>
static void sweep_shape_t(int max_N, int n_disc, int want, long long chunks, int* warps, int* sets) {
    const int top = sweep_max_threads<T>() / 32;
    int fit[3] = {0, 0, 0};
    for (int s = 1; s <= 2; ++s)
        for (int w = 1; w <= top && sweep_smem<T, PPT>(max_N, s, w, n_disc) <= SWEEP_SMEM_LIMIT; ++w) fit[s] = w;
    *sets = 4 * fit[2] >= 3 * fit[1] ? 2 : 1;
    int w = fit[*sets];
    if (want > 0 && want < w) w = want;
    if (chunks < w) w = (int)chunks;
    *warps = w < 4 ? (fit[*sets] < 4 ? fit[*sets] : 4) : w;  // at least 2 fit at any size
}
void sweep_shape(int fp64, int ppt, int max_N, int n_disc, int want, long long chunks, int* warps, int* sets) {
    if (fp64) {
        if (ppt == 2) return sweep_shape_t<double, 2>(max_N, n_disc, want, chunks, warps, sets);
        if (ppt == 8) return sweep_shape_t<double, 8>(max_N, n_disc, want, chunks, warps, sets);
        return sweep_shape_t<double, 4>(max_N, n_disc, want, chunks, warps, sets);
    }
    if (ppt == 2) return sweep_shape_t<float, 2>(max_N, n_disc, want, chunks, warps, sets);
    if (ppt == 8) return sweep_shape_t<float, 8>(max_N, n_disc, want, chunks, warps, sets);
    sweep_shape_t<float, 4>(max_N, n_disc, want, chunks, warps, sets);
}

cudaError_t launch_finalize(int fp64, const Disc* discs, int n_disc, Ctl* ctl, int out_buf, int mode, int max_slices,
                            int max_N, cudaStream_t st) {
    const size_t smem = (mode & 8) ? 0 : sizeof(unsigned long long) * 2 * ((size_t)max_N + 1);
    const int nsl = (mode & 1) ? (max_slices > 0 ? max_slices : 1) : 0;
    const int parts = (mode & 8) ? 1 : max_N / FIELD_NODES + 2;  // field parts (y even), totals and moments parts (odd)
    const dim3 grid(nsl + parts, 2 * n_disc);
    const cudaError_t e = fp64 ? smem_attr(k_post<double>, smem) : smem_attr(k_post<float>, smem);
    if (e != cudaSuccess) return e;
    if (fp64)
        return launch_pdl(k_post<double>, grid, dim3(POST_BLOCK), smem, st, discs, n_disc, ctl, out_buf, mode, nsl,
                          max_N);
    return launch_pdl(k_post<float>, grid, dim3(POST_BLOCK), smem, st, discs, n_disc, ctl, out_buf, mode, nsl, max_N);
}

cudaError_t launch_load(int fp64, const Disc* discs, int n_disc, Ctl* ctl, int buf, unsigned long long seed,
                        int grid_x, cudaStream_t st) {
    dim3 g(grid_x, 2 * n_disc);
    if (fp64) k_load<double><<<g, 256, 0, st>>>(discs, ctl, buf, seed);
    else k_load<float><<<g, 256, 0, st>>>(discs, ctl, buf, seed);
    return cudaGetLastError();
}

cudaError_t launch_load_profile(int fp64, const Disc* discs, int n_disc, Ctl* ctl, int buf, unsigned long long seed,
                                const void* warm, int grid_x, cudaStream_t st) {
    dim3 g(grid_x, 2 * n_disc);
    if (fp64) k_load_profile<double><<<g, 256, 0, st>>>(discs, ctl, buf, seed, (const WarmDev<double>*)warm);
    else k_load_profile<float><<<g, 256, 0, st>>>(discs, ctl, buf, seed, (const WarmDev<float>*)warm);
    return cudaGetLastError();
}

size_t warm_desc_bytes(int fp64) { return fp64 ? sizeof(WarmDev<double>) : sizeof(WarmDev<float>); }

void warm_desc_fill(int fp64, void* out, const void* cdf_e, const void* cdf_i, const void* eps, int P, double scale,
                    double K23) {
    if (fp64) {
        WarmDev<double> w{};
        w.cdf[0] = (const double*)cdf_e;
        w.cdf[1] = (const double*)cdf_i;
        w.eps = (const double*)eps;
        w.P = P;
        w.scale = scale;
        w.K23 = K23;
        *(WarmDev<double>*)out = w;
    } else {
        WarmDev<float> w{};
        w.cdf[0] = (const float*)cdf_e;
        w.cdf[1] = (const float*)cdf_i;
        w.eps = (const float*)eps;
        w.P = P;
        w.scale = (float)scale;
        w.K23 = (float)K23;
        *(WarmDev<float>*)out = w;
    }
}

cudaError_t launch_deposit(int fp64, const Disc* discs, int n_disc, const Ctl* ctl, int buf, int max_N, int grid_x,
                           cudaStream_t st) {
    dim3 g(grid_x, 2 * n_disc);
    const size_t smem = sizeof(unsigned long long) * (max_N + 1);
    if (fp64) k_deposit<double><<<g, 256, smem, st>>>(discs, ctl, buf, max_N);
    else k_deposit<float><<<g, 256, smem, st>>>(discs, ctl, buf, max_N);
    return cudaGetLastError();
}

cudaError_t launch_backkick(int fp64, const Disc* discs, int n_disc, const Ctl* ctl, int buf, int grid_x,
                            cudaStream_t st) {
    dim3 g(grid_x, 2 * n_disc);
    if (fp64) k_backkick<double><<<g, 256, 0, st>>>(discs, ctl, buf);
    else k_backkick<float><<<g, 256, 0, st>>>(discs, ctl, buf);
    return cudaGetLastError();
}

cudaError_t launch_tables(int fp64, int n_pts, int n_proc, double de, double M, const double* se, const double* si,
                          void* Te, void* Ti, unsigned long long* kmax, cudaStream_t st) {
    const int g = (n_pts + 255) / 256;
    if (fp64) k_tables<double><<<g, 256, 0, st>>>(n_pts, n_proc, de, M, se, si, (double*)Te, (double*)Ti, kmax);
    else k_tables<float><<<g, 256, 0, st>>>(n_pts, n_proc, de, M, se, si, (float*)Te, (float*)Ti, kmax);
    return cudaGetLastError();
}

cudaError_t launch_sort(int fp64, const Disc* discs, int n_disc, Ctl* ctl, int src, int dst, unsigned* hist,
                        const long long* hoff, unsigned* tot, unsigned* kr, const long long* eoff, int max_N,
                        long long max_tiles, int sms, cudaStream_t st) {
    // CTAs: what the SMs hold (the counters take 32 bytes a cell), but not more than there can be tiles
    const size_t smem = 2 * (size_t)SORT_NW * ((max_N + 1) / 2 * 2);
    const int per = smem > 100 * 1024 ? 1 : smem > 70 * 1024 ? 2 : 3;
    auto grid = [&](int p) { return dim3((unsigned)(max_tiles < (long long)p * sms ? max_tiles : (long long)p * sms)); };
    cudaError_t e = smem_attr(k_sort_count, smem);
    if (e != cudaSuccess) return e;
    e = launch_pdl(k_sort_count, grid(per), dim3(SORT_BLOCK), smem, st, discs, n_disc, ctl, src, dst, hist, hoff, kr, eoff,
                   max_N);
    if (e != cudaSuccess) return e;
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    e = launch_pdl(k_sort_rows, dim3((max_N + 31) / 32, 2 * n_disc), dim3(1024), 0, st, discs, ctl, src, hist, hoff,
                   tot);
    if (e != cudaSuccess) return e;
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (fp64)
        return launch_pdl(k_sort_scatter<double>, grid(3), dim3(SORT_BLOCK), 0, st, discs, n_disc, ctl, src, dst, hist, hoff,
                          tot, kr, eoff);
    return launch_pdl(k_sort_scatter<float>, grid(3), dim3(SORT_BLOCK), 0, st, discs, n_disc, ctl, src, dst, hist, hoff, tot,
                      kr, eoff);
}

cudaError_t launch_repack(int fp64, const Disc* discs, int n_disc, Ctl* ctl, int src, int dst, int grid_x,
                          cudaStream_t st) {
    const dim3 g(grid_x, 2 * n_disc);
    if (fp64) return launch_pdl(k_repack<double>, g, dim3(256), 0, st, discs, ctl, src, dst);
    return launch_pdl(k_repack<float>, g, dim3(256), 0, st, discs, ctl, src, dst);
}

cudaError_t launch_pack_state(int fp64, const Disc* discs, Ctl* ctl, int d, int sp, int buf, long long n,
                              const int32_t* c, const void* const v[4], unsigned* bad_out, int grid, cudaStream_t st) {
    if (fp64)
        k_pack_state<double><<<grid, 256, 0, st>>>(discs, ctl, d, sp, buf, n, c, (const double*)v[0],
                                                   (const double*)v[1], (const double*)v[2], (const double*)v[3],
                                                   bad_out);
    else
        k_pack_state<float><<<grid, 256, 0, st>>>(discs, ctl, d, sp, buf, n, c, (const float*)v[0], (const float*)v[1],
                                                  (const float*)v[2], (const float*)v[3], bad_out);
    return cudaGetLastError();
}

cudaError_t launch_unpack_state(int fp64, const Disc* discs, const Ctl* ctl, int d, int sp, int buf, long long cap,
                                int32_t* c, void* const v[4], long long* n_out, int grid, cudaStream_t st) {
    if (fp64)
        k_unpack_state<double><<<grid, 256, 0, st>>>(discs, ctl, d, sp, buf, cap, c, (double*)v[0], (double*)v[1],
                                                     (double*)v[2], (double*)v[3], n_out);
    else
        k_unpack_state<float><<<grid, 256, 0, st>>>(discs, ctl, d, sp, buf, cap, c, (float*)v[0], (float*)v[1],
                                                    (float*)v[2], (float*)v[3], n_out);
    return cudaGetLastError();
}

cudaError_t launch_gather(const Gather& g, void* out, int sms, cudaStream_t st) {
    const unsigned ctas = (g.end[g.n - 1] + 255) / 256;
    k_gather<<<ctas < (unsigned)sms ? ctas : (unsigned)sms, 256, 0, st>>>(g, static_cast<unsigned*>(out));
    return cudaGetLastError();
}


long long sort_tile_chunks(int chunk) { return SORT_TILE / chunk; }

// Dynamic shared memory of a k_diag launch: its node arrays and, for a sample, the EEDF (bins > 0).
size_t diag_smem(int max_N, unsigned mask, int bins) {
    return (size_t)__builtin_popcount(mask) * 8 * ((size_t)max_N + 1) + 4 * (size_t)bins;
}

cudaError_t launch_diag(int fp64, const Disc* discs, int n_disc, const Ctl* ctl, int buf, const DiagArgs& A,
                        int max_N, int grid_x, cudaStream_t st) {
    const size_t smem = diag_smem(max_N, A.mask, (A.mode & DIAG_SAMPLE) ? A.bins : 0);
    const dim3 g(grid_x, n_disc);
    if (fp64) {
        cudaError_t e = smem_attr(k_diag<double>, smem);
        if (e != cudaSuccess) return e;
        return launch_pdl(k_diag<double>, g, dim3(DIAG_BLOCK), smem, st, discs, ctl, buf, A);
    }
    cudaError_t e = smem_attr(k_diag<float>, smem);
    if (e != cudaSuccess) return e;
    return launch_pdl(k_diag<float>, g, dim3(DIAG_BLOCK), smem, st, discs, ctl, buf, A);
}

cudaError_t launch_set_dense(const Disc* discs, int n_disc, Ctl* ctl, int buf, cudaStream_t st) {
    return launch_pdl(k_set_dense, dim3(1), dim3(128), 0, st, discs, n_disc, ctl, buf);
}

cudaError_t launch_debug_wait(int arrive, int tries, int* out, cudaStream_t st) {
    k_debug_wait<<<1, 32, 0, st>>>(arrive, tries, out);
    return cudaGetLastError();
}

cudaError_t launch_debug_philox(long long n, const uint32_t* ctr, uint32_t k0, uint32_t k1, uint32_t* out,
                                cudaStream_t st) {
    k_debug_philox<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, ctr, k0, k1, out);
    return cudaGetLastError();
}
cudaError_t launch_debug_math(long long n, const float* x, const float* y, float* lg, float* sn, float* cs,
                              cudaStream_t st) {
    k_debug_math<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, x, y, lg, sn, cs);
    return cudaGetLastError();
}

}  // namespace pic

// mhd_fx.cu -- the FP64 MHD substep with its derivatives in 64-bit fixed point.
//
// Of the 600 FP64 instructions per cell and substep of the kernel in mhd.cu, which kept the FP64
// pipe 80 % busy, 470 are the 57 linear differences of gamma = A B (Eq. 8).  Here they are sums of
// products on the integer pipe (fixed.cuh); the right-hand side of Eqs. A1-A4, the closure and
// the RK update stay in FP64, on the exact cell values.  One RK3 step of 256^3: 60.8 -> 32.6 ms.
//
//   * z-streaming as in mhd.cu: 16 x 8 cells per CTA, planes of all 8 fields in a ring of 8 slots.
//     An arriving plane is converted in place to biased 60-bit integers, one binary scale per plane
//     and field.
//   * Four groups of one thread per cell: three evaluate the derivatives of plane z, 2 to 3 fields each,
//     and convert the arriving plane; one assembles the right-hand side of plane z - 1 from their
//     results in shared memory, so that the FP64 pipe and the integer pipe work at the same time.
//     160^3, one substep: one thread per cell 5.1 ms, two groups 3.75, four groups 3.1 (128 registers
//     a thread).  Bound by the latency of dependent instructions at 4 warps per scheduler (128^3: issue
//     34 %, FP64 pipe 39 %): the ring leaves no shared memory for a second CTA.
//   * One body of code for all fields: unrolled it is 320 KB, and a substep took 24 ms.
//   * A cell uses, per field, the largest scale of the 7 planes of its window.  Where those
//     differ (11 % of the windows), values are shifted as they are read, a branch that is uniform per
//     block and field.  The scales depend on the planes' tiles alone, so results do not depend on
//     the split of z.
//   * Differences of values within 2^6 of the scale are exact before they are weighted, as in FP64,
//     and the sums keep 28 bits below the scale's 2^-60 (FxAcc::wide), so that small differences of
//     large values lose nothing to FP64.  Error of the right-hand side against extended precision:
//     0.03 to 0.95 times that of the FP64 kernel (rms; waves, noise, small waves on large means,
//     components far below their companions).
//   * A field is small at a cell where it and its six neighbours are below 2^-6 of the scale
//     (fixed.cuh says why), and where the scale is out of range, as with infinities and NaN.  A warp
//     with more than 4 such cells of a field takes that field's derivatives in FP64 from global
//     memory, in the operations of mhd.cu; fewer cells are marked unless the gradient shows terms of at
//     least 2^-6 of the scale, and evaluated in FP64 throughout at the end of the CTA.
//   * Accuracy by field, not by axis: next to larger neighbours on one axis, the difference of values
//     far below the scale along another is exact to 2^-60 of the scale only, where FP64 keeps its digits.
//   * One RK3 step in ms, the FP64 pipe's kernel and this one: 256^3 waves 60.8 and 32.6, a vortex of 24
//     cells in 256^3 60.8 and 51.9; 128^3 waves 7.9 and 5.0, a vortex of 6, 10, 16 cells 7.9 and 9.1, 9.0,
//     7.8, a shear layer 7.9 and 8.2 (before fields were taken in FP64 by warps 13.7, 16.9, 14.9, 17.1).
#include <algorithm>

#include "fixed.cuh"
#include "mhd_win.cuh"

namespace stn {
namespace {

constexpr int TX = 16, TY = 8, GROUP = TX * TY, NGROUPS = 4, NT = NGROUPS * GROUP, NSLOT = 8;
// Cells left to FP64: a bit each until the end of the chunk, then in lists of up to LIST cells (7 bits of
// the cell, 7 of the plane).
constexpr int LIST = 1024, MAX_PLANES = 128;
constexpr int FP64_CELLS = 4;  // more small cells of a warp than this: the field's derivatives in FP64
// What the groups of derivatives hand to the group of the right-hand side, per cell: u (Laplacian,
// h, gradient) 3 x 7, A (Laplacian, h, two of the gradient) 3 x 6, lnrho and s (gradient, Laplacian) 2 x 4.
constexpr int EX_A = 21, EX_LNRHO = 39, EX_SS = 43, NEX = 47;
using Cfg = MhdCfg<double, TX, TY, NSLOT>;
constexpr int FE = Cfg::FIELD_ELEMS, RS = Cfg::TXP;
constexpr int FPAIRS = Cfg::TXP * Cfg::ROWS / 2;  // 16-byte pairs of one field's tile
constexpr size_t SMEM = Cfg::SMEM + (size_t)NEX * GROUP * sizeof(double);
static_assert(FE == 2 * FPAIRS, "the tiles of a plane's fields are contiguous");

// Weights as 60-bit integers (2^28 h + l) at the scales 2^e1 (first differences), 2^e2 (second) and
// 2^em (mixed).  Their signs (+, -, + with the distance, centres negative) are compiled in.
struct FxMhd {
    u32 d1h[3][3], d1l[3][3], d2h[3][3], d2l[3][3], dmh[3][3], dml[3][3], ch[3], cl[3];
    int e1, e2, em;
    u64 k1[3], k2[3], km[3], klap;  // biases off the results: first, second and mixed differences, Laplacian
};

struct FxIn {
    const double *f[8];
};

// One field of one cell's window of converted planes; d[k]: how far plane k's scale lies below the
// cell's.
template <bool MIXED> struct FxWin {
    const u64 *p[7];
    int d[7];
    __device__ __forceinline__ u64 at(int k, int dx, int dy) const {
        const u64 v = p[k][dy * RS + dx];
        return MIXED ? fx_shift(v, FX_BIAS, d[k]) : v;
    }
    __device__ __forceinline__ u64 ax(int a, int s) const { return a == 0 ? at(3, s, 0) : a == 1 ? at(3, 0, s) : at(3 + s, 0, 0); }
    __device__ __forceinline__ u64 mx(int pair, int s1, int s2) const {
        return pair == 0 ? at(3, s1, s2) : pair == 1 ? at(3 + s2, s1, 0) : at(3 + s2, 0, s1);
    }
    __device__ __forceinline__ double d1(const FxMhd &w, int a, int sc) const {
        FxAcc acc(0);
#pragma unroll
        for (int k = 1; k <= 3; ++k) {
            const u64 hi = ax(a, k == 2 ? -k : k), lo = ax(a, k == 2 ? k : -k);
            acc.mac(w.d1h[a][k - 1], w.d1l[a][k - 1], hi + (2 * FX_BIAS - lo));
        }
        return acc.wide(w.k1[a], sc + w.e1);
    }
    __device__ __forceinline__ void d2(FxAcc &acc, const FxMhd &w, int a) const {
        acc.mac(w.ch[a], w.cl[a], 2 * FX_BIAS - at(3, 0, 0));
#pragma unroll
        for (int k = 1; k <= 3; ++k) {
            u64 s = ax(a, k) + ax(a, -k);
            if (k == 2) s = 4 * FX_BIAS - s;
            acc.mac(w.d2h[a][k - 1], w.d2l[a][k - 1], s);
        }
    }
    __device__ __forceinline__ double dm(const FxMhd &w, int pair, int sc) const {
        FxAcc acc(0);
#pragma unroll
        for (int k = 1; k <= 3; ++k) {
            const u64 same = mx(pair, k, k) + mx(pair, -k, -k);
            const u64 cross = mx(pair, k, -k) + mx(pair, -k, k);
            acc.mac(w.dmh[pair][k - 1], w.dml[pair][k - 1],
                    k == 2 ? cross + (4 * FX_BIAS - same) : same + (4 * FX_BIAS - cross));
        }
        return acc.wide(w.km[pair], sc + w.em);
    }
};

// Whether a field is below 2^-6 of the scale at a cell and its six neighbours; p: the cell in planes
// -1, 0, 1, whose scales lie d below it.
__device__ __forceinline__ bool field_small(const u64 *const (&p)[3], const int (&d)[3]) {
    bool small = true;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const u32 flag = d[k] < 6 ? FX_FLAG_HI << d[k] : FX_BIAS_HI, lo = FX_BIAS_HI - flag;
        u32 h = (u32)(p[k][0] >> 32) - lo;
        if (k == 1) {
            h = max(h, max((u32)(p[k][1] >> 32) - lo, (u32)(p[k][-1] >> 32) - lo));
            h = max(h, max((u32)(p[k][RS] >> 32) - lo, (u32)(p[k][-RS] >> 32) - lo));
        }
        small = small && h < 2 * flag;
    }
    return small;
}

// The derivatives some term uses of component c of a vector (c < 3; its own gradient component
// only where `own`), or of lnrho and s (c = 3): gradient, Laplacian, and h[a] = d_a d_c.
template <bool MIXED, bool CONDUCT>
__device__ __forceinline__ void field_derivs(const FxWin<MIXED> &w, const FxMhd &k, int sc, int c, bool own,
                                             double (&g)[3], double &lap, double (&h)[3]) {
#pragma unroll
    for (int a = 0; a < 3; ++a)
        if (own || a != c) g[a] = w.d1(k, a, sc);
    if (CONDUCT || c < 3) {
        FxAcc all(0);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            FxAcc one(0);
            w.d2(one, k, a);
            if (a == c) h[a] = one.wide(k.k2[a], sc + k.e2);
            all.add(one);
        }
        lap = all.wide(k.klap, sc + k.e2);
    }
    if (c < 3) {
#pragma unroll
        for (int pair = 0; pair < 3; ++pair) {  // (0,1), (0,2), (1,2)
            const int a = pair == 2 ? 1 : 0, b = pair == 0 ? 1 : 2;
            if (c == a || c == b) {
                const double m = w.dm(k, pair, sc);
                if (c == a) h[b] = m;
                else h[a] = m;
            }
        }
    }
}

// Where the derivatives of field q (component c, or 3) go: Laplacian, h, gradient.
__device__ __forceinline__ int ex_of(int q, int c) { return c == 3 ? (q == F_SS ? EX_SS : EX_LNRHO) : q < F_AX ? 7 * c : EX_A + 6 * c; }
__device__ __forceinline__ void put_derivs(double *e, int c, bool own, bool laplacian, const double (&g)[3], double lap,
                                           const double (&h)[3]) {
    if (c == 3) {
#pragma unroll
        for (int a = 0; a < 3; ++a) e[a * GROUP] = g[a];
        if (laplacian) e[3 * GROUP] = lap;
        return;
    }
    e[0] = lap;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        e[(1 + a) * GROUP] = h[a];
        if (own) e[(4 + a) * GROUP] = g[a];
        else if (a != c) e[(a == (c + 1) % 3 ? 4 : 5) * GROUP] = g[a];
    }
}

// The same derivatives of one field at one cell (f) by FP64 from global memory, in the operations
// of mhd.cu, stored at e.
struct FieldWin : WinOps<double, FieldWin> {
    const double *f;
    int64_t sy, sz;
    __device__ __forceinline__ double at(int, int k, int dx, int dy) const { return f[(k - 3) * sz + dy * sy + dx]; }
};
template <bool CONDUCT>
__device__ __noinline__ void field_fp64(const double *f, int64_t sy, int64_t sz, const MK<double> *k, int c, bool own, double *e) {
    FieldWin w;
    w.f = f;
    w.sy = sy;
    w.sz = sz;
    double g[3], h[3] = {}, lap = 0.0;
#pragma unroll
    for (int a = 0; a < 3; ++a)
        if (own || a != c) g[a] = w.d1(0, a, k->d1[a]);
    if (CONDUCT || c < 3) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const double one = w.d2(0, a, k->d2c[a], k->d2[a]);
            if (a == c) h[a] = one;
            lap = a == 0 ? one : add(lap, one);
        }
    }
    if (c < 3) {
#pragma unroll
        for (int pair = 0; pair < 3; ++pair) {  // (0,1), (0,2), (1,2)
            const int a = pair == 2 ? 1 : 0, b = pair == 0 ? 1 : 2;
            if (c == a || c == b) {
                const double m = w.dmix(0, pair, k->dm[pair]);
                if (c == a) h[b] = m;
                else h[a] = m;
            }
        }
    }
    put_derivs(e, c, own, CONDUCT, g, lap, h);
}

// What follows the right-hand side of one cell: the RK update and its stores, or the dense result.
template <int MODE>
__device__ __forceinline__ void finish_cell(const MK<double> &k, const double (&rhs)[8], const double (&val)[8],
                                            const double (&w)[8], bool first, bool last, double *wbuf, const Ptrs8 &fout,
                                            const Ptrs8 &rbuf, const Geom &g, bool images, bool edge, int64_t cell,
                                            int64_t oidx, int x, int y, int z) {
    if (MODE == 1) {
#pragma unroll
        for (int q = 0; q < 8; ++q) static_cast<double *>(rbuf.p[q])[cell] = rhs[q];
        return;
    }
    double wn[8], fn[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        double kn;
        rk_update<false>(k, first, rhs[q], w[q], 0.0, val[q], wn[q], fn[q], kn, [](double v) { return v; });
    }
    if (!last) store8<double>(wbuf + 8 * cell, wn);
    if (images && edge) {
#pragma unroll
        for (int q = 0; q < 8; ++q) store_with_images(static_cast<double *>(fout.p[q]), g, R6, true, x, y, z, fn[q]);
    } else {
#pragma unroll
        for (int q = 0; q < 8; ++q) static_cast<double *>(fout.p[q])[oidx] = fn[q];
    }
}

// One cell by FP64 throughout, from global memory, as the kernel of mhd.cu evaluates it.
template <int MODE, bool CONDUCT>
__device__ __noinline__ void fp64_cell(const FxIn &in, const Ptrs8 &fout, double *wbuf, const Ptrs8 &rbuf, const Geom &g,
                                       const MK<double> &k, int first, int last, int images, int x, int y, int z) {
    GlobalWin w;
    const int64_t at = g.idx(x, y, z), cell = x + g.n[0] * (y + g.n[1] * z);
#pragma unroll
    for (int q = 0; q < 8; ++q) w.f[q] = in.f[q] + at;
    w.sy = g.pad[0];
    w.sz = g.pad[0] * g.pad[1];
    double rhs[8], val[8], wold[8] = {};
    mhd_rhs_cell<CONDUCT, double>(w, k, rhs, val);
    if (MODE == 0 && !first) load8<double, double>(wbuf + 8 * cell, wold);
    finish_cell<MODE>(k, rhs, val, wold, first != 0, last != 0, wbuf, fout, rbuf, g, images != 0, true, cell, at, x, y, z);
}

template <int MODE, bool CONDUCT>
__global__ void __launch_bounds__(NT, 1)
mhd_fx_kernel(const __grid_constant__ MhdMaps maps, const __grid_constant__ FxIn in, const __grid_constant__ Ptrs8 fout,
              double *wbuf, const __grid_constant__ Ptrs8 rbuf, const __grid_constant__ Geom g,
              const __grid_constant__ MK<double> kp, const __grid_constant__ FxMhd fw, int zc, int first, int last,
              int images, unsigned *err) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    u64 *ring = reinterpret_cast<u64 *>(smem_raw + ((128u - (smem_addr(smem_raw) & 127u)) & 127u));
    __shared__ __align__(8) uint64_t full[NSLOT];
    __shared__ int scale[NSLOT][8];  // exponent codes of each slot's plane, per field
    __shared__ int top[2][8], low[2][8];  // the largest and smallest of a window, by parity
    __shared__ MK<double> ks;  // FP64 operands from registers rather than the constant bank (mhd.cu)
    __shared__ u32 marks[MAX_PLANES][GROUP / 32];
    __shared__ uint16_t list[LIST];
    __shared__ u32 listed, unlisted;
    double *ex = reinterpret_cast<double *>(ring + NSLOT * Cfg::SLOT_ELEMS);
    __shared__ unsigned char exleft[NGROUPS][GROUP];
    const int tid = threadIdx.x, lane = tid & 31, group = tid / GROUP, gt = tid % GROUP, tx = gt % TX, ty = gt / TX;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY, zc0 = blockIdx.z * zc;
    const int nx = (int)g.n[0], ny = (int)g.n[1], nz = (int)g.n[2];
    const int count = min(nz, zc0 + zc) - zc0, nplanes = count + 2 * R6;
    const int x = x0 + tx, y = y0 + ty;
    const bool active = x < nx && y < ny;

    for (int i = tid; i < (int)(sizeof(MK<double>) / sizeof(double)); i += NT)
        reinterpret_cast<double *>(&ks)[i] = reinterpret_cast<const double *>(&kp)[i];
    if (tid == 0) {
        for (int q = 0; q < 8; ++q) tma_prefetch_desc(&maps.m[q]);
        for (int s = 0; s < NSLOT; ++s) {
            mbar_init(&full[s], 1);
            for (int q = 0; q < 8; ++q) scale[s][q] = 0;
        }
        mbar_fence_init();
    }
    __syncthreads();
    const int bx = (int)g.off[0] + x0 - Cfg::HX;
    const int by0 = (int)g.off[1] + y0 - R6;
    const int bz0 = (int)g.off[2] + zc0 - R6;
    int issued = 0;
    auto issue = [&](int j) {
        const int s = j & (NSLOT - 1);
        mbar_arrive_expect_tx(&full[s], 8 * Cfg::BOX_BYTES);
        for (int q = 0; q < 8; ++q)
            tma_load_3d(ring + s * Cfg::SLOT_ELEMS + q * FE, &maps.m[q], &full[s], bx, by0, bz0 + j);
    };
    if (tid == 0)
        for (; issued < NSLOT && issued < nplanes; ++issued) issue(issued);

    // pairs beyond the interior and its halo in x and y are padding or lie outside the field: they
    // count as 0 (tiles inside skip the test)
    const bool rim = x0 + TX + Cfg::HX > nx + R6 || x0 < Cfg::HX || y0 + TY + R6 > ny + R6;
    auto kept = [&](int pair, int u) -> bool {  // pair of one field's tile
        const int row = pair / (RS / 2), gx = x0 - Cfg::HX + 2 * (pair - row * (RS / 2)) + u;
        return gx >= -R6 && gx < nx + R6 && y0 - R6 + row < ny + R6;
    };
    bool ok = true;
    // the largest exponents of plane j's fields
    auto scan = [&](int j, int q0, int nq) {
        const int s = j & (NSLOT - 1);
        ok = ok && mbar_wait_bounded(&full[s], ((unsigned)j / NSLOT) & 1u);
        const double2 *src = reinterpret_cast<const double2 *>(ring + s * Cfg::SLOT_ELEMS);
#pragma unroll 2
        for (int q = q0; q < q0 + nq; ++q) {
            u32 hm = 0u, any = 0u;
#pragma unroll
            for (int i = gt; i < FPAIRS; i += GROUP) {
                double2 v = src[q * FPAIRS + i];
                if (rim) {
                    if (!kept(i, 0)) v.x = 0.0;
                    if (!kept(i, 1)) v.y = 0.0;
                }
                const u32 hx = (u32)__double2hiint(v.x) & 0x7fffffffu, hy = (u32)__double2hiint(v.y) & 0x7fffffffu;
                hm = max(hm, max(hx, hy));
                any |= (u32)__double2loint(v.x) | (u32)__double2loint(v.y);
            }
            hm = __reduce_max_sync(0xffffffffu, hm);
            const bool nonzero = __any_sync(0xffffffffu, (hm | any) != 0u);
            // odd codes only: half as many windows of planes whose scales differ
            const int code = fx_code(hm, nonzero);
            if (lane == 0 && code) atomicMax(&scale[s][q], code | 1);
        }
    };
    auto convert = [&](int j, int q0, int nq) {
        const int s = j & (NSLOT - 1);
        double2 *buf = reinterpret_cast<double2 *>(ring + s * Cfg::SLOT_ELEMS);
#pragma unroll 2
        for (int q = q0; q < q0 + nq; ++q) {
            const int e = max(scale[s][q], FX_EMIN);  // below it nothing shows at a scale the sums use
#pragma unroll
            for (int i = gt; i < FPAIRS; i += GROUP) {
                double2 v = buf[q * FPAIRS + i];
                if (rim) {
                    if (!kept(i, 0)) v.x = 0.0;
                    if (!kept(i, 1)) v.y = 0.0;
                }
                reinterpret_cast<ulonglong2 *>(buf)[q * FPAIRS + i] =
                    make_ulonglong2(fx_from_double(v.x, e), fx_from_double(v.y, e));
            }
        }
    };
    auto window = [&](int m) {  // by 8 threads: the scales of the window of plane m
        if (gt < 8) {
            int hi = 0, lo = 4096;
            for (int k = 0; k < 7; ++k) {
                const int e = scale[(m + k) & (NSLOT - 1)][gt];
                hi = max(hi, e);
                lo = min(lo, e);
            }
            top[m & 1][gt] = hi;
            low[m & 1][gt] = lo;
        }
    };
    for (int j = 0; j < 2 * R6 + 1; ++j) scan(j, 2 * group, 2);
    bool bad = __syncthreads_or(!ok);
    for (int j = 0; j < 2 * R6 + 1; ++j) convert(j, 2 * group, 2);
    if (group == 0) window(0);
    __syncthreads();

    const int64_t nxy = g.n[0] * g.n[1], pitch_z = g.pad[0] * g.pad[1];
    int64_t cell = x + g.n[0] * y + nxy * zc0, oidx = g.idx(x, y, zc0);
    const bool edge_xy = x < R6 || x >= nx - R6 || y < R6 || y >= ny - R6;
    const int own = (ty + R6) * RS + tx + Cfg::HX;
    // Period m: groups 1 to 3 evaluate the derivatives of plane m and convert plane m + 7, while group 0
    // assembles the right-hand side of plane m - 1.
    for (int m = 0; !bad && m <= count; ++m) {
        if (group == 0) {
            if (m > 0 && gt == 0 && m + 1 < count) {  // plane m - 1 has been read for the last time
                fence_proxy_async();  // the block's generic writes to the slot before its next TMA load
                const int s = (m - 1) & (NSLOT - 1);
                for (int q = 0; q < 8; ++q) scale[s][q] = 0;
                issue(issued++);
            }
            double wcur[8] = {}, val[8];
            MhdDerivs<double> d;
            bool left = false;
            const bool some = active && m > 0;
            if (some) {
                if (MODE == 0 && !first) load8<double, double>(wbuf + 8 * cell, wcur);
#pragma unroll
                for (int q = 0; q < 8; ++q) val[q] = in.f[q][oidx];
                const double *e = ex + gt;
                auto get = [&](int i) { return e[i * GROUP]; };
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    const int b = (a + 1) % 3, c = (a + 2) % 3;
                    d.lapu[a] = get(7 * a);
                    d.gdivu[a] = add(add(get(1 + a), get(8 + a)), get(15 + a));
                    d.lapa[a] = get(EX_A + 6 * a);
                    d.gdiva[a] = add(add(get(EX_A + 1 + a), get(EX_A + 7 + a)), get(EX_A + 13 + a));
#pragma unroll
                    for (int k = 0; k < 3; ++k) d.gu[a][k] = get(7 * a + 4 + k);
                    (a == 0 ? d.bx : a == 1 ? d.by : d.bz) = sub(get(EX_A + 6 * c + 5), get(EX_A + 6 * b + 4));
                    d.glr[a] = get(EX_LNRHO + a);
                    d.gs[a] = get(EX_SS + a);
                }
                if constexpr (CONDUCT) {
                    d.laplr = get(EX_LNRHO + 3);
                    d.laps = get(EX_SS + 3);
                }
                left = exleft[1][gt] | exleft[2][gt] | exleft[3][gt];
            }
            asm volatile("bar.arrive 2, %0;" ::"n"(NT) : "memory");  // ex has been read
            const u32 mark = __ballot_sync(0xffffffffu, left);
            if (m > 0 && lane == 0) marks[m - 1][gt / 32] = mark;
            if (some && !left) {
                const int z = zc0 + m - 1;
#pragma unroll
                for (int q = 0; q < 8; ++q) d.val[q] = val[q];
                double rhs[8];
                mhd_rhs_assemble<CONDUCT>(d, ks, rhs);
                finish_cell<MODE>(ks, rhs, val, wcur, first != 0, last != 0, wbuf, fout, rbuf, g, images != 0,
                                  edge_xy || z < R6 || z >= nz - R6, cell, oidx, x, y, z);
            }
            if (m > 0) {
                cell += nxy;
                oidx += pitch_z;
            }
        } else {
            const u64 *plane[7];
#pragma unroll
            for (int k = 0; k < 7; ++k) plane[k] = ring + ((m + k) & (NSLOT - 1)) * Cfg::SLOT_ELEMS + own;
            // group 1: u_x, u_y; 2: u_z, A_x, s; 3: A_y, A_z, lnrho (54, 60 and 57 products)
            const u32 todo = group == 1 ? 0x21u : group == 2 ? 0x743u : 0x065u;
            const int n = group == 1 ? 2 : 3;
            bool left = false;  // to FP64
            // one body of code for all fields: unrolled it is 320 KB and waits for instructions
#pragma unroll 1
            for (int i = 0; i < n; ++i) {
                const int q = (int)(todo >> 4 * i & 15u);
                const int c = q == F_LNRHO || q == F_SS ? 3 : q < F_AX ? q - F_UX : q - F_AX;
                const bool own_grad = q < F_AX;
                double g3[3], lap, h3[3];
                const bool some = active && m < count;
                int sc = top[m & 1][q];
                const bool in_range = sc >= FX_SMIN && sc <= FX_EMAX;  // all zeros count as in range
                bool small = false;
                if (some) {
                    const u64 *const c3[3] = {plane[2] + q * FE, plane[3] + q * FE, plane[4] + q * FE};
                    const int d3[3] = {sc - scale[(m + 2) & (NSLOT - 1)][q], sc - scale[(m + 3) & (NSLOT - 1)][q],
                                       sc - scale[(m + 4) & (NSLOT - 1)][q]};
                    small = in_range ? field_small(c3, d3) : sc != 0;
                }
                // where many cells of a warp are small, its cells' derivatives are taken in FP64
                const bool fp64 = __popc(__ballot_sync(0xffffffffu, small)) > FP64_CELLS;
                if (some && !fp64) {
                    if (low[m & 1][q] == sc || !in_range) {
                        FxWin<false> w;
#pragma unroll
                        for (int k = 0; k < 7; ++k) w.p[k] = plane[k] + q * FE;
                        field_derivs<false, CONDUCT>(w, fw, in_range ? sc : 1023, c, own_grad, g3, lap, h3);
                    } else {
                        FxWin<true> w;
#pragma unroll
                        for (int k = 0; k < 7; ++k) {
                            w.p[k] = plane[k] + q * FE;
                            w.d[k] = sc - scale[(m + k) & (NSLOT - 1)][q];
                        }
                        field_derivs<true, CONDUCT>(w, fw, sc, c, own_grad, g3, lap, h3);
                    }
                    if (small) {  // and its gradient too: the cell goes to FP64
                        int top_g = 0;
#pragma unroll
                        for (int a = 0; a < 3; ++a)
                            if (own_grad || a != c) top_g = max(top_g, __double2hiint(g3[a]) & 0x7fffffff);
                        left = left || !in_range || (top_g >> 20) < sc + fw.e1 - 5;
                    }
                }
                if (i == 0) asm volatile("bar.sync 2, %0;" ::"n"(NT) : "memory");
                if (some) {
                    double *e = ex + ex_of(q, c) * GROUP + gt;
                    if (fp64) field_fp64<CONDUCT>(in.f[q] + oidx + m * pitch_z, g.pad[0], pitch_z, &ks, c, own_grad, e);
                    else put_derivs(e, c, own_grad, CONDUCT, g3, lap, h3);
                }
            }
            exleft[group][gt] = left;
            if (m + 1 < count) {
                const int j = m + 2 * R6 + 1, q0 = group == 1 ? 0 : group == 2 ? 3 : 5, nq = group == 2 ? 2 : 3;
                scan(j, q0, nq);
                asm volatile("bar.sync 1, %0;" ::"n"(NT - GROUP) : "memory");
                if (group == 1) window(m + 1);
                convert(j, q0, nq);
            }
        }
        bad = __syncthreads_or(!ok);
    }
    if (bad) {
        if (tid == 0) {
            atomicOr(err, ERR_TIMEOUT);
            for (int j = max(0, issued - NSLOT); j < issued; ++j)
                (void)mbar_wait_bounded(&full[j & (NSLOT - 1)], ((unsigned)j / NSLOT) & 1u, 100000000ull);
        }
        return;
    }
    // The marked cells by all threads, in lists that the first warp fills (the loop ended with a barrier).
    const u32 *mark = &marks[0][0];
    const int words = count * (GROUP / 32);
    for (int at = 0;;) {
        if (tid < 32) {
            u32 n = 0;
            while (at < words) {  // 32 words at most fill a list
                u32 bits = at + lane < words ? mark[at + lane] : 0u;
                const u32 own_n = __popc(bits);
                u32 upto = own_n;
#pragma unroll
                for (int d = 1; d < 32; d *= 2) {
                    const u32 other = __shfl_up_sync(0xffffffffu, upto, d);
                    if (lane >= d) upto += other;
                }
                const u32 total = __shfl_sync(0xffffffffu, upto, 31);
                if (n + total > (u32)LIST) break;
                for (u32 i = n + upto - own_n; bits; bits &= bits - 1, ++i)
                    list[i] = (uint16_t)((at + lane) * 32 + __ffs((int)bits) - 1);
                n += total;
                at += 32;
            }
            if (lane == 0) {
                listed = n;
                unlisted = at < words;
            }
        }
        __syncthreads();
        const bool again = unlisted;
        for (u32 i = tid; i < listed; i += NT) {
            const int t = (int)(list[i] & (GROUP - 1u)), z = zc0 + (int)(list[i] / GROUP);
            fp64_cell<MODE, CONDUCT>(in, fout, wbuf, rbuf, g, ks, first, last, images, x0 + t % TX, y0 + t / TX, z);
        }
        if (!again) break;
        __syncthreads();
    }
}

// The weights in fixed point; false where they do not fit (spacings of very different size).
bool fx_mhd_weights(const MhdConst &c, FxMhd &o) {
    // sums of the weights' magnitudes: at most 2^60 as integers, so that the accumulators hold them
    // (values enter at most 4 at a time, |results| < 2^62)
    double s1 = 0.0, s2 = 0.0, sm = 0.0, least = INFINITY, most = 0.0;
    for (int a = 0; a < 3; ++a) {
        double t1 = 0.0, tm = 0.0;
        s2 += std::fabs(c.d2c[a]);
        for (int k = 0; k < 3; ++k) {
            t1 += std::fabs(c.d1[a][k]);
            s2 += std::fabs(c.d2[a][k]);
            tm += std::fabs(c.dm[a][k]);
        }
        s1 = std::fmax(s1, t1);
        sm = std::fmax(sm, tm);
        least = std::fmin(least, t1);
        most = std::fmax(most, t1);
    }
    // spacings within a factor of 8: the weights of the coarsest axis keep their bits
    if (!(least > 0.0) || !std::isfinite(s1) || !std::isfinite(s2) || !std::isfinite(sm) || most > 8.0 * least) return false;
    (void)std::frexp(s1, &o.e1);
    (void)std::frexp(s2, &o.e2);
    (void)std::frexp(sm, &o.em);
    for (int e : {o.e1, o.e2, o.em})
        if (e < -100 || e > 100) return false;
    auto put = [](double w, int e, u32 &h, u32 &l) -> u64 {
        const u64 W = (u64)std::llrint(std::ldexp(std::fabs(w), 60 - e));
        h = (u32)(W >> 28);
        l = (u32)(W & 0xfffffffu);
        return W;
    };
    o.klap = 0;
    for (int a = 0; a < 3; ++a) {
        u64 t1 = 0, t2 = 0, tm = 0;
        for (int k = 0; k < 3; ++k) {
            t1 += put(c.d1[a][k], o.e1, o.d1h[a][k], o.d1l[a][k]);
            t2 += put(c.d2[a][k], o.e2, o.d2h[a][k], o.d2l[a][k]);
            tm += put(c.dm[a][k], o.em, o.dmh[a][k], o.dml[a][k]);
        }
        // a bias of 2^60 is a unit of the result per unit of weight
        o.k1[a] = 0ull - 2ull * t1;
        o.k2[a] = 0ull - 2ull * t2 - put(c.d2c[a], o.e2, o.ch[a], o.cl[a]);
        o.km[a] = 0ull - 4ull * tm;
        o.klap += o.k2[a];
    }
    return true;
}

// Planes per z-chunk: the fewest periods over the waves of CTAs (one per SM), when a chunk's start costs
// `start` of them.  Localised fields make some CTAs cost twice what others do, and few long chunks
// leave the SMs unevenly loaded, so chunks have at most 32 planes where the tiles are fewer than two per SM,
// else 64 (128^3, 128 tiles, ms a step in chunks of 128, 64, 32 planes: a vortex of 16 cells 14.8, 10.2,
// 7.8, a shear layer 13.7, 9.6, 8.2, waves 5.05, 5.2, 5.1; 256^3, 512 tiles, in chunks of 64 and 32: waves
// 33.7 and 34.3, a vortex of 24 cells 52.8 and 52.6).
int chunk_planes(int tiles, int nz, int start) {
    const int sms = device_sms();
    int best = 1;
    int64_t least = INT64_MAX;
    const int most = tiles < 2 * sms ? 32 : 64;
    for (int c = (nz + most - 1) / most; c <= nz; ++c) {
        const int zc = (nz + c - 1) / c;
        const int64_t ctas = (int64_t)tiles * ((nz + zc - 1) / zc), cost = (ctas + sms - 1) / sms * (zc + start);
        if (cost < least) {
            least = cost;
            best = zc;
        }
        if (zc == 1) break;
    }
    return best;
}

template <int MODE, bool CONDUCT>
cudaError_t run(int sub, const MhdMaps &maps, const FxIn &in, const Ptrs8 &fo, double *w, const Ptrs8 &rhs, const Geom &g,
                const MK<double> &k, const FxMhd &fw, bool images, unsigned *err, cudaStream_t s, int start,
                int zmode) {
    auto kern = mhd_fx_kernel<MODE, CONDUCT>;
    static int ready[64] = {};  // per device: the shared-memory limit is raised
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!ready[dev]) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM);
        if (e != cudaSuccess) return e;
        ready[dev] = 1;
    }
    const int tx = (int)((g.n[0] + TX - 1) / TX), ty = (int)((g.n[1] + TY - 1) / TY), nz = (int)g.n[2];
    const int zc = std::min(zchunk_len(chunk_planes(tx * ty, nz, start), nz, zmode), MAX_PLANES);
    const dim3 grid(tx, ty, (unsigned)((nz + zc - 1) / zc));
    kern<<<grid, NT, SMEM, s>>>(maps, in, fo, w, rhs, g, k, fw, zc, sub == 0 ? 1 : 0, sub == 2 ? 1 : 0, images ? 1 : 0,
                                err);
    return cudaGetLastError();
}

}  // namespace

// Which fields run here.  A chunk of z costs 6 periods on top of its planes (the first window and
// its conversion, the last plane's right-hand side, the listed cells), 65 us at 10.8 us a plane and
// substep, where the FP64 kernel takes 24 us a plane: chunks of 5 planes and more gain.  The choice
// may not depend on the extent in z, or slabs would differ from the whole field in their last
// bits; with tiles for a third of the SMs and more the thinnest fields get chunks of 4 or more.
// Measured on one RK3 step, FP64 pipe and here: 256^3 60 784 and 33 755 us, 160^3 14 690 and 8885,
// 128 x 128 x 32 2288 and 1535, 128 x 128 x 7 536 and 473; below the line 32^3 174 and 268,
// 48 x 48 x 17 248 and 297 (but 64^3 1164 and 807).
bool mhd_fx_applies(const MhdConst &c, const Geom &g) {
    FxMhd w;
    const int64_t tiles = ((g.n[0] + TX - 1) / TX) * ((g.n[1] + TY - 1) / TY);
    return 3 * tiles > device_sms() && fx_mhd_weights(c, w);
}

cudaError_t launch_mhd_fx(int mode, int sub, const MhdMaps &maps, const Ptrs8 &fi, const Ptrs8 &fo, void *w,
                          const Ptrs8 &rhs, const Geom &g, const MhdConst &c, const MK<double> &k, bool images,
                          unsigned *err, cudaStream_t s, int variant, int zmode) {
    FxMhd fw;
    if (!fx_mhd_weights(c, fw)) return cudaErrorInvalidValue;
    FxIn in;
    for (int q = 0; q < 8; ++q) in.f[q] = static_cast<const double *>(fi.p[q]);
    const bool cond = c.K != 0.0;
    const int start = variant == 0 ? 6 : 2;
    double *wb = static_cast<double *>(w);
    if (mode == 0)
        return cond ? run<0, true>(sub, maps, in, fo, wb, rhs, g, k, fw, images, err, s, start, zmode)
                    : run<0, false>(sub, maps, in, fo, wb, rhs, g, k, fw, images, err, s, start, zmode);
    return cond ? run<1, true>(sub, maps, in, fo, wb, rhs, g, k, fw, images, err, s, start, zmode)
                : run<1, false>(sub, maps, in, fo, wb, rhs, g, k, fw, images, err, s, start, zmode);
}

}  // namespace stn

// diffusion_fx.cu -- FP64 forward-Euler step of the 3D heat equation (Sec. 3.2, Eqs. 4-7) with
// the stencil sum in 64-bit fixed point.
//
// The folded step f' = g0 f + sum_axes sum_{a=1..R} g_{axis,a} (f(+a) + f(-a)) is linear, and on
// the FP64 pipe (2 multiply-adds per clock and SM) its 19 operations took 0.57 ms per 256^3 step,
// 14 times what HBM needs.  Here every plane tile is converted once, in shared memory, to
// integers of one binary scale (fixed.cuh) and the sums run on the integer pipe.
//
//   * 2.5D z-streaming as in diffusion.cu: a CTA owns a 64 x 16 tile of the xy-plane and marches
//     along z; padded plane tiles (72 x (16 + 2R)) arrive by TMA in a ring of 16 slots.
//   * Between two block barriers a CTA works on three planes at once: it converts plane t in place
//     (a thread's share, held in registers since the last interval) to biased 60-bit integers at
//     the plane's scale, loads its share of plane t + 1 and reduces the largest exponent, and
//     computes the outputs of plane t - R - 1.  Half of the warps of each scheduler compute first and
//     half convert first, so that they wait for different things (256^3, r = 3: 244 us per step with all
//     in one order, 235 like this).
//   * A thread owns 2 x-cells.  An output uses the largest scale of the 2R+1 planes its z column
//     spans (S), and values of planes with a smaller one are shifted right, behind branches that
//     are uniform per block.  S depends on nothing but those plane tiles, so results do not
//     depend on how z is split into chunks or slabs.
//   * The pairs' sum runs in fixed point, the centre joins it in one FP64 multiply-add with its
//     exact value: beside g0 f, which is near f when the step is small, the pairs' weights would
//     lose their bits.
//   * With one grid spacing on all axes (ISO) the six values at distance a are summed first: three
//     64 x 64-bit products per cell instead of nine.
//   * The pairs' sum is off by at most 8 units of 2^-60 of 2^ew S (2^ew: above the sum of the
//     weights, one per distance and axis): seven of truncated and shifted values, one of rounding.
//     The weights' own rounding costs 2^-52 of the terms they weigh at r = 3, 2^-50 at r = 4.  A
//     chain of FP64 multiply-adds rounds each of its 1 + 6 R terms, so an output stays within the
//     chain's bound where one of its terms is at least 2^-6 (r = 1), 2^-7 (r = 2), 2^-8 of 2^ew S: the
//     centre's (g0 |f|), one of its six neighbours', or the sum itself.  Outputs that show none of
//     these are listed and evaluated by FP64 multiply-adds from global memory, in the order of
//     diffusion.cu, by all threads, every four planes if they are many and else at the end.
//   * A field that falls by more than the scale holds within a tile (a hot spot, a front) has mostly
//     such outputs.  A plane's outputs are all evaluated in FP64, with coalesced loads and without the
//     fixed-point sums, where a row in the middle of its tile lies 2^-8 and more below the plane's
//     largest value over half its length, and where its window meets infinities, NaN or the ends
//     of the exponent range.
//   * 256^3, r = 3, us per step, the FP64 pipe's kernel and this one: waves 596 and 235; a Gaussian of
//     8, 16, 32 cells 596 and 696, 672, 290; a front of 3 cells 595 and 531; waves at r = 1, 2, 4 221
//     and 194, 424 and 215, 821 and 261; 32^3 14.5 and 9.8.  A field of which nothing fits pays for the
//     exponents and the conversion beside the FP64 pipe's work, at r = 1 up to 1.45 times (221, 321).
#include <algorithm>

#include "fixed.cuh"
#include "internal.h"

namespace stn {
namespace {

template <int R, bool ISO> struct FxCoef {
    static constexpr int N = ISO ? R : 3 * R;
    FxWeights<N> w;       // of the pairs
    double g0, ga[3][R];  // the centre's; the pairs' for the outputs evaluated in FP64
    u32 small_c, small_a[3];  // high words below which the centre and a neighbour on each axis are small
};

template <int R> struct FxCfg {
    static constexpr int BY = 16, NT = 32 * BY, NSLOT = 16;
    static constexpr int TX = 64, TY = BY, HX = 4, TXP = TX + 2 * HX, ROWS = TY + 2 * R;
    static constexpr int PAIRS = TXP / 2 * ROWS;  // 16-byte pairs per plane tile
    static constexpr int KP = (PAIRS + NT - 1) / NT;
    // The last warp has one pair per thread to convert, of one row, and so the time for what is done once per plane.
    static_assert(KP == 2 && PAIRS - NT <= NT - 32, "");
    static constexpr int SLOT = ((TXP * ROWS * 8 + 127) / 128) * 128 / 8;
    static constexpr uint32_t BOX_BYTES = TXP * ROWS * 8;
    static constexpr size_t SMEM = (size_t)NSLOT * SLOT * 8 + 128;
    static constexpr int LIST = 2048, LIST_HIGH = 256;  // listed outputs; more are worked off before the end
    static_assert((NSLOT & (NSLOT - 1)) == 0, "ring depth is a power of two (slot = j & (NSLOT-1))");
    static_assert(NSLOT >= 2 * R + 4, "ring: an output's planes, the two being converted and loaded, one refill");
    static_assert(R >= 1 && R <= 4, "");
};

// One output by FP64 multiply-adds, as the floating-point kernel of diffusion.cu evaluates it.
template <int R, bool ISO>
__device__ __noinline__ double heat_fp64_cell(const double *__restrict__ in, const Geom &g, const FxCoef<R, ISO> &c,
                                              int x, int y, int z) {
    const double *p = in + g.idx(x, y, z);
    const int64_t py = g.pad[0], pz = g.pad[0] * g.pad[1];
    double acc = c.g0 * p[0];
#pragma unroll
    for (int a = 1; a <= R; ++a) {
        acc = fma(c.ga[0][a - 1], p[a] + p[-a], acc);
        acc = fma(c.ga[1][a - 1], p[a * py] + p[-a * py], acc);
        acc = fma(c.ga[2][a - 1], p[a * pz] + p[-a * pz], acc);
    }
    return acc;
}

// Two neighbouring outputs in the same way; p points at the first, 16-byte aligned, w holds g0 and
// ga[axis][distance - 1].
template <int R>
__device__ __noinline__ double2 heat_fp64_pair(const double *__restrict__ p, int64_t py, int64_t pz, const double *w) {
    double x[10];  // cells -4 .. 5
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        if (2 * k + 1 < 4 - R || 2 * k > 5 + R) continue;
        const double2 t = *reinterpret_cast<const double2 *>(p - 4 + 2 * k);
        x[2 * k] = t.x;
        x[2 * k + 1] = t.y;
    }
    double2 n[2][R][2];  // [y, z][distance - 1][+, -]
#pragma unroll
    for (int a = 1; a <= R; ++a) {
        n[0][a - 1][0] = *reinterpret_cast<const double2 *>(p + a * py);
        n[0][a - 1][1] = *reinterpret_cast<const double2 *>(p - a * py);
        n[1][a - 1][0] = *reinterpret_cast<const double2 *>(p + a * pz);
        n[1][a - 1][1] = *reinterpret_cast<const double2 *>(p - a * pz);
    }
    double acc[2] = {w[0] * x[4], w[0] * x[5]};
#pragma unroll
    for (int a = 1; a <= R; ++a) {
#pragma unroll
        for (int u = 0; u < 2; ++u) acc[u] = fma(w[a], x[4 + u + a] + x[4 + u - a], acc[u]);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const double2 hi = n[e][a - 1][0], lo = n[e][a - 1][1];
            acc[0] = fma(w[(e + 1) * R + a], hi.x + lo.x, acc[0]);
            acc[1] = fma(w[(e + 1) * R + a], hi.y + lo.y, acc[1]);
        }
    }
    return make_double2(acc[0], acc[1]);
}

// Whether two biased values' high words are below the threshold t in magnitude.
__device__ __forceinline__ bool fx_below(u32 a, u32 b, u32 t) {
    const u32 lo = FX_BIAS_HI - t;
    return max(a - lo, b - lo) < 2 * t;
}

// Two neighbouring outputs: `cp` points at the first in its centre plane (scale sc - dc), z(k, u)
// gives the value of cell u at plane offset k != 0, at scale sc, f holds the centres' exact values;
// SAME: dc is 0.  Returns bit u set where output u is left to FP64.
template <int R, bool ISO, bool SAME, int TXP, typename Z>
__device__ __forceinline__ int fx_pair(const u64 *cp, const Z &z, int dc, int sc, const FxCoef<R, ISO> &c,
                                       const double2 f, double (&res)[2]) {
    constexpr int LOW = R == 1 ? 54 : R == 2 ? 53 : 52;  // |sum| below 2^LOW: small
    const FxWeights<FxCoef<R, ISO>::N> &w = c.w;
    // the thresholds at the centre plane's scale
    auto at_plane = [&](u32 t) { return SAME ? t : (u32)min((u64)t << min(dc, 28), (u64)FX_BIAS_HI); };
    const u32 tc = at_plane(c.small_c), tx = at_plane(c.small_a[0]), ty = ISO ? tx : at_plane(c.small_a[1]);
    u64 X[10];  // x window: cells -4 .. 5
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        if (2 * k + 1 < 4 - R || 2 * k > 5 + R) continue;
        const ulonglong2 t = *reinterpret_cast<const ulonglong2 *>(cp - 4 + 2 * k);
        X[2 * k] = t.x;
        X[2 * k + 1] = t.y;
    }
    FxAcc acc[2];
    bool small[2];
#pragma unroll
    for (int u = 0; u < 2; ++u)
        small[u] = fx_below((u32)(X[4 + u] >> 32), (u32)(X[4 + u] >> 32), tc) &&
                   fx_below((u32)(X[3 + u] >> 32), (u32)(X[5 + u] >> 32), tx);
    // the in-plane pairs of every distance, moved to the common scale together
#pragma unroll
    for (int u = 0; u < 2; ++u)
        small[u] = small[u] && fx_below((u32)(z(1, u) >> 32), (u32)(z(-1, u) >> 32), c.small_a[ISO ? 0 : 2]);
    u64 sxy[2][R], sy[2][R];
#pragma unroll
    for (int a = 1; a <= R; ++a) {
        const ulonglong2 yp = *reinterpret_cast<const ulonglong2 *>(cp + a * TXP);
        const ulonglong2 ym = *reinterpret_cast<const ulonglong2 *>(cp - a * TXP);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const u64 y1 = u ? yp.y : yp.x, y2 = u ? ym.y : ym.x;
            if (a == 1) small[u] = small[u] && fx_below((u32)(y1 >> 32), (u32)(y2 >> 32), ty);
            sxy[u][a - 1] = X[4 + u + a] + X[4 + u - a];
            sy[u][a - 1] = y1 + y2;
            if (ISO) sxy[u][a - 1] += sy[u][a - 1];
        }
    }
    if (!SAME) {
#pragma unroll
        for (int a = 0; a < R; ++a)
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                sxy[u][a] = fx_shift(sxy[u][a], (ISO ? 4 : 2) * FX_BIAS, dc);
                if (!ISO) sy[u][a] = fx_shift(sy[u][a], 2 * FX_BIAS, dc);
            }
    }
#pragma unroll
    for (int a = 1; a <= R; ++a) {
        const bool neg = a % 2 == 0;  // the weights at even distances are negative
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            if constexpr (ISO) {
                u64 s = sxy[u][a - 1] + z(a, u) + z(-a, u);
                if (neg) s = 12 * FX_BIAS - s;
                acc[u].mac(w.wh[a - 1], w.wl[a - 1], s);
            } else {
                u64 sx = sxy[u][a - 1], s2 = sy[u][a - 1], sz = z(a, u) + z(-a, u);
                if (neg) {
                    sx = 4 * FX_BIAS - sx;
                    s2 = 4 * FX_BIAS - s2;
                    sz = 4 * FX_BIAS - sz;
                }
                acc[u].mac(w.wh[a - 1], w.wl[a - 1], sx);
                acc[u].mac(w.wh[R + a - 1], w.wl[R + a - 1], s2);
                acc[u].mac(w.wh[2 * R + a - 1], w.wl[2 * R + a - 1], sz);
            }
        }
    }
    int left = 0;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const long long v = acc[u].result(w.corr);
        const double sum = fx_big(v) ? fx_to_double(v, sc + w.ew) : fx_small_to_double(v, sc + w.ew);
        res[u] = fma(c.g0, u ? f.y : f.x, sum);
        if (small[u] && (u64)(v + (1ll << LOW)) < (2ull << LOW)) left |= 1 << u;
    }
    return left;
}

template <int R, bool ISO, bool LONG>
__global__ void __launch_bounds__(FxCfg<R>::NT, 1)
heat_fx_kernel(const __grid_constant__ CUtensorMap map, const double *__restrict__ in, double *__restrict__ out,
               const __grid_constant__ Geom g, const __grid_constant__ FxCoef<R, ISO> c, int zc, int images,
               unsigned *err) {
    using Cfg = FxCfg<R>;
    constexpr int NT = Cfg::NT, NSLOT = Cfg::NSLOT, TXP = Cfg::TXP, KP = Cfg::KP;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    // TMA destinations 128-byte aligned (128 spare bytes); an offset, so that loads stay shared loads
    u64 *ring = reinterpret_cast<u64 *>(smem_raw + ((128u - (smem_addr(smem_raw) & 127u)) & 127u));
    __shared__ __align__(8) uint64_t full[NSLOT];
    __shared__ int scale[NSLOT];     // exponent code of each slot's plane
    __shared__ int low[NSLOT];       // how many threads of the last warp hold values far below it
    // of an output plane, by parity: {scale (or FP64, all outputs), planes differ, centre's shift}
    constexpr int FP64 = 4096;
    __shared__ int4 window[2];
    __shared__ double weights[1 + 3 * R];
    __shared__ u32 list[Cfg::LIST];
    __shared__ u32 listed;
    const int tid = threadIdx.x, lane = tid & 31, wy = tid >> 5;
    const int x0 = blockIdx.x * Cfg::TX, y0 = blockIdx.y * Cfg::TY, zc0 = blockIdx.z * zc;
    const int nx = (int)g.n[0], ny = (int)g.n[1], nz = (int)g.n[2];
    const int count = min(nz, zc0 + zc) - zc0;
    const int nplanes = count + 2 * R;
    const int x = x0 + 2 * lane, y = y0 + wy;

    if (tid == 0) {
        tma_prefetch_desc(&map);
        for (int s = 0; s < NSLOT; ++s) {
            mbar_init(&full[s], 1);
            scale[s] = 0;
        }
        mbar_fence_init();
        listed = 0;
    }
    if (tid < 1 + 3 * R) weights[tid] = tid == 0 ? c.g0 : c.ga[(tid - 1) / R][(tid - 1) % R];
    __syncthreads();
    pdl_launch_dependents();
    pdl_wait();

    const int bx = (int)g.off[0] + x0 - Cfg::HX, by0 = (int)g.off[1] + y0 - R, bz0 = (int)g.off[2] + zc0 - R;
    int issued = 0;
    auto issue = [&](int j) {
        const int s = j & (NSLOT - 1);
        mbar_arrive_expect_tx(&full[s], Cfg::BOX_BYTES);
        tma_load_3d(ring + s * Cfg::SLOT, &map, &full[s], bx, by0, bz0 + j);
    };
    if (tid == 0)
        for (; issued < NSLOT && issued < nplanes; ++issued) issue(issued);

    // Cells that enter a plane's scale: those some stencil of the field reads, i.e. the interior
    // and its halo of width R, but not where two axes leave the interior (a star stencil reads no
    // corner, and a caller may leave it unset).  On periodic grids the z-halo planes are images of
    // interior planes and count like them.  Tiles inside the interior skip the test.
    const bool edge = x0 - Cfg::HX < 0 || x0 + Cfg::TX + Cfg::HX > nx || y0 - R < 0 || y0 + Cfg::TY + R > ny || !images;
    u32 keep = ~0u, keep_zhalo = ~0u;  // bits 2 k, 2 k + 1: this thread's k-th pair, in a plane of the interior / beyond
    if (edge) {
        keep = keep_zhalo = 0u;
#pragma unroll
        for (int k = 0; k < KP; ++k)
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int i = tid + k * NT, row = i / (TXP / 2), gx = x0 - Cfg::HX + 2 * (i - row * (TXP / 2)) + u;
                const int gy = y0 - R + row, outside = (gx < 0 || gx >= nx) + (gy < 0 || gy >= ny);
                const bool near = gx >= -R && gx < nx + R && gy < ny + R;
                if (near && outside <= 1) keep |= 1u << (2 * k + u);
                if (near && outside + !images <= 1) keep_zhalo |= 1u << (2 * k + u);
            }
    }
    bool ok = true;
    double2 raw[KP];  // this thread's share of the plane loaded last
    u32 raw_hm = 0u;  // its largest high word
    auto load = [&](int j) {
        const int s = j & (NSLOT - 1);
        ok = ok && mbar_wait_bounded(&full[s], ((unsigned)j / NSLOT) & 1u);
        const double2 *src = reinterpret_cast<const double2 *>(ring + s * Cfg::SLOT);
        u32 hm = 0u;
#pragma unroll
        for (int k = 0; k < KP; ++k) {
            const int i = tid + k * NT;
            raw[k] = make_double2(0.0, 0.0);
            if (i < Cfg::PAIRS) {
                raw[k] = src[i];
                if (edge) {
                    const u32 kp = zc0 - R + j < 0 || zc0 - R + j >= nz ? keep_zhalo : keep;
                    if (!(kp & (1u << (2 * k)))) raw[k].x = 0.0;
                    if (!(kp & (2u << (2 * k)))) raw[k].y = 0.0;
                }
            }
            hm = max(hm, max((u32)__double2hiint(raw[k].x) & 0x7fffffffu, (u32)__double2hiint(raw[k].y) & 0x7fffffffu));
        }
        raw_hm = hm;
        hm = __reduce_max_sync(0xffffffffu, hm);
        int code = (int)(hm >> 20);
        if (hm == 0u) {  // only zeros and the smallest denormals: tell them apart
            u32 any = 0u;
#pragma unroll
            for (int k = 0; k < KP; ++k) any |= (u32)__double2loint(raw[k].x) | (u32)__double2loint(raw[k].y);
            code = __reduce_or_sync(0xffffffffu, any) != 0u;
        } else if (code == 0) {
            code = 1;
        }
        if (lane == 0) atomicMax(&scale[s], code);
    };
    auto convert = [&](int j) {
        const int s = j & (NSLOT - 1);
        // below FX_EMIN nothing shows at a scale the sums use, above FX_EMAX the outputs go to FP64
        const int e = max(scale[s], FX_EMIN);
        ulonglong2 *dst = reinterpret_cast<ulonglong2 *>(ring + s * Cfg::SLOT);
#pragma unroll
        for (int k = 0; k < KP; ++k) {
            const int i = tid + k * NT;
            if (i < Cfg::PAIRS)
                dst[i] = make_ulonglong2(fx_from_double(raw[k].x, e), fx_from_double(raw[k].y, e));
        }
    };

    // Store targets.  Even extents store the images of whole pairs (a neighbour that has none lands
    // in the row padding), odd ones cell by cell.
    const int nv = y < ny ? min(max(nx - x, 0), 2) : 0;
    const int64_t pitch_y = g.pad[0], pitch_z = g.pad[0] * g.pad[1];
    double *optr = out + g.idx(x, y, zc0);
    int mlo = 0, mhi = 0, ys = 0;
    if (images) {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            if (x + u < R) mlo |= 1 << u;
            else if (x + u >= nx - R && x + u < nx) mhi |= 1 << u;
        }
        if (nx % 2 == 0) {
            if (mlo) mlo = 3;
            if (mhi) mhi = 3;
        }
        ys = y < R ? ny : (y >= ny - R ? -ny : 0);
    }
    auto put1 = [](double *p, const double (&v)[2], int mask) {
        if (mask == 3) {
            *reinterpret_cast<double2 *>(p) = make_double2(v[0], v[1]);
        } else {
            if (mask & 1) p[0] = v[0];
            if (mask & 2) p[1] = v[1];
        }
    };
    auto put_image = [](double *p, const double (&v)[2], int mask, bool even) {
        if (even) {
            *reinterpret_cast<double2 *>(p) = make_double2(v[0], v[1]);
        } else {
            if (mask & 1) p[0] = v[0];
            if (mask & 2) p[1] = v[1];
        }
    };
    auto put = [&](double *p, const double (&v)[2]) {
        put1(p, v, nv == 2 ? 3 : 1);
        if (mlo | mhi) {
            if (mlo) put_image(p + nx, v, mlo, nx % 2 == 0);
            if (mhi) put_image(p - nx, v, mhi, nx % 2 == 0);
        }
    };

    const bool plain = nv == 2 && (mlo | mhi) == 0;  // both cells, no x image
    const int own = (wy + R) * TXP + Cfg::HX + 2 * lane;
    const bool early = LONG && ((wy >> 2) & 1);  // computes before it converts
    // the listed outputs, by all threads
    auto work_off = [&]() {
        for (u32 i = tid; i < min(listed, (u32)Cfg::LIST); i += NT) {
            const int cx = x0 + (int)(list[i] & 63u), cy = y0 + (int)((list[i] >> 6) & 15u), cz = zc0 + (int)(list[i] >> 10);
            store_with_images(out, g, R, images != 0, cx, cy, cz, heat_fp64_cell<R, ISO>(in, g, c, cx, cy, cz));
        }
    };
    load(0);
    bool bad = __syncthreads_or(!ok);
    for (int t = 0; !bad && t <= nplanes; ++t) {
        const int m = t - 1 - 2 * R;  // outputs of plane zc0 + m, from planes m .. t - 1
        double2 centre = make_double2(0.0, 0.0);  // exact, for the use below
        if (m >= 0 && nv != 0) centre = *reinterpret_cast<const double2 *>(in + (optr - out));
        auto compute = [&]() {
            if (m < 0 || nv == 0) return;
            const int4 win = window[(t - 1) & 1];
            const int sc = win.x, dc = win.z, z = zc0 + m;
            const u64 *cp = ring + ((m + R) & (NSLOT - 1)) * Cfg::SLOT + own;
            double res[2];
            int left = 0;  // outputs left to FP64
            if (sc != 0 && sc != FP64) {
                u64 Q[2 * R + 1][2];  // the z column at scale sc (its centre is read with the row)
#pragma unroll
                for (int k = 0; k <= 2 * R; ++k) {
                    if (k == R) continue;
                    const ulonglong2 q =
                        *reinterpret_cast<const ulonglong2 *>(ring + ((m + k) & (NSLOT - 1)) * Cfg::SLOT + own);
                    Q[k][0] = q.x;
                    Q[k][1] = q.y;
                }
                auto column = [&](int k, int u) { return Q[R + k][u]; };
                if (!win.y) {
                    left = fx_pair<R, ISO, true, TXP>(cp, column, 0, sc, c, centre, res);
                } else {
#pragma unroll
                    for (int k = 0; k <= 2 * R; ++k) {
                        if (k == R) continue;
                        const int d = sc - scale[(m + k) & (NSLOT - 1)];
                        Q[k][0] = fx_shift(Q[k][0], FX_BIAS, d);
                        Q[k][1] = fx_shift(Q[k][1], FX_BIAS, d);
                    }
                    left = fx_pair<R, ISO, false, TXP>(cp, column, dc, sc, c, centre, res);
                }
            } else if (sc == 0) {
                res[0] = res[1] = 0.0;
            } else {
                const double2 v = heat_fp64_pair<R>(in + (optr - out), pitch_y, pitch_z, weights);
                res[0] = v.x;
                res[1] = v.y;
            }
            left &= (1 << nv) - 1;
            if (left) {
                bool over = false;
#pragma unroll
                for (int u = 0; u < 2; ++u)
                    if (left & (1 << u)) {
                        const u32 at = atomicAdd(&listed, 1u);
                        if (at < (u32)Cfg::LIST) list[at] = (u32)(2 * lane + u) | (u32)wy << 6 | (u32)m << 10;
                        else over = true;
                    }
                if (over) {
                    const double2 v = heat_fp64_pair<R>(in + (optr - out), pitch_y, pitch_z, weights);
                    if (left & 1) res[0] = v.x;
                    if (left & 2) res[1] = v.y;
                }
            }
            const int zs = images ? (z < R ? nz : (z >= nz - R ? -nz : 0)) : 0;
            if (plain) *reinterpret_cast<double2 *>(optr) = make_double2(res[0], res[1]);
            else put(optr, res);
            if (ys | zs) {
                const int64_t dy = (int64_t)ys * pitch_y, dz = (int64_t)zs * pitch_z;
                if (ys) put(optr + dy, res);
                if (zs) put(optr + dz, res);
                if (ys && zs) put(optr + dy + dz, res);
            }
            optr += pitch_z;
        };
        if constexpr (LONG) {
            if (early) compute();
        }
        // the plane's scale is complete since the barrier; its slot is read from the next one on
        if (t < nplanes) {
            convert(t);
            if (wy == Cfg::BY - 1) {
                const u32 far = __ballot_sync(0xffffffffu, keep != 0u && (int)(raw_hm >> 20) + 8 < scale[t & (NSLOT - 1)]);
                if (lane == 31) {
                    low[t & (NSLOT - 1)] = __popc(far);
                    if (t >= 2 * R) {  // the window of the next interval's outputs: planes t - 2R .. t
                        int top = 0, least = 4096;
                        for (int k = t - 2 * R; k <= t; ++k) {
                            const int e = scale[k & (NSLOT - 1)];
                            top = max(top, e);
                            least = min(least, e);
                        }
                        const int centre = (t - R) & (NSLOT - 1);
                        const bool fp64 = top != 0 && (low[centre] > 16 || top < FX_SMIN || top > FX_EMAX);
                        window[t & 1] = make_int4(fp64 ? FP64 : top, least < top, top - scale[centre], 0);
                    }
                }
            }
            if (t + 1 < nplanes) load(t + 1);
        }
        if (!early) compute();
        bad = __syncthreads_or(!ok);
        if (LONG && t % 4 == 3 && !bad) {
            const bool full = listed > (u32)Cfg::LIST_HIGH;
            __syncthreads();  // no thread lists again before all have looked
            if (full) {
                work_off();
                __syncthreads();
                if (tid == 0) listed = 0;
                __syncthreads();
            }
        }
        if (!bad && tid == 0 && issued < nplanes && issued <= m + NSLOT) {  // planes up to m are retired
            fence_proxy_async();  // the block's generic writes to a slot before its next TMA load
            for (; issued < nplanes && issued <= m + NSLOT; ++issued) {
                scale[issued & (NSLOT - 1)] = 0;
                issue(issued);
            }
        }
    }
    if (bad) {
        if (tid == 0) {
            atomicOr(err, ERR_TIMEOUT);
            // drain loads still in flight before the CTA's shared memory is released
            for (int j = max(0, issued - NSLOT); j < issued; ++j)
                (void)mbar_wait_bounded(&full[j & (NSLOT - 1)], ((unsigned)j / NSLOT) & 1u, 100000000ull);
        }
        return;
    }
    work_off();  // the loop ended with a barrier
}

// Chunks of this many planes and more run the LONG body: half of the warps compute first, and the list is
// worked off before the end.  Its two copies of the computation cost a short kernel their fetching: 32^3
// (chunks of one plane) 10.2 us a step, without 9.8; 128^3 (15 planes) 39.5 and 39.4; 200 x 150 x 171 (40)
// 113.6 and 118.9, a Gaussian of 16 cells in 256^3 (37) 672 and 756.
constexpr int FX_LONG = 12;
template <int R, bool ISO>
cudaError_t run(const CUtensorMap *map, const double *in, double *out, const Geom &g, const FxCoef<R, ISO> &c,
                bool images, unsigned *err, cudaStream_t s, double reread, int zmode) {
    using Cfg = FxCfg<R>;
    static int ready[64] = {};  // per device: the shared-memory limit is raised
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!ready[dev]) {
        e = cudaFuncSetAttribute(heat_fx_kernel<R, ISO, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg::SMEM);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(heat_fx_kernel<R, ISO, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg::SMEM);
        if (e != cudaSuccess) return e;
        ready[dev] = 1;
    }
    const int tx = (int)((g.n[0] + Cfg::TX - 1) / Cfg::TX), ty = (int)((g.n[1] + Cfg::TY - 1) / Cfg::TY);
    const int nz = (int)g.n[2];
    const int chunks = choose_zchunks(tx * ty, nz, device_sms(), reread);  // one CTA per SM
    const int zc = zchunk_len((nz + chunks - 1) / chunks, nz, zmode);
    dim3 grid(tx, ty, (unsigned)((nz + zc - 1) / zc));
    const auto k = zc >= FX_LONG ? heat_fx_kernel<R, ISO, true> : heat_fx_kernel<R, ISO, false>;
    return launch_pdl(k, grid, dim3(Cfg::NT), Cfg::SMEM, s, *map, in, out, g, c, zc, images ? 1 : 0, err);
}

// The variants differ in how z is split into chunks: the weight that choose_zchunks gives the
// 2R planes each chunk converts again against SMs left idle in the last wave.
constexpr double FX_REREAD[] = {0.7, 0.35, 1.0, 0.0};

template <int R, bool ISO>
cudaError_t dispatch(int variant, const CUtensorMap *map, const double *in, double *out, const Geom &g,
                     const DiffCoef &dc, bool images, unsigned *err, cudaStream_t s, int zmode) {
    FxCoef<R, ISO> c;
    double w[FxCoef<R, ISO>::N];
    int mult[FxCoef<R, ISO>::N];
    for (int i = 0; i < FxCoef<R, ISO>::N; ++i) {
        w[i] = dc.ga[i / R][i % R];
        mult[i] = ISO ? 6 : 2;
    }
    if (!fx_weights<FxCoef<R, ISO>::N>(w, mult, c.w)) return cudaErrorInvalidValue;
    c.g0 = dc.g0;
    for (int a = 0; a < 3; ++a)
        for (int b = 0; b < R; ++b) c.ga[a][b] = dc.ga[a][b];
    auto threshold = [&](double weight) {  // of a value whose term is below 2^-6, -7, -8 of 2^ew S
        const double t = (FX_FLAG_HI >> std::min(R - 1, 2)) * std::ldexp(1.0, c.w.ew) / weight;
        return t < FX_BIAS_HI ? std::max((u32)t + 1, 4u) : FX_BIAS_HI;  // weight 0: every value is small
    };
    c.small_c = threshold(dc.g0);
    for (int a = 0; a < 3; ++a) c.small_a[a] = threshold(dc.ga[a][0]);
    if (variant < 0 || variant >= 4) return cudaErrorInvalidValue;
    return run<R, ISO>(map, in, out, g, c, images, err, s, FX_REREAD[variant], zmode);
}

template <int R>
cudaError_t dispatch_iso(int variant, const CUtensorMap *map, const double *in, double *out, const Geom &g,
                         const DiffCoef &dc, bool images, unsigned *err, cudaStream_t s, int zmode) {
    bool iso = true;
    for (int b = 0; b < R; ++b) iso = iso && dc.ga[0][b] == dc.ga[1][b] && dc.ga[0][b] == dc.ga[2][b];
    return iso ? dispatch<R, true>(variant, map, in, out, g, dc, images, err, s, zmode)
               : dispatch<R, false>(variant, map, in, out, g, dc, images, err, s, zmode);
}

}  // namespace

// Whether the folded weights of a plan can be held in fixed point (else diffusion.cu runs): in
// range, and with the signs of a forward step that is stable or nearly so (g0 >= 0, positive at
// odd distances, negative at even ones), which the kernel has compiled in.
bool diffusion_fx_fits(const DiffCoef &dc) {
    double w[12];
    const int mult[12] = {};
    bool signs = std::isfinite(dc.g0) && dc.g0 >= 0.0;
    for (int i = 0; i < 12; ++i) {
        const int a = i % 4 + 1;  // distance; weights beyond the radius are 0
        w[i] = dc.ga[i / 4][a - 1];
        signs = signs && (a % 2 == 1 ? w[i] >= 0.0 : w[i] <= 0.0);
    }
    FxWeights<12> o;
    // 2^ew of the launch may be a quarter of this one (ISO)
    return signs && fx_weights<12>(w, mult, o) && o.ew >= 2 - FX_EW;
}

void diffusion_fx_box(int r, int box[3]) {
    box[0] = FxCfg<3>::TXP;
    box[1] = FxCfg<3>::TY + 2 * r;
    box[2] = 1;
}

cudaError_t launch_diffusion_fx(const CUtensorMap *map, const double *in, double *out, const Geom &g,
                                const DiffCoef &dc, bool images, unsigned *err, cudaStream_t s, int variant, int zmode) {
    switch (dc.r) {
    case 1: return dispatch_iso<1>(variant, map, in, out, g, dc, images, err, s, zmode);
    case 2: return dispatch_iso<2>(variant, map, in, out, g, dc, images, err, s, zmode);
    case 3: return dispatch_iso<3>(variant, map, in, out, g, dc, images, err, s, zmode);
    case 4: return dispatch_iso<4>(variant, map, in, out, g, dc, images, err, s, zmode);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace stn

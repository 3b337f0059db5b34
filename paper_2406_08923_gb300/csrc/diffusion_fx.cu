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
//   * ZB new planes per iteration: every thread takes its share of their tiles into registers,
//     the block reduces the largest exponent of each, and the values go back in place as biased
//     60-bit integers at that plane's scale.
//   * A thread owns 2 x-cells and loads their z column (ZB + 2R planes) once per iteration.  An
//     output uses the largest scale of the 2R+1 planes its z column spans (S), and values of
//     planes with a smaller one are shifted right, behind branches that are uniform per block.
//     S depends on nothing but those plane tiles, so results do not depend on how z is split
//     into iterations, chunks or slabs.
//   * With one grid spacing on all axes (ISO) the six values at distance a are summed first: four
//     64 x 64-bit products per cell instead of ten.
//   * Outputs whose stencil is small against S (fixed.cuh), or that meet infinities or NaN, are
//     listed and evaluated at the end of the CTA by FP64 multiply-adds from global memory, in
//     the order of diffusion.cu.
#include <algorithm>

#include "fixed.cuh"
#include "internal.h"

namespace stn {
namespace {

template <int R, bool ISO> struct FxCoef {
    static constexpr int N = ISO ? 1 + R : 1 + 3 * R;
    FxWeights<N> w;
    double g0, ga[3][R];  // for the outputs evaluated in FP64
};

template <int ZB_, int NSLOT_, int R> struct FxCfg {
    static constexpr int BY = 16, NT = 32 * BY, ZB = ZB_, NSLOT = NSLOT_;
    static constexpr int TX = 64, TY = BY, HX = 4, TXP = TX + 2 * HX, ROWS = TY + 2 * R;
    static constexpr int PAIRS = TXP / 2 * ROWS;  // 16-byte pairs per plane tile
    static constexpr int KP = (PAIRS + NT - 1) / NT;
    static constexpr int SLOT = ((TXP * ROWS * 8 + 127) / 128) * 128 / 8;
    static constexpr uint32_t BOX_BYTES = TXP * ROWS * 8;
    static constexpr size_t SMEM = (size_t)NSLOT * SLOT * 8 + 128;
    static constexpr int S = ZB + 2 * R;  // planes of an iteration's z column
    static constexpr int LIST = 1024;
    static_assert((NSLOT & (NSLOT - 1)) == 0, "ring depth is a power of two (slot = j & (NSLOT-1))");
    static_assert(NSLOT >= 2 * ZB + 2 * R, "ring: an iteration's planes and the next ZB");
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

// Two neighbouring outputs: `cp` points at the first in its centre plane (scale sc - dc), z(k, u)
// gives the value of cell u at plane offset k, at scale sc.  Returns bit u set where output u is
// left to FP64: the centre and its four neighbours in the plane are below 2^-6 of the scale.
template <int R, bool ISO, int TXP, typename W, typename Z>
__device__ __forceinline__ int fx_pair(const u64 *cp, const Z &z, int dc, int sc, const W &w, double (&res)[2]) {
    u64 X[10];  // x window: cells -4 .. 5
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        if (2 * k + 1 < 4 - R || 2 * k > 5 + R) continue;
        const ulonglong2 t = *reinterpret_cast<const ulonglong2 *>(cp - 4 + 2 * k);
        X[2 * k] = t.x;
        X[2 * k + 1] = t.y;
    }
    FxAcc acc[2];
    u32 hmx[2], hmn[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const u32 a = (u32)(X[3 + u] >> 32), d = (u32)(X[5 + u] >> 32), e = (u32)(X[4 + u] >> 32);
        hmx[u] = max(max(a, d), e);
        hmn[u] = min(min(a, d), e);
        acc[u].mac(w.wh[0], w.wl[0], z(0, u));
    }
    // the in-plane pairs of every distance, moved to the common scale together
    u64 sxy[2][R], sy[2][R];
#pragma unroll
    for (int a = 1; a <= R; ++a) {
        const ulonglong2 yp = *reinterpret_cast<const ulonglong2 *>(cp + a * TXP);
        const ulonglong2 ym = *reinterpret_cast<const ulonglong2 *>(cp - a * TXP);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const u64 y1 = u ? yp.y : yp.x, y2 = u ? ym.y : ym.x;
            if (a == 1) {
                hmx[u] = max(hmx[u], max((u32)(y1 >> 32), (u32)(y2 >> 32)));
                hmn[u] = min(hmn[u], min((u32)(y1 >> 32), (u32)(y2 >> 32)));
            }
            sxy[u][a - 1] = X[4 + u + a] + X[4 + u - a];
            sy[u][a - 1] = y1 + y2;
            if (ISO) sxy[u][a - 1] += sy[u][a - 1];
        }
    }
    if (dc) {
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
                acc[u].mac(w.wh[a], w.wl[a], s);
            } else {
                u64 sx = sxy[u][a - 1], s2 = sy[u][a - 1], sz = z(a, u) + z(-a, u);
                if (neg) {
                    sx = 4 * FX_BIAS - sx;
                    s2 = 4 * FX_BIAS - s2;
                    sz = 4 * FX_BIAS - sz;
                }
                acc[u].mac(w.wh[a], w.wl[a], sx);
                acc[u].mac(w.wh[R + a], w.wl[R + a], s2);
                acc[u].mac(w.wh[2 * R + a], w.wl[2 * R + a], sz);
            }
        }
    }
    const u32 flag = dc < 6 ? FX_FLAG_HI << dc : FX_BIAS_HI;
    int left = 0;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const long long v = acc[u].result(w.corr);
        res[u] = fx_to_double(v, sc + w.ew);
        if ((hmx[u] < FX_BIAS_HI + flag && hmn[u] >= FX_BIAS_HI - flag) || !fx_big(v)) left |= 1 << u;
    }
    return left;
}

// The same where the output's scale is finer than the one the iteration's z column is held at:
// plane j (its centre) and the others are read again.  Out of line: a tenth of the outputs or fewer.
template <int R, bool ISO, int TXP, int SLOT, int NSLOT, typename W>
__device__ __noinline__ int fx_pair_reread(const u64 *ring, const int *scale, int j, int own, int sc, const W &w,
                                           double *out) {
    double res[2];
    const int left = fx_pair<R, ISO, TXP>(
        ring + (j & (NSLOT - 1)) * SLOT + own,
        [&](int k, int u) {
            const int s = (j + k) & (NSLOT - 1);
            return fx_shift(ring[s * SLOT + own + u], FX_BIAS, sc - scale[s]);
        },
        sc - scale[j & (NSLOT - 1)], sc, w, res);
    out[0] = res[0];
    out[1] = res[1];
    return left;
}

template <int ZB, int NSLOT, int R, bool ISO>
__global__ void __launch_bounds__(FxCfg<ZB, NSLOT, R>::NT, 1)
heat_fx_kernel(const __grid_constant__ CUtensorMap map, const double *__restrict__ in, double *__restrict__ out,
               const __grid_constant__ Geom g, const __grid_constant__ FxCoef<R, ISO> c, int zc, int images,
               unsigned *err) {
    using Cfg = FxCfg<ZB, NSLOT, R>;
    constexpr int NT = Cfg::NT, TXP = Cfg::TXP, S = Cfg::S, KP = Cfg::KP;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    // TMA destinations 128-byte aligned (128 spare bytes); an offset, so that loads stay shared loads
    u64 *ring = reinterpret_cast<u64 *>(smem_raw + ((128u - (smem_addr(smem_raw) & 127u)) & 127u));
    __shared__ __align__(8) uint64_t full[NSLOT];
    __shared__ int scale[NSLOT];  // exponent code of each slot's plane
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
    auto counts = [&](int col, int row, int j) -> bool {
        const int gx = x0 - Cfg::HX + col, gy = y0 - R + row, gz = zc0 - R + j;
        const bool ox = gx < 0 || gx >= nx, oy = gy < 0 || gy >= ny, oz = !images && (gz < 0 || gz >= nz);
        return gx >= -R && gx < nx + R && gy < ny + R && (int)ox + (int)oy + (int)oz <= 1;
    };
    bool ok = true;
    // Converts planes j .. j + ZB - 1 below `end` in place.  Two block barriers: the first also
    // retires what every thread read before the call, so the ring is refilled there, up to plane
    // `refill`.
    auto convert = [&](int j, int end, int refill) -> bool {
        double2 v[ZB][KP];
#pragma unroll
        for (int b = 0; b < ZB; ++b) {
            if (j + b < end) {
                const int s = (j + b) & (NSLOT - 1);
                ok = ok && mbar_wait_bounded(&full[s], ((unsigned)(j + b) / NSLOT) & 1u);
                const double2 *src = reinterpret_cast<const double2 *>(ring + s * Cfg::SLOT);
                u32 hm = 0u;
#pragma unroll
                for (int k = 0; k < KP; ++k) {
                    const int i = tid + k * NT;
                    v[b][k] = make_double2(0.0, 0.0);
                    if (i < Cfg::PAIRS) {
                        v[b][k] = src[i];
                        if (edge) {
                            const int row = i / (TXP / 2), col = 2 * (i - row * (TXP / 2));
                            if (!counts(col, row, j + b)) v[b][k].x = 0.0;
                            if (!counts(col + 1, row, j + b)) v[b][k].y = 0.0;
                        }
                    }
                    hm = max(hm, max((u32)__double2hiint(v[b][k].x) & 0x7fffffffu,
                                     (u32)__double2hiint(v[b][k].y) & 0x7fffffffu));
                }
                hm = __reduce_max_sync(0xffffffffu, hm);
                int code = (int)(hm >> 20);
                if (hm == 0u) {  // only zeros and the smallest denormals: tell them apart
                    u32 any = 0u;
#pragma unroll
                    for (int k = 0; k < KP; ++k) any |= (u32)__double2loint(v[b][k].x) | (u32)__double2loint(v[b][k].y);
                    code = __reduce_or_sync(0xffffffffu, any) != 0u;
                } else if (code == 0) {
                    code = 1;
                }
                if (lane == 0) atomicMax(&scale[s], code);
            }
        }
        const bool bad = __syncthreads_or(!ok);
        if (!bad && tid == 0) {
            fence_proxy_async();  // the block's generic writes to a slot before its next TMA load
            for (; issued < min(nplanes, refill); ++issued) {
                scale[issued & (NSLOT - 1)] = 0;
                issue(issued);
            }
        }
#pragma unroll
        for (int b = 0; b < ZB; ++b) {
            if (j + b < end) {
                const int s = (j + b) & (NSLOT - 1);
                const int e = scale[s];
                ulonglong2 *dst = reinterpret_cast<ulonglong2 *>(ring + s * Cfg::SLOT);
                // outside this range nothing shows at a scale the sums use, or the outputs go to FP64
                const bool in_range = e >= FX_EMIN && e <= FX_EMAX;
#pragma unroll
                for (int k = 0; k < KP; ++k) {
                    const int i = tid + k * NT;
                    if (i < Cfg::PAIRS)
                        dst[i] = in_range ? make_ulonglong2(fx_from_double(v[b][k].x, e), fx_from_double(v[b][k].y, e))
                                          : make_ulonglong2(FX_BIAS, FX_BIAS);
                }
            }
        }
        __syncthreads();
        return bad;
    };

    bool bad = false;
    for (int j = 0; j < 2 * R; j += ZB) bad = convert(j, 2 * R, 0) || bad;

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

    const int own = (wy + R) * TXP + Cfg::HX + 2 * lane;
    for (int m = 0; m < count; m += ZB) {
        bad = convert(m + 2 * R, nplanes, m + NSLOT) || bad;  // planes below m are retired
        if (bad) break;
        if (nv == 0) continue;
        // the z column at one scale: the largest of the iteration's planes
        int E[S];
        u64 Q[S][2];
        int top = 0;
#pragma unroll
        for (int k = 0; k < S; ++k) {
            const int s = (m + k) & (NSLOT - 1);
            E[k] = m + k < nplanes ? scale[s] : 0;
            const ulonglong2 t = *reinterpret_cast<const ulonglong2 *>(ring + s * Cfg::SLOT + own);
            Q[k][0] = t.x;
            Q[k][1] = t.y;
            top = max(top, E[k]);
        }
        bool mixed = false;
#pragma unroll
        for (int k = 0; k < S; ++k) mixed = mixed || E[k] < top;
        if (mixed) {
#pragma unroll
            for (int k = 0; k < S; ++k) {
                const int d = top - E[k];
                Q[k][0] = fx_shift(Q[k][0], FX_BIAS, d);
                Q[k][1] = fx_shift(Q[k][1], FX_BIAS, d);
            }
        }
#pragma unroll
        for (int b = 0; b < ZB; ++b) {
            if (m + b >= count) break;
            int sc = E[b];
#pragma unroll
            for (int k = 1; k <= 2 * R; ++k) sc = max(sc, E[b + k]);
            const int z = zc0 + m + b;
            const u64 *cp = ring + ((m + b + R) & (NSLOT - 1)) * Cfg::SLOT + own;
            double res[2];
            int left = 0;  // outputs left to FP64
            if (sc == top && sc >= FX_SMIN && sc <= FX_EMAX) {
                left = fx_pair<R, ISO, TXP>(cp, [&](int k, int u) { return Q[b + R + k][u]; }, sc - E[b + R], sc, c.w, res);
            } else if (sc >= FX_SMIN && sc <= FX_EMAX) {  // a finer scale than the column's: read it again
                left = fx_pair_reread<R, ISO, TXP, Cfg::SLOT, NSLOT>(ring, scale, m + b + R, own, sc, c.w, res);
            } else {  // zeros only, or infinities, NaN, or near the ends of the exponent range
                res[0] = res[1] = 0.0;
                left = sc == 0 ? 0 : 3;
            }
            left &= (1 << nv) - 1;
            if (left) {
#pragma unroll
                for (int u = 0; u < 2; ++u)
                    if (left & (1 << u)) {
                        const u32 at = atomicAdd(&listed, 1u);
                        if (at < (u32)Cfg::LIST) list[at] = (u32)(2 * lane + u) | (u32)wy << 6 | (u32)(m + b) << 10;
                        else res[u] = heat_fp64_cell<R, ISO>(in, g, c, x + u, y, z);
                    }
            }
            const int zs = images ? (z < R ? nz : (z >= nz - R ? -nz : 0)) : 0;
            double *p = optr + b * pitch_z;
            put(p, res);
            if (ys | zs) {
                const int64_t dy = (int64_t)ys * pitch_y, dz = (int64_t)zs * pitch_z;
                if (ys) put(p + dy, res);
                if (zs) put(p + dz, res);
                if (ys && zs) put(p + dy + dz, res);
            }
        }
        optr += ZB * pitch_z;
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
    __syncthreads();  // the listed cells' first stores and the list itself
    const u32 n = min(listed, (u32)Cfg::LIST);
    for (u32 i = tid; i < n; i += NT) {
        const int cx = x0 + (int)(list[i] & 63u), cy = y0 + (int)((list[i] >> 6) & 15u), cz = zc0 + (int)(list[i] >> 10);
        store_with_images(out, g, R, images != 0, cx, cy, cz, heat_fp64_cell<R, ISO>(in, g, c, cx, cy, cz));
    }
}

template <int ZB, int NSLOT, int R, bool ISO>
cudaError_t run(const CUtensorMap *map, const double *in, double *out, const Geom &g, const FxCoef<R, ISO> &c,
                bool images, unsigned *err, cudaStream_t s, int zmode) {
    using Cfg = FxCfg<ZB, NSLOT, R>;
    auto k = heat_fx_kernel<ZB, NSLOT, R, ISO>;
    static int occ[64] = {};  // resident CTAs per SM, per device
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!occ[dev]) {
        e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg::SMEM);
        if (e != cudaSuccess) return e;
        int o = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, k, Cfg::NT, Cfg::SMEM);
        if (e != cudaSuccess) return e;
        occ[dev] = std::max(o, 1);
    }
    const int tx = (int)((g.n[0] + Cfg::TX - 1) / Cfg::TX), ty = (int)((g.n[1] + Cfg::TY - 1) / Cfg::TY);
    const int nz = (int)g.n[2];
    const int chunks = choose_zchunks(tx * ty, nz, occ[dev] * device_sms(), 0.7);
    const int zc = zchunk_len((nz + chunks - 1) / chunks, nz, zmode);
    dim3 grid(tx, ty, (unsigned)((nz + zc - 1) / zc));
    return launch_pdl(k, grid, dim3(Cfg::NT), Cfg::SMEM, s, *map, in, out, g, c, zc, images ? 1 : 0, err);
}

// Launch shapes over the one 64 x 16 tile: (ZB planes per iteration, NSLOT ring depth).
#define FX_VARIANTS(X) X(1, 16) X(2, 16) X(4, 16) X(3, 16)

template <int R, bool ISO>
cudaError_t dispatch(int variant, const CUtensorMap *map, const double *in, double *out, const Geom &g,
                     const DiffCoef &dc, bool images, unsigned *err, cudaStream_t s, int zmode) {
    FxCoef<R, ISO> c;
    double w[FxCoef<R, ISO>::N];
    int mult[FxCoef<R, ISO>::N];
    w[0] = dc.g0;
    mult[0] = 1;
    for (int i = 1; i < FxCoef<R, ISO>::N; ++i) {
        w[i] = dc.ga[(i - 1) / R][(i - 1) % R];
        mult[i] = ISO ? 6 : 2;
    }
    if (!fx_weights<FxCoef<R, ISO>::N>(w, mult, c.w)) return cudaErrorInvalidValue;
    c.g0 = dc.g0;
    for (int a = 0; a < 3; ++a)
        for (int b = 0; b < R; ++b) c.ga[a][b] = dc.ga[a][b];
    int i = 0;
#define X(ZB, NS) \
    if (i++ == variant) return run<ZB, NS, R, ISO>(map, in, out, g, c, images, err, s, zmode);
    FX_VARIANTS(X)
#undef X
    return cudaErrorInvalidValue;
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
    double w[13];
    int mult[13];
    bool signs = true;
    for (int i = 0; i < 13; ++i) {
        const int a = (i - 1) % 4 + 1;  // distance; weights beyond the radius are 0
        w[i] = i == 0 ? dc.g0 : dc.ga[(i - 1) / 4][a - 1];
        mult[i] = i == 0 ? 1 : 2;
        signs = signs && (i == 0 || a % 2 == 1 ? w[i] >= 0.0 : w[i] <= 0.0);
    }
    FxWeights<13> o;
    return signs && fx_weights<13>(w, mult, o);
}

void diffusion_fx_box(int r, int box[3]) {
    box[0] = FxCfg<4, 16, 3>::TXP;
    box[1] = FxCfg<4, 16, 3>::TY + 2 * r;
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

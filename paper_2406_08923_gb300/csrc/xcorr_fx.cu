// xcorr_fx.cu -- 1D cross-correlation (Sec. 3.1, Eq. 3) in integers: FP64 in fixed point for
// radius 1..1024, and int32 sweeps of radius 1..4 composed into one.
//
// Composition.  k sweeps of a radius-r correlation are one correlation of radius k r whose weights
// are the k-fold convolution of g with itself: 2 k r + 1 multiply-adds per output instead of
// k (2 r + 1), with no halo to shrink, no exchange and no barrier between sweeps.  Modulo 2^32 the
// two are equal bit for bit.  In FP64 the composed sum has fewer roundings than the sweeps; its
// weights are convolved in double-double arithmetic, so that the fixed-point weights are
// as exact as those of a single sweep.  2^20 cells, 10 sweeps, r = 3: int32 12.6 -> 6.6 us on the
// device, FP64 129 -> 33 us.
//
// FP64.  2r+1 FP64 multiply-adds per output ran at 99 % of the FP64 pipe (2 per clock and SM).
// Here a CTA converts its chunk of cells, halo included, to signed 59-bit integers of one binary
// scale, split into two 30-bit limbs, and the weights come as limbs too.  A product is then three
// 32 x 32 + 64-bit multiply-adds (the product of the two low limbs, below 2^-60 of the scale, is
// left out), at 32 per clock and SM: 5.3 times the FP64 rate.  3 M cells, r = 100: 1063 -> 234 us.
//
//   * As in xcorr_wide.cu each thread computes V consecutive outputs (V odd: conflict-free shared
//     loads) and keeps V weights and 2V-1 cells in registers per block of V weights.
//   * An output keeps two 64-bit sums: the high products HH and the cross products M, whose
//     upper part moves to HH every one to four blocks, before 20 terms could overflow it.
//   * Accuracy (fx_wide_weights): the result is off by at most 2 (2r+1) + 4 units of 2^-62 of
//     the largest result the scale admits, which is no more than a chain of FP64 multiply-adds may
//     be off, 2^-53 (2r+1) sum |w f|, wherever sum |w f| is at least 2^-7 of that result.  An output
//     of that size itself shows it; the others are listed, their sum |w f| is accumulated from
//     the high limbs until it passes the bound (a few terms for most), and what stays below is
//     evaluated by FP64 multiply-adds in the order j = -r .. r, unless its window is all zeros.
//   * A chunk with infinities, NaN or exponents near the ends of the range is swept in FP64, one
//     sweep after the other, in shared memory; so is one where 8 of 32 outputs spread over it would stay
//     below the bound (pulses and spikes far above their surroundings).  That is looked at only where a
//     quarter of the threads load mostly small cells.  A chunk of zeros stores zeros.
//     3 M cells, r = 100, in us on the FP64 pipe, here, and with each output by itself: noise 1063, 242,
//     246; pulses of 100 cells 1062, 1035, 1249; a spike every 997 cells 1062, 1066, 1273; zeros 1062, 11,
//     1057. 2^20 cells, 10 sweeps of r = 3: noise 127, 33.2, 33.3; pulses 127, 134, 152; spikes 127,
//     136, 160. Noise over 60 binary orders at r = 1000 is the slowest, 3364, 4063, 4806.
#include <algorithm>
#include <vector>

#include "fixed.cuh"
#include "internal.h"

namespace stn {
namespace {

constexpr int FT = 256;  // threads per CTA
// Weights from which on it pays to look for chunks that FP64 evaluates sooner: 11 weights, 2^20 cells,
// 13.1 us, with the look 14.9, and 31 to 33 at worst where the FP64 pipe takes 29.5.
constexpr int FAR_WEIGHTS = 32;
constexpr uint16_t EMPTY = 0x8000, DONE = 0xffff;  // marks of listed outputs

template <int V_> struct FxWide {
    static constexpr int V = V_, CH = FT * V;
    static constexpr int SPILL = 20 / V;  // blocks between two spills of M: at most 20 terms
    static __host__ __device__ int nwp(int r) { return (2 * r + 1 + V - 1) / V * V; }
    // cells: the chunk, its halo, and zeros for the padded weight blocks
    static __host__ __device__ int cells(int r) { return CH + nwp(r) + V; }
    static __host__ __device__ size_t smem(int r) { return sizeof(int2) * (size_t)(cells(r) + nwp(r)) + sizeof(uint16_t) * CH; }
    static_assert(V % 2 == 1 && SPILL >= 1, "");
    static_assert(CH < 32768, "list entries are 16-bit, one of them a mark");
};

// v as balanced limbs at scale E: v = (2^30 qh + ql) 2^(E - 1081), |2^30 qh + ql| <= 2^59, nearest.
__device__ __forceinline__ int2 fx_limbs(double v, int E) {
    const u32 hi = (u32)__double2hiint(v), lo = (u32)__double2loint(v);
    const int d = min(E - (int)((hi >> 20) & 0x7ffu), 63);
    const u64 m = (((u64)((hi & 0xfffffu) | 0x100000u) << 32) | lo) << 7 >> d;
    const long long a = (long long)((m + 1) >> 1);
    const long long q = (int)hi < 0 ? -a : a;
    const int qh = (int)((q + (1ll << 29)) >> 30);
    return make_int2((int)(u32)q - (int)((u32)qh << 30), qh);  // x: low limb, y: high limb
}

template <int V, int MINB>
__global__ void __launch_bounds__(FT, MINB)
xcorr_wide_fx_kernel(const double *__restrict__ in, double *__restrict__ out, Geom geo, const double *__restrict__ wg,
                     const int2 *__restrict__ wfx, int ew, int r, const double *__restrict__ w1, int r1, int sweeps,
                     int periodic, int images) {
    using B = FxWide<V>;
    constexpr int CH = B::CH;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ u32 red[FT / 32];
    __shared__ u32 listed, far;
    const int tid = threadIdx.x, nw = 2 * r + 1, nwp = B::nwp(r), cells = B::cells(r), len = CH + 2 * r;
    int2 *s = reinterpret_cast<int2 *>(smem_raw);
    double *sd = reinterpret_cast<double *>(smem_raw);  // the results
    int2 *ws = s + cells;
    uint16_t *list = reinterpret_cast<uint16_t *>(ws + nwp);
    const int64_t n = geo.n[0], c0 = (int64_t)blockIdx.x * CH;
    const double *inx = in + geo.off[0];
    double *outx = out + geo.off[0];
    // cell gi of the augmented array (beyond the caller's halo: 0)
    auto cell = [&](int64_t gi) -> double {
        if (gi >= 0 && gi < n) return inx[gi];
        if (periodic) {
            gi %= n;
            return inx[gi < 0 ? gi + n : gi];
        }
        return (gi >= -r && gi < n + r) ? inx[gi] : 0.0;
    };
    if (tid == 0) listed = far = 0u;
    pdl_wait();

    // The cells and their largest exponent; those past the last output's window count as 0.  A
    // thread's first KR cells stay in registers until the scale is known (radius 128 and less:
    // all of them), the rest are read again.
    constexpr int KR = V + 1;
    double kept[KR];
    u32 hm = 0u;
    const bool inside = c0 - r >= 0 && c0 + CH + r <= n;
    const int used = (int)min((int64_t)len, n - c0 + 2 * r);
    const double *src = inx + (c0 - r);
    auto load = [&](int e) -> double { return e < used ? (inside ? src[e] : cell(c0 - r + e)) : 0.0; };
#pragma unroll
    for (int k = 0; k < KR; ++k) kept[k] = load(tid + k * FT);
#pragma unroll
    for (int k = 0; k < KR; ++k) hm = max(hm, (u32)__double2hiint(kept[k]) & 0x7fffffffu);
    for (int e = tid + KR * FT; e < cells; e += FT) hm = max(hm, (u32)__double2hiint(load(e)) & 0x7fffffffu);
    for (int j = tid; j < nwp; j += FT) ws[j] = j < nw ? wfx[j] : make_int2(0, 0);
    hm = __reduce_max_sync(0xffffffffu, hm);
    if ((tid & 31) == 0) red[tid >> 5] = hm;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < FT / 32; ++w) hm = max(hm, red[w]);
    const int E = (int)(hm >> 20);
    bool fixed = E >= FX_SMIN && E <= FX_EMAX;  // uniform per block
    bool zeros = false;
    if (hm == 0u) {  // zeros only, or the smallest denormals too
        u32 any = 0u;
        for (int e = tid; e < used; e += FT) any |= (u32)__double2loint(load(e));
        zeros = !__syncthreads_or(any != 0u);
    }

    // FP64 multiply-adds of output p from global memory
    auto by_fp64 = [&](int p) -> double {
        double acc = 0.0;
        for (int j = 0; j < nw; ++j) acc = fma(wg[j], load(p + j), acc);
        return acc;
    };

    // whether any cell that is not 0 lies so far below the scale that its limbs are 0
    auto faint_cells = [&]() {
        bool any = false;
        for (int e = tid; e < used; e += FT) any = any || ((s[e].x | s[e].y) == 0 && load(e) != 0.0);
        return __syncthreads_or(any) != 0;
    };
    const int base = tid * V;
    double res[V];
    if (fixed) {
#pragma unroll
        for (int k = 0; k < KR; ++k)
            if (tid + k * FT < cells) s[tid + k * FT] = fx_limbs(kept[k], E);
        for (int e = tid + KR * FT; e < cells; e += FT) s[e] = fx_limbs(load(e), E);
        int small = 0;
        if (nw >= FAR_WEIGHTS) {
#pragma unroll
            for (int k = 0; k < KR; ++k)
                small += (int)(((u32)__double2hiint(kept[k]) & 0x7fffffffu) >> 20) + 7 < E && tid + k * FT < used;
        }
        if (__syncthreads_count(2 * small > KR) > FT / 4) {
            // 4 outputs per warp, spread over the chunk, whose sum |w f| is taken whole
            int below = 0;
            const bool faint = faint_cells();
            for (int i = 0; i < 4; ++i) {
                const int p = ((tid >> 5) * 4 + i) * (CH / 32);
                u64 mag = 0;
                int any = 0;
                for (int j = tid & 31; j < nw; j += 32) {
                    mag += (u64)(u32)abs(ws[j].y) * (u32)abs(s[p + j].y);
                    any |= s[p + j].x | s[p + j].y;
                }
                for (int d = 16; d; d >>= 1) mag += __shfl_xor_sync(0xffffffffu, mag, d);
                below += mag < (1ull << 53) && (faint || __any_sync(0xffffffffu, any)) && c0 + p < n;
            }
            if ((tid & 31) == 0 && below) atomicAdd(&far, (u32)below);
            __syncthreads();
            fixed = far < 8u;
        }
    }
    if (fixed) {
        long long hh[V], m[V];
#pragma unroll
        for (int v = 0; v < V; ++v) hh[v] = m[v] = 0;
        int since = 0;
        for (int j0 = 0; j0 < nwp; j0 += V) {
            int2 w[V], x[2 * V - 1];
#pragma unroll
            for (int u = 0; u < V; ++u) w[u] = ws[j0 + u];
#pragma unroll
            for (int q = 0; q < 2 * V - 1; ++q) x[q] = s[base + j0 + q];
#pragma unroll
            for (int u = 0; u < V; ++u)
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    hh[v] += (long long)w[u].y * x[v + u].y;
                    m[v] += (long long)w[u].y * x[v + u].x;
                    m[v] += (long long)w[u].x * x[v + u].y;
                }
            if (++since == B::SPILL) {
                since = 0;
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    hh[v] += m[v] >> 30;
                    m[v] &= (1ll << 30) - 1;
                }
            }
        }
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const long long a = (hh[v] << 2) + ((m[v] + (1ll << 27)) >> 28);
            res[v] = fx_big(a) ? fx_to_double(a, E + ew + 2) : fx_small_to_double(a, E + ew + 2);
            if ((u64)(a + (1ll << 55)) < (1ull << 56) && c0 + base + v < n) list[atomicAdd(&listed, 1u)] = (uint16_t)(base + v);
        }
        __syncthreads();
        // the listed outputs: `res` of most stands; the rest is replaced below
        const u32 nl = listed;
        if (nl) {
            bool empty = false;
            for (u32 i = tid; i < nl; i += FT) {
                const int p = list[i];
                u64 mag = 0;  // sum |w f| in units of 2^2 of the results' last place
                for (int j = 0; j < nw && mag < (1ull << 53); ++j)
                    mag += (u64)(u32)abs(ws[j].y) * (u32)abs(s[p + j].y);
                if (mag >= (1ull << 53)) {
                    list[i] = DONE;
                } else {
                    int any = 0;
                    for (int j = 0; j < nw && !any; ++j) any = s[p + j].x | s[p + j].y;
                    if (!any) {
                        list[i] = (uint16_t)(p | EMPTY);
                        empty = true;
                    }
                }
            }
            if (__syncthreads_or(empty) && !faint_cells()) {  // windows of zeros
                for (u32 i = tid; i < nl; i += FT)
                    if (list[i] & EMPTY) list[i] = DONE;
                __syncthreads();
            }
        }
        // results through shared memory, then coalesced stores
#pragma unroll
        for (int v = 0; v < V; ++v) sd[base + v] = res[v];
    } else if (zeros) {
#pragma unroll
        for (int v = 0; v < V; ++v) sd[base + v] = 0.0;
    } else {
        // every sweep leaves cell e of the sum at e: it reads e .. e + 2 r1, ascending in waves of FT
        for (int e = tid; e < cells; e += FT) sd[e] = load(e);
        __syncthreads();
        for (int k = 1; k <= sweeps; ++k) {
            const int span = len - 2 * r1 * k;
            for (int e0 = 0; e0 < span; e0 += FT) {
                double acc = 0.0;
                if (e0 + tid < span)
                    for (int j = 0; j < 2 * r1 + 1; ++j) acc = fma(w1[j], sd[e0 + tid + j], acc);
                __syncthreads();  // in place: cells below e0 + FT are read by this wave only ...
                if (e0 + tid < span) sd[e0 + tid] = acc;
                __syncthreads();  // ... and the next wave starts at e0 + FT
            }
        }
    }
    __syncthreads();
    if (fixed && listed) {
        for (u32 i = tid; i < listed; i += FT)
            if (list[i] != DONE) sd[list[i] & (EMPTY - 1)] = by_fp64(list[i] & (EMPTY - 1));
        __syncthreads();
    }
    pdl_launch_dependents();  // not earlier: the next launch's CTAs would wait on the SMs
    const int valid = (int)min((int64_t)CH, n - c0);
    if (valid == CH) {
        for (int q = tid; q < CH / 2; q += FT)
            reinterpret_cast<double2 *>(outx + c0)[q] = reinterpret_cast<const double2 *>(sd)[q];
    } else {
        for (int q = tid; q < valid; q += FT) outx[c0 + q] = sd[q];
    }
    if (images && (c0 < r1 || c0 + CH > n - r1))
        for (int q = tid; q < valid; q += FT) {
            const int64_t p = c0 + q;
            if (p < r1) outx[p + n] = sd[q];
            if (p >= n - r1) outx[p - n] = sd[q];
        }
}

__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// int32 sweeps composed into one correlation of radius r <= 64 modulo 2^32.  Shared loads as above;
// bound by the 64 multiply-adds per clock and SM, and at 2^20 cells by the latency of one load,
// compute and store after another.
template <int V>
__global__ void __launch_bounds__(FT)
xcorr_i32_kernel(const uint32_t *__restrict__ in, uint32_t *__restrict__ out, Geom geo,
                 const __grid_constant__ I32Weights wp, int r, int r1, int images) {
    constexpr int CH = FT * V;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    uint32_t *s = reinterpret_cast<uint32_t *>(smem_raw);
    const int tid = threadIdx.x, nwp = (2 * r + 1 + V - 1) / V * V, cells = CH + nwp + V;
    const int64_t n = geo.n[0], c0 = (int64_t)blockIdx.x * CH;
    const uint32_t *inx = in + geo.off[0];
    uint32_t *outx = out + geo.off[0];
    pdl_wait();
    // asynchronous 4-byte copies, all in flight at once: a load and a shared store per cell left
    // the block waiting for one round trip after another
    if (c0 - r >= 0 && c0 - r + cells <= n) {
        const uint32_t *src = inx + (c0 - r);
        for (int e = tid; e < cells; e += FT) cp_async4(s + e, src + e);
    } else {
        for (int e = tid; e < cells; e += FT) {
            int64_t gi = (c0 - r + e) % n;
            cp_async4(s + e, inx + (gi < 0 ? gi + n : gi));
        }
    }
    cp_async_wait_all();
    __syncthreads();
    const int base = tid * V;
    uint32_t acc[V];
#pragma unroll
    for (int v = 0; v < V; ++v) acc[v] = 0u;
    for (int j0 = 0; j0 < nwp; j0 += V) {
        uint32_t x[2 * V - 1];
#pragma unroll
        for (int q = 0; q < 2 * V - 1; ++q) x[q] = s[base + j0 + q];
#pragma unroll
        for (int u = 0; u < V; ++u)
#pragma unroll
            for (int v = 0; v < V; ++v) acc[v] += wp.w[j0 + u] * x[v + u];
    }
    __syncthreads();
#pragma unroll
    for (int v = 0; v < V; ++v) s[base + v] = acc[v];
    __syncthreads();
    // the next launch's CTAs enter here and not earlier: waiting on the SMs from the start, they took
    // 9.7 us per 2^20-cell call against 6.6
    pdl_launch_dependents();
    const int valid = (int)min((int64_t)CH, n - c0);
    if (valid == CH) {
        for (int q = tid; q < CH / 4; q += FT) reinterpret_cast<uint4 *>(outx + c0)[q] = reinterpret_cast<const uint4 *>(s)[q];
    } else {
        for (int q = tid; q < valid; q += FT) outx[c0 + q] = s[q];
    }
    if (images && (c0 < r1 || c0 + CH > n - r1))
        for (int q = tid; q < valid; q += FT) {
            const int64_t p = c0 + q;
            if (p < r1) outx[p + n] = s[q];
            if (p >= n - r1) outx[p - n] = s[q];
        }
}

// Block size V for n cells at radius r: the one with the least estimated time of the busiest SM.
// A CTA costs, in cycles of its SM, its padded multiply-adds (3 V^2 per block for each of 8 warps,
// at 32 lanes per clock), half of the shared loads' wavefronts, which overlap them in part, and
// the conversion and output of its cells (about 300 V).  The estimate is within 20 % of the times
// measured from 11 to 2001 weights and 30 000 to 2^24 cells, and picks the measured best, e.g.
// V = 3 for 30 000 cells and 97 weights (12.4 us; V = 7: 20.6, V = 9: 24.7), V = 9 for 300 001
// cells and 2001 weights (256 us; V = 3: 297, V = 7: 386).
int fx_block(int r, int64_t n) {
    int best = 9;
    double least = 0.0;
    for (int v : {3, 7, 9}) {
        const int nb = (2 * r + 1 + v - 1) / v;
        const double cta = 8.0 * nb * (3.0 * v * v + 0.5 * (5 * v - 2)) + 300.0 * v;
        const int64_t ctas = (n + FT * v - 1) / (FT * v), sms = device_sms();
        const double c = cta * (double)((ctas + sms - 1) / sms);
        if (least == 0.0 || c < least) { least = c; best = v; }
    }
    return best;
}

template <int V, int MINB>
cudaError_t run(const double *in, double *out, const Geom &g, const FxSweep &w, bool periodic, bool images,
                cudaStream_t s) {
    auto k = xcorr_wide_fx_kernel<V, MINB>;
    const size_t smem = FxWide<V>::smem(w.r);
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    const unsigned blocks = (unsigned)((g.n[0] + FxWide<V>::CH - 1) / FxWide<V>::CH);
    return launch_pdl(k, dim3(blocks), dim3(FT), smem, s, in, out, g, w.w, static_cast<const int2 *>(w.limbs), w.ew, w.r,
                      w.w1, w.r1, w.sweeps, periodic ? 1 : 0, images ? 1 : 0);
}

}  // namespace

// The weights hi + lo (lo may be null) as balanced limbs W = 2^30 wh + wl (stored {wl, wh}),
// w = W 2^(ew - 57): |W| <= 2^57 and sum |W| < 2^61, so that with |q| <= 2^59 the result
// sum W q / 2^58 stays below 2^62 and the cross products of 20 terms below 2^63.  Rounding the
// weights and leaving out the low limbs' products costs at most one unit per term each, rounding
// the cells 4 in all.
bool fx_wide_weights(const double *hi, const double *lo, int count, std::vector<int32_t> &limbs, int *ew) {
    double top = 0.0, sum = 0.0;
    for (int i = 0; i < count; ++i) {
        if (!std::isfinite(hi[i])) return false;
        top = std::fmax(top, std::fabs(hi[i]));
        sum += std::fabs(hi[i]);
    }
    if (!(top > 0.0) || !std::isfinite(sum)) return false;
    int e = 0;
    (void)std::frexp(top, &e);
    while (std::ldexp(sum, -e) >= 15.0) ++e;
    if (e < -100 || e > 100) return false;
    limbs.resize(2 * (size_t)count);
    for (int i = 0; i < count; ++i) {
        const double a = std::ldexp(hi[i], 57 - e), whole = std::nearbyint(a);
        const double rest = (a - whole) + (lo ? std::ldexp(lo[i], 57 - e) : 0.0);
        const long long W = (long long)whole + std::llrint(rest);
        const long long h = (W + (1ll << 29)) >> 30;
        limbs[2 * i] = (int32_t)(W - h * (1ll << 30));
        limbs[2 * i + 1] = (int32_t)h;
    }
    *ew = e;
    return true;
}

// (hi + lo) convolved with the 2r+1 weights g, in place, as unevaluated sums.
void fx_convolve(const double *g, int r, std::vector<double> &hi, std::vector<double> &lo) {
    std::vector<double> h(hi.size() + 2 * r, 0.0), l(hi.size() + 2 * r, 0.0);
    for (size_t i = 0; i < hi.size(); ++i)
        for (int j = 0; j < 2 * r + 1; ++j) {
            // h + l += (hi + lo) g: exact product of the leading parts, Knuth's two-sum
            const double p = hi[i] * g[j], e = std::fma(hi[i], g[j], -p) + lo[i] * g[j];
            double &H = h[i + j], &Lo = l[i + j];
            const double t = H + p, z = t - H;
            Lo += ((H - (t - z)) + (p - z)) + e;
            H = t + Lo;
            Lo -= H - t;
        }
    hi.swap(h);
    lo.swap(l);
}

void i32_compose(const int32_t *g, int r, int kmax, std::vector<I32Weights> &o) {
    o.assign(kmax, I32Weights{});
    std::copy(g, g + 2 * r + 1, o[0].w);
    for (int k = 2; k <= kmax; ++k)
        for (int i = 0; i < 2 * r * (k - 1) + 1; ++i)
            for (int j = 0; j < 2 * r + 1; ++j) o[k - 1].w[i + j] += o[k - 2].w[i] * (uint32_t)g[j];
}

cudaError_t launch_xcorr_fx(const double *in, double *out, const Geom &g, const FxSweep &w, bool periodic, bool images,
                            cudaStream_t s) {
    switch (fx_block(w.r, g.n[0])) {
    case 3: return run<3, 5>(in, out, g, w, periodic, images, s);
    case 7:
        // few weights: more CTAs to overlap loads, conversion and output (11 weights, 2^24 cells: 152
        // against 176 us); many: the register budget of two (61 weights, 2^20 cells: 35 against 37 us)
        if (w.r <= 16) return run<7, 4>(in, out, g, w, periodic, images, s);
        return run<7, 2>(in, out, g, w, periodic, images, s);
    default: return run<9, 3>(in, out, g, w, periodic, images, s);
    }
}

cudaError_t launch_xcorr_i32(const int32_t *in, int32_t *out, const Geom &g, const I32Weights &w, int r, int r1,
                             bool images, cudaStream_t s) {
    constexpr int V = 9, CH = FT * V;
    const int nwp = (2 * r + 1 + V - 1) / V * V;
    if (nwp > I32Weights::N) return cudaErrorInvalidValue;
    const unsigned blocks = (unsigned)((g.n[0] + CH - 1) / CH);
    return launch_pdl(xcorr_i32_kernel<V>, dim3(blocks), dim3(FT), sizeof(uint32_t) * (size_t)(CH + nwp + V), s,
                      reinterpret_cast<const uint32_t *>(in), reinterpret_cast<uint32_t *>(out), g, w, r, r1,
                      images ? 1 : 0);
}

}  // namespace stn

// xcorr_fx.cu -- FP64 1D cross-correlation (Sec. 3.1, Eq. 3) of radius 5..1024 in fixed point.
//
// 2r+1 FP64 multiply-adds per output ran at 99 % of the FP64 pipe (2 per clock and SM).  Here a
// CTA converts its chunk of cells, halo included, to signed 59-bit integers of one binary scale,
// split into two 30-bit limbs, and the weights come as limbs too.  A product is then three
// 32 x 32 + 64-bit multiply-adds (the product of the two low limbs, below 2^-60 of the scale, is
// left out), at 64 per clock and SM: 10 times the FP64 rate.
//
//   * As in xcorr_wide.cu each thread computes V consecutive outputs (V odd: conflict-free shared
//     loads) and keeps V weights and 2V-1 cells in registers per block of V weights.
//   * An output keeps two 64-bit sums: the high products HH and the cross products M, whose
//     upper part moves to HH every one to three blocks, before 20 terms could overflow it.
//   * Accuracy (fx_wide_weights): the result is off by at most 2 (2r+1) + 4 units of 2^-62 of
//     the largest result the scale admits, which is no more than a chain of FP64 multiply-adds may
//     be off, 2^-53 (2r+1) sum |w f|, wherever sum |w f| is at least 2^-7 of that result.  An output
//     of that size itself shows it; the others are listed, their sum |w f| is accumulated from
//     the high limbs until it passes the bound (a few terms for most), and what stays below is
//     evaluated by FP64 multiply-adds in the order j = -r .. r.
//   * A chunk with infinities, NaN or exponents near the ends of the range runs FP64
//     multiply-adds throughout.
#include <algorithm>
#include <vector>

#include "fixed.cuh"
#include "internal.h"

namespace stn {
namespace {

constexpr int FT = 256;  // threads per CTA

template <int V_> struct FxWide {
    static constexpr int V = V_, CH = FT * V;
    static constexpr int SPILL = 20 / V;  // blocks between two spills of M: at most 20 terms
    static __host__ __device__ int nwp(int r) { return (2 * r + 1 + V - 1) / V * V; }
    // cells: the chunk, its halo, and zeros for the padded weight blocks
    static __host__ __device__ int cells(int r) { return CH + nwp(r) + V; }
    static __host__ __device__ size_t smem(int r) { return sizeof(int2) * (size_t)(cells(r) + nwp(r)) + sizeof(uint16_t) * CH; }
    static_assert(V % 2 == 1 && SPILL >= 1, "");
    static_assert(CH <= 65536, "list entries are 16-bit");
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

template <int V>
__global__ void __launch_bounds__(FT, 2)
xcorr_wide_fx_kernel(const double *__restrict__ in, double *__restrict__ out, Geom geo, const double *__restrict__ wg,
                     const int2 *__restrict__ wfx, int ew, int r, int periodic, int images) {
    using B = FxWide<V>;
    constexpr int CH = B::CH;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ u32 red[FT / 32];
    __shared__ u32 listed;
    const int tid = threadIdx.x, nw = 2 * r + 1, nwp = B::nwp(r), cells = B::cells(r), len = CH + 2 * r;
    int2 *s = reinterpret_cast<int2 *>(smem_raw);
    double *sd = reinterpret_cast<double *>(smem_raw);  // the cells before conversion, and the results
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
    if (tid == 0) listed = 0u;
    pdl_launch_dependents();
    pdl_wait();

    // stage the cells and find the largest exponent.  Cells past the last output's window count as 0.
    u32 hm = 0u;
    const bool inside = c0 - r >= 0 && c0 + CH + r <= n;
    const int used = (int)min((int64_t)len, n - c0 + 2 * r);
    for (int e = tid; e < cells; e += FT) {
        const double v = e < used ? (inside ? inx[c0 - r + e] : cell(c0 - r + e)) : 0.0;
        sd[e] = v;
        hm = max(hm, (u32)__double2hiint(v) & 0x7fffffffu);
    }
    for (int j = tid; j < nwp; j += FT) ws[j] = j < nw ? wfx[j] : make_int2(0, 0);
    hm = __reduce_max_sync(0xffffffffu, hm);
    if ((tid & 31) == 0) red[tid >> 5] = hm;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < FT / 32; ++w) hm = max(hm, red[w]);
    const int E = (int)(hm >> 20);
    const bool fixed = E >= FX_SMIN && E <= FX_EMAX;  // uniform per block

    // FP64 multiply-adds of output p from global memory
    auto by_fp64 = [&](int p) -> double {
        double acc = 0.0;
        for (int j = 0; j < nw; ++j) acc = fma(wg[j], inside ? inx[c0 - r + p + j] : cell(c0 - r + p + j), acc);
        return acc;
    };

    const int base = tid * V;
    double res[V];
    if (fixed) {
        for (int e = tid; e < cells; e += FT) s[e] = fx_limbs(sd[e], E);  // in place: own elements
        __syncthreads();
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
            for (u32 i = tid; i < nl; i += FT) {
                const int p = list[i];
                u64 mag = 0;  // sum |w f| in units of 2^2 of the results' last place
                for (int j = 0; j < nw && mag < (1ull << 53); ++j)
                    mag += (u64)(u32)abs(ws[j].y) * (u32)abs(s[p + j].y);
                if (mag >= (1ull << 53)) list[i] = 0xffffu;
            }
            __syncthreads();
        }
    } else {
        __syncthreads();
#pragma unroll
        for (int v = 0; v < V; ++v) {
            double acc = 0.0;
            for (int j = 0; j < nw; ++j) acc = fma(wg[j], sd[base + v + j], acc);
            res[v] = acc;
        }
        __syncthreads();
    }
    // results through shared memory, then coalesced stores
#pragma unroll
    for (int v = 0; v < V; ++v) sd[base + v] = res[v];
    __syncthreads();
    if (fixed && listed) {
        for (u32 i = tid; i < listed; i += FT)
            if (list[i] != 0xffffu) sd[list[i]] = by_fp64(list[i]);
        __syncthreads();
    }
    const int valid = (int)min((int64_t)CH, n - c0);
    if (valid == CH) {
        for (int q = tid; q < CH / 2; q += FT)
            reinterpret_cast<double2 *>(outx + c0)[q] = reinterpret_cast<const double2 *>(sd)[q];
    } else {
        for (int q = tid; q < valid; q += FT) outx[c0 + q] = sd[q];
    }
    if (images && (c0 < r || c0 + CH > n - r))
        for (int q = tid; q < valid; q += FT) {
            const int64_t p = c0 + q;
            if (p < r) outx[p + n] = sd[q];
            if (p >= n - r) outx[p - n] = sd[q];
        }
}

// Block size V for radius r: the one with the fewest cycles per output, counting padded
// multiply-adds (3 V^2 per block at 64 per clock and SM, in warp cycles 1.5 V^2) and half of the
// shared loads' (2 (2V - 1) + V wavefronts per block), which overlap them in part.
int fx_block(int r) {
    int best = 9;
    double least = 0.0;
    for (int v : {5, 7, 9}) {
        const int nb = (2 * r + 1 + v - 1) / v;
        const double c = nb * (1.5 * v * v + 0.5 * (5 * v - 2)) / v;
        if (least == 0.0 || c < least) { least = c; best = v; }
    }
    return best;
}

template <int V>
cudaError_t run(int r, const double *in, double *out, const Geom &g, const double *wdev, const int2 *wfx, int ew,
                bool periodic, bool images, cudaStream_t s) {
    auto k = xcorr_wide_fx_kernel<V>;
    const size_t smem = FxWide<V>::smem(r);
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    const unsigned blocks = (unsigned)((g.n[0] + FxWide<V>::CH - 1) / FxWide<V>::CH);
    return launch_pdl(k, dim3(blocks), dim3(FT), smem, s, in, out, g, wdev, wfx, ew, r, periodic ? 1 : 0, images ? 1 : 0);
}

}  // namespace

// The weights as balanced limbs W = 2^30 wh + wl (stored {wl, wh}), w = W 2^(ew - 57): |W| <= 2^57
// and sum |W| < 2^61, so that with |q| <= 2^59 the result sum W q / 2^58 stays below 2^62 and the
// cross products of 20 terms below 2^63.  Rounding the weights and leaving out the low limbs'
// products costs at most one unit per term each, rounding the cells 4 in all.
bool fx_wide_weights(const double *w, int count, std::vector<int32_t> &limbs, int *ew) {
    double top = 0.0, sum = 0.0;
    for (int i = 0; i < count; ++i) {
        if (!std::isfinite(w[i])) return false;
        top = std::fmax(top, std::fabs(w[i]));
        sum += std::fabs(w[i]);
    }
    if (!(top > 0.0) || !std::isfinite(sum)) return false;
    int e = 0;
    (void)std::frexp(top, &e);
    while (std::ldexp(sum, -e) >= 15.0) ++e;
    if (e < -100 || e > 100) return false;
    limbs.resize(2 * (size_t)count);
    for (int i = 0; i < count; ++i) {
        const long long W = std::llrint(std::ldexp(w[i], 57 - e));
        const long long h = (W + (1ll << 29)) >> 30;
        limbs[2 * i] = (int32_t)(W - h * (1ll << 30));
        limbs[2 * i + 1] = (int32_t)h;
    }
    *ew = e;
    return true;
}

cudaError_t launch_xcorr_wide_fx(int r, const double *in, double *out, const Geom &g, const double *wdev,
                                 const void *wfx, int ew, bool periodic, bool images, cudaStream_t s) {
    const int2 *w = static_cast<const int2 *>(wfx);
    switch (fx_block(r)) {
    case 5: return run<5>(r, in, out, g, wdev, w, ew, periodic, images, s);
    case 7: return run<7>(r, in, out, g, wdev, w, ew, periodic, images, s);
    default: return run<9>(r, in, out, g, wdev, w, ew, periodic, images, s);
    }
}

}  // namespace stn

// xcorr_pair.cu -- FP32 1D cross-correlation (Sec. 3.1, Eq. 3) of radius 33..1024 on periodic arrays
// with packed multiply-adds (a caller-filled halo stays with xcorr_wide.cu).
//
// The register-blocked kernel of xcorr_wide.cu issues one instruction per multiply-add and was
// bound by issue: 81 % of the slots for 62 % of the FP32 pipe at r = 64.  Blackwell's packed FP32x2
// multiply-add does two per slot, but takes its operands from aligned register pairs, and
// neighbouring outputs need neighbouring, so mostly unaligned, pairs of cells.  Here the two
// halves of a pair are outputs half a chunk apart: shared memory holds {cell i, cell i + H} in one
// 8-byte slot, so that every window element, weight {w, w} and sum is an aligned pair.
//
//   * A thread computes 2 V outputs (V odd: lanes V slots apart fall on distinct banks), per block
//     of V weights from 2V-1 slots in registers, of which the next block keeps V-1, in the order
//     j = -r .. r with one fused multiply-add each: bit-identical to xcorr_wide.cu.
//   * Cells are staged by 4-byte asynchronous copies into their slots; CTAs of one SM overlap each
//     other's staging and stores.  (Persistent CTAs with the next chunk's copies in flight
//     measured no faster: 98 against 97 us at r = 64 before the window was kept.)
//   * Bound by the FP32 pipe and the shared loads together (58 % and about 50 % busy at r = 64).
//     2^24 cells: r = 64 101.7 -> 91.4 us, r = 256 346 -> 298; 2^20 cells, r = 64 15.6 -> 10.5.
#include <algorithm>

#include "internal.h"

namespace stn {
namespace {

constexpr int PT = 256;  // threads per CTA

template <int V_> struct PairCfg {
    static constexpr int V = V_, H = PT * V, CH = 2 * H;
    static __host__ __device__ int slots(int r) { return H + 2 * r; }
    static __host__ __device__ size_t smem(int r) { return sizeof(float2) * (size_t)(slots(r) + 2 * r + 1); }
    static_assert(V % 2 == 1, "");
};

template <int V, int MINB>
__global__ void __launch_bounds__(PT, MINB)
xcorr_pair_kernel(const float *__restrict__ in, float *__restrict__ out, Geom geo, const float *__restrict__ wg, int r,
                  int images) {
    using B = PairCfg<V>;
    constexpr int H = B::H, CH = B::CH;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int tid = threadIdx.x, nw = 2 * r + 1, slots = B::slots(r);
    float2 *s = reinterpret_cast<float2 *>(smem_raw);
    float *sf = reinterpret_cast<float *>(smem_raw);
    float2 *ws = s + slots;
    const int64_t n = geo.n[0], c0 = (int64_t)blockIdx.x * CH;
    const float *inx = in + geo.off[0];
    float *outx = out + geo.off[0];
    pdl_wait();

    // slot i: cells c0 - r + i and c0 + H - r + i
    if (c0 - r >= 0 && c0 + CH + r <= n) {
        const float *src = inx + (c0 - r);
        for (int i = tid; i < slots; i += PT) {
            cp_async4(&s[i].x, src + i);
            cp_async4(&s[i].y, src + H + i);
        }
    } else {
        auto cell = [&](int64_t gi) -> float {
            if (gi >= 0 && gi < n) return inx[gi];
            if (gi >= n + r) return 0.f;  // no output's window
            gi %= n;
            return inx[gi < 0 ? gi + n : gi];
        };
        for (int i = tid; i < slots; i += PT) s[i] = make_float2(cell(c0 - r + i), cell(c0 + H - r + i));
    }
    for (int j = tid; j < nw; j += PT) ws[j] = make_float2(wg[j], wg[j]);
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();

    const float2 *xp = s + tid * V;
    float2 acc[V], x[2 * V - 1];
#pragma unroll
    for (int v = 0; v < V; ++v) acc[v] = make_float2(0.f, 0.f);
#pragma unroll
    for (int q = 0; q < V - 1; ++q) x[q + V] = xp[q];
    int j0 = 0;
#pragma unroll 2
    for (; j0 <= nw - V; j0 += V) {
        // the window moves by V slots a block: V - 1 of its 2V - 1 stay in registers
#pragma unroll
        for (int q = 0; q < V - 1; ++q) x[q] = x[q + V];
#pragma unroll
        for (int q = V - 1; q < 2 * V - 1; ++q) x[q] = xp[j0 + q];
#pragma unroll
        for (int u = 0; u < V; ++u) {
            const float2 w = ws[j0 + u];
#pragma unroll
            for (int v = 0; v < V; ++v) acc[v] = __ffma2_rn(w, x[v + u], acc[v]);
        }
    }
    // The last, partial block has its own weights only: padded with zeros it would multiply cells
    // beyond an output's window, and 0 x infinity is NaN.
    const int rest = nw - j0;
    if (rest > 0) {
#pragma unroll
        for (int q = 0; q < V - 1; ++q) x[q] = x[q + V];
#pragma unroll
        for (int u = 0; u < V - 1; ++u)
            if (u < rest) {
                x[V - 1 + u] = xp[j0 + V - 1 + u];
                const float2 w = ws[j0 + u];
#pragma unroll
                for (int v = 0; v < V; ++v) acc[v] = __ffma2_rn(w, x[v + u], acc[v]);
            }
    }
    __syncthreads();
    const int base = tid * V;
#pragma unroll
    for (int v = 0; v < V; ++v) {
        sf[base + v] = acc[v].x;
        sf[H + base + v] = acc[v].y;
    }
    __syncthreads();
    pdl_launch_dependents();  // not earlier: the next launch's CTAs would wait on the SMs
    const int valid = (int)min((int64_t)CH, n - c0);
    if (valid == CH) {
        for (int q = tid; q < CH / 4; q += PT) reinterpret_cast<float4 *>(outx + c0)[q] = reinterpret_cast<const float4 *>(sf)[q];
    } else {
        for (int q = tid; q < valid; q += PT) outx[c0 + q] = sf[q];
    }
    if (images && (c0 < r || c0 + CH > n - r))
        for (int q = tid; q < valid; q += PT) {
            const int64_t p = c0 + q;
            if (p < r) outx[p + n] = sf[q];
            if (p >= n - r) outx[p - n] = sf[q];
        }
}

template <int V, int MINB>
cudaError_t run(const float *in, float *out, const Geom &g, const float *wdev, int r, bool images, cudaStream_t s) {
    auto k = xcorr_pair_kernel<V, MINB>;
    const size_t smem = PairCfg<V>::smem(r);
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    const unsigned blocks = (unsigned)((g.n[0] + PairCfg<V>::CH - 1) / PairCfg<V>::CH);
    return launch_pdl(k, dim3(blocks), dim3(PT), smem, s, in, out, g, wdev, r, images ? 1 : 0);
}

}  // namespace

// Block size V for n cells at radius r: the one with the least estimated time of the busiest SM, in
// cycles per CTA: what its 8 warps' blocks and its cells' staging and output (215 V) measured on
// 2^24 cells.  Small inputs take small V, which spread over more SMs (65 536 cells, r = 64: V = 3
// 6.4 us, V = 13 12.4; 300 001 cells, r = 500: V = 5 22.7 us, V = 3 28.8, V = 13 41).
static int pair_block(int r, int64_t n) {
    static constexpr struct { int v; double block; } T[] = {{3, 9.0}, {5, 18.7}, {7, 32.7}, {9, 51.0}, {13, 104.0}};
    int best = 13;
    double least = 0.0;
    for (const auto &t : T) {
        const int nb = (2 * r + 1 + t.v - 1) / t.v;
        const int64_t ch = 2 * PT * t.v, ctas = (n + ch - 1) / ch, sms = device_sms();
        const double c = (8.0 * nb * t.block + 215.0 * t.v) * (double)((ctas + sms - 1) / sms);
        if (least == 0.0 || c < least) { least = c; best = t.v; }
    }
    return best;
}

cudaError_t launch_xcorr_pair(const float *in, float *out, const Geom &g, const float *wdev, int r, bool images,
                              cudaStream_t s) {
    switch (pair_block(r, g.n[0])) {
    case 3: return run<3, 5>(in, out, g, wdev, r, images, s);
    case 5: return run<5, 4>(in, out, g, wdev, r, images, s);
    case 7: return run<7, 3>(in, out, g, wdev, r, images, s);
    case 9: return run<9, 3>(in, out, g, wdev, r, images, s);
    default: return run<13, 3>(in, out, g, wdev, r, images, s);
    }
}

}  // namespace stn

// mhd_win.cuh -- the 6th-order central differences of one cell's window (weights pre-scaled by the
// grid spacing), and the vector access of the RK register, shared by the MHD kernels.
#pragma once

#include "mhd_rhs.cuh"

namespace stn {

// Differences over a window W that supplies at(field, plane 0..6, dx, dy), written out one IEEE
// operation at a time (mhd_rhs.cuh says why).
template <typename C, typename W> struct WinOps {
    __device__ __forceinline__ const W &self() const { return *static_cast<const W *>(this); }
    __device__ __forceinline__ C val(int q) const { return self().at(q, 3, 0, 0); }
    // value at offset s along axis (0: x, 1: y, 2: z)
    __device__ __forceinline__ C ax(int q, int axis, int s) const {
        return axis == 0 ? self().at(q, 3, s, 0) : axis == 1 ? self().at(q, 3, 0, s) : self().at(q, 3 + s, 0, 0);
    }
    // first derivative: c0 (f1 - f-1) + c1 (f2 - f-2) + c2 (f3 - f-3)
    __device__ __forceinline__ C d1(int q, int axis, const C *c) const {
        C a = mul(c[0], sub(ax(q, axis, 1), ax(q, axis, -1)));
        a = fmad(c[1], sub(ax(q, axis, 2), ax(q, axis, -2)), a);
        return fmad(c[2], sub(ax(q, axis, 3), ax(q, axis, -3)), a);
    }
    // second derivative: c0 f0 + c1 (f1 + f-1) + c2 (f2 + f-2) + c3 (f3 + f-3)
    __device__ __forceinline__ C d2(int q, int axis, C c0, const C *c) const {
        C a = mul(c0, ax(q, axis, 0));
        a = fmad(c[0], add(ax(q, axis, 1), ax(q, axis, -1)), a);
        a = fmad(c[1], add(ax(q, axis, 2), ax(q, axis, -2)), a);
        return fmad(c[2], add(ax(q, axis, 3), ax(q, axis, -3)), a);
    }
    // mixed derivative of axes (a1 < a2), diagonal form:
    // sum_a m_a [(f(+a,+a) + f(-a,-a)) - (f(+a,-a) + f(-a,+a))]
    __device__ __forceinline__ C mx(int q, int pair, int s1, int s2) const {
        return pair == 0 ? self().at(q, 3, s1, s2) : pair == 1 ? self().at(q, 3 + s2, s1, 0) : self().at(q, 3 + s2, 0, s1);
    }
    __device__ __forceinline__ C dmix(int q, int pair, const C *m) const {
        C acc = mul(m[0], sub(add(mx(q, pair, 1, 1), mx(q, pair, -1, -1)), add(mx(q, pair, 1, -1), mx(q, pair, -1, 1))));
        acc = fmad(m[1], sub(add(mx(q, pair, 2, 2), mx(q, pair, -2, -2)), add(mx(q, pair, 2, -2), mx(q, pair, -2, 2))),
                   acc);
        return fmad(m[2], sub(add(mx(q, pair, 3, 3), mx(q, pair, -3, -3)), add(mx(q, pair, 3, -3), mx(q, pair, -3, 3))),
                    acc);
    }
};

// The 7-plane window of all fields around one cell in shared memory: p[k] points at the cell
// (field 0) in plane z + k - 3; field q is FE elements further, row neighbours RS elements apart.
template <typename C, typename S, int FE, int RS>
struct Win : WinOps<C, Win<C, S, FE, RS>> {
    const S *p[7];
    __device__ __forceinline__ C at(int q, int k, int dx, int dy) const {
        return to_c<C>(p[k][q * FE + dy * RS + dx]);
    }
};

// The same around one cell of padded fields in global memory.
struct GlobalWin : WinOps<double, GlobalWin> {
    const double *f[8];
    int64_t sy, sz;
    __device__ __forceinline__ double at(int q, int k, int dx, int dy) const {
        return f[q][(k - 3) * sz + dy * sy + dx];
    }
};

// The 8 interleaved values of one cell in the RK register / Kahan arrays (16-byte aligned):
// loaded and stored as 16-byte vectors.
template <typename S, typename C>
__device__ __forceinline__ void load8(const S *p, C (&v)[8]) {
    if constexpr (sizeof(S) == 2) {
        const uint4 a = *reinterpret_cast<const uint4 *>(p);
        const S *e = reinterpret_cast<const S *>(&a);
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = to_c<C>(e[q]);
    } else {
        constexpr int PER = 16 / (int)sizeof(S);  // values per 16-byte vector
#pragma unroll
        for (int h = 0; h < 8 / PER; ++h) {
            const uint4 a = reinterpret_cast<const uint4 *>(p)[h];
            const S *e = reinterpret_cast<const S *>(&a);
#pragma unroll
            for (int u = 0; u < PER; ++u) v[h * PER + u] = to_c<C>(e[u]);
        }
    }
}
template <typename S>
__device__ __forceinline__ void store8(S *p, const S (&v)[8]) {
    constexpr int PER = 16 / (int)sizeof(S);
#pragma unroll
    for (int h = 0; h < 8 / PER; ++h) {
        uint4 a;
        S *e = reinterpret_cast<S *>(&a);
#pragma unroll
        for (int u = 0; u < PER; ++u) e[u] = v[h * PER + u];
        reinterpret_cast<uint4 *>(p)[h] = a;
    }
}

}  // namespace stn

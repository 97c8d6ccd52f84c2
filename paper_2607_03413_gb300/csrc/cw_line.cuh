// cw_line.cuh -- whole x-lines (N consecutive values) in the widest accesses their pitch allows.
//
// A thread that owns an x-line touches N consecutive values, its neighbours the next lines. Read or
// written value by value, every access of a warp spans N times the bytes it uses: N times the L1
// wavefronts and, for stores, partial sectors; from shared memory N-way bank conflicts for even N. With
// one 16-byte access for N = 4 floats (two for N = 8, three 8-byte ones for N = 6, ...) a warp moves the
// span once. Lines start at multiples of N values, so the alignment of a vector's base decides for all of
// its lines; vectors passed in by callers are checked (`aligned`) and read value by value otherwise.
#pragma once
#include <cstdint>
#include <type_traits>

namespace cw {

template <int N, class V>
struct LineVec {
    static constexpr int BYTES = N * (int)sizeof(V);
    static constexpr int VB = BYTES % 16 == 0 ? 16 : BYTES % 8 == 0 ? 8 : BYTES % 4 == 0 ? 4 : 2;
    static constexpr int NW = BYTES / VB;
    static constexpr bool WIDE = VB > (int)sizeof(V);  // else (odd N) value by value is all there is
    using W = std::conditional_t<VB == 16, uint4,
                                 std::conditional_t<VB == 8, uint2, std::conditional_t<VB == 4, uint32_t, uint16_t>>>;
    static_assert(VB >= (int)sizeof(V), "a line is a whole number of accesses");

    static __host__ __device__ __forceinline__ bool aligned(const void *base)
    {
        return (reinterpret_cast<uintptr_t>(base) & (VB - 1)) == 0;
    }
    static __device__ __forceinline__ void ld(const V *p, V (&v)[N])
    {
        W w[NW];
#pragma unroll
        for (int i = 0; i < NW; ++i) w[i] = reinterpret_cast<const W *>(p)[i];
        __builtin_memcpy(v, w, BYTES);
    }
    // read-only data (not written by the kernel through any pointer)
    static __device__ __forceinline__ void ld_nc(const V *p, V (&v)[N])
    {
        W w[NW];
#pragma unroll
        for (int i = 0; i < NW; ++i) w[i] = __ldg(reinterpret_cast<const W *>(p) + i);
        __builtin_memcpy(v, w, BYTES);
    }
    static __device__ __forceinline__ void st(V *p, const V (&v)[N])
    {
        W w[NW];
        __builtin_memcpy(w, v, BYTES);
#pragma unroll
        for (int i = 0; i < NW; ++i) reinterpret_cast<W *>(p)[i] = w[i];
    }
};

// the same for a vector whose alignment is known at run time only (`vec`: aligned(base), uniform)
template <int N, class V>
__device__ __forceinline__ void line_ld(const V *p, V (&v)[N], bool vec)
{
    if (LineVec<N, V>::WIDE && vec) {
        LineVec<N, V>::ld(p, v);
    } else {
#pragma unroll
        for (int m = 0; m < N; ++m) v[m] = p[m];
    }
}
template <int N, class V>
__device__ __forceinline__ void line_st(V *p, const V (&v)[N], bool vec)
{
    if (LineVec<N, V>::WIDE && vec) {
        LineVec<N, V>::st(p, v);
    } else {
#pragma unroll
        for (int m = 0; m < N; ++m) p[m] = v[m];
    }
}

}  // namespace cw

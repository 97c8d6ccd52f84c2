// cw_apply.cuh -- sum-factorised cell-local operator kernels (the hot path).
//
// One CTA owns a tile of CPB consecutive cells; a cell is worked by N*N threads. A thread plays
// three roles in turn: owner of an x-line (j,k), of a y-line (i,k) and of a z-pencil (i,j), with
// (r % N, r / N) as its pair of indices, r in [0, N*N). 1D contractions along the owned line run
// in registers; switching axis goes through shared memory (the odd row pitch PI = N|1 spreads a
// cell's line accesses over the banks; where two cells share a warp, as at N = 5, some conflicts
// remain). The 1D tables are kernel parameters (constant bank) so every contraction coefficient is
// an immediate operand.
//
// Curved cells (Sec. 6, "the general cell-wise Laplacian: evaluate gradients, apply the physics,
// integrate gradients"), per cell with u the nodal values:
//   u_q = (B x B x B) u                 interpolation to the n^3 Gauss points
//   g   = (D u_q along x, y, z)         reference gradient by Gauss-point collocation
//   h   = G_q g,  m_q = c_q u_q         metric G_q = w_q detJ J^-1 J^-T, c_q = w_q detJ
//   y   = (B^T x B^T x B^T)(D_x^T h_x + D_y^T h_y + D_z^T h_z + m_q)
// Cartesian cells (Sec. 6, the factored form (D x B x B + B x D x B + B x B x D) det J J^-2 read
// with D, B the 1D stiffness and mass matrices):
//   y = a_x (M x M x K) u + a_y (M x K x M) u + a_z (K x M x M) u + a_m (M x M x M) u
// evaluated as two x-contractions, three y-contractions and two z-contractions.
#pragma once
#include <type_traits>

#include "cw_arith.cuh"
#include "cw_line.cuh"
#include "cw_tma.cuh"

namespace cw {

// Even-odd form of an N x N matrix M with reflection symmetry M[N-1-a][N-1-b] = s M[a][b]
// (s = +1 for B and B^T, -1 for D and D^T; the Gauss and Gauss-Lobatto points are symmetric about
// 1/2). With e_b = x_b + x_{N-1-b}, o_b = x_b - x_{N-1-b} (b < N/2) and, for odd N, the middle
// entry x_h:  y_a = sum_b E[a][b] e_b + sum_b O[a][b] o_b + Mid[a] x_h  and
// y_{N-1-a} = s (sum_b E[a][b] e_b - sum_b O[a][b] o_b + Mid[a] x_h), for a < (N+1)/2, where
// E[a][b] = (M[a][b] + M[a][N-1-b])/2, O[a][b] = (M[a][b] - M[a][N-1-b])/2, Mid[a] = M[a][h].
// This halves the multiply-adds of a line contraction (Kronbichler and Kormann's even-odd
// decomposition for sum factorisation).
// For double-float tables the same entries are also stored lane-paired, P[a][b] = (E[a][b], O[a][b])
// so that the even and odd sums of an output pair run as one paired multiply-add chain with each
// coefficient pair one 64-bit constant operand; FP32 tables also hold PM[a] = (Mid[a], 0).
template <class C>
struct EOPair {
    struct type {};
};
template <>
struct EOPair<df64> {
    using type = df64p;
};
template <>
struct EOPair<float> {
    using type = float2;
};

template <int N, class C>
struct EOMat {
    static constexpr int H = N / 2, NA = (N + 1) / 2;
    C E[NA][H > 0 ? H : 1];
    C O[NA][H > 0 ? H : 1];
    C Mid[NA];
    typename EOPair<C>::type P[NA][H > 0 ? H : 1];
    typename EOPair<C>::type PM[std::is_same<C, float>::value ? NA : 1];
};

template <int N, class C>
struct TabMetric {
    C B[N][N];  // B[q][m] = l_m(xi_q): Gauss-Lobatto basis at the Gauss points
    C D[N][N];  // D[q][r] = derivative at xi_q of the Lagrange basis on the Gauss points
    EOMat<N, C> Bf, Bt, Df, Dt;  // even-odd forms of B, B^T (s = +1), D, D^T (s = -1)
    C xq[N], wq[N];              // Gauss points and weights on [0,1] (recomputed geometry)
};

// Recomputed geometry: per cell the 21 coefficients a1..a7 (3 components each) of the trilinear
// map x(xi) = a0 + a1 xi + a2 eta + a3 zeta + a4 xi eta + a5 xi zeta + a6 eta zeta + a7 xi eta zeta,
// layout [cell][7][3]; a0 is not needed (only derivatives enter the metric).
constexpr int kTriCoef = 21;

template <int N, class C>
struct TabAffine {
    C M[N][N];  // 1D mass matrix of the Gauss-Lobatto basis on [0,1]
    C K[N][N];  // 1D stiffness matrix
};

// small helpers -------------------------------------------------------------------------------

// sum of two stored values as the structured DSS forms it (BF16: FP32 sum rounded once)
template <class VS>
struct AddOp {
    static __device__ __forceinline__ VS add(VS a, VS b) { return a + b; }
};
template <>
struct AddOp<__nv_bfloat16> {
    static __device__ __forceinline__ __nv_bfloat16 add(__nv_bfloat16 a, __nv_bfloat16 b)
    {
        return __float2bfloat16_rn(__bfloat162float(a) + __bfloat162float(b));
    }
};

template <class S>
__device__ __forceinline__ S ldg_nc(const S *p) { return __ldg(p); }
template <>
__device__ __forceinline__ __nv_bfloat16 ldg_nc<__nv_bfloat16>(const __nv_bfloat16 *p)
{
    return __ushort_as_bfloat16(__ldg(reinterpret_cast<const unsigned short *>(p)));
}

// out[a] = sum_b M[a][b] in[b]  (TR=false)   or   out[a] = sum_b M[b][a] in[b]  (TR=true)
template <int N, bool TR, class Ar>
__device__ __forceinline__ void contract(const typename Ar::C (&M)[N][N], const typename Ar::T (&in)[N],
                                         typename Ar::T (&out)[N])
{
#pragma unroll
    for (int a = 0; a < N; ++a) {
        typename Ar::T s = Ar::mul(in[0], TR ? M[0][a] : M[a][0]);
#pragma unroll
        for (int b = 1; b < N; ++b) Ar::mad(s, in[b], TR ? M[b][a] : M[a][b]);
        out[a] = Ar::norm(s);
    }
}

// out = M in with M in even-odd form (see EOMat), S = +1 or -1 the reflection sign
// NRM: renormalise each double-float output (no effect for the other arithmetics)
template <int N, int S, class Ar, bool NRM = true>
__device__ __forceinline__ void contract_eo(const EOMat<N, typename Ar::C> &M, const typename Ar::T (&in)[N],
                                            typename Ar::T (&out)[N])
{
    using T = typename Ar::T;
    constexpr int H = N / 2;
    // double-float at N = 3: everything renormalised (83 operations per line instead of 68), which makes
    // the form as accurate as the full one with renormalised outputs (93 operations)
    constexpr bool N3 = N == 3 && std::is_same<Ar, ArDF>::value;
    T e[H], o[H];
#pragma unroll
    for (int b = 0; b < H; ++b) {
        e[b] = Ar::add(in[b], in[N - 1 - b]);
        o[b] = Ar::sub(in[b], in[N - 1 - b]);
        if constexpr (N3) e[b] = Ar::norm(e[b]), o[b] = Ar::norm(o[b]);
    }
    if constexpr (std::is_same<Ar, ArDF>::value) {
        // Double-float: the even and odd sums of an output pair run as one chain of paired FP32
        // operations (lane x even, lane y odd), each lane bit-identical to the scalar chain; the middle
        // input of an odd N enters the even sum only, as a scalar operation on lane x. (Pairing the e/o
        // formation and the final add/subtract as well was slower: the lane shuffles cost more.)
        df64p eo[H];
#pragma unroll
        for (int b = 0; b < H; ++b) eo[b] = dfp_pack(e[b], o[b]);
#pragma unroll
        for (int a = 0; a < H; ++a) {
            df64p y2 = dfp_mul(eo[0], M.P[a][0]);
#pragma unroll
            for (int b = 1; b < H; ++b) dfp_mad(y2, eo[b], M.P[a][b]);
            T ye = dfp_x(y2);
            const T yo = dfp_y(y2);
            if constexpr (N % 2 == 1) Ar::mad(ye, in[H], M.Mid[a]);
            // without NRM the outputs stay unnormalised (|lo| a few ulp of hi): every consumer is a
            // double-float operation or the final conversion, which take that form as it is
            const T sum = Ar::add(ye, yo);
            out[a] = NRM || N3 ? Ar::norm(sum) : sum;
            const T d = Ar::sub(ye, yo);
            const T dd = S > 0 ? d : Ar::neg(d);
            out[N - 1 - a] = NRM || N3 ? Ar::norm(dd) : dd;
        }
    } else if constexpr (std::is_same<Ar, ArF32>::value) {
        // FP32: the same pairing with FFMA2 (lane x even, lane y odd)
        float2 eo[H];
#pragma unroll
        for (int b = 0; b < H; ++b) eo[b] = make_float2(e[b], o[b]);
        float2 xm;
        if constexpr (N % 2 == 1) xm = make_float2(in[H], in[H]);
#pragma unroll
        for (int a = 0; a < H; ++a) {
            float2 y2 = __fmul2_rn(eo[0], M.P[a][0]);
#pragma unroll
            for (int b = 1; b < H; ++b) y2 = __ffma2_rn(eo[b], M.P[a][b], y2);
            if constexpr (N % 2 == 1) y2 = __ffma2_rn(xm, M.PM[a], y2);
            out[a] = y2.x + y2.y;
            const T d = y2.x - y2.y;
            out[N - 1 - a] = S > 0 ? d : -d;
        }
    } else {
#pragma unroll
        for (int a = 0; a < H; ++a) {
            T ye = Ar::mul(e[0], M.E[a][0]);
#pragma unroll
            for (int b = 1; b < H; ++b) Ar::mad(ye, e[b], M.E[a][b]);
            if constexpr (N % 2 == 1) Ar::mad(ye, in[H], M.Mid[a]);
            T yo = Ar::mul(o[0], M.O[a][0]);
#pragma unroll
            for (int b = 1; b < H; ++b) Ar::mad(yo, o[b], M.O[a][b]);
            out[a] = Ar::norm(Ar::add(ye, yo));
            const T d = Ar::sub(ye, yo);
            out[N - 1 - a] = Ar::norm(S > 0 ? d : Ar::neg(d));
        }
    }
    if constexpr (N % 2 == 1) {  // middle output: only the even (S = +1) or odd (S = -1) part
        if constexpr (S > 0) {
            T ye = Ar::mul(in[H], M.Mid[H]);
#pragma unroll
            for (int b = 0; b < H; ++b) Ar::mad(ye, e[b], M.E[H][b]);
            out[H] = NRM || N3 ? Ar::norm(ye) : ye;
        } else {
            T yo = Ar::mul(o[0], M.O[H][0]);
#pragma unroll
            for (int b = 1; b < H; ++b) Ar::mad(yo, o[b], M.O[H][b]);
            out[H] = NRM || N3 ? Ar::norm(yo) : yo;
        }
    }
}

// line contraction with B, B^T, D or D^T: even-odd form from N = 4 up (in double-float from N = 3), full
// form below
template <int N, class Ar, int WHICH, bool NRM = true>  // WHICH: 0 B, 1 B^T, 2 D, 3 D^T
__device__ __forceinline__ void sweep(const TabMetric<N, typename Ar::C> &tab, const typename Ar::T (&in)[N],
                                      typename Ar::T (&out)[N])
{
    if constexpr (N >= (std::is_same<Ar, ArDF>::value ? 3 : 4)) {
        if constexpr (WHICH == 0) contract_eo<N, 1, Ar, NRM>(tab.Bf, in, out);
        else if constexpr (WHICH == 1) contract_eo<N, 1, Ar, NRM>(tab.Bt, in, out);
        else if constexpr (WHICH == 2) contract_eo<N, -1, Ar, NRM>(tab.Df, in, out);
        else contract_eo<N, -1, Ar, NRM>(tab.Dt, in, out);
    } else {
        if constexpr (WHICH == 0) contract<N, false, Ar>(tab.B, in, out);
        else if constexpr (WHICH == 1) contract<N, true, Ar>(tab.B, in, out);
        else if constexpr (WHICH == 2) contract<N, false, Ar>(tab.D, in, out);
        else contract<N, true, Ar>(tab.D, in, out);
    }
}

// shared-memory line access: element m of the x-line, y-line or z-pencil owned by (ra, rb)
template <int N>
struct Lines {
    static constexpr int PI = N | 1;  // row pitch (odd)
    static constexpr int CS = PI * N * N;
    static __device__ __forceinline__ int x(int ra, int rb, int m) { return m + PI * (ra + N * rb); }
    static __device__ __forceinline__ int y(int ra, int rb, int m) { return ra + PI * (m + N * rb); }
    static __device__ __forceinline__ int z(int ra, int rb, int m) { return ra + PI * (rb + N * m); }
};

// ---- line buffers of the curved kernels (metric_tile)
// Element (i, j, k) of cell slot c sits at c*CS + i + PI*j + PP*k in each of the three buffers, and
// buffer R starts at element R*RS (RS: CPB*CS rounded up to 16 bytes, so that a bulk copy can land in
// buffer 1). A thread keeps the z-pencil (i, j) = (ra, rb) of its own cell in registers from one step
// to the next, and serves x-line (j, k) = (ra, rb) of its own cell where a step reads the input from
// memory or writes the output (coalesced global accesses). The other x-line steps and the y-line
// steps only load a line from shared memory, contract it and store it back, so any thread may serve
// any cell's line there: with `deal_x` / `deal_y` those lines are dealt to threads in the order of the
// shared-memory bank of their first element, round-robin over the warps, so that a warp touches
// distinct banks wherever the bank counts allow. The pitches come from an exhaustive search over
// (PI, PP, CS <= 1.6 n^3) that minimised the wavefronts of all line accesses of one apply (per
// element: 2 x-line accesses in thread order, 4 dealt, 8 y-line, 9 z-pencil) for 4-byte elements:
// at n = 5 and 8 cells per CTA 1105 instead of 1315 per tile (805 without any conflict). Dealing the
// global x-line steps as well cut more wavefronts but scattered the output stores over the tile's
// cells (2.4x the L2 store sectors) and was slower. Double-float and FP64 tiles (8-byte elements)
// keep odd row pitches with lines in thread order: their kernel is bound by the FP32 pipes, and 22 %
// fewer wavefronts changed nothing in its time.
//
// n = 4 and 8 in 4-byte elements: dense buffers with a swizzle instead of pitches. Element (i, j, k) of cell
// slot c sits at word D(c) ^ A(i) ^ B(j) ^ C(k) (tile_swz): the 16-byte chunks of an x-line keep their four
// elements together, and the chunk bits below 32 words are mixed so that in every warp the 32 x-lines (as
// 16-byte accesses, 8 lanes at a time), the 32 y-lines and the 32 z-pencils each cover all banks: no access of
// the apply has a conflict. With the pitches above (and dealt lines) an n = 4 apply took 1.54 shared-memory
// wavefronts per value (0.94 without conflicts) and kept the L1 data path 91 % busy.
__host__ __device__ constexpr bool tile_swizzled(int N, int ESZ, bool allow_remap)
{
    return allow_remap && ESZ == 4 && (N == 4 || N == 8);
}
template <int N>
struct TileSwz {  // N = 4: a warp holds two cells (c odd and even); N = 8: half a cell
    static __host__ __device__ constexpr int A(int i) { return i; }
    static __host__ __device__ constexpr int B(int j)
    {
        return N == 4 ? 4 * j : (4 * (j >> 2)) ^ (8 * (j & 3)) ^ (32 * (j >> 2));
    }
    static __host__ __device__ constexpr int C(int k)
    {
        return N == 4 ? (4 * (k >> 1)) ^ (16 * (k & 1)) ^ (32 * (k >> 1)) : (8 * (k & 3)) ^ (64 * k);
    }
    static __host__ __device__ constexpr int D(int c) { return N == 4 ? 64 * c ^ ((c & 1) ? 24 : 0) : 512 * c; }
};
// The two claims above, for every warp of a tile: the words are a permutation of the buffer with each 16-byte
// chunk of an x-line whole, and the accesses of 32 lanes (16-byte x accesses: of 8 lanes) cover every bank.
template <int N, int CPB>
constexpr bool tile_swz_ok()
{
    using Z = TileSwz<N>;
    constexpr int N2 = N * N, SIZE = CPB * N2 * N;
    bool seen[SIZE] = {};
    for (int e = 0; e < SIZE; ++e) {
        const int i = e % N, j = e / N % N, k = e / N2 % N, c = e / (N2 * N);
        const int x = Z::D(c) ^ Z::B(j) ^ Z::C(k), w = x ^ Z::A(i);
        if (w < 0 || w >= SIZE || seen[w] || w != (x ^ (i & ~3)) + (i & 3)) return false;
        seen[w] = true;
    }
    for (int t0 = 0; t0 < CPB * N2; t0 += 32)
        for (int m = 0; m < N; ++m) {
            unsigned x[4] = {}, y = 0, z = 0;  // banks (of 8 lanes: 16-byte groups of banks) touched
            for (int l = 0; l < 32; ++l) {
                const int c = (t0 + l) / N2, ra = (t0 + l) % N, rb = (t0 + l) / N % N;
                x[l / 8] |= 1u << ((Z::D(c) ^ Z::B(ra) ^ Z::C(rb) ^ (m & ~3)) / 4 % 8);
                y |= 1u << ((Z::D(c) ^ Z::A(ra) ^ Z::C(rb) ^ Z::B(m)) % 32);
                z |= 1u << ((Z::D(c) ^ Z::A(ra) ^ Z::B(rb) ^ Z::C(m)) % 32);
            }
            for (unsigned q : x)
                if (q != 0xffu) return false;
            if (y != 0xffffffffu || z != 0xffffffffu) return false;
        }
    return true;
}
struct TileGeom {
    int pi, pp, cs;  // row pitch, plane pitch, cell stride (elements)
    bool deal_x, deal_y;
};
__host__ __device__ constexpr TileGeom tile_geom(int N, int CPB, int ESZ, bool allow_remap)
{
    if (tile_swizzled(N, ESZ, allow_remap)) return {N, N * N, N * N * N, false, false};
    if (allow_remap && ESZ == 4) {
        switch (N * 1000 + CPB) {
        case 2016: case 2032: case 2064: return {2, 6, 12, false, true};
        case 3008: case 3016: case 3032: return {3, 10, 41, true, true};
        case 5004: case 5008: return {5, 33, 185, true, true};
        case 6002: case 6004: case 6008: return {6, 37, 228, true, true};
        case 7004: case 7008: return {7, 73, 529, true, true};
        default: break;
        }
    }
    return {N | 1, N * (N | 1), N * N * (N | 1), false, false};
}

template <int N, int CPB, int ESZ, bool REMAP>
struct TileLines {
    static constexpr TileGeom G = tile_geom(N, CPB, ESZ, REMAP);
    static constexpr int PI = G.pi, PP = G.pp, CS = G.cs;
    static constexpr int RS = (CPB * CS * ESZ + 15) / 16 * 16 / ESZ;  // buffer stride (elements)
    static_assert(PI >= N && PP >= N * PI && CS >= N * PP, "tile buffers overlap");
};

// in the shared-memory-only steps thread t serves x-line m[t] >> 16 and y-line m[t] & 0xffff; a line
// l = c N^2 + a + N b is cell slot c's x-line (j, k) = (a, b) or y-line (i, k) = (a, b)
template <int N, int CPB, int ESZ>
struct LineMap {
    uint32_t m[N * N * CPB];
};
template <int N, int CPB, int ESZ, bool REMAP>
constexpr LineMap<N, CPB, ESZ> make_line_map()
{
    constexpr TileGeom G = tile_geom(N, CPB, ESZ, REMAP);
    constexpr int T = N * N * CPB, N2 = N * N;
    constexpr int GRP = ESZ == 4 ? 32 : 16;  // lanes served by one wavefront = banks, in elements
    constexpr int NG = (T + GRP - 1) / GRP;
    LineMap<N, CPB, ESZ> r{};
    for (int dir = 0; dir < 2; ++dir) {
        int order[T] = {};
        int n = 0;
        for (int b = 0; b < GRP; ++b)
            for (int l = 0; l < T; ++l) {
                const int c = l / N2, a = l % N, bb = (l / N) % N;
                const int base = c * G.cs + (dir == 0 ? G.pi * a : a) + G.pp * bb;
                if (base % GRP == b) order[n++] = l;
            }
        n = 0;
        for (int lane = 0; lane < GRP; ++lane)
            for (int g = 0; g < NG; ++g) {
                const int t = g * GRP + lane;
                if (t >= T) continue;
                const uint32_t l = static_cast<uint32_t>((dir == 0 ? G.deal_x : G.deal_y) ? order[n++] : t);
                r.m[t] |= dir == 0 ? (l << 16) : l;
            }
    }
    return r;
}
template <int N, int CPB, int ESZ, bool REMAP>
constexpr bool line_map_is_bijection()
{
    constexpr LineMap<N, CPB, ESZ> M = make_line_map<N, CPB, ESZ, REMAP>();
    constexpr int T = N * N * CPB;
    bool seen_x[T] = {}, seen_y[T] = {};
    for (int t = 0; t < T; ++t) {
        const uint32_t lx = M.m[t] >> 16, ly = M.m[t] & 0xffffu;
        if (lx >= static_cast<uint32_t>(T) || ly >= static_cast<uint32_t>(T) || seen_x[lx] || seen_y[ly]) return false;
        seen_x[lx] = seen_y[ly] = true;
    }
    return true;
}
template <int N, int CPB, int ESZ, bool REMAP>
__device__ constexpr LineMap<N, CPB, ESZ> kLineMap = make_line_map<N, CPB, ESZ, REMAP>();

#define CW_LDX(s, v) _Pragma("unroll") for (int m_ = 0; m_ < N; ++m_) v[m_] = (s)[L::x(ra, rb, m_)]
#define CW_LDY(s, v) _Pragma("unroll") for (int m_ = 0; m_ < N; ++m_) v[m_] = (s)[L::y(ra, rb, m_)]
#define CW_LDZ(s, v) _Pragma("unroll") for (int m_ = 0; m_ < N; ++m_) v[m_] = (s)[L::z(ra, rb, m_)]
#define CW_STX(s, v) _Pragma("unroll") for (int m_ = 0; m_ < N; ++m_) (s)[L::x(ra, rb, m_)] = v[m_]
#define CW_STY(s, v) _Pragma("unroll") for (int m_ = 0; m_ < N; ++m_) (s)[L::y(ra, rb, m_)] = v[m_]
#define CW_STZ(s, v) _Pragma("unroll") for (int m_ = 0; m_ < N; ++m_) (s)[L::z(ra, rb, m_)] = v[m_]

// A thread's share of <x, A x>, accumulated in double-float. FP32 arithmetic: the products of two FP32 values
// have no low parts to carry (10 operations each instead of 12), and those of the x- and y-derivatives run as
// the two lanes of paired instructions with a sum of their own: 20 instructions per point instead of 36,
// beside about 100 for the operator.
struct DotAcc {
    df64 s{0.0f, 0.0f};
    float2 hi2 = make_float2(0.0f, 0.0f), lo2 = make_float2(0.0f, 0.0f);
};
__device__ __forceinline__ void dot_add(DotAcc &d, df64 a, df64 b) { df_mad(d.s, a, b); }
__device__ __forceinline__ void dot_add(DotAcc &d, float a, float b)
{
    const float p = __fmul_rn(a, b), e = __fmaf_rn(a, b, -p);
    float s, t;
    two_sum(d.s.hi, p, s, t);
    d.s.hi = s;
    d.s.lo = __fadd_rn(d.s.lo, __fadd_rn(t, e));
}
__device__ __forceinline__ void dot_add2(DotAcc &d, df64 a, df64 b, df64 a2, df64 b2)
{
    df_mad(d.s, a, b);
    df_mad(d.s, a2, b2);
}
__device__ __forceinline__ void dot_add2(DotAcc &d, float a, float b, float a2, float b2)
{
    const float2 x = make_float2(a, a2), y = make_float2(b, b2), p = __fmul2_rn(x, y);
    const float2 e = __ffma2_rn(x, y, neg2(p));
    float2 s, t;
    two_sum2(d.hi2, p, s, t);
    d.hi2 = s;
    d.lo2 = __fadd2_rn(d.lo2, __fadd2_rn(t, e));
}
__device__ __forceinline__ double dot_value(const DotAcc &d)
{
    df64 t = df_add(d.s, df64{d.hi2.x, d.lo2.x});
    return df_to_double(df_add(t, df64{d.hi2.y, d.lo2.y}));
}

// number of stored metric components per quadrature point for an operator kind
__host__ __device__ constexpr int metric_ncomp(int kind) { return kind == 1 ? 6 : (kind == 2 ? 1 : 7); }

// ------------------------------------------------------------------------ curved kernel ----
// geo layout: [cell][comp][qp] with qp = a + N(b + N c); comps (xx, yy, zz, xy, xz, yz, mass)
// for kind 3, the first six for kind 1, the mass coefficient alone for kind 2.
//
// STAGE: the CTA's input tile and metric tile are moved into shared memory by two 1D bulk copies
// issued at entry (x on barrier 0, metric on barrier 1), so the metric stream overlaps the
// interpolation and gradient sweeps. Tiles that cannot use a bulk copy (ragged last tile,
// misaligned span) and copies that do not complete within the wait bound are read with ordinary
// global loads instead.
// STAGE 0: direct loads; 1: x and metric tiles staged in shared memory by TMA; 2: x tile staged by
// TMA, metric tile prefetched into L2 by a bulk prefetch (a third of the shared memory of mode 1,
// so more CTAs per SM), then read with direct loads; 3: the metric tile in shared memory or on its way
// there (staged by the caller for several right-hand sides: gsm, gcs elements per cell; pb != nullptr: its copy
// completes a phase of *pb, waited for before the physics step), x read directly.
// PERSIST: the caller's CTAs work on one tile after another, on a barrier of their own (pb): an mbarrier must not
// be initialised again while it is live, so the caller initialises it once and passes each tile's state (st);
// in STAGE 2 pb is null for a tile that is not staged.
// Line buffers of metric_tile: three for 4-byte elements; two for 8-byte ones (double-float and FP64
// arithmetic), whose y-derivatives go back into buffer 0 after one more barrier: with the metric staged
// a CTA then needs 72 instead of 80 bytes of shared memory per value (K+M), which is one more CTA per SM
// at n = 5 and 8 (3 instead of 2). In modes 0 and 2, where shared memory is no limit, a third buffer in place of the
// barrier changed nothing (Q5, 3e7 values: 1120 / 1118 us in mode 0, 924 / 922 in mode 2; batches within 1 %).
template <class T>
constexpr int line_buffers()
{
    return sizeof(T) == 8 ? 2 : 3;
}

// Elements between the staged metrics of two cells beyond their own: at n = 4 in FP32 arithmetic the two cells
// of a warp read the same banks (a cell's metric is a multiple of 32 words), so each cell gets 64 bytes more
// and a bulk copy of its own.
template <int N, class T, class GS>
__host__ __device__ constexpr int metric_pad()
{
    return N == 4 && sizeof(T) == 4 ? 64 / (int)sizeof(GS) : 0;
}
// the bulk copies of a tile's metric (CPB cells of gc elements) into shared memory, by one thread
template <int CPB, int PAD, class GS>
__device__ __forceinline__ void metric_copy(GS *dst, const GS *src, int gc, uint64_t *bar)
{
    if constexpr (PAD == 0) {
        bulk_g2s(dst, src, CPB * gc * sizeof(GS), bar);
    } else {
#pragma unroll
        for (int c = 0; c < CPB; ++c) bulk_g2s(dst + c * (gc + PAD), src + c * gc, gc * sizeof(GS), bar);
    }
}

template <int N, int CPB, class T, class GS, bool REMAP = true>
__host__ __device__ constexpr size_t metric_smem_bytes(int nc, int stage)
{
    constexpr size_t lb = line_buffers<T>() * TileLines<N, CPB, sizeof(T), REMAP>::RS * sizeof(T);  // a multiple of 16
    const size_t metric = (CPB * (nc * N * N * N + metric_pad<N, T, GS>()) * sizeof(GS) + 15) / 16 * 16;
    return stage == 1 ? lb + metric + 16 : stage == 2 ? lb + 16 : lb;
}

// whether a whole tile of CPB cells can be moved by one bulk copy from vector x (16-byte alignment and size)
template <int N, int CPB, class VS>
__device__ __forceinline__ bool x_tile_stageable(const VS *x, int64_t cell0, int64_t ncells)
{
    return cell0 + CPB <= ncells && (CPB * N * N * N * sizeof(VS)) % 16 == 0 && aligned16(x + cell0 * (N * N * N));
}

// One tile of `cpt` consecutive cells starting at cell tile*cpt, worked by CPB cell slots of N*N
// threads (cpt <= CPB; slots c >= cpt compute on zeros and store nothing, so a CTA may have more
// threads than the tile needs). STAGE (see metric_smem_bytes; staging needs cpt == CPB).
// DOT: also accumulate this thread's share of <x, A x> into *dot, as the quadrature sum over its
// pencil of (grad u)^T G (grad u) + c u^2 (double-float accumulation): the same quadratic form as
// x^T A_e x cell by cell, read off the quadrature-point step with no extra memory traffic.
// asm_nx > 0 (the mesh's cells per x-row): the x pass of Algorithm struct_dss is applied to the
// x-interfaces between cells of this tile before the store (the two end values of each x-line are
// exchanged through shared memory and summed as that pass sums them); the interfaces between tiles
// are left to the DSS.
// RC: geo holds the trilinear coefficients (kTriCoef per cell) and the metric of every quadrature
// point is recomputed from them (Sec. 6: J, det J, J^-1 at the point), G = (w / det J) [c_a . c_b], applied
// without forming it: G g = (w / det J) c_a . (sum_b c_b g_b), with c_0 = J_eta x J_zeta, c_1 = J_zeta x J_xi,
// c_2 = J_xi x J_eta (the rows of det J J^-1), and the mass coefficient w det J.
// SMOOTH (Algorithm smoother_fused in one pass over the operator's output): y aliases x (= u, updated
// in place), and the stored value is u + D_hat (b - A u) (sb = b, sd = D_hat, cell-wise in the vector
// type), with the x-interfaces inside the tile averaged (the x pass of the averaging DSS:
// (left + right) / 2 to both copies; asm_nx must be the mesh's cells per x-row). Each thread re-reads
// u, b and D_hat on the x-line it stores, with plain loads (y aliases x). The operator output never
// reaches memory.
// An expired wait for a staged copy: record it in the device status word and wait once more (bounded)
// so that the copy is not left in flight. Out of line: the common path carries none of it.
static __device__ __noinline__ void wait_expired(unsigned *status, uint64_t *bar, uint32_t lim)
{
    if (status) atomicOr(status, kDevStatusTimeout);
    mbar_wait_bounded(bar, 0, lim);
}
// The same in a persistent CTA: a wait of some length continues here, up to the limit unless it is an injected
// stall; an expired one is recorded for the CTA's next tiles too.
__device__ __forceinline__ bool stage_wait_long(unsigned *status, StageBar *pb, unsigned st)
{
    const uint32_t phase = st & kTilePhase ? 1u : 0u;
    if (!(st & kTileStalled) && mbar_wait_bounded(&pb->bar, phase, kWaitLimit)) return true;
    if (status) atomicOr(status, kDevStatusTimeout);
    atomicOr(&pb->expired, 1u);
    mbar_wait_bounded(&pb->bar, phase, st & kTileStalled ? kWaitLimitInjected : kWaitLimit);
    return false;
}
static __device__ __noinline__ bool stage_wait_long_call(unsigned *status, StageBar *pb, unsigned st)
{
    return stage_wait_long(status, pb, st);
}
// Whether the long wait stands in the tile's code. The double-float tile is a function of its own, in the middle
// of which a call costs registers (n = 6: 128 instead of 103). In FP32, 8 right-hand sides, inline / call: Q3 40^3
// 158 / 153 us, Q1 64^3 132 / 124, but Q4 40^3 407 / 414 and, 16 of them, Q5 48^3 1932 / 1959.
template <int N, class Ar>
constexpr bool stage_wait_inline()
{
    return std::is_same<Ar, ArDF>::value || N == 5 || N == 6;
}
// Whether the copy behind a persistent CTA's barrier has arrived (bounded wait).
template <bool INL>
__device__ __forceinline__ bool stage_wait(unsigned *status, StageBar *pb, unsigned st)
{
    if (mbar_wait_bounded(&pb->bar, st & kTilePhase ? 1u : 0u, kWaitLimitInjected)) return true;
    if constexpr (INL) return stage_wait_long(status, pb, st);
    else return stage_wait_long_call(status, pb, st);
}

// Staged tiles and their waits: every wait for a bulk copy is bounded. A thread whose wait expired
// never reads the staged data (it takes zeros for the input tile, the global copy of the metric),
// records kDevStatusTimeout in *status (the operator's device status word, reported as
// CW_ERR_TIMEOUT by the next checking call: the outputs of that call are then undefined), and waits
// once more (bounded) so that the copy is not left in flight. Nothing runs on the common path beyond
// the wait itself: deciding the tile's fate block-wide (an early exit, or a flag read before the
// stores) made the common path 2-6 % slower in measurement. A persistent CTA, which has a barrier between its
// tiles and right-hand sides anyway, does decide block-wide there (StageBar::expired). dbg_extra > 0 (fault
// injection for tests) arms the input tile's barrier with dbg_extra bytes more than the copy delivers, so that
// its phase can never complete and the (then short) bounded wait runs out.
template <int N, int CPB, class Ar, class VS, class GS, int STAGE, bool DOT = false, bool RC = false,
          bool SMOOTH = false, bool REMAP = true, bool PERSIST = false>
__device__ __forceinline__ void metric_tile(const VS *x, VS *y, const GS *__restrict__ geo,
                                            int64_t ncells, int kind, const TabMetric<N, typename Ar::C> &tab,
                                            int64_t tile, int cpt, unsigned char *smem_raw, DotAcc *dot = nullptr,
                                            int asm_nx = 0, const VS *sb = nullptr, const VS *sd = nullptr,
                                            unsigned *status = nullptr, uint32_t dbg_extra = 0,
                                            StageBar *pb = nullptr, unsigned st = 0,
                                            const GS *gsm = nullptr, int gcs = 0)
{
    static_assert(!(RC && STAGE == 1), "recomputed geometry has no metric tile to stage");
    static_assert(PERSIST ? STAGE != 1 : STAGE != 3, "staging mode 3 is that of persistent callers");
    static_assert(!(PERSIST && (SMOOTH || DOT)), "persistent callers apply the operator alone");
    // Double-float renormalisation of the intermediate values: kept where the operator serves the
    // solver (DOT), whose attainable accuracy depends on it (at 128^3 Q3 the double-float CG took
    // 1351 instead of 1026 iterations without it); skipped in the plain apply (5 % faster there,
    // errors against the oracle <= 1.0e-13 instead of <= 3e-14).
    constexpr bool NRM = DOT;
    using T = typename Ar::T;
    using TL = TileLines<N, CPB, sizeof(T), REMAP>;
    static_assert(line_map_is_bijection<N, CPB, sizeof(T), REMAP>(), "every line has one thread");
    constexpr int N2 = N * N, N3 = N2 * N, PI = TL::PI, PP = TL::PP, CS = TL::CS, RS = TL::RS;
    constexpr int NB = line_buffers<T>(), YB = NB == 3 ? 2 : 0;  // YB: the buffer of the y-derivatives
    const bool HAS_K = (kind & 1) != 0, HAS_M = (kind & 2) != 0;
    const int NC = metric_ncomp(kind);
    T *S0 = reinterpret_cast<T *>(smem_raw);
    const int t = threadIdx.x;
    const int c = t / N2, r = t - c * N2, ra = r % N, rb = r / N;
    const int64_t cell0 = tile * cpt;
    const int64_t cell = cell0 + c;
    const bool act = c < cpt && cell < ncells;
    // offsets of the first elements of this thread's lines in a buffer: its own cell's x-line
    // (j, k) = (ra, rb) (xi, the steps that read or write memory) and z-pencil (i, j) = (ra, rb) (zo);
    // the dealt x-line (xo) and y-line (yo) of the shared-memory-only steps
    const int xi = c * CS + PI * ra + PP * rb;
    const int zo = c * CS + ra + PI * rb;
    int xo = xi, yo = c * CS + ra + PP * rb;
    if constexpr (TL::G.deal_x || TL::G.deal_y) {
        const uint32_t lm = kLineMap<N, CPB, sizeof(T), REMAP>.m[t];
        const int lx = static_cast<int>(lm >> 16), ly = static_cast<int>(lm & 0xffffu);
        const int xc = lx / N2, xr = lx - xc * N2, yc = ly / N2, yr = ly - yc * N2;
        xo = xc * CS + PI * (xr % N) + PP * (xr / N);
        yo = yc * CS + (yr % N) + PP * (yr / N);
    }

    // whole-line accesses of the input and output (LineVec) where they are wider than a value, but not at n = 6
    // in 8-byte vectors, where they cost the double-float kernel 6 % (Q5, 128e6 values: 33.3 -> 31.2 G values/s)
    constexpr bool WIDE = LineVec<N, VS>::WIDE && !(sizeof(VS) == 8 && N == 6);
    // Lines are loaded (stored) whole before (after) their conversion, also where they are moved value by value.
    // Not in the persistent tiles of n = 6 and 7, where the second copy of the line took the double-float function
    // from 96 to 128 registers (n = 6; 16 right-hand sides on Q5 48^3 12.4 -> 11.2 ms together with the
    // kernel's cap) and 178 to 128 (n = 7, 8 right-hand sides on Q6 24^3 1.58 -> 1.34 ms); at n = 5 it is faster with
    // whole lines (Q4 40^3 1.73 against 1.75 ms), and so is the per-operator kernel (64^3 Q4 718 against 770 us).
    constexpr bool LINES = WIDE || !PERSIST || N < 6;
    // load / store of a line of buffer R (0, 1, 2): x-line (own: the thread's own cell), y-line, z-pencil
    constexpr bool SW = tile_swizzled(N, sizeof(T), REMAP);
    if constexpr (SW) static_assert(tile_swz_ok<N, CPB>(), "swizzled buffers: every word once, no bank conflict");
    using Z = TileSwz<N>;
    [[maybe_unused]] const int sx = Z::D(c) ^ Z::B(ra) ^ Z::C(rb), sy = Z::D(c) ^ Z::A(ra) ^ Z::C(rb);
    [[maybe_unused]] const int sz = Z::D(c) ^ Z::A(ra) ^ Z::B(rb);
    auto ldx = [&](int R, bool own, T(&v)[N]) {
        const T *b = S0 + R * RS;
        if constexpr (SW) {
            T h[4];
#pragma unroll
            for (int m = 0; m < N; m += 4) {
                LineVec<4, T>::ld(b + (sx ^ m), h);
#pragma unroll
                for (int i = 0; i < 4; ++i) v[m + i] = h[i];
            }
        } else {
#pragma unroll
            for (int m = 0; m < N; ++m) v[m] = b[(own ? xi : xo) + m];
        }
    };
    auto stx = [&](int R, bool own, const T(&v)[N]) {
        T *b = S0 + R * RS;
        if constexpr (SW) {
#pragma unroll
            for (int m = 0; m < N; m += 4) {
                const T h[4] = {v[m], v[m + 1], v[m + 2], v[m + 3]};
                LineVec<4, T>::st(b + (sx ^ m), h);
            }
        } else {
#pragma unroll
            for (int m = 0; m < N; ++m) b[(own ? xi : xo) + m] = v[m];
        }
    };
    auto ldy = [&](int R, T(&v)[N]) {
#pragma unroll
        for (int m = 0; m < N; ++m) v[m] = S0[R * RS + (SW ? sy ^ Z::B(m) : yo + PI * m)];
    };
    auto sty = [&](int R, const T(&v)[N]) {
#pragma unroll
        for (int m = 0; m < N; ++m) S0[R * RS + (SW ? sy ^ Z::B(m) : yo + PI * m)] = v[m];
    };
    auto ldz = [&](int R, T(&v)[N]) {
#pragma unroll
        for (int m = 0; m < N; ++m) v[m] = S0[R * RS + (SW ? sz ^ Z::C(m) : zo + PP * m)];
    };
    auto stz = [&](int R, const T(&v)[N]) {
#pragma unroll
        for (int m = 0; m < N; ++m) S0[R * RS + (SW ? sz ^ Z::C(m) : zo + PP * m)] = v[m];
    };

    // ---- tile staging (single right-hand side)
    bool x_smem = false, g_smem = false, x_ok = true;
    const VS *xs = nullptr;
    const GS *gs = nullptr;
    uint64_t *bar = nullptr;
    [[maybe_unused]] const uint32_t lim = dbg_extra ? kWaitLimitInjected : kWaitLimit;
    if constexpr (STAGE == 1) {
        const size_t offg = NB * RS * sizeof(T);
        GS *sG = reinterpret_cast<GS *>(smem_raw + offg);
        constexpr int PAD = metric_pad<N, T, GS>();
        bar = reinterpret_cast<uint64_t *>(smem_raw + offg + (CPB * (NC * N3 + PAD) * sizeof(GS) + 15) / 16 * 16);
        VS *sX = reinterpret_cast<VS *>(S0 + RS);  // buffer 1 is free until the gradients
        const VS *xsrc = x + cell0 * N3;
        const GS *gsrc = geo + cell0 * NC * N3;
        const uint32_t xb = CPB * N3 * sizeof(VS), gb = CPB * NC * N3 * sizeof(GS);
        const bool ok = (cell0 + CPB <= ncells) && aligned16(xsrc) && aligned16(gsrc) && aligned16(sX) &&
                        aligned16(sG) && (xb % 16 == 0) && (gb % 16 == 0);
        if (ok) {  // block-uniform
            if (t == 0) {
                mbar_init(bar, 1);
                mbar_init(bar + 1, 1);
            }
            __syncthreads();
            if (t == 0) {
                mbar_expect_tx(bar, xb + dbg_extra);
                bulk_g2s(sX, xsrc, xb, bar);
                mbar_expect_tx(bar + 1, gb);
                metric_copy<CPB, PAD>(sG, gsrc, NC * N3, bar + 1);
            }
            x_ok = mbar_wait_bounded(bar, 0, lim);
            if (!x_ok) wait_expired(status, bar, lim);
            x_smem = true;
            xs = sX + c * N3;
            gs = sG + c * (NC * N3 + PAD);
            g_smem = true;  // its wait comes before the physics step
        }
    } else if constexpr (STAGE == 3) {
        // the caller passes this tile's metric (gsm): staged in shared memory, where one copy serves
        // several right-hand sides, or in global memory when it could not be staged (cell slots past
        // a ragged tile's end read slot 0's, in bounds, and store nothing)
        gs = gsm + (act ? c : 0) * gcs;
        g_smem = true;
    } else if constexpr (STAGE == 2) {
        bar = reinterpret_cast<uint64_t *>(smem_raw + NB * RS * sizeof(T));
        VS *sX = reinterpret_cast<VS *>(S0 + RS);
        const VS *xsrc = x + cell0 * N3;
        constexpr int GV = RC ? kTriCoef : 0;  // geometry values per cell (RC), else NC * N3
        const int gpc = RC ? GV : NC * N3;
        const GS *gsrc = geo + cell0 * gpc;
        const uint32_t xb = CPB * N3 * sizeof(VS), gb = CPB * gpc * sizeof(GS);
        static_assert(RS * sizeof(T) % 16 == 0, "the staged input tile starts on a 16-byte boundary");
        const bool full = cell0 + CPB <= ncells;
        const bool ok = PERSIST ? pb != nullptr : x_tile_stageable<N, CPB>(x, cell0, ncells);
        if (t == 0 && full && aligned16(gsrc) && (gb % 16 == 0)) bulk_prefetch_l2(gsrc, gb);
        if (ok) {  // block-uniform
            if constexpr (PERSIST) {
                bar = &pb->bar;
            } else {
                if (t == 0) mbar_init(bar, 1);
                __syncthreads();
            }
            if (t == 0) {
                mbar_expect_tx(bar, xb + (PERSIST ? (st & kTileStalled ? kStallBytes : 0u) : dbg_extra));
                bulk_g2s(sX, xsrc, xb, bar);
            }
            if constexpr (PERSIST) {
                x_ok = stage_wait<stage_wait_inline<N, Ar>()>(status, pb, st);
            } else {
                x_ok = mbar_wait_bounded(bar, 0, lim);
                if (!x_ok) wait_expired(status, bar, lim);
            }
            x_smem = true;
            xs = sX + c * N3;
        }
    }

    {
        T v[N], w[N], u[N], acc[N], gx[N], gy[N], gz[N];
        // (1) x-line (j,k) = (ra, rb): N contiguous values of the cell, contracted with B along x
        {
            const bool have = x_smem ? x_ok : act;  // a thread whose wait expired reads nothing staged
            if constexpr (LINES) {
                VS xl[N];
                if (x_smem) {
                    if (have) line_ld<N>(xs + N * r, xl, WIDE);
                } else if (act) {
                    const VS *xg = x + cell * N3 + N * r;
                    if (WIDE && LineVec<N, VS>::aligned(x)) {
                        LineVec<N, VS>::ld_nc(xg, xl);
                    } else {
#pragma unroll
                        for (int m = 0; m < N; ++m) xl[m] = ldg_nc(xg + m);
                    }
                }
#pragma unroll
                for (int m = 0; m < N; ++m) v[m] = have ? Ar::from(xl[m]) : Ar::zero();
            } else if (x_smem) {
#pragma unroll
                for (int m = 0; m < N; ++m) v[m] = have ? Ar::from(xs[N * r + m]) : Ar::zero();
            } else {
                const VS *xg = x + (act ? cell : 0) * N3 + N * r;
#pragma unroll
                for (int m = 0; m < N; ++m) v[m] = have ? Ar::from(ldg_nc(xg + m)) : Ar::zero();
            }
            sweep<N, Ar, 0, NRM>(tab, v, w);
            stx(0, true, w);
        }
        __syncthreads();
        // (2) y-line (i,k): contract with B along y, in place
        {
            ldy(0, v);
            sweep<N, Ar, 0, NRM>(tab, v, w);
            sty(0, w);
        }
        __syncthreads();
        // (3) z-pencil (i,j): contract with B along z -> u at the Gauss points (registers)
        {
            ldz(0, v);
            sweep<N, Ar, 0, NRM>(tab, v, u);
        }
        if (HAS_K) {
            {
                sweep<N, Ar, 2, NRM>(tab, u, gz);
                stz(0, u);
            }
            __syncthreads();
            // x- and y-derivatives by collocation, as line owners
            {
                ldx(0, false, v);
                sweep<N, Ar, 2, NRM>(tab, v, w);
                stx(1, false, w);
                ldy(0, v);
                sweep<N, Ar, 2, NRM>(tab, v, w);
                if constexpr (NB == 2) __syncthreads();  // every line of buffer 0 has been read
                sty(YB, w);
            }
            __syncthreads();
            {
                ldz(1, gx);
                ldz(YB, gy);
            }
        }
        // the metric tile's wait (a thread whose wait expired reads the metric from global memory)
        bool g_ok = true;
        if constexpr (STAGE == 1) {
            if (g_smem) {
                g_ok = mbar_wait_bounded(bar + 1, 0, lim);
                if (!g_ok) wait_expired(status, bar + 1, lim);
            }
        } else if constexpr (STAGE == 3) {
            if (pb)  // block-uniform
                g_ok = stage_wait<stage_wait_inline<N, Ar>()>(status, pb, st);
        }
        // (4) quadrature-point physics on the owned pencil, qp = (ra, rb, k)
        {
            const GS *gc = (g_smem && g_ok) ? gs + r
                                            : geo + (act ? cell : 0) * (RC ? kTriCoef : NC * N3) + (RC ? 0 : r);
            // RC: the pencil's Jacobian columns as J_xi = P0 + zeta P1, J_eta = Q0 + zeta Q1, J_zeta = Z
            T P0[3], P1[3], Q0[3], Q1[3], Z[3], wab;
            if constexpr (RC) {
                T xi = tab.xq[0], eta = tab.xq[0], wa = tab.wq[0], wb = tab.wq[0];
#pragma unroll
                for (int m = 1; m < N; ++m) {
                    if (ra == m) xi = tab.xq[m], wa = tab.wq[m];
                    if (rb == m) eta = tab.xq[m], wb = tab.wq[m];
                }
                wab = Ar::norm(Ar::mul(wa, wb));
                const T xe = Ar::norm(Ar::mul(xi, eta));
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    const T a1 = Ar::from(gc[0 + d]), a2 = Ar::from(gc[3 + d]), a3 = Ar::from(gc[6 + d]);
                    const T a4 = Ar::from(gc[9 + d]), a5 = Ar::from(gc[12 + d]), a6 = Ar::from(gc[15 + d]);
                    const T a7 = Ar::from(gc[18 + d]);
                    T t = a1;
                    Ar::mad(t, a4, eta);
                    P0[d] = Ar::norm(t);
                    t = a5;
                    Ar::mad(t, a7, eta);
                    P1[d] = Ar::norm(t);
                    t = a2;
                    Ar::mad(t, a4, xi);
                    Q0[d] = Ar::norm(t);
                    t = a6;
                    Ar::mad(t, a7, xi);
                    Q1[d] = Ar::norm(t);
                    t = a3;
                    Ar::mad(t, a5, xi);
                    Ar::mad(t, a6, eta);
                    Ar::mad(t, a7, xe);
                    Z[d] = Ar::norm(t);
                }
            }
#pragma unroll
            for (int k = 0; k < N; ++k) {
                const GS *g = gc + N2 * k;
                T gxx, gyy, gzz, gxy, gxz, gyz, cmr, hx, hy, hz;
                if constexpr (RC) {
                    const T zeta = tab.xq[k];
                    T jx[3], jy[3];
#pragma unroll
                    for (int d = 0; d < 3; ++d) {
                        T t = P0[d];
                        Ar::mad(t, P1[d], zeta);
                        jx[d] = Ar::norm(t);
                        t = Q0[d];
                        Ar::mad(t, Q1[d], zeta);
                        jy[d] = Ar::norm(t);
                    }
                    auto cross = [](const T (&a)[3], const T (&b)[3], T (&c)[3]) {
#pragma unroll
                        for (int d = 0; d < 3; ++d) {
                            const int d1 = (d + 1) % 3, d2 = (d + 2) % 3;
                            T t = Ar::mul(a[d1], b[d2]);
                            Ar::mad(t, Ar::neg(a[d2]), b[d1]);
                            c[d] = Ar::norm(t);
                        }
                    };
                    auto dot3 = [](const T (&a)[3], const T (&b)[3]) {
                        T t = Ar::mul(a[0], b[0]);
                        Ar::mad(t, a[1], b[1]);
                        Ar::mad(t, a[2], b[2]);
                        return Ar::norm(t);
                    };
                    T c0[3], c1[3], c2[3];
                    cross(jy, Z, c0);
                    cross(Z, jx, c1);
                    cross(jx, jy, c2);
                    const T det = dot3(jx, c0);
                    const T w = Ar::norm(Ar::mul(wab, tab.wq[k]));
                    cmr = Ar::norm(Ar::mul(w, det));
                    if (HAS_K) {
                        // h_a = (w / det J) c_a . v with v = sum_b c_b g_b: 18 multiply-adds and 3 scalings
                        // where forming G first takes 27 and 6 (41x40x39 Q4 K+M 449 -> 419 us, error 2.8e-14 ->
                        // 1.8e-14)
                        const T sc = Ar::div(w, det);
                        T vv[3];
#pragma unroll
                        for (int d = 0; d < 3; ++d) {
                            T t = Ar::mul(c0[d], gx[k]);
                            Ar::mad(t, c1[d], gy[k]);
                            Ar::mad(t, c2[d], gz[k]);
                            vv[d] = Ar::norm(Ar::mul(sc, Ar::norm(t)));
                        }
                        hx = dot3(c0, vv);
                        hy = dot3(c1, vv);
                        hz = dot3(c2, vv);
                    }
                }
                if (HAS_K) {
                    if constexpr (!RC) {
                        gxx = Ar::from(g[0 * N3]), gyy = Ar::from(g[1 * N3]);
                        gzz = Ar::from(g[2 * N3]), gxy = Ar::from(g[3 * N3]);
                        gxz = Ar::from(g[4 * N3]), gyz = Ar::from(g[5 * N3]);
                    }
                    if constexpr (!RC) {
                        hx = Ar::mul(gx[k], gxx), hy = Ar::mul(gx[k], gxy), hz = Ar::mul(gx[k], gxz);
                        Ar::mad(hx, gy[k], gxy);
                        Ar::mad(hy, gy[k], gyy);
                        Ar::mad(hz, gy[k], gyz);
                        Ar::mad(hx, gz[k], gxz);
                        Ar::mad(hy, gz[k], gyz);
                        Ar::mad(hz, gz[k], gzz);
                    }
                    if constexpr (DOT) {  // (grad u)^T G (grad u) at this point
                        dot_add2(*dot, gx[k], hx, gy[k], hy);
                        dot_add(*dot, gz[k], hz);
                    }
                    gx[k] = NRM ? Ar::norm(hx) : hx;
                    gy[k] = NRM ? Ar::norm(hy) : hy;
                    gz[k] = NRM ? Ar::norm(hz) : hz;
                }
                if (HAS_M) {
                    if constexpr (!RC) cmr = Ar::from(g[(NC - 1) * N3]);
                    const T cm = cmr;
                    acc[k] = NRM ? Ar::norm(Ar::mul(u[k], cm)) : Ar::mul(u[k], cm);
                    if constexpr (DOT) dot_add(*dot, u[k], acc[k]);  // c u^2
                }
            }
        }
        if (HAS_K) {
            // z-part of the transposed derivative in registers, x/y parts as line owners
            {
                sweep<N, Ar, 3, NRM>(tab, gz, v);
#pragma unroll
                for (int k = 0; k < N; ++k) acc[k] = HAS_M ? Ar::add(acc[k], v[k]) : v[k];
                stz(1, gx);  // own pencil only: no other thread reads these pencils now
                stz(YB, gy);
            }
            __syncthreads();
            {
                ldx(1, false, v);
                sweep<N, Ar, 3, NRM>(tab, v, w);
                stx(1, false, w);
                ldy(YB, v);
                sweep<N, Ar, 3, NRM>(tab, v, w);
                sty(YB, w);
            }
            __syncthreads();
            {
                ldz(1, v);
                ldz(YB, w);
#pragma unroll
                for (int k = 0; k < N; ++k) {
                    const T t = Ar::add(acc[k], Ar::add(v[k], w[k]));
                    acc[k] = NRM ? Ar::norm(t) : t;
                }
            }
        }
        // (5) integrate back: B^T along z (registers), y and x as line owners
        {
            sweep<N, Ar, 1, NRM>(tab, acc, w);
            stz(0, w);
        }
        __syncthreads();
        {
            ldy(0, v);
            sweep<N, Ar, 1, NRM>(tab, v, w);
            sty(0, w);
        }
        __syncthreads();
        {
            ldx(0, true, v);
            sweep<N, Ar, 1, NRM>(tab, v, w);
            const int64_t o = (act ? cell : 0) * N3 + N * r;
            if constexpr (!LINES) {  // (persistent callers neither assemble nor smooth)
                if (act) {
#pragma unroll
                    for (int m = 0; m < N; ++m) Ar::to(y[o + m], w[m]);
                }
            } else {
                VS nv[N];  // the values to store
                const bool yvec = WIDE && LineVec<N, VS>::aligned(y);
#pragma unroll
                for (int m = 0; m < N; ++m) Ar::to(nv[m], w[m]);
                if constexpr (SMOOTH) {
                    if (act) {  // (an idle slot must not read u of cell 0, which another CTA updates)
                        VS yl[N], bl[N], dl[N];
                        line_ld<N>(y + o, yl, yvec);
                        line_ld<N>(sb + o, bl, LineVec<N, VS>::aligned(sb));
                        line_ld<N>(sd + o, dl, LineVec<N, VS>::aligned(sd));
#pragma unroll
                        for (int m = 0; m < N; ++m) nv[m] = yl[m] + dl[m] * (bl[m] - nv[m]);
                    }
                }
                if (SMOOTH || asm_nx > 0) {  // kernel-uniform: the x-interfaces inside the tile
                    // buffer 1 is free: its last reads precede the first barrier of step (5)
                    VS *exl = reinterpret_cast<VS *>(S0 + RS), *exr = exl + CPB * N2;
                    exl[c * N2 + r] = nv[0];
                    exr[c * N2 + r] = nv[N - 1];
                    __syncthreads();
                    if (act) {
                        const int64_t ix = cell % asm_nx;
                        if (c + 1 < cpt && cell + 1 < ncells && ix + 1 < asm_nx) {
                            nv[N - 1] = AddOp<VS>::add(nv[N - 1], exl[(c + 1) * N2 + r]);
                            if constexpr (SMOOTH) nv[N - 1] = nv[N - 1] * VS(0.5);
                        }
                        if (c > 0 && ix > 0) {
                            nv[0] = AddOp<VS>::add(exr[(c - 1) * N2 + r], nv[0]);
                            if constexpr (SMOOTH) nv[0] = nv[0] * VS(0.5);
                        }
                    }
                }
                if (act) line_st<N>(y + o, nv, yvec);
            }
        }
    }
}

// Register caps for the double-float kernels (as CTAs per SM for the launch bounds): stored metric
// at n = 5 to 72 registers, which it fits without spilling, so that 4 CTAs of 200 threads fit per
// SM in staging modes 0 and 2 (left alone the allocator takes 78 and loses one; in mode 1, where it starts, shared
// memory allows 3 either way); recomputed geometry to 128 (2 CTAs at n = 5 instead of 1). Other n keep the plain
// kernel: larger n spill under a 72 cap, smaller n already fit and ran slower with the hint (a minimum-blocks hint
// is not neutral, even a hint of 1).
template <class Ar, int N, bool RC>
constexpr bool df_capped()
{
    return std::is_same<Ar, ArDF>::value && (RC || N == 5);
}
template <int THREADS, bool RC>
constexpr int df_min_blocks()
{
    constexpr int warps = (THREADS + 31) / 32;
    constexpr int b = 65536 / (warps * 32 * (RC ? 128 : 72));
    return b > 0 ? b : 1;
}

template <int N, int CPB, class Ar, class VS, class GS, int STAGE, bool RC = false>
__global__ void __launch_bounds__(N *N *CPB) apply_metric_kernel(const VS *__restrict__ x, VS *__restrict__ y,
                                                                  const GS *__restrict__ geo, int64_t ncells,
                                                                  int kind, TabMetric<N, typename Ar::C> tab,
                                                                  int asm_nx, unsigned *status, uint32_t dbg_extra)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    metric_tile<N, CPB, Ar, VS, GS, STAGE, false, RC>(x, y, geo, ncells, kind, tab, blockIdx.x, CPB, smem_raw, nullptr,
                                                      asm_nx, nullptr, nullptr, status, dbg_extra);
}

template <int N, int CPB, class Ar, class VS, class GS, int STAGE, bool RC = false>
__global__ void __launch_bounds__(N *N *CPB, (df_min_blocks<N * N * CPB, RC>()))
    apply_metric_kernel_capped(const VS *__restrict__ x, VS *__restrict__ y, const GS *__restrict__ geo,
                               int64_t ncells, int kind, TabMetric<N, typename Ar::C> tab, int asm_nx,
                               unsigned *status, uint32_t dbg_extra)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    metric_tile<N, CPB, Ar, VS, GS, STAGE, false, RC>(x, y, geo, ncells, kind, tab, blockIdx.x, CPB, smem_raw, nullptr,
                                                      asm_nx, nullptr, nullptr, status, dbg_extra);
}

// Several operators of one degree, kind and precision in one launch (the blocks of a multi-block mesh, each
// too small to fill the GPU): CTA blockIdx.x works on tile blockIdx.x - tile0 of the last operator of the
// table with tile0 <= blockIdx.x. x and y are the concatenated vectors.
struct MultiOp {
    int64_t off, ncells;
    const void *geo;
    unsigned *status;
    unsigned tile0;
    int asm_nx;
    uint32_t dbg_extra;
};
constexpr int kMultiOps = 16;  // operators per launch (the table is a kernel parameter)
struct MultiOps {
    MultiOp o[kMultiOps];
    int count;
};
template <int N, int CPB, class Ar, class VS, class GS, int STAGE>
__global__ void __launch_bounds__(N *N *CPB, (df_capped<Ar, N, false>() ? df_min_blocks<N * N * CPB, false>() : 0))
    apply_multi_kernel(const VS *__restrict__ x, VS *__restrict__ y, int kind, TabMetric<N, typename Ar::C> tab,
                       const __grid_constant__ MultiOps ops)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int b = 0;
    while (b + 1 < ops.count && ops.o[b + 1].tile0 <= blockIdx.x) ++b;
    const MultiOp &o = ops.o[b];
    metric_tile<N, CPB, Ar, VS, GS, STAGE>(x + o.off, y + o.off, static_cast<const GS *>(o.geo), o.ncells, kind, tab,
                                           blockIdx.x - o.tile0, CPB, smem_raw, nullptr, o.asm_nx, nullptr, nullptr,
                                           o.status, o.dbg_extra);
}

// y = A x and the CTA's partial of <x, A x> in part[blockIdx.x] (deterministic: fixed order in a CTA). The
// threads' sums go through shared memory to one warp: 9 FP64 additions of a warp per 128 threads, each 16
// cycles of the SM's FP64 pipe, where shuffles in every warp took 23 (14 us of FP64 pipe per launch of 13824
// CTAs beside a kernel of 47 us). FP32 at n = 4: capped to the registers of the plain apply, which the
// shared memory lets run in 11 CTAs per SM.
template <class Ar, int N, bool RC>
constexpr int dot_min_blocks()
{
    return std::is_same<Ar, ArF32>::value && N == 4 && !RC ? 11 : 0;
}
template <int N, int CPB, class Ar, class VS, class GS, int STAGE, bool RC = false>
__global__ void __launch_bounds__(N *N *CPB, (dot_min_blocks<Ar, N, RC>()))
    apply_metric_dot_kernel(const VS *__restrict__ x, VS *__restrict__ y, const GS *__restrict__ geo, int64_t ncells,
                            int kind, TabMetric<N, typename Ar::C> tab, double *__restrict__ part, unsigned *status,
                            uint32_t dbg_extra)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    DotAcc acc;
    metric_tile<N, CPB, Ar, VS, GS, STAGE, true, RC>(x, y, geo, ncells, kind, tab, blockIdx.x, CPB, smem_raw, &acc, 0,
                                                     nullptr, nullptr, status, dbg_extra);
    constexpr int T = N * N * CPB;
    static_assert(T >= 32, "one whole warp sums");
    double *sh = reinterpret_cast<double *>(smem_raw);  // the line buffers (at least 8 N^3 CPB bytes)
    __syncthreads();                                    // whose last lines have been read
    sh[threadIdx.x] = dot_value(acc);
    __syncthreads();
    if (threadIdx.x < 32) {
        double v = sh[threadIdx.x];
        for (int i = threadIdx.x + 32; i < T; i += 32) v += sh[i];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (threadIdx.x == 0) part[blockIdx.x] = v;
    }
}

// One fused smoothing sweep on a tile (see SMOOTH in metric_tile): u <- x-average(u + D_hat (b - A u)),
// in place; the x pass between tiles and the y and z passes of the averaging DSS follow.
template <int N, int CPB, class Ar, class VS, class GS, int STAGE, bool RC = false>
__global__ void __launch_bounds__(N *N *CPB) smooth_metric_kernel(VS *u, const VS *__restrict__ b,
                                                                   const VS *__restrict__ dhat,
                                                                   const GS *__restrict__ geo, int64_t ncells,
                                                                   int kind, TabMetric<N, typename Ar::C> tab,
                                                                   int asm_nx, unsigned *status, uint32_t dbg_extra)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    metric_tile<N, CPB, Ar, VS, GS, STAGE, false, RC, true>(u, u, geo, ncells, kind, tab, blockIdx.x, CPB, smem_raw,
                                                            nullptr, asm_nx, b, dhat, status, dbg_extra);
}

// ---------------------------------------------------------------------- Cartesian kernel ----
// geo layout: [cell][4] doubles (a_x, a_y, a_z, a_m) = (hy hz/hx, hx hz/hy, hx hy/hz, hx hy hz),
// already multiplied by the kind mask (a_m = 0 for kind 1, a_x = a_y = a_z = 0 for kind 2).
template <int N, int CPB, class Ar, class VS>
__global__ void __launch_bounds__(N *N *CPB) apply_affine_kernel(const VS *__restrict__ x, VS *__restrict__ y,
                                                                  const double *__restrict__ geo, int64_t ncells,
                                                                  int kind, TabAffine<N, typename Ar::C> tab)
{
    using T = typename Ar::T;
    using L = Lines<N>;
    constexpr int N2 = N * N, N3 = N2 * N, CS = L::CS;
    const bool HAS_K = (kind & 1) != 0, HAS_M = (kind & 2) != 0;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *S0 = reinterpret_cast<T *>(smem_raw);
    const int t = threadIdx.x, c = t / N2, r = t - c * N2, ra = r % N, rb = r / N;
    const int64_t cell = static_cast<int64_t>(blockIdx.x) * CPB + c;
    const bool act = cell < ncells;
    T *s0 = S0 + c * CS;
    T *s1 = S0 + (CPB + c) * CS;
    T v[N], P[N], Q[N];
    // x-line: P = M_x u, Q = K_x u
    {
        // (whole-line loads were 6-8 % slower here)
        const VS *xc = x + (act ? cell : 0) * N3 + N * r;
#pragma unroll
        for (int m = 0; m < N; ++m) v[m] = act ? Ar::from(ldg_nc(xc + m)) : Ar::zero();
        contract<N, false, Ar>(tab.M, v, P);
        CW_STX(s0, P);
        if (HAS_K) {
            contract<N, false, Ar>(tab.K, v, Q);
            CW_STX(s1, Q);
        }
    }
    const double *gc = geo + (act ? cell : 0) * 4;
    const T ax = Ar::from(__ldg(gc + 0)), ay = Ar::from(__ldg(gc + 1));
    const T az = Ar::from(__ldg(gc + 2)), am = Ar::from(__ldg(gc + 3));
    __syncthreads();
    // y-line: R1 = M_y P, R2 = K_y P, R3 = M_y Q; W = a_x R3 + a_y R2 + a_m R1
    {
        T R1[N], W[N];
        CW_LDY(s0, v);
        contract<N, false, Ar>(tab.M, v, R1);
        if (HAS_K) {
            T R2[N], R3[N];
            contract<N, false, Ar>(tab.K, v, R2);
            CW_LDY(s1, v);
            contract<N, false, Ar>(tab.M, v, R3);
#pragma unroll
            for (int m = 0; m < N; ++m) {
                T s = Ar::mul(R3[m], ax);
                Ar::mad(s, R2[m], ay);
                if (HAS_M) Ar::mad(s, R1[m], am);
                W[m] = Ar::norm(s);
                R1[m] = Ar::norm(Ar::mul(R1[m], az));
            }
            CW_STY(s1, R1);
        } else {
#pragma unroll
            for (int m = 0; m < N; ++m) W[m] = Ar::norm(Ar::mul(R1[m], am));
        }
        CW_STY(s0, W);
    }
    __syncthreads();
    // z-pencil: y = M_z W + K_z (a_z R1)
    {
        T out[N];
        CW_LDZ(s0, v);
        contract<N, false, Ar>(tab.M, v, out);
        if (HAS_K) {
            T R[N], KR[N];
            CW_LDZ(s1, R);
            contract<N, false, Ar>(tab.K, R, KR);
#pragma unroll
            for (int m = 0; m < N; ++m) out[m] = Ar::norm(Ar::add(out[m], KR[m]));
        }
        if (act) {
            VS *yc = y + cell * N3 + r;
#pragma unroll
            for (int m = 0; m < N; ++m) Ar::to(yc[N2 * m], out[m]);
        }
    }
}

}  // namespace cw

// pkr_sweep.cuh -- the fused stream-and-collide sweep (one time step of the
// high-order kinetic relaxation scheme) as a templated CUDA kernel.
//
// One launch performs, at every site x of the periodic grid:
//   pull-stream   g_i(x) = A_i(x - v_i)                       (all Q velocities)
//   density       Phi(x) = sum_i g_i(x)
//   BGK + source  B_i(x) = (1 - w) g_i(x) + w phi_i Phi(x) + chi_i S(x)
// and, on residual sweeps, compares Phi with the previous step's Phi and
// emits per-block partial sums of |dPhi|^2, |Phi|^2 and max |dPhi|.
//
// Work decomposition.  Sites are taken in the flat order (z*ny + y)*nx + x in
// tiles of 32; one warp owns a tile and all Q velocities of it (one lane per
// site).  Blocks are persistent and stride over the tiles.  Every velocity
// component is a compile-time constant, so the pull address of a velocity is
// two integer adds on per-tile wrapped row/column offsets.  Plane i of an
// array lives at i*V.
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <type_traits>

#include "pkr_internal.h"

namespace pkr {

template <class L>
__host__ __device__ constexpr int vx_of(int i) { return L::T.v[i].x; }
template <class L>
__host__ __device__ constexpr int vy_of(int i) { return L::T.v[i].y; }
template <class L>
__host__ __device__ constexpr int vz_of(int i) { return L::T.v[i].z; }
template <class L>
__host__ __device__ constexpr int cls_of(int i) { return L::T.cls[i]; }
template <class L>
__host__ __device__ constexpr int reach_of() { return L::T.reach; }
template <class L>
__host__ __device__ constexpr int ncls_of() { return L::T.ncls; }
// First velocity of symmetry class c (Q for c = ncls).
template <class L>
__host__ __device__ constexpr int cls_begin(int c)
{
    for (int i = 0; i < L::Q; ++i)
        if (L::T.cls[i] == c) return i;
    return L::Q;
}

template <int I, int N, typename F>
__host__ __device__ __forceinline__ void static_for(F&& f)
{
    if constexpr (I < N) {
        f(std::integral_constant<int, I>{});
        static_for<I + 1, N>(f);
    }
}

template <typename T> struct AccType { using type = T; };
template <> struct AccType<long long> { using type = double; };
// Type of the stored source: binary64 for fixed-point populations.
template <typename T> struct SrcType { using type = T; };
template <> struct SrcType<long long> { using type = double; };

__device__ __forceinline__ int wrap_near(int c, int n)
{
    c = c < 0 ? c + n : c;
    return c >= n ? c - n : c;
}
// c - D wrapped into [0, n) for c in [0, n) and |D| <= n: only one side can
// be crossed, and which one is known at compile time.
template <int D>
__device__ __forceinline__ int wrap_off(int c, int n)
{
    const int v = c - D;
    if constexpr (D > 0) return v < 0 ? v + n : v;
    else if constexpr (D < 0) return v >= n ? v - n : v;
    else return v;
}
__device__ __forceinline__ int wrap_any(int c, int n)
{
    int r = c % n;
    return r < 0 ? r + n : r;
}

__device__ __forceinline__ void store_stream(double* p, double v) { __stcs(p, v); }
__device__ __forceinline__ void store_stream(float* p, float v) { __stcs(p, v); }
__device__ __forceinline__ void store_stream(long long* p, long long v) { __stcs(p, v); }

// ---------------------------------------------------------------------------
// Staged sweep: one warp owns a tile of 32 consecutive sites and all Q
// velocities.  The Q pulled values of the tile are copied global -> shared
// with per-lane asynchronous copies (cp.async, zero-fill for lanes past the
// end and for the first step), so a warp keeps Q x 256 bytes in flight
// without spending registers on them.  Each lane then reads back only its own
// column: no block barrier is needed.  The density is the exact sum above;
// the equilibrium-plus-source term is formed once per symmetry class.
// ---------------------------------------------------------------------------
template <int BYTES>
__device__ __forceinline__ void cp_async(uint32_t dst, const void* src, int src_bytes)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;\n" ::"r"(dst), "l"(src),
                 "n"(BYTES), "r"(src_bytes)
                 : "memory");
}
__device__ __forceinline__ void cp_async_wait_all()
{
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
}
// The copies issued since the last commit form one group.
__device__ __forceinline__ void cp_async_commit()
{
    asm volatile("cp.async.commit_group;\n" ::: "memory");
}
// Every committed group but the most recent one has landed.
__device__ __forceinline__ void cp_async_wait_all_but_last()
{
    asm volatile("cp.async.wait_group 1;\n" ::: "memory");
}
// Every committed group has landed.
__device__ __forceinline__ void cp_async_wait_committed()
{
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
}

// A sweep kernel's dynamic shared memory.  The split of each SM's L1/shared
// array is left to the CUDA driver, which takes the smallest shared part that
// holds the kernel's full occupancy: the rest stays L1, where the 4- and
// 8-byte asynchronous copies of the pull land on their way to shared memory.
// Forcing the largest shared part (228 KB, 28 KB of L1) measured 19% slower
// for the staged sweep at 256^3 in 64-bit fixed point, whose three blocks
// (60.5 KB each) fit the 196 KB split with 60 KB of L1.
template <typename K>
cudaError_t set_sweep_smem(K kern, size_t smem)
{
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}

// Launch geometry of the staged sweep.  A tile's Q velocities are split
// among G warps (velocity groups): splitting cuts the shared memory a warp
// stages by G and so lets an SM hold more warps, at the price of two
// named-barrier meetings per tile.  A block carries TILES tiles.  Several
// (G, TILES) variants are compiled per lattice and storage type; a plan picks
// one (default table below, or pkr_plan_autotune).
template <class L, typename T, int G_, int TILES_>
struct Staged {
    static constexpr int Q = L::Q;
    static constexpr int G = G_;
    static constexpr int TILES = TILES_;
    static constexpr int WARPS = G * TILES;
    static constexpr int CH = (Q + G - 1) / G;     // most velocities a warp stages
    static constexpr size_t smem_bytes() { return (size_t)WARPS * CH * 32 * sizeof(T); }
    static constexpr int lo(int g) { return g * Q / G; }
};

// Variant list: (G, TILES) pairs.  Small sets are never split.
struct Geo {
    int G, TILES;
};
template <class L>
struct Variants {
    static constexpr int N = (L::Q > 64) ? 6 : 2;
    static constexpr Geo at(int k)
    {
        if (L::Q > 64) {
            constexpr Geo big[6] = {{1, 2}, {2, 1}, {2, 2}, {3, 1}, {3, 2}, {4, 1}};
            return big[k];
        }
        constexpr Geo small[2] = {{1, 2}, {1, 4}};
        return small[k];
    }
};

// Density of one site from its Q pulled values in shared memory (stride 32)
// without binary64 additions.  The values are aligned to the largest
// exponent E among them in a 64-bit two's-complement fixed-point sum whose
// unit is 2^(E - 1075 - GB), i.e. GB guard bits below the last place of the
// largest value (GB = 63 - 53 - ceil(log2 Q) leaves room for Q terms).  Each
// term is rounded to that unit (error <= 2^-(GB+1) ulp of the largest value,
// below the half-ulp that every plain binary64 addition may lose), the sum is
// exact, and one conversion plus one exact power-of-two scaling return it to
// binary64.  On this GPU the FP64 pipe issues about two operations per clock
// per SM, so this costs two of its slots per site instead of Q - 1.  Inf/NaN
// inputs, or values all below 2^-1011, take the plain binary64 path.
__host__ __device__ constexpr int ceil_log2(int q)
{
    int r = 0;
    while ((1 << r) < q) ++r;
    return r;
}

// Shared-memory loads issued as volatile asm: a batch of them can go out
// back to back, and the compiler cannot hoist all Q of them into registers.
__device__ __forceinline__ double lds_f64(uint32_t addr)
{
    double v;
    asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ int lds_hi32(uint32_t addr)
{
    int v;
    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(addr + 4));
    return v;
}
__device__ __forceinline__ float lds_f32(uint32_t addr)
{
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr));
    return v;
}

// One term of the fixed-point density at twice its resolution: t = floor(2y)
// for y = v / 2^(emax - 1075 - GB), the mantissa shifted right as a magnitude
// and the sign applied by complement afterwards (for arithmetic shifts
// ~(x >> r) == (~x) >> r, so a negative term becomes floor(2y - 2^-r), which
// moves only exact ties).  floor((t + 1) / 2) = (t + (t & 1)) / 2 is then y
// rounded to the nearest integer, ties away from zero.  A shift of 54 + GB or
// more (zero, subnormal or negligible values) leaves 0 or -1, i.e. a rounded 0.
template <int GB>
__device__ __forceinline__ long long fixed_term2(double v, int emax)
{
    const long long b = __double_as_longlong(v);
    const int hi = (int)(b >> 32);
    const int e = (hi >> 20) & 0x7ff;
    const unsigned long long m =
        ((unsigned long long)(b & 0xfffffffffffffll) | (1ull << 52)) << (GB + 1);
    // PTX shr.b64 clamps shift amounts above 64 to 64 (result 0): no min needed
    unsigned long long r;
    asm("shr.b64 %0, %1, %2;" : "=l"(r) : "l"(m), "r"(emax - e));
    return (long long)r ^ (long long)(hi >> 31);
}

// Largest exponent among N staged binary64 values (VS bytes apart).
template <int N, int VS = 256>
__device__ __forceinline__ int max_exponent(uint32_t col)
{
    int h0 = 0, h1 = 0;
#pragma unroll 2
    for (int k = 0; k + 3 < N; k += 4) {
        h0 = __vimax3_s32(h0, lds_hi32(col + (k + 0) * VS) & 0x7fffffff,
                          lds_hi32(col + (k + 1) * VS) & 0x7fffffff);
        h1 = __vimax3_s32(h1, lds_hi32(col + (k + 2) * VS) & 0x7fffffff,
                          lds_hi32(col + (k + 3) * VS) & 0x7fffffff);
    }
#pragma unroll
    for (int k = N - N % 4; k < N; ++k) h0 = max(h0, lds_hi32(col + k * VS) & 0x7fffffff);
    return max(h0, h1) >> 20;
}

// Fixed-point sum of N staged binary64 values aligned to emax (GB guard bits):
// the sum of the terms rounded to the unit, kept as four partial sums (term k
// in partial k mod 4) of the doubled terms t_k and of their low bits (sum of
// rounded terms = (sum t_k + sum (t_k & 1)) / 2, exact, and even per partial).
// |t_k| < 2^(54 + GB), so a partial of fewer than 2^(9 - GB) terms cannot
// overflow; with GB = 10 - ceil(log2 Q) that holds for every N <= Q.
template <int GB, int N, int VS = 256>
__device__ __forceinline__ long long fixed_sum(uint32_t col, int emax)
{
    constexpr int U = 8;
    static_assert((N + 3) / 4 < (1 << (9 - GB)), "fixed-point partial may overflow");
    long long a[4] = {0, 0, 0, 0};
    int p[4] = {0, 0, 0, 0};
    for (int k = 0; k + U - 1 < N; k += U) {
        double v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) v[u] = lds_f64(col + (k + u) * VS);
        long long t[U];
#pragma unroll
        for (int u = 0; u < U; ++u) t[u] = fixed_term2<GB>(v[u], emax);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            a[u] += t[u] + t[u + 4];
            p[u] += (int)(t[u] & 1) + (int)(t[u + 4] & 1);
        }
    }
#pragma unroll
    for (int k = N - N % U; k < N; ++k) {
        const long long t = fixed_term2<GB>(lds_f64(col + k * VS), emax);
        a[k % 4] += t;
        p[k % 4] += (int)(t & 1);
    }
    return ((a[0] + p[0]) >> 1) + ((a[1] + p[1]) >> 1) + ((a[2] + p[2]) >> 1) +
           ((a[3] + p[3]) >> 1);
}

template <int N, int VS = 256>
__device__ __forceinline__ double plain_sum(uint32_t col)
{
    double s = 0.0;
    for (int k = 0; k < N; ++k) s += lds_f64(col + k * VS);
    return s;
}

// emax out of the range the fixed-point sum handles: Inf/NaN, or every value
// below 2^-960 (take the plain binary64 sum then).
__device__ __forceinline__ bool plain_path(int emax) { return emax == 0x7ff || emax < 64; }

template <int GB>
__device__ __forceinline__ double fixed_value(long long acc, int emax)
{
    // acc x 2^(emax - 1075 - GB): the power of two is added to the exponent
    // field of the converted value on the integer pipe (the binary64 pipe is
    // the scarce one).  emax >= 64 here (plain_path), so a non-zero result is
    // normal; past the binary64 range it is +-inf, as the product would be.
    const double d = (double)acc;
    const long long b = __double_as_longlong(d);
    const int k = emax - 1075 - GB;
    const int be = (int)((b >> 52) & 0x7ff) + k;
    if (acc == 0) return d;
    if (be >= 0x7ff) return acc > 0 ? __longlong_as_double(0x7ff0000000000000ll)
                                    : __longlong_as_double((long long)0xfff0000000000000ull);
    return __longlong_as_double(b + ((long long)k << 52));
}

template <int Q>
__device__ __forceinline__ float density_fixed_f32(uint32_t col)   // stride 128 B
{
    // binary32 storage: plain sum in four interleaved partials (fixed order)
    float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
#pragma unroll 2
    for (int k = 0; k + 3 < Q; k += 4) {
        s0 += lds_f32(col + (k + 0) * 128);
        s1 += lds_f32(col + (k + 1) * 128);
        s2 += lds_f32(col + (k + 2) * 128);
        s3 += lds_f32(col + (k + 3) * 128);
    }
#pragma unroll
    for (int k = Q - Q % 4; k < Q; ++k) s0 += lds_f32(col + k * 128);
    return (s0 + s1) + (s2 + s3);
}

template <typename T> __device__ __forceinline__ T lds_val(uint32_t addr);
template <> __device__ __forceinline__ double lds_val<double>(uint32_t addr) { return lds_f64(addr); }
template <> __device__ __forceinline__ float lds_val<float>(uint32_t addr) { return lds_f32(addr); }
template <> __device__ __forceinline__ long long lds_val<long long>(uint32_t addr)
{
    long long v;
    asm volatile("ld.shared.s64 %0, [%1];" : "=l"(v) : "r"(addr));
    return v;
}

// One grid as a tile step sees it.
template <typename T>
struct TileGrid {
    const T* A;     // populations in (pulled)
    T* B;           // populations out
    const typename SrcType<T>::type* S;   // source
    double* Phi;    // density (written on write/check sweeps)
    int64_t V;
    int nx, ny, nz, small;
    double soff;    // constant added to S in this step (mass correction)
    int fr, fw;     // fixed-point storage: exponents of the read and written arrays
    long long cfx;  // fixed-point storage: round((1 - omega) 2^62)
};

__device__ __forceinline__ long long lds_s64(uint32_t addr)
{
    long long v;
    asm volatile("ld.shared.s64 %0, [%1];" : "=l"(v) : "r"(addr));
    return v;
}

// Sum of N staged 64-bit fixed-point values (VS bytes apart) in four
// interleaved partials: integer addition is exact and associative (two's
// complement wraps cancel), so the split leaves the sum unchanged and cuts
// the dependent chain of 64-bit adds to a quarter.  U: groups of four per
// loop trip (code size against loop overhead; timed per kernel at 256^3).
template <int N, int VS, int U>
__device__ __forceinline__ long long fx_sum(uint32_t col)
{
    long long a0 = 0, a1 = 0, a2 = 0, a3 = 0;
#pragma unroll U
    for (int k = 0; k + 3 < N; k += 4) {
        a0 += lds_s64(col + (k + 0) * VS);
        a1 += lds_s64(col + (k + 1) * VS);
        a2 += lds_s64(col + (k + 2) * VS);
        a3 += lds_s64(col + (k + 3) * VS);
    }
#pragma unroll
    for (int k = N - N % 4; k < N; ++k) a0 += lds_s64(col + k * VS);
    return (a0 + a1) + (a2 + a3);
}

// round(q c / 2^62), rounding half up (c = (1 - omega) 2^62 for the relaxation)
__device__ __forceinline__ long long fx_mul(long long q, long long c)
{
    const __int128 prod = (__int128)q * (__int128)c + ((__int128)1 << 61);
    return (long long)(prod >> 62);
}

// 2^e as a binary64 (|e| < 1000)
__device__ __forceinline__ double pow2(int e)
{
    return __longlong_as_double((long long)(1023 + e) << 52);
}

// The part of a tile step that follows the pull, for velocity group g of G
// (velocities lo(g) .. lo(g + 1) - 1): the group's share of the density
// (the G warps of a tile meet at named barrier `bar`, twice in binary64 and
// once otherwise; every meeting sits outside lane-dependent branches), the
// relaxation and store of the group's velocities, and, in group 0, the
// density output and the residual terms.  sbase: this lane's column of the
// group's staged values (velocity lo(g) first, the next VS bytes further on);
// xacc, xexp: the tile's exchange rows.  after_class(std::integral_constant
// <int, cl>) runs, in every lane, once the group's velocities of symmetry
// class cl are relaxed and stored (classes the group holds, in order).
// SPLIT >= 0: the group's staged values from SPLIT on may still be in flight
// when the call starts; before_tail() (run in every lane) makes them
// visible, and the density reads the values before SPLIT first.  The
// fixed-point and binary64 density sums are exact, so the split leaves them
// unchanged; binary32 runs before_tail() before its ordered sum.
struct NoHook {
    template <class C>
    __device__ __forceinline__ void operator()(C) const {}
};
struct NoTail {
    __device__ __forceinline__ void operator()() const {}
};
template <class L, typename T, int G, int g, int VS = 32 * (int)sizeof(T), int SPLIT = -1,
          class Hook = NoHook, class Tail = NoTail>
__device__ __forceinline__ void group_compute(const TileGrid<T>& tg,
                                              const Coefs<typename AccType<T>::type>& c,
                                              int mode, bool valid, int s,
                                              typename AccType<T>::type Sx, int lane,
                                              uint32_t sbase, int bar, long long (&xacc)[G][32],
                                              int (&xexp)[G][32], double& d2, double& n2,
                                              double& mx, double& ms, unsigned long long& fxm,
                                              const Hook& after_class = Hook{},
                                              const Tail& before_tail = Tail{})
{
    using R = typename AccType<T>::type;
    constexpr int lo = g * L::Q / G;
    constexpr int hi = (g + 1) * L::Q / G;
    constexpr int n = hi - lo;
    constexpr int NC = ncls_of<L>();
    constexpr int GB = 63 - 53 - ceil_log2(L::Q);
    T* __restrict__ B = tg.B;
    const int64_t V = tg.V;
    R Phi;
    if constexpr (std::is_same<T, long long>::value) {
        // fixed point: the density is an exact integer sum (one group of four
        // per trip on the x-pairs rows, four in the staged columns)
        constexpr int FU = VS == 256 ? 4 : 1;
        long long part;
        if constexpr (SPLIT > 0 && SPLIT < n) {
            part = fx_sum<SPLIT, VS, FU>(sbase);
            before_tail();
            part += fx_sum<n - SPLIT, VS, FU>(sbase + SPLIT * VS);
        } else {
            if constexpr (SPLIT >= 0) before_tail();
            part = fx_sum<n, VS, FU>(sbase);
        }
        if constexpr (G > 1) {
            xacc[g][lane] = part;
            asm volatile("bar.sync %0, %1;" ::"r"(bar), "n"(G * 32) : "memory");
            part = 0;
#pragma unroll
            for (int k = 0; k < G; ++k) part += xacc[k][lane];
        }
        Phi = (double)part * pow2(-tg.fr);
    } else if constexpr (std::is_same<T, double>::value) {
        int emax;
        if constexpr (SPLIT > 0 && SPLIT < n) {
            emax = max_exponent<SPLIT, VS>(sbase);
            before_tail();
            emax = max(emax, max_exponent<n - SPLIT, VS>(sbase + SPLIT * VS));
        } else {
            if constexpr (SPLIT >= 0) before_tail();
            emax = max_exponent<n, VS>(sbase);
        }
        if constexpr (G > 1) {
            xexp[g][lane] = emax;
            asm volatile("bar.sync %0, %1;" ::"r"(bar), "n"(G * 32) : "memory");
#pragma unroll
            for (int k = 0; k < G; ++k) emax = max(emax, xexp[k][lane]);
        }
        const bool plain = plain_path(emax);
        long long part = plain ? __double_as_longlong(plain_sum<n, VS>(sbase))
                               : fixed_sum<GB, n, VS>(sbase, emax);
        if constexpr (G > 1) {
            xacc[g][lane] = part;
            asm volatile("bar.sync %0, %1;" ::"r"(bar), "n"(G * 32) : "memory");
            if (plain) {
                double t = 0.0;
#pragma unroll
                for (int k = 0; k < G; ++k) t += __longlong_as_double(xacc[k][lane]);
                Phi = t;
            } else {
                long long t = 0;
#pragma unroll
                for (int k = 0; k < G; ++k) t += xacc[k][lane];
                Phi = fixed_value<GB>(t, emax);
            }
        } else {
            Phi = plain ? __longlong_as_double(part) : fixed_value<GB>(part, emax);
        }
    } else {
        if constexpr (SPLIT >= 0) before_tail();
        float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
#pragma unroll 2
        for (int k = 0; k + 3 < n; k += 4) {
            s0 += lds_f32(sbase + (k + 0) * VS);
            s1 += lds_f32(sbase + (k + 1) * VS);
            s2 += lds_f32(sbase + (k + 2) * VS);
            s3 += lds_f32(sbase + (k + 3) * VS);
        }
#pragma unroll
        for (int k = n - n % 4; k < n; ++k) s0 += lds_f32(sbase + k * VS);
        float part = (s0 + s1) + (s2 + s3);
        if constexpr (G > 1) {
            // binary32 partials meet in group order (fixed, deterministic)
            xacc[g][lane] = (long long)__float_as_int(part);
            asm volatile("bar.sync %0, %1;" ::"r"(bar), "n"(G * 32) : "memory");
            part = 0.f;
#pragma unroll
            for (int k = 0; k < G; ++k) part += __int_as_float((int)xacc[k][lane]);
        }
        Phi = part;
    }

    // relax and store this group's velocities, one symmetry class at a
    // time (velocities of a class are contiguous and share phi_c, chi_c)
    auto relax = [&](auto CI) {
        constexpr int cl = decltype(CI)::value;
        constexpr int cb = cls_begin<L>(cl), ce = cls_begin<L>(cl + 1);
        constexpr int i0 = cb > lo ? cb : lo;
        constexpr int i1 = ce < hi ? ce : hi;
        if constexpr (i0 < i1 && std::is_same<T, long long>::value) {
            const double e = fma(c.wphi[cl], Phi, c.chi[cl] * Sx);
            const long long ei = __double2ll_rn(e * pow2(tg.fw));
            // the written array's scale is 2^-k that of the read one (k >= 0,
            // the rescale only lowers it): fold 2^-k into the coefficient
            const int k = tg.fr - tg.fw;
            const long long cw = k == 0 ? tg.cfx : ((tg.cfx >> (k - 1)) + 1) >> 1;
            T* dst = B + ((int64_t)i0 * V + s);
#pragma unroll 2
            for (int i = i0; i < i1; ++i) {
                const long long p = fx_mul(lds_s64(sbase + (i - lo) * VS), cw) + ei;
                fxm |= (unsigned long long)(p ^ (p >> 63));
                store_stream(dst, (T)p);
                dst += V;
            }
        } else if constexpr (i0 < i1) {
            const R e = fma(c.wphi[cl], Phi, c.chi[cl] * Sx);
            T* dst = B + ((int64_t)i0 * V + s);
            int i = i0;
            for (; i + 3 < i1; i += 4) {
                const R g0 = lds_val<T>(sbase + (i + 0 - lo) * VS);
                const R g1 = lds_val<T>(sbase + (i + 1 - lo) * VS);
                const R g2 = lds_val<T>(sbase + (i + 2 - lo) * VS);
                const R g3 = lds_val<T>(sbase + (i + 3 - lo) * VS);
                store_stream(dst, (T)fma(c.om1, g0, e));
                store_stream(dst + V, (T)fma(c.om1, g1, e));
                store_stream(dst + 2 * V, (T)fma(c.om1, g2, e));
                store_stream(dst + 3 * V, (T)fma(c.om1, g3, e));
                dst += 4 * V;
            }
            for (; i < i1; ++i) {
                const R gi = lds_val<T>(sbase + (i - lo) * VS);
                store_stream(dst, (T)fma(c.om1, gi, e));
                dst += V;
            }
        }
    };
    if constexpr (std::is_same<Hook, NoHook>::value) {
        if (valid) static_for<0, NC>(relax);
    } else {
        static_for<0, NC>([&](auto CI) {
            constexpr int cl = decltype(CI)::value;
            if (valid) relax(CI);
            // classes the group holds velocities of
            if constexpr (cls_begin<L>(cl) < hi && cls_begin<L>(cl + 1) > lo) after_class(CI);
        });
    }
    // density output and residual contributions (one group per tile)
    if (g == 0 && mode != kPlain && valid) {
        const double ph = (double)Phi;
        if (mode == kCheck) {
            const double d = ph - tg.Phi[s];
            d2 += d * d;
            n2 += ph * ph;
            mx = fmax(mx, fabs(d));
            ms += ph;
        }
        tg.Phi[s] = ph;
    }
}

// The pull of one 32-site tile, per lane: wrapped offsets of the lane's
// neighbours, and the copy of one velocity's value into the lane's column
// (dst; zero fill past the grid's end and on the first step).  A lane reads
// back only what it copied itself, so the copies need no barrier.
template <class L, typename T>
struct TilePull {
    static constexpr int RC = reach_of<L>();
    static constexpr int W = 2 * RC + 1;
    int xs[W], yo[W], zo[W];
    int nbytes;

    __device__ __forceinline__ void locate(int tile, int64_t V, int nx, int ny, int nz, int small,
                                           bool zero_in, int lane)
    {
        const int nxy = nx * ny;
        const int64_t s64 = (int64_t)tile * 32 + lane;
        const bool valid = s64 < V;
        const int s = valid ? (int)s64 : 0;
        const int r = (int)((unsigned)s / (unsigned)nx);
        const int x = s - r * nx;
        const int z = (int)((unsigned)r / (unsigned)ny);
        const int y = r - z * ny;
        if (small) {
#pragma unroll
            for (int d = -RC; d <= RC; ++d) {
                xs[d + RC] = wrap_any(x - d, nx);
                yo[d + RC] = wrap_any(y - d, ny) * nx;
                zo[d + RC] = wrap_any(z - d, nz) * nxy;
            }
        } else {
            static_for<0, W>([&](auto DI) {
                constexpr int d = decltype(DI)::value - RC;
                xs[d + RC] = wrap_off<d>(x, nx);
                yo[d + RC] = wrap_off<d>(y, ny) * nx;
                zo[d + RC] = wrap_off<d>(z, nz) * nxy;
            });
        }
        nbytes = (valid && !zero_in) ? (int)sizeof(T) : 0;
    }
    template <int i>
    __device__ __forceinline__ void pull(const T* __restrict__ A, int64_t V, uint32_t dst) const
    {
        const T* src = A + ((int64_t)i * V + (zo[vz_of<L>(i) + RC] + yo[vy_of<L>(i) + RC] +
                                              xs[vx_of<L>(i) + RC]));
        cp_async<sizeof(T)>(dst, src, nbytes);
    }
};

// First velocity of the last symmetry class that velocities lo .. hi - 1 hold.
template <class L>
__host__ __device__ constexpr int tail_begin(int lo, int hi)
{
    const int b = cls_begin<L>(cls_of<L>(hi - 1));
    return b > lo ? b : lo;
}

// Where a tile's copies may start while the one before is relaxed (EARLY
// below): binary64 of the large sets.  GLUPS on 173 x 141 x 100, D3Q111, 2
// groups x 2 tiles, with and without: binary64 2.67 / 2.37, fixed point 2.88 /
// 2.95, binary32 5.15 / 5.81; D3Q19 in binary64 at 256^3 17.9 / 18.1.  D2Q169's
// geometries of few or unpaired warps lose by it (500 x 513, 1 x 2 299 us
// a step with and 294 without, 3 x 1 219 / 206, 4 x 1 243 / 212; 2 x 2 190 / 209).
template <class L, typename T, int G, int TILES>
struct EarlyRefill {
    static constexpr bool value = L::Q > 64 && std::is_same<T, double>::value &&
                                  (L::Q <= 111 || G == 2 || (G == 3 && TILES == 2));
};
// And when it pays: rounds of tiles per resident warp group.  A block's first
// tile overlaps nothing, and a grid of one tile each only runs the longer code:
// time of a step with refill to that without, 2 groups x 2 tiles, by rounds:
// D3Q111 1.04 (0.9), 1.02 (1.35), 0.99 (1.6), 0.95 (2.2), 0.88 (3.3), 0.87 (14);
// D2Q81 0.98 (1.3), 0.92 (1.9), 0.86 (3.5); D2Q169, a third fewer warps per SM,
// 1.09 (1.2), 1.04 (1.5), 1.02 (2.1), 1.01 (3.2), 0.95 (4.6), 0.89 (51).
template <class L>
bool early_refill_pays(int64_t ntiles, int64_t slots)
{
    return 2 * ntiles >= (L::Q > 111 ? 8 : 3) * slots;
}
// One tile of velocity group g.  EARLY: its copies are in flight already, and
// class by class as it is relaxed the copies of the warp's next tile
// (`refill(I)` copies velocity I of it) are started, so the pull of a tile
// overlaps the computation of the one before; each class is a copy group of
// its own, so a tile starts once every class but its last (refilled last) has
// landed, as in the x-pairs sweep.  Else refill copies this tile.
template <class L, typename T, int G, int g, bool EARLY, class Refill>
__device__ __forceinline__ void tile_compute(const TileGrid<T>& tg,
                                             const Coefs<typename AccType<T>::type>& c, int mode,
                                             bool valid, int s, typename AccType<T>::type Sx,
                                             int lane, uint32_t sbase, int bar,
                                             long long (&xacc)[G][32], int (&xexp)[G][32],
                                             double& d2, double& n2, double& mx, double& ms,
                                             unsigned long long& fxm, bool more,
                                             const Refill& refill)
{
    constexpr int lo = g * L::Q / G, hi = (g + 1) * L::Q / G;
    constexpr int VS = 32 * (int)sizeof(T);
    constexpr int tb = tail_begin<L>(lo, hi);
    if constexpr (EARLY) {
        cp_async_wait_all_but_last();
        group_compute<L, T, G, g, VS, tb - lo>(
            tg, c, mode, valid, s, Sx, lane, sbase, bar, xacc, xexp, d2, n2, mx, ms, fxm,
            [&](auto CI) {
                constexpr int cl = decltype(CI)::value;
                constexpr int cb = cls_begin<L>(cl), ce = cls_begin<L>(cl + 1);
                if (more) {
                    static_for<(cb > lo ? cb : lo), (ce < hi ? ce : hi)>(refill);
                    cp_async_commit();
                }
            },
            [&]() { cp_async_wait_committed(); });
    } else {
        static_for<lo, hi>(refill);
        cp_async_wait_all();
        group_compute<L, T, G, g, VS>(tg, c, mode, valid, s, Sx, lane, sbase, bar, xacc, xexp, d2,
                                      n2, mx, ms, fxm);
    }
}

// The first tile's copies, in the groups tile_compute waits for.
template <class L, typename T, int G, int g, class Refill>
__device__ __forceinline__ void tile_first(const Refill& refill)
{
    constexpr int lo = g * L::Q / G, hi = (g + 1) * L::Q / G;
    constexpr int tb = tail_begin<L>(lo, hi);
    static_for<lo, tb>(refill);
    cp_async_commit();
    static_for<tb, hi>(refill);
    cp_async_commit();
}

template <class L, typename T, int G_, int TILES_, bool EARLY>
__global__ void __launch_bounds__(G_ * TILES_ * 32)
sweep_staged_kernel(const SweepArgs a, const Coefs<typename AccType<T>::type> c)
{
    if (a.stop != nullptr && *a.stop != 0) return;   // the run stopped before this step
    constexpr int G = G_;
    constexpr int TILES = TILES_;
    using ST = Staged<L, T, G, TILES>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double rpart[TILES][4];
    // per-group partial densities of a tile, two sets used by turns: a warp
    // writes the next tile's partial only after the exchange barrier of that
    // tile, so a partner still reading this tile's set cannot see it change
    __shared__ long long xacc[2][TILES][G][32];
    __shared__ int xexp[TILES][G][32];         // per-group largest exponents

    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    const int grp = wib % G;     // velocity group of this warp
    const int sub = wib / G;     // tile slot of this warp in the block
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(
        reinterpret_cast<T*>(smem_raw) + (size_t)wib * ST::CH * 32 + lane);
    const bool fx = std::is_same<T, long long>::value;
    const TileGrid<T> tg{static_cast<const T*>(a.A), static_cast<T*>(a.B),
                         static_cast<const typename SrcType<T>::type*>(a.S), a.Phi, a.V, a.nx,
                         a.ny, a.nz, a.small, a.soff, fx ? a.fxF[a.cur] : 0,
                         fx ? a.fxF[a.cur ^ 1] : 0, a.cfx};

    double rd2 = 0.0, rn2 = 0.0, rmx = 0.0, rms = 0.0;
    unsigned long long fxm = 0ull;
    const int nt = gridDim.x * TILES;
    int par = 0;
    using R = typename AccType<T>::type;
    TilePull<L, T> next;
    auto locate = [&](int tile) {
        next.locate(tile, tg.V, tg.nx, tg.ny, tg.nz, tg.small, a.zero_in != 0, lane);
    };
    // one tile of group g; its copies, or those of the next tile, by refill
    auto step = [&](auto GI, int tile, const auto& refill) {
        constexpr int g = decltype(GI)::value;
        const int64_t s64 = (int64_t)tile * 32 + lane;
        const bool valid = s64 < tg.V;
        const int s = valid ? (int)s64 : 0;
        // the source offset (mass correction) is used by binary32 storage only
        R Sx = R(0);
        if (valid) {
            if constexpr (std::is_same<T, float>::value) Sx = (R)((double)tg.S[s] + tg.soff);
            else Sx = (R)tg.S[s];
        }
        const bool more = EARLY && tile + nt < a.ntiles;
        if (more) locate(tile + nt);
        tile_compute<L, T, G, g, EARLY>(tg, c, a.mode, valid, s, Sx, lane, sbase, 1 + sub,
                                        xacc[par][sub], xexp[sub], rd2, rn2, rmx, rms, fxm, more,
                                        refill);
    };
    auto refill_of = [&](auto GI) {
        return [&](auto I) {
            constexpr int i = decltype(I)::value;
            constexpr int lo = decltype(GI)::value * L::Q / G;
            next.template pull<i>(tg.A, tg.V, sbase + (uint32_t)((i - lo) * 32 * sizeof(T)));
        };
    };
    int tile = blockIdx.x * TILES + sub;
    if constexpr (EARLY) {
        // a group's copies run ahead into its own next tile: a loop for each
        static_for<0, G>([&](auto GI) {
            if (grp != decltype(GI)::value) return;
            const auto refill = refill_of(GI);
            if (tile < a.ntiles) {
                locate(tile);
                tile_first<L, T, G, decltype(GI)::value>(refill);
            }
            for (; tile < a.ntiles; tile += nt, par ^= 1) step(GI, tile, refill);
        });
    } else {
        for (; tile < a.ntiles; tile += nt, par ^= 1) {
            locate(tile);
            static_for<0, G>([&](auto GI) {
                if (grp == decltype(GI)::value) step(GI, tile, refill_of(GI));
            });
        }
    }
    if constexpr (std::is_same<T, long long>::value) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            fxm |= __shfl_down_sync(0xffffffffu, fxm, o);
        }
        if (lane == 0 && fxm) atomicOr(a.fxmax, fxm);
    }

    if (a.mode == kCheck) {
        if (grp == 0) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                rd2 += __shfl_down_sync(0xffffffffu, rd2, o);
                rn2 += __shfl_down_sync(0xffffffffu, rn2, o);
                rmx = fmax(rmx, __shfl_down_sync(0xffffffffu, rmx, o));
                rms += __shfl_down_sync(0xffffffffu, rms, o);
            }
            if (lane == 0) {
                rpart[sub][0] = rd2;
                rpart[sub][1] = rn2;
                rpart[sub][2] = rmx;
                rpart[sub][3] = rms;
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            double t0 = 0.0, t1 = 0.0, t2 = 0.0, t3 = 0.0;
            for (int k = 0; k < TILES; ++k) {
                t0 += rpart[k][0];
                t1 += rpart[k][1];
                t2 = fmax(t2, rpart[k][2]);
                t3 += rpart[k][3];
            }
            a.partials[4 * blockIdx.x + 0] = t0;
            a.partials[4 * blockIdx.x + 1] = t1;
            a.partials[4 * blockIdx.x + 2] = t2;
            a.partials[4 * blockIdx.x + 3] = t3;
        }
    }
}

// ---------------------------------------------------------------------------
// Batch sweep: one persistent launch advances every live grid of a batch by
// one step.  Batch-wide tile t belongs to the grid whose tile_begin is the
// largest one <= t (binary search over the descriptors for a warp's first
// tile, a walk from there on).  A grid's age (steps since it joined) picks its
// buffers; it joins at a window's start, so the position k of the step in its
// window of K steps, the same for every grid, gives the residual schedule of
// its own age: Phi is written when (age + 2) % K == 0 and checked when
// (age + 1) % K == 0 (age >= 1), and a grid's trajectory and stopping step do
// not depend on what else is in the batch.  The host passes these as `phase`:
// as three 64-bit remainders per tile and warp they cost as much as a third of
// a binary32 tile.  On check steps each tile leaves its four partial sums in
// tile_partials (with the sum of Phi); batch_reduce_kernel sums them per grid
// in a fixed order.
// ---------------------------------------------------------------------------
template <class L, typename T, int G_, int TILES_>
__global__ void __launch_bounds__(G_ * TILES_ * 32)
sweep_batch_kernel(BatchState* st, int k, int phase)
{
    using R = typename AccType<T>::type;
    constexpr int G = G_;
    constexpr int TILES = TILES_;
    using ST = Staged<L, T, G, TILES>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ long long xacc[2][TILES][G][32];   // two sets used by turns (staged sweep)
    __shared__ int xexp[TILES][G][32];

    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    const int grp = wib % G;
    const int sub = wib / G;
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(
        reinterpret_cast<T*>(smem_raw) + (size_t)wib * ST::CH * 32 + lane);
    const BatchGrid<R>* grids = static_cast<const BatchGrid<R>*>(st->grids);
    const int ngrids = st->ngrids;
    const int ntiles = st->ntiles;
    const long long step = st->step + k;
    double* tpart = st->tile_partials;

    constexpr bool fx = std::is_same<T, long long>::value;
    const int nt = gridDim.x * TILES;
    int par = 0;
    // index of the grid that tile t belongs to
    auto grid_of = [&](int t) {
        int lo = 0, hi = ngrids - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (grids[mid].tile_begin <= t) lo = mid;
            else hi = mid - 1;
        }
        return lo;
    };
    auto mode_of = [&](long long age) {
        if (age >= 1 && (phase & kPhaseCheck)) return (int)kCheck;
        return age == 0 || (phase & kPhaseWrite) ? (int)kWritePhi : (int)kPlain;
    };
    // binary32: the step after a check removes the mass that check measured
    auto soff_of = [&](const BatchGrid<R>& gd, long long age) {
        return gd.soff && age >= 1 && (phase & kPhaseFirst) ? *gd.soff : 0.0;
    };
    auto state_of = [&](const BatchGrid<R>& gd, long long age, double soff) {
        const int cur = (int)(age & 1);
        return TileGrid<T>{static_cast<const T*>(gd.pop[cur]), static_cast<T*>(gd.pop[cur ^ 1]),
                           static_cast<const typename SrcType<T>::type*>(gd.S), gd.Phi, gd.V,
                           gd.nx, gd.ny, gd.nz, gd.small, soff, fx ? gd.fxF[cur] : 0,
                           fx ? gd.fxF[cur ^ 1] : 0, fx ? gd.cfx : 0};
    };
    // a tile's magnitude bound and residual terms
    auto finish = [&](const BatchGrid<R>& gd, int tile, int mode, double d2, double n2, double mx,
                      double ms, unsigned long long fxm) {
        if constexpr (fx) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) fxm |= __shfl_down_sync(0xffffffffu, fxm, o);
            if (lane == 0 && fxm) atomicOr(gd.fxmax, fxm);
        }
        if (mode == kCheck && grp == 0) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                d2 += __shfl_down_sync(0xffffffffu, d2, o);
                n2 += __shfl_down_sync(0xffffffffu, n2, o);
                mx = fmax(mx, __shfl_down_sync(0xffffffffu, mx, o));
                ms += __shfl_down_sync(0xffffffffu, ms, o);
            }
            if (lane == 0) {
                tpart[4 * (int64_t)tile + 0] = d2;
                tpart[4 * (int64_t)tile + 1] = n2;
                tpart[4 * (int64_t)tile + 2] = mx;
                tpart[4 * (int64_t)tile + 3] = ms;
            }
        }
    };
    // this warp's tiles; groups(f) calls f with the warp's velocity group
    auto loop = [&](const auto& groups) {
        int tile = blockIdx.x * TILES + sub;
        if (tile >= ntiles) return;
        int gi = grid_of(tile);
        for (; tile < ntiles; tile += nt, par ^= 1) {
            const BatchGrid<R>& gd = grids[gi];
            const long long age = step - gd.join;
            const int mode = mode_of(age);
            const TileGrid<T> tg = state_of(gd, age, soff_of(gd, age));
            const int64_t s64 = (int64_t)(tile - gd.tile_begin) * 32 + lane;
            const bool valid = s64 < tg.V;
            R Sx = R(0);
            if (valid) {
                if constexpr (std::is_same<T, float>::value)
                    Sx = (R)((double)tg.S[s64] + tg.soff);
                else Sx = (R)tg.S[s64];
            }
            TilePull<L, T> here;
            here.locate(tile - gd.tile_begin, tg.V, tg.nx, tg.ny, tg.nz, tg.small, age == 0, lane);
            double d2 = 0.0, n2 = 0.0, mx = 0.0, ms = 0.0;
            unsigned long long fxm = 0ull;
            groups([&](auto GI) {
                constexpr int g = decltype(GI)::value;
                auto pull = [&](auto I) {
                    constexpr int i = decltype(I)::value;
                    here.template pull<i>(tg.A, tg.V,
                                          sbase + (uint32_t)((i - ST::lo(g)) * 32 * sizeof(T)));
                };
                tile_compute<L, T, G, g, false>(tg, gd.c, mode, valid, (int)s64, Sx, lane, sbase,
                                                1 + sub, xacc[par][sub], xexp[sub], d2, n2, mx, ms,
                                                fxm, false, pull);
            });
            finish(gd, tile, mode, d2, n2, mx, ms, fxm);
            // the next tile's grid is this one or a later one
            if (tile + nt < ntiles)
                while (gi + 1 < ngrids && grids[gi + 1].tile_begin <= tile + nt) ++gi;
        }
    };
    // One loop for all groups in binary64, one for each in the other storages,
    // as measured (us per window of 32 steps, one loop / each its own: D3Q111,
    // 16 grids of 32 x 33 x 34, 2 groups x 2 tiles, binary64 9630 / 9800;
    // binary32 and fixed point up to 5 % the other way).  No copies ahead of a
    // tile (EarlyRefill) here: with them the same batch took 10140 us, 32 grids
    // of 100 x 120 of D2Q169 13560 against 11900.
    if constexpr (std::is_same<T, double>::value) {
        loop([&](const auto& f) {
            static_for<0, G>([&](auto GI) {
                if (grp == decltype(GI)::value) f(GI);
            });
        });
    } else {
        static_for<0, G>([&](auto GI) {
            if (grp == decltype(GI)::value) loop([&](const auto& f) { f(GI); });
        });
    }
}

template <class L, typename T, int K>
int launch_batch_variant(BatchState* st, int k, int phase, int grid, void* stream)
{
    constexpr Geo geo = Variants<L>::at(K);
    using ST = Staged<L, T, geo.G, geo.TILES>;
    sweep_batch_kernel<L, T, geo.G, geo.TILES><<<grid, ST::WARPS * 32, ST::smem_bytes(),
                                                 (cudaStream_t)stream>>>(st, k, phase);
    return (int)cudaGetLastError();
}

template <class L, typename T, int K>
int batch_occupancy_variant(int* blocks)
{
    constexpr Geo geo = Variants<L>::at(K);
    using ST = Staged<L, T, geo.G, geo.TILES>;
    auto kern = sweep_batch_kernel<L, T, geo.G, geo.TILES>;
    cudaError_t e = set_sweep_smem(kern, ST::smem_bytes());
    if (e != cudaSuccess) return (int)e;
    return (int)cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, kern, ST::WARPS * 32,
                                                              ST::smem_bytes());
}

template <class L, typename T>
int launch_batch_t(int variant, BatchState* st, int k, int phase, int grid, void* stream)
{
    int rc = (int)cudaErrorInvalidValue;
    static_for<0, Variants<L>::N>([&](auto K) {
        if (variant == decltype(K)::value)
            rc = launch_batch_variant<L, T, decltype(K)::value>(st, k, phase, grid, stream);
    });
    return rc;
}

template <class L, typename T>
int batch_occupancy_t(int variant, int* blocks)
{
    int rc = (int)cudaErrorInvalidValue;
    static_for<0, Variants<L>::N>([&](auto K) {
        if (variant == decltype(K)::value)
            rc = batch_occupancy_variant<L, T, decltype(K)::value>(blocks);
    });
    return rc;
}

// ---------------------------------------------------------------------------
// binary16 storage.  A population value v lives as the binary16 number
// v / sc[k] in array k, with sc[k] a power of two set before each step so
// that the step's largest |p| has 4x headroom below 65504; every arithmetic
// operation is binary32.  cp.async has no 2-byte form, so each lane copies
// the aligned 4-byte word that holds its value and picks the half by the
// parity of the element index.  One warp per tile, all Q velocities.
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned int lds_b32(uint32_t addr)
{
    unsigned int v;
    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}

template <class L, int TILES>
__global__ void __launch_bounds__(TILES * 32)
sweep_h16_kernel(const SweepArgs a, const Coefs<float> c)
{
    constexpr int Q = L::Q;
    constexpr int RC = reach_of<L>();
    constexpr int W = 2 * RC + 1;
    constexpr int NC = ncls_of<L>();
    constexpr int NPB = (Q + 31) / 32;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double rpart[TILES][4];
    __shared__ float mpart[TILES];

    const int lane = threadIdx.x & 31;
    const int sub = threadIdx.x >> 5;
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(smem_raw) +
                           (uint32_t)((sub * Q * 32 + lane) * 4);
    const __half* __restrict__ A = static_cast<const __half*>(a.A);
    __half* __restrict__ B = static_cast<__half*>(a.B);
    const float* __restrict__ S = static_cast<const float*>(a.S);
    const int64_t V = a.V;
    const int nxy = a.nx * a.ny;
    const float sr = a.sc[a.cur];
    const float inv_sw = 1.0f / a.sc[a.cur ^ 1];
    const int vodd = (int)(V & 1);

    double rd2 = 0.0, rn2 = 0.0, rmx = 0.0, rms = 0.0;
    float pmax = 0.f;
    int of = 0;
    const int nt = gridDim.x * TILES;
    for (int tile = blockIdx.x * TILES + sub; tile < a.ntiles; tile += nt) {
        const int64_t s64 = (int64_t)tile * 32 + lane;
        const bool valid = s64 < V;
        const int s = valid ? (int)s64 : 0;
        const int x = s % a.nx;
        const int r = s / a.nx;
        const int y = r % a.ny;
        const int z = r / a.ny;
        int xs[W], yo[W], zo[W];
#pragma unroll
        for (int d = -RC; d <= RC; ++d) {
            if (a.small) {
                xs[d + RC] = wrap_any(x - d, a.nx);
                yo[d + RC] = wrap_any(y - d, a.ny) * a.nx;
                zo[d + RC] = wrap_any(z - d, a.nz) * nxy;
            } else {
                xs[d + RC] = wrap_near(x - d, a.nx);
                yo[d + RC] = wrap_near(y - d, a.ny) * a.nx;
                zo[d + RC] = wrap_near(z - d, a.nz) * nxy;
            }
        }
        const int nbytes = (valid && !a.zero_in) ? 4 : 0;
        unsigned int pb[NPB];
#pragma unroll
        for (int k = 0; k < NPB; ++k) pb[k] = 0u;
        static_for<0, Q>([&](auto I) {
            constexpr int i = decltype(I)::value;
            constexpr int ox = vx_of<L>(i) + RC;
            constexpr int oy = vy_of<L>(i) + RC;
            constexpr int oz = vz_of<L>(i) + RC;
            const int off = zo[oz] + yo[oy] + xs[ox];
            const int par = (off ^ ((i & 1) & vodd)) & 1;     // parity of i*V + off
            const __half* src = A + ((int64_t)i * V + off - par);
            cp_async<4>(sbase + (uint32_t)(i * 128), src, nbytes);
            pb[i / 32] |= (unsigned int)par << (i % 32);
        });
        cp_async_wait_all();

        // pick each lane's half and rewrite the slot as a binary32 value, so
        // the passes below are those of binary32 storage
#pragma unroll
        for (int w = 0; w < NPB; ++w) {
            const unsigned int bits = pb[w];
            const int nb = (Q - 32 * w) < 32 ? (Q - 32 * w) : 32;
#pragma unroll 4
            for (int b = 0; b < nb; ++b) {
                const uint32_t ad = sbase + (uint32_t)((32 * w + b) * 128);
                const unsigned int wd = lds_b32(ad);
                const unsigned int h = ((bits >> b) & 1u) ? (wd >> 16) : (wd & 0xffffu);
                const float v = __half2float(__ushort_as_half((unsigned short)h));
                asm volatile("st.shared.f32 [%0], %1;" ::"r"(ad), "f"(v) : "memory");
            }
        }
        // the slots hold unscaled values: the array's scale sr (a power of
        // two, so exactly) multiplies the sum and the relaxation factor
        const float Phi = density_fixed_f32<Q>(sbase) * sr;
        const float om1s = c.om1 * sr;
        const float Sx = valid ? (float)((double)S[s] + a.soff) : 0.f;
        if (valid) {
            static_for<0, NC>([&](auto CI) {
                constexpr int cl = decltype(CI)::value;
                constexpr int i0 = cls_begin<L>(cl), i1 = cls_begin<L>(cl + 1);
                const float e = fmaf(c.wphi[cl], Phi, c.chi[cl] * Sx);
                unsigned short* dst = reinterpret_cast<unsigned short*>(B) + ((int64_t)i0 * V + s);
#pragma unroll 4
                for (int i = i0; i < i1; ++i) {
                    const float p = fmaf(om1s, lds_f32(sbase + (uint32_t)(i * 128)), e);
                    pmax = fmaxf(pmax, fabsf(p));
                    __stcs(dst, __half_as_ushort(__float2half_rn(p * inv_sw)));
                    dst += V;
                }
            });
        }
        if (a.mode != kPlain && valid) {
            const double ph = (double)Phi;
            if (a.mode == kCheck) {
                const double d = ph - a.Phi[s];
                rd2 += d * d;
                rn2 += ph * ph;
                rmx = fmax(rmx, fabs(d));
                rms += ph;
            }
            a.Phi[s] = ph;
        }
        __syncwarp();
    }

#pragma unroll
    for (int o = 16; o > 0; o >>= 1) pmax = fmaxf(pmax, __shfl_down_sync(0xffffffffu, pmax, o));
    if (lane == 0) mpart[sub] = pmax;
    if (a.mode == kCheck) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            rd2 += __shfl_down_sync(0xffffffffu, rd2, o);
            rn2 += __shfl_down_sync(0xffffffffu, rn2, o);
            rmx = fmax(rmx, __shfl_down_sync(0xffffffffu, rmx, o));
            rms += __shfl_down_sync(0xffffffffu, rms, o);
        }
        if (lane == 0) {
            rpart[sub][0] = rd2;
            rpart[sub][1] = rn2;
            rpart[sub][2] = rmx;
            rpart[sub][3] = rms;
        }
    }
    // a stored value beyond the binary16 range (it became +-inf) overflowed
    of = !(pmax * inv_sw <= 65504.f);
    if (__any_sync(0xffffffffu, of) && lane == 0) atomicOr(a.oflow, 1);
    __syncthreads();
    if (threadIdx.x == 0) {
        float m = 0.f;
        for (int k = 0; k < TILES; ++k) m = fmaxf(m, mpart[k]);
        atomicMax(a.pmax, __float_as_uint(m));
        if (a.mode == kCheck) {
            double t0 = 0.0, t1 = 0.0, t2 = 0.0, t3 = 0.0;
            for (int k = 0; k < TILES; ++k) {
                t0 += rpart[k][0];
                t1 += rpart[k][1];
                t2 = fmax(t2, rpart[k][2]);
                t3 += rpart[k][3];
            }
            a.partials[4 * blockIdx.x + 0] = t0;
            a.partials[4 * blockIdx.x + 1] = t1;
            a.partials[4 * blockIdx.x + 2] = t2;
            a.partials[4 * blockIdx.x + 3] = t3;
        }
    }
}

// ---------------------------------------------------------------------------
// binary16 storage, two sites per lane.  A warp owns a tile of 64 consecutive
// sites of one x row (nx a multiple of 64, every edge at least the lattice's
// reach) and lane l the pair of sites x0 + 2l, x0 + 2l + 1: one aligned
// 4-byte word of every plane.  For velocity i the pulled elements start at
// x0 - v_x, whose parity is that of v_x, known at compile time: an even start
// is 32 aligned words (lane l's pair is word l), an odd one 33 (lane l's pair
// is the high half of word l and the low half of word l + 1).  Each lane
// copies word l of the run (lane 0 also word 32 of an odd run) into the
// velocity's 33-word slot.  After the copies each odd run is repacked in
// place into aligned pairs, and both passes read one word per velocity and
// lane, converted where it is used.  Per site, the density, relaxation, scaling,
// overflow bound and rounding are those of sweep_h16_kernel, operation for
// operation, so the two give the same results bit for bit.
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned int prmt(unsigned int a, unsigned int b, unsigned int sel)
{
    unsigned int r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(sel));
    return r;
}

// Two binary32 values in one 64-bit register pair, added and multiplied by one
// instruction each; every half rounds as the scalar operation does.
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pack2(float lo, float hi)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float2 unpack2(f32x2 v)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
// max(m, |x|, |y|)
__device__ __forceinline__ float max3_abs(float m, float x, float y)
{
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(m), "f"(fabsf(x)), "f"(fabsf(y)));
    return r;
}

// Lane's pair of a velocity from its slot (sw: this lane's word, 4 l), after
// the repack: one aligned word, low half the even site, high half the odd one.
__device__ __forceinline__ f32x2 h16_pair(uint32_t sw)
{
    const unsigned int w = lds_b32(sw);
    const float2 v = __half22float2(*reinterpret_cast<const __half2*>(&w));
    return pack2(v.x, v.y);
}

// AHEAD: a class's slots take the copies of the warp's next tile as soon as it
// is relaxed.
template <class L, int TILES, int MINB, bool AHEAD>
__global__ void __launch_bounds__(TILES * 32, MINB)
sweep_h16p_kernel(const SweepArgs a, const Coefs<float> c)
{
    constexpr int Q = L::Q;
    constexpr int RC = reach_of<L>();
    constexpr int W = 2 * RC + 1;
    constexpr int NC = ncls_of<L>();
    constexpr int SW = 33 * 4;                 // bytes of one velocity's slot
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double rpart[TILES][4];
    __shared__ float mpart[TILES];

    const int lane = threadIdx.x & 31;
    const int sub = threadIdx.x >> 5;
    const uint32_t slot = (uint32_t)__cvta_generic_to_shared(smem_raw) + (uint32_t)(sub * Q * SW);
    const uint32_t sw = slot + (uint32_t)(lane * 4);
    // one scratch word per lane past the slots of the block's tiles
    const uint32_t dummy = (uint32_t)__cvta_generic_to_shared(smem_raw) +
                           (uint32_t)(TILES * Q * SW + threadIdx.x * 4);
    const unsigned int* __restrict__ A = static_cast<const unsigned int*>(a.A);   // words
    unsigned int* __restrict__ B = static_cast<unsigned int*>(a.B);
    const float* __restrict__ S = static_cast<const float*>(a.S);
    const int64_t V = a.V;
    const int64_t Vw = V >> 1;                 // words per plane (V is even)
    const int nx = a.nx, ny = a.ny, nz = a.nz;
    const int nw = nx >> 1;                    // words per row
    const float sr = a.sc[a.cur];
    const float inv_sw = 1.0f / a.sc[a.cur ^ 1];
    const int ntiles = (int)(V >> 6);

    double rd2 = 0.0, rn2 = 0.0, rmx = 0.0, rms = 0.0;
    float pmax = 0.f;
    const int nt = gridDim.x * TILES;
    const int nb = a.zero_in ? 0 : 4;
    // the tile whose slots are being filled: row offsets, the first x, and the
    // lane's word of the run for each x displacement -R..R (the first word of
    // a run is (x0 - vx) rounded down to even, halved)
    int yo[W], zo[W], wl[W], x0 = 0;
    auto locate = [&](int tile) {
        const int s0 = tile * 64;              // first site: x0 = s0 mod nx, even
        const int r = (int)((unsigned)s0 / (unsigned)nx);
        x0 = s0 - r * nx;
        const int z = (int)((unsigned)r / (unsigned)ny);
        const int y = r - z * ny;
        static_for<0, W>([&](auto DI) {
            constexpr int d = decltype(DI)::value - RC;
            yo[d + RC] = wrap_off<d>(y, ny) * nw;
            zo[d + RC] = wrap_off<d>(z, nz) * (ny * nw);
            int w = ((x0 - d) >> 1) + lane;    // arithmetic shift: floor
            wl[d + RC] = w < 0 ? w + nw : (w >= nw ? w - nw : w);
        });
    };
    auto pull = [&](auto I) {
        constexpr int i = decltype(I)::value;
        constexpr int vx = vx_of<L>(i);
        const unsigned int* row =
            A + ((int64_t)i * Vw + (zo[vz_of<L>(i) + RC] + yo[vy_of<L>(i) + RC]));
        cp_async<4>(sw + (uint32_t)(i * SW), row + wl[vx + RC], nb);
        if constexpr (vx & 1) {
            // word 32 of an odd run, copied by lane 0; the other lanes
            // issue the same instruction with nothing to read, into a
            // word of their own (no branch in the unrolled pull)
            int w1 = ((x0 - vx) >> 1) + 32;
            w1 = w1 >= nw ? w1 - nw : w1;
            cp_async<4>(lane == 0 ? slot + (uint32_t)(i * SW + 128) : dummy, row + w1,
                        lane == 0 ? nb : 0);
        }
    };
    const int first = blockIdx.x * TILES + sub;
    if (AHEAD && first < ntiles) {
        locate(first);
        static_for<0, Q>(pull);
    }
    for (int tile = first; tile < ntiles; tile += nt) {
        if constexpr (!AHEAD) {
            locate(tile);
            static_for<0, Q>(pull);
        }
        const int s = tile * 64 + 2 * lane;
        const float2 S2 = *reinterpret_cast<const float2*>(S + s);
        const bool more = AHEAD && tile + nt < ntiles;
        if (more) locate(tile + nt);
        cp_async_wait_all();
        __syncwarp();
        // repack every odd run in place into aligned pairs: word l := high
        // half of word l, low half of word l + 1 (all lanes read before any
        // writes), so both passes below read one aligned word per velocity
        static_for<0, Q>([&](auto I) {
            constexpr int i = decltype(I)::value;
            if constexpr (vx_of<L>(i) & 1) {
                const uint32_t ad = sw + (uint32_t)(i * SW);
                const unsigned int w = prmt(lds_b32(ad), lds_b32(ad + 4), 0x5432);
                __syncwarp();
                asm volatile("st.shared.b32 [%0], %1;" ::"r"(ad), "r"(w) : "memory");
            }
        });
        __syncwarp();

        // density: per site the four interleaved binary32 partials of
        // density_fixed_f32 (velocity k to partial k mod 4, the last Q mod 4
        // to partial 0), then the array's scale; both sites in one packed add
        f32x2 p0 = 0, p1 = 0, p2 = 0, p3 = 0;
#pragma unroll 2
        for (int k = 0; k + 3 < Q; k += 4) {
            p0 = add2(p0, h16_pair(sw + (uint32_t)((k + 0) * SW)));
            p1 = add2(p1, h16_pair(sw + (uint32_t)((k + 1) * SW)));
            p2 = add2(p2, h16_pair(sw + (uint32_t)((k + 2) * SW)));
            p3 = add2(p3, h16_pair(sw + (uint32_t)((k + 3) * SW)));
        }
#pragma unroll
        for (int k = Q - Q % 4; k < Q; ++k) p0 = add2(p0, h16_pair(sw + (uint32_t)(k * SW)));
        const float2 sum = unpack2(add2(add2(p0, p1), add2(p2, p3)));
        const float PhiA = sum.x * sr;
        const float PhiB = sum.y * sr;
        // the written array's scale inv_sw is a power of two, so it enters the
        // relaxation factor and the per-class terms exactly: the products
        // below are the stored values p / sc, bit for bit those of p * inv_sw
        const float om1w = c.om1 * sr * inv_sw;
        const f32x2 om2 = pack2(om1w, om1w);
        const float SxA = (float)((double)S2.x + a.soff);
        const float SxB = (float)((double)S2.y + a.soff);
        unsigned int* dst = B + (s >> 1);       // plane i's word of the pair, per velocity
        static_for<0, NC>([&](auto CI) {
            constexpr int cl = decltype(CI)::value;
            constexpr int i0 = cls_begin<L>(cl), i1 = cls_begin<L>(cl + 1);
            const f32x2 e = pack2(fmaf(c.wphi[cl], PhiA, c.chi[cl] * SxA) * inv_sw,
                                  fmaf(c.wphi[cl], PhiB, c.chi[cl] * SxB) * inv_sw);
#pragma unroll 4
            for (int i = i0; i < i1; ++i) {
                // p / sc of the written array
                const float2 q = unpack2(fma2(om2, h16_pair(sw + (uint32_t)(i * SW)), e));
                pmax = max3_abs(pmax, q.x, q.y);
                const __half2 h = __floats2half2_rn(q.x, q.y);
                __stcs(dst, *reinterpret_cast<const unsigned int*>(&h));
                dst += Vw;
            }
            // the class's slots take the next tile: its copies are in flight
            // while the other classes and the next tile's repack run
            if constexpr (AHEAD) {
                __syncwarp();
                if (more) static_for<i0, i1>(pull);
            }
        });
        if constexpr (!AHEAD) __syncwarp();   // the slots have been read
        if (a.mode != kPlain) {
            const double phA = (double)PhiA, phB = (double)PhiB;
            if (a.mode == kCheck) {
                const double2 old = *reinterpret_cast<const double2*>(a.Phi + s);
                const double dA = phA - old.x, dB = phB - old.y;
                rd2 += dA * dA;
                rd2 += dB * dB;
                rn2 += phA * phA;
                rn2 += phB * phB;
                rmx = fmax(rmx, fmax(fabs(dA), fabs(dB)));
                rms += phA;
                rms += phB;
            }
            *reinterpret_cast<double2*>(a.Phi + s) = make_double2(phA, phB);
        }
    }

    // pmax holds max |p| / sc (the stored magnitudes): back to max |p|, exactly
    pmax = pmax / inv_sw;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) pmax = fmaxf(pmax, __shfl_down_sync(0xffffffffu, pmax, o));
    if (lane == 0) mpart[sub] = pmax;
    if (a.mode == kCheck) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            rd2 += __shfl_down_sync(0xffffffffu, rd2, o);
            rn2 += __shfl_down_sync(0xffffffffu, rn2, o);
            rmx = fmax(rmx, __shfl_down_sync(0xffffffffu, rmx, o));
            rms += __shfl_down_sync(0xffffffffu, rms, o);
        }
        if (lane == 0) {
            rpart[sub][0] = rd2;
            rpart[sub][1] = rn2;
            rpart[sub][2] = rmx;
            rpart[sub][3] = rms;
        }
    }
    // a stored value beyond the binary16 range (it became +-inf) overflowed
    const int of = !(pmax * inv_sw <= 65504.f);
    if (__any_sync(0xffffffffu, of) && lane == 0) atomicOr(a.oflow, 1);
    __syncthreads();
    if (threadIdx.x == 0) {
        float m = 0.f;
        for (int k = 0; k < TILES; ++k) m = fmaxf(m, mpart[k]);
        atomicMax(a.pmax, __float_as_uint(m));
        if (a.mode == kCheck) {
            double t0 = 0.0, t1 = 0.0, t2 = 0.0, t3 = 0.0;
            for (int k = 0; k < TILES; ++k) {
                t0 += rpart[k][0];
                t1 += rpart[k][1];
                t2 = fmax(t2, rpart[k][2]);
                t3 += rpart[k][3];
            }
            a.partials[4 * blockIdx.x + 0] = t0;
            a.partials[4 * blockIdx.x + 1] = t1;
            a.partials[4 * blockIdx.x + 2] = t2;
            a.partials[4 * blockIdx.x + 3] = t3;
        }
    }
}

}  // namespace pkr

#include "pkr_sweep_h16w.cuh"

namespace pkr {

// binary16 forms (H16Form): one site per lane (any grid), two (nx a multiple of
// 64 and no edge below the reach; the plan checks), two with the next tile's
// copies in flight, four (nx a multiple of 128).  Tiles per block, measured at
// 256 x 256 x 192, D3Q111: two sites, copies ahead, 2 tiles and 6 blocks per SM
// 9.90 GLUPS, 7 blocks (128 registers) 9.25; four sites, 2 tiles 11.51, 1 tile
// 10.41, 3 tiles 11.30, 7 tiles 9.93.  When the plan takes which: see h16_form.
constexpr int kH16Tiles = 2;
template <class L>
constexpr size_t h16_smem(int form)
{
    return form == kH16Four  ? H16w<L>::smem_bytes(kH16Tiles)
           : form == kH16One ? (size_t)kH16Tiles * L::Q * 32 * 4
                             : (size_t)kH16Tiles * (L::Q * 33 * 4 + 32 * 4);
}
template <class L>
auto h16_kernel(int form)
{
    return form == kH16Four       ? sweep_h16w_kernel<L, kH16Tiles>
           : form == kH16TwoAhead ? sweep_h16p_kernel<L, kH16Tiles, 6, true>
           : form == kH16Two      ? sweep_h16p_kernel<L, kH16Tiles, 7, false>
                                  : sweep_h16_kernel<L, kH16Tiles>;
}

template <class L>
int launch_sweep_h16(int form, const SweepArgs& a, const void* coefs, int grid, void* stream)
{
    const Coefs<float>& c = *static_cast<const Coefs<float>*>(coefs);
    h16_kernel<L>(form)<<<grid, kH16Tiles * 32, h16_smem<L>(form), (cudaStream_t)stream>>>(a, c);
    return (int)cudaGetLastError();
}

template <class L>
int occupancy_h16(int form, int* blocks, int* tiles_per_block)
{
    const size_t smem = h16_smem<L>(form);
    auto kern = h16_kernel<L>(form);
    cudaError_t e = set_sweep_smem(kern, smem);
    if (e != cudaSuccess) return (int)e;
    // tiles_per_block counts 32-site tiles
    *tiles_per_block = h16_sites(form) * kH16Tiles;
    return (int)cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, kern, kH16Tiles * 32, smem);
}

}  // namespace pkr

#include "pkr_stencil.cuh"
#include "pkr_sweep_wide.cuh"
#include "pkr_sweep_pair.cuh"
#include "pkr_sweep_ws.cuh"
#include "pkr_resident.cuh"

namespace pkr {

template <class L, typename T, int K>
int launch_variant(const SweepArgs& a, const void* coefs, int grid, void* stream)
{
    using R = typename AccType<T>::type;
    constexpr Geo geo = Variants<L>::at(K);
    using ST = Staged<L, T, geo.G, geo.TILES>;
    auto kern = sweep_staged_kernel<L, T, geo.G, geo.TILES, false>;
    if constexpr (EarlyRefill<L, T, geo.G, geo.TILES>::value) {
        if (early_refill_pays<L>(a.ntiles, (int64_t)grid * geo.TILES))
            kern = sweep_staged_kernel<L, T, geo.G, geo.TILES, true>;
    }
    kern<<<grid, ST::WARPS * 32, ST::smem_bytes(), (cudaStream_t)stream>>>(
        a, *static_cast<const Coefs<R>*>(coefs));
    return (int)cudaGetLastError();
}

template <class L, typename T, int K>
int occupancy_variant(int* blocks, int* tiles_per_block)
{
    constexpr Geo geo = Variants<L>::at(K);
    using ST = Staged<L, T, geo.G, geo.TILES>;
    auto residency = [&](auto kern) {
        int b = 0;
        cudaError_t e = set_sweep_smem(kern, ST::smem_bytes());
        if (e == cudaSuccess)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kern, ST::WARPS * 32,
                                                              ST::smem_bytes());
        if (b < *blocks || *blocks == 0) *blocks = b;
        return e;
    };
    *tiles_per_block = geo.TILES;
    *blocks = 0;
    cudaError_t e = residency(sweep_staged_kernel<L, T, geo.G, geo.TILES, false>);
    if constexpr (EarlyRefill<L, T, geo.G, geo.TILES>::value)
        if (e == cudaSuccess) e = residency(sweep_staged_kernel<L, T, geo.G, geo.TILES, true>);
    return (int)e;
}

// Run-time dispatch over the compiled variants of (L, T): the staged
// geometries of Variants<L>, then the warp-specialised ones of WsVariants<L>.
template <class L, typename T>
int launch_sweep_t(int variant, const SweepArgs& a, const void* coefs, int grid, void* stream)
{
    int rc = (int)cudaErrorInvalidValue;
    static_for<0, Variants<L>::N>([&](auto K) {
        if (variant == decltype(K)::value)
            rc = launch_variant<L, T, decltype(K)::value>(a, coefs, grid, stream);
    });
    static_for<0, WsVariants<L>::N>([&](auto K) {
        if (variant == Variants<L>::N + decltype(K)::value)
            rc = launch_ws_variant<L, T, decltype(K)::value>(a, coefs, grid, stream);
    });
    static_for<0, PairVariant<L>::N>([&](auto K) {
        if (variant == Variants<L>::N + WsVariants<L>::N + decltype(K)::value)
            rc = launch_pair_variant<L, T, decltype(K)::value>(a, coefs, grid, stream);
    });
    return rc;
}

template <class L, typename T>
int occupancy_t(int variant, int* blocks, int* tiles_per_block)
{
    int rc = (int)cudaErrorInvalidValue;
    static_for<0, Variants<L>::N>([&](auto K) {
        if (variant == decltype(K)::value)
            rc = occupancy_variant<L, T, decltype(K)::value>(blocks, tiles_per_block);
    });
    static_for<0, WsVariants<L>::N>([&](auto K) {
        if (variant == Variants<L>::N + decltype(K)::value)
            rc = occupancy_ws_variant<L, T, decltype(K)::value>(blocks, tiles_per_block);
    });
    static_for<0, PairVariant<L>::N>([&](auto K) {
        if (variant == Variants<L>::N + WsVariants<L>::N + decltype(K)::value)
            rc = occupancy_pair_variant<L, T, decltype(K)::value>(blocks, tiles_per_block);
    });
    return rc;
}

// Variants of a plan's sweep (staged, warp-specialised, then the aligned x
// pairs, which need nx a multiple of 64 and every edge at least the reach)
// and of the batch sweep (staged only).
template <class L>
int variant_count_t() { return Variants<L>::N + WsVariants<L>::N + PairVariant<L>::N; }
// first aligned x-pairs variant (they are the last PairVariant<L>::N), or -1
template <class L>
int pair_variant_t() { return PairVariant<L>::N > 0 ? Variants<L>::N + WsVariants<L>::N : -1; }
template <class L>
int batch_variant_count_t() { return Variants<L>::N; }

#define PKR_INSTANTIATE_SWEEP(L)                                                             \
    template int launch_sweep_t<L, double>(int, const SweepArgs&, const void*, int, void*); \
    template int launch_sweep_t<L, long long>(int, const SweepArgs&, const void*, int, void*); \
    template int occupancy_t<L, long long>(int, int*, int*);                                 \
    template int launch_sweep_t<L, float>(int, const SweepArgs&, const void*, int, void*);  \
    template int occupancy_t<L, double>(int, int*, int*);                                    \
    template int occupancy_t<L, float>(int, int*, int*);                                     \
    template int variant_count_t<L>();                                                      \
    template int batch_variant_count_t<L>();                                                \
    template int pair_variant_t<L>();                                                       \
    template int launch_sweep_h16<L>(int, const SweepArgs&, const void*, int, void*);        \
    template int occupancy_h16<L>(int, int*, int*);                                          \
    template int launch_stencil<L>(const double*, double*, const double*, const Coefs<double>&,  \
                                   int64_t, int, int, int, int, int, double*, int, int, void*,  \
                                   const int*);                                                 \
    template int resident_form<L>(int64_t, int, int, int);                                   \
    template int launch_resident<L>(int, const CoopArgs&, const Coefs<double>&, void*);      \
    template int launch_batch_t<L, double>(int, BatchState*, int, int, int, void*);         \
    template int launch_batch_t<L, float>(int, BatchState*, int, int, int, void*);          \
    template int launch_batch_t<L, long long>(int, BatchState*, int, int, int, void*);      \
    template int batch_occupancy_t<L, double>(int, int*);                                    \
    template int batch_occupancy_t<L, long long>(int, int*);                                 \
    template int batch_occupancy_t<L, float>(int, int*);

}  // namespace pkr

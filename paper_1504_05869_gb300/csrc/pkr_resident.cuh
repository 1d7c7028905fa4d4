// pkr_resident.cuh -- runs of per-step-checked binary64 steps that stay on
// the GPU for the whole run (included by pkr_sweep.cuh).
//
// The solves that check every step are small (the paper's 1D lines, a 64 x 64
// plane): one step is a microsecond of work, and launching a sweep and a
// reduction per step, as kernels of a captured graph, took 10 to 20 us.  Here
// one launch runs thousands of steps.  Three forms, all with the arithmetic
// of the one-step kernels (the same Phi bit for bit):
//   stencil_block_kernel   scalar stencil, Phi in one block's shared memory
//   stencil_coop_kernel    scalar stencil, a 32-site tile per block, Phi in L2
//   sweep_coop_kernel      population sweep, a 32-site tile per block, the
//                          arrays in L2
// The last two are cooperative launches whose blocks meet once per step at a
// barrier in device memory.  The residual and the stopping rule are worked
// out behind the steps, off their critical path: a step or two later a warp
// that takes no part in the stencil decides, and the step's result is still
// there (in a third buffer, or in registers).  Whole solves, before and now:
// 64-site D1Q13 line at tau_lb = 1, 4200 steps, 39.2 -> 3.05 ms (5.9 with one
// checking warp); 64^2 D2Q169 at Kn 0.1, 208 steps, 4.6 -> 1.7 ms.
#pragma once

namespace pkr {

// Exponent far enough from the ends of the range that products of two such
// values (and 1e12 times them) are exact enough and do not over- or underflow.
__device__ __forceinline__ bool mid_range(double v)
{
    const int e = (__double2hiint(v) >> 20) & 0x7ff;
    return e > 1023 - 400 && e < 1023 + 400;
}

// a < b for non-negative finite values, on the integer pipe (a binary64
// comparison takes a slot and the latency of the slow binary64 pipe)
__device__ __forceinline__ bool below(double a, double b)
{
    return __double_as_longlong(a) < __double_as_longlong(b);
}

// The stopping rule of pkr_plan_run, one lane, from a check's sums: a =
// |dPhi|^2, b = |Phi|^2, mx = max |dPhi| (b and mx only for the max rule).
// The square roots and the division of the relative residual are left out
// where squares decide the comparisons beyond rounding: one product deep.
struct StopRule {
    int kind, nc, mid;
    double tol, thi, tlo;        // tol, and tol^2 a rounding margin up and down
    double amin, bmin, amin12;   // smallest residual so far: amin (max rule),
                                 // sqrt(amin / bmin); 1e12 amin

    __device__ static double rel(double a, double b)
    {
        return b > 0.0 ? sqrt(a) / sqrt(b) : (a == 0.0 ? 0.0 : INFINITY);
    }
    __device__ double residual(double a, double b, double mx) const
    {
        if (!(a == a) || !(b == b)) return NAN;
        return kind == PKR_TOL_MAX_ABS_DPHI ? mx : rel(a, b);
    }
    __device__ double smallest() const
    {
        return kind == PKR_TOL_MAX_ABS_DPHI ? amin : rel(amin, bmin);
    }
    __device__ void keep(double a, double b)
    {
        amin = a;
        bmin = b;
        amin12 = 1e12 * a;
        mid = kind != PKR_TOL_MAX_ABS_DPHI && mid_range(a) && mid_range(b) && mid_range(tol);
    }
    // 0: go on, 1: converged, 2: diverged
    __device__ int apply(double a, double b, double mx)
    {
        ++nc;
        if (mid && mid_range(a) && mid_range(b)) {
            const double l = a * bmin, r = amin * b, r12 = amin12 * b;
            const double hi = thi * b, lo = tlo * b;
            if (nc > 2 && below(r12, l)) return 2;
            if (below(l, r)) keep(a, b);
            if (below(hi, a)) return 0;
            if (below(a, lo)) return 1;
            return rel(a, b) < tol ? 1 : 0;
        }
        const double r = residual(a, b, mx), m = smallest();
        // (an infinite difference of finite densities comes with b = inf)
        if (!isfinite(b) || !(r == r) || (kind == PKR_TOL_MAX_ABS_DPHI && !isfinite(mx)) ||
            (nc > 2 && r > 1e6 * m && r > 1e-300))
            return 2;
        if (r < m) {
            if (kind == PKR_TOL_MAX_ABS_DPHI) keep(r, 1.0);
            else keep(a, a == 0.0 ? 1.0 : b);
        }
        return tol > 0.0 && r < tol ? 1 : 0;
    }
    __device__ void begin(const RunCtl* ctl, double tol_, int kind_)
    {
        kind = kind_;
        tol = tol_;
        thi = tol * tol * (1.0 + 1e-12);
        tlo = tol * tol * (1.0 - 1e-12);
        nc = ctl->nchecks;
        const double m = ctl->min_res;
        keep(kind == PKR_TOL_MAX_ABS_DPHI ? m : m * m, 1.0);
    }
    // verdict: 0 (ran out of steps), 1, 2; last: 1-based index of the last kept step
    __device__ void end(RunCtl* ctl, int verdict, int last, double res) const
    {
        ctl->stop = verdict != 0;
        ctl->status = verdict == 2 ? PKR_EDIVERGED : PKR_OK;
        ctl->done_at = last - 1;
        ctl->nchecks = nc;
        ctl->min_res = smallest();
        ctl->last_res = res;
    }
};

// Sums a and b (and the maximum mx) over the warp, to every lane; a only for
// the relative rule, mx only for the max rule.  The halves of the warp take
// one of the two sums each, and the maximum goes over the bit patterns.
__device__ __forceinline__ void warp_residual(double& a, double& b, double& mx, int kind)
{
    const bool up = (threadIdx.x & 16) != 0;
    if (kind == PKR_TOL_MAX_ABS_DPHI) {
        long long m = __double_as_longlong(mx);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            b += __shfl_xor_sync(0xffffffffu, b, o);
            const long long t = __shfl_xor_sync(0xffffffffu, m, o);
            m = t > m ? t : m;
        }
        mx = __longlong_as_double(m);
        return;
    }
    double v = up ? b : a;
    v += __shfl_xor_sync(0xffffffffu, up ? a : b, 16);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    a = __shfl_sync(0xffffffffu, v, 0);
    b = __shfl_sync(0xffffffffu, v, 16);
}

// ---------------------------------------------------------------------------
// One block: thread s < V owns site s; Phi of the last steps lives in a ring
// in shared memory.  The check of a step is a longer dependent chain than the
// step (sums over the block, five shuffles, the rule), so four more warps take
// the checks in turn, a step each, while the stencil warps go on: a verdict is
// waited for four steps later, before its buffer is reused.  Hand-offs are
// named barriers met in a fixed order: the stencil warps arrive at kDone + w
// when a step for checking warp w is whole and wait at kSeen + w for its
// verdict; the rule's running state passes from one checking warp to the next
// behind kNext + w.  Bound by the latency of a step's binary64 chain.
// ---------------------------------------------------------------------------
constexpr int kBlockWork = 8192;   // most velocities x sites (resident_form)
constexpr int kCheckers = 4;
// most sites of the one-block form
template <class L>
__host__ __device__ constexpr int block_sites()
{
    const int v = kBlockWork / L::Q / 32 * 32 + 32;
    return v < 512 ? v : 512;
}
constexpr int kRing = kCheckers + 2;

__device__ __forceinline__ void bar_wait(int id, int threads)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int threads)
{
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

template <class L>
__global__ void __launch_bounds__(block_sites<L>() + 32 * kCheckers, 1)
stencil_block_kernel(double* P0, double* P1, const double* __restrict__ St,
                     const Coefs<double> c, int V, int nx, int ny, int nz, int small, int nsteps,
                     double tol, int kind, RunCtl* ctl)
{
    constexpr int kStep = 1, kDone = 2, kSeen = kDone + kCheckers, kNext = kSeen + kCheckers;
    __shared__ double buf[kRing][block_sites<L>()];
    __shared__ int verdict[kCheckers];
    __shared__ StopRule state;      // passed along the checking warps
    __shared__ int stop_at;         // step the rule stopped at, 0: none yet
    const int tid = threadIdx.x, lane = tid & 31;
    const int nt = (int)blockDim.x - 32 * kCheckers;   // stencil threads
    if (tid < V) buf[0][tid] = P0[tid];
    if (tid == 0) {
        state.begin(ctl, tol, kind);
        stop_at = 0;
    }
    __syncthreads();
    if (tid < nt) {
        const bool valid = tid < V;
        Neighbours<L> nb;
        nb.locate(valid ? tid : 0, nx, ny, nz, small);
        const double st = valid ? St[tid] : 0.0;
        int last = 0, w = 0;              // w = step mod kCheckers
        int from = 0, to = 1;             // ring slots of steps j - 1 and j
        for (int j = 1;; ++j) {
            w = w + 1 == kCheckers ? 0 : w + 1;
            if (j > kCheckers) {
                bar_wait(kSeen + w, nt + 32);        // the check of step j - kCheckers
                last = j - kCheckers;
                if (verdict[w] != 0 || last == nsteps) break;
            }
            if (j <= nsteps) {
                const double* in = buf[from];
                if (valid) {
                    double p[kStencilParts];
                    static_for<0, kStencilParts>([&](auto J) {
                        constexpr int q = decltype(J)::value;
                        p[q] = stencil_part<L, q>(c, [&](auto I) {
                            return in[nb.template at<decltype(I)::value>()];
                        });
                    });
                    buf[to][tid] = ((p[0] + p[1]) + (p[2] + p[3])) + st;
                }
                bar_wait(kStep, nt);
                bar_arrive(kDone + w, nt + 32);
                from = to;
                to = to + 1 == kRing ? 0 : to + 1;
            }
        }
        if (valid) ((last & 1) ? P1 : P0)[tid] = buf[last % kRing][tid];
        return;
    }
    const int w = (tid - nt) >> 5;        // checks steps j with j mod kCheckers == w
    for (int j = w > 0 ? w : kCheckers; j <= nsteps; j += kCheckers) {
        bar_wait(kDone + w, nt + 32);
        const double* now = buf[j % kRing];
        const double* old = buf[(j - 1) % kRing];
        double a = 0.0, b = 0.0, mx = 0.0;
        for (int s = lane; s < V; s += 32) {
            const double v = now[s], d = v - old[s];
            b = fma(v, v, b);
            if (kind == PKR_TOL_MAX_ABS_DPHI) mx = fmax(mx, fabs(d));
            else a = fma(d, d, a);
        }
        warp_residual(a, b, mx, kind);
        if (j > 1) bar_wait(kNext + w, 64);
        const bool over = stop_at != 0;   // a step before this one has stopped the run
        int end = over ? stop_at : nsteps;
        if (!over) {
            StopRule r = state;
            const int v = r.apply(a, b, mx);       // every lane alike
            __syncwarp();
            if (lane == 0) {
                state = r;
                verdict[w] = v;
                if (v != 0) stop_at = j;
                if (v != 0 || j == nsteps) r.end(ctl, v, j, r.residual(a, b, mx));
            }
            if (v != 0) end = j;
            __syncwarp();
            bar_arrive(kSeen + w, nt + 32);
        }
        // after a stop the stencil warps still finish kCheckers - 1 steps
        if (end != nsteps || over) end = min(nsteps, end + kCheckers - 1);
        if (j + 1 <= end) bar_arrive(kNext + (w + 1 == kCheckers ? 0 : w + 1), 64);
        if (j + kCheckers > end) break;
    }
}

// ---------------------------------------------------------------------------
// The step barrier of a cooperative launch: every block's thread 0 of the
// caller adds 1 to the counter once the block's step is written (block 0 adds
// a stop bit as well when the rule has stopped the run) and waits for all.
// The stop bit is the barrier's own, by parity: a block still polling barrier
// k - 1 may see block 0's arrival at barrier k.
// Returns the counter (>= target), or 0 after the wait limit, which a
// co-resident grid never reaches: the launch then ends with an error status.
// ---------------------------------------------------------------------------
constexpr unsigned int kCountMask = 0x3fffffffu;
__host__ __device__ constexpr unsigned int stop_bit(int k) { return 0x40000000u << (k & 1); }
constexpr int kWaitLimit = 1 << 23;   // polls of at least 0.3 us each

__device__ __forceinline__ unsigned int step_barrier(unsigned int* counter, unsigned int add,
                                                     unsigned int target)
{
    __threadfence();
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(counter), "r"(add) : "memory");
    for (int w = 0; w < kWaitLimit; ++w) {
        unsigned int v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(counter) : "memory");
        if ((v & kCountMask) >= target) return v;
    }
    return 0u;
}

// What the checking warp of a block does in interval k (the time between
// step barriers k - 1 and k): it reduces the block's tile of step k - 1 to
// the tile's partial sums, and in block 0 sums all tiles of step k - 2 and
// applies the rule to them.  Returns the verdict on step k - 2 (block 0).
struct TileCheck {
    double2 (*val)[32];      // [2][32]: (Phi, dPhi) of the tile by step parity
    double* partials;        // [2][ntiles][4]
    int ntiles, nsteps, kind, lane;

    __device__ __forceinline__ void tile(int k) const
    {
        if (k < 2 || k - 1 > nsteps) return;
        const double2 w = val[(k - 1) & 1][lane];
        double a = kind == PKR_TOL_MAX_ABS_DPHI ? 0.0 : w.y * w.y, b = w.x * w.x, mx = fabs(w.y);
        warp_residual(a, b, mx, kind);
        if (lane == 0) {
            double* p = partials + 4 * ((size_t)((k - 1) & 1) * ntiles + blockIdx.x);
            __stcg(reinterpret_cast<double2*>(p), make_double2(a, b));
            __stcg(p + 2, mx);
        }
    }
    __device__ __forceinline__ int all(int k, StopRule& rule, double& res) const
    {
        if (k < 3 || k - 2 > nsteps) return 0;
        const double* p = partials + 4 * (size_t)((k - 2) & 1) * ntiles;
        double a = 0.0, b = 0.0, mx = 0.0;
#pragma unroll 4
        for (int t = lane; t < ntiles; t += 32) {
            const double2 ab = __ldcg(reinterpret_cast<const double2*>(p + 4 * t));
            a += ab.x;
            b += ab.y;
            mx = fmax(mx, __ldcg(p + 4 * t + 2));
        }
        warp_residual(a, b, mx, kind);
        const int v = rule.apply(a, b, mx);      // every lane alike
        if (v != 0 || k - 2 == nsteps) res = rule.residual(a, b, mx);
        return v;
    }
};

// End of interval k, in the checking warp: block 0's verdict goes with its
// arrival; stop (shared) tells the block what the barrier returned.
__device__ __forceinline__ void interval_end(const CoopArgs& a, int k, int lane, int verdict,
                                             int* stop)
{
    if (lane == 0) {
        const unsigned int v = step_barrier(a.counter, 1u | (verdict ? stop_bit(k) : 0u),
                                            (unsigned int)k * gridDim.x);
        *stop = v == 0u ? 2 : (v & stop_bit(k)) ? 1 : 0;
    }
}

// ---------------------------------------------------------------------------
// Scalar stencil, one 32-site tile per block: four warps take a part of the
// sum each, warp 0 adds them up, warp 4 checks.  The verdict on step m comes
// with barrier m + 2; warp 0 keeps Phi of the last three steps of its sites
// in registers and puts step m's back.
// ---------------------------------------------------------------------------
template <class L>
__global__ void __launch_bounds__(160, 4)
stencil_coop_kernel(const CoopArgs a, const Coefs<double> c)
{
    __shared__ double parts[kStencilParts][32];
    __shared__ double2 val[2][32];
    __shared__ int stop;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t s64 = (int64_t)blockIdx.x * 32 + lane;
    const bool valid = s64 < a.V;
    const int s = valid ? (int)s64 : 0;
    Neighbours<L> nb;
    nb.locate(s, a.nx, a.ny, a.nz, a.small);
    double v0 = 0.0, v1 = 0.0, v2 = 0.0, st = 0.0;
    if (warp == 0 && valid) {
        v0 = __ldcg(a.P[0] + s);
        st = a.S[s];
    }
    StopRule rule;
    rule.begin(a.ctl, a.tol, a.kind);
    double res = 0.0;
    const TileCheck tc{val, a.partials, (int)gridDim.x, a.nsteps, a.kind, lane};
    double *in = a.P[0], *out = a.P[1];
    int k = 1, verdict = 0, halt = 0;
    for (; k <= a.nsteps + 2; ++k) {
        if (warp < kStencilParts) {
            const bool step = k <= a.nsteps;
            nb.hold();
            if (step) {
                static_for<0, kStencilParts>([&](auto J) {
                    constexpr int j = decltype(J)::value;
                    if (warp == j)
                        parts[j][lane] = stencil_part<L, j>(c, [&](auto I) {
                            return __ldcg(in + nb.template at<decltype(I)::value>());
                        });
                });
                asm volatile("bar.sync 1, 128;" ::: "memory");
            }
            if (warp == 0) {
                v2 = v1;
                v1 = v0;
                if (step) {
                    v0 = ((parts[0][lane] + parts[1][lane]) + (parts[2][lane] + parts[3][lane])) +
                         st;
                    if (valid) __stcg(out + s, v0);
                    val[k & 1][lane] = valid ? make_double2(v0, v0 - v1) : make_double2(0.0, 0.0);
                }
            }
        } else {
            tc.tile(k);
            if (blockIdx.x == 0) verdict = tc.all(k, rule, res);
        }
        __syncthreads();
        if (warp == kStencilParts) interval_end(a, k, lane, verdict, &stop);
        __syncthreads();
        halt = stop;
        if (halt) break;
        double* t = in;
        in = out;
        out = t;
    }
    const int last = halt ? k - 2 : a.nsteps;
    // stopped at barrier k: v2 is step k - 2, whose array (out) step k has overwritten
    if (halt == 1 && warp == 0 && valid) __stcg(out + s, v2);
    if (blockIdx.x == 0 && warp == kStencilParts && lane == 0) {
        rule.end(a.ctl, verdict, last, res);
        if (halt == 2) a.ctl->status = PKR_ECUDA;
    }
}

// ---------------------------------------------------------------------------
// Population sweep, one 32-site tile per block: G warps hold Q / G of the
// tile's pulled values each in registers (loaded from L2 in one go), exchange
// the exponent, the exact density sum and the classes' equilibrium-plus-source
// terms, relax and store; warp G checks.  Three population arrays, so that the
// array of step m is whole when the verdict on it comes with barrier m + 2.
//
// A step is run once by each warp, so its code is one for all warps: with the
// velocities as compile-time constants eight warps fetched eight copies of it
// every step (64^2 D2Q169: 10.7 us a step, 6.5 us now; the barrier alone takes
// 1.3 us, with the step's loads and stores 3.7 us).
// ---------------------------------------------------------------------------
template <class L>
struct Coop {
    static constexpr int G = L::Q > 64 ? 15 : L::Q > 16 ? 3 : 1;   // and one that checks
    static constexpr int N = (L::Q + G - 1) / G;   // values of a warp
    static constexpr int THREADS = 32 * G + 32;
};

// fixed_sum of N values in registers
template <int GB, int N>
__device__ __forceinline__ long long fixed_sum_regs(const double (&v)[N], int emax)
{
    static_assert((N + 3) / 4 < (1 << (9 - GB)), "fixed-point partial may overflow");
    long long s[4] = {0, 0, 0, 0};
    int p[4] = {0, 0, 0, 0};
#pragma unroll
    for (int k = 0; k < N; ++k) {
        const long long t = fixed_term2<GB>(v[k], emax);
        s[k % 4] += t;
        p[k % 4] += (int)(t & 1);
    }
    return ((s[0] + p[0]) >> 1) + ((s[1] + p[1]) >> 1) + ((s[2] + p[2]) >> 1) +
           ((s[3] + p[3]) >> 1);
}

template <class L>
__global__ void __launch_bounds__(Coop<L>::THREADS, 2)
sweep_coop_kernel(const CoopArgs a, const Coefs<double> c)
{
    constexpr int Q = L::Q, G = Coop<L>::G, N = Coop<L>::N;
    constexpr int GB = 63 - 53 - ceil_log2(Q);
    constexpr int NC = ncls_of<L>();
    __shared__ long long xacc[G][32];
    __shared__ int xexp[G][32];
    __shared__ double eterm[NC][32];       // equilibrium-plus-source term per class
    __shared__ double2 val[2][32];
    __shared__ int stop;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t s64 = (int64_t)blockIdx.x * 32 + lane;
    const bool valid = s64 < a.V;
    const int s = valid ? (int)s64 : 0;
    const int V = (int)a.V;
    // this warp's velocities: element offsets of the pulled values (Q V fits
    // in 31 bits, see resident_form) and shared-memory offsets of their
    // classes' terms; -1 past the set
    int from[N], term[N];
    {
        Neighbours<L> nb;
        nb.locate(s, a.nx, a.ny, a.nz, a.small);
#pragma unroll
        for (int j = 0; j < N; ++j) from[j] = term[j] = -1;
        static_for<0, Q>([&](auto I) {
            constexpr int i = decltype(I)::value;
            if (warp == i / N) {
                from[i % N] = i * V + nb.template at<i>();
                term[i % N] = cls_of<L>(i) * 32 + lane;
            }
        });
    }
    const double Sx = valid ? a.S[s] : 0.0;
    double v0 = warp == 0 && valid ? a.Phi[s] : 0.0, v1 = 0.0, v2 = 0.0;
    StopRule rule;
    rule.begin(a.ctl, a.tol, a.kind);
    double res = 0.0;
    const TileCheck tc{val, a.partials, (int)gridDim.x, a.nsteps, a.kind, lane};
    double *A = a.P[0], *B = a.P[1], *M = a.P[2];   // read, written, next to write
    int k = 1, verdict = 0, halt = 0;
    for (; k <= a.nsteps + 2; ++k) {
        if (warp < G) {
            v2 = v1;
            v1 = v0;
            if (k <= a.nsteps) {
                double v[N];
#pragma unroll
                for (int j = 0; j < N; ++j) v[j] = from[j] >= 0 ? __ldcg(A + from[j]) : 0.0;
                int emax = 0;
#pragma unroll
                for (int j = 0; j < N; ++j) emax = max(emax, __double2hiint(v[j]) & 0x7fffffff);
                emax >>= 20;
                if constexpr (G > 1) {
                    xexp[warp][lane] = emax;
                    asm volatile("bar.sync 1, %0;" ::"n"(G * 32) : "memory");
#pragma unroll
                    for (int q = 0; q < G; ++q) emax = max(emax, xexp[q][lane]);
                }
                const bool plain = plain_path(emax);
                long long part;
                if (plain) {
                    double t = 0.0;
#pragma unroll
                    for (int j = 0; j < N; ++j) t += v[j];
                    part = __double_as_longlong(t);
                } else {
                    part = fixed_sum_regs<GB, N>(v, emax);
                }
                double Phi;
                if constexpr (G > 1) {
                    xacc[warp][lane] = part;
                    asm volatile("bar.sync 1, %0;" ::"n"(G * 32) : "memory");
                    if (plain) {
                        double t = 0.0;
#pragma unroll
                        for (int q = 0; q < G; ++q) t += __longlong_as_double(xacc[q][lane]);
                        Phi = t;
                    } else {
                        long long t = 0;
#pragma unroll
                        for (int q = 0; q < G; ++q) t += xacc[q][lane];
                        Phi = fixed_value<GB>(t, emax);
                    }
                } else {
                    Phi = plain ? __longlong_as_double(part) : fixed_value<GB>(part, emax);
                }
                for (int cl = warp; cl < NC; cl += G)
                    eterm[cl][lane] = fma(c.wphi[cl], Phi, c.chi[cl] * Sx);
                if constexpr (G > 1) asm volatile("bar.sync 1, %0;" ::"n"(G * 32) : "memory");
                else __syncwarp();
                double* dst = B + (int64_t)warp * N * V + s;
#pragma unroll
                for (int j = 0; j < N; ++j) {
                    if (valid && term[j] >= 0)
                        __stcg(dst, fma(c.om1, v[j], (&eterm[0][0])[term[j]]));
                    dst += V;
                }
                v0 = Phi;
                if (warp == 0)
                    val[k & 1][lane] = valid ? make_double2(Phi, Phi - v1) : make_double2(0.0, 0.0);
            }
        } else {
            tc.tile(k);
            if (blockIdx.x == 0) verdict = tc.all(k, rule, res);
        }
        __syncthreads();
        if (warp == G) interval_end(a, k, lane, verdict, &stop);
        __syncthreads();
        halt = stop;
        if (halt) break;
        double* t = A;
        A = B;
        B = M;
        M = t;
    }
    // stopped at barrier k: the verdict was on step k - 2, whose density is
    // v2; out of steps: two intervals past the last step it is v2 too
    const int last = halt ? k - 2 : a.nsteps;
    if (warp == 0 && valid) a.Phi[s] = v2;
    if (blockIdx.x == 0 && warp == G && lane == 0) {
        rule.end(a.ctl, verdict, last, res);
        if (halt == 2) a.ctl->status = PKR_ECUDA;
    }
}

// Form of a resident run: 0 none, 1 stencil in one block, 2 stencil over
// blocks, 3 sweep over blocks.  One block while its binary64 work per step
// (Q operations per site at 16 clocks per warp) stays under the cost of the
// step barrier (about 2 us): Q V <= kBlockWork.  The other forms take a tile per
// block, all of them on the GPU at once (a cooperative launch must be), and
// no more than `most` tiles: beyond that the one-step kernels fill the GPU.
template <class L>
int resident_form(int64_t V, int stencil, int nsm, int most)
{
    if (stencil && V <= block_sites<L>() && V * L::Q <= kBlockWork) return 1;
    const int64_t tiles = (V + 31) / 32;
    int bps = 0;
    if (tiles > most || (int64_t)L::Q * V > 0x7fffffff) return 0;
    const cudaError_t e =
        stencil ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, stencil_coop_kernel<L>, 160, 0)
                : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, sweep_coop_kernel<L>,
                                                                Coop<L>::THREADS, 0);
    if (e != cudaSuccess || tiles > (int64_t)bps * nsm) return 0;
    return stencil ? 2 : 3;
}

template <class L>
int launch_resident(int form, const CoopArgs& a, const Coefs<double>& c, void* stream)
{
    cudaStream_t st = (cudaStream_t)stream;
    if (form == 1) {
        const int threads = 32 * (int)((a.V + 31) / 32) + 32 * kCheckers;
        stencil_block_kernel<L><<<1, threads, 0, st>>>(a.P[0], a.P[1], a.S, c, (int)a.V, a.nx,
                                                       a.ny, a.nz, a.small, a.nsteps, a.tol,
                                                       a.kind, a.ctl);
        return (int)cudaGetLastError();
    }
    const int grid = (int)((a.V + 31) / 32);
    void* args[2] = {const_cast<CoopArgs*>(&a), const_cast<Coefs<double>*>(&c)};
    if (form == 2)
        return (int)cudaLaunchCooperativeKernel(stencil_coop_kernel<L>, dim3(grid), dim3(160),
                                                args, 0, st);
    return (int)cudaLaunchCooperativeKernel(sweep_coop_kernel<L>, dim3(grid),
                                            dim3(Coop<L>::THREADS), args, 0, st);
}

}  // namespace pkr

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
// 64-site D1Q13 line at tau_lb = 1, 4200 steps, 38.8 -> 5.9 ms; 64^2 D2Q169
// at Kn 0.1, 208 steps, 4.6 -> 3.1 ms.
#pragma once

namespace pkr {

// Exponent far enough from the ends of the range that products of two such
// values (and 1e12 times them) are exact enough and do not over- or underflow.
__device__ __forceinline__ bool mid_range(double v)
{
    const int e = (__double2hiint(v) >> 20) & 0x7ff;
    return e > 1023 - 400 && e < 1023 + 400;
}

// The stopping rule of pkr_plan_run, one lane, from a check's sums: a =
// |dPhi|^2, b = |Phi|^2, mx = max |dPhi| (b and mx only for the max rule).
// The square roots and the division of the relative residual are left out
// where squares decide the comparisons beyond rounding.
struct StopRule {
    int kind, nc;
    double tol;
    double amin, bmin;   // smallest residual so far: amin (max rule), sqrt(amin / bmin)

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
    // 0: go on, 1: converged, 2: diverged
    __device__ int apply(double a, double b, double mx)
    {
        ++nc;
        if (kind != PKR_TOL_MAX_ABS_DPHI && mid_range(a) && mid_range(b) && mid_range(amin) &&
            mid_range(bmin) && mid_range(tol)) {
            const double l = a * bmin, r = amin * b;
            if (nc > 2 && l > 1e12 * r) return 2;
            if (l < r) {
                amin = a;
                bmin = b;
            }
            const double t = tol * tol * b;
            if (a > t * (1.0 + 1e-12)) return 0;
            if (a < t * (1.0 - 1e-12)) return 1;
            return rel(a, b) < tol ? 1 : 0;
        }
        const double r = residual(a, b, mx), m = smallest();
        // (an infinite difference of finite densities comes with b = inf)
        if (!isfinite(b) || !(r == r) || (kind == PKR_TOL_MAX_ABS_DPHI && !isfinite(mx)) ||
            (nc > 2 && r > 1e6 * m && r > 1e-300))
            return 2;
        if (r < m) {
            amin = kind == PKR_TOL_MAX_ABS_DPHI ? r : a;
            bmin = kind == PKR_TOL_MAX_ABS_DPHI || a == 0.0 ? 1.0 : b;
        }
        return tol > 0.0 && r < tol ? 1 : 0;
    }
    __device__ void begin(const RunCtl* ctl, double tol_, int kind_)
    {
        kind = kind_;
        tol = tol_;
        nc = ctl->nchecks;
        const double m = ctl->min_res;
        amin = kind == PKR_TOL_MAX_ABS_DPHI ? m : m * m;
        bmin = 1.0;
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

__device__ __forceinline__ void warp_residual(double& a, double& b, double& mx, int kind)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        b += __shfl_xor_sync(0xffffffffu, b, o);
        if (kind == PKR_TOL_MAX_ABS_DPHI) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        else a += __shfl_xor_sync(0xffffffffu, a, o);
    }
}

// ---------------------------------------------------------------------------
// One block: thread s < V owns site s, Phi of the last three steps lives in
// shared memory, one barrier per step.  The block's last warp checks step
// k - 1 while the others compute step k.  Bound by the binary64 pipe: Q
// operations per site plus about 20 per 32 sites for the check, 16 clocks
// each per warp.
// ---------------------------------------------------------------------------
constexpr int kBlockSites = 512;

template <class L>
__global__ void __launch_bounds__(kBlockSites + 32)
stencil_block_kernel(double* P0, double* P1, const double* __restrict__ St,
                     const Coefs<double> c, int V, int nx, int ny, int nz, int small, int nsteps,
                     double tol, int kind, RunCtl* ctl)
{
    __shared__ double buf[3][kBlockSites];
    __shared__ int verdict[2];
    const int tid = threadIdx.x;
    const int nw = (blockDim.x >> 5) - 1;          // stencil warps
    const bool checker = (tid >> 5) == nw;
    const int lane = tid & 31;
    const bool valid = !checker && tid < V;
    Neighbours<L> nb;
    nb.locate(valid ? tid : 0, nx, ny, nz, small);
    const double st = valid ? St[tid] : 0.0;
    if (valid) buf[0][tid] = P0[tid];
    StopRule rule;
    rule.begin(ctl, tol, kind);
    double res = 0.0, a = 0.0, b = 0.0, mx = 0.0;
    // step k's verdict (lane 0 of the checking warp)
    auto check = [&](int k) {
        const double* now = buf[k % 3];
        const double* old = buf[(k + 2) % 3];
        a = b = mx = 0.0;
        for (int s = lane; s < V; s += 32) {
            const double v = now[s], d = v - old[s];
            b = fma(v, v, b);
            if (kind == PKR_TOL_MAX_ABS_DPHI) mx = fmax(mx, fabs(d));
            else a = fma(d, d, a);
        }
        warp_residual(a, b, mx, kind);
        if (lane == 0) verdict[k & 1] = rule.apply(a, b, mx);
    };
    __syncthreads();
    int k = 1, stopped = 0;
    for (; k <= nsteps; ++k) {
        if (checker) {
            if (k > 1) check(k - 1);
        } else if (valid) {
            const double* in = buf[(k + 2) % 3];
            double p[kStencilParts];
            static_for<0, kStencilParts>([&](auto J) {
                constexpr int j = decltype(J)::value;
                p[j] = stencil_part<L, j>(c, [&](auto I) {
                    return in[nb.template at<decltype(I)::value>()];
                });
            });
            buf[k % 3][tid] = ((p[0] + p[1]) + (p[2] + p[3])) + st;
        }
        __syncthreads();
        if (k > 1 && verdict[(k - 1) & 1]) {
            stopped = verdict[(k - 1) & 1];
            break;
        }
    }
    int last = k - 1;              // stopped at k: step k - 1 is the last one kept
    if (!stopped) {
        last = nsteps;
        if (checker) check(nsteps);
        __syncthreads();
        stopped = verdict[nsteps & 1];
    }
    if (valid) ((last & 1) ? P1 : P0)[tid] = buf[last % 3][tid];
    if (checker && lane == 0) rule.end(ctl, stopped, last, rule.residual(a, b, mx));
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
__global__ void __launch_bounds__(160)
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
// the exponent and the exact density sum as the staged sweep does, relax and
// store; warp G checks.  Three population arrays, so that the array of step m
// is whole when the verdict on it comes with barrier m + 2.
// ---------------------------------------------------------------------------
template <class L>
struct Coop {
    static constexpr int G = L::Q > 64 ? 8 : L::Q > 16 ? 2 : 1;
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
__global__ void __launch_bounds__(Coop<L>::THREADS)
sweep_coop_kernel(const CoopArgs a, const Coefs<double> c)
{
    constexpr int G = Coop<L>::G;
    constexpr int GB = 63 - 53 - ceil_log2(L::Q);
    constexpr int NC = ncls_of<L>();
    __shared__ long long xacc[G][32];
    __shared__ int xexp[G][32];
    __shared__ double2 val[2][32];
    __shared__ int stop;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t s64 = (int64_t)blockIdx.x * 32 + lane;
    const bool valid = s64 < a.V;
    const int s = valid ? (int)s64 : 0;
    const int64_t V = a.V;
    Neighbours<L> nb;
    nb.locate(s, a.nx, a.ny, a.nz, a.small);
    const double Sx = valid ? a.S[s] : 0.0;
    double v0 = warp == 0 && valid ? a.Phi[s] : 0.0, v1 = 0.0, v2 = 0.0;
    StopRule rule;
    rule.begin(a.ctl, a.tol, a.kind);
    double res = 0.0;
    const TileCheck tc{val, a.partials, (int)gridDim.x, a.nsteps, a.kind, lane};
    double *A = a.P[0], *B = a.P[1], *N = a.P[2];   // read, written, next to write
    int k = 1, verdict = 0, halt = 0;
    for (; k <= a.nsteps + 2; ++k) {
        if (warp < G) {
            if (warp == 0) {
                v2 = v1;
                v1 = v0;
            }
            if (k <= a.nsteps) {
                static_for<0, G>([&](auto GI) {
                    constexpr int g = decltype(GI)::value;
                    constexpr int lo = g * L::Q / G, hi = (g + 1) * L::Q / G, n = hi - lo;
                    if (warp != g) return;
                    double v[n];
                    static_for<lo, hi>([&](auto I) {
                        constexpr int i = decltype(I)::value;
                        v[i - lo] = __ldcg(A + ((int64_t)i * V + nb.template at<i>()));
                    });
                    int emax = 0;
#pragma unroll
                    for (int q = 0; q < n; ++q)
                        emax = max(emax, __double2hiint(v[q]) & 0x7fffffff);
                    emax >>= 20;
                    if constexpr (G > 1) {
                        xexp[g][lane] = emax;
                        asm volatile("bar.sync 1, %0;" ::"n"(G * 32) : "memory");
#pragma unroll
                        for (int q = 0; q < G; ++q) emax = max(emax, xexp[q][lane]);
                    }
                    const bool plain = plain_path(emax);
                    long long part;
                    if (plain) {
                        double t = 0.0;
#pragma unroll
                        for (int q = 0; q < n; ++q) t += v[q];
                        part = __double_as_longlong(t);
                    } else {
                        part = fixed_sum_regs<GB, n>(v, emax);
                    }
                    double Phi;
                    if constexpr (G > 1) {
                        xacc[g][lane] = part;
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
                    if (valid) {
                        static_for<0, NC>([&](auto CI) {
                            constexpr int cl = decltype(CI)::value;
                            constexpr int cb = cls_begin<L>(cl), ce = cls_begin<L>(cl + 1);
                            constexpr int i0 = cb > lo ? cb : lo, i1 = ce < hi ? ce : hi;
                            if constexpr (i0 < i1) {
                                const double e = fma(c.wphi[cl], Phi, c.chi[cl] * Sx);
#pragma unroll
                                for (int i = i0; i < i1; ++i)
                                    __stcg(B + ((int64_t)i * V + s), fma(c.om1, v[i - lo], e));
                            }
                        });
                    }
                    if constexpr (g == 0) {
                        v0 = Phi;
                        val[k & 1][lane] =
                            valid ? make_double2(Phi, Phi - v1) : make_double2(0.0, 0.0);
                    }
                });
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
        B = N;
        N = t;
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
// step barrier (about 2 us): Q V <= 8192.  The other forms take a tile per
// block, all of them on the GPU at once (a cooperative launch must be), and
// no more than `most` tiles: beyond that the one-step kernels fill the GPU.
template <class L>
int resident_form(int64_t V, int stencil, int nsm, int most)
{
    if (stencil && V <= kBlockSites && V * L::Q <= 8192) return 1;
    const int64_t tiles = (V + 31) / 32;
    int bps = 0;
    if (tiles > most) return 0;
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
        const int threads = 32 * (int)((a.V + 31) / 32) + 32;
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

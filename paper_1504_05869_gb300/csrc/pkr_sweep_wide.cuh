// pkr_sweep_wide.cuh -- the aligned x-pairs sweep of binary32 storage with
// two sites per lane (included by pkr_sweep.cuh; same step and arithmetic, in
// the same order, as the two velocity groups of sweep_pair_kernel<L, float>).
//
// What holds the narrow storages is the number of memory requests: a copy of
// the sweep's planes reaches 6.2 TB/s in 8-byte lanes, 5.5 in 4-byte and 4.2
// in 2-byte ones, a warp's 32 lanes making one request whatever they carry.
// Here a warp owns 64 sites of an x row and a velocity group, a lane two
// adjacent sites: 8-byte copies, shared-memory reads and stores.  The rows
// hold the aligned run x0 .. x0 + 63 unshifted, with 4 values of halo on the
// side v_x needs, and are read at x - v_x: one 8-byte read for an even v_x,
// two 4-byte ones for an odd one.  The rows are the warp's own (no barrier but
// the density exchange of the two groups), and a class's rows take the next
// pair's copies as soon as it is relaxed.
#pragma once

namespace pkr {

template <class L>
struct Wide {
    static constexpr int Q = L::Q;
    static constexpr int G = 2;
    static constexpr int HL = (reach_of<L>() + 3) / 4 * 4;   // halo values per side
    static constexpr int RL = 64 + 2 * HL;
    static constexpr int ROWB = RL * 4;
    // 64-site pairs per block: one block of 12 warps per SM.  Measured on D3Q111
    // (D2Q81 takes the same; D2Q169's rows leave room for 3).  GB/s at 192^3 and
    // 256 x 256 x 160: 6 pairs 5905 / 5807, 4 pairs 5898 / 5748 (8
    // warps), 3 pairs x 2 blocks 5713 / 5697, 2 pairs x 3 blocks 4877 / 4875,
    // 7 pairs 4631 / 4570 (too little of the SM left for L1).
    static constexpr int PAIRS = L::Q > 111 ? 3 : 6;
    static constexpr int THREADS = PAIRS * G * 32;
    static constexpr size_t smem_bytes() { return (size_t)PAIRS * Q * ROWB; }
};

__device__ __forceinline__ f32x2 lds_2f32(uint32_t addr)
{
    f32x2 v;
    asm volatile("ld.shared.b64 %0, [%1];" : "=l"(v) : "r"(addr));
    return v;
}
// The two values of a lane at row position a (in floats from the row's
// start), a even at compile time or not.
template <bool EVEN>
__device__ __forceinline__ f32x2 row_pair(uint32_t addr)
{
    if constexpr (EVEN) return lds_2f32(addr);
    else return pack2(lds_f32(addr), lds_f32(addr + 4));
}

template <class L>
__global__ void __launch_bounds__(Wide<L>::THREADS, 1)
sweep_wide_kernel(const SweepArgs a, const Coefs<float> c)
{
    if (a.stop != nullptr && *a.stop != 0) return;   // the run stopped before this step
    using WD = Wide<L>;
    constexpr int Q = L::Q, G = WD::G, HL = WD::HL, ROWB = WD::ROWB, PAIRS = WD::PAIRS;
    constexpr int RC = reach_of<L>(), W = 2 * RC + 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double rpart[PAIRS][4];
    // per-group partial densities, two sets used by turns
    __shared__ float2 xacc[2][PAIRS][G][32];

    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    const int grp = wib % G, sub = wib / G;
    const float* __restrict__ A = static_cast<const float*>(a.A);
    float* __restrict__ B = static_cast<float*>(a.B);
    const float* __restrict__ S = static_cast<const float*>(a.S);
    const int64_t V = a.V;
    const int nx = a.nx, ny = a.ny, nz = a.nz, nxy = nx * ny;
    const int npairs = (int)(V >> 6);
    const int nt = gridDim.x * PAIRS;
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(smem_raw) + (uint32_t)(sub * Q * ROWB);
    double rd2 = 0.0, rn2 = 0.0, rmx = 0.0, rms = 0.0;

    static_for<0, G>([&](auto GI) {
        constexpr int g = decltype(GI)::value;
        constexpr int lo = g * Q / G, hi = (g + 1) * Q / G, n = hi - lo;
        if (grp != g) return;
        // the pair whose rows are being filled
        int yo[W], zo[W], x0 = 0, xl = 0, xr = 0;
        auto locate = [&](int p) {
            const int s0 = p * 64;
            const int r = (int)((unsigned)s0 / (unsigned)nx);
            x0 = s0 - r * nx;
            const int z = (int)((unsigned)r / (unsigned)ny);
            const int y = r - z * ny;
            static_for<0, W>([&](auto DI) {
                constexpr int d = decltype(DI)::value - RC;
                yo[d + RC] = wrap_off<d>(y, ny) * nx;
                zo[d + RC] = wrap_off<d>(z, nz) * nxy;
            });
            xl = (x0 > 0 ? x0 : nx) - HL + lane;
            xr = (x0 + 64 < nx ? x0 + 64 : 0) + lane;
        };
        const int nbytes = a.zero_in ? 0 : 8, hbytes = a.zero_in ? 0 : 4;
        auto pull = [&](auto I) {
            constexpr int i = decltype(I)::value;
            constexpr int vx = vx_of<L>(i);
            const float* row = A + ((int64_t)i * V + (zo[vz_of<L>(i) + RC] + yo[vy_of<L>(i) + RC]));
            const uint32_t rb = base + (uint32_t)(i * ROWB);
            cp_async<8>(rb + (uint32_t)((HL + 2 * lane) * 4), row + (x0 + 2 * lane), nbytes);
            if constexpr (vx > 0) {
                if (lane < HL) cp_async<4>(rb + (uint32_t)(lane * 4), row + xl, hbytes);
            } else if constexpr (vx < 0) {
                if (lane < HL) cp_async<4>(rb + (uint32_t)((HL + 64 + lane) * 4), row + xr, hbytes);
            }
        };
        // this lane's two values of velocity i
        auto value = [&](auto I) {
            constexpr int i = decltype(I)::value;
            constexpr int vx = vx_of<L>(i);
            return row_pair<vx % 2 == 0>(base +
                                         (uint32_t)(i * ROWB + (HL + 2 * lane - vx) * 4));
        };
        int pr = blockIdx.x * PAIRS + sub;
        if (pr < npairs) {
            locate(pr);
            static_for<lo, hi>(pull);
        }
        int par = 0;
        for (; pr < npairs; pr += nt, par ^= 1) {
            const int s = pr * 64 + 2 * lane;
            const float2 S2 = *reinterpret_cast<const float2*>(S + s);
            const bool more = pr + nt < npairs;
            if (more) locate(pr + nt);
            cp_async_wait_all();
            __syncwarp();   // a lane reads values its neighbours copied
            f32x2 p[4] = {0, 0, 0, 0};
            static_for<lo, hi>([&](auto I) {
                constexpr int k = decltype(I)::value - lo;
                constexpr int q = k < n - n % 4 ? k % 4 : 0;
                p[q] = add2(p[q], value(I));
            });
            xacc[par][sub][g][lane] = unpack2(add2(add2(p[0], p[1]), add2(p[2], p[3])));
            asm volatile("bar.sync %0, %1;" ::"r"(1 + sub), "n"(G * 32) : "memory");
            f32x2 sum = 0;
#pragma unroll
            for (int k = 0; k < G; ++k) {
                const float2 t = xacc[par][sub][k][lane];
                sum = add2(sum, pack2(t.x, t.y));
            }
            const float2 Phi = unpack2(sum);
            const float Sa = (float)((double)S2.x + a.soff), Sb = (float)((double)S2.y + a.soff);
            const f32x2 om1 = pack2(c.om1, c.om1);
            static_for<cls_of<L>(lo), cls_of<L>(hi - 1) + 1>([&](auto CI) {
                constexpr int cl = decltype(CI)::value;
                constexpr int cb = cls_begin<L>(cl), ce = cls_begin<L>(cl + 1);
                constexpr int i0 = cb > lo ? cb : lo, i1 = ce < hi ? ce : hi;
                const f32x2 e = pack2(fmaf(c.wphi[cl], Phi.x, c.chi[cl] * Sa),
                                      fmaf(c.wphi[cl], Phi.y, c.chi[cl] * Sb));
                static_for<i0, i1>([&](auto I) {
                    constexpr int i = decltype(I)::value;
                    const float2 q = unpack2(fma2(om1, value(I), e));
                    __stcs(reinterpret_cast<float2*>(B + ((int64_t)i * V + s)), q);
                });
                __syncwarp();   // every lane has read the class's rows
                if (more) static_for<i0, i1>(pull);
            });
            if (g == 0 && a.mode != kPlain) {
                const double phA = (double)Phi.x, phB = (double)Phi.y;
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
    });
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
            for (int k = 0; k < PAIRS; ++k) {
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

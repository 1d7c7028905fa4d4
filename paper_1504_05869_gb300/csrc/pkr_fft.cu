// pkr_fft.cu -- the scheme's exact fixed point by FFT (a direct comparator).
//
// The kinetic relaxation scheme is linear and translation invariant on the
// periodic grid, so each Fourier mode k of the populations evolves on its own:
//     g(k) <- E(k) [ (1 - w) g(k) + w phi (1^T g(k)) + chi S(k) ],
// E(k) = diag(e_i), e_i = exp(-i k.v_i).  At the fixed point, with
// q_i = e_i / (1 - (1 - w) e_i) (Sherman-Morrison on the rank-one collision),
//     Phi(k) = T(k) S(k),  T(k) = sum_i chi_i q_i / (1 - w sum_i phi_i q_i),
// and Phi(0) = 0 (the gauge the iteration from zero keeps).  The velocity sets
// are symmetric (v and -v with equal weights), so q(-v) = conj(q(v)) and both
// sums are real: 2 Re over one velocity of each pair (the rest velocity once).
// The denominator is small near k = 0 (it vanishes like |k|^2); since the phi_i
// sum to one it is written as sum_i phi_i Re[(1 - e_i) / (1 - (1 - w) e_i)]
// with 1 - cos(theta) = 2 sin^2(theta / 2), so nothing cancels there; nor does
// it near theta = pi, where 1 - (1 - w) e_i vanishes as w nears 2 (see
// transfer_kernel).  The phase theta = k.v_i is reduced exactly on the integers
// (m v mod n) and its half angle built from per-axis tables of exp(-i pi j / n).
// The inverse transform's 1 / V goes into T.
// The transforms are cuFFT's; the transfer function T(k) is this file's kernel.
#include <cuda_runtime.h>
#include <cufft.h>

#include <chrono>
#include <cmath>
#include <cstring>
#include <type_traits>

#include "pkr_internal.h"

namespace pkr {
namespace {

// Weights per symmetry class and the relaxation of one transfer.
struct FftCoefs {
    double phi[kMaxClasses], chi[kMaxClasses];
    double omega, scale;
};

// H[j] = exp(-i pi j / n), j < n: the half-angle phase of one axis.
__global__ void half_phase_kernel(double2* __restrict__ H, int n)
{
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
        double sn, cs;
        sincospi((double)j / n, &sn, &cs);
        H[j] = make_double2(cs, -sn);
    }
}

// Multiply the half spectrum S(k) (nx/2 + 1 modes along x) by T(k) * scale.
//
// With theta = k.v, s = sin(theta / 2), C = cos(theta / 2), c = 1 - w and
// d = 1 + c = 2 - w,
//     |1 - c e|^2 = w^2 + 4 c s^2 = d^2 - 4 c C^2 =: m,
//     Re q = (w - 2 s^2) / m,   Re[(1 - e) / (1 - c e)] = 2 d s^2 / m.
// Each sum is taken in the form whose terms have one sign: for w <= 1 m from s,
// and per class W = sum 1 / m and U = sum s^2 / m (sum Re q = w W - 2 U); for
// w > 1 (OVER) m from C, and U alone: since w^2 W = n + 4 (w - 1) U for n
// velocities, sum Re q = (n - 2 d U) / w.  With the first form for w > 1, m is
// the difference of two numbers near 4 where theta nears pi and w nears 2: T
// of D3Q111, order 1, at tau_lb = 0.5005 would be off by up to 4e-10 of its
// value, against 2e-14 (binary64 against 60 digits, modes of 24 x 20 x 18).
// The sets are symmetric under the reflection of every axis: T is too, and one
// thread forms it for the modes (mx, +-my, +-mz); and the sines and cosines of
// a triple's sign images (+-a, +-b, +-c) share their products.  Bound by the
// binary64 pipe: about 16 operations per +-v pair, 18 for w > 1 (35 when each
// mode and pair multiplied three phases and divided), for a quarter of the
// half spectrum.  pkr_fixed_point_fft on 200 x 180 x 150, D3Q111: 12.8 ms
// before, 3.7 ms now, most of it cuFFT and its plans.
template <class L>
struct Triples {   // velocities with no negative component
    static constexpr int reach = L::T.reach;
    static constexpr int count()
    {
        int n = 0;
        for (int i = 0; i < L::Q; ++i)
            if (L::T.v[i].x >= 0 && L::T.v[i].y >= 0 && L::T.v[i].z >= 0) ++n;
        return n;
    }
    static constexpr int at(int k)   // index of the k-th one in the set's order
    {
        for (int i = 0; i < L::Q; ++i)
            if (L::T.v[i].x >= 0 && L::T.v[i].y >= 0 && L::T.v[i].z >= 0 && k-- == 0) return i;
        return -1;
    }
    static constexpr int cls(int k) { return k < count() ? L::T.cls[at(k)] : -1; }
    static constexpr V3 v(int k) { return L::T.v[at(k)]; }
};

template <int I, int N, typename F>
__device__ __forceinline__ void unroll(F&& f)
{
    if constexpr (I < N) {
        f(std::integral_constant<int, I>{});
        unroll<I + 1, N>(f);
    }
}

// cos and sin of a pi m v / n for v = 0 .. R (the index reduced on the integers)
template <int R>
__device__ __forceinline__ void axis_phases(const double2* __restrict__ H, int m, int n,
                                            double (&cs)[R + 1], double (&sn)[R + 1])
{
    cs[0] = 1.0;
    sn[0] = 0.0;
    unsigned int j = 0;
#pragma unroll
    for (int v = 1; v <= R; ++v) {
        j += (unsigned int)m;
        if (j >= (unsigned int)n) j -= (unsigned int)n;
        const double2 h = __ldg(H + j);
        cs[v] = h.x;
        sn[v] = -h.y;
    }
}

template <class L, bool OVER>
__global__ void __launch_bounds__(128)
transfer_kernel(cufftDoubleComplex* __restrict__ sk, int nx, int ny, int nz, const FftCoefs c,
                const double2* __restrict__ Hx, const double2* __restrict__ Hy,
                const double2* __restrict__ Hz)
{
    constexpr int R = Triples<L>::reach, RY = L::DIM >= 2 ? R : 0, RZ = L::DIM >= 3 ? R : 0;
    const int nxh = nx / 2 + 1, nyh = ny / 2 + 1, nzh = nz / 2 + 1;
    const int64_t total = (int64_t)nxh * nyh * nzh;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const double w = c.omega, cw = 1.0 - w, d = 2.0 - w, d4 = 4.0 * d;
    const double m0 = OVER ? d * d : w * w, m1 = OVER ? -4.0 * cw : 4.0 * cw;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += stride) {
        const int mx = (int)(t % nxh);
        const int64_t r = t / nxh;
        const int my = (int)(r % nyh), mz = (int)(r / nyh);
        double cx[R + 1], sx[R + 1], cy[RY + 1], sy[RY + 1], cz[RZ + 1], sz[RZ + 1];
        axis_phases<R>(Hx, mx, nx, cx, sx);
        axis_phases<RY>(Hy, my, ny, cy, sy);
        axis_phases<RZ>(Hz, mz, nz, cz, sz);
        double num = 0.0, den = 0.0, U = 0.0, W = 0.0;
        int count = 0;   // velocities of the class so far
        // one half angle (s, C); two share their reciprocal
        auto one = [&](double s, double C) {
            const double q = s * s, inv = 1.0 / fma(m1, OVER ? C * C : q, m0);
            U = fma(q, inv, U);
            if constexpr (!OVER) W += inv;
        };
        auto two = [&](double s, double C, double p, double D) {
            const double qs = s * s, qp = p * p;
            const double ms = fma(m1, OVER ? C * C : qs, m0);
            const double mp = fma(m1, OVER ? D * D : qp, m0);
            const double inv = 1.0 / (ms * mp);
            const double is = inv * mp, ip = inv * ms;
            U = fma(qs, is, fma(qp, ip, U));
            if constexpr (!OVER) W += is + ip;
        };
        unroll<0, Triples<L>::count()>([&](auto K) {
            constexpr int k = decltype(K)::value;
            constexpr int cl = Triples<L>::cls(k);
            constexpr int a = Triples<L>::v(k).x, b = Triples<L>::v(k).y, e = Triples<L>::v(k).z;
            constexpr int axes = (a > 0) + (b > 0) + (e > 0);
            if constexpr (axes == 0) {
                if constexpr (!OVER) num = c.chi[cl] / w;   // the rest velocity: s = 0, m = w^2
            } else if constexpr (axes == 1) {
                one(a > 0 ? sx[a] : b > 0 ? sy[b] : sz[e], a > 0 ? cx[a] : b > 0 ? cy[b] : cz[e]);
            } else if constexpr (axes == 2) {
                const double c1 = a > 0 ? cx[a] : cy[b], s1 = a > 0 ? sx[a] : sy[b];
                const double c2 = e > 0 ? cz[e] : cy[b], s2 = e > 0 ? sz[e] : sy[b];
                const double p = s1 * c2, q = c1 * s2, u = c1 * c2, v = s1 * s2;
                two(p + q, u - v, p - q, u + v);
            } else {
                // y and z first: angles b + e and b - e, then both with +-a
                const double p = sy[b] * cz[e], q = cy[b] * sz[e];
                const double u = cy[b] * cz[e], v = sy[b] * sz[e];
                const double sp = p + q, sm = p - q, cp = u - v, cm = u + v;
                const double f1 = sx[a] * cp, f2 = cx[a] * sp, g1 = cx[a] * cp, g2 = sx[a] * sp;
                two(f1 + f2, g1 - g2, f1 - f2, g1 + g2);
                const double h1 = sx[a] * cm, h2 = cx[a] * sm, i1 = cx[a] * cm, i2 = sx[a] * sm;
                two(h1 + h2, i1 - i2, h1 - h2, i1 + i2);
            }
            // the class is complete: 2^axes velocities per triple, two per half angle
            count += 1 << axes;
            if constexpr (Triples<L>::cls(k + 1) != cl) {
                if constexpr (OVER) num = fma(c.chi[cl], count - d4 * U, num);   // w num
                else if constexpr (axes > 0) num += 2.0 * c.chi[cl] * (w * W - 2.0 * U);
                den += c.phi[cl] * U;
                U = W = 0.0;
                count = 0;
            }
        });
        const bool zero = mx == 0 && my == 0 && mz == 0;
        const double T = zero ? 0.0 : num / ((OVER ? w * d4 : d4) * den) * c.scale;
        const int ya = my, yb = my == 0 || 2 * my == ny ? my : ny - my;
        const int za = mz, zb = mz == 0 || 2 * mz == nz ? mz : nz - mz;
        auto apply = [&](int y, int z) {
            cufftDoubleComplex* p = sk + ((int64_t)z * ny + y) * nxh + mx;
            cufftDoubleComplex v = *p;
            v.x = zero ? 0.0 : v.x * T;
            v.y = zero ? 0.0 : v.y * T;
            *p = v;
        };
        apply(ya, za);
        if (yb != ya) apply(yb, za);
        if (zb != za) {
            apply(ya, zb);
            if (yb != ya) apply(yb, zb);
        }
    }
}

template <class L>
void launch_transfer(cufftDoubleComplex* sk, int nx, int ny, int nz, const FftCoefs& c,
                     const double2* h, cudaStream_t s)
{
    const int64_t total = (int64_t)(nx / 2 + 1) * (ny / 2 + 1) * (nz / 2 + 1);
    int64_t blocks = (total + 127) / 128;
    if (blocks > 152 * 64) blocks = 152 * 64;
    const auto kern = c.omega > 1.0 ? transfer_kernel<L, true> : transfer_kernel<L, false>;
    kern<<<(int)blocks, 128, 0, s>>>(sk, nx, ny, nz, c, h, h + nx, h + nx + ny);
}

}  // namespace
}  // namespace pkr

using namespace pkr;

extern "C" int pkr_fixed_point_fft(const pkr_problem* p, const double* rho, double* phi,
                                   int host_buffers, pkr_stats* st, void* stream)
{
    if (!p || !rho || !phi) return PKR_EINVAL;
    LatticeInfo li;
    int rc = build_lattice(p->lattice, p->order, &li);
    if (rc != PKR_OK) return rc;
    if (li.dim != p->dim) return PKR_EINVAL;
    int64_t V = 1;
    for (int k = 0; k < 3; ++k) {
        if (p->n[k] < 1 || (k >= p->dim && p->n[k] != 1)) return PKR_EINVAL;
        V *= p->n[k];
    }
    if (V > (int64_t)0x7fffffff) return PKR_EINVAL;
    double tau = p->tau_lb;
    if (!(tau > 0.0) && pkr_tau_from_knudsen(p->lattice, p->knudsen, p->n, &tau) != PKR_OK)
        return PKR_EINVAL;
    if (!(tau > 0.5) || !std::isfinite(tau)) return PKR_EINVAL;
    if (unstable(li, 1.0 / tau)) return PKR_EUNSTABLE;
    const double eps = p->epsilon == 0.0 ? 1.0 : p->epsilon;
    const int nx = (int)p->n[0], ny = (int)p->n[1], nz = (int)p->n[2];
    cudaStream_t s = (cudaStream_t)stream;

    FftCoefs c{};
    c.omega = 1.0 / tau;
    c.scale = 1.0 / (double)V;   // of the forward and inverse transforms together
    for (int k = 0; k < li.ncls; ++k) {
        c.phi[k] = li.cls_phi[k];
        c.chi[k] = li.cls_chi[k];
    }

    const int nxh = nx / 2 + 1;
    const size_t nspec = (size_t)nxh * ny * nz;
    // one device block: source, then Phi; half spectrum (first holds host rho:
    // 16 nspec >= 8 V); half-angle phase tables of x, y, z; mean, flag, partials
    const int red_blocks = 152 * 4;
    const size_t rb = ((size_t)V * 8 + 255) / 256 * 256;
    const size_t kb = (nspec * sizeof(cufftDoubleComplex) + 255) / 256 * 256;
    const size_t hb = ((size_t)nx + ny + nz) * sizeof(double2);
    unsigned char* block = nullptr;
    if (cudaMalloc((void**)&block, rb + kb + hb + 16 + red_blocks * 8) != cudaSuccess) {
        cudaGetLastError();
        return PKR_ENOMEM;
    }
    double* d_r = reinterpret_cast<double*>(block);
    cufftDoubleComplex* d_k = reinterpret_cast<cufftDoubleComplex*>(block + rb);
    double2* d_h = reinterpret_cast<double2*>(block + rb + kb);
    double* d_mean = reinterpret_cast<double*>(block + rb + kb + hb);
    int* d_flag = reinterpret_cast<int*>(d_mean + 1);
    double* d_part = d_mean + 2;
    cufftHandle fwd = 0, inv = 0;
    bool ok = true;
    double back[2] = {0.0, 0.0};   // mean, then the flag
    int flag = 0;
    const auto t0 = std::chrono::steady_clock::now();
    {
        const double* rd = rho;
        if (host_buffers) {
            ok = cudaMemcpyAsync(d_k, rho, (size_t)V * 8, cudaMemcpyHostToDevice, s) == cudaSuccess;
            rd = reinterpret_cast<const double*>(d_k);
        }
        // S = (rho - <rho>) c_s^2 (tau_lb - 1/2) / eps, into d_r
        const bool prepared =
            ok && cudaMemsetAsync(d_flag, 0, sizeof(int), s) == cudaSuccess &&
            launch_rho_partials(rd, V, d_part, red_blocks, d_flag, s) == 0 &&
            launch_finalize_mean(d_part, red_blocks, V, d_mean, s) == 0 &&
            launch_make_source(rd, d_mean, li.cs2 * (tau - 0.5) / eps, V, d_r, PKR_FP64, s) == 0;
        ok = prepared;
        // the transforms of a non-finite rho run for nothing, or fail for want
        // of work space: phi is written only after the flag has been read, and
        // the flag decides the status first.  The inverse plan is built while
        // the GPU works on the forward transform.
        int n3[3] = {nz, ny, nx};
        const int rank = p->dim;
        int* dims = n3 + (3 - rank);
        ok = ok &&
             cufftPlanMany(&fwd, rank, dims, nullptr, 1, 0, nullptr, 1, 0, CUFFT_D2Z, 1) ==
                 CUFFT_SUCCESS &&
             cufftSetStream(fwd, s) == CUFFT_SUCCESS;
        ok = ok && cufftExecD2Z(fwd, d_r, d_k) == CUFFT_SUCCESS;
        if (ok) {
            half_phase_kernel<<<(nx + 255) / 256, 256, 0, s>>>(d_h, nx);
            half_phase_kernel<<<(ny + 255) / 256, 256, 0, s>>>(d_h + nx, ny);
            half_phase_kernel<<<(nz + 255) / 256, 256, 0, s>>>(d_h + nx + ny, nz);
            switch (p->lattice) {
            case PKR_D1Q5: launch_transfer<D1Q5>(d_k, nx, ny, nz, c, d_h, s); break;
            case PKR_D1Q9: launch_transfer<D1Q9>(d_k, nx, ny, nz, c, d_h, s); break;
            case PKR_D1Q13: launch_transfer<D1Q13>(d_k, nx, ny, nz, c, d_h, s); break;
            case PKR_D2Q25: launch_transfer<D2Q25>(d_k, nx, ny, nz, c, d_h, s); break;
            case PKR_D2Q81: launch_transfer<D2Q81>(d_k, nx, ny, nz, c, d_h, s); break;
            case PKR_D2Q169: launch_transfer<D2Q169>(d_k, nx, ny, nz, c, d_h, s); break;
            case PKR_D3Q19: launch_transfer<D3Q19>(d_k, nx, ny, nz, c, d_h, s); break;
            case PKR_D3Q111: launch_transfer<D3Q111>(d_k, nx, ny, nz, c, d_h, s); break;
            }
            ok = cudaGetLastError() == cudaSuccess;
        }
        ok = ok &&
             cufftPlanMany(&inv, rank, dims, nullptr, 1, 0, nullptr, 1, 0, CUFFT_Z2D, 1) ==
                 CUFFT_SUCCESS &&
             cufftSetStream(inv, s) == CUFFT_SUCCESS &&
             cufftExecZ2D(inv, d_k, d_r) == CUFFT_SUCCESS;
        const bool read = prepared &&
                          cudaMemcpyAsync(back, d_mean, sizeof(back), cudaMemcpyDeviceToHost, s) ==
                              cudaSuccess &&
                          cudaStreamSynchronize(s) == cudaSuccess;
        std::memcpy(&flag, back + 1, sizeof(int));
        ok = ok && read && !flag;
        ok = ok && cudaMemcpyAsync(phi, d_r, (size_t)V * 8,
                                   host_buffers ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice,
                                   s) == cudaSuccess &&
             cudaStreamSynchronize(s) == cudaSuccess;
    }
    const double ms =
        std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
    if (fwd) cufftDestroy(fwd);
    if (inv) cufftDestroy(inv);
    cudaFree(block);
    if (!ok) cudaGetLastError();   // an allocation cuFFT was refused is not the next call's error
    if (flag) return PKR_EINVAL;
    if (!ok) return PKR_ECUDA;
    if (st) {
        std::memset(st, 0, sizeof(*st));
        st->rho_mean_removed = back[0];
        st->tau_lb = tau;
        st->cs2 = li.cs2;
        st->wall_ms = ms;
        st->residual = 0.0;
        st->variant = -1;
    }
    return PKR_OK;
}

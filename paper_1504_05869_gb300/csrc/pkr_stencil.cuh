// pkr_stencil.cuh -- the scalar stencil of omega = 1 (included by
// pkr_sweep.cuh).
//
// At tau_lb = 1 (the paper's setting) the collision forgets the pulled
// populations, f_i = phi_i Phi + chi_i S, so one step is the scalar stencil
//     Phi'(x) = sum_i w_i Phi(x - v_i) + St(x)
// with w_i = phi_i and St = sum_i chi_i S(x - v_i) (the same kernels with
// w_i = chi_i, St = 0, build St once).  The state is Phi alone.
//
// Every form is bound by the binary64 pipe (two operations per clock and SM),
// not by memory (24 bytes per site), so what counts is the number of binary64
// operations per site.  The velocities of a symmetry class share their
// weight, so values are added first and weighted once per class.
#pragma once

namespace pkr {

// ---------------------------------------------------------------------------
// One site from its Q neighbours: the classes fall into kStencilParts
// contiguous parts of about Q / kStencilParts velocities; part j is
// sum_c w_c (sum of the class), and the site's value ((a0 + a1) + (a2 + a3)) +
// St.  The resident forms and stencil_kernel with SPLIT evaluate exactly this, so
// they agree bit for bit whether one thread takes all parts or four warps take
// one each; stencil_kernel without it (one chain) and the plane form add in
// orders of their own.
// ---------------------------------------------------------------------------
constexpr int kStencilParts = 4;

template <class L>
__host__ __device__ constexpr int part_begin(int j)   // first class of part j
{
    if (j >= kStencilParts) return ncls_of<L>();
    for (int c = 0; c < ncls_of<L>(); ++c)
        if (cls_begin<L>(c) * kStencilParts >= j * L::Q) return c;
    return ncls_of<L>();
}

template <class L, int j, class Get>
__device__ __forceinline__ double stencil_part(const Coefs<double>& c, const Get& get)
{
    double acc = 0.0;
    static_for<part_begin<L>(j), part_begin<L>(j + 1)>([&](auto CI) {
        constexpr int cl = decltype(CI)::value;
        constexpr int i0 = cls_begin<L>(cl), i1 = cls_begin<L>(cl + 1);
        // two interleaved sums: half the dependent chain
        double s0 = get(std::integral_constant<int, i0>{});
        if constexpr (i1 - i0 > 1) {
            double s1 = get(std::integral_constant<int, i0 + 1>{});
            static_for<i0 + 2, i1>([&](auto I) {
                constexpr int i = decltype(I)::value;
                if constexpr ((i - i0) % 2 == 0) s0 += get(I);
                else s1 += get(I);
            });
            s0 += s1;
        }
        acc = fma(c.wphi[cl], s0, acc);
    });
    return acc;
}

// Wrapped offsets of a site's neighbours, one entry per displacement -R..R.
template <class L>
struct Neighbours {
    static constexpr int RC = reach_of<L>();
    static constexpr int W = 2 * RC + 1;
    static constexpr int WY = L::DIM >= 2 ? W : 1, WZ = L::DIM >= 3 ? W : 1;
    int xs[W], yo[WY], zo[WZ];

    __device__ __forceinline__ void locate(int s, int nx, int ny, int nz, int small)
    {
        const int x = s % nx, r = s / nx, y = r % ny, z = r / ny;
        const int nxy = nx * ny;
        yo[0] = y * nx;
        zo[0] = z * nxy;
        if (small) {
#pragma unroll
            for (int d = -RC; d <= RC; ++d) {
                xs[d + RC] = wrap_any(x - d, nx);
                if constexpr (L::DIM >= 2) yo[d + RC] = wrap_any(y - d, ny) * nx;
                if constexpr (L::DIM >= 3) zo[d + RC] = wrap_any(z - d, nz) * nxy;
            }
        } else {
#pragma unroll
            for (int d = -RC; d <= RC; ++d) {
                xs[d + RC] = wrap_near(x - d, nx);
                if constexpr (L::DIM >= 2) yo[d + RC] = wrap_near(y - d, ny) * nx;
                if constexpr (L::DIM >= 3) zo[d + RC] = wrap_near(z - d, nz) * nxy;
            }
        }
    }
    // Keeps the compiler from forming all Q sums of at() ahead of a loop that
    // uses them (it would spill them).
    __device__ __forceinline__ void hold()
    {
#pragma unroll
        for (int d = 0; d < W; ++d) asm volatile("" : "+r"(xs[d]));
        if constexpr (WY > 1) {
#pragma unroll
            for (int d = 0; d < W; ++d) asm volatile("" : "+r"(yo[d]));
        }
    }
    // flat index of x - v_i
    template <int i>
    __device__ __forceinline__ int at() const
    {
        constexpr int oy = L::DIM >= 2 ? vy_of<L>(i) + RC : 0;
        constexpr int oz = L::DIM >= 3 ? vz_of<L>(i) + RC : 0;
        return zo[oz] + yo[oy] + xs[vx_of<L>(i) + RC];
    }
};

// The block's residual terms of a check step to partials (4 doubles per
// block): |dPhi|^2, |Phi|^2, max |dPhi|, sum Phi, summed in a fixed order.
__device__ __forceinline__ void stencil_partials(double d2, double n2, double mx, double ms,
                                                 double* partials)
{
    __shared__ double red[8][4];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        d2 += __shfl_down_sync(0xffffffffu, d2, o);
        n2 += __shfl_down_sync(0xffffffffu, n2, o);
        mx = fmax(mx, __shfl_down_sync(0xffffffffu, mx, o));
        ms += __shfl_down_sync(0xffffffffu, ms, o);
    }
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) {
        red[w][0] = d2;
        red[w][1] = n2;
        red[w][2] = mx;
        red[w][3] = ms;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double t0 = 0.0, t1 = 0.0, t2 = 0.0, t3 = 0.0;
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) {
            t0 += red[k][0];
            t1 += red[k][1];
            t2 = fmax(t2, red[k][2]);
            t3 += red[k][3];
        }
        partials[4 * blockIdx.x + 0] = t0;
        partials[4 * blockIdx.x + 1] = t1;
        partials[4 * blockIdx.x + 2] = t2;
        partials[4 * blockIdx.x + 3] = t3;
    }
}

// One thread per site; the Q neighbour reads hit L1/L2.  Any grid and set.
// SPLIT: the parts of the resident forms, four short chains, for grids that
// those take (they wait on latency).  Else the binary64 pipe is the bound and
// one chain of Q multiply-adds from St on has the fewest operations (D3Q111:
// 111 against 115, D3Q19: 19 against 23).
template <class L, bool SPLIT>
__global__ void __launch_bounds__(256)
stencil_kernel(const double* __restrict__ Pin, double* __restrict__ Pout,
               const double* __restrict__ St, const Coefs<double> c, int64_t V, int nx, int ny,
               int nz, int small, int check, double* partials, const int* stop)
{
    if (stop != nullptr && *stop != 0) return;   // the run stopped before this step
    double d2 = 0.0, n2 = 0.0, mx = 0.0, ms = 0.0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t s64 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s64 < V; s64 += stride) {
        const int s = (int)s64;
        double acc;
        if constexpr (SPLIT) {
            Neighbours<L> nb;
            nb.locate(s, nx, ny, nz, small);
            acc = St ? St[s] : 0.0;
            double a[kStencilParts];
            static_for<0, kStencilParts>([&](auto J) {
                constexpr int j = decltype(J)::value;
                a[j] = stencil_part<L, j>(c, [&](auto I) {
                    return __ldg(Pin + nb.template at<decltype(I)::value>());
                });
            });
            acc = ((a[0] + a[1]) + (a[2] + a[3])) + acc;
        } else {
            // (offsets on three axes for every set, and a choice per offset: as
            // Neighbours forms them D2Q81 took 9.0 us a step for 8.3 on 150 x 150,
            // the other sets the same within 1 %)
            constexpr int RC = reach_of<L>(), W = 2 * RC + 1;
            const int nxy = nx * ny;
            const int x = s % nx, r = s / nx, y = r % ny, z = r / ny;
            int xs[W], yo[W], zo[W];
#pragma unroll
            for (int d = -RC; d <= RC; ++d) {
                if (small) {
                    xs[d + RC] = wrap_any(x - d, nx);
                    yo[d + RC] = wrap_any(y - d, ny) * nx;
                    zo[d + RC] = wrap_any(z - d, nz) * nxy;
                } else {
                    xs[d + RC] = wrap_near(x - d, nx);
                    yo[d + RC] = wrap_near(y - d, ny) * nx;
                    zo[d + RC] = wrap_near(z - d, nz) * nxy;
                }
            }
            acc = St ? St[s] : 0.0;
            static_for<0, L::Q>([&](auto I) {
                constexpr int i = decltype(I)::value;
                const int at = zo[vz_of<L>(i) + RC] + yo[vy_of<L>(i) + RC] + xs[vx_of<L>(i) + RC];
                acc = fma(c.wphi[cls_of<L>(i)], __ldg(Pin + at), acc);
            });
        }
        Pout[s] = acc;
        if (check) {
            const double d = acc - Pin[s];
            d2 += d * d;
            n2 += acc * acc;
            mx = fmax(mx, fabs(d));
            ms += acc;
        }
    }
    if (check) stencil_partials(d2, n2, mx, ms, partials);
}

// ---------------------------------------------------------------------------
// 3D sets on grids of some size: a block marches through the planes of a
// chunk of z.  In a plane it forms, per site, the sums X_a of the values at
// x - a and x + a (shared memory), from them the ring sums R_ab over the
// images of (+-a, +-b) in x and y, and from those, weighted, T_c: what the
// plane adds to the results c planes above and below it.  Each site's seven
// (2 R + 1) open results live in registers.
//
// binary64 operations per site of D3Q111: 3 (X) + 15 (R) + 19 (T) + 8, about
// 47 with the X sums of the rows around the tile, against 111 multiply-adds
// in the per-site form: 256^3 takes 1.69 ms a step (9.9 GLUPS) against 3.56 ms
// (4.7).  The tile is 32 x 16 sites, 256 threads of two sites: wide enough
// that those rows cost 3 x 6/16 operations more, small enough that several
// blocks share an SM and cover each other's barriers; or 32 x 8, one site a
// thread, a few percent dearer per site and twice as fine, which fills the SMs
// more evenly on mid-size grids (100^3: 171 us a step against 179 and, one
// thread per site, 235; 62 x 163 x 53: 87 against 97 and 124).
// ---------------------------------------------------------------------------
// weight class of (a, b, c), any order and sign; -1: not in the set
template <class L>
__host__ __device__ constexpr int cls_at(int a, int b, int c)
{
    for (int i = 0; i < L::Q; ++i)
        if (vx_of<L>(i) == a && vy_of<L>(i) == b && vz_of<L>(i) == c) return cls_of<L>(i);
    return -1;
}
// some velocity has components (+-a, +-b) in x and y
template <class L>
__host__ __device__ constexpr bool ring_used(int a, int b)
{
    for (int c = 0; c <= reach_of<L>(); ++c)
        if (cls_at<L>(a, b, c) >= 0) return true;
    return false;
}

template <class L, int TY_>
struct Planes {
    static constexpr int RC = reach_of<L>();
    static constexpr int TX = 32, TY = TY_, NT = 256, NH = TX * TY / NT;
    static constexpr int PX = TX + 2 * RC, PY = TY + 2 * RC;
    static constexpr int NLD = (PX * PY + NT - 1) / NT;   // values a thread loads per plane
    static constexpr int NXS = (TX * PY + NT - 1) / NT;   // X positions a thread forms
};

template <class L, int TY_>
__global__ void __launch_bounds__(256, 3)
stencil_planes_kernel(const double* __restrict__ Pin, double* __restrict__ Pout,
                      const double* __restrict__ St, const Coefs<double> c, int nx, int ny,
                      int nz, int tx, int ty, int cz, int items, int check, double* partials,
                      const int* stop)
{
    if (stop != nullptr && *stop != 0) return;   // the run stopped before this step
    using PL = Planes<L, TY_>;
    constexpr int NH = PL::NH, RC = PL::RC, TX = PL::TX, TY = PL::TY, NT = PL::NT, PX = PL::PX, PY = PL::PY;
    constexpr int W = 2 * RC + 1;
    __shared__ double ph[PY][PX];
    __shared__ double xsum[RC][PY][TX];
    const int tid = threadIdx.x;
    const int lx = tid & 31, ly = tid >> 5;     // site (lx, ly), and (lx, ly + 8) of 16 rows
    const int64_t nxy = (int64_t)nx * ny;
    double d2 = 0.0, n2 = 0.0, mx = 0.0, ms = 0.0;

    for (int item = blockIdx.x; item < items; item += gridDim.x) {
        const int bx = item % tx, by = (item / tx) % ty, bz = item / (tx * ty);
        const int x0 = bx * TX, y0 = by * TY;
        const int z0 = bz * cz, z1 = min(nz, z0 + cz);
        // in-plane offsets of the values this thread loads (the same in every plane)
        int off[PL::NLD];
#pragma unroll
        for (int k = 0; k < PL::NLD; ++k) {
            const int p = tid + k * NT;
            const int px = p % PX, py = p / PX;
            off[k] = wrap_any(y0 - RC + py, ny) * nx + wrap_any(x0 - RC + px, nx);
        }
        double next[PL::NLD];
        auto fetch = [&](int z) {
            const double* src = Pin + nxy * wrap_any(z, nz);
#pragma unroll
            for (int k = 0; k < PL::NLD; ++k)
                if (tid + k * NT < PX * PY) next[k] = __ldg(src + off[k]);
        };
        double acc[NH][W];   // open results of planes z - R .. z + R
#pragma unroll
        for (int h = 0; h < NH; ++h)
#pragma unroll
            for (int q = 0; q < W; ++q) acc[h][q] = 0.0;
        fetch(z0 - RC);
        for (int z = z0 - RC; z < z1 + RC; ++z) {
            __syncthreads();   // the previous plane's sums have been read
#pragma unroll
            for (int k = 0; k < PL::NLD; ++k)
                if (tid + k * NT < PX * PY) (&ph[0][0])[tid + k * NT] = next[k];
            __syncthreads();
            if (z + 1 < z1 + RC) fetch(z + 1);
#pragma unroll
            for (int k = 0; k < PL::NXS; ++k) {
                const int p = tid + k * NT;
                const int px = p % TX, py = p / TX;
                if (p < TX * PY) {
#pragma unroll
                    for (int a = 1; a <= RC; ++a)
                        xsum[a - 1][py][px] = ph[py][px + RC - a] + ph[py][px + RC + a];
                }
            }
            __syncthreads();
            // the plane's terms are needed by results z - c and z + c in the chunk
            bool need[RC + 1];
#pragma unroll
            for (int q = 0; q <= RC; ++q)
                need[q] = (z - q >= z0 && z - q < z1) || (z + q >= z0 && z + q < z1);
#pragma unroll
            for (int h = 0; h < NH; ++h) {
                const int ry = ly + 8 * h + RC, cx = lx + RC;
                // R_ab, a >= b: the images of (+-a, +-b) and (+-b, +-a)
                double R[RC + 1][RC + 1];
                static_for<0, RC + 1>([&](auto AI) {
                    constexpr int a = decltype(AI)::value;
                    static_for<0, a + 1>([&](auto BI) {
                        constexpr int b = decltype(BI)::value;
                        if constexpr (ring_used<L>(a, b)) {
                            if constexpr (a == 0) R[0][0] = ph[ry][cx];
                            else if constexpr (b == 0)
                                R[a][0] = xsum[a - 1][ry][lx] + (ph[ry - a][cx] + ph[ry + a][cx]);
                            else if constexpr (a == b)
                                R[a][a] = xsum[a - 1][ry - a][lx] + xsum[a - 1][ry + a][lx];
                            else
                                R[a][b] = (xsum[a - 1][ry - b][lx] + xsum[a - 1][ry + b][lx]) +
                                          (xsum[b - 1][ry - a][lx] + xsum[b - 1][ry + a][lx]);
                        }
                    });
                });
                static_for<0, RC + 1>([&](auto QI) {
                    constexpr int q = decltype(QI)::value;
                    if (need[q]) {
                        double T = 0.0;
                        static_for<0, RC + 1>([&](auto AI) {
                            constexpr int a = decltype(AI)::value;
                            static_for<0, a + 1>([&](auto BI) {
                                constexpr int b = decltype(BI)::value;
                                constexpr int cl = cls_at<L>(a, b, q);
                                if constexpr (cl >= 0) T = fma(c.wphi[cl], R[a][b], T);
                            });
                        });
                        acc[h][RC - q] += T;
                        if constexpr (q > 0) acc[h][RC + q] += T;
                    }
                });
            }
            // the result of plane z - R is complete
            const int zo = z - RC;
#pragma unroll
            for (int h = 0; h < NH; ++h) {
                const int x = x0 + lx, y = y0 + ly + 8 * h;
                if (zo >= z0 && x < nx && y < ny) {
                    const int64_t s = nxy * zo + (int64_t)y * nx + x;
                    const double v = acc[h][0] + (St ? St[s] : 0.0);
                    Pout[s] = v;
                    if (check) {
                        const double d = v - Pin[s];
                        d2 += d * d;
                        n2 += v * v;
                        mx = fmax(mx, fabs(d));
                        ms += v;
                    }
                }
#pragma unroll
                for (int q = 0; q + 1 < W; ++q) acc[h][q] = acc[h][q + 1];
                acc[h][W - 1] = 0.0;
            }
        }
    }
    if (check) {
        __syncthreads();
        stencil_partials(d2, n2, mx, ms, partials);
    }
}

template <class L>
int launch_stencil(const double* Pin, double* Pout, const double* St, const Coefs<double>& c,
                   int64_t V, int nx, int ny, int nz, int small, int check, double* partials,
                   int grid, int form, void* stream, const int* stop)
{
    if constexpr (L::DIM == 3) {
        if (form > 0) {
            const int cz = stencil_cz(form), rows = stencil_ty(form);
            const int tx = (nx + 31) / 32, ty = (ny + rows - 1) / rows;
            const int items = tx * ty * ((nz + cz - 1) / cz);
            const auto kern =
                rows == 16 ? stencil_planes_kernel<L, 16> : stencil_planes_kernel<L, 8>;
            kern<<<grid, 256, 0, (cudaStream_t)stream>>>(Pin, Pout, St, c, nx, ny, nz, tx, ty,
                                                         cz, items, check, partials, stop);
            return (int)cudaGetLastError();
        }
    }
    const int block = (int64_t)grid * 64 >= V ? 64 : 256;   // see stencil_block
    const auto kern = form == kStencilParts4 ? stencil_kernel<L, true> : stencil_kernel<L, false>;
    kern<<<grid, block, 0, (cudaStream_t)stream>>>(Pin, Pout, St, c, V, nx, ny, nz, small, check,
                                                   partials, stop);
    return (int)cudaGetLastError();
}

}  // namespace pkr

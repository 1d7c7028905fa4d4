// pkr_sweep_h16w.cuh -- binary16 storage with four sites per lane (included by
// pkr_sweep.cuh).
//
// As sweep_h16p_kernel (two sites per lane), with a warp's tile of 128 sites of
// one x row: every copy and store of a warp is one 256-byte request instead of
// two of 128 bytes and, for odd v_x, a third of one word.  A row holds the
// aligned run of 128 values unshifted and a halo of 4 (8 for reaches above 4)
// on the side v_x needs; before the density each row with v_x != 0 is shifted
// in place by v_x, so that both passes read one 8-byte word per velocity.  Per
// site the operations and their order are those of sweep_h16_kernel: the same
// results bit for bit.  Needs nx a multiple of 128 and no edge below the reach.
#pragma once

namespace pkr {

template <class L>
struct H16w {
    static constexpr int HL = (reach_of<L>() + 3) / 4 * 4;   // halo sites per side
    static constexpr int ROWB = (128 + 2 * HL) * 2;          // bytes per row (multiple of 16)
    static constexpr size_t smem_bytes(int tiles) { return (size_t)tiles * L::Q * ROWB; }
};

// Four binary16 values (8 bytes) as two pairs of binary32.
struct Quad {
    f32x2 a, b;
};
__device__ __forceinline__ f32x2 h16_unpack(unsigned int w)
{
    const float2 v = __half22float2(*reinterpret_cast<const __half2*>(&w));
    return pack2(v.x, v.y);
}
__device__ __forceinline__ uint2 lds_2b32(uint32_t addr)
{
    uint2 v;
    asm volatile("ld.shared.v2.b32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(addr));
    return v;
}
__device__ __forceinline__ Quad h16_quad(uint32_t addr)
{
    const uint2 w = lds_2b32(addr);
    return Quad{h16_unpack(w.x), h16_unpack(w.y)};
}

// Words of the four sites 4 l - VX .. 4 l - VX + 3 of a row from its aligned
// words (own: address of the lane's words 4 l .. 4 l + 3).
template <int VX>
__device__ __forceinline__ uint2 h16_shifted(uint32_t own)
{
    static_assert(VX >= -8 && VX <= 8, "halo of at most 8 sites");
    constexpr int o = -VX;                              // first site, relative to 4 l
    constexpr int q = (o >= 0 ? o : o - 3) / 4;         // its aligned group of four
    constexpr int r = o - 4 * q;                        // 0 .. 3 inside the group
    const uint32_t at = own + (uint32_t)(8 * q);
    if constexpr (r == 0) return lds_2b32(at);
    else if constexpr (r == 2) return make_uint2(lds_b32(at + 4), lds_b32(at + 8));
    else if constexpr (r == 1) {
        const uint2 w = lds_2b32(at);
        const unsigned int n = lds_b32(at + 8);
        return make_uint2(prmt(w.x, w.y, 0x5432), prmt(w.y, n, 0x5432));
    } else {
        const unsigned int w = lds_b32(at + 4);
        const uint2 n = lds_2b32(at + 8);
        return make_uint2(prmt(w, n.x, 0x5432), prmt(n.x, n.y, 0x5432));
    }
}

template <class L, int TILES>
__global__ void __launch_bounds__(TILES * 32)
sweep_h16w_kernel(const SweepArgs a, const Coefs<float> c)
{
    constexpr int Q = L::Q;
    constexpr int RC = reach_of<L>(), W = 2 * RC + 1;
    constexpr int NC = ncls_of<L>();
    constexpr int HL = H16w<L>::HL, ROWB = H16w<L>::ROWB;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double rpart[TILES][4];
    __shared__ float mpart[TILES];

    const int lane = threadIdx.x & 31;
    const int sub = threadIdx.x >> 5;
    // row 0, and this lane's words of it
    const uint32_t rows = (uint32_t)__cvta_generic_to_shared(smem_raw) + (uint32_t)(sub * Q * ROWB);
    const uint32_t own = rows + (uint32_t)(HL * 2 + lane * 8);
    const unsigned short* __restrict__ A = static_cast<const unsigned short*>(a.A);
    unsigned short* __restrict__ B = static_cast<unsigned short*>(a.B);
    const float* __restrict__ S = static_cast<const float*>(a.S);
    const int64_t V = a.V;
    const int nx = a.nx, ny = a.ny, nz = a.nz;
    const float sr = a.sc[a.cur];
    const float inv_sw = 1.0f / a.sc[a.cur ^ 1];
    const int ntiles = (int)(V >> 7);

    double rd2 = 0.0, rn2 = 0.0, rmx = 0.0, rms = 0.0;
    float pmax = 0.f;
    const int nt = gridDim.x * TILES;
    const int nb = a.zero_in ? 0 : 8;
    // the tile whose rows are being filled
    int yo[W], zo[W], x0 = 0, xl = 0, xr = 0;
    auto locate = [&](int tile) {
        const int s0 = tile * 128;
        const int r = (int)((unsigned)s0 / (unsigned)nx);
        x0 = s0 - r * nx;
        const int z = (int)((unsigned)r / (unsigned)ny);
        const int y = r - z * ny;
        static_for<0, W>([&](auto DI) {
            constexpr int d = decltype(DI)::value - RC;
            yo[d + RC] = wrap_off<d>(y, ny) * nx;
            zo[d + RC] = wrap_off<d>(z, nz) * (nx * ny);
        });
        xl = (x0 > 0 ? x0 : nx) - HL + 4 * lane;
        xr = (x0 + 128 < nx ? x0 + 128 : 0) + 4 * lane;
    };
    auto pull = [&](auto I) {
        constexpr int i = decltype(I)::value;
        constexpr int vx = vx_of<L>(i);
        const unsigned short* row =
            A + ((int64_t)i * V + (zo[vz_of<L>(i) + RC] + yo[vy_of<L>(i) + RC]));
        cp_async<8>(own + (uint32_t)(i * ROWB), row + (x0 + 4 * lane), nb);
        if constexpr (vx > 0) {
            if (lane < HL / 4) cp_async<8>(rows + (uint32_t)(i * ROWB + lane * 8), row + xl, nb);
        } else if constexpr (vx < 0) {
            if (lane < HL / 4)
                cp_async<8>(rows + (uint32_t)(i * ROWB + (HL + 128) * 2 + lane * 8), row + xr, nb);
        }
    };
    const int first = blockIdx.x * TILES + sub;
    if (first < ntiles) {
        locate(first);
        static_for<0, Q>(pull);
    }
    for (int tile = first; tile < ntiles; tile += nt) {
        const int s = tile * 128 + 4 * lane;
        const float4 S4 = *reinterpret_cast<const float4*>(S + s);
        const bool more = tile + nt < ntiles;
        if (more) locate(tile + nt);
        cp_async_wait_all();
        __syncwarp();
        // shift the rows in place, a class at a time: every lane reads the
        // class's rows before any lane writes them
        static_for<0, NC>([&](auto CI) {
            constexpr int cl = decltype(CI)::value;
            constexpr int i0 = cls_begin<L>(cl), n = cls_begin<L>(cl + 1) - i0;
            uint2 w[n];
            static_for<0, n>([&](auto K) {
                constexpr int k = decltype(K)::value;
                constexpr int vx = vx_of<L>(i0 + k);
                if constexpr (vx != 0)
                    w[k] = h16_shifted<vx>(own + (uint32_t)((i0 + k) * ROWB));
            });
            __syncwarp();
            static_for<0, n>([&](auto K) {
                constexpr int k = decltype(K)::value;
                if constexpr (vx_of<L>(i0 + k) != 0)
                    asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(
                                     own + (uint32_t)((i0 + k) * ROWB)),
                                 "r"(w[k].x), "r"(w[k].y)
                                 : "memory");
            });
        });
        // (a lane reads back only its own words from here on)
        // density: per site the four interleaved binary32 partials of
        // density_fixed_f32, then the array's scale
        f32x2 pa[4] = {0, 0, 0, 0}, pb[4] = {0, 0, 0, 0};
#pragma unroll 2
        for (int k = 0; k + 3 < Q; k += 4) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const Quad v = h16_quad(own + (uint32_t)((k + j) * ROWB));
                pa[j] = add2(pa[j], v.a);
                pb[j] = add2(pb[j], v.b);
            }
        }
#pragma unroll
        for (int k = Q - Q % 4; k < Q; ++k) {
            const Quad v = h16_quad(own + (uint32_t)(k * ROWB));
            pa[0] = add2(pa[0], v.a);
            pb[0] = add2(pb[0], v.b);
        }
        const float2 sa = unpack2(add2(add2(pa[0], pa[1]), add2(pa[2], pa[3])));
        const float2 sb = unpack2(add2(add2(pb[0], pb[1]), add2(pb[2], pb[3])));
        const float Phi[4] = {sa.x * sr, sa.y * sr, sb.x * sr, sb.y * sr};
        // the written array's scale is a power of two: see sweep_h16p_kernel
        const float om1w = c.om1 * sr * inv_sw;
        const f32x2 om2 = pack2(om1w, om1w);
        const float Sx[4] = {(float)((double)S4.x + a.soff), (float)((double)S4.y + a.soff),
                             (float)((double)S4.z + a.soff), (float)((double)S4.w + a.soff)};
        unsigned short* dst = B + s;
        static_for<0, NC>([&](auto CI) {
            constexpr int cl = decltype(CI)::value;
            constexpr int i0 = cls_begin<L>(cl), i1 = cls_begin<L>(cl + 1);
            float e[4];
#pragma unroll
            for (int j = 0; j < 4; ++j)
                e[j] = fmaf(c.wphi[cl], Phi[j], c.chi[cl] * Sx[j]) * inv_sw;
            const f32x2 ea = pack2(e[0], e[1]), eb = pack2(e[2], e[3]);
#pragma unroll 4
            for (int i = i0; i < i1; ++i) {
                // p / sc of the written array
                const Quad v = h16_quad(own + (uint32_t)(i * ROWB));
                const float2 qa = unpack2(fma2(om2, v.a, ea)), qb = unpack2(fma2(om2, v.b, eb));
                pmax = max3_abs(max3_abs(pmax, qa.x, qa.y), qb.x, qb.y);
                const __half2 ha = __floats2half2_rn(qa.x, qa.y);
                const __half2 hb = __floats2half2_rn(qb.x, qb.y);
                __stcs(reinterpret_cast<uint2*>(dst),
                       make_uint2(*reinterpret_cast<const unsigned int*>(&ha),
                                  *reinterpret_cast<const unsigned int*>(&hb)));
                dst += V;
            }
            // the class's rows take the next tile's copies
            if (more) static_for<i0, i1>(pull);
        });
        if (a.mode != kPlain) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const double ph = (double)Phi[j];
                if (a.mode == kCheck) {
                    const double d = ph - a.Phi[s + j];
                    rd2 += d * d;
                    rn2 += ph * ph;
                    rmx = fmax(rmx, fabs(d));
                    rms += ph;
                }
                a.Phi[s + j] = ph;
            }
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

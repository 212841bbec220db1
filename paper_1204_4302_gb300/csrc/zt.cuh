// Fused z pass of the tensor method for FP32 plans of z length 32, 64 and 128:
// forward z transforms of the three components, H^ = -N^ M^, inverse z transforms
// (as k_z_conv2), one small CTA per tile of TC columns kx of one ky row.
//
// What bounds it is the instructions per point and the latency between its
// barriers, so the tile is small and several CTAs per SM interleave their phases
// (points a component, threads, shared memory, CTAs and warps per SM: L = 32, 16 columns
// 512, 64, 19 KB, 8, 16; 8 columns 256, 32, 11 KB, 16, 16; L = 64, 8 columns 512, 64, 20 KB,
// 8, 16; L = 128, 16 columns 2048, 128, 73 KB, 3, 12; 8 columns 1024, 64, 38 KB, 5, 10),
// L = R1 x 8 is a compile-time pair, a row of the tile is a whole 64- to 256-byte segment
// (conflict-free exchange without a swizzle), the tensor block arrives from the
// tile-ordered copy by 16-byte asynchronous copies while stage 1 runs, and the
// product's terms are packed FP32x2 multiply-adds. Against the two-stage kernel with an
// 8-point second stage: 128 x 128 x 16 24 -> 14.5 us, 128 x 128 x 32 33 -> 21.6 (97 -> 55
// instructions per point), 128 x 128 x 64 58 -> 47. Asking for 20 or 24 warps per SM (96 or
// 80 registers) changed nothing: the L1 and shared-memory accesses are at 70% of their rate.
#pragma once
#include "mix2.cuh"
#include "zws.cuh"

namespace demag {

// TC columns per tile: 16, 8 and 16 at L = 32, 64 and 128, or 8 where the wide
// tiles would leave SMs without work. Kx = 2^k + 1, so a wider tile is emptier in a
// row's last tile (L = 64: 21.6 us with 8 columns, 22.3 with 16 at 128 x 128 x 32; L = 128:
// 49.5 and 47.5 at 128 x 128 x 64; L = 32: 14.5 either way at 128 x 128 x 16). RP: exchange rows per stage-1 group (one more where a row is
// shorter than a 128-byte line, so that two rows of a half warp use different banks).
// TZB floats per 4-column sub-block of the tensor tile, TZS floats apart in shared
// memory: the sub-blocks of a row start 128 / TC banks apart.
template <int L, int TC> struct ZtShape {
    static constexpr int R2 = 8, R1 = L / 8;
    static constexpr int NT = R1 * TC < R2 * TC ? R1 * TC : R2 * TC;
    static constexpr int RP = TC >= 16 ? R1 : R1 + 1;
    static constexpr int EXS = R2 * RP * TC;  // one component of the exchange
    static constexpr int HZ = L / 2 + 1, NSUB = TC / 4;
    static constexpr int TZB = 24 * HZ, TZS = TZB + (128 / TC - TZB % 32 + 64) % 32;
    static constexpr size_t SMEM = (size_t)3 * EXS * sizeof(float2) + (size_t)NSUB * TZS * sizeof(float);
    // 16 warps per SM, or what the shared memory (with a reserved kilobyte per CTA and the
    // static sums) admits: 3 or 5 at L = 128, where asking for 4 or 8 changed nothing
    // (128 x 128 x 64: 43.0 us)
    static constexpr int FIT = (int)(228 * 1024 / (SMEM + 1024 + NT * sizeof(double)));
    static constexpr int MIN_CTAS = 512 / NT < FIT ? 512 / NT : FIT;
    static_assert((R2 * TC) % NT == 0 && (R1 * TC) % NT == 0, "whole rounds of butterflies");
    static_assert(TZS % 4 == 0, "16-byte copies");
};

template <int L> constexpr int kZtCols = L == 64 ? 8 : 16;

enum ZtMode { ZT_FIELD = 0, ZT_ENERGY = 1, ZT_BOTH = 2 };

// One tile by NT threads: the CTA, or with GRP one of its 256 / NT thread groups
// (each group a tile of its own in its own slice of shared memory, its barriers
// named barriers 1 + group, so the persistent batch kernel runs the same tiles; the
// spectrum, which other CTAs of that launch wrote, is then read past L1 as in its
// other passes, ldp).
// ntile: the tile-ordered tensor copy (zws_ntx4(Kx) sub-blocks per ky
// row). ZT_ENERGY: nothing is written back, the CTA's part of the spectral energy
// sum_k w(kx) m^H N^ m goes to partials[tile]; ZT_BOTH: the field and that sum,
// taken as -Re(m^H h).
template <int L, int TC, int MODE, bool GRP = false>
__device__ __forceinline__ void zt_tile(float2 *__restrict__ S, int Kx, int Py, int64_t ss, int64_t rs, int64_t cs, int nrows,
                                        const float *__restrict__ ntile, const float2 *__restrict__ tw, int ntx, int tile,
                                        unsigned char *smraw, double *partials)
{
    using Sh = ZtShape<L, TC>;
    constexpr int R1 = Sh::R1, R2 = Sh::R2, NT = Sh::NT, RP = Sh::RP, EXS = Sh::EXS, HZ = Sh::HZ, TZB = Sh::TZB,
                  TZS = Sh::TZS, H1 = (R1 + 1) / 2;
    constexpr int Q1 = R2 * TC / NT, Q2 = R1 * TC / NT;  // rounds of a component's outer stages, of the middle
    static_assert(!GRP || (256 % NT == 0 && 256 / NT <= 15 && Sh::SMEM % 16 == 0), "thread groups");
    const int tid = GRP ? (int)threadIdx.x % NT : (int)threadIdx.x, grp = GRP ? (int)threadIdx.x / NT : 0;
    __shared__ double red[GRP ? 256 : NT];
    auto sync = [&]() {
        if constexpr (GRP) asm volatile("bar.sync %0, %1;\n" ::"r"(1 + grp), "n"(NT) : "memory");
        else __syncthreads();
    };
    // the CTA's (group's) FP64 sum, as block_partial
    auto partial = [&](double v) {
        double *r = red + grp * NT;
        r[tid] = v;
        sync();
        if (tid < 32) {
            double e = r[tid];
#pragma unroll
            for (int w = 1; w < NT / 32; ++w) e += r[tid + 32 * w];
            for (int off = 16; off > 0; off >>= 1) e += __shfl_down_sync(0xffffffffu, e, off);
            if (tid == 0) partials[tile] = e;
        }
    };
    float2 *ex = reinterpret_cast<float2 *>(smraw + (size_t)grp * Sh::SMEM);
    float *tz = reinterpret_cast<float *>(ex + 3 * EXS);
    const int c = tid % TC, j0 = tid / TC;
    const int kyi = tile / ntx, kxt = tile - kyi * ntx, kx0 = kxt * TC;
    const int ky = ky_pair_order(kyi, Py), kyf = ky > Py / 2 ? Py - ky : ky;
    const bool ok = kx0 + c < Kx;
    {
        const int ntx4 = zws_ntx4(Kx), have = ntx4 - kxt * Sh::NSUB;  // sub-blocks the row still has
        const float *src = ntile + ((size_t)kyf * ntx4 + kxt * Sh::NSUB) * TZB;
#pragma unroll
        for (int h = 0; h < Sh::NSUB; ++h)
            if (h < have)
                for (int i = tid * 4; i < TZB; i += NT * 4) cp_async16(tz + h * TZS + i, src + h * TZB + i);
    }
    float2 *col = S + (int64_t)ky * ss + kx0 + c;
    // stage 1: R1-point DFTs (upper half zero); the loads of several butterflies first
    constexpr int QB = R1 <= 8 ? 3 * Q1 : 1;
#pragma unroll
    for (int q0 = 0; q0 < 3 * Q1; q0 += QB) {
        float2 u[QB][R1];
#pragma unroll
        for (int i = 0; i < QB; ++i) {
            const int q = q0 + i, j = j0 + (q % Q1) * (NT / TC);
            const float2 *p = col + (q / Q1) * cs + j * rs;
#pragma unroll
            for (int r = 0; r < H1; ++r) {
                u[i][r] = make_float2(0.f, 0.f);
                if (ok && j + r * R2 < nrows) u[i][r] = ldp<GRP>(p + (int64_t)r * R2 * rs);
            }
        }
#pragma unroll
        for (int i = 0; i < QB; ++i) {
            const int q = q0 + i, j = j0 + (q % Q1) * (NT / TC);
            mx::DFT<R1, H1, false, float2>::run(u[i]);
            float2 *s = ex + (q / Q1) * EXS + j * RP * TC + c;
#pragma unroll
            for (int r = 0; r < R1; ++r) s[r * TC] = u[i][r];
        }
    }
    cp_async_wait_all();
    sync();
    // middle: R2-point DFTs of the three components, product, inverse DFTs, in place
    double eacc = 0.0;
#pragma unroll 1
    for (int q = 0; q < Q2; ++q) {
        const int j = j0 + q * (NT / TC);
        float2 *s = ex + j * TC + c;
        constexpr int step = RP * TC;
        float2 a[R2], b[R2], d[R2];
#pragma unroll
        for (int r = 0; r < R2; ++r) {
            a[r] = s[r * step];
            b[r] = s[EXS + r * step];
            d[r] = s[2 * EXS + r * step];
        }
#pragma unroll
        for (int r = 1; r < R2; ++r) {
            const float2 w = __ldg(&tw[r * j]);
            a[r] = zw::mul(a[r], w);
            b[r] = zw::mul(b[r], w);
            d[r] = zw::mul(d[r], w);
        }
        mx::DFT<R2, R2, false, float2>::run(a);
        mx::DFT<R2, R2, false, float2>::run(b);
        mx::DFT<R2, R2, false, float2>::run(d);
        const float *tb = tz + (c >> 2) * TZS + (c & 3);
        const float szm = j == 0 ? 1.f : -1.f;  // kz = L/2 + j: folded unless j = 0
        float2 e0 = make_float2(0.f, 0.f), e1 = e0, e2 = e0;
        auto prod_all = [&](auto syneg) {
            constexpr bool SN = decltype(syneg)::value;
#pragma unroll
            for (int m = 0; m < R2; ++m) {
                const int kzf = m < R2 / 2 ? j + R1 * m : L - j - R1 * m;
                const float *t = tb + kzf * 4;
                float txz = t[4 * HZ * 4], tyz = t[5 * HZ * 4];
                if (m == R2 / 2) {
                    txz *= szm;
                    tyz *= szm;
                } else if (m > R2 / 2) {
                    txz = -txz;
                    tyz = -tyz;
                }
                const float2 mx_ = a[m], my_ = b[m], mz_ = d[m];
                zw::product<SN>(a[m], b[m], d[m], t[0], t[HZ * 4], t[2 * HZ * 4], t[3 * HZ * 4], txz, tyz);
                if constexpr (MODE != ZT_FIELD) {
                    e0 = __ffma2_rn(mx_, a[m], e0);
                    e1 = __ffma2_rn(my_, b[m], e1);
                    e2 = __ffma2_rn(mz_, d[m], e2);
                }
            }
        };
        if (ky > Py / 2) prod_all(std::true_type{});
        else prod_all(std::false_type{});
        if constexpr (MODE != ZT_FIELD)
            if (ok) eacc -= (double)(((e0.x + e0.y) + (e1.x + e1.y) + (e2.x + e2.y)) * kx_weight<float>(kx0 + c, Kx));
        if constexpr (MODE != ZT_ENERGY) {
            mx::DFT<R2, R2, true, float2>::run(a);
            mx::DFT<R2, R2, true, float2>::run(b);
            mx::DFT<R2, R2, true, float2>::run(d);
#pragma unroll
            for (int r = 0; r < R2; ++r) {
                const float2 w = __ldg(&tw[r * j]);
                s[r * step] = r ? zw::mulc(a[r], w) : a[r];
                s[EXS + r * step] = r ? zw::mulc(b[r], w) : b[r];
                s[2 * EXS + r * step] = r ? zw::mulc(d[r], w) : d[r];
            }
        }
    }
    if constexpr (MODE == ZT_ENERGY) {
        partial(eacc);
        return;
    }
    sync();
    // stage 3: R1-point inverse DFTs, rows z < nrows stored
#pragma unroll (R1 <= 8 ? 3 * Q1 : 1)
    for (int q = 0; q < 3 * Q1; ++q) {
        const int j = j0 + (q % Q1) * (NT / TC);
        float2 u[R1];
        const float2 *s = ex + (q / Q1) * EXS + j * RP * TC + c;
#pragma unroll
        for (int r = 0; r < R1; ++r) u[r] = s[r * TC];
        mx::DFT<R1, R1, true, float2>::run(u);
        float2 *p = col + (q / Q1) * cs + j * rs;
#pragma unroll
        for (int r = 0; r < R1 / 2; ++r)
            if (ok && j + r * R2 < nrows) p[(int64_t)r * R2 * rs] = u[r];
    }
    if constexpr (MODE == ZT_BOTH) partial(eacc);
}

template <int L, int TC, int MODE>
__global__ void __launch_bounds__(ZtShape<L, TC>::NT, ZtShape<L, TC>::MIN_CTAS)
k_z_t(float2 *__restrict__ S, int Kx, int Py, int64_t ss, int64_t rs, int64_t cs, int nrows, const float *__restrict__ ntile,
      const float2 *__restrict__ tw, int ntx, double *__restrict__ partials)
{
    extern __shared__ __align__(16) unsigned char smraw[];
    zt_tile<L, TC, MODE>(S, Kx, Py, ss, rs, cs, nrows, ntile, tw, ntx, blockIdx.x, smraw, partials);
}

}  // namespace demag

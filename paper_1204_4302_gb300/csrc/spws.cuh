// Fused SP z pass for FP32 plans of z length 256 and 512 (the pass of k_sp_z2: three
// forward z transforms, the product with the kernel tables and the half-cell
// phase to one potential spectrum, one inverse z transform to the node rows), in the
// manner of k_z_ws: persistent CTAs over 8-column tiles whose input rows
// arrive by one TMA tensor copy and whose kernel block arrives by bulk copies of a
// tile-ordered copy of the tables, both one tile ahead on mbarriers (bounded waits).
//
// The three components meet in one sum, so they run one after another through one
// exchange tile: a thread keeps the 16 accumulated products of its frequencies and
// the 16 values of the current component, and the shared memory of a tile (input 48 KB,
// exchange 33 KB, kernel block 25 KB at L = 512) admits two CTAs of 256 threads per
// SM, whose phases overlap; k_sp_z2 held three exchange tiles and three components in
// registers with one CTA of 384 threads per SM. 256^3: 782 -> 406 us (DRAM floor 190).
#pragma once
#include "zt.cuh"

namespace demag {

// A read-only load that is not merged with an earlier one of the same address: the
// twiddles come from L1 four times a tile instead of holding 30 registers.
__device__ __forceinline__ float2 ld_again(const float2 *p)
{
    float2 v;
    asm volatile("ld.global.nc.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
    return v;
}

template <int L> struct SpwsShape {
    static_assert(L == 256 || L == 512, "the persistent SP z pass is built for L = 256 and 512");
    static constexpr int TC = 8, R1 = L / 16, RP = R1 + 1, NT = R1 * TC, HZ = L / 2 + 1;
    static constexpr int EX = 16 * RP * TC;                 // exchange, complex values
    static constexpr int TZB = 12 * HZ, TZS = TZB + 4;      // HZ odd, 12 HZ = 12 mod 32: TZS = 16 mod 32 banks
    static constexpr int MIN_CTAS = L == 512 ? 2 : 4;
    static_assert(TZS % 32 == 16, "the two 4-column sub-blocks in different bank halves");
};

template <int L> inline size_t spws_smem_bytes(int nrows)
{
    using Sh = SpwsShape<L>;
    const size_t stg = ((size_t)3 * nrows * Sh::TC * sizeof(float2) + 127) / 128 * 128;
    return 128 + stg + (size_t)Sh::EX * sizeof(float2) + (size_t)2 * Sh::TZS * sizeof(float) + 2 * sizeof(uint64_t);
}

// Tile t: columns kx = (t % ntx) 8 .. + 7 of the ky row ky_pair_order(t / ntx). map: S2
// [3][nz][Py][Kxp] as reals, box (16, 1, nz, 3). ttile: [Py/2+1][ntx4][3][HZ][4].
// phx, phy, phz: exp(-pi i k / P). nout = nrows + 1 <= L/2 + 1 node rows are
// stored over component 0 (the last on component 1's first plane, whose columns of
// this tile have been read).
template <int L>
__global__ void __launch_bounds__(SpwsShape<L>::NT, SpwsShape<L>::MIN_CTAS)
k_sp_ws(const __grid_constant__ CUtensorMap map, float2 *__restrict__ S, int Kx, int Py, int64_t ss, int64_t rs, int nrows,
        int nout, const float *__restrict__ ttile, const float2 *__restrict__ twg, const float2 *__restrict__ phx,
        const float2 *__restrict__ phy, const float2 *__restrict__ phz, int ntx, int ntiles)
{
    using Sh = SpwsShape<L>;
    constexpr int TC = Sh::TC, R1 = Sh::R1, RP = Sh::RP, HZ = Sh::HZ, TZB = Sh::TZB, TZS = Sh::TZS;
    constexpr unsigned TZ_BYTES = (unsigned)(2 * TZB * sizeof(float));
    extern __shared__ __align__(16) unsigned char smraw[];
    unsigned char *base = smraw + ((128 - (smem_u32(smraw) & 127)) & 127);
    const unsigned in_bytes = 3u * (unsigned)nrows * TC * (unsigned)sizeof(float2);
    const size_t stg_bytes = ((size_t)in_bytes + 127) / 128 * 128;
    float2 *stg = reinterpret_cast<float2 *>(base);            // [3][nrows][TC]
    float2 *ex = reinterpret_cast<float2 *>(base + stg_bytes);  // [16 RP][TC]
    float *tz = reinterpret_cast<float *>(ex + Sh::EX);         // [2][TZS]: [3][HZ][4] each
    uint64_t *bar = reinterpret_cast<uint64_t *>(tz + 2 * TZS);  // [0] input, [1] kernel block
    __shared__ int s_fail;
    const int tid = threadIdx.x, c = tid & (TC - 1), j2 = tid / TC;
    const int ntx4 = zws_ntx4(Kx);
    if (tid == 0) {
        s_fail = 0;
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        mbar_fence_init();
    }
    __syncthreads();
    auto tile_ky = [&](int t) { return ky_pair_order(t / ntx, Py); };
    auto issue_in = [&](int t) {
        mbar_expect_tx(&bar[0], in_bytes);
        tma_load_4d(stg, &map, 2 * (t % ntx) * TC, tile_ky(t), 0, 0, &bar[0]);
    };
    auto issue_tz = [&](int t) {
        const int ky = tile_ky(t), kyf = ky > Py / 2 ? Py - ky : ky;
        mbar_expect_tx(&bar[1], TZ_BYTES);
        const float *src = ttile + ((size_t)kyf * ntx4 + (t % ntx) * 2) * TZB;
        bulk_g2s(tz, src, TZB * (unsigned)sizeof(float), &bar[1]);
        bulk_g2s(tz + TZS, src + TZB, TZB * (unsigned)sizeof(float), &bar[1]);
    };
    int t = blockIdx.x;
    if (tid == 0 && t < ntiles) {
        issue_in(t);
        issue_tz(t);
    }
    const float2 pz = __ldg(&phz[j2]);
    const float szm = j2 == 0 ? 1.f : -1.f;  // kz = L/2 + j2: folded unless j2 = 0
    for (int k = 0; t < ntiles; t += gridDim.x, ++k) {
        const int next = t + gridDim.x;
        const unsigned par = (unsigned)(k & 1);
        const int ky = tile_ky(t), kx0 = (t % ntx) * TC;
        const float sy = ky > Py / 2 ? -1.f : 1.f;
        if (!mbar_wait_bounded(&bar[0], par, kPipeWaitCycles)) s_fail = 1;
        float2 acc[16];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            // T_x and T_z change sign with sy: they are summed first and T_y
            // takes sy instead, the common sign goes into the phase
            const int comp = i == 0 ? 0 : (i == 1 ? 2 : 1);
            // ---- stage 1 of the component (rows and outputs as in k_z_ws)
            {
                const int j1 = (tid / TC) & 15, p = L == 512 ? tid / (16 * TC) : 0;
                float2 v[16];
                const float2 *src = stg + ((size_t)comp * nrows + j1) * TC + c;
#pragma unroll
                for (int r = 0; r < 16; ++r)
                    v[r] = (r < L / 32 && j1 + 16 * r < nrows) ? src[16 * r * TC] : make_float2(0.f, 0.f);
                float2 *dst = ex + (RP * j1 + p) * TC + c;
                if constexpr (L == 512) {
                    if (p) zw::tw32_half(v);
                    zw::dft16<false>(v);
#pragma unroll
                    for (int m = 0; m < 16; ++m) dst[2 * m * TC] = v[m];
                } else {
                    zw::dft16_half_in(v);
#pragma unroll
                    for (int m = 0; m < 16; ++m) dst[m * TC] = v[m];
                }
            }
            __syncthreads();  // exchange written (and after the last component the staged input read)
            if (i == 0 && s_fail) {  // the input copy timed out; the kernel block's copy was issued
                if (tid == 0) {
                    mbar_wait_bounded(&bar[0], par, kPipeWaitCycles);
                    mbar_wait_bounded(&bar[1], par, kPipeWaitCycles);
                    atomicExch(&g_xpipe_error, 1);
                }
                return;
            }
            if (i == 2 && tid == 0 && next < ntiles) {
                fence_proxy_async_smem();
                issue_in(next);
            }
            // ---- stage 2: rows RP r + j2, twiddles, 16-point DFT, kz = j2 + R1 m
            {
                float2 v[16];
                const float2 *s = ex + j2 * TC + c;
#pragma unroll
                for (int r = 0; r < 16; ++r) v[r] = s[RP * r * TC];
#pragma unroll
                for (int r = 1; r < 16; ++r) v[r] = zw::mul(v[r], ld_again(&twg[r * j2]));
                zw::dft16<false>(v);
                if (i == 0 && !mbar_wait_bounded(&bar[1], par, kPipeWaitCycles)) s_fail = 1;
                const float *tb = tz + (c >> 2) * TZS + comp * HZ * 4 + (c & 3);
#pragma unroll
                for (int m = 0; m < 16; ++m) {
                    const int kzf = m < 8 ? j2 + R1 * m : L - j2 - R1 * m;
                    float q = tb[kzf * 4];
                    if (comp != 2) q = m < 8 ? q : (m == 8 ? q * szm : -q);  // kz flips T_x and T_y
                    if (comp == 1) q *= sy;
                    const float2 qq = make_float2(q, q);
                    acc[m] = i == 0 ? __fmul2_rn(qq, v[m]) : __ffma2_rn(qq, v[m], acc[m]);
                }
            }
            if (i < 2) __syncthreads();  // exchange read before the next component writes it
            if (i == 0 && s_fail) {  // the kernel block's copy timed out; nothing else is in flight
                if (tid == 0) {
                    mbar_wait_bounded(&bar[1], par, kPipeWaitCycles);
                    atomicExch(&g_xpipe_error, 1);
                }
                return;
            }
        }
        // phase -i Phi(kx, ky, kz) = p0 W32^m, inverse 16-point DFT, the stage-3 twiddles,
        // back to the rows this thread read
        {
            const float2 pxy = zw::mul(__ldg(&phx[min(kx0 + c, Kx - 1)]), __ldg(&phy[ky]));
            const float2 p0 = zw::mul(make_float2(sy * pxy.y, -sy * pxy.x), pz);
#pragma unroll
            for (int m = 0; m < 16; ++m) acc[m] = zw::mul(acc[m], p0);
            zw::tw32_half(acc);
            zw::dft16<true>(acc);
#pragma unroll
            for (int r = 1; r < 16; ++r) acc[r] = zw::mulc(acc[r], ld_again(&twg[r * j2]));
            float2 *o = ex + j2 * TC + c;
#pragma unroll
            for (int r = 0; r < 16; ++r) o[RP * r * TC] = acc[r];
        }
        __syncthreads();  // kernel block consumed, exchange written
        if (tid == 0 && next < ntiles) {
            fence_proxy_async_smem();
            issue_tz(next);
        }
        // ---- stage 3: rows RP n1 + k1, R1-point inverse DFT of the outputs n2 <= R1/2;
        // L = 512: the even (p = 0) or odd outputs of the 32-point DFT
        {
            const int n1 = (tid / TC) & 15, p = L == 512 ? tid / (16 * TC) : 0;
            const float2 *s = ex + RP * n1 * TC + c;
            float2 a[16];
            float2 last = make_float2(0.f, 0.f);  // output n2 = R1/2 of n1 = 0: the row z = L/2
            if constexpr (L == 512) {
                if (p == 0) {
#pragma unroll
                    for (int q = 0; q < 16; ++q) a[q] = zw::add(s[q * TC], s[(q + 16) * TC]);
                } else {
#pragma unroll
                    for (int q = 0; q < 16; ++q) a[q] = zw::sub(s[q * TC], s[(q + 16) * TC]);
                    SFor<1, 16>::run([&](auto qq) {
                        constexpr int q = decltype(qq)::value;
                        a[q] = zw::tw<32, q, true>(a[q]);
                    });
                }
            } else {
#pragma unroll
                for (int q = 0; q < 16; ++q) a[q] = s[q * TC];
            }
            const bool edge = nout > L / 2 && n1 == 0 && p == 0;
            if (edge) {
#pragma unroll
                for (int q = 0; q < 16; ++q) last = (q & 1) ? zw::sub(last, a[q]) : zw::add(last, a[q]);
            }
            zw::idft16_lo(a);
            if (kx0 + c < Kx) {
                float2 *col = S + (int64_t)ky * ss + kx0 + c;
#pragma unroll
                for (int m = 0; m < 8; ++m) {
                    const int z = n1 + 16 * (L == 512 ? 2 * m + p : m);
                    if (z < nout) col[(int64_t)z * rs] = a[m];
                }
                if (edge) col[(int64_t)(L / 2) * rs] = last;
            }
        }
        __syncthreads();  // exchange read before the next tile's stage 1 writes it
    }
}

}  // namespace demag

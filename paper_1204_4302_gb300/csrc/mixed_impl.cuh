// Launchers of the mixed-radix passes (transform lengths that are not
// powers of two): stage plans and launches of the kernels in mixed.cuh.
#pragma once
#include <string.h>

#include "launch_util.cuh"
#include "mix2.cuh"
#include "mixed.cuh"
#include "plan.h"

namespace demag {

namespace {

// ceil(2^32 / d): n / d == umulhi(n, magic) for n d < 2^32 (d == 1 apart)
unsigned magic_of(int d) { return d <= 1 ? 0u : (unsigned)(((1ull << 32) + (unsigned)d - 1) / (unsigned)d); }

// Elements per tile of the mixed-radix kernels: the column and row passes
// hold two buffers, the z pass six (three components, ping-pong).
template <typename T> constexpr int gen_tile_elems(bool zpass)
{
    return sizeof(T) == 4 ? (zpass ? 2048 : 4096) : (zpass ? 1024 : 2048);
}

// Stage radices of the mixed-radix passes: every length <= 32 with prime
// factors 2, 3, 5, 7 (the in-register DFTs that mixed.cuh instantiates).
bool gen_stage_radix(int r)
{
    if (r < 2 || r > 32) return false;
    for (int f : {2, 3, 5, 7})
        while (r % f == 0) r /= f;
    return r == 1;
}

// Fewest stages (at most `depth`), then the smallest largest radix, radices
// in non-increasing order; false if L has no such split.
bool gen_split(int m, int maxr, int depth, int *cur, int n, int *best, int &bn, int &bmax)
{
    if (m == 1) {
        int mx = 0;
        for (int i = 0; i < n; ++i) mx = cur[i] > mx ? cur[i] : mx;
        if (bn == 0 || n < bn || (n == bn && mx < bmax)) {
            for (int i = 0; i < n; ++i) best[i] = cur[i];
            bn = n;
            bmax = mx;
        }
        return true;
    }
    if (depth == 0) return false;
    bool any = false;
    for (int r = maxr; r >= 2; --r)
        if (m % r == 0 && gen_stage_radix(r)) {
            cur[n] = r;
            any |= gen_split(m / r, r, depth - 1, cur, n + 1, best, bn, bmax);
        }
    return any;
}

// Stage plan of a mixed-radix transform of length L (a product of 2, 3, 5
// and 7, L < 2048) over tiles of about `tile` elements, radices <= maxr;
// comps components per grid column share the tile (z pass: 3).
bool gen_plan(int L, int tile, GenRadix &g, int maxr, int comps = 1)
{
    memset(&g, 0, sizeof g);
    if (L < 2 || L >= 2048) return false;
    g.L = L;
    const int cols = tile / L > 1 ? tile / L : 1;  // grid columns (rows of the x passes) per tile
    g.TC = comps * cols;                             // tile columns: the components side by side
    g.mCols = magic_of(cols);
    int cur[4], r[4], n = 0, mx = 0;
    if (!gen_split(L, maxr, 4, cur, 0, r, n, mx) || n == 0) return false;
    int NS = 1;
    for (int s = 0; s < n; ++s) {
        g.r[s] = r[s];
        g.NS[s] = NS;
        g.mNS[s] = magic_of(NS);
        g.mPer[s] = magic_of(L / r[s] * g.TC);
        g.mNB[s] = magic_of(L / r[s]);
        NS *= r[s];
    }
    g.n = n;
    g.mTC = magic_of(g.TC);
    g.mL = magic_of(L);
    g.mL1 = magic_of(L + 1);
    return true;
}

// Largest stage radix of the general z passes. FP32: 32 where that saves a stage
// against 16 above length 128 (an exchange and a barrier per direction; us of the z pass
// with 16 and with 32: SP 200^3 106 / 97, 270^3 267 / 224, 300^3 371 / 319, DM
// 128 x 128 x 600 207 / 185), else 16, whose kernel is the smaller (SP 120^3 26.7, 28.6
// with 32). FP64: 16, as a thread of the larger radices holds twice the registers
// (SP 200^3 1068, 1523 with 32; 300^3 4194, 5938).
template <typename T> int gen_z_radix(int L)
{
    if (sizeof(T) == 8 || L <= 128) return 16;
    GenRadix a, b;
    const bool big = gen_plan(L, gen_tile_elems<T>(true), b, 32, 3) && b.r[b.n - 1] >= gen_min_radix(32);
    return big && !(gen_plan(L, gen_tile_elems<T>(true), a, 16, 3) && a.n <= b.n) ? 32 : 16;
}

// Two-stage plan L = R1 R2 with radices <= maxr: the smallest largest radix,
// the larger one first (forward: its inputs are half empty) or last (inverse: half
// of its outputs are not formed). False where L has no such split.
bool mix2_split(int L, int maxr, bool larger_first, Mix2 &g)
{
    int best = 0;
    for (int r = 2; r <= maxr; ++r)
        if (L % r == 0 && gen_stage_radix(r) && gen_stage_radix(L / r) && L / r <= r && (best == 0 || r < best)) best = r;
    if (!best) return false;
    memset(&g, 0, sizeof g);
    g.L = L;
    g.R1 = larger_first ? best : L / best;
    g.R2 = L / g.R1;
    g.m1 = magic_of(g.R1);
    g.m2 = magic_of(g.R2);
    return true;
}

// Column passes: groups of TC threads, G <= gmax of them in whole warps, the
// choice that leaves the fewest butterfly slots of both stages empty (the
// larger G of two equal ones).
void mix2_groups(Mix2 &g, int TC, int gmax)
{
    double best = -1;
    for (int G = 1; G <= gmax; ++G) {
        if ((G * TC) % 32) continue;
        const int n1 = (g.R2 + G - 1) / G, n2 = (g.R1 + G - 1) / G;
        const double use = 2.0 * g.L / ((double)G * (n1 * g.R1 + n2 * g.R2)) + (G * TC >= 96 ? 0.2 : 0.0) + 1e-3 * G;
        if (use > best) {
            best = use;
            g.G = G;
        }
    }
}

// Row passes: rows per CTA, one butterfly per thread and stage.
void mix2_rows(Mix2 &g)
{
    const int big = g.R1 > g.R2 ? g.R1 : g.R2;
    g.G = kMix2RowThreads / big;
    g.RP = g.R1 | 1;
}
constexpr int kMix2RowRadix = 28;  // largest radix of the row passes' two-stage lengths (up to 512)

template <typename T, int TC, int MAXR>
cudaError_t mix2_col_launch(bool inv, const typename Cplx<T>::type *in, typename Cplx<T>::type *out, int width, int nslabs,
                            int64_t iss, int64_t irs, int nin, int64_t oss, int64_t ors, int nout,
                            const typename Cplx<T>::type *tw, Mix2 g, cudaStream_t st)
{
    using C = typename Cplx<T>::type;
    // 64-byte rows: an odd group stride keeps two rows of a half warp apart
    g.RP = TC * sizeof(C) >= 128 ? g.R1 : (g.R1 | 1);
    mix2_groups(g, TC, (sizeof(T) == 4 ? 256 : 128) / TC);
    // tiles within a slab where rounding its width up to the tile costs
    // little, so that a tile's rows start on the rows' own alignment
    const int up = (width + TC - 1) / TC * TC;
    const int vw = up * 8 <= width * 9 ? up : width;
    const int64_t grid = ((int64_t)vw * nslabs + TC - 1) / TC;
    const size_t sm = (size_t)g.R2 * g.RP * TC * sizeof(C);
    cudaError_t e;
    if (inv) {
        if ((e = allow_smem<k_mix2_col<T, true, TC, MAXR>>(sm)) != cudaSuccess) return e;
        k_mix2_col<T, true, TC, MAXR><<<(unsigned)grid, g.G * TC, sm, st>>>(in, out, vw, width, nslabs, iss, (int)irs, nin, oss,
                                                                          (int)ors, nout, tw, g);
    } else {
        if ((e = allow_smem<k_mix2_col<T, false, TC, MAXR>>(sm)) != cudaSuccess) return e;
        k_mix2_col<T, false, TC, MAXR><<<(unsigned)grid, g.G * TC, sm, st>>>(in, out, vw, width, nslabs, iss, (int)irs, nin, oss,
                                                                           (int)ors, nout, tw, g);
    }
    return cudaGetLastError();
}

// Two-stage plan of the z pass: R1 <= 32 and R2 <= 16 with the least of
// max(R1, 3 R2), the values a thread holds in the outer and in the middle stages.
bool mix2_zsplit(int L, Mix2 &g)
{
    int best = 0, cost = 0;
    for (int r = 2; r <= 32; ++r)
        if (L % r == 0 && gen_stage_radix(r) && gen_stage_radix(L / r) && L / r <= 16) {
            const int c = r > 3 * (L / r) ? r : 3 * (L / r);
            if (!best || c < cost) {
                best = r;
                cost = c;
            }
        }
    if (!best) return false;
    memset(&g, 0, sizeof g);
    g.L = L;
    g.R1 = best;
    g.R2 = L / best;
    g.RP = g.R1 | 1;
    return true;
}

template <typename T, int MAXR2>
cudaError_t mix2_z_launch(typename Cplx<T>::type *S, int Kx, int Py, int64_t ss, int64_t rs, int64_t cs, int nrows,
                          const T *nhat, const T *ntile, const typename Cplx<T>::type *tw, const Mix2 &g, cudaStream_t st)
{
    constexpr int TC = sizeof(T) == 4 ? 8 : 4;
    using C = typename Cplx<T>::type;
    const size_t sm = (size_t)3 * g.R2 * g.RP * TC * sizeof(C) +
                      (sizeof(T) == 4 ? 2 * (size_t)mix2_tensor_stride(g.L / 2 + 1) * sizeof(T) : 0);
    cudaError_t e = allow_smem<k_mix2_z<T, TC, MAXR2>>(sm);
    if (e != cudaSuccess) return e;
    const int ntx = (Kx + TC - 1) / TC;
    k_mix2_z<T, TC, MAXR2><<<(unsigned)(ntx * Py), g.R1 * TC, sm, st>>>(S, Kx, Py, ss, rs, cs, nrows, nhat, ntile, tw, ntx, g);
    return cudaGetLastError();
}

}  // namespace

template <typename T, int MAXR>
cudaError_t gen_z_launch(int L, typename Cplx<T>::type *S, int ncols, int width, int64_t ss, int64_t rs, int64_t cs, int nrows,
                         const T *nhat, int Py, int Kx, const typename Cplx<T>::type *tw, int twstride, cudaStream_t st)
{
    GenRadix g;
    if (!gen_plan(L, gen_tile_elems<T>(true), g, MAXR, 3)) return cudaErrorInvalidValue;
    const int cols = g.TC / 3;
    const size_t sm = 2 * swsize(L * g.TC) * sizeof(typename Cplx<T>::type);
    cudaError_t e = allow_smem<k_gen_zconv<T, MAXR>>(sm);
    if (e != cudaSuccess) return e;
    k_gen_zconv<T, MAXR><<<(ncols + cols - 1) / cols, kGenThreads, sm, st>>>(
        S, ncols, width, magic_of(width), ss, rs, cs, nrows, nhat, Py, Kx, tw, twstride, g);
    return cudaGetLastError();
}

template <typename T, int MAXR>
cudaError_t gen_sp_z_launch(int L, typename Cplx<T>::type *S, int ncols, int width, int64_t ss, int64_t rs, int64_t cs,
                            int nrows, int nout, const T *that, int Py, int Kx, const typename Cplx<T>::type *tw,
                            const typename Cplx<T>::type *phx, const typename Cplx<T>::type *phy,
                            const typename Cplx<T>::type *phz, cudaStream_t st)
{
    GenRadix g3, g1;
    if (!gen_plan(L, gen_tile_elems<T>(true), g3, MAXR, 3)) return cudaErrorInvalidValue;
    if (!gen_plan(L, gen_tile_elems<T>(true), g1, MAXR, 1)) return cudaErrorInvalidValue;
    const int cols = g1.TC;
    const size_t sm = 2 * swsize(L * g3.TC) * sizeof(typename Cplx<T>::type);
    cudaError_t e = allow_smem<k_gen_sp_zconv<T, MAXR>>(sm);
    if (e != cudaSuccess) return e;
    k_gen_sp_zconv<T, MAXR><<<(ncols + cols - 1) / cols, kGenThreads, sm, st>>>(
        S, ncols, width, magic_of(width), ss, rs, cs, nrows, nout, that, Py, Kx, tw, phx, phy, phz, g3, g1);
    return cudaGetLastError();
}

// the FP32 kernels of largest radix 32: a translation unit of their own (compile time)
extern template cudaError_t gen_z_launch<float, 32>(int, float2 *, int, int, int64_t, int64_t, int64_t, int, const float *,
                                                    int, int, const float2 *, int, cudaStream_t);
extern template cudaError_t gen_sp_z_launch<float, 32>(int, float2 *, int, int, int64_t, int64_t, int64_t, int, int,
                                                       const float *, int, int, const float2 *, const float2 *,
                                                       const float2 *, const float2 *, cudaStream_t);

template <typename T>
bool MixedPasses<T>::z_tiled(int L)
{
    Mix2 g;
    return sizeof(T) == 4 && mix2_zsplit(L, g);
}

template <typename T>
cudaError_t MixedPasses<T>::x_fwd(int L, const XIn<T> &a, int nrows, int nvalid, C *out, int64_t out_rs,
                                  const C *twx, cudaStream_t st)
{
    if (nrows <= 0) return cudaSuccess;
    Mix2 m;
    if (nvalid <= L && mix2_split(L, kMix2RowRadix, true, m)) {
        mix2_rows(m);
        const size_t sm = (size_t)m.G * m.R2 * m.RP * sizeof(C);
        const int grid = (nrows + m.G - 1) / m.G;
        const unsigned mh = magic_of(L / 2 + 1);
        cudaError_t e;
        if (m.R1 <= 16) {
            if ((e = allow_smem<k_mix2_x_fwd<T, 16>>(sm)) != cudaSuccess) return e;
            k_mix2_x_fwd<T, 16><<<grid, kMix2RowThreads, sm, st>>>(a, nrows, nvalid, out, out_rs, twx, m, mh);
        } else {
            if ((e = allow_smem<k_mix2_x_fwd<T, kMix2RowRadix>>(sm)) != cudaSuccess) return e;
            k_mix2_x_fwd<T, kMix2RowRadix><<<grid, kMix2RowThreads, sm, st>>>(a, nrows, nvalid, out, out_rs, twx, m, mh);
        }
        return cudaGetLastError();
    }
    GenRadix g;
    if (!gen_plan(L, gen_tile_elems<T>(false), g, kGenMaxRadixRows)) return cudaErrorInvalidValue;
    const size_t sm = gen_io_buffers(g.n, false) * swsize(L * g.TC) * sizeof(C);
    cudaError_t e = allow_smem<k_gen_x_fwd<T>>(sm);
    if (e != cudaSuccess) return e;
    k_gen_x_fwd<T><<<(nrows + g.TC - 1) / g.TC, kGenThreads, sm, st>>>(a, nrows, nvalid, out, out_rs, twx, g);
    return cudaGetLastError();
}

template <typename T>
int MixedPasses<T>::x_blocks(int L, int nrows)
{
    Mix2 m;
    if (mix2_split(L, kMix2RowRadix, false, m)) {  // the inverse pass's CTAs
        mix2_rows(m);
        return (nrows + m.G - 1) / m.G;
    }
    GenRadix g;
    if (!gen_plan(L, gen_tile_elems<T>(false), g, kGenMaxRadixRows)) return 1;
    return (nrows + g.TC - 1) / g.TC;
}

template <typename T>
cudaError_t MixedPasses<T>::x_inv(int L, const C *in, int64_t in_rs, int nrows, int nvalid, const XOut<T> &o,
                                  const C *twx, cudaStream_t st, int *blocks)
{
    int unused, &grid = blocks ? *blocks : unused;
    grid = 0;
    if (nrows <= 0) return cudaSuccess;
    Mix2 m;
    if (mix2_split(L, kMix2RowRadix, false, m)) {
        if (nvalid > L + 1) return cudaErrorInvalidValue;
        mix2_rows(m);
        const size_t sm = (size_t)m.G * m.R2 * m.RP * sizeof(C);
        grid = (nrows + m.G - 1) / m.G;
        cudaError_t e;
        if (m.R2 <= 16) {
            if ((e = allow_smem<k_mix2_x_inv<T, 16>>(sm)) != cudaSuccess) return e;
            k_mix2_x_inv<T, 16><<<grid, kMix2RowThreads, sm, st>>>(in, in_rs, nrows, nvalid, o, twx, m);
        } else {
            if ((e = allow_smem<k_mix2_x_inv<T, kMix2RowRadix>>(sm)) != cudaSuccess) return e;
            k_mix2_x_inv<T, kMix2RowRadix><<<grid, kMix2RowThreads, sm, st>>>(in, in_rs, nrows, nvalid, o, twx, m);
        }
        return cudaGetLastError();
    }
    GenRadix g;
    if (!gen_plan(L, gen_tile_elems<T>(false), g, kGenMaxRadixRows)) return cudaErrorInvalidValue;
    const size_t sm = gen_io_buffers(g.n, true) * swsize(L * g.TC) * sizeof(C);
    cudaError_t e = allow_smem<k_gen_x_inv<T>>(sm);
    if (e != cudaSuccess) return e;
    grid = (nrows + g.TC - 1) / g.TC;
    k_gen_x_inv<T><<<grid, kGenThreads, sm, st>>>(in, in_rs, nrows, nvalid, o, twx, g);
    return cudaGetLastError();
}

template <typename T>
cudaError_t MixedPasses<T>::col(int L, bool inv, const C *in, C *out, int ncols, int width, int64_t iss, int64_t irs,
                                int nin, int64_t oss, int64_t ors, int nout, const C *tw, int twstride, cudaStream_t st)
{
    if (ncols <= 0) return cudaSuccess;
    Mix2 m;
    // the pruned field passes (the setup's full transforms take the general kernel)
    if (twstride == 1 && ncols % width == 0 && irs * L < (1ll << 31) && ors * L < (1ll << 31) &&
        (inv ? nin == L && 2 * (nout - 1) <= L : nout == L && 2 * nin <= L) && mix2_split(L, 32, !inv, m)) {
        constexpr int TCL = 128 / (int)sizeof(C);  // a 128-byte line; half of it where the tile would leave room for few CTAs
        const int nslabs = ncols / width, big = m.R1 > m.R2 ? m.R1 : m.R2;
        if (big <= 16) return mix2_col_launch<T, TCL, 16>(inv, in, out, width, nslabs, iss, irs, nin, oss, ors, nout, tw, m, st);
        if (L <= 576) return mix2_col_launch<T, TCL, 28>(inv, in, out, width, nslabs, iss, irs, nin, oss, ors, nout, tw, m, st);
        return mix2_col_launch<T, TCL / 2, 32>(inv, in, out, width, nslabs, iss, irs, nin, oss, ors, nout, tw, m, st);
    }
    GenRadix g;
    if (!gen_plan(L, gen_tile_elems<T>(false), g, kGenMaxRadixRows)) return cudaErrorInvalidValue;
    const size_t sm = gen_io_buffers(g.n, true) * swsize(L * g.TC) * sizeof(C);
    const unsigned mw = magic_of(width);
    const int grid = (ncols + g.TC - 1) / g.TC;
    cudaError_t e;
    if (inv) {
        if ((e = allow_smem<k_gen_col<T, true>>(sm)) != cudaSuccess) return e;
        k_gen_col<T, true><<<grid, kGenThreads, sm, st>>>(in, out, ncols, width, mw, iss, irs, nin, oss, ors, nout, tw,
                                                          twstride, g);
    } else {
        if ((e = allow_smem<k_gen_col<T, false>>(sm)) != cudaSuccess) return e;
        k_gen_col<T, false><<<grid, kGenThreads, sm, st>>>(in, out, ncols, width, mw, iss, irs, nin, oss, ors, nout,
                                                           tw, twstride, g);
    }
    return cudaGetLastError();
}

template <typename T>
cudaError_t MixedPasses<T>::zconv(int L, C *S, int ncols, int width, int64_t ss, int64_t rs, int64_t cs, int nrows,
                                  const T *nhat, int Py, int Kx, const C *tw, int twstride, cudaStream_t st,
                                  const T *ntile)
{
    if (ncols <= 0) return cudaSuccess;
    if (nrows > L) return cudaErrorInvalidValue;
    Mix2 m;
    if (twstride == 1 && width == Kx && ncols == Py * Kx && 2 * nrows <= L && (Py == 1 || Py % 2 == 0) &&
        (sizeof(T) != 4 || (ntile && ((uintptr_t)ntile & 15) == 0)) && mix2_zsplit(L, m))
        return m.R2 <= 10 ? mix2_z_launch<T, 10>(S, Kx, Py, ss, rs, cs, nrows, nhat, ntile, tw, m, st)
                          : mix2_z_launch<T, 16>(S, Kx, Py, ss, rs, cs, nrows, nhat, ntile, tw, m, st);
    if constexpr (sizeof(T) == 4)
        if (gen_z_radix<T>(L) == 32)
            return gen_z_launch<T, 32>(L, S, ncols, width, ss, rs, cs, nrows, nhat, Py, Kx, tw, twstride, st);
    return gen_z_launch<T, 16>(L, S, ncols, width, ss, rs, cs, nrows, nhat, Py, Kx, tw, twstride, st);
}

template <typename T>
cudaError_t MixedPasses<T>::sp_zconv(int L, C *S, int ncols, int width, int64_t ss, int64_t rs, int64_t cs,
                                     int nrows, int nout, const T *that, int Py, int Kx, const C *tw, const C *phx,
                                     const C *phy, const C *phz, cudaStream_t st)
{
    if (ncols <= 0) return cudaSuccess;
    if (2 * nrows > L || nout != nrows + 1 || cs != (int64_t)nrows * rs) return cudaErrorInvalidValue;
    if constexpr (sizeof(T) == 4)
        if (gen_z_radix<T>(L) == 32)
            return gen_sp_z_launch<T, 32>(L, S, ncols, width, ss, rs, cs, nrows, nout, that, Py, Kx, tw, phx, phy, phz, st);
    return gen_sp_z_launch<T, 16>(L, S, ncols, width, ss, rs, cs, nrows, nout, that, Py, Kx, tw, phx, phy, phz, st);
}

}  // namespace demag

// Two-stage mixed-radix passes: transforms of length L = R1 R2 with
// R1, R2 <= 32 products of 2, 3, 5 and 7 (every even 7-smooth length up to
// 1024 but seven, see mix2_plan). Same inputs, outputs and epilogues as the
// general kernels of mixed.cuh, which keep the lengths of three and more stages and
// the unpruned transforms of the tensor setup.
//
// What bounds these passes is the instructions per point, so the runtime
// length costs as few as it can:
//  * a thread keeps its column (or its row and butterfly) for a whole stage;
//    addresses advance by one constant per element, with no division per element;
//  * one shared-memory exchange between the stages, its rows padded to an odd
//    stride where needed for conflict-free access, and no swizzle arithmetic;
//  * the zero padding is a property of the in-register DFTs: the first
//    stage's inputs r >= (R1 + 1) / 2 are zero at compile time (rows j + r R2 with
//    j < R2 are then at or beyond L / 2), and only the outputs r <= R2 / 2 of an
//    inverse last stage are formed.
// Against the general kernels (120-190 instructions per point, now 40-90), FP32: 130^3
// padded to 270^3, x forward 67 -> 29 us, y 74 -> 39 and 80 -> 49, z 300 -> 137, x inverse
// 66 -> 40; 300 x 260 x 100 padded to 600 x 540 x 256, x forward 196 -> 92, y 226 -> 142
// and 226 -> 173, x inverse 127 -> 97. Still latency-bound: 35-50% of the issue slots.
#pragma once
#include "mixed.cuh"
#include "fft2.cuh"

namespace demag {

// Stage plan of a pass. RP: exchange rows per first-stage group (R1, or R1 + 1).
struct Mix2 {
    int L, R1, R2, RP;
    int G;        // butterfly groups per CTA (column passes), rows per CTA (row passes)
    unsigned m1;  // row passes: division by R1, and by R2
    unsigned m2;
};

namespace mx {

// a + c t with a real constant c, one packed instruction for float2
template <typename C> __device__ __forceinline__ C cfma(decltype(C::x) c, C t, C a)
{
    return cmk<C>(a.x + c * t.x, a.y + c * t.y);
}
template <> __device__ __forceinline__ float2 cfma<float2>(float c, float2 t, float2 a)
{
    return __ffma2_rn(make_float2(c, c), t, a);
}
template <typename C> __device__ __forceinline__ C cscale(decltype(C::x) c, C t) { return cmk<C>(c * t.x, c * t.y); }
template <> __device__ __forceinline__ float2 cscale<float2>(float c, float2 t) { return __fmul2_rn(make_float2(c, c), t); }
// a - i b and a + i b
template <typename C> __device__ __forceinline__ C add_mi(C a, C b) { return cmk<C>(a.x + b.y, a.y - b.x); }
template <typename C> __device__ __forceinline__ C add_pi(C a, C b) { return cmk<C>(a.x - b.y, a.y + b.x); }

__host__ __device__ constexpr int split_of(int R) { return R % 4 == 0 && R > 4 ? 4 : small_prime_factor(R); }
__host__ __device__ constexpr int imin(int a, int b) { return a < b ? a : b; }
__host__ __device__ constexpr int nz_of(int NZ, int q, int P) { return NZ > q ? (NZ - q + P - 1) / P : 0; }

// DFT of R points of which the inputs v[NZ..R) are zero (not read), natural
// order in and out; outputs that are not used cost nothing.
template <int R, int NZ, bool INV, typename C> struct DFT {
    static __device__ __forceinline__ void run(C *v)
    {
        using T = decltype(C::x);
        if constexpr (R == 1) {
            return;
        } else if constexpr (NZ == 0) {
#pragma unroll
            for (int k = 0; k < R; ++k) v[k] = cmk<C>(0, 0);
        } else if constexpr (NZ == 1) {
#pragma unroll
            for (int k = 1; k < R; ++k) v[k] = v[0];
        } else if constexpr (R == 2) {
            const C a = v[0], b = v[1];
            v[0] = cadd(a, b);
            v[1] = csub(a, b);
        } else if constexpr (R == 4) {
            const C a0 = v[0], a1 = v[1];
            C s0 = a0, d0 = a0, s1 = a1, d1 = a1;
            if constexpr (NZ > 2) {
                s0 = cadd(a0, v[2]);
                d0 = csub(a0, v[2]);
            }
            if constexpr (NZ > 3) {
                s1 = cadd(a1, v[3]);
                d1 = csub(a1, v[3]);
            }
            v[0] = cadd(s0, s1);
            v[2] = csub(s0, s1);
            v[1] = INV ? add_pi(d0, d1) : add_mi(d0, d1);
            v[3] = INV ? add_mi(d0, d1) : add_pi(d0, d1);
        } else if constexpr (split_of(R) == R) {
            // odd prime: the pair form of dft_odd
            constexpr int H = (R - 1) / 2;
            C t[H], u[H];
#pragma unroll
            for (int k = 0; k < H; ++k) {
                t[k] = u[k] = cmk<C>(0, 0);
                if (R - 1 - k < NZ) {
                    t[k] = cadd(v[k + 1], v[R - 1 - k]);
                    u[k] = csub(v[k + 1], v[R - 1 - k]);
                } else if (k + 1 < NZ) {
                    t[k] = u[k] = v[k + 1];
                }
            }
            const C x0 = v[0];
            C y0 = x0;
#pragma unroll
            for (int k = 0; k < H; ++k)
                if (k + 1 < NZ) y0 = cadd(y0, t[k]);
            v[0] = y0;
#pragma unroll
            for (int m = 1; m <= H; ++m) {
                C a = x0, b = cmk<C>(0, 0);
#pragma unroll
                for (int k = 1; k <= H; ++k) {
                    if (k >= NZ) continue;
                    const int q = (k * m) % R;
                    const T cq = (T)(q <= H ? cos_tab<R>(q) : cos_tab<R>(R - q));
                    const T sq = (T)(q <= H ? sin_tab<R>(q) : -sin_tab<R>(R - q));
                    a = cfma(cq, t[k - 1], a);
                    b = k == 1 ? cscale(sq, u[0]) : cfma(sq, u[k - 1], b);
                }
                v[m] = INV ? add_pi(a, b) : add_mi(a, b);
                v[R - m] = INV ? add_mi(a, b) : add_pi(a, b);
            }
        } else {
            constexpr int P = split_of(R), Q = R / P;
            C sub[P][Q];
#pragma unroll
            for (int q = 0; q < P; ++q)
#pragma unroll
                for (int m = 0; m < Q; ++m)
                    if (m * P + q < NZ) sub[q][m] = v[m * P + q];
            SFor<0, P>::run([&](auto qq) {
                constexpr int q = decltype(qq)::value;
                if constexpr (q < NZ) DFT<Q, nz_of(NZ, q, P), INV, C>::run(sub[q]);
            });
            SFor<0, Q>::run([&](auto kk) {
                constexpr int k = decltype(kk)::value;
                C t[P];
                if constexpr (P == 2 && 4 * k == R && NZ > 1) {  // the twiddle is -+i: folded into the adds
                    v[k] = INV ? add_pi(sub[0][k], sub[1][k]) : add_mi(sub[0][k], sub[1][k]);
                    v[k + Q] = INV ? add_mi(sub[0][k], sub[1][k]) : add_pi(sub[0][k], sub[1][k]);
                } else {
                    SFor<0, P>::run([&](auto qq) {
                        constexpr int q = decltype(qq)::value;
                        if constexpr (q < NZ) t[q] = twmul<R, q * k, INV>(sub[q][k]);
                    });
                    DFT<P, imin(P, NZ), INV, C>::run(t);
#pragma unroll
                    for (int s2 = 0; s2 < P; ++s2) v[k + Q * s2] = t[s2];
                }
            });
        }
    }
};

// f(std::integral_constant<int, R>) for the stage radix R (<= MAXR) of a plan, or
// for the compile-time radix FIXED where it is not 0
template <int MAXR, int FIXED = 0, typename F> __device__ __forceinline__ void with_radix(int R, F &&f)
{
    if constexpr (FIXED != 0) {
        f(std::integral_constant<int, FIXED>{});
        return;
    }
#define DEMAG_R(N) case N: if constexpr (N <= MAXR) f(std::integral_constant<int, N>{}); break;
    switch (R) {
        DEMAG_R(2) DEMAG_R(3) DEMAG_R(4) DEMAG_R(5) DEMAG_R(6) DEMAG_R(7) DEMAG_R(8) DEMAG_R(9) DEMAG_R(10)
        DEMAG_R(12) DEMAG_R(14) DEMAG_R(15) DEMAG_R(16) DEMAG_R(18) DEMAG_R(20) DEMAG_R(21) DEMAG_R(24)
        DEMAG_R(25) DEMAG_R(27) DEMAG_R(28) DEMAG_R(30) DEMAG_R(32)
    default: break;
    }
#undef DEMAG_R
}

// v[r] *= W_L^(r k) (or its conjugate), r = 1 .. R - 1
template <int R, bool INV, typename C>
__device__ __forceinline__ void twiddle(C *v, int kstep, const C *__restrict__ tw)
{
#pragma unroll
    for (int r = 1; r < R; ++r) {
        const C w = __ldg(&tw[r * kstep]);
        v[r] = INV ? cmulc(v[r], w) : cmul(v[r], w);
    }
}

}  // namespace mx

// Column pass: TC columns per CTA (one 128-byte line of complex values), tile
// column f = slab * vw + off with off < width (vw is width, or width rounded
// up to the tile so that tiles start on the row's alignment). HALF_IN: forward,
// rows >= L / 2 are zero (nin <= L / 2); otherwise the inverse, of which rows
// <= L / 2 are formed. Thread (g, c): butterflies g, g + G, ... of column c.
// C1, C2: the radices where they are known at compile time (the power-of-two
// lengths 512 and 1024), else 0 and the plan's.
template <typename T, bool INV, int TC, int MAXR, int C1 = 0, int C2 = 0>
__global__ void __launch_bounds__(sizeof(T) == 4 ? 256 : 128, MAXR <= 16 ? (sizeof(T) == 4 ? 3 : 4) : 2)
k_mix2_col(const typename Cplx<T>::type *__restrict__ in, typename Cplx<T>::type *__restrict__ out, int vw, int width,
           int nslabs, int64_t iss, int irs, int nin, int64_t oss, int ors, int nout,
           const typename Cplx<T>::type *__restrict__ tw, const Mix2 g)
{
    using C = typename Cplx<T>::type;
    extern __shared__ __align__(16) unsigned char smraw[];
    C *ex = reinterpret_cast<C *>(smraw);
    const int c = threadIdx.x % TC, j0 = threadIdx.x / TC;
    const int f = blockIdx.x * TC + c, slab = f / vw, off = f - slab * vw;
    const bool ok = slab < nslabs && off < width;
    const C *src = in + (int64_t)slab * iss + off;
    C *dst = out + (int64_t)slab * oss + off;
    const int R1 = C1 ? C1 : g.R1, R2 = C2 ? C2 : g.R2, G = C1 ? 256 / TC : g.G;
    const int RP = C1 ? (TC * (int)sizeof(C) >= 128 ? C1 : (C1 | 1)) : g.RP;
    mx::with_radix<MAXR, C1>(R1, [&](auto rr) {
        constexpr int R = decltype(rr)::value, H = INV ? R : (R + 1) / 2;
        const unsigned step = (unsigned)(R2 * irs);
        for (int j = j0; j < R2; j += G) {
            C u[R];
            unsigned a = (unsigned)(j * irs);
            int row = j;
#pragma unroll
            for (int r = 0; r < H; ++r) {
                u[r] = cmk<C>(0, 0);
                if (ok && row < nin) u[r] = src[a];
                a += step;
                row += R2;
            }
            mx::DFT<R, H, INV, C>::run(u);
            C *s = ex + j * RP * TC + c;
#pragma unroll
            for (int r = 0; r < R; ++r) s[r * TC] = u[r];
        }
    });
    __syncthreads();
    mx::with_radix<MAXR, C2>(R2, [&](auto rr) {
        constexpr int R = decltype(rr)::value, H = INV ? R / 2 + 1 : R;
        const int step = RP * TC;
        const unsigned ostep = (unsigned)(R1 * ors);
        for (int j = j0; j < R1; j += G) {
            C v[R];
            const C *s = ex + j * TC + c;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                v[r] = *s;
                s += step;
            }
            mx::twiddle<R, INV>(v, j, tw);
            mx::DFT<R, R, INV, C>::run(v);
            unsigned a = (unsigned)(j * ors);
            int row = j;
#pragma unroll
            for (int r = 0; r < (H < R ? H : R); ++r) {
                if (ok && row < nout) dst[a] = v[r];
                a += ostep;
                row += R1;
            }
        }
    });
}

// Floats between the two 4-column sub-blocks of a tensor tile in shared
// memory: 16 modulo 32 banks, so that the eight columns of four frequencies are
// read without conflicts.
__host__ __device__ inline int mix2_tensor_stride(int HZ) { return 24 * HZ + (16 - 24 * HZ % 32 + 32) % 32; }

// Threads of a row-pass CTA: with 256 the three barriers of fewer, larger CTAs left the
// scheduler idle (x forward at 130^3: 41 us with 256 and serial loads, 29 with 128 and the
// loads issued together).
constexpr int kMix2RowThreads = 128;

// Real-to-complex rows (as k_gen_x_fwd): g.G rows per CTA, one butterfly of
// one row per thread and stage (g.G R1 and g.G R2 <= the CTA), the packed
// transform back in the exchange in natural order, then the split by pairs
// (k, L - k), which share both values, the sums and the twiddle.
template <typename T, int MAXR>
__global__ void __launch_bounds__(kMix2RowThreads, (sizeof(T) == 4 ? (MAXR <= 16 ? 3 : 2) : 1) * 256 / kMix2RowThreads)
k_mix2_x_fwd(XIn<T> a, int nrows, int nvalid, typename Cplx<T>::type *__restrict__ out, int64_t out_rs,
             const typename Cplx<T>::type *__restrict__ twx, const Mix2 g, unsigned mh)
{
    using C = typename Cplx<T>::type;
    extern __shared__ __align__(16) unsigned char smraw[];
    C *ex = reinterpret_cast<C *>(smraw);
    const int L = g.L, R1 = g.R1, R2 = g.R2, RP = g.RP, TR = g.G;
    const int RS = R2 * RP;  // exchange row (>= L)
    const int row0 = blockIdx.x * TR;
    // rows of whole pairs on pair boundaries: one vector load per pair
    const bool pairs = (a.in_rs & 1) == 0 && (nvalid & 1) == 0 && ((uintptr_t)a.in & (sizeof(C) - 1)) == 0;
    const int rr1 = udiv(threadIdx.x, R2, g.m2), j1 = threadIdx.x - rr1 * R2;
    const bool act1 = rr1 < TR;
    mx::with_radix<MAXR>(R1, [&](auto rc) {
        constexpr int R = decltype(rc)::value, H = (R + 1) / 2;
        if (!act1) return;
        const int row = row0 + rr1;
        // the loads of all inputs first (independent, predicated), then the scaling
        C u[R];
        const T *p = a.in + (int64_t)row * a.in_rs;
        const int left = row < nrows ? nvalid : 0;
        if (pairs) {
#pragma unroll
            for (int r = 0; r < H; ++r) {
                const int x0 = 2 * (j1 + r * R2);
                u[r] = cmk<C>(0, 0);
                if (x0 < left) u[r] = *reinterpret_cast<const C *>(p + x0);
            }
        } else {
#pragma unroll
            for (int r = 0; r < H; ++r) {
                const int x0 = 2 * (j1 + r * R2);
                u[r] = cmk<C>(0, 0);
                if (x0 < left) u[r].x = p[x0];
                if (x0 + 1 < left) u[r].y = p[x0 + 1];
            }
        }
        if (a.wcell) {
            const T *w = a.wcell + (int64_t)(row % a.rows_per_comp) * a.in_rs;
#pragma unroll
            for (int r = 0; r < H; ++r) {
                const int x0 = 2 * (j1 + r * R2);
                T w0 = 0, w1 = 0;
                if (x0 < left) w0 = __ldg(&w[x0]);
                if (x0 + 1 < left) w1 = __ldg(&w[x0 + 1]);
                u[r].x *= a.wscalar * w0;
                u[r].y *= a.wscalar * w1;
            }
        } else {
#pragma unroll
            for (int r = 0; r < H; ++r) u[r] = mx::cscale(a.wscalar, u[r]);
        }
        mx::DFT<R, H, false, C>::run(u);
        C *s = ex + rr1 * RS + j1 * RP;
#pragma unroll
        for (int r = 0; r < R; ++r) s[r] = u[r];
    });
    __syncthreads();
    const int rr2 = udiv(threadIdx.x, R1, g.m1), j2 = threadIdx.x - rr2 * R1;
    const bool act2 = rr2 < TR;
    mx::with_radix<MAXR>(R2, [&](auto rc) {
        constexpr int R = decltype(rc)::value;
        C v[R];
        if (act2) {
            const C *s = ex + rr2 * RS + j2;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                v[r] = *s;
                s += RP;
            }
            mx::twiddle<R, false>(v, 2 * j2, twx);
            mx::DFT<R, R, false, C>::run(v);
        }
        __syncthreads();  // every exchange value is read before any is replaced
        if (act2) {
            C *s = ex + rr2 * RS + j2;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                *s = v[r];
                s += R1;
            }
        }
    });
    __syncthreads();
    const T h = (T)0.5;
    const int HP = L / 2 + 1;  // pairs k = 0 .. L / 2 per row
    for (int e = threadIdx.x; e < HP * TR; e += blockDim.x) {
        const int rr = udiv(e, HP, mh), k = e - rr * HP, row = row0 + rr;
        if (row >= nrows) break;
        const C p = ex[rr * RS + k], q = ex[rr * RS + (k == 0 ? 0 : L - k)];
        const C E = cmk<C>(h * (p.x + q.x), h * (p.y - q.y));
        const C O = cmk<C>(h * (p.y + q.y), -h * (p.x - q.x));
        const C wo = cmul(O, __ldg(&twx[k]));
        C *o = out + (int64_t)row * out_rs;
        o[k] = cadd(E, wo);
        if (2 * k != L) o[L - k] = cmk<C>(E.x - wo.x, wo.y - E.y);
    }
}

// Complex-to-real rows (as k_gen_x_inv): g.G rows per CTA, one butterfly per
// thread and stage; the first stage forms the packed spectrum from X[k] and
// X[L - k], the last forms the outputs n <= L / 2 and applies the XOut epilogue.
template <typename T, int MAXR>
__global__ void __launch_bounds__(kMix2RowThreads, (sizeof(T) == 4 ? (MAXR <= 16 ? 3 : 2) : 1) * 256 / kMix2RowThreads)
k_mix2_x_inv(const typename Cplx<T>::type *__restrict__ in, int64_t in_rs, int nrows, int nvalid, XOut<T> o,
             const typename Cplx<T>::type *__restrict__ twx, const Mix2 g)
{
    using C = typename Cplx<T>::type;
    extern __shared__ __align__(16) unsigned char smraw[];
    C *ex = reinterpret_cast<C *>(smraw);
    const int L = g.L, R1 = g.R1, R2 = g.R2, RP = g.RP, TR = g.G;
    const int RS = R2 * RP;
    const int row0 = blockIdx.x * TR;
    const int rr1 = udiv(threadIdx.x, R2, g.m2), j1 = threadIdx.x - rr1 * R2;
    mx::with_radix<MAXR>(R1, [&](auto rc) {
        constexpr int R = decltype(rc)::value;
        if (rr1 >= TR) return;
        const int row = row0 + rr1;
        C u[R];
        if (row < nrows) {
            const C *p = in + (int64_t)row * in_rs;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int k = j1 + r * R2;
                const C x = p[k], y = p[L - k];
                const C E2 = cmk<C>(x.x + y.x, x.y - y.y);
                const C D = cmk<C>(x.x - y.x, x.y + y.y);
                const C O2 = cmulc(D, __ldg(&twx[k]));
                u[r] = cmk<C>(E2.x - O2.y, E2.y + O2.x);
            }
        } else {
#pragma unroll
            for (int r = 0; r < R; ++r) u[r] = cmk<C>(0, 0);
        }
        mx::DFT<R, R, true, C>::run(u);
        C *s = ex + rr1 * RS + j1 * RP;
#pragma unroll
        for (int r = 0; r < R; ++r) s[r] = u[r];
    });
    __syncthreads();
    const int rr2 = udiv(threadIdx.x, R1, g.m1), j2 = threadIdx.x - rr2 * R1;
    const T oscale = o.oscale * (o.gdev ? (T)(*o.gdev) : (T)1);
    T acc = 0;
    mx::with_radix<MAXR>(R2, [&](auto rc) {
        constexpr int R = decltype(rc)::value, H = R / 2 + 1;
        const int row = row0 + rr2;
        if (rr2 >= TR || row >= nrows) return;
        const int64_t ro = (int64_t)row * o.out_rs;
        // rows of whole pairs on pair boundaries: vector stores and loads
        const bool pairs = (o.out_rs & 1) == 0 && (nvalid & 1) == 0 && ((uintptr_t)o.out & (sizeof(C) - 1)) == 0 &&
                           ((uintptr_t)o.Mref & (sizeof(C) - 1)) == 0;
        C m[H];  // the energy's M, loaded ahead of the transform
        if (o.partials) {
            const T *mp = o.Mref + ro;
#pragma unroll
            for (int r = 0; r < H; ++r) {
                const int x0 = 2 * (j2 + r * R1);
                m[r] = cmk<C>(0, 0);
                if (pairs) {
                    if (x0 < nvalid) m[r] = *reinterpret_cast<const C *>(mp + x0);
                } else {
                    if (x0 < nvalid) m[r].x = mp[x0];
                    if (x0 + 1 < nvalid) m[r].y = mp[x0 + 1];
                }
            }
        }
        C v[R];
        const C *s = ex + rr2 * RS + j2;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            v[r] = *s;
            s += RP;
        }
        mx::twiddle<R, true>(v, 2 * j2, twx);
        mx::DFT<R, R, true, C>::run(v);
#pragma unroll
        for (int r = 0; r < H; ++r) v[r] = mx::cscale(o.scale, v[r]);
        if (o.wcell) {
            const T *wc = o.wcell + (int64_t)(row % o.rows_per_comp) * o.out_rs;
#pragma unroll
            for (int r = 0; r < H; ++r) {
                const int x0 = 2 * (j2 + r * R1);
                T w0 = 0, w1 = 0;
                if (x0 < nvalid) w0 = __ldg(&wc[x0]);
                if (x0 + 1 < nvalid) w1 = __ldg(&wc[x0 + 1]);
                if (o.partials) acc += o.mscale * (w0 * m[r].x * v[r].x + w1 * m[r].y * v[r].y);
                v[r] = cmk<C>(v[r].x * oscale * w0, v[r].y * oscale * w1);
            }
        } else {
#pragma unroll
            for (int r = 0; r < H; ++r) {
                // m is zero where x >= nvalid
                if (o.partials) acc += o.mscale * (m[r].x * v[r].x + m[r].y * v[r].y);
                v[r] = mx::cscale(oscale, v[r]);
            }
        }
        if (!o.out) return;
        T *op = o.out + ro;
#pragma unroll
        for (int r = 0; r < H; ++r) {
            const int x0 = 2 * (j2 + r * R1);
            if (pairs) {
                if (x0 < nvalid) *reinterpret_cast<C *>(op + x0) = v[r];
            } else {
                if (x0 < nvalid) op[x0] = v[r].x;
                if (x0 + 1 < nvalid) op[x0 + 1] = v[r].y;
            }
        }
    });
    if (o.partials) block_partial<kMix2RowThreads>((double)acc, o.partials, blockIdx.x);
}

// Fused z pass (as k_gen_zconv) for L = R1 R2, R2 <= MAXR2: one CTA per TC columns
// kx of one ky row, R1 TC threads. Stage 1: R1-point DFTs of the half-empty
// input rows j + r R2 of the three components into the exchange rows j RP + m.
// Middle, one thread per (m, column): the three components' R2-point DFTs
// in registers, the product at kz = m + R1 q, the inverse DFTs and both
// twiddles, in place. Stage 3: R1-point inverse DFTs, rows z < nrows stored. The middle
// holds three components, so R2 is the smaller radix (130^3 -> 270^3, 30 x 9: 137 us at
// two CTAs per SM, 51% of the issue slots; DRAM floor 43 us). FP32: the tile's tensor block (two
// 4-column sub-blocks of the tile-ordered copy) is copied to shared memory with
// 16-byte asynchronous copies while stage 1 runs; FP64 reads the octant table.
template <typename T, int TC, int MAXR2>
__global__ void __launch_bounds__(32 * TC, sizeof(T) == 4 && MAXR2 <= 10 ? 2 : 1)
k_mix2_z(typename Cplx<T>::type *__restrict__ S, int Kx, int Py, int64_t ss, int64_t rs, int64_t cs, int nrows,
         const T *__restrict__ nhat, const T *__restrict__ ntile, const typename Cplx<T>::type *__restrict__ tw, int ntx,
         const Mix2 g)
{
    using C = typename Cplx<T>::type;
    constexpr bool TILE = sizeof(T) == 4;
    extern __shared__ __align__(16) unsigned char smraw[];
    C *ex = reinterpret_cast<C *>(smraw);
    const int L = g.L, R1 = g.R1, R2 = g.R2, RP = g.RP, HZ = L / 2 + 1;
    const int EXS = R2 * RP * TC;  // one component
    T *tz = reinterpret_cast<T *>(ex + 3 * EXS);
    const int TZB = 24 * HZ, TZS = mix2_tensor_stride(HZ);
    const int kyi = blockIdx.x / ntx, kx0 = (blockIdx.x - kyi * ntx) * TC;
    const int ky = ky_pair_order(kyi, Py), kyf = ky > Py / 2 ? Py - ky : ky;
    const int tid = threadIdx.x, c = tid % TC, j0 = tid / TC;
    const bool ok = kx0 + c < Kx;
    if constexpr (TILE) {
        const T *src = ntile + ((size_t)kyf * ((Kx + 7) / 8 * 2) + kx0 / 4) * TZB;
#pragma unroll
        for (int h = 0; h < TC / 4; ++h)
            for (int i = tid * 4; i < TZB; i += (int)blockDim.x * 4) cp_async16(tz + h * TZS + i, src + h * TZB + i);
    }
    C *col = S + (int64_t)ky * ss + kx0 + c;
    // R1 groups of threads over the 3 R2 butterflies
    mx::with_radix<32>(R1, [&](auto rc) {
        constexpr int R = decltype(rc)::value, H = (R + 1) / 2;
        const int64_t step = R2 * rs;
        for (int b = j0; b < 3 * R2; b += R) {
            const int comp = b >= 2 * R2 ? 2 : (b >= R2 ? 1 : 0), j = b - comp * R2;
            C u[R];
            const C *p = col + comp * cs + j * rs;
            int row = j;
#pragma unroll
            for (int r = 0; r < H; ++r) {
                u[r] = cmk<C>(0, 0);
                if (ok && row < nrows) u[r] = *p;
                p += step;
                row += R2;
            }
            mx::DFT<R, H, false, C>::run(u);
            C *s = ex + comp * EXS + j * RP * TC + c;
#pragma unroll
            for (int r = 0; r < R; ++r) s[r * TC] = u[r];
        }
    });
    cp_async_wait_all();
    __syncthreads();
    mx::with_radix<MAXR2>(R2, [&](auto rc) {
        constexpr int R = decltype(rc)::value;
        const int step = RP * TC;
        C v0[R], v1[R], v2[R];
        C *s = ex + j0 * TC + c;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            v0[r] = s[r * step];
            v1[r] = s[r * step + EXS];
            v2[r] = s[r * step + 2 * EXS];
        }
#pragma unroll
        for (int r = 1; r < R; ++r) {
            const C w = __ldg(&tw[r * j0]);
            v0[r] = cmul(v0[r], w);
            v1[r] = cmul(v1[r], w);
            v2[r] = cmul(v2[r], w);
        }
        mx::DFT<R, R, false, C>::run(v0);
        mx::DFT<R, R, false, C>::run(v1);
        mx::DFT<R, R, false, C>::run(v2);
        const T sy = ky > Py / 2 ? (T)-1 : (T)1;
#pragma unroll
        for (int q = 0; q < R; ++q) {
            const int kz = j0 + R1 * q;
            const bool fz = 2 * kz > L;
            const int kzf = fz ? L - kz : kz;
            const T sz = fz ? (T)-1 : (T)1;
            T n[6];
            if constexpr (TILE) {
                const T *t = tz + (c >> 2) * TZS + kzf * 4 + (c & 3);
#pragma unroll
                for (int i = 0; i < 6; ++i) n[i] = t[i * HZ * 4];
            } else {
                const int hy = Py / 2 + 1;
                const T *t = nhat + ((int64_t)kzf * hy + kyf) * Kx + (ok ? kx0 + c : 0);
#pragma unroll
                for (int i = 0; i < 6; ++i) n[i] = __ldg(&t[(int64_t)i * HZ * hy * Kx]);
            }
            const T xy = sy * n[3], xz = sz * n[4], yz = sy * sz * n[5];
            const C mx_ = v0[q], my_ = v1[q], mz_ = v2[q];
            v0[q] = mx::cfma(-xz, mz_, mx::cfma(-xy, my_, mx::cscale(-n[0], mx_)));
            v1[q] = mx::cfma(-yz, mz_, mx::cfma(-n[1], my_, mx::cscale(-xy, mx_)));
            v2[q] = mx::cfma(-n[2], mz_, mx::cfma(-yz, my_, mx::cscale(-xz, mx_)));
        }
        mx::DFT<R, R, true, C>::run(v0);
        mx::DFT<R, R, true, C>::run(v1);
        mx::DFT<R, R, true, C>::run(v2);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const C w = __ldg(&tw[r * j0]);
            s[r * step] = r ? cmulc(v0[r], w) : v0[r];
            s[r * step + EXS] = r ? cmulc(v1[r], w) : v1[r];
            s[r * step + 2 * EXS] = r ? cmulc(v2[r], w) : v2[r];
        }
    });
    __syncthreads();
    mx::with_radix<32>(R1, [&](auto rc) {
        constexpr int R = decltype(rc)::value, H = R / 2 + 1;
        const int64_t step = R2 * rs;
        for (int b = j0; b < 3 * R2; b += R) {
            const int comp = b >= 2 * R2 ? 2 : (b >= R2 ? 1 : 0), n1 = b - comp * R2;
            C u[R];
            const C *s = ex + comp * EXS + n1 * RP * TC + c;
#pragma unroll
            for (int r = 0; r < R; ++r) u[r] = s[r * TC];
            mx::DFT<R, R, true, C>::run(u);
            C *p = col + comp * cs + n1 * rs;
            int row = n1;
#pragma unroll
            for (int r = 0; r < (H < R ? H : R); ++r) {
                if (ok && row < nrows) *p = u[r];
                p += step;
                row += R2;
            }
        }
    });
}

}  // namespace demag

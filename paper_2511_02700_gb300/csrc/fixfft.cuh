// FP64 transforms in 64-bit block fixed point.
//
// GB300 issues two FP64 lanes per SM and clock: a warp's FP64 instruction occupies
// the SM for 16 clocks, an integer one the issue slot of one of four schedulers.  A
// length-P transform therefore runs on 64-bit integers with one exponent for the
// whole transform: doubles are quantised in the first stage (to 2^-58 of the largest
// magnitude with radix 8), every stage adds, subtracts and rotates integers, and the
// last stage writes doubles.  Between stages the integers are shifted so that their
// largest uses the word (block floating point), which keeps each stage's rounding
// at 2^-58 of its largest value; an FP64 butterfly rounds every value at 2^-53 of
// itself.  Against long double, over noise, payoff-like, decaying and peaked sequences of
// 128 to 8192 values, the error is half that of a radix-2 FP64 transform (equal for a
// single spike at 8192).  A spectrum column keeps its entries to 2^-61 of its largest and the
// product its values to 2^-62 of the two maxima's, below the transforms' own errors: jump
// sums with spectra that fall by 1e-8 within a column, or peak where the field's do not, are
// off by 0.04 to 0.51 of what they were with FP64 butterflies (N = 64 to 256, against 128 bits).
// Subnormal values count as zero, so fields below about 1e-288 lose digits.
//
// Measured, one fixed-point iteration of a solve with FP64 transforms against these:
// N = 256 75 -> 56 us, N = 512 213 -> 113 us, N = 1024 755 -> 339 us (column pass 297 -> 90,
// and 82 us with nothing converted between its transforms).  What bounds them now: latency
// (barriers, shared memory, twiddle loads) and integer issue.  Tried and slower: twiddles
// loaded before a stage's barrier (N = 1024 326 -> 335 us), the spectrum column fetched before
// the last barrier (330).  Units smaller than a warp (P < 128) keep FP64 butterflies.
//
//   q in [-2^B, 2^B] at the input of a radix-R butterfly, B = 61 - log2 R: a complex
//   value then stays below 2^61.5 through the butterfly (|z| grows by R at most).
//   Products with a twiddle (Q62) use 32-bit halves, v = h 2^32 + l and w = wh 2^32 + wl
//   with signed l, wl: v w / 2^62 = 4 h wh + (h wl + l wh) / 2^30, dropping l wl / 2^62
//   (at most one unit); every partial sum of a complex product stays below 2^63.
//
// A non-finite input makes every output NaN.
#pragma once

#include "common.cuh"

namespace pide {

using fx2 = longlong2;

// v = h 2^32 + l with l a signed 32-bit value
struct FxHalf {
    int h, l;
};
__host__ __device__ __forceinline__ FxHalf fx_split(long long v) {
    const int l = (int)(unsigned)(unsigned long long)v;
    return FxHalf{(int)(v >> 32) - (l >> 31), l};
}

// v c / 2^62 for a Q62 constant
__host__ __device__ __forceinline__ long long fx_mulc(FxHalf v, FxHalf c) {
    const long long hh = (long long)v.h * c.h;
    const long long cr = (long long)v.h * c.l + (long long)v.l * c.h + (1LL << 29);
    return hh * 4 + (cr >> 30);
}

// v times w (CONJ = false) or its conjugate; w = (re h, re l, im h, im l) in Q62
template <bool CONJ>
__host__ __device__ __forceinline__ fx2 fx_cmul(fx2 v, int4 w) {
    const FxHalf x = fx_split(v.x), y = fx_split(v.y);
    const long long xr_hh = (long long)x.h * w.x, xr_cr = (long long)x.h * w.y + (long long)x.l * w.x + (1LL << 29);
    const long long yi_hh = (long long)y.h * w.z, yi_cr = (long long)y.h * w.w + (long long)y.l * w.z;
    const long long yr_hh = (long long)y.h * w.x, yr_cr = (long long)y.h * w.y + (long long)y.l * w.x + (1LL << 29);
    const long long xi_hh = (long long)x.h * w.z, xi_cr = (long long)x.h * w.w + (long long)x.l * w.z;
    fx2 o;
    if (CONJ) {
        o.x = (xr_hh + yi_hh) * 4 + ((xr_cr + yi_cr) >> 30);
        o.y = (yr_hh - xi_hh) * 4 + ((yr_cr - xi_cr) >> 30);
    } else {
        o.x = (xr_hh - yi_hh) * 4 + ((xr_cr - yi_cr) >> 30);
        o.y = (yr_hh + xi_hh) * 4 + ((yr_cr + xi_cr) >> 30);
    }
    return o;
}

// a b / 2^62 rounded, for Q62 values
__host__ __device__ __forceinline__ long long fx_mul62(long long a, long long b) {
#ifdef __CUDA_ARCH__
    const long long hi = __mul64hi(a, b);
#else
    const long long hi = (long long)(((__int128)a * b) >> 64);
#endif
    const unsigned long long lo = (unsigned long long)a * (unsigned long long)b;
    return (long long)(((unsigned long long)hi << 2) + (lo >> 62) + ((lo >> 61) & 1));
}
// e^{-2 pi i k / P} in Q62: the product over the bits of k of e^{-2 pi i / 2^m}, whose sines
// and cosines are given to the last bit; each product rounds at 2^-62, so the result is within
// 2^-58, where a twiddle rounded to double is within 2^-54 and would dominate the transform's
// error (N = 64 jump sum against 64-bit arithmetic 2.8e-16 -> 2.6e-16, N = 256 2.7e-16 -> 2.3e-16)
__host__ __device__ inline fx2 fx_twiddle(int k, int P) {
    const long long cs[14][2] = {{4611686018427387904, 0}, {-4611686018427387904, 0}, {0, 4611686018427387904},
                                 {3260954456333195553, 3260954456333195553}, {4260642322793532497, 1764815834521887442},
                                 {4523073764714963030, 899695310372275547}, {4589479489746651964, 452024275624069880},
                                 {4606131040650197959, 226284707652502141}, {4610297064819661174, 113176440454146016},
                                 {4611338766951757487, 56592481536850979}, {4611599204741358747, 28296773447188932},
                                 {4611664314954810277, 14148453308909941}, {4611680592556051597, 7074234977634094},
                                 {4611684661959354334, 3537118529214896}};
    fx2 w{cs[0][0], 0};
    int m = 0;
    while ((1 << m) < P) ++m;
    for (; k; k >>= 1, --m)
        if (k & 1) {
            const long long c = cs[m][0], s = -cs[m][1];
            w = fx2{fx_mul62(w.x, c) - fx_mul62(w.y, s), fx_mul62(w.x, s) + fx_mul62(w.y, c)};
        }
    return w;
}

// v e^{DIR 2 pi i m / 16} for a compile-time m
template <int DIR, int M>
__host__ __device__ __forceinline__ fx2 fx_w16(fx2 v) {
    constexpr int m = M & 15;
    // cos(2 pi k/16) in Q62
    constexpr long long c16[4] = {4611686018427387904, 4260642322793532497, 3260954456333195553, 1764815834521887442};
    if constexpr (m == 0) {
        return v;
    } else if constexpr (m == 8) {
        return fx2{-v.x, -v.y};
    } else if constexpr (m == 4 || m == 12) {            // times +-i
        if constexpr ((m == 4) == (DIR > 0)) return fx2{-v.y, v.x};
        else return fx2{v.y, -v.x};
    } else if constexpr (m > 8) {
        const fx2 u = fx_w16<DIR, M - 8>(v);
        return fx2{-u.x, -u.y};
    } else if constexpr (m > 4) {
        return fx_w16<DIR, 4>(fx_w16<DIR, M - 4>(v));
    } else if constexpr (m == 2) {                       // (1 + DIR i) / sqrt 2
        const FxHalf c = fx_split(c16[2]);
        const long long s = v.x + v.y, d = v.x - v.y;
        if constexpr (DIR > 0) return fx2{fx_mulc(fx_split(d), c), fx_mulc(fx_split(s), c)};
        else return fx2{fx_mulc(fx_split(s), c), fx_mulc(fx_split(-d), c)};
    } else {
        const FxHalf c = fx_split(c16[m]), s = fx_split(c16[4 - m]);
        return fx_cmul<(DIR < 0)>(v, int4{c.h, c.l, s.h, s.l});
    }
}

// X[k] = sum_n v[n] e^{DIR 2 pi i n k / RAD} in natural order, as dft_small
template <int DIR, int RAD, int LEN, int I, int K>
__host__ __device__ __forceinline__ void fx_bfly(fx2* v) {
    if constexpr (I < RAD) {
        if constexpr (K < LEN / 2) {
            const fx2 a = v[I + K], b = fx_w16<DIR, K*(16 / LEN)>(v[I + K + LEN / 2]);
            v[I + K] = fx2{a.x + b.x, a.y + b.y};
            v[I + K + LEN / 2] = fx2{a.x - b.x, a.y - b.y};
            fx_bfly<DIR, RAD, LEN, I, K + 1>(v);
        } else {
            fx_bfly<DIR, RAD, LEN, I + LEN, 0>(v);
        }
    }
}
template <int DIR, int RAD, int LEN>
__host__ __device__ __forceinline__ void fx_layers(fx2* v) {
    if constexpr (LEN <= RAD) {
        fx_bfly<DIR, RAD, LEN, 0, 0>(v);
        fx_layers<DIR, RAD, LEN * 2>(v);
    }
}
template <int RAD, int I>
__host__ __device__ __forceinline__ void fx_bitrev(fx2* v) {
    if constexpr (I < RAD) {
        constexpr int J = brev_t<I, log2_t<RAD>::value>::value;
        if constexpr (J > I) {
            const fx2 t = v[I];
            v[I] = v[J];
            v[J] = t;
        }
        fx_bitrev<RAD, I + 1>(v);
    }
}
template <int DIR, int RAD>
__host__ __device__ __forceinline__ void fx_dft(fx2* v) {
    fx_bitrev<RAD, 0>(v);
    fx_layers<DIR, RAD, 2>(v);
}

__host__ __device__ constexpr int fx_bits(int rad) { return rad == 16 ? 57 : (rad == 8 ? 58 : (rad == 4 ? 59 : 60)); }

// round(d 2^k) for |d| 2^k < 2^61 (integer instructions only; magnitudes below the normal
// range count as zero)
__host__ __device__ __forceinline__ long long fx_quantise(unsigned hi, unsigned lo, int k) {
    const int e = (int)((hi >> 20) & 0x7ffu);
    const unsigned long long m = ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 41) | ((unsigned long long)lo << 9);
    int r = 1084 - e - k;                                 // m 2^-r is the value (m < 2^62)
    r = r > 63 ? 63 : r;
    const unsigned long long q = e ? ((m >> (r - 1)) + 1) >> 1 : 0;
    const long long s = (long long)((int)hi >> 31);
    return (long long)(q ^ (unsigned long long)s) - s;
}

// q 2^e as a double, rounded to nearest (ties away), |q| < 2^63; magnitudes outside the
// normal range become 0 or infinity
__host__ __device__ __forceinline__ unsigned long long fx_double_bits(long long q, int e) {
    const unsigned long long s = (unsigned long long)(q >> 63);
    const unsigned long long a = ((unsigned long long)q ^ s) - s;
#ifdef __CUDA_ARCH__
    const int lz = __clzll((long long)a);
#else
    const int lz = a ? __builtin_clzll(a) : 64;
#endif
    const int ex = e + 1085 - lz;                         // biased exponent - 1 of the leading bit, at 2^(63 - lz)
    unsigned long long m = a << (lz & 63);
    m = (m >> 11) + ((m >> 10) & 1);                      // 53 bits, leading one included (it adds 1 to the exponent)
    unsigned long long b = m + ((unsigned long long)(unsigned)ex << 52);
    if (a == 0 || ex < 0) b = 0;
    if (ex >= 2046) b = 0x7ff0000000000000ull;
    return b | (s << 63);
}

#ifdef __CUDACC__
// values of a unit's warps: the largest exponent word of the input (slots 0..15), the
// OR of the sign-folded high words of a stage's output (slots 16..31)
__device__ __forceinline__ unsigned* fx_slots(double2* buf, int P) {
    return reinterpret_cast<unsigned*>(buf + padded_len(P) + 4);
}

template <int P, int RAD, int NS, class F>
__device__ __forceinline__ void fx_store_smem(fx2* buf, int base, const fx2* v, const F& note) {
    if constexpr (NS % 16 == 0 || (NS == 1 && (RAD == 16 || RAD == 8))) {
        const int pb = padi(base);
#pragma unroll
        for (int r = 0; r < RAD; ++r) {
            note(v[r]);
            buf[pb + r * (NS + NS / 16)] = v[r];
        }
    } else {
#pragma unroll
        for (int r = 0; r < RAD; ++r) {
            note(v[r]);
            buf[padi(base + r * NS)] = v[r];
        }
    }
}

// A column of a weight spectrum as the column passes multiply with it: entry k2 holds the
// halves of w q, w = q 2^(e - 62) with |q| < 2^61 and one exponent e for the column; the low
// bits of the first 16 real parts hold e + 2^15 (0xffff: the column is not finite); the low bit
// of every real part is dropped in the product, so a scaled column gives the scaled product.
__device__ __forceinline__ int fx_spectrum_code(const int4* w, bool valid) {
    return valid ? (int)(__ballot_sync(0xffffffffu, w[threadIdx.x & 15].y & 1) & 0xffffu) : 1 << 15;
}
__device__ __forceinline__ int4 fx_spectrum_entry(double2 w, int k, int k2, int code) {
    long long re = fx_quantise((unsigned)__double2hiint(w.x), (unsigned)__double2loint(w.x), k);
    const long long im = fx_quantise((unsigned)__double2hiint(w.y), (unsigned)__double2loint(w.y), k);
    if (k2 < 16) re = (re & ~1LL) | ((code >> k2) & 1);
    const FxHalf r = fx_split(re), i = fx_split(im);
    return make_int4(r.h, r.l, i.h, i.l);
}
// Storer of a forward transform that goes on, still in integers, as the inverse transform of
// its product with a spectrum column, whose outputs `next` takes
template <class S2> struct FxThen {
    const int4* w;
    int code;
    bool valid;
    const S2& next;
    static constexpr bool fx_then = true;
};
template <class T, class = void> struct is_fx_then { static constexpr bool value = false; };
template <class T> struct is_fx_then<T, decltype((void)T::fx_then, void())> { static constexpr bool value = true; };

// the stages with span NS, NS V, ...: integers in buf, exponent E (value = q 2^E)
template <int DIR, int P, int NS, class S>
__device__ __forceinline__ void fx_rest(fx2* buf, unsigned* red, int t, const int4* __restrict__ twi, int E, bool bad,
                                        const S& store) {
    constexpr int V = fft_values<double>(P), NT = P / V, NW = NT / 32;
    constexpr int RAD = (NS * V <= P) ? V : P / NS;
    constexpr int NB = V / RAD, STRIDE = P / RAD, TWS = P / (NS * RAD);
    constexpr bool LAST = NS * RAD == P;
    unsigned any = 0;
#pragma unroll
    for (int u = 0; u < NW; ++u) any |= red[16 + u];
    const int s = (any ? 64 - __clz(any) : 32) - fx_bits(RAD);
    E += s;
    fx2 v[V];
#pragma unroll
    for (int b = 0; b < NB; ++b) {
        const int j = t + b * NT;
        if constexpr (STRIDE % 16 == 0) {
            const int pj = padi(j);
#pragma unroll
            for (int r = 0; r < RAD; ++r) v[b * RAD + r] = buf[pj + r * (STRIDE + STRIDE / 16)];
        } else {
#pragma unroll
            for (int r = 0; r < RAD; ++r) v[b * RAD + r] = buf[padi(j + r * STRIDE)];
        }
    }
    if (s > 0) {
        const long long half = 1LL << (s - 1);
#pragma unroll
        for (int i = 0; i < V; ++i) v[i] = fx2{(v[i].x + half) >> s, (v[i].y + half) >> s};
    } else {
#pragma unroll
        for (int i = 0; i < V; ++i)
            v[i] = fx2{(long long)((unsigned long long)v[i].x << -s), (long long)((unsigned long long)v[i].y << -s)};
    }
#pragma unroll
    for (int b = 0; b < NB; ++b) {
        const int k = (t + b * NT) & (NS - 1);
        if constexpr (NS > 1) {
#pragma unroll
            for (int r = 1; r < RAD; ++r) v[b * RAD + r] = fx_cmul<(DIR > 0)>(v[b * RAD + r], __ldg(&twi[k * (r * TWS)]));
        }
        fx_dft<DIR, RAD>(&v[b * RAD]);
    }
    __syncthreads();
    if constexpr (LAST && is_fx_then<S>::value) {
        unsigned o = 0;
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            const int j = t + b * NT;
            const int k = j & (NS - 1);
            const int base = (j - k) * RAD + k;
#pragma unroll
            for (int r = 0; r < RAD; ++r) {
                const int k2 = base + r * NS;
                int4 w = store.valid ? __ldg(&store.w[k2]) : make_int4(0, 0, 0, 0);
                w.y &= ~1;                            // (fx_spectrum_code)
                const fx2 q = fx_cmul<false>(v[b * RAD + r], w);
                const int hx = (int)(q.x >> 32), hy = (int)(q.y >> 32);
                o |= (unsigned)(hx ^ (hx >> 31)) | (unsigned)(hy ^ (hy >> 31));
                buf[padi(k2)] = q;
            }
        }
        o = __reduce_or_sync(0xffffffffu, o);
        if ((t & 31) == 0) red[16 + (t >> 5)] = o;
        __syncthreads();
        fx_rest<-DIR, P, 1>(buf, red, t, twi, E + store.code - (1 << 15), bad || store.code == 0xffff, store.next);
    } else if constexpr (LAST) {
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            const int j = t + b * NT;
            const int k = j & (NS - 1);
            const int base = (j - k) * RAD + k;
            auto val = [&](int r) {
                const double x = __longlong_as_double((long long)fx_double_bits(v[b * RAD + r].x, E));
                const double y = __longlong_as_double((long long)fx_double_bits(v[b * RAD + r].y, E));
                const double nan = __longlong_as_double(0x7ff8000000000000LL);
                return bad ? make_double2(nan, nan) : make_double2(x, y);
            };
            if constexpr (is_smem_io<S>::value && NS % 16 == 0) {
                const int pb = padi(base);
#pragma unroll
                for (int r = 0; r < RAD; ++r) store.at(pb, r * (NS + NS / 16), val(r));
            } else {
#pragma unroll
                for (int r = 0; r < RAD; ++r) store(base + r * NS, val(r));
            }
        }
        __syncthreads();
    } else {
        unsigned o = 0;
        auto note = [&](fx2 q) {
            const int hx = (int)(q.x >> 32), hy = (int)(q.y >> 32);
            o |= (unsigned)(hx ^ (hx >> 31)) | (unsigned)(hy ^ (hy >> 31));
        };
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            const int j = t + b * NT;
            const int k = j & (NS - 1);
            fx_store_smem<P, RAD, NS>(buf, (j - k) * RAD + k, &v[b * RAD], note);
        }
        o = __reduce_or_sync(0xffffffffu, o);
        if ((t & 31) == 0) red[16 + (t >> 5)] = o;
        __syncthreads();
        fx_rest<DIR, P, NS * RAD>(buf, red, t, twi, E, bad, store);
    }
}

// lengths whose units are whole warps
__host__ __device__ constexpr bool fx_length(int P) { return P / fft_values<double>(P) >= 32; }

// the first stage of values v in registers (value = v 2^E), and the rest
template <int DIR, int P, class S>
__device__ __forceinline__ void fx_first(fx2* buf, unsigned* red, int t, const int4* __restrict__ twi, fx2* v, int E, bool bad,
                                         const S& store) {
    constexpr int V = fft_values<double>(P);
    fx_dft<DIR, V>(v);
    unsigned o = 0;
    auto note = [&](fx2 q) {
        const int hx = (int)(q.x >> 32), hy = (int)(q.y >> 32);
        o |= (unsigned)(hx ^ (hx >> 31)) | (unsigned)(hy ^ (hy >> 31));
    };
    fx_store_smem<P, V, 1>(buf, t * V, v, note);
    o = __reduce_or_sync(0xffffffffu, o);
    if ((t & 31) == 0) red[16 + (t >> 5)] = o;
    __syncthreads();
    fx_rest<DIR, P, V>(buf, red, t, twi, E, bad, store);
}

// block_fft in block fixed point (same contract)
template <int DIR, int P, class L, class S>
__device__ __forceinline__ void fx_fft(double2* bufd, int t, const double2* __restrict__ tw, const L& load, const S& store) {
    constexpr int V = fft_values<double>(P), NT = P / V, NW = NT / 32;
    static_assert(NT % 32 == 0 && NW <= 16, "whole warps");
    fx2* buf = reinterpret_cast<fx2*>(bufd);
    unsigned* red = fx_slots(bufd, P);
    const int4* twi = reinterpret_cast<const int4*>(tw + P);
    fx2 v[V];
    unsigned big = 0;
    constexpr unsigned ZM = zero_mask_of<L>::value;
    {
        const int pj = padi(t);
#pragma unroll
        for (int r = 0; r < V; ++r) {
            double2 d = make_double2(0.0, 0.0);
            if (!((ZM >> r) & 1u)) {
                if constexpr (is_smem_io<L>::value && NT % 16 == 0) d = load.at(pj, r * (NT + NT / 16));
                else d = load(t + r * NT);
            }
            v[r] = fx2{__double_as_longlong(d.x), __double_as_longlong(d.y)};
            big = max(big, max((unsigned)(v[r].x >> 32) & 0x7fffffffu, (unsigned)(v[r].y >> 32) & 0x7fffffffu));
        }
    }
    big = __reduce_max_sync(0xffffffffu, big);
    if ((t & 31) == 0) red[t >> 5] = big;
    __syncthreads();                          // also: every input of the stage is read before any store
#pragma unroll
    for (int u = 0; u < NW; ++u) big = max(big, red[u]);
    const bool bad = big >= 0x7ff00000u;
    // every |d| < 2^(exponent + 1)
    const int k = fx_bits(V) - ((int)(big >> 20) - 1022);
#pragma unroll
    for (int r = 0; r < V; ++r)
        if (!((ZM >> r) & 1u))
            v[r] = fx2{fx_quantise((unsigned)(v[r].x >> 32), (unsigned)v[r].x, k),
                       fx_quantise((unsigned)(v[r].y >> 32), (unsigned)v[r].y, k)};
    fx_first<DIR, P>(buf, red, t, twi, v, -k, bad, store);
}

// The transform of the midpoints of P + 2 nodes x[i] = node(i): input j is the cubic midpoint
// (9 (x[j+1] + x[j+2]) - x[j] - x[j+3]) / 16 for j <= P - 2, and 0 at P - 1.  The nodes are
// quantised once and the midpoints are integer, at 2^-57 of the largest node; in FP64 they are
// eight instructions a point, which held the SM longer than the butterflies.  Nodes that
// are all zero give zero outputs without a transform (the far field of a put above the strike).
// `node` may read buf.
template <int DIR, int P, class L, class S>
__device__ __forceinline__ void fx_fft_mid(double2* bufd, int t, const double2* __restrict__ tw, const L& node, const S& store) {
    constexpr int V = fft_values<double>(P), NT = P / V, NW = NT / 32;
    static_assert(NT % 32 == 0 && NW <= 16, "whole warps");
    fx2* buf = reinterpret_cast<fx2*>(bufd);
    unsigned* red = fx_slots(bufd, P);
    const int4* twi = reinterpret_cast<const int4*>(tw + P);
    fx2 x[V + 1];
    unsigned big = 0;
#pragma unroll
    for (int r = 0; r <= V; ++r) {
        const double2 d = (r < V || t < 2) ? node(t + r * NT) : make_double2(0.0, 0.0);
        x[r] = fx2{__double_as_longlong(d.x), __double_as_longlong(d.y)};
        big = max(big, max((unsigned)(x[r].x >> 32) & 0x7fffffffu, (unsigned)(x[r].y >> 32) & 0x7fffffffu));
    }
    big = __reduce_max_sync(0xffffffffu, big);
    if ((t & 31) == 0) red[t >> 5] = big;
    __syncthreads();                          // also: every node is read before any store
#pragma unroll
    for (int u = 0; u < NW; ++u) big = max(big, red[u]);
    if constexpr (!is_fx_then<S>::value) {
        if (__syncthreads_or(big != 0) == 0) {
#pragma unroll
            for (int r = 0; r < V; ++r) store(t + r * NT, make_double2(0.0, 0.0));
            __syncthreads();
            return;
        }
    }
    const bool bad = big >= 0x7ff00000u;
    const int k = fx_bits(V) - 1 - ((int)(big >> 20) - 1022);
#pragma unroll
    for (int r = 0; r <= V; ++r)
        if (r < V || t < 2)
            buf[padi(t + r * NT)] = fx2{fx_quantise((unsigned)(x[r].x >> 32), (unsigned)x[r].x, k),
                                        fx_quantise((unsigned)(x[r].y >> 32), (unsigned)x[r].y, k)};
    __syncthreads();
    fx2 v[V];
#pragma unroll
    for (int r = 0; r < V; ++r) {
        const int j = t + r * NT;
        const fx2 a = buf[padi(j)], b = buf[padi(j + 1)], c = buf[padi(j + 2)];
        const fx2 d = j <= P - 2 ? buf[padi(j + 3)] : fx2{0, 0};
        v[r] = j <= P - 2 ? fx2{(9 * (b.x + c.x) - (a.x + d.x) + 8) >> 4, (9 * (b.y + c.y) - (a.y + d.y) + 8) >> 4} : fx2{0, 0};
    }
    __syncthreads();
    fx_first<DIR, P>(buf, red, t, twi, v, -k, bad, store);
}
// Unscaled length-P complex DFT (DIR = -1: e^{-2 pi i jk/P}, DIR = +1: e^{+...})
// with input x[j] = load(j) and output X[k] handed to store(k, X[k]);
// tw is the twiddle table laid out as in common.cuh.  FUSE2 = false keeps a remainder of 2 as its own
// stage (for store functors heavy enough that the radix-32 stage spills).  Every thread of the block must call it (it
// synchronises the block); inputs read from `buf` must have been written and
// synchronised before the call.
template <typename R, int DIR, int P, bool FUSE2 = true, class L, class S>
__device__ __forceinline__ void block_fft(cpx<R>* buf, int t, const cpx<R>* __restrict__ tw, const L& load,
                                          const S& store) {
    if constexpr (sizeof(R) == 8 && fx_length(P)) fx_fft<DIR, P>(buf, t, tw, load, store);
    else fft_from<R, DIR, P, 1, FUSE2>(buf, t, tw, load, store);
}
// A loader marked `mid` gives P + 2 nodes; the transform's inputs are their midpoints.
template <class T, class = void> struct is_mid { static constexpr bool value = false; };
template <class T> struct is_mid<T, decltype((void)T::mid, void())> { static constexpr bool value = true; };
// Forward transform of load(j), product with the spectrum column w (0 where !valid), inverse
// transform into `store`: the column passes.  In block fixed point the column is in
// integers (fx_spectrum_entry) and nothing is converted between the transforms: jump sum N = 512 112 -> 96 us, N = 1024
// 284 -> 250, N = 2048 1019 -> 830, with the integer midpoints of fx_fft_mid.
template <typename R, int P, class L, class S>
__device__ __forceinline__ void block_conv(cpx<R>* buf, int t, const cpx<R>* __restrict__ tw, const cpx<R>* w, bool valid,
                                           const L& load, const S& store) {
    if constexpr (sizeof(R) == 8 && fx_length(P)) {
        const int4* wi = reinterpret_cast<const int4*>(w);
        const FxThen<S> then{wi, fx_spectrum_code(wi, valid), valid, store};
        if constexpr (is_mid<L>::value) fx_fft_mid<-1, P>(buf, t, tw, load, then);
        else fx_fft<-1, P>(buf, t, tw, load, then);
    } else {
        auto product = [&](int k2, cpx<R> v) { buf[padi(k2)] = cmul(v, valid ? __ldg(&w[k2]) : mk<R>(R(0), R(0))); };
        if constexpr (is_mid<L>::value) {
            // nodes staged in buf (constant trip count with a guard: the loop unrolls and its
            // loads go out together)
            constexpr int NT = P / fft_values<R>(P);
#pragma unroll
            for (int q = 0; q < (P + 2 + NT - 1) / NT; ++q) {
                const int i = t + q * NT;
                if (i < P + 2) buf[padi(i)] = load(i);
            }
            __syncthreads();
            auto mid = [&](int i) -> cpx<R> {
                if (i > P - 2) return mk<R>(R(0), R(0));
                const cpx<R> x0 = buf[padi(i)], x1 = buf[padi(i + 1)], x2 = buf[padi(i + 2)], x3 = buf[padi(i + 3)];
                return mk<R>(R(-0.0625) * (x0.x + x3.x) + R(0.5625) * (x1.x + x2.x),
                             R(-0.0625) * (x0.y + x3.y) + R(0.5625) * (x1.y + x2.y));
            };
            block_fft<R, -1, P>(buf, t, tw, mid, product);
        } else {
            block_fft<R, -1, P>(buf, t, tw, load, product);
        }
        block_fft<R, +1, P>(buf, t, tw, SmemLoad<R>{buf}, store);
    }
}
#endif

}  // namespace pide

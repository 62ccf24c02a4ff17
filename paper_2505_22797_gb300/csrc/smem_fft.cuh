// Mixed-radix DFTs of several sequences of one length in a block's shared
// memory (the transforms of the gridded operator, field_ops.cu).
//
// NC sequences lie interleaved, element e of sequence c at
// [smem_fft_pad(e) * NC + c], and move between two buffers, one Stockham pass
// per radix (16, 8, 5, 4, 3, 2; a length is a product of these).  One element of
// padding per eight keeps the first pass's stride-8 writes off one bank: for
// FP32 pairs and NC = 4, consecutive butterflies are then 36 words apart in
// 8-byte units instead of 32.
#pragma once

#include "common.cuh"

namespace mpi {

constexpr int kFftMaxPasses = 12;

struct SmemFft {
    int n = 1, np = 0;
    int rad[kFftMaxPasses];
    unsigned mag[kFftMaxPasses];  // j / Ns = (j * mag) >> 32, Ns = product of the earlier radices
};

// Radices of a length, or np = 0 for n > 1 when it has another prime factor.
inline SmemFft smem_fft_plan(int n)
{
    SmemFft p;
    p.n = n;
    int m = n, two = 0, r[kFftMaxPasses], k = 0;
    while (m % 2 == 0) m /= 2, ++two;
    // 2^two as 16s and 8s, as few as possible (4 or 2 where that leaves a rest)
    int n16 = two / 4;
    while (n16 > 0 && (two - 4 * n16) % 3 != 0) --n16;
    if ((two - 4 * n16) % 3 != 0) n16 = 0;
    two -= 4 * n16;
    while (n16-- > 0) r[k++] = 16;
    while (two >= 3 && two != 4) r[k++] = 8, two -= 3;
    while (two >= 2) r[k++] = 4, two -= 2;
    int one2 = two;
    while (m % 5 == 0 && k < kFftMaxPasses) r[k++] = 5, m /= 5;
    while (m % 3 == 0 && k < kFftMaxPasses) r[k++] = 3, m /= 3;
    while (one2-- > 0 && k < kFftMaxPasses) r[k++] = 2;
    if (m != 1) return p;
    p.np = k;
    int64_t ns = 1;
    for (int q = 0; q < k; ++q) {
        p.rad[q] = r[q];
        p.mag[q] = ns > 1 ? unsigned((int64_t(1) << 32) / ns + 1) : 0u;
        ns *= r[q];
    }
    return p;
}

__host__ __device__ inline int smem_fft_pad(int e) { return e + (e >> 3); }
// Elements of one buffer of NC sequences of length n.
inline size_t smem_fft_elems(int n, int nc) { return size_t(smem_fft_pad(n - 1) + 1) * nc; }

#ifdef __CUDACC__

template <typename R> __device__ __forceinline__ V2<R> cadd(V2<R> a, V2<R> b) { return V2<R>{a.x + b.x, a.y + b.y}; }
template <typename R> __device__ __forceinline__ V2<R> csub(V2<R> a, V2<R> b) { return V2<R>{a.x - b.x, a.y - b.y}; }
template <typename R> __device__ __forceinline__ V2<R> cmul(V2<R> a, V2<R> b)
{
    return V2<R>{fmx(a.x, b.x, -a.y * b.y), fmx(a.x, b.y, a.y * b.x)};
}
// a times i (SGN > 0) or -i (SGN < 0).
template <int SGN, typename R> __device__ __forceinline__ V2<R> cmuli(V2<R> a)
{
    return SGN > 0 ? V2<R>{-a.y, a.x} : V2<R>{a.y, -a.x};
}

template <int SGN, typename R> __device__ __forceinline__ void dft2(V2<R> &a, V2<R> &b)
{
    const V2<R> t = csub(a, b);
    a = cadd(a, b);
    b = t;
}
template <int SGN, typename R> __device__ __forceinline__ void dft4(V2<R> &a, V2<R> &b, V2<R> &c, V2<R> &d)
{
    const V2<R> s = cadd(a, c), t = csub(a, c), u = cadd(b, d), w = cmuli<SGN>(csub(b, d));
    a = cadd(s, u);
    b = cadd(t, w);
    c = csub(s, u);
    d = csub(t, w);
}
template <int RAD, int SGN, typename R> __device__ __forceinline__ void dft(V2<R> (&v)[RAD])
{
    if constexpr (RAD == 2) {
        dft2<SGN>(v[0], v[1]);
    } else if constexpr (RAD == 3) {
        const R h = R(0.86602540378443864676);  // sin(pi/3)
        const V2<R> s = cadd(v[1], v[2]), d = cmuli<SGN>(csub(v[1], v[2]));
        const V2<R> m = V2<R>{fmx(R(-0.5), s.x, v[0].x), fmx(R(-0.5), s.y, v[0].y)};
        v[0] = cadd(v[0], s);
        v[1] = V2<R>{fmx(h, d.x, m.x), fmx(h, d.y, m.y)};
        v[2] = V2<R>{fmx(-h, d.x, m.x), fmx(-h, d.y, m.y)};
    } else if constexpr (RAD == 4) {
        dft4<SGN>(v[0], v[1], v[2], v[3]);
    } else if constexpr (RAD == 5) {
        const R c1 = R(0.30901699437494742410), s1 = R(0.95105651629515357212);   // cos, sin of 2 pi/5
        const R c2 = R(-0.80901699437494742410), s2 = R(0.58778525229247312917);  // cos, sin of 4 pi/5
        const V2<R> a = cadd(v[1], v[4]), b = cadd(v[2], v[3]);
        const V2<R> d = cmuli<SGN>(csub(v[1], v[4])), e = cmuli<SGN>(csub(v[2], v[3]));
        const V2<R> m1 = V2<R>{fmx(c2, b.x, fmx(c1, a.x, v[0].x)), fmx(c2, b.y, fmx(c1, a.y, v[0].y))};
        const V2<R> m2 = V2<R>{fmx(c1, b.x, fmx(c2, a.x, v[0].x)), fmx(c1, b.y, fmx(c2, a.y, v[0].y))};
        const V2<R> n1 = V2<R>{fmx(s2, e.x, s1 * d.x), fmx(s2, e.y, s1 * d.y)};
        const V2<R> n2 = V2<R>{fmx(-s1, e.x, s2 * d.x), fmx(-s1, e.y, s2 * d.y)};
        v[0] = cadd(v[0], cadd(a, b));
        v[1] = cadd(m1, n1);
        v[4] = csub(m1, n1);
        v[2] = cadd(m2, n2);
        v[3] = csub(m2, n2);
    } else if constexpr (RAD == 16) {
        // 4 x 4: DFTs over n1 of v[4 n1 + n2], twiddles w16^(n2 k1), DFTs over n2
        const R c1 = R(0.92387953251128675613), s1 = R(0.38268343236508977173), h = R(0.70710678118654752440);
#pragma unroll
        for (int n2 = 0; n2 < 4; ++n2) dft4<SGN>(v[n2], v[4 + n2], v[8 + n2], v[12 + n2]);
        // v[4 k1 + n2]
        const R S = R(SGN);
        v[5] = cmul(v[5], V2<R>{c1, S * s1});
        v[6] = cmul(v[6], V2<R>{h, S * h});
        v[7] = cmul(v[7], V2<R>{s1, S * c1});
        v[9] = cmul(v[9], V2<R>{h, S * h});
        v[10] = cmuli<SGN>(v[10]);
        v[11] = cmul(v[11], V2<R>{-h, S * h});
        v[13] = cmul(v[13], V2<R>{s1, S * c1});
        v[14] = cmul(v[14], V2<R>{-h, S * h});
        v[15] = cmul(v[15], V2<R>{-c1, -S * s1});
#pragma unroll
        for (int k1 = 0; k1 < 4; ++k1) dft4<SGN>(v[4 * k1], v[4 * k1 + 1], v[4 * k1 + 2], v[4 * k1 + 3]);
        // v[4 k1 + k2] is output k1 + 4 k2: transpose
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = i + 1; j < 4; ++j) {
                const V2<R> t = v[4 * i + j];
                v[4 * i + j] = v[4 * j + i];
                v[4 * j + i] = t;
            }
    } else {
        static_assert(RAD == 8, "radix");
        const R h = R(0.70710678118654752440);
        dft4<SGN>(v[0], v[2], v[4], v[6]);
        dft4<SGN>(v[1], v[3], v[5], v[7]);
        // v[1], v[3], v[5], v[7] now hold the odd half's outputs 0, 1, 2, 3
        const V2<R> o1 = v[3], o2 = cmuli<SGN>(v[5]), o3 = v[7];
        const V2<R> w1 = SGN > 0 ? V2<R>{h * (o1.x - o1.y), h * (o1.x + o1.y)} : V2<R>{h * (o1.x + o1.y), h * (o1.y - o1.x)};
        const V2<R> w3 = SGN > 0 ? V2<R>{-h * (o3.x + o3.y), h * (o3.x - o3.y)} : V2<R>{h * (o3.y - o3.x), -h * (o3.x + o3.y)};
        const V2<R> e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1];
        v[0] = cadd(e0, o0);
        v[4] = csub(e0, o0);
        v[1] = cadd(e1, w1);
        v[5] = csub(e1, w1);
        v[2] = cadd(e2, o2);
        v[6] = csub(e2, o2);
        v[3] = cadd(e3, w3);
        v[7] = csub(e3, w3);
    }
}

// One pass of radix RAD after passes of product ns.  tw: exp(-2 pi i t / n).
template <int RAD, int NC, int SGN, typename R>
__device__ __forceinline__ void smem_fft_pass(const V2<R> *__restrict__ a, V2<R> *__restrict__ b, int n, int ns,
                                              unsigned mag, const V2<R> *__restrict__ tw)
{
    const int m = n / RAD;
    const int ts = m / ns;  // twiddle step: n / (ns RAD)
    for (int t = threadIdx.x; t < NC * m; t += blockDim.x) {
        const int c = t % NC, j = t / NC;
        const int q = ns > 1 ? int(__umulhi(unsigned(j), mag)) : j;
        const int k = j - q * ns;
        V2<R> v[RAD];
        if ((m & 7) == 0) {  // padded strides are uniform
            const V2<R> *s = a + smem_fft_pad(j) * NC + c;
            const int ms = (m + (m >> 3)) * NC;
#pragma unroll
            for (int r = 0; r < RAD; ++r) v[r] = s[r * ms];
        } else {
#pragma unroll
            for (int r = 0; r < RAD; ++r) v[r] = a[smem_fft_pad(j + r * m) * NC + c];
        }
        if (ns > 1) {
#pragma unroll
            for (int r = 1; r < RAD; ++r) {
                V2<R> w = tw[k * ts * r];
                if (SGN > 0) w.y = -w.y;
                v[r] = cmul(v[r], w);
            }
        }
        dft<RAD, SGN>(v);
        const int base = q * ns * RAD + k;
        V2<R> *o = b + smem_fft_pad(base) * NC + c;
        if ((ns & 7) == 0) {
            const int os = (ns + (ns >> 3)) * NC;
#pragma unroll
            for (int r = 0; r < RAD; ++r) o[r * os] = v[r];
        } else if (RAD % 8 == 0 && ns == 1) {
#pragma unroll
            for (int r = 0; r < RAD; ++r) o[(r + (r >> 3)) * NC] = v[r];
        } else {
#pragma unroll
            for (int r = 0; r < RAD; ++r) b[smem_fft_pad(base + r * ns) * NC + c] = v[r];
        }
    }
}

// The DFT (SGN -1: exp(-2 pi i ..), +1: the unscaled inverse) of the NC
// sequences in a; b is the second buffer.  All threads of the block call it
// after the data in a are visible; returns the buffer that holds the result
// (visible to all threads).
template <int NC, int SGN, typename R>
__device__ V2<R> *smem_fft(V2<R> *a, V2<R> *b, const SmemFft &p, const V2<R> *__restrict__ tw)
{
    int ns = 1;
#pragma unroll 1
    for (int q = 0; q < p.np; ++q) {
        const int r = p.rad[q];
        const unsigned mag = p.mag[q];
        if (r == 16) smem_fft_pass<16, NC, SGN, R>(a, b, p.n, ns, mag, tw);
        else if (r == 8) smem_fft_pass<8, NC, SGN, R>(a, b, p.n, ns, mag, tw);
        else if (r == 4) smem_fft_pass<4, NC, SGN, R>(a, b, p.n, ns, mag, tw);
        else if (r == 5) smem_fft_pass<5, NC, SGN, R>(a, b, p.n, ns, mag, tw);
        else if (r == 3) smem_fft_pass<3, NC, SGN, R>(a, b, p.n, ns, mag, tw);
        else smem_fft_pass<2, NC, SGN, R>(a, b, p.n, ns, mag, tw);
        ns *= r;
        __syncthreads();
        V2<R> *s = a;
        a = b;
        b = s;
    }
    return a;
}

#endif

}  // namespace mpi

// Transforms of a few hundred to a few thousand points in shared memory, in
// the Stockham form: natural order in and out, two buffers used in turn, each
// pass giving every thread one sub-transform of radix 8, 6, 5, 4, 3 or 2 in
// registers (the in-plane grid transforms and the FP32 line transforms).
#pragma once

#include <cstdint>
#include <vector>

namespace fbc {

constexpr int kMaxPass = 8;

// One transform length and its passes: pass p has radix R[p], Ns[p] = the product of the earlier
// radices, NR[p] = N / R[p] work items per sequence, twiddle step N / (Ns R); divisions by NR and Ns
// as multiply-high, add and shift (m, l).
struct Fft1D {
    int N = 0, np = 0;
    int R[kMaxPass], Ns[kMaxPass], NR[kMaxPass], tstep[kMaxPass];
    unsigned mNR[kMaxPass], mNs[kMaxPass];
    int lNR[kMaxPass], lNs[kMaxPass];
};

namespace fft {

// n / d for 0 <= n < 2^31 with (m, l) from div_magic(d)
__device__ __forceinline__ int fdiv(int n, unsigned m, int l) {
    return (int)((__umulhi((unsigned)n, m) + (unsigned)n) >> l);
}

inline void div_magic(int d, unsigned* m, int* l) {
    int s = 0;
    while ((1LL << s) < d) s++;
    *l = s;
    *m = (unsigned)((((unsigned long long)1 << 32) * (((unsigned long long)1 << s) - (unsigned long long)d)) /
                    (unsigned long long)d + 1ULL);
}

// fewest passes of radix 8, 6, 5, 4, 3, 2 with product n (empty if n has another prime factor)
inline std::vector<int> radix_passes(int n) {
    static const int kRad[6] = {8, 6, 5, 4, 3, 2};
    std::vector<std::vector<int>> best(n + 1);
    std::vector<bool> ok(n + 1, false);
    ok[1] = true;
    for (int m = 2; m <= n; m++) {
        if (n % m) continue;
        for (int R : kRad)
            if (m % R == 0 && ok[m / R] && (!ok[m] || best[m / R].size() + 1 < best[m].size())) {
                best[m] = best[m / R];
                best[m].push_back(R);
                ok[m] = true;
            }
    }
    return ok[n] ? best[n] : std::vector<int>();
}

// The passes of a transform of exactly N points (np = 0 if N has a prime factor above 5).
inline Fft1D make_fft(int N) {
    Fft1D F;
    const std::vector<int> p = radix_passes(N);
    F.N = N;
    F.np = (int)p.size() <= kMaxPass ? (int)p.size() : 0;
    int Ns = 1;
    for (int q = 0; q < F.np; q++) {
        F.R[q] = p[q], F.Ns[q] = Ns, F.NR[q] = N / p[q], F.tstep[q] = N / (Ns * p[q]);
        div_magic(F.NR[q], &F.mNR[q], &F.lNR[q]);
        div_magic(Ns, &F.mNs[q], &F.lNs[q]);
        Ns *= p[q];
    }
    return F;
}

__device__ __forceinline__ float fmx(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fmx(double a, double b, double c) { return __fma_rn(a, b, c); }

template <typename C> __device__ __forceinline__ C mkc(decltype(C::x) x, decltype(C::x) y) {
    C c;
    c.x = x, c.y = y;
    return c;
}

template <typename C> __device__ __forceinline__ C cmul(C a, C w) {
    return mkc<C>(fmx(a.x, w.x, -a.y * w.y), fmx(a.x, w.y, a.y * w.x));
}

// Shared-memory index with one pad slot after every 8 complex numbers: the early Stockham passes store
// with strides of 8 and 64 elements, which would otherwise hit the same banks.
__device__ __forceinline__ int sx(int i) { return i + (i >> 3); }
__host__ __device__ inline int padded(int n) { return n + (n >> 3) + 1; }

template <bool INV, typename C> __device__ __forceinline__ C add(C a, C b) { return mkc<C>(a.x + b.x, a.y + b.y); }
template <bool INV, typename C> __device__ __forceinline__ C sub(C a, C b) { return mkc<C>(a.x - b.x, a.y - b.y); }
// times -i (forward) or +i (inverse)
template <bool INV, typename C> __device__ __forceinline__ C rot(C a) {
    return INV ? mkc<C>(-a.y, a.x) : mkc<C>(a.y, -a.x);
}

template <bool INV, typename C> __device__ __forceinline__ void dft2(C* v) {
    const C t = v[0];
    v[0] = add<INV>(t, v[1]), v[1] = sub<INV>(t, v[1]);
}

template <bool INV, typename C> __device__ __forceinline__ void dft4(C& v0, C& v1, C& v2, C& v3) {
    const C a0 = add<INV>(v0, v2), a1 = sub<INV>(v0, v2), a2 = add<INV>(v1, v3), a3 = rot<INV>(sub<INV>(v1, v3));
    v0 = add<INV>(a0, a2), v1 = add<INV>(a1, a3), v2 = sub<INV>(a0, a2), v3 = sub<INV>(a1, a3);
}

// 8-point transform from two 4-point ones (even and odd inputs) and the factors exp(-+ i pi k / 4)
template <bool INV, typename C> __device__ __forceinline__ void dft8(C* v) {
    using R = decltype(C::x);
    const R h = (R)0.70710678118654752440;
    C e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
    dft4<INV>(e0, e1, e2, e3);
    dft4<INV>(o0, o1, o2, o3);
    o1 = INV ? mkc<C>((o1.x - o1.y) * h, (o1.x + o1.y) * h) : mkc<C>((o1.x + o1.y) * h, (o1.y - o1.x) * h);
    o2 = rot<INV>(o2);
    o3 = INV ? mkc<C>(-(o3.x + o3.y) * h, (o3.x - o3.y) * h) : mkc<C>((o3.y - o3.x) * h, -(o3.x + o3.y) * h);
    v[0] = add<INV>(e0, o0), v[4] = sub<INV>(e0, o0);
    v[1] = add<INV>(e1, o1), v[5] = sub<INV>(e1, o1);
    v[2] = add<INV>(e2, o2), v[6] = sub<INV>(e2, o2);
    v[3] = add<INV>(e3, o3), v[7] = sub<INV>(e3, o3);
}

template <bool INV, typename C> __device__ __forceinline__ void dft3(C& v0, C& v1, C& v2) {
    using R = decltype(C::x);
    const R h = (R)0.86602540378443864676;  // sin(2 pi / 3)
    const C t1 = add<INV>(v1, v2), d = sub<INV>(v1, v2);
    const C t2 = INV ? mkc<C>(-d.y * h, d.x * h) : mkc<C>(d.y * h, -d.x * h);  // -+ i h (v1 - v2)
    const C m = mkc<C>(v0.x - (R)0.5 * t1.x, v0.y - (R)0.5 * t1.y);
    v0 = add<INV>(v0, t1), v1 = add<INV>(m, t2), v2 = sub<INV>(m, t2);
}

template <bool INV, typename C> __device__ __forceinline__ void dft5(C* v) {
    using R = decltype(C::x);
    const R c1 = (R)0.30901699437494742410, c2 = (R)-0.80901699437494742410;  // cos(2 pi / 5), cos(4 pi / 5)
    const R s1 = (R)0.95105651629515357212, s2 = (R)0.58778525229247312917;   // sin(2 pi / 5), sin(4 pi / 5)
    const C t1 = add<INV>(v[1], v[4]), t2 = add<INV>(v[2], v[3]), t3 = sub<INV>(v[1], v[4]), t4 = sub<INV>(v[2], v[3]);
    const C a1 = mkc<C>(v[0].x + c1 * t1.x + c2 * t2.x, v[0].y + c1 * t1.y + c2 * t2.y);
    const C a2 = mkc<C>(v[0].x + c2 * t1.x + c1 * t2.x, v[0].y + c2 * t1.y + c1 * t2.y);
    const C b1 = mkc<C>(s1 * t3.x + s2 * t4.x, s1 * t3.y + s2 * t4.y);
    const C b2 = mkc<C>(s2 * t3.x - s1 * t4.x, s2 * t3.y - s1 * t4.y);
    // forward: y1 = a1 - i b1, y2 = a2 - i b2, y3 = a2 + i b2, y4 = a1 + i b1 (inverse: i -> -i)
    const C ib1 = rot<INV>(b1), ib2 = rot<INV>(b2);
    v[0] = mkc<C>(v[0].x + t1.x + t2.x, v[0].y + t1.y + t2.y);
    v[1] = add<INV>(a1, ib1), v[4] = sub<INV>(a1, ib1);
    v[2] = add<INV>(a2, ib2), v[3] = sub<INV>(a2, ib2);
}

// 6 points from two 3-point transforms (even and odd inputs) and the factors exp(-+ i pi k / 3)
template <bool INV, typename C> __device__ __forceinline__ void dft6(C* v) {
    using R = decltype(C::x);
    const R h = (R)0.86602540378443864676;
    C e0 = v[0], e1 = v[2], e2 = v[4], o0 = v[1], o1 = v[3], o2 = v[5];
    dft3<INV>(e0, e1, e2);
    dft3<INV>(o0, o1, o2);
    // w1 = 1/2 -+ i h, w2 = -1/2 -+ i h
    const R sg = INV ? (R)1 : (R)-1;
    o1 = mkc<C>((R)0.5 * o1.x - sg * h * o1.y, (R)0.5 * o1.y + sg * h * o1.x);
    o2 = mkc<C>((R)-0.5 * o2.x - sg * h * o2.y, (R)-0.5 * o2.y + sg * h * o2.x);
    v[0] = add<INV>(e0, o0), v[3] = sub<INV>(e0, o0);
    v[1] = add<INV>(e1, o1), v[4] = sub<INV>(e1, o1);
    v[2] = add<INV>(e2, o2), v[5] = sub<INV>(e2, o2);
}

// ---- FP64 butterflies with the twiddles folded in -----------------------------------------------------------------
// The FP64 pipe (two lanes a cycle and SM) bounds the in-plane FP64 transforms, so these count operations: a twiddled
// pair a +- w b is four fused multiply-adds and 2 a - (a + w b), two more (a product and the sums: eight); six points
// are three pairs and two three-point transforms without factors between them (2 and 3 are coprime); the factors of
// three- and eight-point transforms go into fused operations.  Six points with their twiddles: 50 operations (68),
// without 36 (48), and 24 with the upper half of the inputs zero; eight: 80 (84), 52 (56) and 36 (their pairs take eight
// operations: with six the rounding error of 512 points grew by 2 %).  Rms error against 80-bit sums, 20 normal vectors
// forward: 216 points 3.37e-16 (3.54e-16), 320 points 2.48e-16 (2.50e-16), 512 points 2.65e-16 (2.66e-16).

__device__ __forceinline__ double2 axpy2(double2 a, double h, double2 b) {  // a + h b
    return make_double2(__fma_rn(h, b.x, a.x), __fma_rn(h, b.y, a.y));
}
// p = a + w b, m = a - w b (EXACT: m by products of its own)
template <bool TW, bool EXACT = false> __device__ __forceinline__ void pair64(double2 a, double2 b, double2 w, double2& p, double2& m) {
    if (TW) {
        p = make_double2(__fma_rn(-w.y, b.y, __fma_rn(w.x, b.x, a.x)), __fma_rn(w.y, b.x, __fma_rn(w.x, b.y, a.y)));
        m = EXACT ? make_double2(__fma_rn(w.y, b.y, __fma_rn(-w.x, b.x, a.x)), __fma_rn(-w.y, b.x, __fma_rn(-w.x, b.y, a.y)))
                  : make_double2(__fma_rn(2.0, a.x, -p.x), __fma_rn(2.0, a.y, -p.y));
    } else {
        p = add<false>(a, b), m = sub<false>(a, b);
    }
}
template <bool INV> __device__ __forceinline__ void dft3_64(double2& v0, double2& v1, double2& v2) {
    const double h = INV ? -0.86602540378443864676 : 0.86602540378443864676;  // sin(2 pi / 3)
    const double2 t = add<false>(v1, v2), d = sub<false>(v1, v2), q = make_double2(d.y, -d.x), m = axpy2(v0, -0.5, t);
    v0 = add<false>(v0, t), v1 = axpy2(m, h, q), v2 = axpy2(m, -h, q);
}
// R points v, with TW times the twiddles w[1 .. R-1] first (already conjugated for the inverse); HALF: v[R/2 ..] are zero
template <int R, bool INV, bool TW, bool HALF> __device__ __forceinline__ void bfly64(double2* v, const double2* w) {
    static_assert(!(TW && HALF) && (!HALF || R == 6 || R == 8), "only first passes read zeros");
    auto tw = [&](int r) { return TW ? cmul(v[r], w[r]) : v[r]; };
    const double2 one = make_double2(1.0, 0.0);
    auto wr = [&](int r) { return TW ? w[r] : one; };
    if constexpr (R == 6) {
        double2 s0, s1, s2, d0, d1, d2;
        if (HALF) {
            s0 = d0 = v[0], s1 = d1 = v[2], s2 = v[1], d2 = make_double2(-v[1].x, -v[1].y);
        } else {
            pair64<TW>(v[0], v[3], wr(3), s0, d0);
            pair64<TW>(tw(2), v[5], wr(5), s1, d1);
            pair64<TW>(tw(4), v[1], wr(1), s2, d2);
        }
        dft3_64<INV>(s0, s1, s2);
        dft3_64<INV>(d0, d1, d2);
        v[0] = s0, v[4] = s1, v[2] = s2, v[3] = d0, v[1] = d1, v[5] = d2;
    } else if constexpr (R == 8) {
        const double h = 0.70710678118654752440;
        double2 e0, e1, e2, e3, o0, o1, o2, o3;
        if (HALF) {
            e0 = e1 = v[0], e2 = e3 = v[2], o0 = o1 = v[1], o2 = o3 = v[3];
        } else {
            pair64<TW, true>(v[0], v[4], wr(4), e0, e1);
            pair64<TW, true>(tw(2), v[6], wr(6), e2, e3);
            pair64<TW, true>(tw(1), v[5], wr(5), o0, o1);
            pair64<TW, true>(tw(3), v[7], wr(7), o2, o3);
        }
        e3 = rot<INV>(e3), o3 = rot<INV>(o3);
        const double2 a0 = add<false>(e0, e2), a2 = sub<false>(e0, e2), a1 = add<false>(e1, e3), a3 = sub<false>(e1, e3);
        const double2 b0 = add<false>(o0, o2), b2 = rot<INV>(sub<false>(o0, o2)), c1 = add<false>(o1, o3), c3 = sub<false>(o1, o3);
        // exp(-+ i pi / 4) c1 = h b1, exp(-+ 3 i pi / 4) c3 = h b3
        const double2 b1 = INV ? make_double2(c1.x - c1.y, c1.x + c1.y) : make_double2(c1.x + c1.y, c1.y - c1.x);
        const double2 b3 = INV ? make_double2(-(c3.x + c3.y), c3.x - c3.y) : make_double2(c3.y - c3.x, -(c3.x + c3.y));
        v[0] = add<false>(a0, b0), v[4] = sub<false>(a0, b0), v[2] = add<false>(a2, b2), v[6] = sub<false>(a2, b2);
        v[1] = axpy2(a1, h, b1), v[5] = axpy2(a1, -h, b1), v[3] = axpy2(a3, h, b3), v[7] = axpy2(a3, -h, b3);
    } else if constexpr (R == 4) {
        double2 a0, a1, a2, a3;
        pair64<TW, true>(v[0], v[2], wr(2), a0, a1);
        pair64<TW, true>(tw(1), v[3], wr(3), a2, a3);
        a3 = rot<INV>(a3);
        v[0] = add<false>(a0, a2), v[1] = add<false>(a1, a3), v[2] = sub<false>(a0, a2), v[3] = sub<false>(a1, a3);
    } else if constexpr (R == 2) {
        double2 p, m;
        pair64<TW>(v[0], v[1], wr(1), p, m);
        v[0] = p, v[1] = m;
    } else {
#pragma unroll
        for (int r = 1; r < R; r++) v[r] = tw(r);
        if constexpr (R == 3) dft3_64<INV>(v[0], v[1], v[2]);
        else dft5<INV>(v);
    }
}

// One Stockham pass (pass q of F, radix R) over nseq sequences of length N: work item j of a
// sequence reads x[j + r N/R], twiddles by exp(-+2 pi i r k / (Ns R)) with k = j mod Ns, transforms
// in registers and writes y[(j - k) R + k + r Ns].  tw[m] = exp(-2 pi i m / N), m < N.  FAST: the
// FP64 butterflies above; HALF: x[N/2 ..] are zero and not read.
template <int R, bool INV, bool FAST, bool HALF, typename C>
__device__ __forceinline__ void stockham_pass(const C* in, C* out, int nseq, const Fft1D& F, int q,
                                              const C* __restrict__ tw) {
    const int N = F.N, NR = F.NR[q], Ns = F.Ns[q], tstep = F.tstep[q];
    const unsigned mNR = F.mNR[q], mNs = F.mNs[q];
    const int lNR = F.lNR[q], lNs = F.lNs[q];
    for (int t = threadIdx.x; t < nseq * NR; t += blockDim.x) {
        const int seq = fdiv(t, mNR, lNR), j = t - seq * NR, k = j - fdiv(j, mNs, lNs) * Ns;
        const int x0 = seq * N + j;
        C v[R];
#pragma unroll
        for (int r = 0; r < (HALF ? R / 2 : R); r++) v[r] = in[sx(x0 + r * NR)];
        if constexpr (FAST) {
            if (!HALF && Ns > 1) {
                C w[R];
#pragma unroll
                for (int r = 1; r < R; r++) {
                    w[r] = __ldg(tw + r * k * tstep);
                    if (INV) w[r].y = -w[r].y;
                }
                bfly64<R, INV, true, false>(v, w);
            } else {
                bfly64<R, INV, false, HALF>(v, v);
            }
        } else {
            if (Ns > 1) {
#pragma unroll
                for (int r = 1; r < R; r++) {
                    C w = __ldg(tw + r * k * tstep);
                    if (INV) w.y = -w.y;
                    v[r] = cmul(v[r], w);
                }
            }
            if (R == 8) dft8<INV>(v);
            else if (R == 6) dft6<INV>(v);
            else if (R == 5) dft5<INV>(v);
            else if (R == 4) dft4<INV>(v[0], v[1], v[2], v[3]);
            else if (R == 3) dft3<INV>(v[0], v[1], v[2]);
            else dft2<INV>(v);
        }
        const int y0 = seq * N + (j - k) * R + k;
#pragma unroll
        for (int r = 0; r < R; r++) out[sx(y0 + r * Ns)] = v[r];
    }
}

// nseq transforms of length F.N in a (natural order, padded index); b is scratch
// of the same size.  Returns the buffer that holds the result.  Starts and ends at a barrier.
// half: the upper half of every sequence is zero (taken up by FAST where the first radix is 6 or 8).
template <bool INV, bool FAST = false, typename C>
__device__ C* fft_smem(C* a, C* b, int nseq, const Fft1D& F, const C* __restrict__ tw, bool half = false) {
    for (int q = 0; q < F.np; q++) {
        switch (F.R[q]) {
            case 8:
                if (FAST && half && q == 0) stockham_pass<8, INV, FAST, FAST>(a, b, nseq, F, q, tw);
                else stockham_pass<8, INV, FAST, false>(a, b, nseq, F, q, tw);
                break;
            case 6:
                if (FAST && half && q == 0) stockham_pass<6, INV, FAST, FAST>(a, b, nseq, F, q, tw);
                else stockham_pass<6, INV, FAST, false>(a, b, nseq, F, q, tw);
                break;
            case 5: stockham_pass<5, INV, FAST, false>(a, b, nseq, F, q, tw); break;
            case 4: stockham_pass<4, INV, FAST, false>(a, b, nseq, F, q, tw); break;
            case 3: stockham_pass<3, INV, FAST, false>(a, b, nseq, F, q, tw); break;
            default: stockham_pass<2, INV, FAST, false>(a, b, nseq, F, q, tw); break;
        }
        __syncthreads();
        C* t = a;
        a = b, b = t;
    }
    return a;
}

}  // namespace fft
}  // namespace fbc

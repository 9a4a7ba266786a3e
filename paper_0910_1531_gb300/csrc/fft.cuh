// Shared-memory Stockham FFT of many independent lines.
//
// A CTA holds `lines` transforms of length n in shared memory; element e of
// line l sits at buf[e * es + l * ls].  Tiles of columns of the y / z axes use
// es = T (tile width), ls = 1 so that consecutive threads touch consecutive
// addresses; rows of the x axis use es = 1 and an odd line pitch (free of bank
// conflicts for 8-byte elements).
//
// Stage with radix R and Ns = product of the earlier radices (self-sorting,
// out of place):  for butterfly j of n/R,
//     v[r] = src[j + r n/R] * w^( (j mod Ns) r n/(Ns R) ),  w = exp(-+2 pi i / n)
//     v    = DFT_R(v)
//     dst[(j / Ns) Ns R + (j mod Ns) + r Ns] = v[r]
// After all stages the result is in natural order.  The twiddle table holds
// exp(-2 pi i m / n), m < n, computed in double on the host.
#pragma once

#include <utility>

#include "common.cuh"

// Complex sum and difference of a butterfly.  FP32 uses the packed instructions, one for both parts
// (same rounding: the difference as b (-1) + a).  128^3, S = 3, one iteration 751 -> 743 us, 160^3 2.03 ->
// 1.97 ms: the passes issue in half of their cycles.
template <typename C> __device__ __forceinline__ C badd(C a, C b) { return cadd(a, b); }
template <typename C> __device__ __forceinline__ C bsub(C a, C b) { return csub(a, b); }
__device__ __forceinline__ unsigned long long pack2(float2 a) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a.x), "f"(a.y));
    return r;
}
__device__ __forceinline__ float2 unpack2(unsigned long long r) {
    float2 a;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a.x), "=f"(a.y) : "l"(r));
    return a;
}
template <> __device__ __forceinline__ float2 badd(float2 a, float2 b) {
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(b)));
    return unpack2(r);
}
template <> __device__ __forceinline__ float2 bsub(float2 a, float2 b) {
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(pack2(b)), "l"(pack2(make_float2(-1.0f, -1.0f))), "l"(pack2(a)));
    return unpack2(r);
}

template <bool INV, typename C> __device__ __forceinline__ void dft2(C* v) {
    C a = v[0], b = v[1];
    v[0] = badd(a, b);
    v[1] = bsub(a, b);
}

// rotate by -i (forward) or +i (inverse)
template <bool INV, typename C> __device__ __forceinline__ C rot(C a) { return INV ? cmul_i(a) : cmul_mi(a); }

template <bool INV, typename C> __device__ __forceinline__ void dft3(C* v) {
    using R = decltype(C().x);
    const R h = R(0.86602540378443864676);   // sqrt(3)/2
    C s = cadd(v[1], v[2]);
    C d = csub(v[1], v[2]);
    C m = csub(v[0], cscale(s, R(0.5)));
    C t = rot<INV>(cscale(d, h));              // -i h d (forward)
    v[0] = cadd(v[0], s);
    v[1] = cadd(m, t);
    v[2] = csub(m, t);
}

template <bool INV, typename C> __device__ __forceinline__ void dft4(C& x0, C& x1, C& x2, C& x3) {
    C a0 = badd(x0, x2), a1 = bsub(x0, x2);
    C a2 = badd(x1, x3), a3 = rot<INV>(bsub(x1, x3));
    x0 = badd(a0, a2);
    x2 = bsub(a0, a2);
    x1 = cadd(a1, a3);
    x3 = csub(a1, a3);
}

template <bool INV, typename C> __device__ __forceinline__ void dft4(C* v) { dft4<INV>(v[0], v[1], v[2], v[3]); }

template <bool INV, typename C> __device__ __forceinline__ void dft8(C* v) {
    using R = decltype(C().x);
    const R s = R(0.70710678118654752440);
    C e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6];
    C o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
    dft4<INV>(e0, e1, e2, e3);
    dft4<INV>(o0, o1, o2, o3);
    // o_k *= W8^k, W8 = exp(-+ 2 pi i / 8)
    o1 = INV ? cmake<C>((o1.x - o1.y) * s, (o1.x + o1.y) * s) : cmake<C>((o1.x + o1.y) * s, (o1.y - o1.x) * s);
    o2 = rot<INV>(o2);
    o3 = INV ? cmake<C>((-o3.x - o3.y) * s, (o3.x - o3.y) * s) : cmake<C>((o3.y - o3.x) * s, (-o3.x - o3.y) * s);
    v[0] = badd(e0, o0); v[4] = bsub(e0, o0);
    v[1] = cadd(e1, o1); v[5] = csub(e1, o1);
    v[2] = cadd(e2, o2); v[6] = csub(e2, o2);
    v[3] = cadd(e3, o3); v[7] = csub(e3, o3);
}

template <bool INV, typename C> __device__ __forceinline__ void dft16(C* v) {
    using R = decltype(C().x);
    // Y_r = DFT4(v[r], v[r+4], v[r+8], v[r+12]);  X[k1 + 4 k2] = DFT4_r(W16^(r k1) Y_r[k1])
    C y[16];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        C a = v[r], b = v[r + 4], c = v[r + 8], d = v[r + 12];
        dft4<INV>(a, b, c, d);
        y[r * 4 + 0] = a; y[r * 4 + 1] = b; y[r * 4 + 2] = c; y[r * 4 + 3] = d;
    }
    const R c1 = R(0.92387953251128675613), s1 = R(0.38268343236508977173), c2 = R(0.70710678118654752440);
    const R sg = INV ? R(1) : R(-1);
    // W16^m for m = r k1 in {0..9}: (cos(2 pi m/16), sg sin(2 pi m/16))
    const R wc[10] = {R(1), c1, c2, s1, R(0), -s1, -c2, -c1, R(-1), -c1};
    const R ws[10] = {R(0), s1, c2, c1, R(1), c1, c2, s1, R(0), -s1};
#pragma unroll
    for (int r = 1; r < 4; ++r) {
#pragma unroll
        for (int k1 = 1; k1 < 4; ++k1) {
            const int m = r * k1;
            if (m == 4) y[r * 4 + k1] = rot<INV>(y[r * 4 + k1]);
            else y[r * 4 + k1] = cmul(y[r * 4 + k1], cmake<C>(wc[m], sg * ws[m]));
        }
    }
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) {
        C a = y[0 * 4 + k1], b = y[1 * 4 + k1], c = y[2 * 4 + k1], d = y[3 * 4 + k1];
        dft4<INV>(a, b, c, d);
        v[k1] = a; v[k1 + 4] = b; v[k1 + 8] = c; v[k1 + 12] = d;
    }
}

// cos(2 pi p / q) and sin(2 pi p / q) in double at compile time: the angle reduced to [0, pi/4]
// by symmetry, then the Taylor series.
__host__ __device__ constexpr double ct_taylor(double x, int first) {
    double term = first ? x : 1.0, sum = term;
    for (int k = first + 1; k < 30; k += 2) {
        term *= -x * x / (double(k) * double(k + 1));
        sum += term;
    }
    return sum;
}
__host__ __device__ constexpr double ct_sin2pi(int p, int q);
__host__ __device__ constexpr double ct_cos2pi(int p, int q) {
    p = ((p % q) + q) % q;
    if (2 * p > q) p = q - p;
    if (4 * p > q) return -ct_cos2pi(q - 2 * p, 2 * q);
    if (8 * p > q) return ct_sin2pi(q - 4 * p, 4 * q);
    return ct_taylor(6.28318530717958647692 * double(p) / double(q), 0);
}
__host__ __device__ constexpr double ct_sin2pi(int p, int q) {
    p = ((p % q) + q) % q;
    if (2 * p > q) return -ct_sin2pi(q - p, q);
    if (4 * p > q) return ct_sin2pi(q - 2 * p, 2 * q);
    if (8 * p > q) return ct_cos2pi(q - 4 * p, 4 * q);
    return ct_taylor(6.28318530717958647692 * double(p) / double(q), 1);
}

template <int... I, typename F> __device__ __forceinline__ void ct_for_impl(std::integer_sequence<int, I...>, F&& f) {
    (f(std::integral_constant<int, I>{}), ...);
}
template <int N, typename F> __device__ __forceinline__ void ct_for(F&& f) {
    ct_for_impl(std::make_integer_sequence<int, N>{}, f);
}

// DFT of odd prime length R by pairs: with a_r = v_r + v_(R-r), b_r = v_r - v_(R-r), r = 1..(R-1)/2,
// X_q, X_(R-q) = v_0 + sum_r a_r cos(2 pi r q / R) -+ i sum_r b_r sin(2 pi r q / R).
template <int R, bool INV, typename C> __device__ __forceinline__ void dft_odd(C* v) {
    using T = decltype(C().x);
    constexpr int H = (R - 1) / 2;
    C a[H], b[H];
#pragma unroll
    for (int r = 0; r < H; ++r) {
        a[r] = badd(v[r + 1], v[R - 1 - r]);
        b[r] = bsub(v[r + 1], v[R - 1 - r]);
    }
    const C v0 = v[0];
#pragma unroll
    for (int r = 0; r < H; ++r) v[0] = badd(v[0], a[r]);
    ct_for<H>([&](auto qc) {
        constexpr int q = decltype(qc)::value + 1;
        C m = v0, t = cmake<C>(T(0), T(0));
        ct_for<H>([&](auto rc) {
            constexpr int r = decltype(rc)::value + 1;
            constexpr double c = ct_cos2pi(r * q, R), s = ct_sin2pi(r * q, R);
            m = cmake<C>(m.x + a[r - 1].x * T(c), m.y + a[r - 1].y * T(c));
            t = cmake<C>(t.x + b[r - 1].x * T(s), t.y + b[r - 1].y * T(s));
        });
        const C it = rot<INV>(t);
        v[q] = cadd(m, it);
        v[R - q] = csub(m, it);
    });
}

template <int R, bool INV, typename C> __device__ __forceinline__ void dft_small(C* v);

// DFT of length N1 N2 (coprime) without twiddles (Good-Thomas): inputs taken at N2 n1 + N1 n2 mod N,
// outputs at the index congruent to k1 mod N1 and k2 mod N2.
template <int N1, int N2, bool INV, typename C> __device__ __forceinline__ void dft_coprime(C* v) {
    constexpr int N = N1 * N2;
    C y[N];
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) {
        C u[N1];
#pragma unroll
        for (int n1 = 0; n1 < N1; ++n1) u[n1] = v[(N2 * n1 + N1 * n2) % N];
        dft_small<N1, INV>(u);
#pragma unroll
        for (int k1 = 0; k1 < N1; ++k1) y[k1 * N2 + n2] = u[k1];
    }
#pragma unroll
    for (int k1 = 0; k1 < N1; ++k1) {
        C u[N2];
#pragma unroll
        for (int n2 = 0; n2 < N2; ++n2) u[n2] = y[k1 * N2 + n2];
        dft_small<N2, INV>(u);
#pragma unroll
        for (int k = 0; k < N; ++k)
            if (k % N1 == k1) v[k] = u[k % N2];
    }
}

// DFT of length 9 as three by three with the twiddles W9^(n2 k1).
template <bool INV, typename C> __device__ __forceinline__ void dft9(C* v) {
    using T = decltype(C().x);
    C y[9];
#pragma unroll
    for (int n2 = 0; n2 < 3; ++n2) {
        C u[3] = {v[n2], v[n2 + 3], v[n2 + 6]};
        dft3<INV>(u);
#pragma unroll
        for (int k1 = 0; k1 < 3; ++k1) y[k1 * 3 + n2] = u[k1];
    }
    ct_for<2>([&](auto kc) {
        ct_for<2>([&](auto nc) {
            constexpr int k1 = decltype(kc)::value + 1, n2 = decltype(nc)::value + 1;
            constexpr double c = ct_cos2pi(k1 * n2, 9), s = ct_sin2pi(k1 * n2, 9);
            y[k1 * 3 + n2] = cmul(y[k1 * 3 + n2], cmake<C>(T(c), T(INV ? s : -s)));
        });
    });
#pragma unroll
    for (int k1 = 0; k1 < 3; ++k1) {
        C u[3] = {y[k1 * 3], y[k1 * 3 + 1], y[k1 * 3 + 2]};
        dft3<INV>(u);
#pragma unroll
        for (int k2 = 0; k2 < 3; ++k2) v[k1 + 3 * k2] = u[k2];
    }
}

template <int R, bool INV, typename C> __device__ __forceinline__ void dft_small(C* v) {
    if constexpr (R == 2) dft2<INV>(v);
    else if constexpr (R == 3) dft3<INV>(v);
    else if constexpr (R == 4) dft4<INV>(v);
    else if constexpr (R == 5 || R == 7) dft_odd<R, INV>(v);
    else if constexpr (R == 6) dft_coprime<2, 3, INV>(v);
    else if constexpr (R == 8) dft8<INV>(v);
    else if constexpr (R == 9) dft9<INV>(v);
    else if constexpr (R == 10) dft_coprime<2, 5, INV>(v);
    else if constexpr (R == 12) dft_coprime<4, 3, INV>(v);
    else if constexpr (R == 14) dft_coprime<2, 7, INV>(v);
    else if constexpr (R == 15) dft_coprime<3, 5, INV>(v);
    else dft16<INV>(v);
}

// What a stage does with an element it loads (first stages) or stores (last ones); e: its index on
// the axis.
struct PreNone {
    template <typename C> __device__ __forceinline__ void operator()(C&, int) const {}
};
struct PostStore {
    template <typename C> __device__ __forceinline__ void operator()(C* p, C v, int) const { *p = v; }
};

// ------------------------------------------------------------------------------------
// Run-time transforms: the Stockham stages of an AxisPlan.  NT: threads of the block.  Divisions by
// run-time constants are multiplications (FastDiv).  Lines are the rows of RtRows or the columns of
// RtCols; either maps a task (one butterfly of one line) to the butterfly j and the shared-memory
// offset of the line's element 0, and gives the distance between its elements.
// ------------------------------------------------------------------------------------
// `lines` rows: element e of line l at e + l ls, ls odd; line index fastest across threads, so that
// the butterflies of a half-warp fall into distinct banks.
struct RtRows {
    int lines, ls;
    FastDiv dl;
    __device__ __forceinline__ RtRows(int n, int pitch) : lines(n), ls(pitch), dl(n) {}
    __device__ __forceinline__ int count() const { return lines; }
    __device__ __forceinline__ int stride() const { return 1; }
    __device__ __forceinline__ void split(int task, const AxisPlan&, int, int& j, int& off) const {
        j = dl.div(task);
        off = (task - j * lines) * ls;
    }
};
// Tiles of T columns by P planes of the other axis.  Along y the planes follow one another (element
// e of column t of plane p at (p n + e) T + t), along z they are interleaved ((e P + p) T + t): the
// orders in which a TMA box lands.  Threads run over t, then over what is contiguous next.
template <int T> struct RtCols {
    int P, es, ps;
    bool zax;
    FastDiv dp;
    __device__ __forceinline__ RtCols(int planes, int n, bool z)
        : P(planes), es(z ? planes * T : T), ps(z ? T : n * T), zax(z), dp(planes) {}
    __device__ __forceinline__ int count() const { return P * T; }
    __device__ __forceinline__ int stride() const { return es; }
    __device__ __forceinline__ void split(int task, const AxisPlan& a, int s, int& j, int& off) const {
        const int t = task % T, rest = task / T;
        int p = 0;
        if (P == 1) j = rest;
        else if (zax) { j = dp.div(rest); p = rest - j * P; }
        else { p = a.dm[s].div(rest); j = rest - p * a.m[s]; }
        off = p * ps + t;
    }
};

template <int R, bool INV, int NT, typename L, typename Pre, typename Post, typename C>
__device__ __forceinline__ void rt_stage(const C* __restrict__ src, C* __restrict__ dst, const AxisPlan& p, int s,
                                         const L& lines, const C* __restrict__ tw, Pre pre, Post post) {
    const int ES = lines.stride();
    const int m = p.m[s], ns = p.ns[s].d, tws = p.tws[s];
    const FastDiv dns = p.ns[s];
    const int total = m * lines.count();
    for (int task = threadIdx.x; task < total; task += NT) {
        int j, off;
        lines.split(task, p, s, j, off);
        const int q = dns.div(j), k = j - q * ns;
        const C* s0 = src + off + j * ES;
        C v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            v[r] = s0[r * m * ES];
            pre(v[r], j + r * m);
        }
        if (ns > 1) {
            const C* w0 = tw + k * tws;
#pragma unroll
            for (int r = 1; r < R; ++r) {
                C w = w0[(r - 1) * k * tws];
                if (INV) w.y = -w.y;
                v[r] = cmul(v[r], w);
            }
        }
        dft_small<R, INV>(v);
        C* d0 = dst + off + (q * ns * R + k) * ES;
#pragma unroll
        for (int r = 0; r < R; ++r) post(d0 + r * ns * ES, v[r], q * ns * R + k + r * ns);
    }
}

// Stage of a prime radix R >= 11 (the pairs of dft_odd), its outputs spread over threads: a thread
// forms X_q and X_(R-q) of QG consecutive q of one butterfly (and X_0 with the first ones).  The
// roots W_R^(r q) = tw[(r q mod R) m] are the same for a whole butterfly and mostly for a warp.
template <int R, bool INV, int NT, typename L, typename Pre, typename Post, typename C>
__device__ __noinline__ void rt_stage_prime(const C* __restrict__ src, C* __restrict__ dst, const AxisPlan& p, int s,
                                            const L& lines, const C* __restrict__ tw, Pre pre, Post post) {
    using F = decltype(C().x);
    const int ES = lines.stride();
    constexpr int H = (R - 1) / 2, QG = 4, NG = (H + QG - 1) / QG;
    const int m = p.m[s], ns = p.ns[s].d, tws = p.tws[s];
    const FastDiv dns = p.ns[s];
    const int per = m * lines.count();
    for (int task = threadIdx.x; task < per * NG; task += NT) {
        int grp = 0, rem = task;
        while (rem >= per) { rem -= per; ++grp; }
        int j, off;
        lines.split(rem, p, s, j, off);
        const int q = dns.div(j), k = j - q * ns;
        const C* s0 = src + off + j * ES;
        C v0 = s0[0];
        pre(v0, j);
        C a[H], b[H], x0 = v0;
#pragma unroll
        for (int r = 1; r <= H; ++r) {
            C u = s0[r * m * ES], w = s0[(R - r) * m * ES];
            pre(u, j + r * m);
            pre(w, j + (R - r) * m);
            if (ns > 1) {
                C t = tw[r * k * tws], t2 = tw[(R - r) * k * tws];
                if (INV) { t.y = -t.y; t2.y = -t2.y; }
                u = cmul(u, t);
                w = cmul(w, t2);
            }
            a[r - 1] = cadd(u, w);
            b[r - 1] = csub(u, w);
            x0 = cadd(x0, a[r - 1]);
        }
        const int e0 = q * ns * R + k;
        C* d0 = dst + off + e0 * ES;
        if (grp == 0) post(d0, x0, e0);
        const int q1 = grp * QG + QG < H ? grp * QG + QG : H;
#pragma unroll 1
        for (int o = grp * QG + 1; o <= q1; ++o) {
            C c = v0, t = cmake<C>(F(0), F(0));
            int e = 0;
#pragma unroll
            for (int r = 0; r < H; ++r) {
                e += o;
                if (e >= R) e -= R;
                const C w = tw[e * m];         // (cos, -sin)
                c = cmake<C>(c.x + a[r].x * w.x, c.y + a[r].y * w.x);
                t = cmake<C>(t.x - b[r].x * w.y, t.y - b[r].y * w.y);
            }
            const C it = rot<INV>(t);
            post(d0 + o * ns * ES, cadd(c, it), e0 + o * ns);
            post(d0 + (R - o) * ns * ES, csub(c, it), e0 + (R - o) * ns);
        }
    }
}

// Stage s of a plan.  BIG: lengths with a prime factor of 17..31 (kernels of their own, whose
// register budget the other lengths do not pay).
template <bool INV, int NT, bool BIG, typename L, typename Pre = PreNone, typename Post = PostStore, typename C>
__device__ __forceinline__ void rt_stage_any(const C* src, C* dst, const AxisPlan& p, int s, const L& lines,
                                             const C* tw, Pre pre = Pre{}, Post post = Post{}) {
#define DFT_RT(R) case R: rt_stage<R, INV, NT>(src, dst, p, s, lines, tw, pre, post); break;
#define DFT_RTP(R) case R: rt_stage_prime<R, INV, NT>(src, dst, p, s, lines, tw, pre, post); break;
    switch (p.radix[s]) {
        DFT_RT(2) DFT_RT(3) DFT_RT(4) DFT_RT(5) DFT_RT(6) DFT_RT(7) DFT_RT(8) DFT_RT(9) DFT_RT(10) DFT_RT(12)
        DFT_RT(14) DFT_RT(15) DFT_RT(16)
        DFT_RTP(11) DFT_RTP(13)
        default:
            if constexpr (BIG) {
                switch (p.radix[s]) { DFT_RTP(17) DFT_RTP(19) DFT_RTP(23) DFT_RTP(29) DFT_RTP(31) }
            }
    }
#undef DFT_RT
#undef DFT_RTP
}

// Transform the `lines` rows held in `a` (b is scratch of the same size) by the stages of a plan.
// The caller must __syncthreads() before the call (data in a visible).  Returns the buffer holding
// the result; all threads see it on return.
template <bool INV, bool BIG, int NT, typename C>
__device__ C* rt_fft_rows(C* a, C* b, const AxisPlan& p, int lines, int ls, const C* tw) {
    const RtRows rows(lines, ls);
    for (int s = 0; s < p.nstages; ++s) {
        rt_stage_any<INV, NT, BIG>(a, b, p, s, rows, tw);
        __syncthreads();
        C* t = a; a = b; b = t;
    }
    return a;
}

// ------------------------------------------------------------------------------------
// Compile-time transforms.  The same Stockham stages with the length, the radix plan and
// (for column tiles) the tile width known at compile time, so that index arithmetic is by
// constants and every loop unrolls.  Radix plans: two stages of near-equal radices, the larger
// first, so that both stages have butterflies for a block's threads (64 as 8 x 8 has eight per
// line in both, as 16 x 4 four, which leaves most lanes of a small block's warps idle; FP64, bound
// by whole warps on its pipe, most of all).  Line-search iteration, two species, against 16 first:
// 96^3 FP32 492 -> 369 us (there were three stages), 64^3 145 -> 139, 48^3 113 -> 99, 32^3 81 -> 75;
// FP64 32^3 408 -> 307, 48^3 1026 -> 714, 64^3 1856 -> 1566, 96^3 6254 -> 4952.
// ------------------------------------------------------------------------------------
__host__ __device__ constexpr int ct_radix_at(int n, int s) {
    const int r0 = n == 32 ? 8 : n == 48 ? 8 : n == 64 ? 8 : n == 96 ? 12 : 16;
    return s == 0 ? r0 : (s == 1 ? n / r0 : 0);
}
__host__ __device__ constexpr int ct_nstages(int n) { int s = 0; while (ct_radix_at(n, s) != 0) ++s; return s; }
__host__ __device__ constexpr int ct_ns_at(int n, int s) { int p = 1; for (int i = 0; i < s; ++i) p *= ct_radix_at(n, i); return p; }

constexpr int kFftThreads = 256;

// Compile-time x passes keep element e of a row at position e + floor(e / 16): the first
// Stockham stage writes its outputs with a stride of R (16) elements across threads, which the
// pad turns into 17 so the eight-byte stores of a half-warp hit distinct banks.
__host__ __device__ constexpr int ct_xpad(int e) { return e + (e >> 4); }

// Row pitch (elements) of the compile-time x passes: at least the padded row length, and,
// when a stage has M < 16 butterflies per row (16/M rows in one half-warp), congruent to M
// modulo 16 so that those rows fall into disjoint bank groups.
__host__ __device__ constexpr int ct_row_pitch(int n) {
    int msmall = 0;
    for (int s = 0; s < ct_nstages(n); ++s) {
        const int m = n / ct_radix_at(n, s);
        if (m < 16 && (msmall == 0 || m < msmall)) msmall = m;
    }
    const int len = ct_xpad(n - 1) + 1;
    if (msmall == 0) return len | 1;
    return len + (((msmall - len) % 16) + 16) % 16;
}

// One stage.  COLS: lines are tile columns (element e of line l at e*T + l, line index fastest
// across threads); otherwise lines are rows (element e of line l at e + l*ls, e fastest).
// Rows: the padded position ct_xpad(a + r s) of the r-th element a butterfly touches splits
// into a per-thread part and a compile-time part when s is a multiple of 16 (then (a + r s) >> 4
// = (a >> 4) + r s / 16), or when every a + r s stays inside one block of 16 positions past a
// multiple of 16 (loads: a < M, 16 % M == 0; stores: 16 % (NS R) == 0).  The butterfly then
// addresses its elements at one base pointer plus constants.
template <int M, int R> __host__ __device__ constexpr bool ct_split_loads() { return M % 16 == 0 || 16 % M == 0; }
template <int NS, int R> __host__ __device__ constexpr bool ct_split_stores() { return NS % 16 == 0 || 16 % (NS * R) == 0; }

template <int N, int R, int NS, bool INV, bool COLS, int T, typename C>
__device__ __forceinline__ void ct_stage(const C* __restrict__ src, C* __restrict__ dst, int lines, int ls,
                                         const C* __restrict__ tw) {
    constexpr int M = N / R;
    constexpr int TWSTEP = N / (NS * R);
    const int total = COLS ? M * T : M * lines;
    if constexpr (!COLS && ct_split_loads<M, R>() && ct_split_stores<NS, R>()) {
#pragma unroll 2
        for (int task = threadIdx.x; task < total; task += kFftThreads) {
            const int j = task % M, line = task / M;
            const int k = j % NS;
            // loads: element j + r M at pad(j) + r (M + M / 16) (M a multiple of 16), or at
            // j + pad(r M) (j < M <= 16, 16 % M == 0)
            const C* s0 = src + line * ls + (M % 16 == 0 ? ct_xpad(j) : j);
            C v[R];
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = s0[M % 16 == 0 ? r * (M + M / 16) : ct_xpad(r * M)];
            if constexpr (NS > 1) {
#pragma unroll
                for (int r = 1; r < R; ++r) {
                    C w = tw[k * r * TWSTEP];
                    if (INV) w.y = -w.y;
                    v[r] = cmul(v[r], w);
                }
            }
            dft_small<R, INV>(v);
            // stores: element b + r NS, b = (j / NS) NS R + k, at pad(b) + r (NS + NS / 16) (NS a
            // multiple of 16), or at b + b / 16 + r NS (b a multiple of NS R, a divisor of 16, plus k < NS)
            const int b = (j / NS) * (NS * R) + k;
            C* d0 = dst + line * ls + ct_xpad(b);
#pragma unroll
            for (int r = 0; r < R; ++r) d0[NS % 16 == 0 ? r * (NS + NS / 16) : r * NS] = v[r];
        }
        return;
    }
#pragma unroll 2
    for (int task = threadIdx.x; task < total; task += kFftThreads) {
        int line, j;
        if constexpr (COLS) { line = task % T; j = task / T; }
        else { j = task % M; line = task / M; }
        const int k = j % NS;
        const int off = COLS ? line : line * ls;
        constexpr int ES = COLS ? T : 1;
        C v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int e = j + r * M;
            v[r] = src[(COLS ? e * ES : ct_xpad(e)) + off];
        }
        if constexpr (NS > 1) {
#pragma unroll
            for (int r = 1; r < R; ++r) {
                C w = tw[k * r * TWSTEP];
                if (INV) w.y = -w.y;
                v[r] = cmul(v[r], w);
            }
        }
        dft_small<R, INV>(v);
        const int base = (j / NS) * (NS * R) + k;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int e = base + r * NS;
            dst[(COLS ? e * ES : ct_xpad(e)) + off] = v[r];
        }
    }
}

template <int N, bool INV, bool COLS, int T, int S, typename C>
__device__ __forceinline__ void ct_stages(C*& a, C*& b, int lines, int ls, const C* tw) {
    if constexpr (S < ct_nstages(N)) {
        constexpr int R = ct_radix_at(N, S);
        constexpr int NS = ct_ns_at(N, S);
        ct_stage<N, R, NS, INV, COLS, T>(a, b, lines, ls, tw);
        __syncthreads();
        C* t = a; a = b; b = t;
        ct_stages<N, INV, COLS, T, S + 1>(a, b, lines, ls, tw);
    }
}

// Compile-time counterpart of rt_fft_rows (same contract).  COLS with tile width T, or rows
// with `lines` rows of pitch ls.
template <int N, bool INV, bool COLS, int T, typename C>
__device__ __forceinline__ C* ct_fft(C* a, C* b, int lines, int ls, const C* tw) {
    ct_stages<N, INV, COLS, T, 0>(a, b, lines, ls, tw);
    return a;
}

// Rows of a length N > 0 by the compile-time stages, of any length (N = 0; N = -1 with a prime
// factor of 17..31) by those of the plan.
template <int N, bool INV, typename C>
__device__ __forceinline__ C* any_fft(C* a, C* b, const AxisPlan& p, int lines, int ls, const C* tw) {
    if constexpr (N > 0) return ct_fft<N, INV, false, 0>(a, b, lines, ls, tw);
    else return rt_fft_rows<INV, (N < 0), kFftThreads>(a, b, p, lines, ls, tw);
}

// ------------------------------------------------------------------------------------
// Grouped column transforms: `groups` tiles of T columns x N rows, tile g at offset g * GSTR,
// transformed together so that every stage has groups * T * N / R butterflies for the CTA's
// NT threads.  Inside a tile, element e of column t sits at T * ct_xpad(e) + t (padded: the
// first stage's outputs, R rows apart across threads, then fall into distinct bank groups);
// SRC_DENSE / DST_DENSE make the first stage read, or the last stage write, the dense layout
// e * T + t of a TMA box instead.
// ------------------------------------------------------------------------------------
__host__ __device__ constexpr int ct_gpos(int e, int T) { return T * ct_xpad(e); }
__host__ __device__ constexpr int ct_gtile(int n, int T) { return T * (ct_xpad(n - 1) + 1); }
// group stride: the padded tile rounded up to 128 bytes (TMA destinations are 128-byte aligned)
__host__ __device__ constexpr int ct_gstride(int n, int T, int csize) {
    return (ct_gtile(n, T) + 128 / csize - 1) / (128 / csize) * (128 / csize);
}

template <int N, int R, int NS, bool INV, int T, int GSTR, bool SD, bool DD, int NT, typename Pre = PreNone,
          typename Post = PostStore, typename C>
__device__ __forceinline__ void ct_stage_grouped(const C* __restrict__ src, C* __restrict__ dst, int groups,
                                                 const C* __restrict__ tw, Pre pre = Pre{}, Post post = Post{},
                                                 bool single = false) {
    constexpr int M = N / R;
    constexpr int TWSTEP = N / (NS * R);
    constexpr int PERG = M * T;
    const int total = single ? M : PERG * groups;
    for (int task = threadIdx.x; task < total; task += NT) {
        const int g = task / PERG;
        const int rem = task - g * PERG;
        const int t = single ? 0 : rem % T, j = single ? task : rem / T;
        const int k = j % NS;
        const int off = single ? 0 : g * GSTR + t;
        C v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int e = j + r * M;
            v[r] = src[(SD ? e * T : ct_gpos(e, T)) + off];
            pre(v[r], e);
        }
        if constexpr (NS > 1) {
#pragma unroll
            for (int r = 1; r < R; ++r) {
                C w = tw[k * r * TWSTEP];
                if (INV) w.y = -w.y;
                v[r] = cmul(v[r], w);
            }
        }
        dft_small<R, INV>(v);
        const int base = (j / NS) * (NS * R) + k;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int e = base + r * NS;
            post(dst + (DD ? e * T : ct_gpos(e, T)) + off, v[r], e);
        }
    }
}

template <int N, bool INV, int T, int GSTR, bool SD, bool DD, int NT, int S, typename C>
__device__ __forceinline__ void ct_stages_grouped(C*& a, C*& b, int groups, const C* tw) {
    if constexpr (S < ct_nstages(N)) {
        constexpr int R = ct_radix_at(N, S);
        constexpr int NS = ct_ns_at(N, S);
        constexpr bool last = (S + 1 == ct_nstages(N));
        ct_stage_grouped<N, R, NS, INV, T, GSTR, SD && S == 0, DD && last, NT>(a, b, groups, tw);
        __syncthreads();
        C* t = a; a = b; b = t;
        ct_stages_grouped<N, INV, T, GSTR, SD, DD, NT, S + 1>(a, b, groups, tw);
    }
}

// Transform `groups` tiles held in a (b: scratch of the same size); the caller syncs before;
// returns the buffer holding the result (synced).
template <int N, bool INV, int T, int GSTR, bool SD = false, bool DD = false, int NT = kFftThreads, typename C>
__device__ __forceinline__ C* ct_fft_grouped(C* a, C* b, int groups, const C* tw) {
    ct_stages_grouped<N, INV, T, GSTR, SD, DD, NT, 0>(a, b, groups, tw);
    return a;
}

// ------------------------------------------------------------------------------------
// In-place grouped column transforms (same layouts, SRC_DENSE / DST_DENSE meaning and twiddle
// table as ct_fft_grouped).  Each thread takes one butterfly of a stage, holds its R inputs in
// registers across a barrier and then writes its outputs over the same tile, so that no scratch
// tiles are needed; the groups are taken in chunks of NT / (T N / R) per pass of the threads
// (chunks touch disjoint groups, so one barrier per chunk orders its reads before its writes).
// The caller syncs before the call; the last stage is NOT followed by a barrier, so the caller
// syncs (after any proxy fence its TMA stores need) before reading the result.
// ------------------------------------------------------------------------------------
// barrier among the first `count` threads of the CTA (a multiple of 32), named barrier 1
__device__ __forceinline__ void bar_sync_first(int count) {
    asm volatile("bar.sync 1, %0;" ::"r"(count) : "memory");
}

template <int N, int R, int NS, bool INV, int T, int GSTR, bool SD, bool DD, int NT, bool END_SYNC, typename C>
__device__ __forceinline__ void ct_stage_grouped_ip(C* buf, int groups, const C* __restrict__ tw) {
    constexpr int M = N / R;
    constexpr int TWSTEP = N / (NS * R);
    constexpr int PERG = M * T;
    static_assert(PERG <= NT, "the butterflies of one group fit the threads of a pass");
    constexpr int GCH = NT / PERG;
    // the thread index read through a volatile move: the compiler would otherwise hoist every
    // stage's butterfly offsets (loop invariants of a persistent kernel's tile loop) and keep
    // them all live across the loop
    int tid;
    asm volatile("mov.u32 %0, %%tid.x;" : "=r"(tid));
    const int gl = tid / PERG;
    const int rem = tid - gl * PERG;
    const int t = rem % T, j = rem / T;
    const int k = j % NS;
    const int base = (j / NS) * (NS * R) + k;
    for (int g0 = 0; g0 < groups; g0 += GCH) {
        const int ng = groups - g0 < GCH ? groups - g0 : GCH;
        // the warps that hold this chunk's butterflies take part (named barrier among them);
        // their idle lanes transform a copy of the chunk's first group and do not store it
        const int nthr = (ng * PERG + 31) & ~31;
        if (tid < nthr) {
            const bool act = gl < ng;
            const int g = g0 + (act ? gl : 0);
            const int off = g * GSTR + t;
            C v[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int e = j + r * M;
                v[r] = buf[(SD ? e * T : ct_gpos(e, T)) + off];
            }
            if constexpr (NS > 1) {
#pragma unroll
                for (int r = 1; r < R; ++r) {
                    C w = tw[k * r * TWSTEP];
                    if (INV) w.y = -w.y;
                    v[r] = cmul(v[r], w);
                }
            }
            dft_small<R, INV>(v);
            bar_sync_first(nthr);
            if (act) {
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int e = base + r * NS;
                    buf[(DD ? e * T : ct_gpos(e, T)) + off] = v[r];
                }
            }
        }
    }
    if constexpr (END_SYNC) __syncthreads();
}

template <int N, bool INV, int T, int GSTR, bool SD, bool DD, int NT, int S, typename C>
__device__ __forceinline__ void ct_stages_grouped_ip(C* a, int groups, const C* tw) {
    if constexpr (S < ct_nstages(N)) {
        constexpr int R = ct_radix_at(N, S);
        constexpr int NS = ct_ns_at(N, S);
        constexpr bool last = (S + 1 == ct_nstages(N));
        ct_stage_grouped_ip<N, R, NS, INV, T, GSTR, SD && S == 0, DD && last, NT, !last>(a, groups, tw);
        ct_stages_grouped_ip<N, INV, T, GSTR, SD, DD, NT, S + 1>(a, groups, tw);
    }
}

// Transform `groups` tiles held in a, in place; the caller syncs before and after.
template <int N, bool INV, int T, int GSTR, bool SD = false, bool DD = false, int NT = kFftThreads, typename C>
__device__ __forceinline__ void ct_fft_grouped_ip(C* a, int groups, const C* tw) {
    ct_stages_grouped_ip<N, INV, T, GSTR, SD, DD, NT, 0>(a, groups, tw);
}

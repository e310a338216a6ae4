// Register-resident DFTs of the lengths 1, 2, 4, 6, 8, 10, 12 and 16, natural order in and out, fully
// unrolled. 6, 10 and 12 split into coprime factors by the prime-factor map (Good 1958, Thomas 1963:
// no twiddles between the factors); 8 and 16 by one Cooley-Tukey step. Operation counts per complex
// transform: 6: 36 additions + 8 products, 8: 52 + 4, 10: 88 + 24, 12: 96 + 16, 16: 144 + 24.
#pragma once

#include "vie_internal.cuh"

namespace vie {

#define VIE_HD __host__ __device__ __forceinline__

template <class C> VIE_HD C cscale(C a, typename real_of<C>::type s) { return mk(a.x * s, a.y * s); }
// a * (-i) forward, a * i inverse
template <bool FWD, class C> VIE_HD C rot(C a) { return FWD ? mul_mi(a) : mul_i(a); }

template <bool FWD, class C> VIE_HD void dft2(C& a, C& b) {
    const C t = a - b;
    a = a + b;
    b = t;
}

template <bool FWD, class C> VIE_HD void dft3(C& a, C& b, C& c) {
    typedef typename real_of<C>::type R;
    const R h = (R)0.86602540378443864676;               // sin(pi / 3)
    const C s = b + c, d = rot<FWD>(b - c), m = cfmas(s, (R)-0.5, a);
    a = a + s;
    b = cfmas(d, h, m);
    c = cfmas(d, -h, m);
}

template <bool FWD, class C> VIE_HD void dft4(C& a, C& b, C& c, C& d) {
    const C s = a + c, t = a - c, u = b + d, v = rot<FWD>(b - d);
    a = s + u;
    c = s - u;
    b = t + v;
    d = t - v;
}

template <bool FWD, class C> VIE_HD void dft5(C& a, C& b, C& c, C& d, C& e) {
    typedef typename real_of<C>::type R;
    const R c1 = (R)0.30901699437494742410, c2 = (R)-0.80901699437494742410;   // cos(2 pi / 5), cos(4 pi / 5)
    const R s1 = (R)0.95105651629515357212, s2 = (R)0.58778525229247312917;    // sin of the same
    const C p = b + e, q = c + d, u = b - e, v = c - d;
    const C m1 = cfmas(q, c2, cfmas(p, c1, a)), m2 = cfmas(q, c1, cfmas(p, c2, a));
    const C n1 = rot<FWD>(mk(s1 * u.x + s2 * v.x, s1 * u.y + s2 * v.y));
    const C n2 = rot<FWD>(mk(s2 * u.x - s1 * v.x, s2 * u.y - s1 * v.y));
    a = a + p + q;
    b = m1 + n1;
    e = m1 - n1;
    c = m2 + n2;
    d = m2 - n2;
}

template <int H, bool FWD, class C> VIE_HD void dft(C (&a)[H]) {
    typedef typename real_of<C>::type R;
    if constexpr (H == 1) {
    } else if constexpr (H == 2) {
        dft2<FWD>(a[0], a[1]);
    } else if constexpr (H == 4) {
        dft4<FWD>(a[0], a[1], a[2], a[3]);
    } else if constexpr (H == 6 || H == 10 || H == 12) {
        // n = (N2 n1 + N1 n2) mod H in, k = k1 (mod N1), k = k2 (mod N2) out
        constexpr int N1 = H == 12 ? 4 : 2, N2 = H / N1;
        C b[N1][N2];
#pragma unroll
        for (int n1 = 0; n1 < N1; ++n1) {
#pragma unroll
            for (int n2 = 0; n2 < N2; ++n2) b[n1][n2] = a[(N2 * n1 + N1 * n2) % H];
            if constexpr (N2 == 3) dft3<FWD>(b[n1][0], b[n1][1], b[n1][2]);
            else dft5<FWD>(b[n1][0], b[n1][1], b[n1][2], b[n1][3], b[n1][4]);
        }
#pragma unroll
        for (int k2 = 0; k2 < N2; ++k2) {
            if constexpr (N1 == 2) dft2<FWD>(b[0][k2], b[1][k2]);
            else dft4<FWD>(b[0][k2], b[1][k2], b[2][k2], b[3][k2]);
        }
#pragma unroll
        for (int k = 0; k < H; ++k) a[k] = b[k % N1][k % N2];
    } else if constexpr (H == 8) {
        const R r = (R)0.70710678118654752440;
        dft4<FWD>(a[0], a[2], a[4], a[6]);
        dft4<FWD>(a[1], a[3], a[5], a[7]);
        // W_8^k of the odd half: 1, (1 - i) / sqrt 2, -i, -(1 + i) / sqrt 2 (conjugates inverse)
        const C t1 = FWD ? mk(r * (a[3].x + a[3].y), r * (a[3].y - a[3].x)) : mk(r * (a[3].x - a[3].y), r * (a[3].y + a[3].x));
        const C t2 = rot<FWD>(a[5]);
        const C t3 = FWD ? mk(r * (a[7].y - a[7].x), -r * (a[7].x + a[7].y)) : mk(-r * (a[7].x + a[7].y), r * (a[7].x - a[7].y));
        const C e0 = a[0], e1 = a[2], e2 = a[4], e3 = a[6], o0 = a[1];
        a[0] = e0 + o0; a[4] = e0 - o0;
        a[1] = e1 + t1; a[5] = e1 - t1;
        a[2] = e2 + t2; a[6] = e2 - t2;
        a[3] = e3 + t3; a[7] = e3 - t3;
    } else {
        static_assert(H == 16, "dft: no such length");
        const R c = (R)0.92387953251128675613, s = (R)0.38268343236508977173, r = (R)0.70710678118654752440;
#pragma unroll
        for (int n2 = 0; n2 < 4; ++n2) dft4<FWD>(a[n2], a[n2 + 4], a[n2 + 8], a[n2 + 12]);
        // a[n2 + 4 k1] *= W_16^{n2 k1}
        auto tw = [](C v, R wr, R wi) {                   // v * (wr - i wi) forward, v * (wr + i wi) inverse
            return FWD ? mk(v.x * wr + v.y * wi, v.y * wr - v.x * wi) : mk(v.x * wr - v.y * wi, v.y * wr + v.x * wi);
        };
        auto w2 = [r](C v) { return FWD ? mk(r * (v.x + v.y), r * (v.y - v.x)) : mk(r * (v.x - v.y), r * (v.y + v.x)); };
        a[5] = tw(a[5], c, s);
        a[6] = w2(a[6]);
        a[7] = tw(a[7], s, c);
        a[9] = w2(a[9]);
        a[10] = rot<FWD>(a[10]);
        a[11] = rot<FWD>(w2(a[11]));
        a[13] = tw(a[13], s, c);
        a[14] = rot<FWD>(w2(a[14]));
        a[15] = tw(a[15], -c, -s);
#pragma unroll
        for (int k1 = 0; k1 < 4; ++k1) dft4<FWD>(a[4 * k1], a[4 * k1 + 1], a[4 * k1 + 2], a[4 * k1 + 3]);
        // position 4 k1 + k2 holds frequency k1 + 4 k2
#pragma unroll
        for (int k1 = 0; k1 < 4; ++k1)
#pragma unroll
            for (int k2 = k1 + 1; k2 < 4; ++k2) {
                const C t = a[4 * k1 + k2];
                a[4 * k1 + k2] = a[4 * k2 + k1];
                a[4 * k2 + k1] = t;
            }
    }
}

// s += a b, s -= a b, as four fused multiply-adds (the product's own sum first would take six operations)
template <class C> VIE_HD void cmac(C& s, C a, C b) {
    s.x = fma(-a.y, b.y, fma(a.x, b.x, s.x));
    s.y = fma(a.y, b.x, fma(a.x, b.y, s.y));
}
template <class C> VIE_HD void cmacn(C& s, C a, C b) {
    s.x = fma(a.y, b.y, fma(-a.x, b.x, s.x));
    s.y = fma(-a.y, b.x, fma(-a.x, b.y, s.y));
}

// The symmetric 3x3 Green multiply of one frequency with the entries v (xx, xy, xz, yy, yz, zz), the
// frequency being in the upper half of the axis AXIS (0: x, 2: z; the two off-diagonal components odd along
// that axis change sign) when FLIP is set.
template <int AXIS, bool FLIP, class C> VIE_HD void green3(C& X, C& Y, C& Z, const C (&v)[6]) {
    C ox = cmul(v[0], X), oy = cmul(v[3], Y), oz = cmul(v[5], Z);
    auto mac = [](bool neg, C& s, C a, C b) {
        if (neg) cmacn(s, a, b);
        else cmac(s, a, b);
    };
    mac(FLIP && AXIS == 0, ox, v[1], Y);
    mac(FLIP && AXIS == 0, oy, v[1], X);
    mac(FLIP, ox, v[2], Z);
    mac(FLIP, oz, v[2], X);
    mac(FLIP && AXIS == 2, oy, v[4], Z);
    mac(FLIP && AXIS == 2, oz, v[4], Y);
    X = ox;
    Y = oy;
    Z = oz;
}

}  // namespace vie

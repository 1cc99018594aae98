// Exact signs of the orientation and in-circle determinants with fixed-width
// integers, for host and device code.
//
// A few double coordinates whose exponents differ by at most kSpan are
// integers of at most 126 bits on their common grid (the smallest ulp among
// them), so their differences, the 2x2 minors and lifted heights (257 bits)
// and the in-circle determinant (517 bits) are computed without rounding in
// sign-magnitude words: about a hundred 64-bit products and under 1 KB of
// locals.  The floating-point expansions of predicates.cpp hold up to 31 KB
// on the stack, which a GPU would reserve for every resident thread.
// Coordinates spread over more exponents are reported as unknown (the caller
// then leaves the mesh to the host builder).
#pragma once

#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define RICH_HD __host__ __device__
#else
#define RICH_HD
#endif

namespace rich {
namespace exactint {

constexpr int kUnknown = 2;  // the coordinates do not fit the integer grid
constexpr int kSpan = 72;    // exponents a grid covers beyond a mantissa
constexpr int kImageSpan = 68;  // with multiples of a box's sides

template <int N> struct Big {  // s * sum_k w[k] 2^(64 k), s in {-1, 0, 1}
    uint64_t w[N];
    int s;
};

RICH_HD inline uint64_t bits_of(double v)
{
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(v);
#else
    uint64_t b;
    std::memcpy(&b, &v, 8);
    return b;
#endif
}

// 2^k for |k| <= 1022
RICH_HD inline double pow2(int k)
{
    const uint64_t b = (uint64_t)(1023 + k) << 52;
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)b);
#else
    double v;
    std::memcpy(&v, &b, 8);
    return v;
#endif
}

RICH_HD inline uint64_t mul_hi(uint64_t a, uint64_t b)
{
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}

// exponent of a value's last mantissa bit (zero: a large number)
RICH_HD inline int low_exp(double v)
{
    const uint64_t b = bits_of(v);
    const int e = (int)((b >> 52) & 0x7ff);
    if ((b << 1) == 0) return 1 << 20;
    return (e ? e : 1) - 1075;
}

// The common grid of k values: its exponent, or false when they are not
// finite or spread too far.
RICH_HD inline bool grid_of(const double *v, int k, int &E, int span = kSpan)
{
    int lo = 1 << 20, hi = -(1 << 20);
    for (int i = 0; i < k; i++) {
        if (((bits_of(v[i]) >> 52) & 0x7ff) == 0x7ff) return false;
        const int e = low_exp(v[i]);
        if (e == 1 << 20) continue;
        if (e < lo) lo = e;
        if (e > hi) hi = e;
    }
    E = lo == 1 << 20 ? 0 : lo;
    return hi < lo || hi - lo <= span;
}

// a - b + k c on the grid 2^E (|k| <= 8; c counts only where k does)
RICH_HD inline Big<2> diff(double a, double b, int E, int k = 0, double c = 0.0)
{
    uint64_t lo = 0, hi = 0;
    for (int t = 0; t < (k ? 3 : 2); t++) {
        const double v = t == 0 ? a : (t == 1 ? b : c);
        const uint64_t u = bits_of(v);
        if ((u << 1) == 0) continue;
        uint64_t m = u & 0xfffffffffffffull;
        if ((u >> 52) & 0x7ff) m |= 1ull << 52;
        if (t == 2) m *= (uint64_t)(k < 0 ? -k : k);
        const int sh = low_exp(v) - E;  // 0 .. the span
        uint64_t l, h;
        if (sh == 0) { l = m; h = 0; }
        else if (sh < 64) { l = m << sh; h = m >> (64 - sh); }
        else { l = 0; h = m << (sh - 64); }
        const bool neg = ((u >> 63) != 0) != (t == 1 || (t == 2 && k < 0));
        if (neg) {  // two's complement
            l = ~l + 1;
            h = ~h + (l == 0 ? 1 : 0);
        }
        const uint64_t s = lo + l;
        hi += h + (s < lo ? 1 : 0);
        lo = s;
    }
    Big<2> r;
    if (hi >> 63) {
        lo = ~lo + 1;
        hi = ~hi + (lo == 0 ? 1 : 0);
        r.s = -1;
    } else {
        r.s = (lo | hi) ? 1 : 0;
    }
    r.w[0] = lo;
    r.w[1] = hi;
    return r;
}

template <int A, int B> RICH_HD inline Big<A + B> mul(const Big<A> &a, const Big<B> &b)
{
    Big<A + B> r;
    for (int i = 0; i < A + B; i++) r.w[i] = 0;
    r.s = a.s * b.s;
    if (!r.s) return r;
    for (int i = 0; i < A; i++) {
        uint64_t carry = 0;
        for (int j = 0; j < B; j++) {
            uint64_t lo = a.w[i] * b.w[j], hi = mul_hi(a.w[i], b.w[j]);
            uint64_t t = r.w[i + j] + lo;
            hi += t < lo ? 1 : 0;
            t += carry;
            hi += t < carry ? 1 : 0;
            r.w[i + j] = t;
            carry = hi;
        }
        r.w[i + B] = carry;
    }
    return r;
}

// a + sb * b for two numbers of N words (the sum has N + 1)
template <int N> RICH_HD inline Big<N + 1> add(const Big<N> &a, const Big<N> &b, int sb)
{
    Big<N + 1> r;
    const int bs = b.s * sb;
    r.w[N] = 0;
    if (a.s == 0 || bs == 0) {
        r.s = a.s ? a.s : bs;
        for (int i = 0; i < N; i++) r.w[i] = a.s ? a.w[i] : (bs ? b.w[i] : 0);
        return r;
    }
    if (a.s == bs) {
        uint64_t c = 0;
        for (int i = 0; i < N; i++) {
            uint64_t t = a.w[i] + c;
            c = t < c ? 1 : 0;
            t += b.w[i];
            c += t < b.w[i] ? 1 : 0;
            r.w[i] = t;
        }
        r.w[N] = c;
        r.s = a.s;
        return r;
    }
    int cmp = 0;
    for (int i = N - 1; i >= 0 && cmp == 0; i--) cmp = a.w[i] > b.w[i] ? 1 : (a.w[i] < b.w[i] ? -1 : 0);
    uint64_t br = 0;
    for (int i = 0; i < N; i++) {
        const uint64_t p = cmp >= 0 ? a.w[i] : b.w[i], q = cmp >= 0 ? b.w[i] : a.w[i];
        const uint64_t t = p - q;
        const uint64_t nb = (p < q ? 1 : 0) + (t < br ? 1 : 0);
        r.w[i] = t - br;
        br = nb;
    }
    r.s = cmp == 0 ? 0 : (cmp > 0 ? a.s : bs);
    return r;
}

// Sign of (b - a) x (c - a), or kUnknown.
RICH_HD inline int orient_sign(double ax, double ay, double bx, double by, double cx, double cy)
{
    const double v[6] = {ax, ay, bx, by, cx, cy};
    int E;
    if (!grid_of(v, 6, E)) return kUnknown;
    return add(mul(diff(bx, ax, E), diff(cy, ay, E)), mul(diff(by, ay, E), diff(cx, ax, E)), -1).s;
}

// the in-circle determinant of differences from the fourth point
RICH_HD inline int incircle_of(const Big<2> p[3], const Big<2> q[3])
{
    Big<12> sum;
    for (int i = 0; i < 12; i++) sum.w[i] = 0;
    sum.s = 0;
    for (int k = 0; k < 3; k++) {
        const int i = (k + 1) % 3, j = (k + 2) % 3;
        const Big<5> lift = add(mul(p[k], p[k]), mul(q[k], q[k]), 1);
        const Big<5> minor = add(mul(p[i], q[j]), mul(p[j], q[i]), -1);
        const Big<10> t = mul(lift, minor);
        Big<12> w;
        for (int c = 0; c < 10; c++) w.w[c] = t.w[c];
        w.w[10] = w.w[11] = 0;
        w.s = t.s;
        const Big<13> s = add(sum, w, 1);
        for (int c = 0; c < 12; c++) sum.w[c] = s.w[c];
        sum.s = s.s;
    }
    return sum.s;
}

// Sign of the in-circle determinant of counter-clockwise a, b, c against d
// (> 0: d strictly inside), or kUnknown.
RICH_HD inline int incircle_sign(double ax, double ay, double bx, double by, double cx, double cy, double dx,
                                 double dy)
{
    const double v[8] = {ax, ay, bx, by, cx, cy, dx, dy};
    int E;
    if (!grid_of(v, 8, E)) return kUnknown;
    const Big<2> p[3] = {diff(ax, dx, E), diff(bx, dx, E), diff(cx, dx, E)};
    const Big<2> q[3] = {diff(ay, dy, E), diff(by, dy, E), diff(cy, dy, E)};
    return incircle_of(p, q);
}

// Points of a periodic plane: cell positions x, y and shifts by kx, ky box
// sides Lx, Ly, taken exactly.  (The coordinates of an image in floating point
// are rounded, differently in each copy of the same four points.)
struct Images {
    double x[4], y[4], Lx, Ly;
    int8_t kx[4], ky[4];  // -2 .. 2
    RICH_HD bool grid(int &E) const
    {
        double v[10];
        for (int k = 0; k < 4; k++) {
            v[2 * k] = x[k];
            v[2 * k + 1] = y[k];
        }
        v[8] = Lx;
        v[9] = Ly;
        return grid_of(v, 10, E, kImageSpan);
    }
    RICH_HD Big<2> dx(int a, int b, int E) const { return diff(x[a], x[b], E, kx[a] - kx[b], Lx); }
    RICH_HD Big<2> dy(int a, int b, int E) const { return diff(y[a], y[b], E, ky[a] - ky[b], Ly); }
    RICH_HD int orient(int a, int b, int c, int E) const
    {
        return add(mul(dx(b, a, E), dy(c, a, E)), mul(dy(b, a, E), dx(c, a, E)), -1).s;
    }
};

// Orientation of its first three points, or kUnknown.
RICH_HD inline int orient_images(const Images &m)
{
    int E;
    return m.grid(E) ? m.orient(0, 1, 2, E) : kUnknown;
}

// In-circle of its counter-clockwise first three points against the fourth
// (> 0: inside) with the symbolic tie-break of predicates.h, or kUnknown.
RICH_HD inline int incircle_images(const Images &m)
{
    int E;
    if (!m.grid(E)) return kUnknown;
    {
        const Big<2> p[3] = {m.dx(0, 3, E), m.dx(1, 3, E), m.dx(2, 3, E)};
        const Big<2> q[3] = {m.dy(0, 3, E), m.dy(1, 3, E), m.dy(2, 3, E)};
        const int s = incircle_of(p, q);
        if (s) return s;
    }
    int k = 0;  // the lexicographically smallest
    for (int c = 1; c < 4; c++) {
        const int sx = m.dx(c, k, E).s;
        if (sx < 0 || (sx == 0 && m.dy(c, k, E).s < 0)) k = c;
    }
    switch (k) {
    case 0: return m.orient(1, 2, 3, E);
    case 1: return -m.orient(0, 2, 3, E);
    case 2: return m.orient(0, 1, 3, E);
    default: return -m.orient(0, 1, 2, E);
    }
}

}  // namespace exactint
}  // namespace rich

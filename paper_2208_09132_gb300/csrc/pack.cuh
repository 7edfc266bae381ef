// pack.cuh -- four velocities of one place (a chunk) as packed pairs.
//
// The FP32 sweeps are bound by instruction issue before HBM; sm_103a issues
// one instruction for two FP32 operations on a register pair (add / mul /
// fma .f32x2, each rounded like the scalar operation).  Pk<float> keeps a
// chunk as two such pairs; Pk<double> is four plain values.
#pragma once

#include "kernels.cuh"

namespace cdg {

template <typename T> struct Pk;

template <>
struct alignas(16) Pk<float> {
    unsigned long long p[2];
    static __device__ __forceinline__ unsigned long long pair(float a, float b) {
        unsigned long long r;
        asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
        return r;
    }
    static __device__ __forceinline__ Pk bc(float x) {
        Pk r;
        r.p[0] = r.p[1] = pair(x, x);
        return r;
    }
    static __device__ __forceinline__ Pk of(const float (&x)[VC]) {
        Pk r;
        r.p[0] = pair(x[0], x[1]);
        r.p[1] = pair(x[2], x[3]);
        return r;
    }
    __device__ __forceinline__ void get(float (&x)[VC]) const {
        asm("mov.b64 {%0, %1}, %2;" : "=f"(x[0]), "=f"(x[1]) : "l"(p[0]));
        asm("mov.b64 {%0, %1}, %2;" : "=f"(x[2]), "=f"(x[3]) : "l"(p[1]));
    }
};
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ unsigned long long sub2(unsigned long long a, unsigned long long b) {
    unsigned long long r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b) {
    unsigned long long r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ Pk<float> operator+(const Pk<float>& a, const Pk<float>& b) {
    return {{add2(a.p[0], b.p[0]), add2(a.p[1], b.p[1])}};
}
__device__ __forceinline__ Pk<float> operator-(const Pk<float>& a, const Pk<float>& b) {
    return {{sub2(a.p[0], b.p[0]), sub2(a.p[1], b.p[1])}};
}
__device__ __forceinline__ Pk<float> operator*(const Pk<float>& a, const Pk<float>& b) {
    return {{mul2(a.p[0], b.p[0]), mul2(a.p[1], b.p[1])}};
}
__device__ __forceinline__ Pk<float> fma4(const Pk<float>& a, const Pk<float>& b, const Pk<float>& c) {
    return {{fma2(a.p[0], b.p[0], c.p[0]), fma2(a.p[1], b.p[1], c.p[1])}};
}
// the sum of the four values: (0 + 2) + (1 + 3)
__device__ __forceinline__ float sum4(const Pk<float>& a) {
    float x, y;
    const unsigned long long s = add2(a.p[0], a.p[1]);
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(s));
    return Ar<float>::add(x, y);
}
// sum of a_v b_v, the pairs' products chained by fma
__device__ __forceinline__ float dot4(const Pk<float>& a, const Pk<float>& b) {
    float x, y;
    const unsigned long long s = fma2(a.p[1], b.p[1], mul2(a.p[0], b.p[0]));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(s));
    return Ar<float>::add(x, y);
}

template <>
struct alignas(16) Pk<double> {
    double v[VC];
    static __device__ __forceinline__ Pk bc(double x) { return {{x, x, x, x}}; }
    static __device__ __forceinline__ Pk of(const double (&x)[VC]) { return {{x[0], x[1], x[2], x[3]}}; }
    __device__ __forceinline__ void get(double (&x)[VC]) const {
#pragma unroll
        for (int i = 0; i < VC; ++i) x[i] = v[i];
    }
};
__device__ __forceinline__ Pk<double> operator+(const Pk<double>& a, const Pk<double>& b) {
    Pk<double> r;
#pragma unroll
    for (int i = 0; i < VC; ++i) r.v[i] = __dadd_rn(a.v[i], b.v[i]);
    return r;
}
__device__ __forceinline__ Pk<double> operator-(const Pk<double>& a, const Pk<double>& b) {
    Pk<double> r;
#pragma unroll
    for (int i = 0; i < VC; ++i) r.v[i] = __dsub_rn(a.v[i], b.v[i]);
    return r;
}
__device__ __forceinline__ Pk<double> operator*(const Pk<double>& a, const Pk<double>& b) {
    Pk<double> r;
#pragma unroll
    for (int i = 0; i < VC; ++i) r.v[i] = __dmul_rn(a.v[i], b.v[i]);
    return r;
}
__device__ __forceinline__ Pk<double> fma4(const Pk<double>& a, const Pk<double>& b, const Pk<double>& c) {
    Pk<double> r;
#pragma unroll
    for (int i = 0; i < VC; ++i) r.v[i] = __fma_rn(a.v[i], b.v[i], c.v[i]);
    return r;
}
__device__ __forceinline__ double sum4(const Pk<double>& a) {
    return __dadd_rn(__dadd_rn(a.v[0], a.v[2]), __dadd_rn(a.v[1], a.v[3]));
}
__device__ __forceinline__ double dot4(const Pk<double>& a, const Pk<double>& b) {
    return __dadd_rn(__fma_rn(a.v[2], b.v[2], __dmul_rn(a.v[0], b.v[0])),
                     __fma_rn(a.v[3], b.v[3], __dmul_rn(a.v[1], b.v[1])));
}

// One cell's chunk of the state or of a face array (g then b, 32 B in FP32, one
// sector): whole-sector 256-bit accesses.  NC as in Chunk.
template <bool NC>
__device__ __forceinline__ void ld256(const void* p, unsigned long long (&x)[4]) {
    if constexpr (NC)
        asm volatile("ld.global.nc.v4.b64 {%0, %1, %2, %3}, [%4];"
                     : "=l"(x[0]), "=l"(x[1]), "=l"(x[2]), "=l"(x[3])
                     : "l"(p));
    else
        asm volatile("ld.global.v4.b64 {%0, %1, %2, %3}, [%4];"
                     : "=l"(x[0]), "=l"(x[1]), "=l"(x[2]), "=l"(x[3])
                     : "l"(p)
                     : "memory");
}
__device__ __forceinline__ void st256(void* p, unsigned long long a, unsigned long long b, unsigned long long c,
                                      unsigned long long d) {
    asm volatile("st.global.v4.b64 [%0], {%1, %2, %3, %4};" ::"l"(p), "l"(a), "l"(b), "l"(c), "l"(d) : "memory");
}
template <bool NC>
__device__ __forceinline__ void load_gb(const float* p, Pk<float>& g, Pk<float>& b) {
    unsigned long long x[4];
    ld256<NC>(p, x);
    g.p[0] = x[0]; g.p[1] = x[1]; b.p[0] = x[2]; b.p[1] = x[3];
}
template <bool NC>
__device__ __forceinline__ void load_gb(const double* p, Pk<double>& g, Pk<double>& b) {
    unsigned long long x[4], y[4];
    ld256<NC>(p, x);
    ld256<NC>(p + VC, y);
#pragma unroll
    for (int i = 0; i < VC; ++i) {
        g.v[i] = __longlong_as_double((long long)x[i]);
        b.v[i] = __longlong_as_double((long long)y[i]);
    }
}
__device__ __forceinline__ void store_gb(float* p, const Pk<float>& g, const Pk<float>& b) {
    st256(p, g.p[0], g.p[1], b.p[0], b.p[1]);
}
__device__ __forceinline__ void store_gb(double* p, const Pk<double>& g, const Pk<double>& b) {
    unsigned long long x[VC], y[VC];
#pragma unroll
    for (int i = 0; i < VC; ++i) {
        x[i] = (unsigned long long)__double_as_longlong(g.v[i]);
        y[i] = (unsigned long long)__double_as_longlong(b.v[i]);
    }
    st256(p, x[0], x[1], x[2], x[3]);
    st256(p + VC, y[0], y[1], y[2], y[3]);
}
// 16-byte-aligned read-only loads of a chunk-wide vector
__device__ __forceinline__ Pk<float> ldg4(const float* p) {
    const ulonglong2 a = __ldg(reinterpret_cast<const ulonglong2*>(p));
    return {{a.x, a.y}};
}
__device__ __forceinline__ Pk<double> ldg4(const double* p) {
    const double2 a = __ldg(reinterpret_cast<const double2*>(p)), b = __ldg(reinterpret_cast<const double2*>(p + 2));
    return {{a.x, a.y, b.x, b.y}};
}

// The van Leer limiter of the sweeps with upwind owners.  FP64: the quotient p / s
// for p > 0 by residual correction with one FMA (P. Markstein, IBM J. Res. Dev. 34
// (1990) 111): with an approximate reciprocal y of s and q = p y, twice
// q <- q + (p - s q) y.  y is the FP32 reciprocal of the leading 24 bits of s (an
// error of at most 2^-23 for the rest of s, 2^-23 for the 1 ulp of the instruction)
// with the exponent of s put back, so a correction takes a relative error e to
// 2^-22 e: 2^-22, 2^-44, 2^-66, each but the last beside its rounding of 2^-53.  The
// result is the rounding of a value within 2^-65 of the quotient, off by at most
// (1/2 + 2^-12) ulp: the correctly rounded quotient, or its neighbour where the
// quotient lies within 2^-12 ulp of the middle between the two.  That takes products
// whose residuals do not underflow and an s whose reciprocal is normal; all others
// are divided.  Five operations of the FP64 pipe, which bounds sweep A in FP64, instead of
// the divide's, and none where no lane's differences share a sign (flat flows):
// sweep A at 256 x 256 cells x 32 x 32 velocities 8.67 ms, with the divide 10.64; 1D 8192 x
// 129 0.152 with either.  (k_sweep and k_shslope keep the divide.)
__device__ __forceinline__ float vanleer1(float s1, float s2) { return Num<float>::vanleer(s1, s2); }
static __device__ __noinline__ double vanleer_divide(double p, double s) { return p / s; }
__device__ __forceinline__ double vanleer1(double s1, double s2) {
    const double p = s1 * s2, s = s1 + s2;
    const unsigned hp = (unsigned)__double2hiint(p), hs = (unsigned)__double2hiint(s), ls = (unsigned)__double2loint(s);
    const unsigned es = hs & 0x7ff00000u;
    double q = 0.0;
    if (hp - 0x01700000u < 0x7e800000u && es < 0x7fc00000u) {       // 2^-1000 <= p < infinity, |s| < 2^1021
        const unsigned r = __float_as_uint(Num<float>::rcp(__uint_as_float(0x3f800000u | (hs & 0xfffffu) << 3 | ls >> 29)));
        // its exponent from FP32's bias to FP64's, less that of s
        const double y = __hiloint2double((int)(((r >> 3) + 0x77f00000u - es) | (hs & 0x80000000u)), (int)(r << 29));
        q = p * y;
        q = __fma_rn(__fma_rn(-s, q, p), y, q);
        q = __fma_rn(__fma_rn(-s, q, p), y, q);
    } else if (hp < 0x7ff00001u && (hp | (unsigned)__double2loint(p)) != 0u) {   // positive all the same
        q = vanleer_divide(p, s);
    }
    return q;
}
// Half van Leer slope times dx of four velocities: s1 s2 / (s1 + s2) where the
// one-sided differences share a sign, else 0 (eq. VanLeer).
__device__ __forceinline__ Pk<float> vanleer4(const Pk<float>& s1, const Pk<float>& s2) {
    const Pk<float> p = s1 * s2, s = s1 + s2;
    float pv[VC], sv[VC];
    s.get(sv);
    p.get(pv);
#pragma unroll
    for (int i = 0; i < VC; ++i) sv[i] = Num<float>::rcp(sv[i]);
    const Pk<float> q = p * Pk<float>::of(sv);
    float qv[VC];
    q.get(qv);
#pragma unroll
    for (int i = 0; i < VC; ++i) qv[i] = pv[i] > 0.f ? qv[i] : 0.f;
    return Pk<float>::of(qv);
}
__device__ __forceinline__ Pk<double> vanleer4(const Pk<double>& s1, const Pk<double>& s2) {
    Pk<double> r;
#pragma unroll
    for (int i = 0; i < VC; ++i) r.v[i] = vanleer1(s1.v[i], s2.v[i]);
    return r;
}
template <typename T>
__device__ __forceinline__ Pk<T> expo4(const Pk<T>& x) {
    T v[VC];
    x.get(v);
#pragma unroll
    for (int i = 0; i < VC; ++i) v[i] = Num<T>::expo(v[i]);
    return Pk<T>::of(v);
}

// The equilibria of a chunk's velocities xi (hx = |xi|^2 / 2) at a place with
// the constants c: u (D), cexp, pref, eb, hu2, three more, with SK sq (D) and
// e2.  hL as in shakhov_point.  One exponential per velocity: a chunk's four
// values by the recurrence of equally spaced nodes from the first would take two
// exponentials (FP64 1D, 8192 x 129: a step 0.325 ms instead of 0.372), but lose
// what it climbs, exp(dxi^2 / RT): 1e-9 of the largest value at nodes four
// thermal widths apart, all digits from six on.
template <typename T, int D, bool SK>
__device__ __forceinline__ void eq4(const T* c, const Pk<T>* xi, const Pk<T>& hx, T hL, Pk<T>& ge, Pk<T>& be) {
    using K = Pk<T>;
    K c2, cq;
#pragma unroll
    for (int a = 0; a < D; ++a) {
        const K d = xi[a] - K::bc(c[a]);
        c2 = a == 0 ? d * d : fma4(d, d, c2);
        if constexpr (SK) cq = a == 0 ? K::bc(c[D + 7]) * d : fma4(K::bc(c[D + 7 + a]), d, cq);
    }
    const K gM = K::bc(c[D + 1]) * expo4<T>(K::bc(c[D]) * c2);
    if constexpr (SK) {              // as shakhov_point
        const K P1 = fma4(c2, K::bc(c[D] * Num<T>::irt_scale()), K::bc(T(-(D + 2))));
        const K in = fma4(hx, P1, fma4(K::bc(hL), c2, K::bc(-c[2 * D + 7])));
        be = gM * fma4(cq, in, hx + K::bc(c[D + 2]));
        ge = fma4(gM * cq, P1, gM);
    } else {
        ge = gM;
        be = (hx + K::bc(c[D + 2])) * gM;
    }
}
// How many values those constants are.
template <typename T, int D, bool SK>
struct EqPack {
    static constexpr int N = D + 7 + (SK ? D + 1 : 0);
    static constexpr int NV = (N + 3) / 4;
};

// Keeps a loop constant in its register (the compiler would convert it from
// double again in every iteration, on the FP64 pipe).
__device__ __forceinline__ void keep(float& x) { asm volatile("" : "+f"(x)); }
__device__ __forceinline__ void keep(double& x) { asm volatile("" : "+d"(x)); }
__device__ __forceinline__ void keep(int& x) { asm volatile("" : "+r"(x)); }

// N running sums: Kahan pairs in FP32 (folded two at a time), plain in FP64.
template <typename T, int N> struct Sums;
template <int N>
struct Sums<float, N> {
    static constexpr int M = (N + 1) / 2;
    unsigned long long s[M], c[M];
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int i = 0; i < M; ++i) s[i] = c[i] = 0ull;
    }
    // add x[k] to sum k; called as the values [k0, k1) become known (k0, k1
    // compile-time constants after unrolling): a pair is folded once it is complete
    __device__ __forceinline__ void add(const float (&x)[N], int k0, int k1) {
#pragma unroll
        for (int i = 0; i < M; ++i) {
            const int top = 2 * i + 1 < N ? 2 * i + 1 : 2 * i;
            if (top < k0 || top >= k1) continue;
            const unsigned long long y = sub2(Pk<float>::pair(x[2 * i], top > 2 * i ? x[top] : 0.f), c[i]);
            const unsigned long long t = add2(s[i], y);
            c[i] = sub2(sub2(t, s[i]), y);
            s[i] = t;
        }
    }
    __device__ __forceinline__ double value(int k) const {      // k a compile-time constant after unrolling
        float s0, s1, c0, c1;
        asm("mov.b64 {%0, %1}, %2;" : "=f"(s0), "=f"(s1) : "l"(s[k / 2]));
        asm("mov.b64 {%0, %1}, %2;" : "=f"(c0), "=f"(c1) : "l"(c[k / 2]));
        return k % 2 ? (double)s1 - (double)c1 : (double)s0 - (double)c0;
    }
};
template <int N>
struct Sums<double, N> {
    double s[N];
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int i = 0; i < N; ++i) s[i] = 0.0;
    }
    __device__ __forceinline__ void add(const double (&x)[N], int k0, int k1) {
#pragma unroll
        for (int i = 0; i < N; ++i)
            if (i >= k0 && i < k1) s[i] = __dadd_rn(s[i], x[i]);
    }
    __device__ __forceinline__ double value(int k) const { return s[k]; }
};

}  // namespace cdg

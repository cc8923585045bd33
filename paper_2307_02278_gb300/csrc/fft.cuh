// Mesh-stage device code shared by the operator kernels (kernels_mesh.cu) and
// the compile-time FFT passes (fft_sizes_*.cu): vector loads, complex
// arithmetic, the in-register DFTs, the Stockham passes with compile-time
// mesh size, and the spreading fused with the first forward pass.
#pragma once

#include <algorithm>
#include <atomic>

#include "mbd_internal.cuh"

namespace mbd {

template <class T> struct FFTArgs {
    typename Cplx<T>::type *data;   // complex view of the mesh
    const typename Cplx<T>::type *tw;   // exp(-2 pi i n / K), n = 0..K-1
    const T *G;          // influence function (fused pass only)
    int K;
    int inner;           // complex elements per row (contiguous)
    int W;               // tile width (complex columns)
    int nst;
    unsigned long long radices;   // stage s radix = (radices >> 4 s) & 15
    int V;               // complex probe pairs per mesh point (fused pass: G index = e / V)
    int early;           // compile-time passes: programmatic dependent launch (1; 2: of every double pass too) or plain (0)
    int sms;             // multiprocessors
};

// Compile-time passes for the smooth sizes listed below (fft_sizes_*.cu) over
// [outer][K][inner]; mode 0 forward, 1 inverse, 2 forward x G inverse (outer =
// 1).  Return 1 when launched, 0 when the launch could not be configured, -1
// when there is no compile-time pass for the size.
//   a.W: the tile width in complex columns of float passes, 32 or 16 (double
//   passes have one width).
template <class T> int launch_fft_ct_sized(const FFTArgs<T> &a, int mode, unsigned outer, cudaStream_t st);
bool fft_ct_size(int K);

// Arguments of the spreading by pencil records (PencilRec) into the mesh.
template <class T> struct SpreadArgs {
    const T *d;          // dipoles [N][3][ld]
    T *mesh;             // [K1][K2][K3][ld]
    int R, ld;           // probes (the rest of ld is written as zero)
    int K1, K2, K3, p;
    const int *prow;     // [K1 K2 K3 + 1] records by point (k1, k2, top3)
    const PencilRec<T> *prec;
    const T *k3w;        // [N][2p] M3, M3'
    const typename Cplx<T>::type *tw;   // twiddles of k3
    int sms;             // multiprocessors
};
// Spreading fused with the forward transform along k3; same return values.
template <class T> int launch_spp_sized(const SpreadArgs<T> &a, cudaStream_t st);

// Sizes with a compile-time pass and their radices (first stage first), in
// groups of one translation unit each.  The largest radix comes last: the last
// stage has no twiddles to multiply by, and the stages before it keep more
// threads busy.  us per pass (mean of the four of a convolution), largest first
// and largest last: 192^3 x 64 probes 661 and 640, 162^3 x 16 122 and 107, 75^3 x 32
// 24.2 and 20.5, 60^3 x 64 17.6 and 16.8, 40^3 x 16 in double 35.3 and 32.1; spreading
// with its k3 transform at 180^3 x 64 793 and 708.  45, 72, 80, 108 and 150 are
// the other way round: in double 72^3 x 16 takes 166 and 173, the spreading at 45^3 x 8 49 and
// 55; the others differ by less than 1 %, in favour of this order.
#define MBD_FFT_GROUP0(X) X(16, 4, 4) X(18, 3, 6) X(20, 4, 5) X(24, 4, 6) X(25, 5, 5) X(27, 3, 9) X(30, 5, 6)
#define MBD_FFT_GROUP1(X) X(32, 4, 8) X(36, 6, 6) X(40, 5, 8) X(45, 9, 5) X(48, 6, 8) X(50, 5, 10) X(54, 6, 9)
#define MBD_FFT_GROUP2(X) X(60, 6, 10) X(64, 8, 8) X(72, 9, 8) X(75, 5, 15) X(80, 10, 8) X(81, 9, 9) X(90, 9, 10)
#define MBD_FFT_GROUP3(X) X(96, 8, 12) X(100, 10, 10) X(108, 12, 9) X(120, 10, 12) X(125, 5, 5, 5) X(128, 8, 16) \
    X(135, 9, 15)
#define MBD_FFT_GROUP4(X) X(144, 12, 12) X(150, 15, 10) X(160, 10, 16) X(162, 3, 6, 9) X(180, 12, 15) \
    X(192, 12, 16) X(200, 4, 5, 10)
#define MBD_FFT_GROUP5(X) X(216, 6, 6, 6) X(225, 15, 15) X(240, 15, 16) X(243, 3, 9, 9) X(250, 5, 5, 10) \
    X(256, 16, 16)
#define MBD_FFT_NUM_GROUPS 6

template <class T> int launch_fft_ct_group0(const FFTArgs<T> &, int, unsigned, cudaStream_t);
template <class T> int launch_fft_ct_group1(const FFTArgs<T> &, int, unsigned, cudaStream_t);
template <class T> int launch_fft_ct_group2(const FFTArgs<T> &, int, unsigned, cudaStream_t);
template <class T> int launch_fft_ct_group3(const FFTArgs<T> &, int, unsigned, cudaStream_t);
template <class T> int launch_fft_ct_group4(const FFTArgs<T> &, int, unsigned, cudaStream_t);
template <class T> int launch_fft_ct_group5(const FFTArgs<T> &, int, unsigned, cudaStream_t);
template <class T> int launch_spp_group0(const SpreadArgs<T> &, cudaStream_t);
template <class T> int launch_spp_group1(const SpreadArgs<T> &, cudaStream_t);
template <class T> int launch_spp_group2(const SpreadArgs<T> &, cudaStream_t);
template <class T> int launch_spp_group3(const SpreadArgs<T> &, cudaStream_t);
template <class T> int launch_spp_group4(const SpreadArgs<T> &, cudaStream_t);
template <class T> int launch_spp_group5(const SpreadArgs<T> &, cudaStream_t);

namespace {

// Vector loads/stores of VEC consecutive values (VEC in {1, 2, 4}).
template <class T, int VEC> struct VecT;
template <> struct VecT<float, 2> { using type = float2; };
template <> struct VecT<float, 4> { using type = float4; };
template <> struct VecT<double, 1> { using type = double; };
template <> struct VecT<double, 2> { using type = double2; };

template <class T, int VEC> __device__ __forceinline__ void vload(const T *p, T *v) {
    if constexpr (VEC == 4 && sizeof(T) == 8) {
        const double2 a = reinterpret_cast<const double2 *>(p)[0], b = reinterpret_cast<const double2 *>(p)[1];
        v[0] = a.x;
        v[1] = a.y;
        v[2] = b.x;
        v[3] = b.y;
        return;
    } else {
    using V = typename VecT<T, VEC>::type;
    const V x = *reinterpret_cast<const V *>(p);
    if constexpr (VEC == 1) {
        v[0] = x;
    } else if constexpr (VEC == 2) {
        v[0] = x.x;
        v[1] = x.y;
    } else {
        v[0] = x.x;
        v[1] = x.y;
        v[2] = x.z;
        v[3] = x.w;
    }
    }
}
template <class T, int VEC> __device__ __forceinline__ void vstore(T *p, const T *v) {
    if constexpr (VEC == 4 && sizeof(T) == 8) {
        reinterpret_cast<double2 *>(p)[0] = make_double2(v[0], v[1]);
        reinterpret_cast<double2 *>(p)[1] = make_double2(v[2], v[3]);
        return;
    } else {
    using V = typename VecT<T, VEC>::type;
    V x;
    if constexpr (VEC == 1) {
        x = v[0];
    } else if constexpr (VEC == 2) {
        x.x = v[0];
        x.y = v[1];
    } else {
        x.x = v[0];
        x.y = v[1];
        x.z = v[2];
        x.w = v[3];
    }
    *reinterpret_cast<V *>(p) = x;
    }
}

// ---------------------------------------------------------------- FFT
// Complex values Cx<F>: F = double holds one complex probe pair, F = float2 two of
// them, (x0, x1) in x and (y0, y1) in y, on which every
// operation is one packed instruction (add, multiply, FMA of two floats).
// FP32 meshes hold a multiple of four probes per point, and four consecutive
// probes p0 .. p3 are read as the two complex pairs p0 + i p2 and p1 + i p3,
// which needs no shuffle and half the FP32 instructions of the scalar form.
// Any pairing of the probes gives the same convolution (the influence function
// is real and even); every pass of one mesh uses the same pairing.
template <class F> struct __align__(2 * sizeof(F)) Cx {
    F x, y;
};
// The packed form of a real type's columns.
template <class T> struct PackOf { using type = T; };
template <> struct PackOf<float> { using type = float2; };
template <class F> struct Scal { using type = F; };
template <> struct Scal<float2> { using type = float; };

__device__ __forceinline__ double fadd(double a, double b) { return a + b; }
__device__ __forceinline__ float2 fadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ double fsub(double a, double b) { return a - b; }
__device__ __forceinline__ float2 fsub(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ double fmulc(double a, double c) { return a * c; }
__device__ __forceinline__ float2 fmulc(float2 a, float c) { return __fmul2_rn(a, make_float2(c, c)); }
// a c + b with a scalar c
__device__ __forceinline__ double fmac(double a, double c, double b) { return fma(a, c, b); }
__device__ __forceinline__ float2 fmac(float2 a, float c, float2 b) { return __ffma2_rn(a, make_float2(c, c), b); }

template <class F> __device__ __forceinline__ Cx<F> cadd(Cx<F> a, Cx<F> b) { return {fadd(a.x, b.x), fadd(a.y, b.y)}; }
template <class F> __device__ __forceinline__ Cx<F> csub(Cx<F> a, Cx<F> b) { return {fsub(a.x, b.x), fsub(a.y, b.y)}; }
// a + s i b and a - s i b, s = -1 (forward transforms) or +1 (INV)
template <bool INV, class F> __device__ __forceinline__ Cx<F> cadd_i(Cx<F> a, Cx<F> b) {
    if constexpr (INV) return {fsub(a.x, b.y), fadd(a.y, b.x)};
    else return {fadd(a.x, b.y), fsub(a.y, b.x)};
}
template <bool INV, class F> __device__ __forceinline__ Cx<F> csub_i(Cx<F> a, Cx<F> b) { return cadd_i<!INV>(a, b); }
// a c + b, a scalar c; and b + s i c a
template <class F, class S> __device__ __forceinline__ Cx<F> cfma(Cx<F> a, S c, Cx<F> b) {
    return {fmac(a.x, c, b.x), fmac(a.y, c, b.y)};
}
template <bool INV, class F, class S> __device__ __forceinline__ Cx<F> cfma_i(Cx<F> a, S c, Cx<F> b) {
    const S d = INV ? c : -c;
    return {fmac(a.y, -d, b.x), fmac(a.x, d, b.y)};
}
// a (c + s i t) for constants c, t (the twiddle exp(s i angle) with c = cos, t = sin)
template <bool INV, class F, class S> __device__ __forceinline__ Cx<F> crot(Cx<F> a, S c, S t) {
    const S d = INV ? t : -t;
    return {fmac(a.y, -d, fmulc(a.x, c)), fmac(a.x, d, fmulc(a.y, c))};
}

// In-register R-point DFTs  X_t = sum_q x_q exp(s 2 pi i q t / R), natural
// order in and out.
template <class F, int R, bool INV> struct Dft;
template <class F, bool INV> struct Dft<F, 2, INV> {
    static __device__ __forceinline__ void run(Cx<F> *v) {
        const Cx<F> a = v[0], b = v[1];
        v[0] = cadd(a, b);
        v[1] = csub(a, b);
    }
};
template <class F, bool INV> struct Dft<F, 3, INV> {
    static __device__ __forceinline__ void run(Cx<F> *v) {
        using S = typename Scal<F>::type;
        const Cx<F> t = cadd(v[1], v[2]), u = csub(v[1], v[2]);
        const Cx<F> m = cfma(t, S(-0.5), v[0]);
        v[0] = cadd(v[0], t);
        v[1] = cfma_i<INV>(u, S(0.86602540378443864676), m);
        v[2] = cfma_i<!INV>(u, S(0.86602540378443864676), m);
    }
};
template <class F, bool INV> struct Dft<F, 4, INV> {
    static __device__ __forceinline__ void run(Cx<F> *v) {
        const Cx<F> s02 = cadd(v[0], v[2]), d02 = csub(v[0], v[2]);
        const Cx<F> s13 = cadd(v[1], v[3]), d13 = csub(v[1], v[3]);
        v[0] = cadd(s02, s13);
        v[2] = csub(s02, s13);
        v[1] = cadd_i<INV>(d02, d13);
        v[3] = csub_i<INV>(d02, d13);
    }
};
template <class F, bool INV> struct Dft<F, 5, INV> {
    static __device__ __forceinline__ void run(Cx<F> *v) {
        using S = typename Scal<F>::type;
        // cos and sin of 2 pi / 5 and 4 pi / 5
        const S c1 = S(0.30901699437494742410), c2 = S(-0.80901699437494742410);
        const S s1 = S(0.95105651629515357212), s2 = S(0.58778525229247312917);
        const Cx<F> a = v[0];
        const Cx<F> t1 = cadd(v[1], v[4]), t2 = cadd(v[2], v[3]);
        const Cx<F> u1 = csub(v[1], v[4]), u2 = csub(v[2], v[3]);
        v[0] = cadd(cadd(a, t1), t2);
        const Cx<F> m1 = cfma(t2, c2, cfma(t1, c1, a)), m2 = cfma(t2, c1, cfma(t1, c2, a));
        v[1] = cfma_i<INV>(u2, s2, cfma_i<INV>(u1, s1, m1));
        v[4] = cfma_i<!INV>(u2, s2, cfma_i<!INV>(u1, s1, m1));
        v[2] = cfma_i<!INV>(u2, s1, cfma_i<INV>(u1, s2, m2));
        v[3] = cfma_i<INV>(u2, s1, cfma_i<!INV>(u1, s2, m2));
    }
};
template <class F, bool INV> struct Dft<F, 8, INV> {
    static __device__ __forceinline__ void run(Cx<F> *v) {
        using S = typename Scal<F>::type;
        const S h = S(0.70710678118654752440);
        Cx<F> e[4] = {v[0], v[2], v[4], v[6]};
        Cx<F> o[4] = {v[1], v[3], v[5], v[7]};
        Dft<F, 4, INV>::run(e);
        Dft<F, 4, INV>::run(o);
        // odd outputs times exp(s 2 pi i t / 8) = h (1 + s i), s i, h (-1 + s i)
        const Cx<F> p1 = cadd_i<INV>(o[1], o[1]), p3 = csub_i<INV>(o[3], o[3]);
        v[0] = cadd(e[0], o[0]);
        v[4] = csub(e[0], o[0]);
        v[1] = cfma(p1, h, e[1]);
        v[5] = cfma(p1, -h, e[1]);
        v[2] = cadd_i<INV>(e[2], o[2]);
        v[6] = csub_i<INV>(e[2], o[2]);
        v[3] = cfma(p3, -h, e[3]);
        v[7] = cfma(p3, h, e[3]);
    }
};
// R = A B with A, B coprime: two dimensions of DFTs and no twiddles.  Input
// n = (B a + A b) mod R, output k with k mod A = ka and k mod B = kb.
template <class F, int A, int B, bool INV> struct DftCoprime {
    static constexpr int out(int ka, int kb) {
        for (int k = 0; k < A * B; ++k)
            if (k % A == ka && k % B == kb) return k;
        return 0;
    }
    static __device__ __forceinline__ void run(Cx<F> *v) {
        Cx<F> t[A * B];
#pragma unroll
        for (int b = 0; b < B; ++b) {
            Cx<F> u[A];
#pragma unroll
            for (int a = 0; a < A; ++a) u[a] = v[(B * a + A * b) % (A * B)];
            Dft<F, A, INV>::run(u);
#pragma unroll
            for (int a = 0; a < A; ++a) t[a * B + b] = u[a];
        }
#pragma unroll
        for (int a = 0; a < A; ++a) {
            Dft<F, B, INV>::run(t + a * B);
#pragma unroll
            for (int b = 0; b < B; ++b) v[out(a, b)] = t[a * B + b];
        }
    }
};
template <class F, bool INV> struct Dft<F, 6, INV> : DftCoprime<F, 2, 3, INV> {};
template <class F, bool INV> struct Dft<F, 10, INV> : DftCoprime<F, 2, 5, INV> {};
template <class F, bool INV> struct Dft<F, 12, INV> : DftCoprime<F, 4, 3, INV> {};
template <class F, bool INV> struct Dft<F, 15, INV> : DftCoprime<F, 3, 5, INV> {};
// 9 = 3 x 3 and 16 = 4 x 4: x[B a + b] -> DFT over a, twiddle exp(s 2 pi i b ka / R), DFT over b -> k = ka + A kb
template <class F, bool INV> struct Dft<F, 9, INV> {
    static __device__ __forceinline__ void run(Cx<F> *v) {
        using S = typename Scal<F>::type;
        Cx<F> t[3][3];
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            Cx<F> u[3] = {v[b], v[3 + b], v[6 + b]};
            Dft<F, 3, INV>::run(u);
#pragma unroll
            for (int a = 0; a < 3; ++a) t[a][b] = u[a];
        }
        // cos and sin of 40, 80 and 160 degrees
        const S c2 = S(0.17364817766693034885), s2 = S(0.98480775301220805937);
        t[1][1] = crot<INV>(t[1][1], S(0.76604444311897803520), S(0.64278760968653932632));
        t[1][2] = crot<INV>(t[1][2], c2, s2);
        t[2][1] = crot<INV>(t[2][1], c2, s2);
        t[2][2] = crot<INV>(t[2][2], S(-0.93969262078590838405), S(0.34202014332566873304));
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            Dft<F, 3, INV>::run(t[a]);
#pragma unroll
            for (int b = 0; b < 3; ++b) v[a + 3 * b] = t[a][b];
        }
    }
};
template <class F, bool INV> struct Dft<F, 16, INV> {
    static __device__ __forceinline__ void run(Cx<F> *v) {
        using S = typename Scal<F>::type;
        Cx<F> t[4][4];
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            Cx<F> u[4] = {v[b], v[4 + b], v[8 + b], v[12 + b]};
            Dft<F, 4, INV>::run(u);
#pragma unroll
            for (int a = 0; a < 4; ++a) t[a][b] = u[a];
        }
        const S h = S(0.70710678118654752440), c = S(0.92387953251128675613), d = S(0.38268343236508977173);
        t[1][1] = crot<INV>(t[1][1], c, d);
        t[1][2] = crot<INV>(t[1][2], h, h);
        t[1][3] = crot<INV>(t[1][3], d, c);
        t[2][1] = crot<INV>(t[2][1], h, h);
        t[2][2] = crot<INV>(t[2][2], S(0), S(1));
        t[2][3] = crot<INV>(t[2][3], -h, h);
        t[3][1] = crot<INV>(t[3][1], d, c);
        t[3][2] = crot<INV>(t[3][2], -h, h);
        t[3][3] = crot<INV>(t[3][3], -c, -d);
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            Dft<F, 4, INV>::run(t[a]);
#pragma unroll
            for (int b = 0; b < 4; ++b) v[a + 4 * b] = t[a][b];
        }
    }
};

// Twiddles exp(-2 pi i n / K) in shared memory: as complex values, or for the
// packed form with each component doubled.
template <class F> struct TwOf { using type = Cx<F>; };
template <> struct TwOf<float2> { using type = float4; };
__device__ __forceinline__ void tw_set(Cx<double> &t, double2 w) { t = {w.x, w.y}; }
__device__ __forceinline__ void tw_set(float4 &t, float2 w) { t = make_float4(w.x, w.x, w.y, w.y); }
// v times the twiddle (its conjugate for INV)
template <bool INV> __device__ __forceinline__ Cx<double> ctw(Cx<double> v, Cx<double> w) {
    const double wy = INV ? -w.y : w.y;
    return {fma(v.x, w.x, -(v.y * wy)), fma(v.x, wy, v.y * w.x)};
}
template <bool INV> __device__ __forceinline__ Cx<float2> ctw(Cx<float2> v, float4 w) {
    const float2 wx = make_float2(w.x, w.y), wy = make_float2(w.z, w.w), nwy = make_float2(-w.z, -w.w);
    return {__ffma2_rn(v.x, wx, __fmul2_rn(v.y, INV ? wy : nwy)), __ffma2_rn(v.x, INV ? nwy : wy, __fmul2_rn(v.y, wx))};
}
// A complex value in one 16-byte access.
template <class F> union CxBits {
    float4 v;
    Cx<F> c;
};
template <class F> __device__ __forceinline__ Cx<F> cld(const Cx<F> *p) {
    static_assert(sizeof(Cx<F>) == 16, "one pair in double, two in float");
    CxBits<F> u;
    u.v = *reinterpret_cast<const float4 *>(p);
    return u.c;
}
template <class F> __device__ __forceinline__ void cst(Cx<F> *p, Cx<F> c) {
    CxBits<F> u;
    u.c = c;
    *reinterpret_cast<float4 *>(p) = u.v;
}

// ---------------------------------------------------------------- compile-time passes
// A transform of K = r_1 r_2 ... r_n rows, in place on a K x W tile in shared
// memory.  Forward (decimation in frequency): stage s splits every block of
// B = r_s M rows into r_s-point DFTs over the rows m + M q, multiplied by the
// twiddles exp(-2 pi i m q / B), leaving r_s blocks of M rows; the last stage
// (M = 1) leaves the row of frequency k at the digit-reversed place, so its
// thread writes the frequencies it holds straight to their rows of the mesh.
// A butterfly is read and written by one thread, so a stage needs no second
// buffer and one barrier follows it: for almost all sizes n = 2 (radices up
// to 16), that is a tile written once, read, written and read.  The pass fused
// with the influence function multiplies the frequencies that a thread of the
// last stage holds by G, transforms them back at once (inverse r_n-point DFT)
// and runs the remaining stages backwards (decimation in time) in the same
// places: three exchanges instead of the six of a forward and an inverse pass.
template <int... RS> struct Plan {
    static constexpr int n = sizeof...(RS);
    static constexpr int r[n] = {RS...};
    static constexpr int K = (RS * ... * 1);
    static constexpr int M(int s) {          // rows of the blocks that stage s leaves
        int m = 1;
        for (int t = s + 1; t < n; ++t) m *= r[t];
        return m;
    }
    static constexpr int last() { return r[n - 1]; }
    static constexpr int rmin() {
        int m = r[0];
        for (int t = 1; t < n; ++t) m = r[t] < m ? r[t] : m;
        return m;
    }
    static constexpr int before(int s) {     // product of the radices before stage s
        int m = 1;
        for (int t = 0; t < s; ++t) m *= r[t];
        return m;
    }
    // lowest frequency of the last stage's block `blk`: digits k_1 .. k_{n-1}, first digit fastest
    template <int S = n - 2> static __device__ __forceinline__ int rev(int blk) {
        constexpr int R = r[S], mult = before(S);
        if constexpr (S == 0) return blk;
        else return (blk % R) * mult + rev<S - 1>(blk / R);
    }
};

// Threads of a pass: one butterfly each in the stage with the most, at most 256.
template <class P, int W> constexpr int ct_threads() {
    constexpr int t = ((P::K / P::rmin()) * W + 31) / 32 * 32;
    return t < 256 ? t : 256;
}

// Stage S (not the last) of the forward transform in place, and the same stage
// of the inverse (twiddles first) in place or, for S = 0, to the rows of the
// mesh column gout (row stride gs) of a valid column.
template <class P, int S, class F, int W, int NT, bool INV>
__device__ __forceinline__ void ct_fwd_stage(Cx<F> *tile, const typename TwOf<F>::type *tw) {
    constexpr int R = P::r[S], M = P::M(S), K = P::K, B = R * M, NB = K / R;
    const int col = threadIdx.x % W;
#pragma unroll
    for (int it = 0; it < (NB * W + NT - 1) / NT; ++it) {
        const int j = it * (NT / W) + (int)threadIdx.x / W;
        if (NB % (NT / W) != 0 && j >= NB) break;
        const int m = j % M;
        Cx<F> *t = tile + ((j / M) * B + m) * W + col;
        Cx<F> v[R];
#pragma unroll
        for (int q = 0; q < R; ++q) v[q] = cld(t + q * M * W);
        Dft<F, R, INV>::run(v);
        cst(t, v[0]);
#pragma unroll
        for (int q = 1; q < R; ++q) cst(t + q * M * W, ctw<INV>(v[q], tw[(K / B) * m * q]));
    }
}
template <class P, int S, class F, int W, int NT>
__device__ __forceinline__ void ct_inv_stage(Cx<F> *tile, const typename TwOf<F>::type *tw, Cx<F> *gout, size_t gs,
                                             bool valid) {
    constexpr int R = P::r[S], M = P::M(S), K = P::K, B = R * M, NB = K / R;
    const int col = threadIdx.x % W;
#pragma unroll
    for (int it = 0; it < (NB * W + NT - 1) / NT; ++it) {
        const int j = it * (NT / W) + (int)threadIdx.x / W;
        if (NB % (NT / W) != 0 && j >= NB) break;
        const int m = j % M;
        Cx<F> *t = tile + ((j / M) * B + m) * W + col;
        Cx<F> v[R];
        v[0] = cld(t);
#pragma unroll
        for (int q = 1; q < R; ++q) v[q] = ctw<true>(cld(t + q * M * W), tw[(K / B) * m * q]);
        Dft<F, R, true>::run(v);
        if constexpr (S == 0) {
            if (valid) {
#pragma unroll
                for (int q = 0; q < R; ++q) cst(gout + (size_t)(m + M * q) * gs, v[q]);
            }
        } else {
#pragma unroll
            for (int q = 0; q < R; ++q) cst(t + q * M * W, v[q]);
        }
    }
}
// The last stage of a pass: frequencies to the mesh column gout.
template <class P, class F, int W, int NT, bool INV>
__device__ __forceinline__ void ct_last_stage(const Cx<F> *tile, Cx<F> *gout, size_t gs, bool valid) {
    constexpr int R = P::r[P::n - 1], K = P::K, NB = K / R;
    const int col = threadIdx.x % W;
#pragma unroll
    for (int it = 0; it < (NB * W + NT - 1) / NT; ++it) {
        const int j = it * (NT / W) + (int)threadIdx.x / W;
        if (NB % (NT / W) != 0 && j >= NB) break;
        const Cx<F> *t = tile + j * R * W + col;
        Cx<F> v[R];
#pragma unroll
        for (int q = 0; q < R; ++q) v[q] = cld(t + q * W);
        Dft<F, R, INV>::run(v);
        if (valid) {
            Cx<F> *o = gout + (size_t)P::template rev<>(j) * gs;
#pragma unroll
            for (int q = 0; q < R; ++q) cst(o + (size_t)(q * NB) * gs, v[q]);
        }
    }
}
// The G of one butterfly of the mid stage: rows rev(j) + NB q of the column.
template <class P, class S> __device__ __forceinline__ void ct_load_g(const S *__restrict__ gcol, size_t gstride, int j,
                                                                      S *g) {
    constexpr int R = P::r[P::n - 1], NB = P::K / R;
    const S *gr = gcol + (size_t)P::template rev<>(j) * gstride;
#pragma unroll
    for (int q = 0; q < R; ++q) g[q] = gr[(size_t)(q * NB) * gstride];
}
// Whether a thread has one butterfly of the mid stage per tile, whose G it then
// loads before it waits for the tile.
template <class P, int W, int NT> constexpr bool ct_g_early() { return (P::K / P::r[P::n - 1]) * W <= NT; }

// The last forward stage, the product with G (gcol: G of the column, row
// stride gstride; g: the values already loaded, ct_g_early) and the first
// inverse stage, in place.
template <class P, class F, int W, int NT>
__device__ __forceinline__ void ct_mid_stage(Cx<F> *tile, const typename Scal<F>::type *__restrict__ gcol,
                                             size_t gstride, const typename Scal<F>::type *gearly) {
    using S = typename Scal<F>::type;
    constexpr int R = P::r[P::n - 1], K = P::K, NB = K / R;
    const int col = threadIdx.x % W;
#pragma unroll
    for (int it = 0; it < (NB * W + NT - 1) / NT; ++it) {
        const int j = it * (NT / W) + (int)threadIdx.x / W;
        if (NB % (NT / W) != 0 && j >= NB) break;
        Cx<F> *t = tile + j * R * W + col;
        S g[R];
        if constexpr (ct_g_early<P, W, NT>()) {
#pragma unroll
            for (int q = 0; q < R; ++q) g[q] = gearly[q];
        } else {
            ct_load_g<P>(gcol, gstride, j, g);
        }
        Cx<F> v[R];
#pragma unroll
        for (int q = 0; q < R; ++q) v[q] = cld(t + q * W);
        Dft<F, R, false>::run(v);
#pragma unroll
        for (int q = 0; q < R; ++q) v[q] = {fmulc(v[q].x, g[q]), fmulc(v[q].y, g[q])};
        Dft<F, R, true>::run(v);
#pragma unroll
        for (int q = 0; q < R; ++q) cst(t + q * W, v[q]);
    }
}
template <class P, int S, class F, int W, int NT, bool INV>
__device__ __forceinline__ void ct_forward(Cx<F> *tile, const typename TwOf<F>::type *tw) {
    if constexpr (S < P::n - 1) {
        ct_fwd_stage<P, S, F, W, NT, INV>(tile, tw);
        __syncthreads();
        ct_forward<P, S + 1, F, W, NT, INV>(tile, tw);
    }
}
template <class P, int S, class F, int W, int NT>
__device__ __forceinline__ void ct_inverse(Cx<F> *tile, const typename TwOf<F>::type *tw, Cx<F> *gout, size_t gs,
                                           bool valid) {
    ct_inv_stage<P, S, F, W, NT>(tile, tw, gout, gs, valid);
    if constexpr (S > 0) {
        __syncthreads();
        ct_inverse<P, S - 1, F, W, NT>(tile, tw, gout, gs, valid);
    }
}
// The unfused transform of a tile already in shared memory (visible to every
// thread), to the mesh column gout.
template <class P, class F, int W, int NT, bool INV>
__device__ __forceinline__ void ct_transform(Cx<F> *tile, const typename TwOf<F>::type *tw, Cx<F> *gout, size_t gs,
                                             bool valid) {
    ct_forward<P, 0, F, W, NT, INV>(tile, tw);
    ct_last_stage<P, F, W, NT, INV>(tile, gout, gs, valid);
}

// Asynchronous copies from global to shared memory (cp.async) of one complex
// value, and the group fences of those copies.
template <int BYTES> __device__ __forceinline__ void cp_async(void *smem, const void *gmem) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    if constexpr (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sa), "l"(gmem) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(sa), "l"(gmem), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// One 1D pass along the middle axis of [outer][K][inner] (values Cx<F>), MODE
// 0 forward, 1 inverse, 2 forward x G inverse.  The outer x inner columns are
// cut into tiles of W consecutive ones (a tile may span several outer slabs,
// so narrow rows fill tiles too; only the last tile is partial).  A block
// takes tiles blockIdx.x, blockIdx.x + gridDim.x, ...; while it transforms one,
// the next arrives in its second buffer by cp.async.  A thread works on one
// column of every tile.
// Bound: HBM (each pass reads and writes the mesh once); the FP32 issue and the
// shared-memory exchanges are what the packed form and the two stages cut.
template <class T, class F, class P, int MODE, int W, int NT>
__global__ void __launch_bounds__(NT) k_fft_ct(FFTArgs<T> a, unsigned ncols, unsigned ntiles) {
    using C = Cx<F>;
    using TW = typename TwOf<F>::type;
    constexpr int K = P::K, RL = P::last();
    constexpr int TR = NT / W;                // rows copied per step
    static_assert(P::n >= 2 && NT % W == 0, "two stages at least; whole rows of threads");
    extern __shared__ __align__(16) unsigned char smem_ct[];
    TW *tw = reinterpret_cast<TW *>(smem_ct);
    C *buf = reinterpret_cast<C *>(tw + K);
    for (int i = threadIdx.x; i < K; i += NT) tw_set(tw[i], a.tw[i]);   // set up once per system
    pdl_wait();
    pdl_launch_dependents();
    const int col = threadIdx.x % W, row0 = threadIdx.x / W;
    C *data = reinterpret_cast<C *>(a.data);
    const size_t gs = (size_t)a.inner;
    auto column = [&](unsigned cg) {
        const unsigned o = cg / (unsigned)a.inner;
        return data + (size_t)o * K * gs + (cg - o * (unsigned)a.inner);
    };
    auto fetch = [&](unsigned t, C *to) {
        const unsigned cg = t * W + col;
        if (cg < ncols) {
            const C *src = column(cg) + (size_t)row0 * gs;
            for (int row = row0; row < K; row += TR, src += TR * gs) cp_async<(int)sizeof(C)>(to + row * W + col, src);
        }
    };
    unsigned t = blockIdx.x;
    if (t < ntiles) fetch(t, buf);
    cp_async_commit();
    for (int b = 0; t < ntiles; t += gridDim.x, b ^= 1) {
        C *cur = buf + b * (K * W);
        __syncthreads();                      // every thread is done with the other buffer
        if (t + gridDim.x < ntiles) fetch(t + gridDim.x, buf + (b ^ 1) * (K * W));
        cp_async_commit();
        const unsigned cg = t * W + col;
        const bool valid = cg < ncols;
        C *out = column(valid ? cg : 0);
        const T *gcol = MODE == 2 ? a.G + (valid ? cg : 0) / (unsigned)a.V : nullptr;
        const size_t gstride = MODE == 2 ? gs / a.V : 0;
        T g[RL];
        if constexpr (MODE == 2 && ct_g_early<P, W, NT>()) {
            if (row0 < K / RL) ct_load_g<P>(gcol, gstride, row0, g);
        }
        cp_async_wait<1>();                   // this thread's copies of tile t are done
        __syncthreads();                      // and every thread's
        if constexpr (MODE == 2) {
            ct_forward<P, 0, F, W, NT, false>(cur, tw);
            ct_mid_stage<P, F, W, NT>(cur, gcol, gstride, g);
            __syncthreads();
            ct_inverse<P, P::n - 2, F, W, NT>(cur, tw, out, gs, valid);
        } else {
            ct_transform<P, F, W, NT, MODE == 1>(cur, tw, out, gs, valid);
        }
    }
    cp_async_wait<0>();                       // no copy in flight at exit
}

// Launch of one pass: a block per tile when all tiles are resident at once
// (one buffer), persistent blocks with two buffers otherwise.
template <class T, class F, class P, int MODE, int W> int launch_ct(const FFTArgs<T> &a, unsigned outer,
                                                                    cudaStream_t st) {
    constexpr int NT = ct_threads<P, W>();
    auto kern = k_fft_ct<T, F, P, MODE, W, NT>;
    const size_t tile = sizeof(Cx<F>) * (size_t)P::K * W, fixed = sizeof(typename TwOf<F>::type) * P::K;
    const size_t most = fixed + 2 * tile;
    static std::atomic<int> per_sm[2];        // resident blocks per SM with one and two buffers (one architecture)
    int resident[2];
    for (int k = 0; k < 2; ++k) {
        resident[k] = per_sm[k].load(std::memory_order_relaxed);
        if (resident[k] > 0) continue;
        if (allow_smem(kern, most, most) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&resident[k], kern, NT, fixed + (k + 1) * tile) != cudaSuccess ||
            resident[k] < 1)
            return 0;
        per_sm[k].store(resident[k], std::memory_order_relaxed);
    }
    const unsigned ncols = outer * (unsigned)a.inner, ntiles = (ncols + W - 1) / W;
    const unsigned sms = (unsigned)std::max(1, a.sms);
    const bool once = ntiles <= resident[0] * sms;
    const unsigned grid = once ? ntiles : std::min(ntiles, resident[1] * sms);
    const size_t smem = fixed + (once ? 1 : 2) * tile;
    if (allow_smem(kern, smem, most) != cudaSuccess) return 0;
    // double passes of a few blocks per SM are bound by the FP64 units: blocks
    // launched early land unevenly on the SMs (64 atoms, 32^3 x 16 probes: 4.2 ms
    // per energy + forces against 3.6); one block per SM or persistent blocks
    // are even in any case
    const bool early = a.early == 2 || (a.early == 1 && (sizeof(T) == 4 || !once || grid <= sms));
    launch_pdl(early, kern, dim3(grid), dim3(NT), smem, st, a, ncols, ntiles);
    return 1;
}

// The passes of one size: packed float tiles of 16 or 8 column pairs (a.W = 32
// or 16 complex columns; V is even), double tiles of 8.
template <class T, class F, class P, int W> int ct_mode(const FFTArgs<T> &a, int mode, unsigned outer, cudaStream_t st) {
    if (mode == 0) return launch_ct<T, F, P, 0, W>(a, outer, st);
    if (mode == 1) return launch_ct<T, F, P, 1, W>(a, outer, st);
    return launch_ct<T, F, P, 2, W>(a, outer, st);
}
template <class T, class P> int ct_size(const FFTArgs<T> &a, int mode, unsigned outer, cudaStream_t st) {
    if constexpr (sizeof(T) == 8) {
        return ct_mode<T, double, P, 8>(a, mode, outer, st);
    } else {
        FFTArgs<T> q = a;
        q.inner /= 2;
        q.V /= 2;
        return a.W == 32 ? ct_mode<T, float2, P, 16>(q, mode, outer, st) : ct_mode<T, float2, P, 8>(q, mode, outer, st);
    }
}

// ---------------------------------------------------------------- spreading by pencil records
// Spline orders the spreading is compiled for.
#define MBD_SPLINE_ORDERS(X) X(4) X(6) X(8) X(10)

// a c + b over the probes of a lane (packed for two floats), scalar c.
template <class T, int PPL> __device__ __forceinline__ void lane_fma(const T *a, T c, T *b) {
    if constexpr (PPL % 2 == 0 && sizeof(T) == 4) {
#pragma unroll
        for (int e = 0; e < PPL; e += 2) {
            const float2 r = __ffma2_rn(make_float2(a[e], a[e + 1]), make_float2(c, c), make_float2(b[e], b[e + 1]));
            b[e] = r.x;
            b[e + 1] = r.y;
        }
    } else {
#pragma unroll
        for (int e = 0; e < PPL; ++e) b[e] += a[e] * c;
    }
}

// A lane's walk along one pencil (k1, k2) for its PPL probes (d: the dipole
// rows at those probes): the records of the points (k1, k2, t) for t = t1 - 1
// down to t0 (records q0 .. q1 - 1, begins(t) the first of point t), each adding
// M3(j) (e0 . d) + M3'(j) (e1 . d) to the rows t - j, j < P.  Row t is complete
// after point t and goes to row_done; the P - 1 rows below t0 stay in
// registers and go to tail after between() (a barrier where they belong to
// another warp).  The window of P open rows is a register array whose origin
// moves with t, unrolled by P so that it never shifts; each row is a sum in a
// fixed order.  The next record is loaded one ahead.  STARTS: the record starts of
// P points are loaded together (where they come from global memory).
template <class T, int P, int PPL, bool STARTS, class Begins, class Done, class Between, class Tail>
__device__ __forceinline__ void pencil_walk(const T *__restrict__ d, int ld, const PencilRec<T> *__restrict__ prec,
                                            const T *__restrict__ k3w, int t0, int t1, int q0, int q1, Begins &&begins,
                                            Done &&row_done, Between &&between, Tail &&tail) {
    T acc[P][PPL];                              // row r in slot (t1 - 1 - r) mod P
#pragma unroll
    for (int j = 0; j < P; ++j)
#pragma unroll
        for (int e = 0; e < PPL; ++e) acc[j][e] = T(0);
    int q = q1 - 1;
    PencilRec<T> rc{};
    if (q >= q0) rc = prec[q];
    const int n = t1 - t0;
    for (int sb = 0; sb < n; sb += P) {
        int starts[P];
        if constexpr (STARTS) {
#pragma unroll
            for (int u = 0; u < P; ++u) starts[u] = begins(max(t0, t1 - 1 - sb - u));
        }
#pragma unroll
        for (int u = 0; u < P; ++u) {
            if (sb + u >= n) break;
            const int t = t1 - 1 - sb - u, qb = STARTS ? starts[u] : begins(t);
            while (q >= qb) {
                T x[PPL], y[PPL], z[PPL], w[2 * P];
                const T *dj = d + (size_t)(3 * rc.atom) * ld;
                vload<T, PPL>(dj, x);
                vload<T, PPL>(dj + ld, y);
                vload<T, PPL>(dj + 2 * (size_t)ld, z);
                constexpr int U = 16 / (int)sizeof(T);
                const T *kw = k3w + (size_t)rc.atom * (2 * P);
#pragma unroll
                for (int b = 0; b < 2 * P; b += U) vload<T, U>(kw + b, w + b);
                T fu[PPL], fv[PPL];
#pragma unroll
                for (int e = 0; e < PPL; ++e) fu[e] = fv[e] = T(0);
                lane_fma<T, PPL>(x, rc.e0[0], fu);
                lane_fma<T, PPL>(y, rc.e0[1], fu);
                lane_fma<T, PPL>(z, rc.e0[2], fu);
                lane_fma<T, PPL>(x, rc.e1[0], fv);
                lane_fma<T, PPL>(y, rc.e1[1], fv);
                lane_fma<T, PPL>(z, rc.e1[2], fv);
                if (--q >= q0) rc = prec[q];
#pragma unroll
                for (int j = 0; j < P; ++j) {
                    lane_fma<T, PPL>(fu, w[j], acc[(u + j) % P]);
                    lane_fma<T, PPL>(fv, w[P + j], acc[(u + j) % P]);
                }
            }
            row_done(t, acc[u]);
#pragma unroll
            for (int e = 0; e < PPL; ++e) acc[u][e] = T(0);
        }
    }
    between();
    const int phase = n % P;                    // slot of row t0 - 1
#pragma unroll
    for (int k = 0; k < 2 * P - 2; ++k)
        if (k >= phase && k < phase + P - 1) tail(t0 - 1 - (k - phase), acc[k % P]);
}

// Probes per lane and complex columns per tile (a warp's width) of the spreading.
template <class T> constexpr int spread_ppl() { return sizeof(T) == 4 ? 2 : 1; }
template <class T> constexpr int spread_w() { return 16 * spread_ppl<T>(); }
// Warps of a block: one per segment of the pencil, each at least P - 1 rows.  Few
// long segments add fewer rows twice and balance their records better, as
// long as the blocks' warps fill the SM (short pencils: many blocks); long
// pencils have fewer blocks in shared memory and take more warps per block.  us
// per launch: 120^3 x 64 probes 207 with 4 segments and 221 with 6, 128^3 x 128
// 490 and 498; 144^3 x 64 363 with 6 and 379 with 5, 160^3 x 64 547 and 556; 192^3
// x 64 921 with 8, 986 with 6 and 1012 with 10 (before the order of the radices).  Grids of few tiles are bound by a
// warp's own chain of records: 8 (40^3 x 8: 9.9 against 10.3).
template <int K, int P> constexpr int spread_segs(bool few_tiles) {
    constexpr int want = K <= 128 ? 4 : (K <= 160 ? 6 : 8), most = K / (P - 1);
    return (few_tiles ? 8 : want) < most ? (few_tiles ? 8 : want) : most;
}

// Shared memory of a block whose tile touches `pens` pencils, and the blocks
// per SM asked of the compiler: 32 warps (64 registers) in float and 24 in
// double as far as shared memory holds them (resident warps hide the latency
// of the dipole loads: loading them one record ahead takes the registers of a
// third of the warps, 64^3 x 64 probes 49 -> 62 us).
template <class T, int K> constexpr size_t spread_smem(int pens) {
    return sizeof(typename TwOf<typename PackOf<T>::type>::type) * K +
           sizeof(T) * 2 * (size_t)spread_w<T>() * K +
           sizeof(int) * ((size_t)pens * K + 1);
}
template <class T, int K, int NSEG> constexpr int spread_blocks() {
    constexpr int by_smem = (int)(227 * 1024 / (spread_smem<T, K>(2) + 1024)), by_regs = (sizeof(T) == 4 ? 32 : 24) / NSEG;
    return by_smem < by_regs ? by_smem : by_regs;
}

// Spreading fused with the forward FFT along k3.  A block owns a tile of W
// consecutive complex columns (pencil, probe pair) of the mesh: one pencil's
// when the probes fill a warp, several pencils' otherwise; lane l holds the
// tile's probes l PPL .. and so its own pencil.  The K points of the pencil
// are cut into one segment per warp; a warp walks the records of its segment's
// points once, its rows go to the shared tile, and after a barrier it adds the
// P - 1 rows below its segment, which belong to the warp before (cyclically).
// Then the block transforms the tile and writes it.  Probes >= R are zero.
// Bound: instruction issue and the latency of the dipole loads (L2).  Walking
// every record that reaches a warp's rows, and a second buffer for the
// transform: 192^3 x 64 probes 1507 us per launch; each record once, the rows
// below a segment through a halo in shared memory: 1139; those rows kept in
// registers (the walk runs downwards), one block more per SM: 921, and 900 with
// the largest radix last.  128^3 x 128: 862, 552 and 490; 64^3 x 64: 56, 41 and 37.
template <class T, class PL, int P, int NSEG>
__global__ void __launch_bounds__(32 * NSEG, (spread_blocks<T, PL::K, NSEG>()))
    k_spread_pencil_fft3(const T *__restrict__ d, T *__restrict__ mesh, int R, int ld, unsigned ncols,
                         const int *__restrict__ prow, const PencilRec<T> *__restrict__ prec,
                         const T *__restrict__ k3w, const typename Cplx<T>::type *__restrict__ twg) {
    using F = typename PackOf<T>::type;
    using C = Cx<F>;
    constexpr int K = PL::K, PPL = spread_ppl<T>(), W = spread_w<T>(), NT = 32 * NSEG;
    constexpr int WF = W * 2 * (int)sizeof(T) / (int)sizeof(C);
    static_assert(NT % WF == 0 && NSEG >= 2, "whole rows of threads, two segments at least");
    extern __shared__ __align__(16) unsigned char smem_spp[];
    auto *tw = reinterpret_cast<typename TwOf<F>::type *>(smem_spp);
    T *tile = reinterpret_cast<T *>(tw + K);          // [K][2W] reals
    int *rp = reinterpret_cast<int *>(tile + 2 * (size_t)K * W);   // record starts of the tile's pencils
    const int V = ld / 2;
    const unsigned c0 = blockIdx.x * W;
    const unsigned pen0 = c0 / V, pen1 = min(c0 + W, ncols) - 1;   // first pencil, last column
    const int nrp = (int)(pen1 / V - pen0 + 1) * K;
    for (int i = threadIdx.x; i < K; i += NT) tw_set(tw[i], twg[i]);   // set up once per system
    for (int i = threadIdx.x; i <= nrp; i += NT) rp[i] = prow[(size_t)pen0 * K + i];
    pdl_wait();
    pdl_launch_dependents();
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int r0 = warp * K / NSEG, r1 = (warp + 1) * K / NSEG;
    const unsigned cl = min(c0 + lane * PPL / 2, ncols - 1);      // the lane's column (the last one again past the end)
    const unsigned pen = cl / V;
    const int pr0 = 2 * (int)(cl - pen * V) + (lane * PPL & 1);   // its first probe
    const int *rpp = rp + (pen - pen0) * K;
    T *mine = tile + lane * PPL;
    pencil_walk<T, P, PPL, false>(
        d + pr0, ld, prec, k3w, r0, r1, rpp[r0], rpp[r1], [&](int t) { return rpp[t]; },
        [&](int row, const T *v) {
            T o[PPL];
#pragma unroll
            for (int e = 0; e < PPL; ++e) o[e] = pr0 + e < R ? v[e] : T(0);
            vstore<T, PPL>(mine + row * 2 * W, o);
        },
        [] { __syncthreads(); },
        [&](int row, const T *v) {
            T *o = mine + (row < 0 ? row + K : row) * 2 * W;
            T y[PPL];
            vload<T, PPL>(o, y);
#pragma unroll
            for (int e = 0; e < PPL; ++e) y[e] += pr0 + e < R ? v[e] : T(0);
            vstore<T, PPL>(o, y);
        });
    __syncthreads();
    const unsigned VF = (unsigned)((size_t)ld * sizeof(T) / sizeof(C)), nf = ncols / V * VF;
    const unsigned cg = blockIdx.x * WF + threadIdx.x % WF;
    const bool valid = cg < nf;
    const unsigned pf = (valid ? cg : 0) / VF;
    ct_transform<PL, F, WF, NT, false>(reinterpret_cast<C *>(tile), tw,
                                       reinterpret_cast<C *>(mesh) + (size_t)pf * K * VF + ((valid ? cg : 0) - pf * VF),
                                       VF, valid);
}

template <class T, class PL, int P, int NSEG>
int launch_spp_segs(const SpreadArgs<T> &a, cudaStream_t st) {
    constexpr int K = PL::K, W = spread_w<T>();
    auto kern = k_spread_pencil_fft3<T, PL, P, NSEG>;
    const int V = a.ld / 2;
    const int pens = (W - 1) / V + 2;              // pencils that a tile can touch; most at the smallest V
    const size_t smem = spread_smem<T, K>(pens);
    constexpr int vmin = probe_ld<T>(1) / 2;
    if (allow_smem(kern, smem, spread_smem<T, K>((W - 1) / vmin + 2)) != cudaSuccess) return 0;
    const unsigned ncols = (unsigned)((size_t)a.K1 * a.K2 * V);
    launch_pdl(true, kern, dim3((ncols + W - 1) / W), dim3(32 * NSEG), smem, st, a.d, a.mesh, a.R, a.ld, ncols, a.prow,
               a.prec, a.k3w, a.tw);
    return 1;
}
template <class T, class PL, int P> int launch_spp(const SpreadArgs<T> &a, cudaStream_t st) {
    constexpr int many = spread_segs<PL::K, P>(false), few = spread_segs<PL::K, P>(true);
    const size_t tiles = (size_t)a.K1 * a.K2 * (a.ld / 2) / spread_w<T>();
    if (many != few && tiles < 8 * (size_t)a.sms) return launch_spp_segs<T, PL, P, few>(a, st);
    return launch_spp_segs<T, PL, P, many>(a, st);
}
template <class T, class PL> int spp_size(const SpreadArgs<T> &a, cudaStream_t st) {
#define MBD_SPP_ORDER(P) \
    case P: \
        if constexpr (PL::K >= 2 * (P)) return launch_spp<T, PL, P>(a, st); \
        break;
    switch (a.p) { MBD_SPLINE_ORDERS(MBD_SPP_ORDER) }
#undef MBD_SPP_ORDER
    return -1;
}

}  // namespace

// The translation unit of group g: dispatch over its sizes.
#define MBD_CT_CASE(K, ...) \
    case K: return ct_size<T, Plan<__VA_ARGS__>>(a, mode, outer, st);
#define MBD_SPP_CASE(K, ...) \
    case K: return spp_size<T, Plan<__VA_ARGS__>>(a, st);
#define MBD_FFT_GROUP_TU(g)                                                                                       \
    template <class T> int launch_fft_ct_group##g(const FFTArgs<T> &a, int mode, unsigned outer, cudaStream_t st) { \
        switch (a.K) { MBD_FFT_GROUP##g(MBD_CT_CASE) default: return -1; }                                         \
    }                                                                                                              \
    template <class T> int launch_spp_group##g(const SpreadArgs<T> &a, cudaStream_t st) {                          \
        switch (a.K3) { MBD_FFT_GROUP##g(MBD_SPP_CASE) default: return -1; }                                       \
    }                                                                                                              \
    template int launch_fft_ct_group##g<float>(const FFTArgs<float> &, int, unsigned, cudaStream_t);               \
    template int launch_fft_ct_group##g<double>(const FFTArgs<double> &, int, unsigned, cudaStream_t);             \
    template int launch_spp_group##g<float>(const SpreadArgs<float> &, cudaStream_t);                              \
    template int launch_spp_group##g<double>(const SpreadArgs<double> &, cudaStream_t);

}  // namespace mbd

// Force kernels.  The paper computes energies only (its Conclusions name the
// gradients as the next step); with alpha and omega position-independent,
//   dE/dR = (1/4) Tr(C^{-1/2} dC/dR) ~ (1/4)(D/R) sum_l grad_R [p_l^T T'(R) q_l],
// p_l = g . w_l, q_l = g . v_l, w_l = C^{-1/2} v_l = sum_k c_{lk} y_{lk}.
// The probes' p and q are interleaved as 2R "probes" (p_l, q_l in columns 2l, 2l + 1),
// so the SPME part reuses the spread and FFT convolution kernels, which transform
// pairs of them as one complex vector (G is real and even: any pairing is exact):
//   phi_p = F^-1[G F[D_p]], phi_q = F^-1[G F[D_q]],
// and grad_i = sum_k H_i(k) [p_i phi_q(k) + q_i phi_p(k)] with H_i the Hessian
// of the stencil weight W_i(k) wrt R_i; the real-space part contracts the
// derivative of the pair tensor, dA_ab/dr_c, with p_i q_j + p_j q_i.
#include "fft.cuh"

#include <algorithm>

namespace mbd {

namespace {

constexpr int kWarps = 8;

template <class T>
__global__ void k_force_dipoles(int rows, const double *__restrict__ Y, const double *__restrict__ coef,
                                const int *__restrict__ length, const double *__restrict__ g, int R, int ld, int m,
                                T *__restrict__ dpq, int ld2) {
    const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (size_t)rows * R) return;
    const int row = (int)(idx / R), r = (int)(idx % R);
    const size_t stride = (size_t)rows * ld;
    const int n = length[r];
    double w = 0.0;
    for (int k = 0; k < n; ++k) w += coef[(size_t)k * ld + r] * Y[(size_t)k * stride + (size_t)row * ld + r];
    const double gi = g[row / 3];
    dpq[(size_t)row * ld2 + 2 * r] = T(gi * w);
    dpq[(size_t)row * ld2 + 2 * r + 1] = T(gi * Y[(size_t)row * ld + r]);
}

// The same from w = sum_k c_k y_k accumulated during a rerun of the recurrence
// (recomputed basis) and y_0 = v.
template <class T>
__global__ void k_force_dipoles_w(int rows, const double *__restrict__ w, const double *__restrict__ v,
                                  const double *__restrict__ g, int R, int ld, T *__restrict__ dpq, int ld2) {
    const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (size_t)rows * R) return;
    const int row = (int)(idx / R), r = (int)(idx % R);
    const double gi = g[row / 3];
    dpq[(size_t)row * ld2 + 2 * r] = T(gi * w[(size_t)row * ld + r]);
    dpq[(size_t)row * ld2 + 2 * r + 1] = T(gi * v[(size_t)row * ld + r]);
}

template <class T> struct ForceArgs {
    const T *dpq;        // [N][3][ld2] (p_l, q_l) interleaved
    const T *mesh;       // [K^3][ld2] (phi_p, phi_q) interleaved
    int R, ld2;
    Geom g;
    const int *order;    // atoms in the Morton order of the bricks
    const int *top;
    const T *w, *dw, *d2w;
    const int *row, *col;
    const T *dA;         // [nnz][18] dA_ab/dr_c of the real-space pair tensor
    double scale;
    double *forces;      // [N][3] FP64
    int lanes;           // lanes that hold a chunk of 32 VEC values of a row (or all of it)
    int wpa;             // warps per atom
};

// One atom's force, wpa warps each: `lanes` lanes with 16-byte accesses hold the
// probes' (p, q) values (chunks of 32 VEC of them, one after another), and the
// groups of the atom's warps share out the p^2 pencils of its stencil and its
// neighbours.  Along a pencil the Hessian of the weight factorises like the
// weight: s_n = sum_t M3^(n)(t) phi, n = 0, 1, 2 (three FMAs per mesh value), and
// six sums over the pencils, G_ab = sum H_ab phi, take two products of M1, M2 and
// their derivatives times s_n each; the dipoles enter once per atom, h_a = sum_b
// (G^q_ab e_p,b + G^p_ab e_q,b).  Partial gradients are summed in FP64 in a fixed
// order (lanes, then warps).
// Bound: load latency (FP32), the FP64 units (FP64).  100,002 atoms x 64 probes
// 6.4 -> 3.1 ms per launch, 3000 x 64 258 -> 135 us, 501 x 7 FP64 391 -> 86 us, 64
// x 16 FP64 124 -> 25 us against the Hessian per mesh value and a lane per probe.
template <class T, int P>
__global__ void __launch_bounds__(kWarps * 32, 2) k_force_gather(ForceArgs<T> a) {
    constexpr int VEC = 16 / (int)sizeof(T);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int idx = blockIdx.x * (kWarps / a.wpa) + warp / a.wpa;
    const int S = 32 / a.lanes, sub = lane / a.lanes, lid = lane - sub * a.lanes;
    const int member = (warp % a.wpa) * S + sub, members = a.wpa * S;
    const bool valid = idx < a.g.N;
    __shared__ double part[kWarps][3];
    double gx = 0.0, gy = 0.0, gz = 0.0;
    const int i = valid ? a.order[idx] : 0;
    if (valid && sub < S) {
        const double *cm = a.g.cmat;
        const int top1 = a.top[3 * i], top2 = a.top[3 * i + 1], top3 = a.top[3 * i + 2];
        const T *w = a.w + (size_t)3 * P * i, *dw = a.dw + (size_t)3 * P * i, *d2w = a.d2w + (size_t)3 * P * i;
        T w3[3][P];
#pragma unroll
        for (int t = 0; t < P; t += 2) {
            vload<T, 2>(w + 2 * P + t, w3[0] + t);
            vload<T, 2>(dw + 2 * P + t, w3[1] + t);
            vload<T, 2>(d2w + 2 * P + t, w3[2] + t);
        }
        T g[3] = {T(0), T(0), T(0)};
        double acc[3] = {0.0, 0.0, 0.0};
        const int nb0 = a.row[i], nb1 = a.row[i + 1];
        for (int c0 = 0; c0 < a.ld2; c0 += 32 * VEC) {
            const int r0 = c0 + lid * VEC;
            if (r0 >= a.ld2) break;
            // the lane's own dipoles; values past the last probe are zero
            T own[3][VEC];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                vload<T, VEC>(a.dpq + (size_t)(3 * i + c) * a.ld2 + r0, own[c]);
#pragma unroll
                for (int v = 0; v < VEC; ++v)
                    if (r0 + v >= 2 * a.R) own[c][v] = T(0);
            }
            // ---- SPME: G_ab (00, 11, 22, 01, 02, 12) of this member's pencils
            T G[6][VEC];
#pragma unroll
            for (int q = 0; q < 6; ++q)
#pragma unroll
                for (int v = 0; v < VEC; ++v) G[q][v] = T(0);
            for (int u = member; u < P * P; u += members) {
                const int t1 = u % P, t2 = u / P;
                int k1 = top1 - t1, k2 = top2 - t2;
                if (k1 < 0) k1 += a.g.K1;
                if (k2 < 0) k2 += a.g.K2;
                const T *rowp = a.mesh + ((size_t)k1 * a.g.K2 + k2) * a.g.K3 * a.ld2 + r0;
                T phi[P][VEC], s[3][VEC];
#pragma unroll
                for (int t = 0; t < P; ++t)
                    vload<T, VEC>(rowp + (size_t)(top3 - t + (top3 < t ? a.g.K3 : 0)) * a.ld2, phi[t]);
                const T wa = w[t1], da = dw[t1], ea = d2w[t1], wb = w[P + t2], db = dw[P + t2], eb = d2w[P + t2];
#pragma unroll
                for (int n = 0; n < 3; ++n) {
#pragma unroll
                    for (int v = 0; v < VEC; ++v) s[n][v] = T(0);
#pragma unroll
                    for (int t = 0; t < P; ++t) lane_fma<T, VEC>(phi[t], w3[n][t], s[n]);
                }
                lane_fma<T, VEC>(s[0], ea * wb, G[0]);
                lane_fma<T, VEC>(s[0], wa * eb, G[1]);
                lane_fma<T, VEC>(s[2], wa * wb, G[2]);
                lane_fma<T, VEC>(s[0], da * db, G[3]);
                lane_fma<T, VEC>(s[1], da * wb, G[4]);
                lane_fma<T, VEC>(s[1], wa * db, G[5]);
            }
            // scaled-fractional components e = C x of p_i and q_i, and h
#pragma unroll
            for (int v = 0; v < VEC; v += 2) {
                T ep[3], eq[3];
#pragma unroll
                for (int b = 0; b < 3; ++b) {
                    ep[b] = T(cm[3 * b]) * own[0][v] + T(cm[3 * b + 1]) * own[1][v] + T(cm[3 * b + 2]) * own[2][v];
                    eq[b] = T(cm[3 * b]) * own[0][v + 1] + T(cm[3 * b + 1]) * own[1][v + 1] +
                            T(cm[3 * b + 2]) * own[2][v + 1];
                }
                auto h = [&](int x, int y, int z) {   // row of G against the other probe vector's components
                    return G[x][v + 1] * ep[0] + G[x][v] * eq[0] + G[y][v + 1] * ep[1] + G[y][v] * eq[1] +
                           G[z][v + 1] * ep[2] + G[z][v] * eq[2];
                };
                acc[0] += double(h(0, 3, 4));
                acc[1] += double(h(3, 1, 5));
                acc[2] += double(h(4, 5, 2));
            }
            // ---- real space: sum_j dA_ab/dr_c sum_l (p_ia q_jb + p_ja q_ib), dA precomputed per pair
            for (int nb = nb0 + member; nb < nb1; nb += members) {
                const int j = a.col[nb];
                T o[3][VEC], M[6] = {T(0), T(0), T(0), T(0), T(0), T(0)};
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    vload<T, VEC>(a.dpq + (size_t)(3 * j + c) * a.ld2 + r0, o[c]);
#pragma unroll
                    for (int v = 0; v < VEC; ++v)
                        if (r0 + v >= 2 * a.R) o[c][v] = T(0);
                }
                T dA[18];
#pragma unroll
                for (int q = 0; q < 18; q += 2) vload<T, 2>(a.dA + 18 * (size_t)nb + q, dA + q);
#pragma unroll
                for (int v = 0; v < VEC; v += 2) {
                    int e = 0;
#pragma unroll
                    for (int x = 0; x < 3; ++x)
#pragma unroll
                        for (int y = x; y < 3; ++y) {
                            T m = own[x][v] * o[y][v + 1] + o[x][v] * own[y][v + 1];
                            if (x != y) m += own[y][v] * o[x][v + 1] + o[y][v] * own[x][v + 1];
                            M[e++] += m;
                        }
                }
#pragma unroll
                for (int ab = 0; ab < 6; ++ab)
#pragma unroll
                    for (int c = 0; c < 3; ++c) g[c] += dA[3 * ab + c] * M[ab];
            }
        }
        // Cartesian: grad_alpha = sum_beta C_{beta alpha} acc_beta
        gx = cm[0] * acc[0] + cm[3] * acc[1] + cm[6] * acc[2] + double(g[0]);
        gy = cm[1] * acc[0] + cm[4] * acc[1] + cm[7] * acc[2] + double(g[1]);
        gz = cm[2] * acc[0] + cm[5] * acc[1] + cm[8] * acc[2] + double(g[2]);
    }
    for (int off = 16; off > 0; off >>= 1) {
        gx += __shfl_down_sync(0xffffffffu, gx, off);
        gy += __shfl_down_sync(0xffffffffu, gy, off);
        gz += __shfl_down_sync(0xffffffffu, gz, off);
    }
    if (lane == 0) {
        part[warp][0] = gx;
        part[warp][1] = gy;
        part[warp][2] = gz;
    }
    __syncthreads();
    if (valid && warp % a.wpa == 0 && lane < 3) {
        double t = 0.0;
        for (int q = 0; q < a.wpa; ++q) t += part[warp + q][lane];
        a.forces[3 * i + lane] = -a.scale * t;
    }
}

template <class T> PrecData<T> &prec(mbd_system *s);
template <> PrecData<double> &prec<double>(mbd_system *s) { return s->f64; }
template <> PrecData<float> &prec<float>(mbd_system *s) { return s->f32; }

}  // namespace

template <class T>
mbd_status launch_force_dipoles_t(mbd_system *s, const double *Y, const double *coef, const int *length, int R,
                                  int ld, int m, T *dpq, int ld2) {
    const int rows = 3 * s->N;
    const size_t n = (size_t)rows * R;
    k_force_dipoles<T><<<(unsigned)((n + 255) / 256), 256, 0, s->stream>>>(rows, Y, coef, length, s->g_d.as<double>(),
                                                                          R, ld, m, dpq, ld2);
    MBD_LAUNCH_CHECK();
    return MBD_OK;
}

template <class T>
mbd_status launch_force_dipoles_w_t(mbd_system *s, const double *w, const double *v, int R, int ld, T *dpq,
                                    int ld2) {
    const int rows = 3 * s->N;
    const size_t n = (size_t)rows * R;
    k_force_dipoles_w<T><<<(unsigned)((n + 255) / 256), 256, 0, s->stream>>>(rows, w, v, s->g_d.as<double>(), R,
                                                                            ld, dpq, ld2);
    MBD_LAUNCH_CHECK();
    return MBD_OK;
}

template <class T>
mbd_status launch_force_gather_t(mbd_system *s, const T *dpq, const T *mesh, int R, int ld2, double scale,
                                 double *forces) {
    PrecData<T> &P = prec<T>(s);
    ForceArgs<T> a;
    a.dpq = dpq;
    a.mesh = mesh;
    a.R = R;
    a.ld2 = ld2;
    a.g.N = s->N;
    a.g.K1 = s->K[0];
    a.g.K2 = s->K[1];
    a.g.K3 = s->K[2];
    a.g.p = s->p;
    for (int b = 0; b < 3; ++b)
        for (int c = 0; c < 3; ++c) a.g.cmat[3 * b + c] = s->K[b] * s->recip[3 * b + c];
    for (int k = 0; k < 9; ++k) a.g.cell[k] = s->cell[k];
    a.top = s->top_d.as<int>();
    a.w = P.w.template as<T>();
    a.dw = P.dw.template as<T>();
    a.d2w = P.d2w.template as<T>();
    a.row = s->row_d.as<int>();
    a.col = s->col_d.as<int>();
    a.dA = P.pairdA.template as<T>();
    a.scale = scale;
    a.forces = forces;
    constexpr int VEC = 16 / (int)sizeof(T);
    a.order = s->order_d.as<int>();
    a.lanes = std::min(32, ld2 / VEC);
    // warps per atom: more for small systems, whose one warp per atom would
    // leave most of the SMs' warp slots empty
    a.wpa = s->N <= 2048 ? 8 : (s->N <= 8192 ? 4 : (s->N <= 65536 ? 2 : 1));
    const int per = kWarps / a.wpa;
    const unsigned grid = (unsigned)((s->N + per - 1) / per);
    switch (s->p) {
#define MBD_FORCE_ORDER(P) \
    case P: k_force_gather<T, P><<<grid, kWarps * 32, 0, s->stream>>>(a); break;
        MBD_SPLINE_ORDERS(MBD_FORCE_ORDER)
#undef MBD_FORCE_ORDER
        default: return MBD_ERR_UNSUPPORTED;
    }
    MBD_LAUNCH_CHECK();
    return MBD_OK;
}

template mbd_status launch_force_dipoles_t<double>(mbd_system *, const double *, const double *, const int *, int, int,
                                                   int, double *, int);
template mbd_status launch_force_dipoles_t<float>(mbd_system *, const double *, const double *, const int *, int, int,
                                                  int, float *, int);
template mbd_status launch_force_dipoles_w_t<double>(mbd_system *, const double *, const double *, int, int,
                                                     double *, int);
template mbd_status launch_force_dipoles_w_t<float>(mbd_system *, const double *, const double *, int, int, float *,
                                                    int);
template mbd_status launch_force_gather_t<double>(mbd_system *, const double *, const double *, int, int, double,
                                                  double *);
template mbd_status launch_force_gather_t<float>(mbd_system *, const float *, const float *, int, int, double,
                                                 double *);

}  // namespace mbd

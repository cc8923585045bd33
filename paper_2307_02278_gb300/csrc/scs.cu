// Self-consistent screening of the atomic polarisabilities (the MBD@rsSCS
// front end).  arXiv 2307.02278 names this step in its review of the MBD model
// (the polarisabilities, made frequency-dependent, are screened by a Dyson-like
// equation solved at a set of frequencies) and keeps it out of its own scope;
// the published range-separated scheme is restated:
//   alpha_i(iu) = alpha_i / (1 + (u/omega_i)^2),  sigma_i(u) = (sqrt(2/pi) alpha_i(iu) / 3)^(1/3)
//   T_SR_ij(u)  = sum'_n (1 - f(|r+n|)) T_GG(r+n; sqrt(sigma_i^2 + sigma_j^2)),  |r+n| < damp_cut
//   T_GG(r; s)  = grad_i grad_j erf(|r|/s)/|r| = c_id I - c_rr r r^T,  f = the Fermi damping s(R; beta)
//   (A(u)^-1 + T_SR(u)) X_c = 1_c  (c = x, y, z),   alpha_i^SCS(iu) = (1/3) sum_c X_c[i, c]
//   C6_i = (3/pi) int_0^inf alpha_i^SCS(iu)^2 du,  omega_i^SCS = 4 C6_i / (3 alpha_i^SCS(0)^2),
//   Rvdw_i^SCS = Rvdw_i (alpha_i^SCS(0) / alpha_i)^(1/3).
//
// GB300 layout: the columns of the solve are (direction c, frequency k), the
// frequency innermost in 32 lanes (k = 0 static, 1..n the quadrature nodes).
// A warp owns an atom, lane k its frequency, and the three directions share
// the lane's tensor.  Mixed systems evaluate T_SR in FP32 inside every product
// from a 16-byte record per pair {r, (1 - f) [r < damp_cut]} and the squared
// widths sigma_j(u_k)^2 (one coalesced row per neighbour): the product then
// costs arithmetic, not a pass over stored tensors (32 x 6 values per pair).
// FP64 systems evaluate T_SR once per call in FP64 and keep it, [nnz][6][32],
// streamed once per step.  Vectors are FP64 [N][3 a][3 c][32]; the search
// direction also in the operator precision for the neighbour gathers.  Jacobi
// preconditioner diag(alpha_i(iu)).  Column sums are deterministic: fixed
// grid, warps take atoms in a fixed stride, block partials summed in block
// order.
#include "mbd_internal.cuh"

#include <algorithm>
#include <cmath>
#include <vector>

namespace mbd {
namespace {

constexpr int kLanes = 32;                  // frequency columns per direction
constexpr int kCols = 3 * kLanes;           // (c, k)
constexpr int kVec = 9 * kLanes;            // values per atom: [a][c][k]
constexpr int kWarps = 8;                   // warps per block
constexpr double kU0 = 0.5;                 // centre of the frequency map (Ha)
constexpr double kPiD = 3.14159265358979323846;

// Gauss-Legendre nodes and weights on (-1, 1) by Newton's method on the
// Legendre polynomial P_n (three-term recurrence), started from the
// asymptotic guesses cos(pi (i - 1/4) / (n + 1/2)); w = 2 / ((1 - t^2) P_n'(t)^2).
void gauss_legendre(int n, std::vector<double> &t, std::vector<double> &w) {
    t.assign(n, 0.0);
    w.assign(n, 0.0);
    for (int i = 0; i < n; ++i) {
        double x = std::cos(kPiD * (i + 0.75) / (n + 0.5));
        double dp = 1.0;
        for (int it = 0; it < 100; ++it) {
            double p0 = 1.0, p1 = x;
            for (int k = 2; k <= n; ++k) {
                const double p2 = ((2.0 * k - 1.0) * x * p1 - (k - 1.0) * p0) / k;
                p0 = p1;
                p1 = p2;
            }
            double pn = n == 1 ? x : p1, pm = n == 1 ? 1.0 : p0;
            dp = n * (x * pn - pm) / (x * x - 1.0);
            const double dx = pn / dp;
            x -= dx;
            if (std::fabs(dx) < 1e-16) break;
        }
        double p0 = 1.0, p1 = x;
        for (int k = 2; k <= n; ++k) {
            const double p2 = ((2.0 * k - 1.0) * x * p1 - (k - 1.0) * p0) / k;
            p0 = p1;
            p1 = p2;
        }
        const double pn = n == 1 ? x : p1, pm = n == 1 ? 1.0 : p0;
        dp = n * (x * pn - pm) / (x * x - 1.0);
        t[n - 1 - i] = x;                    // ascending
        w[n - 1 - i] = 2.0 / ((1.0 - x * x) * dp * dp);
    }
}

struct ScsArgs {
    int N, ncol;
    const double *alpha, *omega, *rvdw, *pos;
    const int *row, *col, *shift;
    double cell[9];
    double damp_cut, damp_beta, damp_d;
    const double *u;            // [32] frequencies (0 beyond ncol)
};

// Per atom and column: 1 / alpha_i(iu_k), alpha_i(iu_k), sigma_i(u_k) and
// sigma_i(u_k)^2 in FP32; zeros beyond ncol.
__global__ void k_scs_atoms(ScsArgs a, double *__restrict__ ainv, double *__restrict__ aiu, double *__restrict__ sig,
                            float *__restrict__ sig2f) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= a.N * kLanes) return;
    const int i = idx / kLanes, k = idx % kLanes;
    double inv = 0.0, au = 0.0, s = 0.0;
    if (k < a.ncol) {
        const double q = a.u[k] / a.omega[i];
        au = a.alpha[i] / (1.0 + q * q);
        inv = 1.0 / au;
        s = cbrt(sqrt(2.0 / kPiD) * au / 3.0);
    }
    ainv[idx] = inv;
    aiu[idx] = au;
    sig[idx] = s;
    sig2f[idx] = float(s * s);
}

// Pair records of the FP32 product: {r_x, r_y, r_z, (1 - f(r)) [r < damp_cut]},
// r = R_i - R_j - n (FP64 from the positions and the image shift); a warp per
// atom, lanes over its entries.
__global__ void k_scs_geometry(ScsArgs a, float4 *__restrict__ geo) {
    const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (i >= a.N) return;
    const double xi = a.pos[3 * i], yi = a.pos[3 * i + 1], zi = a.pos[3 * i + 2];
    for (int e = a.row[i] + lane; e < a.row[i + 1]; e += 32) {
        const int j = a.col[e];
        const int sh = a.shift[e];
        const double n1 = double((sh & 255) - 128), n2 = double(((sh >> 8) & 255) - 128),
                     n3 = double(((sh >> 16) & 255) - 128);
        const double rx = xi - a.pos[3 * j] - (n1 * a.cell[0] + n2 * a.cell[3] + n3 * a.cell[6]);
        const double ry = yi - a.pos[3 * j + 1] - (n1 * a.cell[1] + n2 * a.cell[4] + n3 * a.cell[7]);
        const double rz = zi - a.pos[3 * j + 2] - (n1 * a.cell[2] + n2 * a.cell[5] + n3 * a.cell[8]);
        const double r = sqrt(rx * rx + ry * ry + rz * rz);
        double oms = 0.0;
        if (r < a.damp_cut)
            oms = 1.0 / (1.0 + exp(a.damp_d * (r / (a.damp_beta * (a.rvdw[i] + a.rvdw[j])) - 1.0)));
        geo[e] = make_float4(float(rx), float(ry), float(rz), float(oms));
    }
}

// T_SR per (pair entry, frequency): `parts` warps per atom i walk its entries, 32
// at a time: lane l first takes entry l's geometry and damping, which all
// frequencies share, then lane k evaluates the frequency-k tensor of each entry
// (FP64) and stores it in T.
template <class T>
__global__ void k_scs_tensors(ScsArgs a, const double *__restrict__ sig, T *__restrict__ tsr, int parts) {
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int k = threadIdx.x & 31, i = w / parts, sub = w - i * parts;
    if (i >= a.N) return;
    const double xi = a.pos[3 * i], yi = a.pos[3 * i + 1], zi = a.pos[3 * i + 2];
    const double si = sig[(size_t)i * kLanes + k];
    const int r0 = a.row[i], n = a.row[i + 1] - r0, e1 = r0 + n * (sub + 1) / parts;
    const double kk = 2.0 / sqrt(kPiD);
    for (int eb = r0 + n * sub / parts; eb < e1; eb += 32) {
        const int cnt = min(32, e1 - eb);
        int lj = i;
        double lx = 1.0, ly = 0.0, lz = 0.0, lr2 = 1.0, lr = 1.0, lir = 1.0, loms = 0.0;
        if (k < cnt) {
            lj = a.col[eb + k];
            const int sh = a.shift[eb + k];
            const double n1 = double((sh & 255) - 128), n2 = double(((sh >> 8) & 255) - 128),
                         n3 = double(((sh >> 16) & 255) - 128);
            lx = xi - a.pos[3 * lj] - (n1 * a.cell[0] + n2 * a.cell[3] + n3 * a.cell[6]);
            ly = yi - a.pos[3 * lj + 1] - (n1 * a.cell[1] + n2 * a.cell[4] + n3 * a.cell[7]);
            lz = zi - a.pos[3 * lj + 2] - (n1 * a.cell[2] + n2 * a.cell[5] + n3 * a.cell[8]);
            lr2 = lx * lx + ly * ly + lz * lz;
            lr = sqrt(lr2);
            lir = 1.0 / lr;
            if (lr < a.damp_cut)
                loms = 1.0 / (1.0 + exp(a.damp_d * (lr / (a.damp_beta * (a.rvdw[i] + a.rvdw[lj])) - 1.0)));
        }
        for (int e = 0; e < cnt; ++e) {
            const int j = __shfl_sync(0xffffffffu, lj, e);
            const double rx = __shfl_sync(0xffffffffu, lx, e), ry = __shfl_sync(0xffffffffu, ly, e),
                         rz = __shfl_sync(0xffffffffu, lz, e), r = __shfl_sync(0xffffffffu, lr, e),
                         inv_r = __shfl_sync(0xffffffffu, lir, e), oms = __shfl_sync(0xffffffffu, loms, e);
            double v[6] = {0, 0, 0, 0, 0, 0};
            if (k < a.ncol && oms > 0.0) {
                const double sj = sig[(size_t)j * kLanes + k];
                const double inv_s = 1.0 / sqrt(si * si + sj * sj);
                const double x = r * inv_s;
                const double ke = kk * exp(-x * x) * inv_s;
                const double inv_r2 = inv_r * inv_r;
                const double be = erf(x) * inv_r2 * inv_r - ke * inv_r2;
                const double cid = oms * be;
                const double crr = oms * (3.0 * be - 2.0 * ke * inv_s * inv_s) * inv_r2;
                v[0] = cid - crr * rx * rx;
                v[1] = -crr * rx * ry;
                v[2] = -crr * rx * rz;
                v[3] = cid - crr * ry * ry;
                v[4] = -crr * ry * rz;
                v[5] = cid - crr * rz * rz;
            }
            T *o = tsr + (size_t)(eb + e) * 6 * kLanes + k;
#pragma unroll
            for (int c = 0; c < 6; ++c) o[c * kLanes] = T(v[c]);
        }
    }
}

// Block partial sums of per-lane column values acc[c] (c = 0..2) over the
// block's warps, in warp order: partial[blockIdx.x][c * 32 + lane].
__device__ __forceinline__ void block_columns(const double acc[3], double *__restrict__ partial) {
    __shared__ double s_acc[kWarps][kCols];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int c = 0; c < 3; ++c) s_acc[warp][c * kLanes + lane] = acc[c];
    __syncthreads();
    for (int t = threadIdx.x; t < kCols; t += blockDim.x) {
        double s = 0.0;
        for (int w = 0; w < kWarps; ++w) s += s_acc[w][t];
        partial[(size_t)blockIdx.x * kCols + t] = s;
    }
}

// The FP64 tail of a product for rows t of atom i, the sums over its pairs in
// f: q = A^-1 p + T_SR p and, with PQ, p.q per column.  WPA warps of a block
// share the atom's pairs: their sums are added in order in s_acc and row t is
// warp t mod WPA's.
template <class F, bool PQ, int WPA>
__device__ __forceinline__ void matvec_tail(const F (&acc)[9], F (*s_acc)[9][kLanes], int sub, int lane, int i,
                                            const double *__restrict__ p, const double *__restrict__ ainv,
                                            double *__restrict__ q, double *dot) {
    const double ai = ainv[(size_t)i * kLanes + lane];
    if (WPA > 1) {
#pragma unroll
        for (int t = 0; t < 9; ++t) s_acc[sub][t][lane] = acc[t];
        __syncthreads();
    }
#pragma unroll
    for (int t = 0; t < 9; ++t) {
        if (WPA > 1 && t % WPA != sub) continue;
        F f = acc[t];
        if (WPA > 1) {
            f = s_acc[0][t][lane];
#pragma unroll
            for (int v = 1; v < WPA; ++v) f += s_acc[v][t][lane];
        }
        const size_t o = (size_t)i * kVec + t * kLanes + lane;
        const double pv = p[o];
        const double qv = ai * pv + double(f);
        q[o] = qv;
        if (PQ) dot[t % 3] += pv * qv;
    }
    if (WPA > 1) __syncthreads();
}

// q = (A^-1 + T_SR) p; with PQ, also the block partials of p.q per column.  WPA
// warps per atom (1, or the block's in small systems).
template <class T, bool PQ, int WPA>
__global__ void __launch_bounds__(kWarps * 32) k_scs_matvec(int N, const int *__restrict__ row,
                                                            const int *__restrict__ col, const T *__restrict__ tsr,
                                                            const T *__restrict__ pT, const double *__restrict__ p,
                                                            const double *__restrict__ ainv, double *__restrict__ q,
                                                            double *__restrict__ partial,
                                                            const int *__restrict__ flags) {
    if (flags[1]) return;
    __shared__ T s_acc[WPA > 1 ? WPA : 1][9][kLanes];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sub = WPA == 1 ? 0 : warp;
    const int first = WPA == 1 ? blockIdx.x * kWarps + warp : blockIdx.x, step = WPA == 1 ? gridDim.x * kWarps : gridDim.x;
    double dot[3] = {0.0, 0.0, 0.0};
    for (int i = first; i < N; i += step) {
        T acc[9];
#pragma unroll
        for (int t = 0; t < 9; ++t) acc[t] = T(0);
        const int r0 = row[i], n = row[i + 1] - r0, e1 = r0 + n * (sub + 1) / WPA;
        for (int e = r0 + n * sub / WPA; e < e1; ++e) {
            const int j = col[e];
            const T *te = tsr + (size_t)e * 6 * kLanes + lane;
            const T t0 = te[0], t1 = te[kLanes], t2 = te[2 * kLanes], t3 = te[3 * kLanes], t4 = te[4 * kLanes],
                    t5 = te[5 * kLanes];
            const T *pj = pT + (size_t)j * kVec + lane;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const T x = pj[(0 * 3 + c) * kLanes], y = pj[(1 * 3 + c) * kLanes], z = pj[(2 * 3 + c) * kLanes];
                acc[0 * 3 + c] += t0 * x + t1 * y + t2 * z;
                acc[1 * 3 + c] += t1 * x + t3 * y + t4 * z;
                acc[2 * 3 + c] += t2 * x + t4 * y + t5 * z;
            }
        }
        matvec_tail<T, PQ, WPA>(acc, s_acc, sub, lane, i, p, ainv, q, dot);
    }
    if (PQ) block_columns(dot, partial);
}

// D(x) = erf(x) - (2/sqrt(pi)) x exp(-x^2), the combination the Gaussian
// dipole tensor needs (c_id = D/r^3), in FP32 from e = exp(-x^2):
//   x < 1: its Maclaurin series (2/sqrt(pi)) sum_{n>=1} (-1)^(n+1) 2n x^(2n+1) / (n! (2n+1)),
//          ten terms (truncation below 6e-8 relative), free of the cancellation
//          of the difference at small x;
//   x >= 1: Hastings' rational approximation of erf (Abramowitz & Stegun 7.1.26,
//          |error| <= 1.5e-7), erf = 1 - t (a1 + t (a2 + t (a3 + t (a4 + t a5)))) e,
//          t = 1 / (1 + 0.3275911 x); D >= 0.43 there (relative error below 2.5e-7).
// Two pairs at a time, packed (each operation below is one instruction for
// both); the series is skipped when no lane of the warp needs it.
__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 gauss_dipole_d(const float2 x, const float2 e) {
    const float kk = 1.1283791670955126f;   // 2 / sqrt(pi)
    const float2 den = fma2(f2(0.3275911f), x, f2(1.0f));
    const float2 t = make_float2(__frcp_rn(den.x), __frcp_rn(den.y));
    float2 poly = fma2(t, f2(1.061405429f), f2(-1.453152027f));
    poly = fma2(t, poly, f2(1.421413741f));
    poly = fma2(t, poly, f2(-0.284496736f));
    poly = mul2(t, fma2(t, poly, f2(0.254829592f)));
    float2 d = fma2(mul2(f2(-kk), x), e, fma2(mul2(f2(-1.0f), poly), e, f2(1.0f)));
    if (__any_sync(0xffffffffu, x.x < 1.0f || x.y < 1.0f)) {
        const float2 x2 = mul2(x, x);
        float2 sr = f2(-2.624506592760561e-07f);
        sr = fma2(sr, x2, f2(2.6106934001670845e-06f));
        sr = fma2(sr, x2, f2(-2.334267040149393e-05f));
        sr = fma2(sr, x2, f2(1.8518518518518518e-04f));
        sr = fma2(sr, x2, f2(-1.282051282051282e-03f));
        sr = fma2(sr, x2, f2(7.575757575757576e-03f));
        sr = fma2(sr, x2, f2(-3.7037037037037035e-02f));
        sr = fma2(sr, x2, f2(1.4285714285714285e-01f));
        sr = fma2(sr, x2, f2(-0.4f));
        sr = fma2(sr, x2, f2(0.6666666666666666f));
        const float2 m = mul2(mul2(f2(kk), x), mul2(x2, sr));
        d.x = x.x < 1.0f ? m.x : d.x;
        d.y = x.y < 1.0f ? m.y : d.y;
    }
    return d;
}

// acc += T_SR(g; s2) x for two pairs (components .x and .y): g = {r, 1 - f},
// s2 the squared widths.  A lane beyond the columns has s2 = 0 and x = 0 (its
// width is floored, its terms vanish with x); a pair beyond the cutoff has
// 1 - f = 0; r is never zero.
__device__ __forceinline__ void pair_apply(const float4 ga, const float4 gb, float2 s2, const float2 x[9],
                                           float2 acc[9]) {
    const float kk = 1.1283791670955126f;   // 2 / sqrt(pi)
    const float2 gx = make_float2(ga.x, gb.x), gy = make_float2(ga.y, gb.y), gz = make_float2(ga.z, gb.z),
                 gw = make_float2(ga.w, gb.w);
    const float2 r2 = fma2(gx, gx, fma2(gy, gy, mul2(gz, gz)));
    const float2 inv_r = make_float2(rsqrtf(r2.x), rsqrtf(r2.y));
    const float2 inv_s = make_float2(rsqrtf(fmaxf(s2.x, 1e-30f)), rsqrtf(fmaxf(s2.y, 1e-30f)));
    const float2 inv_r2 = mul2(inv_r, inv_r);
    const float2 xr = mul2(mul2(r2, inv_r), inv_s);
    const float2 xx = mul2(xr, xr);
    const float2 e = make_float2(expf(-xx.x), expf(-xx.y));
    const float2 ke = mul2(mul2(f2(kk), e), inv_s);
    const float2 base = mul2(mul2(gauss_dipole_d(xr, e), inv_r), inv_r2);
    const float2 cid = mul2(gw, base);
    const float2 w = mul2(mul2(f2(-2.0f), ke), mul2(inv_s, inv_s));
    const float2 mcrr = mul2(mul2(mul2(f2(-1.0f), gw), fma2(f2(3.0f), base, w)), inv_r2);   // -c_rr
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float2 px = x[0 * 3 + c], py = x[1 * 3 + c], pz = x[2 * 3 + c];
        const float2 rd = mul2(mcrr, fma2(gx, px, fma2(gy, py, mul2(gz, pz))));
        acc[0 * 3 + c] = fma2(gx, rd, fma2(cid, px, acc[0 * 3 + c]));
        acc[1 * 3 + c] = fma2(gy, rd, fma2(cid, py, acc[1 * 3 + c]));
        acc[2 * 3 + c] = fma2(gz, rd, fma2(cid, pz, acc[2 * 3 + c]));
    }
}

// The same product with T_SR evaluated in FP32 per (pair, frequency):
//   s^2 = sigma_i^2 + sigma_j^2, x = r/s, ke = (2/sqrt(pi)) exp(-x^2)/s,
//   c_id = (1 - f) D(x)/r^3,  c_rr = (1 - f) (3 D(x)/r^3 - 2 ke/s^2)/r^2,
//   T_SR p = c_id p - c_rr r (r . p).
// Two pairs per packed instruction.  WPA warps share an atom: each walks a
// contiguous part of its entries (neighbour indices 32 at a time, one per
// lane), the parts are added in order in shared memory and the warps share out
// the nine rows of the FP64 tail.
// Bound: instruction issue (FP32) on large systems (12,000 atoms: 9.3 -> 7.7 ms
// per call); on small ones the chain of dependent loads along an atom's
// entries, which WPA = 8 cuts.
template <bool PQ, int WPA>
__global__ void __launch_bounds__(kWarps * 32, 3) k_scs_matvec_fly(int N, const int *__restrict__ order,
                                                                   const int *__restrict__ row,
                                                                   const int *__restrict__ col,
                                                                   const float4 *__restrict__ geo,
                                                                   const float *__restrict__ sig2,
                                                                   const float *__restrict__ pT,
                                                                   const double *__restrict__ p,
                                                                   const double *__restrict__ ainv,
                                                                   double *__restrict__ q,
                                                                   double *__restrict__ partial,
                                                                   const int *__restrict__ flags) {
    if (flags[1]) return;                       // converged: the call's remaining launches do nothing
    static_assert(WPA == 1 || WPA == kWarps, "a warp or a block per atom");
    __shared__ float s_acc[WPA > 1 ? WPA : 1][9][kLanes];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int first = WPA == 1 ? blockIdx.x * kWarps + warp : blockIdx.x, step = WPA == 1 ? gridDim.x * kWarps : gridDim.x;
    double dot[3] = {0.0, 0.0, 0.0};
    for (int w = first; w < N; w += step) {
        const int i = order[w];
        float2 acc[9];
#pragma unroll
        for (int t = 0; t < 9; ++t) acc[t] = make_float2(0.0f, 0.0f);
        const float si2 = sig2[(size_t)i * kLanes + lane];
        const int r0 = row[i], n = row[i + 1] - r0, sub = WPA == 1 ? 0 : warp;
        const int e0 = r0 + n * sub / WPA, e1 = r0 + n * (sub + 1) / WPA;
        for (int eb = e0; eb < e1; eb += 32) {
            const int cnt = min(32, e1 - eb);
            const int cv = lane < cnt ? col[eb + lane] : i;
            for (int k = 0; k < cnt; k += 2) {
                const bool two = k + 1 < cnt;
                const int ja = __shfl_sync(0xffffffffu, cv, k), jb = __shfl_sync(0xffffffffu, cv, two ? k + 1 : k);
                const float4 ga = geo[eb + k], gb = two ? geo[eb + k + 1] : make_float4(1.f, 0.f, 0.f, 0.f);
                const float2 s2 =
                    make_float2(si2 + sig2[(size_t)ja * kLanes + lane], si2 + sig2[(size_t)jb * kLanes + lane]);
                const float *pa = pT + (size_t)ja * kVec + lane, *pb = pT + (size_t)jb * kVec + lane;
                float2 x[9];
#pragma unroll
                for (int t = 0; t < 9; ++t) x[t] = make_float2(pa[t * kLanes], pb[t * kLanes]);
                pair_apply(ga, gb, s2, x, acc);
            }
        }
        float f[9];
#pragma unroll
        for (int t = 0; t < 9; ++t) f[t] = acc[t].x + acc[t].y;
        matvec_tail<float, PQ, WPA>(f, s_acc, sub, lane, i, p, ainv, q, dot);
    }
    if (PQ) block_columns(dot, partial);
}

// Sum of one column of the block partials: lane l adds the blocks l, l + 32,
// ... in order, then a fixed shuffle tree.
__device__ __forceinline__ double column_sum(const double *__restrict__ partial, int nblk, int colx) {
    double s = 0.0;
    for (int b = threadIdx.x; b < nblk; b += 32) s += partial[(size_t)b * kCols + colx];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

// CG scalars, a warp per column.  st[0..95] rho = r.z, st[96..191] alpha step,
// st[192..287] beta, st[288..383] r.r; flags[0] set when p.q <= 0 on a live
// column, flags[1] when every column has converged, flags[2] the iterations
// taken (so that the host can queue several iterations without asking).
__global__ void k_scs_alpha(const double *__restrict__ partial, int nblk, double *__restrict__ st,
                            int *__restrict__ flags) {
    if (flags[1]) return;
    const int t = blockIdx.x;
    const double g = column_sum(partial, nblk, t);
    if (threadIdx.x != 0) return;
    const double rho = st[t];
    double al = 0.0;
    if (rho > 0.0) {
        if (g > 0.0) al = rho / g;
        else atomicOr(flags, 1);
    }
    st[kCols + t] = al;
}
// beta, and by the last of its warps to finish the convergence: ||r_c,k|| <=
// tol ||1_c|| = tol sqrt(N) on every live column; worst[0] the largest relative
// residual (NaN when one is not finite, which ends the iteration too).
__global__ void k_scs_beta(const double *__restrict__ partial, int nblk, double *__restrict__ st, int first, int ncol,
                           double bnorm2, double tol, int *__restrict__ flags, double *__restrict__ worst) {
    if (flags[1]) return;
    const int t = blockIdx.x, k = threadIdx.x;
    const double rho_new = column_sum(partial, nblk, t);
    const double rr_t = column_sum(partial + (size_t)nblk * kCols, nblk, t);
    int last = 0;
    if (k == 0) {
        const double rho_old = st[t];
        st[2 * kCols + t] = (first || rho_old <= 0.0) ? 0.0 : rho_new / rho_old;
        st[t] = rho_new;
        st[3 * kCols + t] = rr_t;
        __threadfence();
        last = atomicAdd(&flags[4], 1) == kCols - 1;
    }
    if (!__shfl_sync(0xffffffffu, last, 0)) return;
    __threadfence();
    double w = 0.0;
    int bad = 0;
    if (k < ncol)
        for (int c = 0; c < 3; ++c) {
            const double rr = __ldcg(&st[3 * kCols + c * kLanes + k]);
            bad |= isfinite(rr) ? 0 : 1;
            w = fmax(w, sqrt(fmax(rr, 0.0) / bnorm2));
        }
    for (int o = 16; o > 0; o >>= 1) {
        w = fmax(w, __shfl_xor_sync(0xffffffffu, w, o));
        bad |= __shfl_xor_sync(0xffffffffu, bad, o);
    }
    if (k == 0) {
        worst[0] = bad ? nan("") : w;
        flags[4] = 0;
        if (!first) flags[2] += 1;
        if (bad || w <= tol) flags[1] = 1;
    }
}

// x += a p, r -= a q (first: x = x0 = p, r = b - q), with the block partials of
// r.z (z = alpha_i(iu) r) and r.r per column.
__global__ void __launch_bounds__(kWarps * 32) k_scs_update(int N, int first, const double *__restrict__ st,
                                                            const double *__restrict__ p,
                                                            const double *__restrict__ q,
                                                            const double *__restrict__ aiu, double *__restrict__ x,
                                                            double *__restrict__ r, double *__restrict__ partial,
                                                            int nblk, const int *__restrict__ flags) {
    if (flags[1]) return;
    const int lane = threadIdx.x & 31;
    const int gw = blockIdx.x * kWarps + (threadIdx.x >> 5), nw = gridDim.x * kWarps;
    double rz[3] = {0.0, 0.0, 0.0}, rr[3] = {0.0, 0.0, 0.0};
    double al[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) al[c] = first ? 0.0 : st[kCols + c * kLanes + lane];
    for (int w = gw; w < 3 * N; w += nw) {      // a warp per (atom, a): its three directions c
        const int i = w / 3, ax = w - 3 * i;
        const double zscale = aiu[(size_t)i * kLanes + lane];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const size_t o = (size_t)i * kVec + (3 * ax + c) * kLanes + lane;
            double rv;
            if (first) {
                x[o] = p[o];
                rv = (ax == c && zscale > 0.0 ? 1.0 : 0.0) - q[o];
            } else {
                x[o] += al[c] * p[o];
                rv = r[o] - al[c] * q[o];
            }
            r[o] = rv;
            rz[c] += rv * (rv * zscale);
            rr[c] += rv * rv;
        }
    }
    block_columns(rz, partial);
    __syncthreads();
    block_columns(rr, partial + (size_t)nblk * kCols);
}

// p = z + beta p (first: p = x0 = alpha_i(iu) delta_ac), and its copy in T.
template <class T>
__global__ void k_scs_direction(int N, int mode, const double *__restrict__ st, const double *__restrict__ r,
                                const double *__restrict__ aiu, double *__restrict__ p, T *__restrict__ pT,
                                const int *__restrict__ flags) {
    if (flags[1]) return;
    const size_t o = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (o >= (size_t)N * kVec) return;
    const int lane = (int)(o % kLanes), t = (int)((o / kLanes) % 9), i = (int)(o / kVec);
    const int a = t / 3, c = t % 3;
    const double zs = aiu[(size_t)i * kLanes + lane];
    double v;
    if (mode == 0) v = (a == c) ? zs : 0.0;                                       // x0 = A 1_c
    else v = r[o] * zs + st[2 * kCols + c * kLanes + lane] * p[o];
    p[o] = v;
    pT[o] = T(v);
}

// Screened outputs per atom from the solutions x.
__global__ void k_scs_finish(int N, int ncol, const double *__restrict__ x, const double *__restrict__ alpha,
                             const double *__restrict__ rvdw, const double *__restrict__ wq,
                             double *__restrict__ out, double *__restrict__ aiu, int *__restrict__ flags) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    double a0 = 0.0, c6 = 0.0;
    for (int k = 0; k < ncol; ++k) {
        const size_t b = (size_t)i * kVec + k;
        const double ak = (x[b + 0 * kLanes] + x[b + 4 * kLanes] + x[b + 8 * kLanes]) / 3.0;
        aiu[(size_t)k * N + i] = ak;
        if (!isfinite(ak)) flags[3] = 1;
        if (k == 0) a0 = ak;
        else c6 += wq[k] * ak * ak;
    }
    c6 *= 3.0 / kPiD;
    out[i] = a0;
    out[N + i] = 4.0 * c6 / (3.0 * a0 * a0);
    out[2 * N + i] = rvdw[i] * cbrt(a0 / alpha[i]);
    out[3 * N + i] = c6;
    for (int q = 0; q < 4; ++q)
        if (!isfinite(out[q * N + i])) flags[3] = 1;
}

template <class T>
mbd_status screen(mbd_system *s, int n_freq, double tol, int max_iter, double *alpha_out, double *omega_out,
                  double *rvdw_out, double *c6_out, double *aiu_out, int32_t *iters_out, double *res_out) {
    const int N = s->N, ncol = n_freq + 1;
    const cudaStream_t st = s->stream;
    std::vector<double> t, w;
    gauss_legendre(n_freq, t, w);
    std::vector<double> u(kLanes, 0.0), wq(kLanes, 0.0);
    for (int k = 0; k < n_freq; ++k) {
        u[k + 1] = kU0 * (1.0 + t[k]) / (1.0 - t[k]);
        wq[k + 1] = w[k] * 2.0 * kU0 / ((1.0 - t[k]) * (1.0 - t[k]));
    }
    const long long nnz = s->nnz;
    constexpr bool kFly = sizeof(T) == 4;   // FP32 operator: T_SR evaluated inside each product
    const size_t nv = (size_t)N * kVec;
    // persistent grid: the resident blocks of the product kernel on every SM
    int per_sm = 0;
    if constexpr (kFly)
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_scs_matvec_fly<true, 1>, kWarps * 32, 0);
    else
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_scs_matvec<T, true, 1>, kWarps * 32, 0);
    cudaGetLastError();
    per_sm = std::max(1, std::min(8, per_sm));
    const int per_block = (N + kWarps - 1) / kWarps, sms = std::max(1, s->num_sms);
    // fewer atoms than resident warps: a block per atom
    const bool split = N <= per_sm * sms * kWarps;
    const int nblk = std::max(1, std::min(split ? N : per_block, per_sm * sms));
    // the vector updates stream from L2 and HBM: more blocks, more loads in flight
    const int ublk = std::max(1, std::min((3 * N + kWarps - 1) / kWarps, 5 * sms));
    // one allocation for the call, cut into its arrays
    DevBuf mem;
    size_t used = 0;
    auto take = [&](size_t bytes) {
        const size_t at = used;
        used += (bytes + 255) / 256 * 256;
        return at;
    };
    const size_t D = sizeof(double), col = (size_t)N * kLanes;
    const size_t o_q = take(2 * kLanes * D), o_al = take(N * D), o_om = take(N * D), o_ainv = take(col * D),
                 o_aiuc = take(col * D), o_sig = take(col * D), o_sig2 = take(col * sizeof(float)),
                 o_pair = take(std::max<size_t>(1, (size_t)nnz) * (kFly ? sizeof(float4) : 6 * kLanes * sizeof(T))),
                 o_x = take(nv * D), o_r = take(nv * D), o_p = take(nv * D), o_qv = take(nv * D),
                 o_pT = take(nv * sizeof(T)), o_part = take((size_t)std::max(nblk, 2 * ublk) * kCols * D), o_st = take(4 * kCols * D),
                 o_flag = take(6 * sizeof(int) + D), o_out = take(4 * (size_t)N * D), o_aiu = take((size_t)ncol * N * D);
    MBD_TRY(mem.ensure(used));
    unsigned char *m0 = mem.as<unsigned char>();
    auto dbl = [&](size_t at) { return reinterpret_cast<double *>(m0 + at); };
    double *d_u = dbl(o_q), *d_wq = d_u + kLanes, *d_ainv = dbl(o_ainv), *d_aiu_c = dbl(o_aiuc), *d_sig = dbl(o_sig),
           *d_x = dbl(o_x), *d_r = dbl(o_r), *d_p = dbl(o_p), *d_q = dbl(o_qv), *d_part = dbl(o_part),
           *st_d = dbl(o_st), *d_out = dbl(o_out), *d_aiu = dbl(o_aiu);
    float *d_sig2 = reinterpret_cast<float *>(m0 + o_sig2);
    T *d_pT = reinterpret_cast<T *>(m0 + o_pT);
    int *d_flag = reinterpret_cast<int *>(m0 + o_flag);
    double *d_worst = reinterpret_cast<double *>(d_flag + 6);
    u.insert(u.end(), wq.begin(), wq.end());
    MBD_CUDA_TRY(cudaMemcpyAsync(d_u, u.data(), 2 * kLanes * D, cudaMemcpyHostToDevice, st));
    MBD_CUDA_TRY(cudaMemcpyAsync(m0 + o_al, s->alpha.data(), N * D, cudaMemcpyHostToDevice, st));
    MBD_CUDA_TRY(cudaMemcpyAsync(m0 + o_om, s->omega.data(), N * D, cudaMemcpyHostToDevice, st));
    MBD_CUDA_TRY(cudaMemsetAsync(d_flag, 0, 6 * sizeof(int) + D, st));
    MBD_CUDA_TRY(cudaMemsetAsync(st_d, 0, 4 * kCols * D, st));

    ScsArgs a{};
    a.N = N;
    a.ncol = ncol;
    a.alpha = dbl(o_al);
    a.omega = dbl(o_om);
    a.rvdw = s->rvdw_d.as<double>();
    a.pos = s->pos_d.as<double>();
    a.row = s->row_d.as<int>();
    a.col = s->col_d.as<int>();
    a.shift = s->shift_d.as<int>();
    for (int c = 0; c < 9; ++c) a.cell[c] = s->cell[c];
    a.damp_cut = s->damp_cut;
    a.damp_beta = s->damp_beta;
    a.damp_d = s->damp_d;
    a.u = d_u;

    k_scs_atoms<<<(N * kLanes + 255) / 256, 256, 0, st>>>(a, d_ainv, d_aiu_c, d_sig, d_sig2);
    MBD_LAUNCH_CHECK();
    if constexpr (kFly)
        k_scs_geometry<<<(N + 7) / 8, 256, 0, st>>>(a, reinterpret_cast<float4 *>(m0 + o_pair));
    else
        k_scs_tensors<T><<<split ? N : (N + 7) / 8, 256, 0, st>>>(a, d_sig, reinterpret_cast<T *>(m0 + o_pair),
                                                                  split ? kWarps : 1);
    MBD_LAUNCH_CHECK();
    auto matvec = [&](bool pq) {
        if constexpr (kFly) {
            auto kern = split ? (pq ? k_scs_matvec_fly<true, kWarps> : k_scs_matvec_fly<false, kWarps>)
                              : (pq ? k_scs_matvec_fly<true, 1> : k_scs_matvec_fly<false, 1>);
            kern<<<nblk, kWarps * 32, 0, st>>>(N, s->order_d.as<int>(), a.row, a.col,
                                               reinterpret_cast<const float4 *>(m0 + o_pair), d_sig2, d_pT, d_p, d_ainv,
                                               d_q, d_part, d_flag);
        } else {
            auto kern = split ? (pq ? k_scs_matvec<T, true, kWarps> : k_scs_matvec<T, false, kWarps>)
                              : (pq ? k_scs_matvec<T, true, 1> : k_scs_matvec<T, false, 1>);
            kern<<<nblk, kWarps * 32, 0, st>>>(N, a.row, a.col, reinterpret_cast<const T *>(m0 + o_pair), d_pT, d_p,
                                               d_ainv, d_q, d_part, d_flag);
        }
    };

    const unsigned vgrid = (unsigned)((nv + 255) / 256);
    const double bnorm2 = (double)N;
    auto update = [&](int first) {              // x, r, their sums, beta, convergence, the next direction
        k_scs_update<<<ublk, kWarps * 32, 0, st>>>(N, first, st_d, d_p, d_q, d_aiu_c, d_x, d_r, d_part, ublk, d_flag);
        k_scs_beta<<<kCols, 32, 0, st>>>(d_part, ublk, st_d, first, ncol, bnorm2, tol, d_flag, d_worst);
        k_scs_direction<T><<<vgrid, 256, 0, st>>>(N, 1, st_d, d_r, d_aiu_c, d_p, d_pT, d_flag);
    };
    // x0 = A 1_c, r0 = 1_c - M x0, p0 = z0
    k_scs_direction<T><<<vgrid, 256, 0, st>>>(N, 0, st_d, d_r, d_aiu_c, d_p, d_pT, d_flag);
    matvec(false);
    update(1);
    MBD_LAUNCH_CHECK();

    // iterations are queued four at a time; those after convergence do nothing
    struct {
        int flag[6];                            // see k_scs_alpha; [4] is k_scs_beta's counter
        double worst;
    } h{};
    auto read = [&]() -> mbd_status {
        MBD_CUDA_TRY(cudaMemcpyAsync(&h, d_flag, 6 * sizeof(int) + D, cudaMemcpyDeviceToHost, st));
        MBD_CUDA_TRY(cudaStreamSynchronize(st));
        return std::isfinite(h.worst) ? MBD_OK : MBD_ERR_NONFINITE;
    };
    constexpr int kAhead = 4;
    for (int iters = 0; iters < max_iter;) {
        const int n = std::min(kAhead, max_iter - iters);
        for (int k = 0; k < n; ++k) {
            matvec(true);
            k_scs_alpha<<<kCols, 32, 0, st>>>(d_part, nblk, st_d, d_flag);
            update(0);
        }
        MBD_LAUNCH_CHECK();
        iters += n;
        MBD_TRY(read());
        if (h.flag[0]) return MBD_ERR_NOT_POSITIVE_DEFINITE;   // a stalled column need never converge
        if (h.flag[1]) break;
    }
    k_scs_finish<<<(N + 127) / 128, 128, 0, st>>>(N, ncol, d_x, a.alpha, a.rvdw, d_wq, d_out, d_aiu, d_flag);
    MBD_LAUNCH_CHECK();
    MBD_TRY(read());
    if (h.flag[3]) return MBD_ERR_NONFINITE;
    double *const to[4] = {alpha_out, omega_out, rvdw_out, c6_out};
    for (int q = 0; q < 4; ++q)
        if (to[q]) MBD_CUDA_TRY(cudaMemcpyAsync(to[q], d_out + (size_t)q * N, N * D, cudaMemcpyDeviceToHost, st));
    if (aiu_out) MBD_CUDA_TRY(cudaMemcpyAsync(aiu_out, d_aiu, (size_t)ncol * N * D, cudaMemcpyDeviceToHost, st));
    MBD_CUDA_TRY(cudaStreamSynchronize(st));
    if (iters_out) *iters_out = h.flag[2];
    if (res_out) *res_out = h.worst;
    return MBD_OK;
}

}  // namespace
}  // namespace mbd

extern "C" mbd_status mbd_scs_screen(mbd_system *s, int32_t n_freq, double tol, int32_t max_iter, double *alpha_out,
                                     double *omega_out, double *r_vdw_out, double *c6_out, double *alpha_iu_out,
                                     int32_t *iterations, double *residual) {
    if (!s || !alpha_out || !omega_out || !r_vdw_out) return MBD_ERR_INVALID_ARG;
    if (n_freq < 1 || n_freq > 31 || !(tol > 0.0) || !std::isfinite(tol) || max_iter < 0 || max_iter > 100000)
        return MBD_ERR_INVALID_ARG;
    MBD_TRY(mbd::check_geometry(s));
    if (s->precision == MBD_FP64)
        return mbd::screen<double>(s, n_freq, tol, max_iter, alpha_out, omega_out, r_vdw_out, c6_out, alpha_iu_out,
                                   iterations, residual);
    return mbd::screen<float>(s, n_freq, tol, max_iter, alpha_out, omega_out, r_vdw_out, c6_out, alpha_iu_out,
                              iterations, residual);
}

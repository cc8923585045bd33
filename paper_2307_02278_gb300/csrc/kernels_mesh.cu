// Per-step operator kernels: SPME spreading (Eq. dipolarr), the batched 3D FFT
// convolution with the influence function (Eq. spme), and the fused field
// kernel (SPME gather + real-space pairs + self term, Eqs. spme, fld_ewald,
// fld_ewald1) with the Lanczos epilogue l_k = Omega y_k + Diag(g) E*_k and
// a_k = y_k^T l_k (Eqs. lk3, recurs2).
#include "fft.cuh"

#include <algorithm>

namespace mbd {

namespace {

// ---------------------------------------------------------------- spreading
// The dipole array D(k) = sum_j d_j . grad W_j(k) (Eq. dipolarr) from the
// pencil records, built once per geometry in a fixed atom order, so every mesh
// value is a sum in a fixed order: spreading is deterministic and writes each
// mesh point once.

// Pencil records (PencilRec): a thread per mesh point (k1, k2, k3) finds the
// atoms whose top stencil point is (k1 + t1, k2 + t2, k3), t1, t2 < p (mod K),
// in the bricks that hold those tops, visited in a fixed order (candidate
// bricks in order, atoms of a brick by index), so the records of a point come
// in a fixed order.  FILL = false counts, FILL = true writes e0 and e1 from
// the FP64 stencil weights.
template <class T, bool FILL>
__global__ void k_pencil_rows(Geom g, BinView B, const int *__restrict__ top, const double *__restrict__ w64,
                              const double *__restrict__ dw64, int *__restrict__ cnt_or_row,
                              PencilRec<T> *__restrict__ rec) {
    const size_t npts = (size_t)g.K1 * g.K2 * g.K3;
    const size_t pt = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (pt >= npts) return;
    const int g3 = (int)(pt % g.K3), g2 = (int)((pt / g.K3) % g.K2), g1 = (int)(pt / ((size_t)g.K2 * g.K3));
    const int p = g.p;
    // bricks holding tops in [g1, g1 + p - 1] (and likewise along k2), the one holding k3
    const int b1 = g1 / B.bs1, b2 = g2 / B.bs2, b3 = g3 / B.bs3;
    const int n1 = min(B.nb1, (g1 + p - 1) / B.bs1 - b1 + 1);
    const int n2 = min(B.nb2, (g2 + p - 1) / B.bs2 - b2 + 1);
    int c = 0;
    const int base = FILL ? cnt_or_row[pt] : 0;
    for (int c1 = 0; c1 < n1; ++c1) {
        const int t1b = (b1 + c1) % B.nb1;
        for (int c2 = 0; c2 < n2; ++c2) {
            const int t2b = (b2 + c2) % B.nb2;
            const int bin = (t1b * B.nb2 + t2b) * B.nb3 + b3;
            for (int s = B.start[bin]; s < B.start[bin + 1]; ++s) {
                const int j = B.atoms[s];
                if (top[3 * j + 2] != g3) continue;
                int u1 = top[3 * j] - g1;
                if (u1 < 0) u1 += g.K1;
                int u2 = top[3 * j + 1] - g2;
                if (u2 < 0) u2 += g.K2;
                if (u1 >= p || u2 >= p) continue;
                if (FILL) {
                    const double *w = w64 + (size_t)3 * p * j, *dw = dw64 + (size_t)3 * p * j;
                    const double m1 = w[u1], m2 = w[p + u2], n1v = dw[u1], n2v = dw[p + u2];
                    const double a = n1v * m2, b = m1 * n2v, cc = m1 * m2;
                    PencilRec<T> r;
#pragma unroll
                    for (int al = 0; al < 3; ++al) {
                        r.e0[al] = T(g.cmat[al] * a + g.cmat[3 + al] * b);
                        r.e1[al] = T(g.cmat[6 + al] * cc);
                    }
                    r.atom = j;
                    r.top3 = g3;
                    rec[base + c] = r;
                }
                ++c;
            }
        }
    }
    if (!FILL) cnt_or_row[pt] = c;
}

// The k3 stencil of each atom for the pencil spreading: k3w[j][t] = M3(t),
// k3w[j][p + t] = M3'(t).
template <class T>
__global__ void k_pencil_k3w(int N, int p, const double *__restrict__ w64, const double *__restrict__ dw64,
                             T *__restrict__ k3w) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= 2 * p * N) return;
    const int j = idx / (2 * p), t = idx % (2 * p);
    k3w[idx] = T(t < p ? w64[(size_t)(3 * j + 2) * p + t] : dw64[(size_t)(3 * j + 2) * p + t - p]);
}

// Exclusive scan of n counts (blocks of 4096), the block sums, and the fix-up.  Sums
// stop at 2^31 - 1 instead of wrapping to negative starts: kernels may read the
// starts of a scan that has overflowed before the host sees its total, -1.
__device__ __forceinline__ int sat_add(int a, int b) {   // a, b >= 0
    const unsigned s = (unsigned)a + (unsigned)b;
    return s > 0x7fffffffu ? 0x7fffffff : (int)s;
}
__global__ void __launch_bounds__(1024) k_scan_block(const int *__restrict__ in, int *__restrict__ out,
                                                     int *__restrict__ bsum, int n) {
    __shared__ int sh[1024];
    const int tid = threadIdx.x;
    const long long base = (long long)blockIdx.x * 4096 + tid * 4;
    int v[4], tsum = 0;
    for (int k = 0; k < 4; ++k) {
        v[k] = (base + k < n) ? in[base + k] : 0;
        tsum = sat_add(tsum, v[k]);
    }
    sh[tid] = tsum;
    __syncthreads();
    for (int off = 1; off < 1024; off <<= 1) {
        const int t = tid >= off ? sh[tid - off] : 0;
        __syncthreads();
        sh[tid] = sat_add(sh[tid], t);
        __syncthreads();
    }
    int excl = tid > 0 ? sh[tid - 1] : 0;
    for (int k = 0; k < 4; ++k) {
        if (base + k < n) out[base + k] = excl;
        excl = sat_add(excl, v[k]);
    }
    if (tid == 1023) bsum[blockIdx.x] = sh[1023];
}
__global__ void k_scan_sums(int *__restrict__ bsum, int nb, int *__restrict__ total) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    long long acc = 0;
    for (int b = 0; b < nb; ++b) {
        const int t = bsum[b];
        bsum[b] = (int)min(acc, 0x7fffffffLL);
        acc += t;
    }
    *total = acc >= 0x7fffffffLL ? -1 : (int)acc;
}
__global__ void k_scan_add(int *__restrict__ out, const int *__restrict__ bsum, int n) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = sat_add(out[i], bsum[i / 4096]);
}

// The spreading alone, for mesh lengths without a fused pass and for the
// stage-level call: a tile of W complex columns per nseg warps (nseg = 1: per warp of a
// block of four), each warp walking its segment of the tile's pencils downwards
// and, after a barrier, adding the P - 1 rows below it to the segment before (cyclically),
// which the block has written.  Bound: a warp's chain of records where there
// are few tiles.  12^3 x 64 probes and 3000 atoms: 262 us per launch with one segment and
// 144 with two, 15^3 x 16 203 and 78 with three.
template <class T, int P>
__global__ void __launch_bounds__(256) k_spread_pencil(SpreadArgs<T> a, unsigned ncols, int nseg) {
    constexpr int PPL = spread_ppl<T>(), W = spread_w<T>();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, K = a.K3, V = a.ld / 2;
    const unsigned c = (blockIdx.x * (blockDim.x >> 5) + warp) / nseg * W + lane * PPL / 2;
    const bool on = c < ncols;
    const int seg = warp % nseg, r0 = on ? seg * K / nseg : 0, r1 = on ? (seg + 1) * K / nseg : 0;
    const unsigned pen = (on ? c : 0) / V;
    const int pr0 = on ? 2 * (int)(c - pen * V) + (lane * PPL & 1) : 0;
    const int *rp = a.prow + (size_t)pen * K;
    T *out = a.mesh + (size_t)pen * K * a.ld + pr0;
    pencil_walk<T, P, PPL, true>(
        a.d + pr0, a.ld, a.prec, a.k3w, r0, r1, rp[r0], rp[r1], [&](int t) { return rp[t]; },
        [&](int row, const T *v) {
            T o[PPL];
#pragma unroll
            for (int e = 0; e < PPL; ++e) o[e] = pr0 + e < a.R ? v[e] : T(0);
            vstore<T, PPL>(out + (size_t)row * a.ld, o);
        },
        [] { __syncthreads(); },
        [&](int row, const T *v) {
            if (!on) return;
            T *o = out + (size_t)(row < 0 ? row + K : row) * a.ld;
            T y[PPL];
            vload<T, PPL>(o, y);
#pragma unroll
            for (int e = 0; e < PPL; ++e) y[e] += pr0 + e < a.R ? v[e] : T(0);
            vstore<T, PPL>(o, y);
        });
}

// One radix-R Stockham stage over the K rows of a K x W tile in shared memory
// (R compile-time, so the butterfly stays in registers).
template <class F, int R, bool INV>
__device__ __forceinline__ void stockham_stage(const Cx<F> *__restrict__ in, Cx<F> *__restrict__ out,
                                               const typename TwOf<F>::type *__restrict__ tw, int K, int W, int Ns) {
    const int nb = K / R;
    const int step = K / (Ns * R);
    for (int idx = threadIdx.x; idx < nb * W; idx += blockDim.x) {
        const int j = idx / W, col = idx - j * W;
        Cx<F> v[R];
#pragma unroll
        for (int q = 0; q < R; ++q) v[q] = cld(in + (j + q * nb) * W + col);
        const int jm = j % Ns;
        if (jm != 0) {
#pragma unroll
            for (int q = 1; q < R; ++q) v[q] = ctw<INV>(v[q], tw[q * jm * step]);
        }
        Dft<F, R, INV>::run(v);
        const int base = (j / Ns) * Ns * R + jm;
#pragma unroll
        for (int q = 0; q < R; ++q) cst(out + (base + q * Ns) * W + col, v[q]);
    }
}

// Mixed-radix Stockham passes over the K rows of a K x W tile held in shared
// memory; returns the buffer that holds the result (natural order).
template <class T, class F, bool INV>
__device__ Cx<F> *stockham(Cx<F> *in, Cx<F> *out, const FFTArgs<T> &a, const typename TwOf<F>::type *tw) {
    int Ns = 1;
    for (int s = 0; s < a.nst; ++s) {
        const int R = (int)((a.radices >> (4 * s)) & 15ull);
        switch (R) {
            case 2: stockham_stage<F, 2, INV>(in, out, tw, a.K, a.W, Ns); break;
            case 3: stockham_stage<F, 3, INV>(in, out, tw, a.K, a.W, Ns); break;
            case 4: stockham_stage<F, 4, INV>(in, out, tw, a.K, a.W, Ns); break;
            case 5: stockham_stage<F, 5, INV>(in, out, tw, a.K, a.W, Ns); break;
            default: stockham_stage<F, 8, INV>(in, out, tw, a.K, a.W, Ns); break;
        }
        __syncthreads();
        Cx<F> *t = in;
        in = out;
        out = t;
        Ns *= R;
    }
    return in;
}

// One 1D FFT pass along the middle axis of [outer][K][inner] (values Cx<F>)
// for the lengths without a compile-time pass; MODE 0 forward, 1 inverse, 2
// forward, multiplied by G(k1, k2, k3), inverse.  A tile is W columns of one
// outer slab or, where a slab has fewer than W (one or two probes along k3), the
// whole columns of `slabs` slabs, which are contiguous.
template <class T, class F, int MODE>
__global__ void __launch_bounds__(256) k_fft_pass(FFTArgs<T> a, unsigned outer, int slabs) {
    using C = Cx<F>;
    using TW = typename TwOf<F>::type;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TW *tw = reinterpret_cast<TW *>(smem_raw);
    C *b0 = reinterpret_cast<C *>(tw + a.K);
    C *b1 = b0 + a.K * a.W;
    for (int i = threadIdx.x; i < a.K; i += blockDim.x) tw_set(tw[i], a.tw[i]);
    const int ncb = slabs > 1 ? 1 : (a.inner + a.W - 1) / a.W;
    const size_t o0 = (size_t)(blockIdx.x / ncb) * slabs;
    const int c0 = (int)(blockIdx.x % ncb) * a.W;
    const int wc = min(a.W, a.inner - c0), ns = (int)min((size_t)slabs, outer - o0);   // columns of a slab, slabs
    C *base = reinterpret_cast<C *>(a.data) + o0 * (size_t)a.K * a.inner + c0;
    // element e of the tile: column e % wc, row, slab
    auto each = [&](auto &&f) {
        for (int e = threadIdx.x; e < ns * a.K * wc; e += blockDim.x) {
            const int q = e / wc, col = e - q * wc, sl = slabs > 1 ? q / a.K : 0, row = q - sl * a.K;
            f(row * a.W + sl * wc + col, base + ((size_t)sl * a.K + row) * a.inner + col, row, col);
        }
    };
    each([&](int t, const C *g, int, int) { cst(b0 + t, cld(g)); });
    __syncthreads();
    C *res;
    if (MODE == 2) {
        res = stockham<T, F, false>(b0, b1, a, tw);
        C *other = (res == b0) ? b1 : b0;
        // one slab; G index: (row, (c0 + col) / V)
        each([&](int t, const C *, int row, int col) {
            const T gv = a.G[(size_t)row * (a.inner / a.V) + (c0 + col) / a.V];
            res[t] = {fmulc(res[t].x, gv), fmulc(res[t].y, gv)};
        });
        __syncthreads();
        res = stockham<T, F, true>(res, other, a, tw);
    } else {
        res = stockham<T, F, MODE == 1>(b0, b1, a, tw);
    }
    each([&](int t, C *g, int, int) { cst(g, cld(res + t)); });
}

// The generic pass over columns of Cx<F> (a.inner, a.V and a.W in that unit).  The
// tile narrows until two blocks fit an SM (one block of 16 columns left it at eight
// warps); slabs narrower than a tile are taken together up to four blocks per SM, as
// far as that leaves two blocks for each.  us for the five passes of 288^3: FP32,
// up to 4 probes 4236 -> 2439, 8 probes 7239 -> 4913; FP64, 2 probes 10840 -> 8084.
constexpr size_t kGenericPassSmem = 100 * 1024;
template <class T, class F> mbd_status launch_fft_generic(FFTArgs<T> a, int mode, unsigned outer, cudaStream_t st) {
    auto bytes = [&](int w) { return sizeof(typename TwOf<F>::type) * a.K + 2 * sizeof(Cx<F>) * (size_t)a.K * w; };
    a.W = std::min(a.inner, 16);
    while (a.W > 1 && bytes(a.W) > kGenericPassSmem) a.W = (a.W + 1) / 2;
    int slabs = 1;
    if (a.W == a.inner && mode != 2) {
        slabs = (int)std::max(1u, std::min(16u / a.W, outer / (2u * (unsigned)std::max(1, a.sms))));
        while (slabs > 1 && bytes(slabs * a.W) > kGenericPassSmem / 2) --slabs;
        a.W *= slabs;
    }
    auto kern = mode == 0 ? k_fft_pass<T, F, 0> : (mode == 1 ? k_fft_pass<T, F, 1> : k_fft_pass<T, F, 2>);
    const unsigned grid = slabs > 1 ? (outer + slabs - 1) / slabs : outer * (unsigned)((a.inner + a.W - 1) / a.W);
    MBD_CUDA_TRY(allow_smem(kern, bytes(a.W), kGenericPassSmem));
    kern<<<grid, 256, bytes(a.W), st>>>(a, outer, slabs);
    MBD_LAUNCH_CHECK();
    return MBD_OK;
}

// ---------------------------------------------------------------- real space on clusters
template <class T> struct RealArgs {
    const T *d;          // [N][3][ld]
    T *out;              // [N][3][ld] E_real
    int ld, N;
    const int *order;    // cluster c = atoms order[16c .. 16c + 15]
    const int *pstart, *ecnt, *rcnt, *entries;
    const RealDuo<T> *recs;
    int np;              // probes of a chunk (blockIdx.y)
    int ce;              // entries staged at a time
};

// The real-space field E_real = sum over pairs A(r) d_j (Eq. fld_ewald with
// the damping correction) on clusters: a block per cluster of 16 atoms and
// chunk of np probes, warp w for the cluster's atoms 2w and 2w + 1.  The block
// stages the dipoles of the cluster's distinct neighbours in shared memory, ce
// entries at a time (cp.async, 16 bytes per lane), so each neighbour's dipoles
// come from L2 once per cluster.  A warp walks the records of its two atoms in
// entry order, in double-buffered batches of 32 (cp.async), and counts by a
// ballot those whose entries are staged; np / VEC lanes hold the probes, and
// the S groups of a warp take the records in turn.  A record applies one
// neighbour's dipoles, read from shared memory once, to both atoms: close atoms
// share three quarters of their neighbours, and the reads of shared memory and
// the instructions beside the packed FMAs are what bound the kernel (100,002
// atoms x 64 probes: 677 -> 559 us per launch; with 64 registers and four
// blocks per SM it spills, 605 us).
// An atom's field is a sum in a fixed order (per group, then the groups).
constexpr int kRealBatch = 32;
constexpr int kRealStageBytes = 36 * 1024;
constexpr int kRealMaxEntries = 192;      // staged at a time
// MASKED: an atom that has no pair with the neighbour of a record is left out.  FP64 is
// bound by its FMAs and gains by it.  FP32 gives it the record's zero tensor, which
// is quicker (24,000 atoms x 64 probes 147 against 174 us), but not the same when the
// neighbour's dipole is not finite: only right where one such dipole reaches
// every atom anyway, by the mesh.
template <class T, bool MASKED>
__global__ void __launch_bounds__(16 * kClusterSize, sizeof(T) == 4 ? 3 : 2) k_real_clusters(RealArgs<T> a) {
    constexpr int VEC = 16 / (int)sizeof(T), NW = kClusterSize / 2;
    constexpr int RC = (int)sizeof(RealDuo<T>) / 16;       // 16-byte pieces of a record
    extern __shared__ __align__(16) unsigned char real_smem[];
    RealDuo<T> *sp = reinterpret_cast<RealDuo<T> *>(real_smem);              // [NW][2][kRealBatch]
    int *ent = reinterpret_cast<int *>(sp + NW * 2 * kRealBatch);            // [2][ce]
    T *sd = reinterpret_cast<T *>(real_smem + sizeof(RealDuo<T>) * NW * 2 * kRealBatch + 16 * ((8 * a.ce + 15) / 16));
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c = blockIdx.x, pb = blockIdx.y * a.np, np = min(a.np, a.ld - pb);
    const int lanes = a.np / VEC, S = 32 / lanes, sub = lane / lanes, lid = lane - sub * lanes;
    const bool on = sub < S && lid * VEC < np;
    const int p0 = a.pstart[c * kClusterSize], ne = a.ecnt[c];
    const int *entries = a.entries + p0;
    const RealDuo<T> *recs = a.recs + a.pstart[c * kClusterSize + 2 * warp];
    const int nrec = a.rcnt[c * NW + warp];
    RealDuo<T> *mine = sp + warp * 2 * kRealBatch;
    auto fetch_batch = [&](int first, int b) {
        const int nq = min(kRealBatch, nrec - first) * RC;
        const float4 *src = reinterpret_cast<const float4 *>(recs + first);
        float4 *dst = reinterpret_cast<float4 *>(mine + b * kRealBatch);
        for (int q = lane; q < nq; q += 32) cp_async<16>(dst + q, src + q);
        cp_async_commit();
    };
    if (nrec > 0) fetch_batch(0, 0);
    for (int q = threadIdx.x; q < min(a.ce, ne); q += blockDim.x) ent[q] = entries[q];
    int first = -kRealBatch, bn = kRealBatch, bi = kRealBatch, buf = 1;   // current batch: none yet
    int ev = 0x7fffffff;                           // entry of the batch's record held by this lane
    T E[2][3][VEC];
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int k = 0; k < 3; ++k)
#pragma unroll
            for (int v = 0; v < VEC; ++v) E[h][k][v] = T(0);
    for (int c0 = 0, eb = 0; c0 < ne; c0 += a.ce, eb ^= 1) {
        const int m = min(a.ce, ne - c0);
        __syncthreads();                           // the previous chunk is consumed; its successor's entries are there
        for (int r = warp * S + sub; r < 3 * m && on; r += NW * S) {
            const int q = r / 3, k = r - 3 * q;
            cp_async<16>(sd + (size_t)r * a.np + lid * VEC,
                         a.d + (size_t)(3 * ent[eb * a.ce + q] + k) * a.ld + pb + lid * VEC);
        }
        for (int q = threadIdx.x; q < min(a.ce, ne - c0 - m); q += blockDim.x)
            ent[(eb ^ 1) * a.ce + q] = entries[c0 + m + q];
        cp_async_commit();
        cp_async_wait<0>();                        // the chunk (and the records on their way)
        __syncthreads();
        const int lim = c0 + m;                    // entries staged: [c0, lim)
        for (;;) {
            if (bi == bn) {                        // the next batch of records
                first += bn;
                if (first >= nrec) {
                    first = nrec;
                    bn = bi = 0;
                    break;
                }
                buf ^= 1;
                bn = min(kRealBatch, nrec - first);
                bi = 0;
                cp_async_wait<0>();
                __syncwarp();
                ev = lane < bn ? mine[buf * kRealBatch + lane].e : 0x7fffffff;
                if (first + bn < nrec) fetch_batch(first + bn, buf ^ 1);
            }
            // the records bi .. bi + cnt - 1 of the batch have their entries
            // staged (entries increase along the batch)
            const int cnt = __popc(__ballot_sync(0xffffffffu, lane >= bi && ev < lim));
            if (on) {
                for (int t = sub; t < cnt; t += S) {
                    const RealDuo<T> &cur = mine[buf * kRealBatch + bi + t];
                    const T *x0 = sd + (size_t)(cur.e - c0) * 3 * a.np + lid * VEC;
                    T x[VEC], y[VEC], z[VEC], A[12];
                    vload<T, VEC>(x0, x);
                    vload<T, VEC>(x0 + a.np, y);
                    vload<T, VEC>(x0 + 2 * a.np, z);
#pragma unroll
                    for (int q = 0; q < 12; q += VEC) vload<T, VEC>(cur.a + q, A + q);
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        if (MASKED && !(cur.mask & (1 << h))) continue;
                        const T *B = A + 6 * h;
                        lane_fma<T, VEC>(x, B[0], E[h][0]);
                        lane_fma<T, VEC>(y, B[1], E[h][0]);
                        lane_fma<T, VEC>(z, B[2], E[h][0]);
                        lane_fma<T, VEC>(x, B[1], E[h][1]);
                        lane_fma<T, VEC>(y, B[3], E[h][1]);
                        lane_fma<T, VEC>(z, B[4], E[h][1]);
                        lane_fma<T, VEC>(x, B[2], E[h][2]);
                        lane_fma<T, VEC>(y, B[4], E[h][2]);
                        lane_fma<T, VEC>(z, B[5], E[h][2]);
                    }
                }
            }
            __syncwarp();                          // the batch is read before a later one takes its buffer
            bi += cnt;
            if (bi < bn) break;                    // the next record waits for a later chunk
        }
    }
    cp_async_wait<0>();                            // no copy in flight at exit
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int idx = c * kClusterSize + 2 * warp + h;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            T o[VEC];
#pragma unroll
            for (int v = 0; v < VEC; ++v) {
                o[v] = E[h][k][v];
                for (int g = 1; g < S; ++g) o[v] += __shfl_sync(0xffffffffu, E[h][k][v], lid + g * lanes);
            }
            if (sub == 0 && on && idx < a.N)
                vstore<T, VEC>(a.out + (size_t)(3 * a.order[idx] + k) * a.ld + pb + lid * VEC, o);
        }
    }
}

// ---------------------------------------------------------------- field
template <class T> struct FieldArgs {
    const T *d;          // [N][3][ld]
    const T *mesh;       // [K^3][ld]
    int R, ld;
    Geom g;
    PairView<T> pr;
    const unsigned char *rec;   // FieldRec of every atom in processing order
    const double *g_at;  // [N] w sqrt(alpha)
    const double *w2;    // [N] w^2
    double self_coef;
    const T *ereal;      // real-space field from k_real_clusters [N][3][ld] (kernels without the pair loop)
    FieldOut<T> o;
    int lanes;           // lanes of a warp that share an atom (VEC probes each)
    int teams;           // atoms that a block works on at once
    int apb;             // atoms per block
};

// What the field kernel reads of an atom, in processing order (Morton order of
// the bricks): {atom, top1, top2, top3}, then M1, M1', M2, M2', M3, M3' (P values each).
template <class T, int P> constexpr int field_rec_bytes() { return 16 + 6 * P * (int)sizeof(T); }
template <class T>
__global__ void k_field_rec(int N, int p, const int *__restrict__ order, const int *__restrict__ top,
                            const double *__restrict__ w64, const double *__restrict__ dw64,
                            unsigned char *__restrict__ rec) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x, per = 6 * p + 4;
    if (idx >= N * per) return;
    const int pos = idx / per, k = idx - pos * per, i = order[pos];
    unsigned char *r = rec + (size_t)pos * (16 + 6 * p * sizeof(T));
    if (k < 4) {
        reinterpret_cast<int *>(r)[k] = k == 0 ? i : top[3 * i + k - 1];
    } else {
        const int dim = (k - 4) / (2 * p), t = (k - 4) % (2 * p);
        reinterpret_cast<T *>(r + 16)[k - 4] =
            T(t < p ? w64[(size_t)(3 * i + dim) * p + t] : dw64[(size_t)(3 * i + dim) * p + t - p]);
    }
}

// Warps of a field block: as many as divide the p^2 pencils of a stencil evenly.
template <int P> constexpr int field_warps() { return P == 6 ? 6 : (P == 10 ? 10 : 8); }
template <class T> constexpr int field_vec() { return 16 / (int)sizeof(T); }

// The epilogue of one iteration of the field kernels, one thread per (atom,
// component, probe) slot: the warps' partial fields red[NW][OUT] summed in
// order, then the output selected by o.mode; part: y.l of the thread's slots.
template <class T, int NW, int OUT, int OPT>
__device__ __forceinline__ void field_epilogue(const FieldArgs<T> &a, const T *red, int rec_bytes, int nloc, int nout,
                                               int rbase, int ib, int i1, double *part) {
#pragma unroll
    for (int k = 0; k < OPT; ++k) {
        const int slot = threadIdx.x + k * NW * 32;
        if (slot >= nout) break;
        const int tc = slot / nloc, t = slot - tc * nloc, tm = tc / 3, c = tc - 3 * tm;
        const int r = rbase + t;
        if (r >= a.ld || ib + tm >= i1) continue;
        const int i = *reinterpret_cast<const int *>(a.rec + (size_t)(ib + tm) * rec_bytes);
        T sum = T(0);
#pragma unroll
        for (int w = 0; w < NW; ++w) sum += red[w * OUT + slot];
        const double En = double(sum);
        const size_t o = (size_t)(3 * i + c) * a.ld + r;
        if (a.o.mode == kFieldOut) {
            a.o.out[o] = En;
        } else if (a.o.mode == kFieldApply) {
            a.o.out[o] = a.w2[i] * a.o.xin[o] + a.g_at[i] * En;
        } else {
            const double invb = a.o.lz.invb[r];
            double *Yk = a.o.lz.Y + lz_slot(a.o.lz, a.o.k) * (size_t)(3 * a.g.N) * a.ld;
            const double ys = Yk[o];
            const double y = ys * invb, l = (a.w2[i] * ys + a.g_at[i] * En) * invb;
            Yk[o] = y;
            a.o.lz.L[o] = l;
            if (a.o.lz.W) a.o.lz.W[o] += a.o.lz.coef[(size_t)a.o.k * a.ld + r] * y;
            part[k] += y * l;
        }
    }
}
// a_k = y_k^T l_k: per probe, the teams and components in order, then a
// deterministic reduction over blocks.  pall [OUT], bsum and tot [probes of a
// chunk] are shared scratch.
template <class T, int NW, int OPT>
__device__ __forceinline__ void field_reduce_a(const FieldArgs<T> &a, int nloc, int nout, int rbase, const double *part,
                                               double *pall, double *bsum, double *tot) {
#pragma unroll
    for (int k = 0; k < OPT; ++k)
        if ((int)threadIdx.x + k * NW * 32 < nout) pall[threadIdx.x + k * NW * 32] = part[k];
    __syncthreads();
    for (int t = threadIdx.x; t < nloc; t += NW * 32) {
        double sum = 0.0;
        for (int q = 0; q < 3 * a.teams; ++q) sum += pall[q * nloc + t];
        bsum[t] = sum;
    }
    __syncthreads();
    if (grid_reduce(bsum, nloc, rbase, a.R, a.ld, a.o.lz, tot)) {
        for (int k = threadIdx.x; k < nloc; k += NW * 32)
            if (rbase + k < a.R) a.o.lz.a[(size_t)a.o.k * a.ld + rbase + k] = tot[k];
    }
}

// Field kernel.  `lanes` lanes with VEC probes each (16-byte accesses) hold the
// probes of an atom (of a chunk of 32 VEC probes, blockIdx.y), so a warp holds
// S = 32 / lanes groups.  A block works on `teams` atoms at once; the groups of
// a team (S / teams per warp, in every warp) split the p^2 pencils of the
// atom's stencil and, with PAIRS, its neighbours.  With many probes (S = teams
// = 1) a warp gathers whole planes of the stencil; with few, a warp's groups take
// several atoms or, in small systems, share one.  Along a pencil the field
// factorises like the weights: s0 = sum_t M3(t) phi, s1 = sum_t M3'(t) phi
// (two FMAs per mesh value), then f += (M1' M2 s0, M1 M2' s0, M1 M2 s1) once.
// The partial fields are summed in a fixed order (shuffles within a warp,
// then the warps in shared memory) and the epilogue selected by o.mode runs
// with one thread per (atom, component, probe): E* = E^rec + E^dir + E^self
// (Eqs. ewalddip, spme, fld_ewald, fld_ewald1), l_k = Omega y_k + Diag(g) E*_k
// and a_k = y_k^T l_k (Eqs. lk3, recurs2).
// Bound: load latency (FP32), the FP64 units (FP64).  Against a lane per probe
// with six FMAs and three products per mesh value: 288 atoms x 1 FP64 68 -> 23
// us per launch, 1371 x 33 order 8 127 -> 34, 3000 x 32 FP64 544 -> 295, 15,000
// x 2 order 8 331 -> 76.
template <class T, int P, bool PAIRS>
__global__ void __launch_bounds__(field_warps<P>() * 32, sizeof(T) == 8 ? 2 : (PAIRS ? 3 : 4) * 6 / field_warps<P>())
    k_field(FieldArgs<T> a) {
    constexpr int VEC = field_vec<T>(), NW = field_warps<P>(), NTH = NW * 32;
    constexpr int RB = field_rec_bytes<T, P>();
    constexpr int OUT = 32 * VEC * 3;            // (team, component, probe) slots of an iteration, at most
    constexpr int OPT = (OUT + NTH - 1) / NTH;   // of them per thread, at most
    pdl_wait();
    pdl_launch_dependents();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int S = 32 / a.lanes, nloc = a.lanes * VEC, per = S / a.teams;   // groups of a team in a warp
    const int sub = lane / a.lanes, lid = lane - sub * a.lanes;
    const int team = sub % a.teams, member = warp + NW * (sub / a.teams), members = NW * per;
    const int rbase = blockIdx.y * 32 * VEC;
    const int r0 = rbase + lid * VEC;
    const bool on = sub < S && r0 < a.ld;
    const int nout = a.teams * 3 * nloc;
    // partial fields of the warps, double-buffered by iteration: the barrier
    // after one iteration's writes also orders the previous epilogue's reads
    // before the buffer is written again, so one barrier per iteration
    __shared__ __align__(16) T red[2][NW][OUT];
    __shared__ double pall[OUT], bsum[32 * VEC], tot[32 * VEC];
    double part[OPT];                            // y.l of the slots this thread owns
#pragma unroll
    for (int k = 0; k < OPT; ++k) part[k] = 0.0;
    const int i0 = blockIdx.x * a.apb, i1 = min(i0 + a.apb, a.g.N);
    int buf = 0;
    for (int ib = i0; ib < i1; ib += a.teams, buf ^= 1) {
        T E[3][VEC];
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int v = 0; v < VEC; ++v) E[c][v] = T(0);
        if (on && ib + team < i1) {
            const unsigned char *rec = a.rec + (size_t)(ib + team) * RB;
            const int4 hd = *reinterpret_cast<const int4 *>(rec);
            const int i = hd.x;
            if (a.o.terms & MBD_TERM_RECIP) {
                T f[3][VEC];
#pragma unroll
                for (int c = 0; c < 3; ++c)
#pragma unroll
                    for (int v = 0; v < VEC; ++v) f[c][v] = T(0);
                const T *w = reinterpret_cast<const T *>(rec + 16);
                T w3[2 * P];
#pragma unroll
                for (int b = 0; b < 2 * P; b += VEC) vload<T, VEC>(w + 4 * P + b, w3 + b);
                int off[P];
#pragma unroll
                for (int t = 0; t < P; ++t) off[t] = (hd.w - t + (hd.w < t ? a.g.K3 : 0)) * a.ld;
                for (int u = member; u < P * P; u += members) {
                    const int t1 = u % P, t2 = u / P;
                    int k1 = hd.y - t1, k2 = hd.z - t2;
                    if (k1 < 0) k1 += a.g.K1;
                    if (k2 < 0) k2 += a.g.K2;
                    const T *rowp = a.mesh + ((size_t)k1 * a.g.K2 + k2) * a.g.K3 * a.ld + r0;
                    T phi[P][VEC];
#pragma unroll
                    for (int t = 0; t < P; ++t) vload<T, VEC>(rowp + off[t], phi[t]);
                    const T wa = w[t1], da = w[P + t1], wb = w[2 * P + t2], db = w[3 * P + t2];
                    T s0[VEC], s1[VEC];
#pragma unroll
                    for (int v = 0; v < VEC; ++v) s0[v] = s1[v] = T(0);
#pragma unroll
                    for (int t = 0; t < P; ++t) {
                        lane_fma<T, VEC>(phi[t], w3[t], s0);
                        lane_fma<T, VEC>(phi[t], w3[P + t], s1);
                    }
                    lane_fma<T, VEC>(s0, da * wb, f[0]);
                    lane_fma<T, VEC>(s0, wa * db, f[1]);
                    lane_fma<T, VEC>(s1, wa * wb, f[2]);
                }
                // E^rec_alpha = sum_beta C_{beta alpha} f_beta
#pragma unroll
                for (int c = 0; c < 3; ++c)
#pragma unroll
                    for (int b = 0; b < 3; ++b) lane_fma<T, VEC>(f[b], T(a.g.cmat[3 * b + c]), E[c]);
            }
            if (a.o.terms & MBD_TERM_REAL) {
                if constexpr (PAIRS) {
                    const int nb1 = a.pr.row[i + 1];
                    constexpr int B = 2;
                    for (int nb = a.pr.row[i] + member; nb < nb1; nb += B * members) {
                        int jj[B];
                        T x[B][VEC], y[B][VEC], z[B][VEC];
#pragma unroll
                        for (int u = 0; u < B; ++u) jj[u] = nb + u * members < nb1 ? a.pr.col[nb + u * members] : -1;
#pragma unroll
                        for (int u = 0; u < B; ++u)
                            if (jj[u] >= 0) {
                                const T *dj = a.d + (size_t)(3 * jj[u]) * a.ld + r0;
                                vload<T, VEC>(dj, x[u]);
                                vload<T, VEC>(dj + a.ld, y[u]);
                                vload<T, VEC>(dj + 2 * (size_t)a.ld, z[u]);
                            }
#pragma unroll
                        for (int u = 0; u < B; ++u)
                            if (jj[u] >= 0) {
                                T A[6];
#pragma unroll
                                for (int e = 0; e < 6; e += 2)
                                    vload<T, 2>(a.pr.A + 6 * (size_t)(nb + u * members) + e, A + e);
                                lane_fma<T, VEC>(x[u], A[0], E[0]);
                                lane_fma<T, VEC>(y[u], A[1], E[0]);
                                lane_fma<T, VEC>(z[u], A[2], E[0]);
                                lane_fma<T, VEC>(x[u], A[1], E[1]);
                                lane_fma<T, VEC>(y[u], A[3], E[1]);
                                lane_fma<T, VEC>(z[u], A[4], E[1]);
                                lane_fma<T, VEC>(x[u], A[2], E[2]);
                                lane_fma<T, VEC>(y[u], A[4], E[2]);
                                lane_fma<T, VEC>(z[u], A[5], E[2]);
                            }
                    }
                } else if (member == NW - 1) {
                    T x[VEC];
                    const T *ei = a.ereal + (size_t)(3 * i) * a.ld + r0;
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        vload<T, VEC>(ei + (size_t)c * a.ld, x);
#pragma unroll
                        for (int v = 0; v < VEC; ++v) E[c][v] += x[v];
                    }
                }
            }
            if ((a.o.terms & MBD_TERM_SELF) && member == 0) {
                T x[VEC];
                const T *di = a.d + (size_t)(3 * i) * a.ld + r0;
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    vload<T, VEC>(di + (size_t)c * a.ld, x);
                    lane_fma<T, VEC>(x, T(a.self_coef), E[c]);
                }
            }
        }
        // the groups of a team within the warp (S is a power of two when per > 1)
        for (int h = S / 2; h >= a.teams && per > 1; h >>= 1) {
#pragma unroll
            for (int c = 0; c < 3; ++c)
#pragma unroll
                for (int v = 0; v < VEC; ++v) E[c][v] += __shfl_down_sync(0xffffffffu, E[c][v], h * a.lanes);
        }
        if (sub < a.teams) {
#pragma unroll
            for (int c = 0; c < 3; ++c) vstore<T, VEC>(&red[buf][warp][(team * 3 + c) * nloc + lid * VEC], E[c]);
        }
        __syncthreads();
        field_epilogue<T, NW, OUT, OPT>(a, &red[buf][0][0], RB, nloc, nout, rbase, ib, i1, part);
    }
    if (a.o.mode != kFieldLanczos) return;
    field_reduce_a<T, NW, OPT>(a, nloc, nout, rbase, part, pall, bsum, tot);
}

// The field kernel for large FP32 systems with the real space on clusters: the
// same split (a group per warp and atom, so members = NW, and p^2 / NW pencils
// per group in a fixed order), with the mesh values streamed through shared
// memory.  Each thread copies its own 16 bytes of a pencil's P points by
// cp.async, kFieldDepth pencils ahead of the one it works on and across atoms,
// and reads back only what it copied itself, so no barrier is involved and no
// register holds a value in flight: the loads in flight per SM, which bound the
// kernel (ncu: DRAM and L2 far from their peaks, long-scoreboard stalls), no
// longer depend on registers.  The atoms' weights for the next iteration are
// copied to shared memory meanwhile.
constexpr int kFieldDepth = 2;
template <int P> constexpr size_t field_stream_smem(int teams) {
    constexpr int NTH = field_warps<P>() * 32;
    return 16 * (size_t)kFieldDepth * P * NTH + 4 * (size_t)field_warps<P>() * 384 + 2 * (size_t)teams * 24 * P;
}
template <int P>
__global__ void __launch_bounds__(field_warps<P>() * 32, P == 6 ? 4 : 2) k_field_stream(FieldArgs<float> a) {
    constexpr int VEC = 4, NW = field_warps<P>(), NTH = NW * 32, PP = P * P / NW, D = kFieldDepth;
    constexpr int OUT = 32 * VEC * 3, OPT = (OUT + NTH - 1) / NTH, RB = field_rec_bytes<float, P>(), W4 = 6 * P / 4;
    static_assert(P * P % NW == 0 && PP % D == 0 && 6 * P % 4 == 0, "whole pencils per warp and ring");
    pdl_wait();
    pdl_launch_dependents();
    extern __shared__ __align__(16) unsigned char smem_fs[];
    float4 *ring = reinterpret_cast<float4 *>(smem_fs);                  // [D][P][NTH]
    float *red = reinterpret_cast<float *>(ring + D * P * NTH);          // [NW][OUT]
    float4 *wts = reinterpret_cast<float4 *>(red + NW * OUT);            // [2][teams][W4]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nloc = a.lanes * VEC, sub = lane / a.lanes, lid = lane - sub * a.lanes;
    const int rbase = blockIdx.y * 32 * VEC, r0 = rbase + lid * VEC;
    const bool on = sub < a.teams && r0 < a.ld;
    const int nout = a.teams * 3 * nloc;
    double part[OPT];
#pragma unroll
    for (int k = 0; k < OPT; ++k) part[k] = 0.0;
    const int i0 = blockIdx.x * a.apb, i1 = min(i0 + a.apb, a.g.N);
    auto header = [&](int pos) {
        return pos < i1 ? *reinterpret_cast<const int4 *>(a.rec + (size_t)pos * RB) : make_int4(-1, 0, 0, 0);
    };
    auto fetch_weights = [&](int ib, int b) {   // the weights of the teams' atoms from ib on
        for (int q = threadIdx.x; q < a.teams * W4; q += NTH)
            if (ib + q / W4 < i1)
                cp_async<16>(wts + b * a.teams * W4 + q, a.rec + (size_t)(ib + q / W4) * RB + 16 + 16 * (q % W4));
    };
    int off[P];
    auto offsets = [&](int4 hd) {
#pragma unroll
        for (int t = 0; t < P; ++t) off[t] = (hd.w - t + (hd.w < t ? a.g.K3 : 0)) * a.ld;
    };
    auto fetch = [&](int4 hd, int j) {          // pencil j of the atom into ring slot j % D
        if (on && hd.x >= 0) {
            const int u = warp + NW * j, t1 = u % P, t2 = u / P;
            int k1 = hd.y - t1, k2 = hd.z - t2;
            if (k1 < 0) k1 += a.g.K1;
            if (k2 < 0) k2 += a.g.K2;
            const float *rowp = a.mesh + ((size_t)k1 * a.g.K2 + k2) * a.g.K3 * a.ld + r0;
#pragma unroll
            for (int t = 0; t < P; ++t) cp_async<16>(ring + ((j % D) * P + t) * NTH + threadIdx.x, rowp + off[t]);
        }
        cp_async_commit();
    };
    int4 hd = header(i0 + sub);
    fetch_weights(i0, 0);
    cp_async_commit();
    offsets(hd);
#pragma unroll
    for (int j = 0; j < D; ++j) fetch(hd, j);
    cp_async_wait<D>();                          // the first weights, made visible by the barrier
    __syncthreads();
    int b = 0;
    for (int ib = i0; ib < i1; ib += a.teams, b ^= 1) {
        const int4 next = header(ib + a.teams + sub);
        fetch_weights(ib + a.teams, b ^ 1);      // joins the group of the next pencil
        const float *w = reinterpret_cast<const float *>(wts + (b * a.teams + (sub < a.teams ? sub : 0)) * W4);
        float f[3][VEC];
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int v = 0; v < VEC; ++v) f[c][v] = 0.f;
#pragma unroll
        for (int j = 0; j < PP; ++j) {
            cp_async_wait<D - 1>();              // this thread's copies of pencil j are done
            float s0[VEC], s1[VEC];
#pragma unroll
            for (int v = 0; v < VEC; ++v) s0[v] = s1[v] = 0.f;
#pragma unroll
            for (int t = 0; t < P; ++t) {
                float phi[VEC];
                vload<float, VEC>(reinterpret_cast<const float *>(ring + ((j % D) * P + t) * NTH + threadIdx.x), phi);
                lane_fma<float, VEC>(phi, w[4 * P + t], s0);
                lane_fma<float, VEC>(phi, w[5 * P + t], s1);
            }
            if (j + D == PP) offsets(next);
            if (j + D < PP) fetch(hd, j + D);
            else fetch(next, j + D - PP);
            const int u = warp + NW * j, t1 = u % P, t2 = u / P;
            const float wa = w[t1], da = w[P + t1], wb = w[2 * P + t2], db = w[3 * P + t2];
            lane_fma<float, VEC>(s0, da * wb, f[0]);
            lane_fma<float, VEC>(s0, wa * db, f[1]);
            lane_fma<float, VEC>(s1, wa * wb, f[2]);
        }
        float E[3][VEC];
        const bool act = on && hd.x >= 0;
        // E^rec_alpha = sum_beta C_{beta alpha} f_beta
#pragma unroll
        for (int c = 0; c < 3; ++c) {
#pragma unroll
            for (int v = 0; v < VEC; ++v) E[c][v] = 0.f;
#pragma unroll
            for (int q = 0; q < 3; ++q) lane_fma<float, VEC>(f[q], float(a.g.cmat[3 * q + c]), E[c]);
        }
        if (act && warp == NW - 1 && (a.o.terms & MBD_TERM_REAL)) {
            const float *ei = a.ereal + (size_t)(3 * hd.x) * a.ld + r0;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                float x[VEC];
                vload<float, VEC>(ei + (size_t)c * a.ld, x);
#pragma unroll
                for (int v = 0; v < VEC; ++v) E[c][v] += x[v];
            }
        }
        if (act && warp == 0 && (a.o.terms & MBD_TERM_SELF)) {
            const float *di = a.d + (size_t)(3 * hd.x) * a.ld + r0;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                float x[VEC];
                vload<float, VEC>(di + (size_t)c * a.ld, x);
                lane_fma<float, VEC>(x, float(a.self_coef), E[c]);
            }
        }
        if (sub < a.teams) {
#pragma unroll
            for (int c = 0; c < 3; ++c) vstore<float, VEC>(red + warp * OUT + (sub * 3 + c) * nloc + lid * VEC, E[c]);
        }
        if constexpr (PP == D) cp_async_wait<D - 1>();   // (they came with the next atom's first pencil)
        __syncthreads();                         // the partial fields, and the next weights
        field_epilogue<float, NW, OUT, OPT>(a, red, RB, nloc, nout, rbase, ib, i1, part);
        __syncthreads();                         // red is written again
        hd = next;
    }
    cp_async_wait<0>();                          // no copy in flight at exit
    if (a.o.mode != kFieldLanczos) return;
    double *pall = reinterpret_cast<double *>(smem_fs);
    __syncthreads();                             // the ring is scratch from here on
    field_reduce_a<float, NW, OPT>(a, nloc, nout, rbase, part, pall, pall + OUT, pall + OUT + 32 * VEC);
}

template <class T> PrecData<T> &prec(mbd_system *s);
template <> PrecData<double> &prec<double>(mbd_system *s) { return s->f64; }
template <> PrecData<float> &prec<float>(mbd_system *s) { return s->f32; }

Geom geom_of(const mbd_system *s) {
    Geom g;
    g.N = s->N;
    g.K1 = s->K[0];
    g.K2 = s->K[1];
    g.K3 = s->K[2];
    g.p = s->p;
    for (int b = 0; b < 3; ++b)
        for (int a = 0; a < 3; ++a) g.cmat[3 * b + a] = s->K[b] * s->recip[3 * b + a];
    for (int k = 0; k < 9; ++k) g.cell[k] = s->cell[k];
    return g;
}

}  // namespace

mbd_status launch_exclusive_scan(const int *in, int *out, int n, DevBuf &bsum, cudaStream_t st) {
    const int nb = (n + 4095) / 4096;
    MBD_TRY(bsum.ensure(sizeof(int) * (size_t)std::max(1, nb)));
    if (n > 0) {
        k_scan_block<<<nb, 1024, 0, st>>>(in, out, bsum.as<int>(), n);
        MBD_LAUNCH_CHECK();
    }
    k_scan_sums<<<1, 32, 0, st>>>(bsum.as<int>(), nb, out + n);
    MBD_LAUNCH_CHECK();
    if (n > 0) {
        k_scan_add<<<(n + 255) / 256, 256, 0, st>>>(out, bsum.as<int>(), n);
        MBD_LAUNCH_CHECK();
    }
    return MBD_OK;
}

// The spreading records of the current geometry: counts, CSR starts, records,
// and the per-atom k3 stencils; and the field kernel's records.
template <class T> mbd_status build_spread_records(mbd_system *s) {
    PrecData<T> &P = prec<T>(s);
    const Geom g = geom_of(s);
    const size_t npts = (size_t)s->K[0] * s->K[1] * s->K[2];
    const size_t nnz = (size_t)s->p * s->p * (size_t)s->N;   // each atom covers p^2 pencils (K >= 2p)
    if (npts >= 0x7fffffffULL || nnz >= 0x7fffffffULL) return MBD_ERR_UNSUPPORTED;
    MBD_TRY(P.prow.ensure(sizeof(int) * (npts + 1)));
    MBD_TRY(P.prec.ensure(sizeof(PencilRec<T>) * std::max<size_t>(1, nnz)));
    MBD_TRY(P.k3w.ensure(sizeof(T) * 2 * s->p * std::max(1, s->N)));
    DevBuf &cnt = s->scan_cnt, &bsum = s->scan_bsum;
    MBD_TRY(cnt.ensure(sizeof(int) * npts));
    const int threads = 256;
    const unsigned blocks = (unsigned)((npts + threads - 1) / threads);
    k_pencil_rows<T, false><<<blocks, threads, 0, s->stream>>>(g, s->bins, s->top_d.as<int>(), s->w64_d.as<double>(),
                                                              s->dw64_d.as<double>(), cnt.as<int>(), nullptr);
    MBD_LAUNCH_CHECK();
    MBD_TRY(launch_exclusive_scan(cnt.as<int>(), P.prow.template as<int>(), (int)npts, bsum, s->stream));
    k_pencil_rows<T, true><<<blocks, threads, 0, s->stream>>>(g, s->bins, s->top_d.as<int>(), s->w64_d.as<double>(),
                                                             s->dw64_d.as<double>(), P.prow.template as<int>(),
                                                             P.prec.template as<PencilRec<T>>());
    MBD_LAUNCH_CHECK();
    MBD_TRY(P.frec.ensure((16 + 6 * (size_t)s->p * sizeof(T)) * std::max(1, s->N)));
    if (s->N > 0) {
        const int nrec = s->N * (6 * s->p + 4);
        k_field_rec<T><<<(nrec + threads - 1) / threads, threads, 0, s->stream>>>(
            s->N, s->p, s->order_d.as<int>(), s->top_d.as<int>(), s->w64_d.as<double>(), s->dw64_d.as<double>(),
            P.frec.template as<unsigned char>());
        MBD_LAUNCH_CHECK();
        k_pencil_k3w<T><<<(2 * s->p * s->N + threads - 1) / threads, threads, 0, s->stream>>>(
            s->N, s->p, s->w64_d.as<double>(), s->dw64_d.as<double>(), P.k3w.template as<T>());
        MBD_LAUNCH_CHECK();
    }
    return MBD_OK;
}

template <class T> SpreadArgs<T> spread_args(mbd_system *s, const T *d, T *mesh, int R, int ld) {
    PrecData<T> &P = prec<T>(s);
    return {d, mesh, R, ld, s->K[0], s->K[1], s->K[2], s->p, P.prow.template as<int>(),
            P.prec.template as<PencilRec<T>>(), P.k3w.template as<T>(),
            P.tw3.template as<typename Cplx<T>::type>(), std::max(1, s->num_sms)};
}

template <class T> mbd_status launch_spread(mbd_system *s, const T *d, T *mesh, int R, int ld) {
    const SpreadArgs<T> a = spread_args(s, d, mesh, R, ld);
    const unsigned ncols = (unsigned)((size_t)a.K1 * a.K2 * (ld / 2));
    const unsigned tiles = (ncols + spread_w<T>() - 1) / spread_w<T>();
    // segments of at least p - 1 rows where one warp per tile would leave the GPU idle
    const int nseg = tiles < 8 * (unsigned)a.sms ? std::min(8, a.K3 / (s->p - 1)) : 1;
    const int warps = nseg > 1 ? nseg : 4;
    const unsigned grid = (tiles * nseg + warps - 1) / warps;
    switch (s->p) {
#define MBD_SPREAD_ORDER(P) \
    case P: k_spread_pencil<T, P><<<grid, 32 * warps, 0, s->stream>>>(a, ncols, nseg); break;
        MBD_SPLINE_ORDERS(MBD_SPREAD_ORDER)
#undef MBD_SPREAD_ORDER
        default: return MBD_ERR_UNSUPPORTED;
    }
    MBD_LAUNCH_CHECK();
    return MBD_OK;
}

// Meshes of at most this many bytes (three quarters of the 129 MB L2) launch
// their FFT passes with programmatic dependence; larger ones plainly.
constexpr size_t kEarlyFFTMaxBytes = 96u << 20;
// A convolution on its own launches its double passes early as well while the mesh is
// small: us per mbd_convolve, plain and early, 16^3 x 32 probes 64 and 49, 20^3 x 32 80
// and 69, 32^3 x 16 104 and 90, 40^3 x 16 (8 MB) 193 and 209.
constexpr size_t kEarlyAloneMaxBytes = 4u << 20;

#define MBD_HAS_CASE(K, ...) case K:
bool fft_ct_size(int K) {
    switch (K) {
        MBD_FFT_GROUP0(MBD_HAS_CASE)
        MBD_FFT_GROUP1(MBD_HAS_CASE)
        MBD_FFT_GROUP2(MBD_HAS_CASE)
        MBD_FFT_GROUP3(MBD_HAS_CASE)
        MBD_FFT_GROUP4(MBD_HAS_CASE)
        MBD_FFT_GROUP5(MBD_HAS_CASE)
        return true;
        default: return false;
    }
}
#undef MBD_HAS_CASE

template <class T> int launch_fft_ct_sized(const FFTArgs<T> &a, int mode, unsigned outer, cudaStream_t st) {
    int r;
    if ((r = launch_fft_ct_group0<T>(a, mode, outer, st)) >= 0) return r;
    if ((r = launch_fft_ct_group1<T>(a, mode, outer, st)) >= 0) return r;
    if ((r = launch_fft_ct_group2<T>(a, mode, outer, st)) >= 0) return r;
    if ((r = launch_fft_ct_group3<T>(a, mode, outer, st)) >= 0) return r;
    if ((r = launch_fft_ct_group4<T>(a, mode, outer, st)) >= 0) return r;
    return launch_fft_ct_group5<T>(a, mode, outer, st);
}

template <class T> int launch_spp_sized(const SpreadArgs<T> &a, cudaStream_t st) {
    int r;
    if ((r = launch_spp_group0<T>(a, st)) >= 0) return r;
    if ((r = launch_spp_group1<T>(a, st)) >= 0) return r;
    if ((r = launch_spp_group2<T>(a, st)) >= 0) return r;
    if ((r = launch_spp_group3<T>(a, st)) >= 0) return r;
    if ((r = launch_spp_group4<T>(a, st)) >= 0) return r;
    return launch_spp_group5<T>(a, st);
}

// Spreading fused with the first forward FFT pass when the k3 size has a
// compile-time pass.
bool spread_fft3_supported(const mbd_system *s) { return fft_ct_size(s->K[2]); }

// Returns MBD_ERR_UNSUPPORTED (nothing launched) when spread_fft3_supported is false.
template <class T> mbd_status launch_spread_fft3(mbd_system *s, const T *d, T *mesh, int R, int ld) {
    const int r = launch_spp_sized<T>(spread_args(s, d, mesh, R, ld), s->stream);
    if (r < 0) return MBD_ERR_UNSUPPORTED;
    if (r == 0) {
        set_last_error("fused spreading: shared-memory size", cudaGetLastError());
        return MBD_ERR_CUDA;
    }
    MBD_LAUNCH_CHECK();
    return MBD_OK;
}

template <class T> mbd_status launch_convolve(mbd_system *s, T *mesh, int ld, bool skip_first, bool alone) {
    using C = typename Cplx<T>::type;
    PrecData<T> &P = prec<T>(s);
    const int V = ld / 2;
    const int K1 = s->K[0], K2 = s->K[1], K3 = s->K[2];
    const size_t npts_bytes = sizeof(T) * (size_t)K1 * K2 * K3 * ld;
    auto run = [&](int dim, int outer, int inner, int mode) -> mbd_status {
        FFTArgs<T> a;
        a.data = reinterpret_cast<C *>(mesh);
        a.tw = (dim == 0 ? P.tw1 : (dim == 1 ? P.tw2 : P.tw3)).template as<C>();
        a.G = P.G.template as<T>();
        a.K = s->fft[dim].K;
        a.nst = s->fft[dim].nst;
        a.radices = 0ull;
        for (int k = 0; k < a.nst; ++k) a.radices |= (unsigned long long)s->fft[dim].radix[k] << (4 * k);
        a.inner = inner;
        a.V = V;
        // early launch of the passes while the mesh fits in three quarters of L2
        a.early = npts_bytes > kEarlyFFTMaxBytes ? 0 : (alone && npts_bytes <= kEarlyAloneMaxBytes ? 2 : 1);
        a.sms = s->num_sms;
        // wide tiles unless they are too few for four blocks per SM
        a.W = (size_t)outer * inner >= (size_t)128 * a.sms ? 32 : 16;
        if (s->tune_fft_w != 0 && tuned_for<T>(s, ld)) a.W = s->tune_fft_w;
        const int r = launch_fft_ct_sized<T>(a, mode, (unsigned)outer, s->stream);
        if (r == 0) {
            set_last_error("FFT pass: shared-memory size", cudaGetLastError());
            return MBD_ERR_CUDA;
        }
        if (r == 1) {
            MBD_LAUNCH_CHECK();
            return MBD_OK;
        }
        if (sizeof(T) == 4) {
            a.inner /= 2;
            a.V /= 2;
        }
        return launch_fft_generic<T, typename PackOf<T>::type>(a, mode, (unsigned)outer, s->stream);
    };
    if (!skip_first) MBD_TRY(run(2, K1 * K2, V, 0));   // forward along k3
    MBD_TRY(run(1, K1, K3 * V, 0));            // forward along k2
    MBD_TRY(run(0, 1, K2 * K3 * V, 2));         // forward k1, x G, inverse k1
    MBD_TRY(run(1, K1, K3 * V, 1));            // inverse along k2
    MBD_TRY(run(2, K1 * K2, V, 1));            // inverse along k3
    return MBD_OK;
}

// On small meshes the field kernel and the prologue are launched before the
// kernel in front of them has ended: their own launch then hides behind it, and
// a step of 36 us (96 atoms, 24^3, 1 probe) takes 31, one of 45 (1,200 atoms,
// 45^3, 4 probes) 42, one of 76.5 (32 probes, 12 MB) 73.8.  With longer kernels
// their waiting blocks hold registers and shared memory that the running one
// has a use for: nothing is gained at 23 MB, and 64^3 x 32 probes (34 MB) goes
// from 111 to 118 us.
constexpr size_t kEarlyStepMaxBytes = 16u << 20;
bool step_early(const mbd_system *s, int ld, int real_bytes) {
    return (size_t)real_bytes * s->K[0] * s->K[1] * s->K[2] * ld <= kEarlyStepMaxBytes;
}

// How a field launch is laid out: lanes per atom, atoms at once and in all per
// block, blocks.
struct FieldShape {
    int lanes, teams, apb, blocks, chunks;
};
namespace {
// Resident blocks per SM of one field-kernel variant (the same on every
// device of one architecture), asked of the occupancy calculator once.
template <class T, int P, bool PAIRS> int field_occupancy() {
    static std::atomic<int> nb;
    int x = nb.load(std::memory_order_relaxed);
    if (x == 0) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&x, k_field<T, P, PAIRS>, field_warps<P>() * 32, 0) !=
                cudaSuccess ||
            x < 1) {
            cudaGetLastError();
            return 1;
        }
        nb.store(x, std::memory_order_relaxed);
    }
    return x;
}

// Lanes per atom: just enough for the probes of a chunk (32 VEC at most).  In
// systems with fewer atoms than the resident blocks can take S at a time, the
// groups of a warp share atoms instead (lanes a power of two): as many atoms
// at once per block as give the resident blocks one iteration each.  Otherwise
// the blocks fill whole waves of the resident capacity, with at most 64
// atoms per block (more waves beyond that, for balance).
template <class T> FieldShape field_shape(const mbd_system *s, int ld, int terms = MBD_TERM_ALL) {
    constexpr int VEC = field_vec<T>();
    const bool pairs = !real_on_clusters(s, ld, (int)sizeof(T), terms);
    int occ = 1;
    switch (s->p) {
#define MBD_FIELD_OCC(P) \
    case P: occ = pairs ? field_occupancy<T, P, true>() : field_occupancy<T, P, false>(); break;
        MBD_SPLINE_ORDERS(MBD_FIELD_OCC)
#undef MBD_FIELD_OCC
        default: break;
    }
    FieldShape f;
    f.chunks = (ld + 32 * VEC - 1) / (32 * VEC);
    f.lanes = std::min(32, ld / VEC);
    const long long per_wave = std::max(1, occ * std::max(1, s->num_sms) / f.chunks);
    f.teams = 32 / f.lanes;
    const long long want = (s->N + per_wave - 1) / per_wave;   // atoms per resident block
    if (want < f.teams) {
        int l = 1;
        while (l < f.lanes) l *= 2;
        f.lanes = l;
        f.teams = 32 / l;
        while (f.teams > 1 && f.teams / 2 >= want) f.teams /= 2;
    }
    if (s->tune_field_apb > 0 && tuned_for<T>(s, ld)) {
        f.apb = s->tune_field_apb;
    } else {
        // at most 64 in whole iterations of `teams` atoms (launch choices hold no more)
        const long long most = 64 / f.teams * f.teams * per_wave, waves = (s->N + most - 1) / most;
        f.apb = (int)std::max<long long>(1, (s->N + waves * per_wave - 1) / (waves * per_wave));
    }
    f.apb = (f.apb + f.teams - 1) / f.teams * f.teams;
    f.blocks = (s->N + f.apb - 1) / f.apb;
    return f;
}
// The streaming kernel: FP32 with the real space on clusters, at least 32
// probes (four groups per warp at most), whole iterations' worth of atoms, the
// mesh term wanted.
constexpr int kFieldStreamLanes = 8;
bool field_streams(const mbd_system *s, int ld, const FieldShape &f, int terms) {
    return s->precision != MBD_FP64 && real_on_clusters(s, ld, 4, terms) && f.lanes >= kFieldStreamLanes && f.teams == 32 / f.lanes &&
           (terms & MBD_TERM_RECIP);
}
}  // namespace

template <class T>
mbd_status launch_field(mbd_system *s, const T *d, const T *mesh, int R, int ld, const FieldOut<T> &o) {
    PrecData<T> &P = prec<T>(s);
    const FieldShape f = field_shape<T>(s, ld, o.terms);
    FieldArgs<T> a;
    a.d = d;
    a.mesh = mesh;
    a.R = R;
    a.ld = ld;
    a.g = geom_of(s);
    a.pr = PairView<T>{s->row_d.as<int>(), s->col_d.as<int>(), s->shift_d.as<int>(), P.pairA.template as<T>()};
    a.rec = P.frec.template as<unsigned char>();
    a.g_at = s->g_d.as<double>();
    a.w2 = s->w2_d.as<double>();
    a.self_coef = -4.0 * s->ewald_beta * s->ewald_beta * s->ewald_beta / (3.0 * 1.77245385090551602730);
    const bool pairs = !real_on_clusters(s, ld, (int)sizeof(T), o.terms);
    a.ereal = pairs ? nullptr : P.ereal.template as<T>();
    a.o = o;
    a.lanes = f.lanes;
    a.teams = f.teams;
    a.apb = f.apb;
    const dim3 grid(f.blocks, f.chunks);
    const bool early = step_early(s, ld, (int)sizeof(T));
    if constexpr (sizeof(T) == 4) {
        if (field_streams(s, ld, f, o.terms)) {
            switch (s->p) {
#define MBD_FIELD_ORDER(P)                                                                                        \
    case P: {                                                                                                     \
        const size_t smem = field_stream_smem<P>(f.teams);                                                        \
        MBD_CUDA_TRY(allow_smem(k_field_stream<P>, smem, field_stream_smem<P>(32 / kFieldStreamLanes)));          \
        launch_pdl(early, k_field_stream<P>, grid, dim3(field_warps<P>() * 32), smem, s->stream, a);               \
        break;                                                                                                    \
    }
                MBD_SPLINE_ORDERS(MBD_FIELD_ORDER)
#undef MBD_FIELD_ORDER
            }
            MBD_LAUNCH_CHECK();
            return MBD_OK;
        }
    }
    switch (s->p) {
#define MBD_FIELD_ORDER(P)                                                                \
    case P:                                                                               \
        launch_pdl(early, pairs ? k_field<T, P, true> : k_field<T, P, false>, grid,       \
                   dim3(field_warps<P>() * 32), 0, s->stream, a);                         \
        break;
        MBD_SPLINE_ORDERS(MBD_FIELD_ORDER)
#undef MBD_FIELD_ORDER
        default: return MBD_ERR_UNSUPPORTED;
    }
    MBD_LAUNCH_CHECK();
    return MBD_OK;
}

int field_apb(const mbd_system *s, int ld) {
    return s->precision == MBD_FP64 ? field_shape<double>(s, ld).apb : field_shape<float>(s, ld).apb;
}
int field_blocks(const mbd_system *s, int ld) {
    return s->precision == MBD_FP64 ? field_shape<double>(s, ld).blocks : field_shape<float>(s, ld).blocks;
}

// Chunks of probes of the cluster kernel: at most 64 probes each (FP64: 32), and
// down to 16 where fewer would leave less than two blocks per SM.
template <class T> int real_chunks(const mbd_system *s, int ld) {
    constexpr int most = 256 / (int)sizeof(T);
    const int least = (ld + most - 1) / most, want = (2 * std::max(1, s->num_sms) + s->n_clusters - 1) /
                                                     std::max(1, s->n_clusters);
    return std::max(least, std::min(want, ld / 16));
}
// The real-space field runs on the clusters when they were built and atoms x
// probes are enough to fill the GPU with them; smaller systems keep the pair
// loop of the field kernel, whose groups split the neighbours of one atom.
// Measured per Lanczos step, pairs against clusters: 1200 atoms x 128 probes 188
// and 195 us; 3000 x 32 122 and 131, x 64 224 and 210; 6000 x 16 156 and 157, x 32
// 260 and 240; 15,000 x 2 (padded to 4) 203 and 240.  Without the mesh term the pair loop
// has the kernel to itself and keeps up for longer (us per mbd_field of the real space,
// r_cut 9: 1500 x 128 52 and 62, 3000 x 128 66 and 76, 12,000 x 32 68 and 81, x 64 128 and 115,
// 24,000 x 32 145 and 136).  FP64, bound by its arithmetic either way, takes them with
// four blocks per SM.
constexpr long long kRealMinValues = 160 * 1024, kRealMinValuesLocal = 512 * 1024;
bool real_on_clusters(const mbd_system *s, int ld, int real_bytes, int terms) {
    if (!s->real_clusters || s->real_method == MBD_REAL_PAIRS) return false;
    if (s->real_method == MBD_REAL_CLUSTERS) return true;
    if (real_bytes == 8) return (long long)s->n_clusters * ((ld + 31) / 32) >= 4LL * std::max(1, s->num_sms);
    return (long long)s->N * ld >= (terms & MBD_TERM_RECIP ? kRealMinValues : kRealMinValuesLocal);
}

// E_real of every atom from the clusters (the caller runs this before
// launch_field whenever real_on_clusters holds and the real-space term is wanted).
template <class T>
mbd_status launch_real_clusters(mbd_system *s, const T *d, T *ereal, int ld, cudaStream_t st, bool local) {
    PrecData<T> &P = prec<T>(s);
    constexpr int VEC = 16 / (int)sizeof(T);
    if (s->n_clusters == 0) return MBD_OK;
    const int chunks = real_chunks<T>(s, ld);
    RealArgs<T> a;
    a.d = d;
    a.out = ereal;
    a.ld = ld;
    a.N = s->N;
    a.order = s->order_d.as<int>();
    a.pstart = s->cl_pstart.as<int>();
    a.ecnt = s->cl_ecnt.as<int>();
    a.rcnt = s->cl_rcnt.as<int>();
    a.entries = s->cl_entries.as<int>();
    a.recs = P.cA.template as<RealDuo<T>>();
    a.np = ((ld + chunks - 1) / chunks + VEC - 1) / VEC * VEC;
    a.ce = std::min(kRealMaxEntries, kRealStageBytes / (3 * a.np * (int)sizeof(T)));
    dim3 grid((unsigned)s->n_clusters, (unsigned)((ld + a.np - 1) / a.np));
    auto bytes = [](size_t ce, size_t dipoles) {
        return sizeof(RealDuo<T>) * kClusterSize * kRealBatch + 16 * ((8 * ce + 15) / 16) + dipoles;
    };
    const size_t smem = bytes(a.ce, sizeof(T) * 3 * (size_t)a.np * a.ce);
    auto kern = sizeof(T) == 8 || local ? k_real_clusters<T, true> : k_real_clusters<T, sizeof(T) == 8>;
    MBD_CUDA_TRY(allow_smem(kern, smem, bytes(kRealMaxEntries, kRealStageBytes)));
    kern<<<grid, 16 * kClusterSize, smem, st>>>(a);
    MBD_LAUNCH_CHECK();
    return MBD_OK;
}

template mbd_status build_spread_records<double>(mbd_system *);
template mbd_status build_spread_records<float>(mbd_system *);
template mbd_status launch_spread<double>(mbd_system *, const double *, double *, int, int);
template mbd_status launch_spread<float>(mbd_system *, const float *, float *, int, int);
template mbd_status launch_convolve<double>(mbd_system *, double *, int, bool, bool);
template mbd_status launch_convolve<float>(mbd_system *, float *, int, bool, bool);
template mbd_status launch_spread_fft3<double>(mbd_system *, const double *, double *, int, int);
template mbd_status launch_spread_fft3<float>(mbd_system *, const float *, float *, int, int);
template mbd_status launch_field<double>(mbd_system *, const double *, const double *, int, int,
                                         const FieldOut<double> &);
template mbd_status launch_field<float>(mbd_system *, const float *, const float *, int, int,
                                        const FieldOut<float> &);
template mbd_status launch_real_clusters<double>(mbd_system *, const double *, double *, int, cudaStream_t, bool);
template mbd_status launch_real_clusters<float>(mbd_system *, const float *, float *, int, cudaStream_t, bool);

}  // namespace mbd

// K10: batched Krylov vector operations on B independent bases
// (the outer image step has B = 1; Solve-OF has one basis per frame pair).
//
// A basis is stored as V[b][j][N] (vector j of problem b contiguous), with
// the current size K[b] in device memory, so kernel grids never depend on
// the basis size and a whole solver iteration can be replayed as a graph.
//
// Reductions (dot products, norms) are deterministic: products in the
// storage precision, summed in a fixed tree within a chunk of CHUNK
// elements, chunk partials written out and combined in FP64 in chunk order.
#include "common.cuh"
#include "solver.cuh"

#include <atomic>
#include <type_traits>

namespace mof {

constexpr int KT = 256;                    // threads per block
constexpr int KE = 8;                      // elements per thread per chunk (norms, scalar paths)
constexpr int CHUNK = KT * KE;             // elements per chunk of the scalar kernels
constexpr int DCH_BYTES = 16384;           // bytes of one staged right-hand chunk of the multi-dot
template <typename real>
constexpr int dch() { return DCH_BYTES / (int)sizeof(real); }  // elements per multi-dot chunk

long long krylov_chunks(long long N) { return (N + CHUNK - 1) / CHUNK; }
template <typename real>
long long mdot_chunks(long long N) { return (N + dch<real>() - 1) / dch<real>(); }

// block-wide sum of one value per thread into thread 0's return (FP64 across warps)
template <typename acc_t>
__device__ __forceinline__ double block_sum_to_double(acc_t v, double *sh) {
    if constexpr (sizeof(acc_t) == 4) v = warp_sumf(v);
    else v = warp_sum(v);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) sh[w] = (double)v;
    __syncthreads();
    double r = 0.0;
    if (threadIdx.x == 0)
        for (int i = 0; i < KT / 32; ++i) r += sh[i];
    __syncthreads();
    return r;
}

// partial[b][chunk][v][j] = sum_{i in chunk} V[b][j][i] * x_v[b][i], j < K[b], v < NV.
// EXACT (FP32 data only): error-free accumulation per lane (DFAcc), lanes summed in FP64;
// used for the Gram matrices whose projected residual subtracts nearly equal terms.
// The NV right-hand chunks are staged in shared memory; warp w streams the
// basis vectors j = w, w + 8, ... of the chunk (16-byte loads when VEC) and
// reduces each dot once.
template <typename real, int NV, bool VEC, bool EXACT = false>
__global__ void __launch_bounds__(KT) k_mdot(const real *__restrict__ V, long long N, int Kmax, const int *__restrict__ K,
                                             const int *__restrict__ act, DotVecs<real> xs, double *__restrict__ partial,
                                             int nchunk) {
    constexpr int DCH = dch<real>();
    __shared__ __align__(16) real sx[NV][DCH];
    const int b = blockIdx.y, chunk = blockIdx.x;
    if (act && !act[b]) return;
    const int Kb = min(K[b], Kmax);
    const long long c0 = (long long)chunk * DCH;
    const int len = (int)min((long long)DCH, N - c0);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        const real *xb = xs.x[v] + b * xs.stride[v] + c0;
        for (int i = threadIdx.x; i < DCH; i += KT) sx[v][i] = i < len ? xb[i] : (real)0;
    }
    __syncthreads();
    const real *Vb = V + (long long)b * Kmax * N + c0;
    if constexpr (EXACT && sizeof(real) == 4) {
        for (int j = w; j < Kb; j += KT / 32) {
            const real *vj = Vb + (long long)j * N;
            DFAcc a[NV];
            for (int i = l; i < len; i += 32) {
                const float q = vj[i];
#pragma unroll
                for (int v = 0; v < NV; ++v) a[v].add_prod(q, sx[v][i]);
            }
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                const double t = warp_sum(a[v].value());
                if (l == 0) partial[(((long long)b * nchunk + chunk) * NV + v) * Kmax + j] = t;
            }
        }
        return;
    }
    for (int j = w; j < Kb; j += KT / 32) {
        const real *vj = Vb + (long long)j * N;
        if constexpr (VEC) {
            // FP32: each step's 16 products per right-hand side summed in FP32, the steps'
            // partials accumulated with their rounding errors (DFAcc::add), lanes in FP64
            DFAcc a[NV];
            const float4 *v4 = reinterpret_cast<const float4 *>(vj);
            const int n4 = len >> 2;
            int i = l;
#pragma unroll 1
            for (; i + 96 < n4; i += 128) {
                const float4 q0 = __ldcs(v4 + i), q1 = __ldcs(v4 + i + 32), q2 = __ldcs(v4 + i + 64), q3 = __ldcs(v4 + i + 96);
#pragma unroll
                for (int v = 0; v < NV; ++v) {
                    const float4 *x4 = reinterpret_cast<const float4 *>(sx[v]);
                    const float4 y0 = x4[i], y1 = x4[i + 32], y2 = x4[i + 64], y3 = x4[i + 96];
                    float t = q0.x * y0.x + q0.y * y0.y + q0.z * y0.z + q0.w * y0.w;
                    t += q1.x * y1.x + q1.y * y1.y + q1.z * y1.z + q1.w * y1.w;
                    t += q2.x * y2.x + q2.y * y2.y + q2.z * y2.z + q2.w * y2.w;
                    t += q3.x * y3.x + q3.y * y3.y + q3.z * y3.z + q3.w * y3.w;
                    a[v].add(t);
                }
            }
            for (; i < n4; i += 32) {
                const float4 q = __ldcs(v4 + i);
#pragma unroll
                for (int v = 0; v < NV; ++v) {
                    const float4 y = reinterpret_cast<const float4 *>(sx[v])[i];
                    a[v].add(q.x * y.x + q.y * y.y + q.z * y.z + q.w * y.w);
                }
            }
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                const double t = warp_sum(a[v].value());
                if (l == 0) partial[(((long long)b * nchunk + chunk) * NV + v) * Kmax + j] = t;
            }
        } else {
            real a[NV];
#pragma unroll
            for (int v = 0; v < NV; ++v) a[v] = 0;
            for (int i = l; i < len; i += 32) {
                const real q = vj[i];
#pragma unroll
                for (int v = 0; v < NV; ++v) a[v] += q * sx[v][i];
            }
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                real t = a[v];
                if constexpr (sizeof(real) == 4) t = warp_sumf(t);
                else t = warp_sum(t);
                if (l == 0) partial[(((long long)b * nchunk + chunk) * NV + v) * Kmax + j] = (double)t;
            }
        }
    }
}

// out_v[b*bstride + i*istride + col*jstride] = sign * sum_chunk partial[b][chunk][v][i], i < K[b];
// col = K[b] - 1 when last_col, else 0. One warp per output (lanes stride
// over the chunks, then a fixed tree), blockIdx.y = problem.
constexpr int SUMT = 256;
__global__ void __launch_bounds__(SUMT) k_sum_chunks(const double *__restrict__ partial, int nchunk, int NV, int Kmax,
                                                     const int *__restrict__ K, const int *__restrict__ act, DotOuts outs) {
    const int b = blockIdx.y;
    if (act && !act[b]) return;
    const int Kb = min(K[b], Kmax);
    const int e = blockIdx.x * (SUMT / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (e >= NV * Kb) return;
    const int v = e / Kb, i = e - (e / Kb) * Kb;
    const DotOut &o = outs.o[v];
    if (!o.out) return;
    double s = 0.0;
#pragma unroll 8
    for (int c = lane; c < nchunk; c += 32) s += partial[(((long long)b * nchunk + c) * NV + v) * Kmax + i];
    s = warp_sum(s);
    if (lane == 0) {
        const long long col = o.last_col ? (long long)(Kb - 1) : 0;
        o.out[b * o.bstride + (long long)i * o.istride + col * o.jstride] = o.sign * s;
    }
}

// out[b] = sum_j V[b][j] c[b][j] (mode 0), x[b] - sum_j V[b][j] c[b][j] (mode 1),
// sum_j V[b][j] c[b][j] - x[b] (mode 2); optionally ||out[b]||^2 per block.
// One thread per 4 consecutive elements (16-byte loads when VEC), basis
// vectors streamed four at a time.
constexpr int CT = 256;
template <typename real, int MODE, bool VEC>
__global__ void __launch_bounds__(CT) k_combine(const real *__restrict__ V, long long N, int Kmax, const int *__restrict__ K,
                                                const int *__restrict__ act, const double *__restrict__ c, long long cstride,
                                                const real *__restrict__ x, long long xstride, real *__restrict__ out,
                                                long long ostride, double *__restrict__ nrm_partial, int nblk) {
    __shared__ real sc[64];
    __shared__ double sh[CT / 32];
    const int b = blockIdx.y;
    if (act && !act[b]) return;
    const int Kb = min(K[b], Kmax);
    for (int j = threadIdx.x; j < Kb; j += CT) sc[j] = (real)c[b * cstride + j];
    __syncthreads();
    const long long i4 = ((long long)blockIdx.x * CT + threadIdx.x) * 4;
    const real *Vb = V + (long long)b * Kmax * N;
    real n2 = 0;
    if (i4 < N) {
        real acc[4] = {0, 0, 0, 0};
        if (VEC && i4 + 3 < N) {
            int j = 0;
            for (; j + 3 < Kb; j += 4) {
                const float4 q0 = __ldcs(reinterpret_cast<const float4 *>(Vb + (long long)j * N + i4));
                const float4 q1 = __ldcs(reinterpret_cast<const float4 *>(Vb + (long long)(j + 1) * N + i4));
                const float4 q2 = __ldcs(reinterpret_cast<const float4 *>(Vb + (long long)(j + 2) * N + i4));
                const float4 q3 = __ldcs(reinterpret_cast<const float4 *>(Vb + (long long)(j + 3) * N + i4));
                const real c0 = sc[j], c1 = sc[j + 1], c2 = sc[j + 2], c3 = sc[j + 3];
                acc[0] += q0.x * c0 + q1.x * c1 + q2.x * c2 + q3.x * c3;
                acc[1] += q0.y * c0 + q1.y * c1 + q2.y * c2 + q3.y * c3;
                acc[2] += q0.z * c0 + q1.z * c1 + q2.z * c2 + q3.z * c3;
                acc[3] += q0.w * c0 + q1.w * c1 + q2.w * c2 + q3.w * c3;
            }
            for (; j < Kb; ++j) {
                const float4 q = __ldcs(reinterpret_cast<const float4 *>(Vb + (long long)j * N + i4));
                const real cj = sc[j];
                acc[0] += q.x * cj;
                acc[1] += q.y * cj;
                acc[2] += q.z * cj;
                acc[3] += q.w * cj;
            }
        } else {
            for (int j = 0; j < Kb; ++j) {
                const real cj = sc[j];
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (i4 + e < N) acc[e] += Vb[(long long)j * N + i4 + e] * cj;
            }
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const long long i = i4 + e;
            if (i < N) {
                const real v = MODE == 1 ? x[b * xstride + i] - acc[e] : (MODE == 2 ? acc[e] - x[b * xstride + i] : acc[e]);
                out[b * ostride + i] = v;
                n2 += v * v;
            }
        }
    }
    if (nrm_partial) {
        const double s = block_sum_to_double(n2, sh);
        if (threadIdx.x == 0) nrm_partial[(long long)b * nblk + blockIdx.x] = s;
    }
}

// ------------------------------------------------------------ fused CGS2 middle pass
// x'[b] = x[b] - V[b] c[b] and the chunk partials of V[b]^T x'[b] in one pass
// over V: a CTA owns one 1 KB chunk of every basis vector of its problem and
// of x, brought into shared memory by 1D bulk copies (TMA) that complete on
// an mbarrier; it forms x' for the chunk, writes it, and takes the dots from
// the same staged tile. Classical Gram-Schmidt twice then reads V three times
// instead of four. Products in the storage precision, summed per chunk in a
// fixed order (deterministic), chunks combined in FP64 by k_sum_chunks.
constexpr int SDT = 64;        // threads per CTA
constexpr int SD_BYTES = 1024; // bytes of one vector's chunk (small tiles: many CTAs per SM keep copies in flight)
template <typename real>
constexpr int sdch() { return SD_BYTES / (int)sizeof(real); }
constexpr long long MBAR_MAX_POLLS = 1LL << 22;

long long subdot_chunks(long long N, int elem_bytes) { return (N * elem_bytes + SD_BYTES - 1) / SD_BYTES; }
long long krylov_partial_doubles(long long N, int Kmax) {
    // multi-dot (<= 3 right-hand sides), norms and combines; fused pass, whose fixed-size
    // chunks hold the fewest elements (so are the most numerous) for FP64
    const long long a = krylov_chunks(N) * 3 * Kmax, b = subdot_chunks(N, 8) * (Kmax + 1);
    return a > b ? a : b;
}

__device__ __forceinline__ unsigned smem_u32(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, unsigned bytes, unsigned bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}
// Bound of the first wait of a tile (polls of the mbarrier); mof_debug_set_wait_limit
// lowers it to make the timeout path run in tests. The wait after a timeout, which only
// keeps the CTA alive until its own copies have landed, always uses MBAR_MAX_POLLS.
__device__ long long g_wait_polls = MBAR_MAX_POLLS;

// poll the mbarrier phase with a bound; false when the bound ran out
__device__ __forceinline__ bool mbar_wait(unsigned bar, unsigned phase, long long limit = MBAR_MAX_POLLS) {
    for (long long it = 0; it < limit; ++it) {
        unsigned done;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(bar), "r"(phase)
            : "memory");
        if (done) return true;
    }
    return false;
}

template <typename real>
__global__ void __launch_bounds__(SDT) k_sub_dot(const real *__restrict__ V, long long N, int Kmax, const int *__restrict__ K,
                                                 const int *__restrict__ act, const double *__restrict__ c, long long cstride,
                                                 const real *x, long long xstride, real *out, long long ostride,
                                                 double *__restrict__ partial, int nchunk, int *__restrict__ err, int kcap,
                                                 double *__restrict__ nrm_partial) {
    constexpr int CH = sdch<real>();
    constexpr int EPT = CH / SDT;  // elements per thread: 4 (FP32) or 2 (FP64), 16 bytes
    using vec_t = typename std::conditional<sizeof(real) == 4, float4, double2>::type;
    extern __shared__ __align__(128) unsigned char sd_smem[];
    real *sx = reinterpret_cast<real *>(sd_smem);  // [CH]
    real *sV = sx + CH;                            // [Kmax][CH]
    __shared__ real sc[64];
    __shared__ __align__(8) unsigned long long bar;
    const int b = blockIdx.y, chunk = blockIdx.x, tid = threadIdx.x;
    if (act && !act[b]) return;
    int Kb = min(K[b], Kmax);
    if (Kb > kcap) {  // the tile holds kcap vectors: a caller's bound was wrong
        if (tid == 0 && err) atomicOr(err, 8);
        Kb = kcap;
    }
    const long long c0 = (long long)chunk * CH;
    const int len = (int)min((long long)CH, N - c0);
    const unsigned bar_a = smem_u32(&bar);
    // the copies go out first (the thread that initialised the barrier issues them);
    // the coefficients are read while they are in flight
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar_a) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        const unsigned bytes = (unsigned)len * (unsigned)sizeof(real);
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar_a), "r"(bytes * (unsigned)(Kb + 1))
                     : "memory");
        bulk_g2s(sx, x + b * xstride + c0, bytes, bar_a);
        const real *Vb = V + (long long)b * Kmax * N + c0;
        for (int j = 0; j < Kb; ++j) bulk_g2s(sV + (long long)j * CH, Vb + (long long)j * N, bytes, bar_a);
    }
    for (int j = tid; j < Kb; j += SDT) sc[j] = (real)c[b * cstride + j];
    __syncthreads();  // sc complete, and the barrier's initialisation visible to every thread
    if (!mbar_wait(bar_a, 0, g_wait_polls)) {
        if (tid == 0 && err) atomicOr(err, 4);
        mbar_wait(bar_a, 0);  // do not leave while copies may still land
        return;
    }
    // x' = x - V c on this thread's EPT consecutive elements
    const int i0 = tid * EPT;
    real acc[EPT];
#pragma unroll
    for (int e = 0; e < EPT; ++e) acc[e] = 0;
    for (int j = 0; j < Kb; ++j) {
        const vec_t q = *reinterpret_cast<const vec_t *>(sV + (long long)j * CH + i0);
        const real cj = sc[j];
        const real *qq = reinterpret_cast<const real *>(&q);
#pragma unroll
        for (int e = 0; e < EPT; ++e) acc[e] += qq[e] * cj;
    }
    {
        vec_t xv = *reinterpret_cast<const vec_t *>(sx + i0);
        real *xx = reinterpret_cast<real *>(&xv);
#pragma unroll
        for (int e = 0; e < EPT; ++e) xx[e] = (i0 + e < len) ? xx[e] - acc[e] : (real)0;
        *reinterpret_cast<vec_t *>(sx + i0) = xv;
        real *ob = out + b * ostride + c0;
        if (i0 + EPT <= len) {
            *reinterpret_cast<vec_t *>(ob + i0) = xv;
        } else {
#pragma unroll
            for (int e = 0; e < EPT; ++e)
                if (i0 + e < len) ob[i0 + e] = xx[e];
        }
        if (nrm_partial) {  // ||x'||^2 of the chunk (the padding is zero), FP64 across the warps
            real q = 0;
#pragma unroll
            for (int e = 0; e < EPT; ++e) q += xx[e] * xx[e];
            double dq;
            if constexpr (sizeof(real) == 4) dq = (double)warp_sumf(q);
            else dq = warp_sum(q);
            __shared__ double s_nq[SDT / 32];
            if ((tid & 31) == 0) s_nq[tid >> 5] = dq;
            __syncthreads();
            if (tid == 0) {
                double t = 0.0;
                for (int wq = 0; wq < SDT / 32; ++wq) t += s_nq[wq];
                nrm_partial[(long long)b * nchunk + chunk] = t;
            }
        }
    }
    __syncthreads();
    // partial dots V_j^T x' of the chunk: warp w takes j = w, w + 4, ...
    const int w = tid >> 5, l = tid & 31;
    for (int j = w; j < Kb; j += SDT / 32) {
        real a = 0;
#pragma unroll
        for (int q = 0; q < CH / (32 * EPT); ++q) {
            const int i = (q * 32 + l) * EPT;
            const vec_t v = *reinterpret_cast<const vec_t *>(sV + (long long)j * CH + i);
            const vec_t y = *reinterpret_cast<const vec_t *>(sx + i);
            const real *vv = reinterpret_cast<const real *>(&v);
            const real *yy = reinterpret_cast<const real *>(&y);
#pragma unroll
            for (int e = 0; e < EPT; ++e)
                if (i + e < len) a += vv[e] * yy[e];
        }
        if constexpr (sizeof(real) == 4) a = warp_sumf(a);
        else a = warp_sum(a);
        if (l == 0) partial[((long long)b * nchunk + chunk) * Kmax + j] = (double)a;
    }
}

// ------------------------------------------------ Solve-OF: projection and new Gram column in one pass
// For every frame pair b (p = q = 2 GKS, one basis V of K vectors of [2][ns] values):
//   x' = r - V d                                (d = Mg^-1 V^T r, the projection coefficients)
//   y  = Ups^T Ups x'                           (pointwise: u_c (u_x x'_x + u_y x'_y))
//   dots  V^T x', V^T y, V^T q                  (q = L^T L r, the graph Laplacian of r, precomputed)
//   scalars ||x'||^2, x'^T y, x'^T q, x'^T Ups^T b
// A CTA is one warp and owns every nparts-th tile of 512 bytes per component (128 FP32 pixels):
// bulk copies stage, for each basis vector and for r, q and Ups^T b, the two segments of those
// pixels, and the segments of u_x and u_y, on one mbarrier (bounded wait). A lane holds 16 bytes of
// each component, so x', y and the dots need no barrier; the lanes' sums of eight vectors are
// reduced together (9 shuffles each instead of 40), to one vector per lane, and are accumulated in
// FP64 over the warp's tiles. Those totals (3 Kmax + 4 per warp) are reduced by k_of_pass_finish.
// Bound by HBM once enough tiles are in flight, which one warp per tile gives: (K + 4) KB of shared
// memory each, 6 to 16 warps per SM that load, compute and start the next load independently. 63
// pairs of 1024^2, K = 10 to 28: 3.4 ms per pass (0.55 of the measured copy rate) with 128-thread
// CTAs of one tile each, which loaded K, waited, and met at five barriers; 2.2 ms (0.87) so.
// 31 pairs of 256^2: 135 -> 106 us. With x' = r - V d the new vector is v = x' / ||x'|| and its Gram
// column follows from these without another pass over the basis (k_of_pass_finish):
//   G_A[i][v] = (V^T y)_i / ||x'||,   G_L[i][v] = ((V^T q)_i - (G_L d)_i) / ||x'||,
//   g[v] = x'^T Ups^T b / ||x'||,     G_A[v][v] = x'^T y / ||x'||^2,
//   G_L[v][v] = (x'^T q - d^T V^T q + d^T G_L d) / ||x'||^2,   Mg[i][v] = (V^T x')_i / ||x'||.
template <typename real>
constexpr int opx() { return 512 / (int)sizeof(real); }  // pixels per tile: 128 (FP32), 64 (FP64)

// Warps per frame pair: each takes up to OP_TILES tiles, fewer where the pairs together would not
// give the GPU's 152 x 32 warp slots one each (64^2 x 7 pairs: one tile per warp, 448 warps; 1024^2 x
// 63: eight, which spreads the start of a warp and shortens the reduction behind). A function of the
// problem alone: the sums do not depend on how the pairs are grouped.
constexpr int OP_TILES = 8;
static int of_pass_parts_of(long long ns, int pairs, int elem_bytes) {
    const long long nt = (ns * elem_bytes + 511) / 512;
    const long long T = std::max(1LL, std::min<long long>(OP_TILES, nt * pairs / (152 * 32)));
    return (int)((nt + T - 1) / T);
}
long long of_pass_parts(long long ns, int pairs) { return std::max(of_pass_parts_of(ns, pairs, 4), of_pass_parts_of(ns, pairs, 8)); }
int of_pass_stride(int Kmax) { return 3 * Kmax + 4; }

// 8 bytes of values: two FP32 or one FP64
template <typename real>
using half_t = typename std::conditional<sizeof(real) == 4, F2, double>::type;
__device__ __forceinline__ double fma2(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ double mul2(double a, double b) { return a * b; }
__device__ __forceinline__ double sub2(double a, double b) { return a - b; }
__device__ __forceinline__ float hsum(F2 a) {
    float x, y;
    unpack2(a, x, y);
    return x + y;
}
__device__ __forceinline__ double hsum(double a) { return a; }

// The sums over the warp of eight values per lane: value lane >> 2 is returned (equal in the four
// lanes of a group).
template <typename real>
__device__ __forceinline__ real warp_sums8(real (&t)[8], int lane) {
#pragma unroll
    for (int h = 4; h > 0; h >>= 1) {
        const bool up = lane & (h << 2);
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const real send = up ? t[i] : t[i + h];
            t[i] = (up ? t[i + h] : t[i]) + __shfl_xor_sync(0xffffffffu, send, h << 2);
        }
    }
    real v = t[0];
    v += __shfl_xor_sync(0xffffffffu, v, 2);
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    return v;
}

template <typename real>
__global__ void __launch_bounds__(32) k_of_proj_gram_pass(const real *V, long long ns, int Kmax, const int *__restrict__ K,
                                                         const int *__restrict__ act, const double *__restrict__ d,
                                                         const real *__restrict__ x, const real *__restrict__ q, real *to,
                                                         const real *__restrict__ AtB, const real *__restrict__ ux,
                                                         const real *__restrict__ uy, double *__restrict__ partial, int nparts,
                                                         int *__restrict__ err, int kcap) {
    constexpr int PX = opx<real>(), EPL = 16 / (int)sizeof(real);
    using half = half_t<real>;
    struct __align__(16) Q {  // a lane's 16 bytes of a segment
        half h[2];
    };
    extern __shared__ __align__(128) unsigned char op_smem[];  // segments of 512 bytes: r, q, Ups^T b (2 each), u_x, u_y, V_j (2 each)
    __shared__ half sd[64];
    __shared__ __align__(8) unsigned long long bar;
    const int b = blockIdx.y, part = blockIdx.x, lane = threadIdx.x;
    if (act && !act[b]) return;
    const int K0 = K[b];
    int Kb = min(K0, Kmax);
    if (Kb > kcap) {
        if (lane == 0 && err) atomicOr(err, 8);
        Kb = kcap;
    }
    const unsigned bar_a = smem_u32(&bar);
    if (lane == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar_a) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    const long long N2 = 2 * ns;
    const int ntile = (int)((ns + PX - 1) / PX);
    const real *Vb = V + (long long)b * Kmax * N2;
    auto fetch = [&](int tile) {
        const long long p0 = (long long)tile * PX;
        const unsigned bytes = (unsigned)min((long long)PX, ns - p0) * (unsigned)sizeof(real);  // (a multiple of 16)
        if (lane == 0)
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar_a), "r"(bytes * (unsigned)(2 * Kb + 8))
                         : "memory");
        __syncwarp();
        for (int i = lane; i < 2 * Kb + 8; i += 32) {
            const long long c = (i & 1) ? ns : 0;
            const real *src;
            if (i >= 8) src = Vb + (long long)((i - 8) >> 1) * N2 + c;
            else if (i >= 6) src = (i == 6 ? ux : uy) + b * ns;
            else src = (i < 2 ? x : (i < 4 ? q : AtB)) + b * N2 + c;
            bulk_g2s(op_smem + i * 512, src + p0, bytes, bar_a);
        }
    };
    fetch(part);
    for (int j = lane; j < Kb; j += 32) {
        if constexpr (sizeof(real) == 4) sd[j] = both((float)d[(long long)b * Kmax + j]);
        else sd[j] = d[(long long)b * Kmax + j];
    }
    __syncwarp();
    const Q *seg = reinterpret_cast<const Q *>(op_smem) + lane;  // segment i: seg[i * 32]
    double acc[3][2] = {}, acs = 0.0;
    unsigned phase = 0;
    for (int tile = part; tile < ntile; tile += nparts) {
        const long long p = (long long)tile * PX + lane * EPL;
        const bool in = p < ns;  // all of a lane's pixels or none
        if (!in) {
            Q zero;
            if constexpr (sizeof(real) == 4) zero.h[0] = zero.h[1] = both(0.f);
            else zero.h[0] = zero.h[1] = 0.0;
            for (int i = 0; i < 2 * Kb + 8; ++i) const_cast<Q *>(seg)[i * 32] = zero;
        }
        // (the warp leaves as one: a lane that went on would wait for a tile that not all lanes fetch)
        if (!__all_sync(0xffffffffu, mbar_wait(bar_a, phase, g_wait_polls))) {
            if (lane == 0 && err) atomicOr(err, 4);
            mbar_wait(bar_a, phase);  // do not leave while copies may still land
            return;
        }
        phase ^= 1;
        const Q *sv = seg + 8 * 32;
        Q xa = seg[0], xb = seg[32];
        {  // x' = r - V d
            half s[4];
            if constexpr (sizeof(real) == 4) s[0] = s[1] = s[2] = s[3] = both(0.f);
            else s[0] = s[1] = s[2] = s[3] = 0.0;
#pragma unroll 4
            for (int j = 0; j < Kb; ++j) {
                const Q va = sv[j * 64], vb = sv[j * 64 + 32];
                const half dj = sd[j];
                s[0] = fma2(va.h[0], dj, s[0]);
                s[1] = fma2(va.h[1], dj, s[1]);
                s[2] = fma2(vb.h[0], dj, s[2]);
                s[3] = fma2(vb.h[1], dj, s[3]);
            }
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                xa.h[e] = sub2(xa.h[e], s[e]);
                xb.h[e] = sub2(xb.h[e], s[2 + e]);
            }
        }
        if (in && K0 < Kmax) {  // into the slot behind the basis, where an append finds it (a full basis appends nothing)
            real *ob = to + ((long long)b * Kmax + Kb) * N2 + p;
            *reinterpret_cast<Q *>(ob) = xa;
            *reinterpret_cast<Q *>(ob + ns) = xb;
        }
        // y = Ups^T Ups x' and the four scalars
        Q ya, yb;
        const Q qa = seg[64], qb = seg[96];
        {
            const Q fx = seg[6 * 32], fy = seg[7 * 32], aa = seg[4 * 32], ab = seg[5 * 32];
            half s[4];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const half w = fma2(fx.h[e], xa.h[e], mul2(fy.h[e], xb.h[e]));
                ya.h[e] = mul2(fx.h[e], w);
                yb.h[e] = mul2(fy.h[e], w);
                s[0] = e ? fma2(xa.h[e], xa.h[e], s[0]) : mul2(xa.h[e], xa.h[e]);
                s[1] = e ? fma2(xa.h[e], ya.h[e], s[1]) : mul2(xa.h[e], ya.h[e]);
                s[2] = e ? fma2(xa.h[e], qa.h[e], s[2]) : mul2(xa.h[e], qa.h[e]);
                s[3] = e ? fma2(xa.h[e], aa.h[e], s[3]) : mul2(xa.h[e], aa.h[e]);
                s[0] = fma2(xb.h[e], xb.h[e], s[0]);
                s[1] = fma2(xb.h[e], yb.h[e], s[1]);
                s[2] = fma2(xb.h[e], qb.h[e], s[2]);
                s[3] = fma2(xb.h[e], ab.h[e], s[3]);
            }
            real t[8] = {hsum(s[0]), hsum(s[1]), hsum(s[2]), hsum(s[3]), 0, 0, 0, 0};
            acs += (double)warp_sums8(t, lane);
        }
        // dots of the basis vectors with x', y and q: eight vectors at a time, four such blocks to a
        // value per lane (lane l: vector 8 (l & 3) + (l >> 2) of the 32)
#pragma unroll
        for (int jb = 0; jb < 2; ++jb) {
            if (jb * 32 >= Kb) break;
            real v1 = 0, v2 = 0, v3 = 0;
#pragma unroll 1
            for (int g = 0; g < 4; ++g) {
                const int j0 = jb * 32 + g * 8;
                if (j0 >= Kb) break;
                real t1[8], t2[8], t3[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    t1[i] = t2[i] = t3[i] = 0;
                    if (j0 + i < Kb) {
                        const Q va = sv[(j0 + i) * 64], vb = sv[(j0 + i) * 64 + 32];
                        t1[i] = hsum(fma2(vb.h[1], xb.h[1], fma2(vb.h[0], xb.h[0], fma2(va.h[1], xa.h[1], mul2(va.h[0], xa.h[0])))));
                        t2[i] = hsum(fma2(vb.h[1], yb.h[1], fma2(vb.h[0], yb.h[0], fma2(va.h[1], ya.h[1], mul2(va.h[0], ya.h[0])))));
                        t3[i] = hsum(fma2(vb.h[1], qb.h[1], fma2(vb.h[0], qb.h[0], fma2(va.h[1], qa.h[1], mul2(va.h[0], qa.h[0])))));
                    }
                }
                const real u1 = warp_sums8(t1, lane), u2 = warp_sums8(t2, lane), u3 = warp_sums8(t3, lane);
                const bool mine = (lane & 3) == g;
                v1 = mine ? u1 : v1;
                v2 = mine ? u2 : v2;
                v3 = mine ? u3 : v3;
            }
            acc[0][jb] += (double)v1;
            acc[1][jb] += (double)v2;
            acc[2][jb] += (double)v3;
        }
        if (tile + nparts < ntile) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();  // every lane has read the tile
            fetch(tile + nparts);
        }
    }
    // stored output-major, [b][output][warp], so that the reduction reads each output contiguously
    double *out = partial + (long long)b * (3 * Kmax + 4) * nparts + part;
#pragma unroll
    for (int jb = 0; jb < 2; ++jb) {
        const int j = jb * 32 + 8 * (lane & 3) + (lane >> 2);
        if (j < Kb)
#pragma unroll
            for (int c = 0; c < 3; ++c) out[(long long)(c * Kmax + j) * nparts] = acc[c][jb];
    }
    if (lane < 16 && !(lane & 3)) out[(long long)(3 * Kmax + (lane >> 2)) * nparts] = acs;
}

// ||x[b]||^2 per chunk
template <typename real, bool EXACT = false>
__global__ void __launch_bounds__(KT) k_norm2(const real *__restrict__ x, long long N, long long xstride,
                                              double *__restrict__ partial, int nchunk) {
    __shared__ double sh[KT / 32];
    const int b = blockIdx.y, chunk = blockIdx.x;
    const long long i0 = (long long)chunk * CHUNK + threadIdx.x;
    if constexpr (EXACT && sizeof(real) == 4) {
        DFAcc a;
#pragma unroll
        for (int e = 0; e < KE; ++e) {
            const long long i = i0 + (long long)e * KT;
            if (i < N) {
                const float v = x[b * xstride + i];
                a.add_prod(v, v);
            }
        }
        const double s = block_sum_to_double(a.value(), sh);
        if (threadIdx.x == 0) partial[(long long)b * nchunk + chunk] = s;
        return;
    }
    real n2 = 0;
#pragma unroll
    for (int e = 0; e < KE; ++e) {
        const long long i = i0 + (long long)e * KT;
        if (i < N) {
            const real v = x[b * xstride + i];
            n2 += v * v;
        }
    }
    const double s = block_sum_to_double(n2, sh);
    if (threadIdx.x == 0) partial[(long long)b * nchunk + chunk] = s;
}

// out[b] = sum_chunk partial[b][chunk], one warp per problem
__global__ void k_sum_scalar_chunks(const double *__restrict__ partial, int nchunk, double *__restrict__ out, int B) {
    const int b = blockIdx.x, lane = threadIdx.x;
    if (b >= B) return;
    double s = 0.0;
#pragma unroll 8
    for (int c = lane; c < nchunk; c += 32) s += partial[(long long)b * nchunk + c];
    s = warp_sum(s);
    if (lane == 0) out[b] = s;
}

// Append x[b] / ||x[b]|| as vector K[b] when ||x[b]|| > tol * scale[b] and the
// problem is still growing (scale == null: only ||x|| > 0 is required); the
// new vector is also written to stage[b] when stage != null.
__device__ __forceinline__ bool append_ok(int grow, int Kb, int Kmax, double nrm2, const double *scale, int b, double tol) {
    const double nr = sqrt(nrm2);
    const double sc = scale ? scale[b] : 0.0;
    return grow && Kb < Kmax && (nr > tol * sc) && (nr > 0.0) && isfinite(nr);
}

// The per-problem decision and scale of an append, once per problem (FP64):
// slot[b] = K[b] and inv[b] = 1/||x[b]|| when the vector is appended (then
// K[b] += 1), slot[b] = -1 and grow[b] = 0 otherwise; appended[b] (may be
// null) records which. k_append's threads then do no FP64 arithmetic.
template <typename real>
__global__ void k_append_prep(int *__restrict__ K, int Kmax, const double *__restrict__ nrm2, const double *__restrict__ scale,
                              double tol, int *__restrict__ grow, int B, int *__restrict__ slot, real *__restrict__ inv,
                              int *__restrict__ appended) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B) return;
    const int Kb = K[b];
    const bool ok = append_ok(grow[b], Kb, Kmax, nrm2[b], scale, b, tol);
    slot[b] = ok ? Kb : -1;
    inv[b] = ok ? (real)(1.0 / sqrt(nrm2[b])) : (real)0;
    if (ok) K[b] = Kb + 1;
    else grow[b] = 0;
    if (appended) appended[b] = ok;
}

// The same with ||x[b]||^2 summed here from the per-block partials of the update
// that formed x (one warp per problem, lanes over the partials, then a fixed tree:
// the order of k_sum_scalar_chunks), written to nrm2_out, and sqrt(||x[b]||^2)
// written to sq1[b] and sq2[b] (each may be null) for problems still growing
// (grow[b] as it was on entry).
template <typename real>
__global__ void k_append_prep_sum(int *__restrict__ K, int Kmax, const double *__restrict__ parts, int nparts,
                                  double *__restrict__ nrm2_out, const double *__restrict__ scale, double tol,
                                  int *__restrict__ grow, int B, int *__restrict__ slot, real *__restrict__ inv,
                                  int *__restrict__ appended, double *__restrict__ sq1, double *__restrict__ sq2) {
    const int b = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (b >= B) return;
    double s = 0.0;
#pragma unroll 8
    for (int c = lane; c < nparts; c += 32) s += parts[(long long)b * nparts + c];
    s = warp_sum(s);
    if (lane != 0) return;
    nrm2_out[b] = s;
    const int g = grow[b];
    if (g) {
        const double r = sqrt(s);
        if (sq1) sq1[b] = r;
        if (sq2) sq2[b] = r;
    }
    const int Kb = K[b];
    const bool ok = append_ok(g, Kb, Kmax, s, scale, b, tol);
    slot[b] = ok ? Kb : -1;
    inv[b] = ok ? (real)(1.0 / sqrt(s)) : (real)0;
    if (ok) K[b] = Kb + 1;
    else grow[b] = 0;
    if (appended) appended[b] = ok;
}

template <typename real>
__global__ void __launch_bounds__(KT) k_append(real *__restrict__ V, long long N, int Kmax, const int *__restrict__ slot,
                                               const real *__restrict__ inv, const real *__restrict__ x, long long xstride,
                                               real *__restrict__ stage) {
    const int b = blockIdx.y;
    const int sl = slot[b];
    if (sl < 0) return;
    const real iv = inv[b];
    real *vd = V + ((long long)b * Kmax + sl) * N;
    for (long long i = blockIdx.x * (long long)KT + threadIdx.x; i < N; i += (long long)gridDim.x * KT) {
        const real v = x[b * xstride + i] * iv;
        vd[i] = v;
        if (stage) stage[b * N + i] = v;
    }
}

// ------------------------------------------------------------ Golub-Kahan half-steps
// A half-step forms x = (operator applied to the other side's vector) - c v_prev, takes it out of
// the basis once more (x' = x - V V^T x; V^T x = 0 by the recurrence) and appends x' / ||x'||.
// k_gk_dots forms x (by FRONT, below) and V^T x, k_gk_sub forms x' in the slot behind the basis and
// ||x'||; the last CTA of a problem to finish (counter done[b], left at zero) adds the partials and,
// in k_gk_sub, takes the append decision (as k_append_prep_sum). The vector's scale 1 / ||x'|| is
// applied by the next half-step's front, which reads the vector anyway, or by k_gk_scale. Two
// launches and 11 + 4 K passes over ns values per half-step on the V side of Solve-OF instead of six
// and 17 + 4 K: bound by HBM on large frames (63 pairs of 1024^2, 10 steps: 31.4 -> 23.3 ms), by the
// launches and the last CTA on small ones (31 pairs of 256^2: 1.74 -> 0.99 ms; image step of 64^2 x 8
// in FP64 with its projections: 1.90 -> 1.52 ms).
//   FRONT 0: x = a - coef prev (prev may be null: x = a, which is then not written)
//   FRONT 1: x = Ups^T u - coef prev, u of N / 2 values (prev may be null)
//   FRONT 2: x = Ups v - coef prev, v of 2 N values
// FRONT 1, 2: u / v is multiplied by inv[b] and written back first when inv is given.
template <typename real, int FRONT, bool VEC>
__global__ void __launch_bounds__(KT) k_gk_dots(const real *V, long long N, int Kmax, const int *__restrict__ K,
                                                const int *__restrict__ act, GkFront<real> f, double *__restrict__ partial,
                                                int nchunk, double *__restrict__ out, int *done) {
    // a chunk: FRONT 1: the same DCH / 2 pixels of both components
    constexpr int DCH = dch<real>(), SEG = FRONT == 1 ? 2 : 1, PER = DCH / SEG, W = VEC ? 4 : 1;
    __shared__ __align__(16) real sx[DCH];
    __shared__ int s_last;
    const int b = blockIdx.y, chunk = blockIdx.x, tid = threadIdx.x, w = tid >> 5, l = tid & 31;
    if (act && !act[b]) return;
    const int Kb = min(K[b], Kmax);
    const long long L = N / SEG, c0 = (long long)chunk * PER;
    const int len = (int)min((long long)PER, L - c0);
    struct __align__(W * sizeof(real)) Vec {
        real v[W];
    };
    auto ld = [](const real *q) { return *reinterpret_cast<const Vec *>(q); };
    auto st = [](real *q, const Vec &v) { *reinterpret_cast<Vec *>(q) = v; };
    const real cf = f.prev ? (real)f.coef[b] : (real)0, iv = f.inv ? f.inv[b] : (real)1;
    const real *pb = f.prev ? f.prev + b * f.pstride + c0 : nullptr;
    real *xb = f.x + b * f.xstride + c0;
    for (int i = tid * W; i < PER; i += KT * W) {
        Vec x[SEG];
#pragma unroll
        for (int g = 0; g < SEG; ++g)
#pragma unroll
            for (int e = 0; e < W; ++e) x[g].v[e] = 0;
        if (i < len) {
            if constexpr (FRONT == 0) {
                x[0] = ld(f.a + b * f.astride + c0 + i);
            } else {
                const Vec ax = ld(f.ux + b * f.fstride + c0 + i), ay = ld(f.uy + b * f.fstride + c0 + i);
                real *ab = f.s + b * f.astride + c0 + i;
                Vec u = ld(ab);
                if constexpr (FRONT == 1) {
                    if (f.inv) {
#pragma unroll
                        for (int e = 0; e < W; ++e) u.v[e] *= iv;
                        st(ab, u);
                    }
#pragma unroll
                    for (int e = 0; e < W; ++e) {
                        x[0].v[e] = ax.v[e] * u.v[e];
                        x[SEG - 1].v[e] = ay.v[e] * u.v[e];
                    }
                } else {
                    Vec u1 = ld(ab + N);
                    if (f.inv) {
#pragma unroll
                        for (int e = 0; e < W; ++e) {
                            u.v[e] *= iv;
                            u1.v[e] *= iv;
                        }
                        st(ab, u);
                        st(ab + N, u1);
                    }
#pragma unroll
                    for (int e = 0; e < W; ++e) x[0].v[e] = ax.v[e] * u.v[e] + ay.v[e] * u1.v[e];
                }
            }
            if (pb) {
#pragma unroll
                for (int g = 0; g < SEG; ++g) {
                    const Vec q = ld(pb + g * L + i);
#pragma unroll
                    for (int e = 0; e < W; ++e) x[g].v[e] -= cf * q.v[e];
                }
            }
            if (FRONT != 0 || pb)
#pragma unroll
                for (int g = 0; g < SEG; ++g) st(xb + g * L + i, x[g]);
        }
#pragma unroll
        for (int g = 0; g < SEG; ++g) st(sx + g * PER + i, x[g]);
    }
    __syncthreads();
    double *pt = partial + (long long)b * Kmax * nchunk;  // [vector][chunk]
    const real *Vb = V + (long long)b * Kmax * N + c0;
    for (int j = w; j < Kb; j += KT / 32) {
        const real *vj = Vb + (long long)j * N;
        double t;
        if constexpr (VEC) {  // (sums as in k_mdot)
            DFAcc a;
#pragma unroll
            for (int g = 0; g < SEG; ++g) {
                const float4 *v4 = reinterpret_cast<const float4 *>(vj + g * L), *x4 = reinterpret_cast<const float4 *>(sx + g * PER);
                const int n4 = len >> 2;
                int i = l;
#pragma unroll 1
                for (; i + 96 < n4; i += 128) {
                    const float4 q0 = v4[i], q1 = v4[i + 32], q2 = v4[i + 64], q3 = v4[i + 96];
                    const float4 y0 = x4[i], y1 = x4[i + 32], y2 = x4[i + 64], y3 = x4[i + 96];
                    float t4 = q0.x * y0.x + q0.y * y0.y + q0.z * y0.z + q0.w * y0.w;
                    t4 += q1.x * y1.x + q1.y * y1.y + q1.z * y1.z + q1.w * y1.w;
                    t4 += q2.x * y2.x + q2.y * y2.y + q2.z * y2.z + q2.w * y2.w;
                    t4 += q3.x * y3.x + q3.y * y3.y + q3.z * y3.z + q3.w * y3.w;
                    a.add(t4);
                }
                for (; i < n4; i += 32) {
                    const float4 q = v4[i], y = x4[i];
                    a.add(q.x * y.x + q.y * y.y + q.z * y.z + q.w * y.w);
                }
            }
            t = warp_sum(a.value());
        } else {
            real a = 0;
#pragma unroll
            for (int g = 0; g < SEG; ++g)
                for (int i = l; i < len; i += 32) a += vj[g * L + i] * sx[g * PER + i];
            if constexpr (sizeof(real) == 4) t = (double)warp_sumf(a);
            else t = warp_sum(a);
        }
        if (l == 0) pt[(long long)j * nchunk + chunk] = t;
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) {
        s_last = atomicAdd(done + b, 1) == (int)gridDim.x - 1;
        if (s_last) done[b] = 0;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    for (int j = w; j < Kb; j += KT / 32) {
        const double *src = pt + (long long)j * nchunk;
        double t = 0.0;
#pragma unroll 8
        for (int c = l; c < nchunk; c += 32) t += __ldcg(src + c);
        t = warp_sum(t);
        if (l == 0) out[(long long)b * Kmax + j] = t;
    }
}

template <typename real, bool VEC>
__global__ void __launch_bounds__(CT) k_gk_sub(real *V, long long N, int Kmax, int *K, const int *act, const double *__restrict__ c,
                                               const real *__restrict__ x, long long xstride, double *__restrict__ partial,
                                               int nblk, double *__restrict__ nrm2_out, const double *__restrict__ scale, double tol,
                                               int *grow, int *__restrict__ slot, real *__restrict__ inv, double *__restrict__ sq1,
                                               double *__restrict__ sq2, int *done) {
    __shared__ real sc[64];
    __shared__ double sh[CT / 32];
    __shared__ int s_last;
    const int b = blockIdx.y, tid = threadIdx.x;
    if (act && !act[b]) return;
    const int Kb = min(K[b], Kmax);
    for (int j = tid; j < Kb; j += CT) sc[j] = (real)c[(long long)b * Kmax + j];
    __syncthreads();
    const long long i4 = ((long long)blockIdx.x * CT + tid) * 4;
    const real *Vb = V + (long long)b * Kmax * N;
    real *ob = V + ((long long)b * Kmax + Kb) * N;
    const real *xb = x + b * xstride;
    const bool put = Kb < Kmax;  // a full basis appends nothing
    real n2 = 0;
    if (i4 < N) {
        real acc[4] = {0, 0, 0, 0}, v[4];
        if (VEC) {
            int j = 0;
            for (; j + 3 < Kb; j += 4) {
                const float4 q0 = *reinterpret_cast<const float4 *>(Vb + (long long)j * N + i4);
                const float4 q1 = *reinterpret_cast<const float4 *>(Vb + (long long)(j + 1) * N + i4);
                const float4 q2 = *reinterpret_cast<const float4 *>(Vb + (long long)(j + 2) * N + i4);
                const float4 q3 = *reinterpret_cast<const float4 *>(Vb + (long long)(j + 3) * N + i4);
                const real c0 = sc[j], c1 = sc[j + 1], c2 = sc[j + 2], c3 = sc[j + 3];
                acc[0] += q0.x * c0 + q1.x * c1 + q2.x * c2 + q3.x * c3;
                acc[1] += q0.y * c0 + q1.y * c1 + q2.y * c2 + q3.y * c3;
                acc[2] += q0.z * c0 + q1.z * c1 + q2.z * c2 + q3.z * c3;
                acc[3] += q0.w * c0 + q1.w * c1 + q2.w * c2 + q3.w * c3;
            }
            for (; j < Kb; ++j) {
                const float4 q = *reinterpret_cast<const float4 *>(Vb + (long long)j * N + i4);
                const real cj = sc[j];
                acc[0] += q.x * cj;
                acc[1] += q.y * cj;
                acc[2] += q.z * cj;
                acc[3] += q.w * cj;
            }
            const float4 y = *reinterpret_cast<const float4 *>(xb + i4);
            v[0] = y.x - acc[0];
            v[1] = y.y - acc[1];
            v[2] = y.z - acc[2];
            v[3] = y.w - acc[3];
            if (put) *reinterpret_cast<float4 *>(ob + i4) = make_float4(v[0], v[1], v[2], v[3]);
#pragma unroll
            for (int e = 0; e < 4; ++e) n2 += v[e] * v[e];
        } else {
            for (int j = 0; j < Kb; ++j) {
                const real cj = sc[j];
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (i4 + e < N) acc[e] += Vb[(long long)j * N + i4 + e] * cj;
            }
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (i4 + e < N) {
                    v[e] = xb[i4 + e] - acc[e];
                    if (put) ob[i4 + e] = v[e];
                    n2 += v[e] * v[e];
                }
        }
    }
    const double t = block_sum_to_double(n2, sh);
    if (tid == 0) {
        partial[(long long)b * nblk + blockIdx.x] = t;
        __threadfence();
        s_last = atomicAdd(done + b, 1) == (int)gridDim.x - 1;
        if (s_last) done[b] = 0;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    const double *src = partial + (long long)b * nblk;
    double s = 0.0;
#pragma unroll 8
    for (int q = tid; q < nblk; q += CT) s += __ldcg(src + q);
    s = block_sum_to_double(s, sh);
    if (tid != 0) return;
    nrm2_out[b] = s;
    const int g = grow[b];
    if (g) {
        const double r = sqrt(s);
        if (sq1) sq1[b] = r;
        if (sq2) sq2[b] = r;
    }
    const bool ok = append_ok(g, Kb, Kmax, s, scale, b, tol);
    slot[b] = ok ? Kb : -1;
    inv[b] = ok ? (real)(1.0 / sqrt(s)) : (real)0;
    if (ok) K[b] = Kb + 1;
    else grow[b] = 0;
}

// the vector in slot[b] (-1: none) times inv[b]
template <typename real>
__global__ void __launch_bounds__(KT) k_gk_scale(real *__restrict__ V, long long N, int Kmax, const int *__restrict__ slot,
                                                 const real *__restrict__ inv) {
    const int b = blockIdx.y, sl = slot[b];
    if (sl < 0) return;
    const real iv = inv[b];
    real *vd = V + ((long long)b * Kmax + sl) * N;
    const long long i0 = ((long long)blockIdx.x * KT + threadIdx.x) * 4;
    if (sizeof(real) == 4 && i0 + 3 < N && (reinterpret_cast<uintptr_t>(vd + i0) & 15) == 0) {
        float4 q = *reinterpret_cast<float4 *>(vd + i0);
        q.x *= (float)iv;
        q.y *= (float)iv;
        q.z *= (float)iv;
        q.w *= (float)iv;
        *reinterpret_cast<float4 *>(vd + i0) = q;
    } else {
        for (long long i = i0; i < min(i0 + 4, N); ++i) vd[i] *= iv;
    }
}

mof_status set_wait_polls(long long polls) {
    const long long v = polls < 0 ? MBAR_MAX_POLLS : (polls > MBAR_MAX_POLLS ? MBAR_MAX_POLLS : polls);
    MOF_CUDA(cudaMemcpyToSymbol(g_wait_polls, &v, sizeof(v)));
    MOF_CUDA(cudaDeviceSynchronize());
    return MOF_OK;
}

// ------------------------------------------------------------ host launchers
template <typename real>
void Krylov<real>::dots(const BasisRef<real> &B, const real *x, long long xstride, double *out, long long ostride, double sign,
                        cudaStream_t st) const {
    DotVecs<real> xs{};
    xs.x[0] = x;
    xs.stride[0] = xstride;
    DotOuts o{};
    o.o[0] = DotOut{out, ostride, 1, 0, 0, sign};
    multidot(B, 1, xs, o, st);
}

template <typename real>
static bool vec_ok(const void *base, long long N, long long stride) {
    return sizeof(real) == 4 && (N % 4) == 0 && (stride % 4) == 0 && (reinterpret_cast<uintptr_t>(base) % 16) == 0;
}

template <typename real>
void Krylov<real>::multidot(const BasisRef<real> &B, int nv, const DotVecs<real> &xs, const DotOuts &outs,
                            cudaStream_t st, bool exact) const {
    const int nc = (int)mdot_chunks<real>(B.N);
    const dim3 grid(nc, B.B);
    const bool vec = vec_ok<real>(B.V, B.N, (long long)B.Kmax * B.N);
#define MDOT(NVv)                                                                                                       \
    if (exact) ::mof::count_launch(), k_mdot<real, NVv, false, true><<<grid, KT, 0, st>>>(B.V, B.N, B.Kmax, B.K, B.act, xs, partial, nc); \
    else if (vec) ::mof::count_launch(), k_mdot<real, NVv, true><<<grid, KT, 0, st>>>(B.V, B.N, B.Kmax, B.K, B.act, xs, partial, nc); \
    else ::mof::count_launch(), k_mdot<real, NVv, false><<<grid, KT, 0, st>>>(B.V, B.N, B.Kmax, B.K, B.act, xs, partial, nc);
    if (nv == 1) {
        MDOT(1)
    } else if (nv == 2) {
        MDOT(2)
    } else {
        MDOT(3)
    }
#undef MDOT
    ::mof::count_launch(), k_sum_chunks<<<dim3((nv * B.Kmax + SUMT / 32 - 1) / (SUMT / 32), B.B), SUMT, 0, st>>>(partial, nc, nv, B.Kmax, B.K, B.act, outs);
}

template <typename real>
void Krylov<real>::combine(const BasisRef<real> &B, const double *c, long long cstride, real *out, long long ostride,
                           cudaStream_t st) const {
    const int nb = (int)((B.N + 4LL * CT - 1) / (4LL * CT));
    const bool vec = vec_ok<real>(B.V, B.N, (long long)B.Kmax * B.N) && (ostride % 4 == 0);
    if (vec)
        ::mof::count_launch(), k_combine<real, 0, true><<<dim3(nb, B.B), CT, 0, st>>>(B.V, B.N, B.Kmax, B.K, B.act, c, cstride,
                                                                                   nullptr, 0, out, ostride, nullptr, nb);
    else
        ::mof::count_launch(), k_combine<real, 0, false><<<dim3(nb, B.B), CT, 0, st>>>(B.V, B.N, B.Kmax, B.K, B.act, c, cstride,
                                                                                    nullptr, 0, out, ostride, nullptr, nb);
}

template <typename real>
void Krylov<real>::combine_minus(const BasisRef<real> &B, const double *c, long long cstride, const real *x, long long xstride,
                                 real *out, long long ostride, double *nrm2_out, cudaStream_t st) const {
    const int nb = (int)((B.N + 4LL * CT - 1) / (4LL * CT));
    const bool vec = vec_ok<real>(B.V, B.N, (long long)B.Kmax * B.N) && (ostride % 4 == 0);
    double *np = nrm2_out ? partial : nullptr;
    if (vec)
        ::mof::count_launch(), k_combine<real, 2, true><<<dim3(nb, B.B), CT, 0, st>>>(B.V, B.N, B.Kmax, B.K, B.act, c, cstride, x,
                                                                                   xstride, out, ostride, np, nb);
    else
        ::mof::count_launch(), k_combine<real, 2, false><<<dim3(nb, B.B), CT, 0, st>>>(B.V, B.N, B.Kmax, B.K, B.act, c, cstride, x,
                                                                                    xstride, out, ostride, np, nb);
    if (nrm2_out) ::mof::count_launch(), k_sum_scalar_chunks<<<B.B, 32, 0, st>>>(partial, nb, nrm2_out, B.B);
}

template <typename real>
void Krylov<real>::subtract(const BasisRef<real> &B, const double *c, long long cstride, const real *x, long long xstride,
                            real *out, long long ostride, double *nrm2_out, cudaStream_t st) const {
    const int nb = (int)((B.N + 4LL * CT - 1) / (4LL * CT));
    const bool vec = vec_ok<real>(B.V, B.N, (long long)B.Kmax * B.N) && (ostride % 4 == 0);
    double *np = nrm2_out ? partial : nullptr;
    if (vec)
        ::mof::count_launch(), k_combine<real, 1, true><<<dim3(nb, B.B), CT, 0, st>>>(B.V, B.N, B.Kmax, B.K, B.act, c, cstride, x,
                                                                                   xstride, out, ostride, np, nb);
    else
        ::mof::count_launch(), k_combine<real, 1, false><<<dim3(nb, B.B), CT, 0, st>>>(B.V, B.N, B.Kmax, B.K, B.act, c, cstride, x,
                                                                                    xstride, out, ostride, np, nb);
    if (nrm2_out) ::mof::count_launch(), k_sum_scalar_chunks<<<B.B, 32, 0, st>>>(partial, nb, nrm2_out, B.B);
}

template <typename real>
void Krylov<real>::norm2(const real *x, long long N, long long xstride, int nb, double *out, cudaStream_t st,
                         bool exact) const {
    const int nc = (int)krylov_chunks(N);
    if (exact) ::mof::count_launch(), k_norm2<real, true><<<dim3(nc, nb), KT, 0, st>>>(x, N, xstride, partial, nc);
    else ::mof::count_launch(), k_norm2<real><<<dim3(nc, nb), KT, 0, st>>>(x, N, xstride, partial, nc);
    ::mof::count_launch(), k_sum_scalar_chunks<<<nb, 32, 0, st>>>(partial, nc, out, nb);
}

template <typename real>
bool Krylov<real>::sub_dot(const BasisRef<real> &B, const double *c, long long cstride, real *x, long long xstride,
                           double *out, cudaStream_t st, int kcap, int *nparts) const {
    const long long es = sizeof(real);
    const bool ok = B.Kmax <= 64 && (B.N * es) % 16 == 0 && (xstride * es) % 16 == 0 &&
                    (reinterpret_cast<uintptr_t>(B.V) % 16) == 0 && (reinterpret_cast<uintptr_t>(x) % 16) == 0;
    if (!ok) return false;
    static std::atomic<bool> configured{false};
    if (!configured.load()) {  // the largest tile this instantiation can need (65 chunks)
        if (cudaFuncSetAttribute(k_sub_dot<real>, cudaFuncAttributeMaxDynamicSharedMemorySize, 65 * SD_BYTES) != cudaSuccess)
            return false;
        configured.store(true);
    }
    const int nc = (int)subdot_chunks(B.N, (int)es);
    const int kc = kcap > 0 ? std::min(kcap, B.Kmax) : B.Kmax;  // vectors the tile holds
    const size_t smem = (size_t)(kc + 1) * SD_BYTES;
    ::mof::count_launch(), k_sub_dot<real><<<dim3(nc, B.B), SDT, smem, st>>>(B.V, B.N, B.Kmax, B.K, B.act, c, cstride, x, xstride,
                                                                         x, xstride, partial, nc, err, kc,
                                                                         nparts ? partial + (long long)B.B * nc * B.Kmax : nullptr);
    DotOuts o{};
    o.o[0] = DotOut{out, B.Kmax, 1, 0, 0, 1.0};
    ::mof::count_launch(), k_sum_chunks<<<dim3((B.Kmax + SUMT / 32 - 1) / (SUMT / 32), B.B), SUMT, 0, st>>>(partial, nc, 1, B.Kmax,
                                                                                                          B.K, B.act, o);
    if (nparts) *nparts = nc;
    return true;
}

template <typename real>
void Krylov<real>::gk_half_step(const BasisRef<real> &B, int *Kmut, int front, const GkFront<real> &f, double *coef, double *nrm2_out,
                                const double *scale, double tol, int *grow, double *sq1, double *sq2, int *done, bool scaled,
                                cudaStream_t st) const {
    const long long L = front == 1 ? B.N / 2 : B.N;
    const int per = front == 1 ? dch<real>() / 2 : dch<real>(), nc = (int)((L + per - 1) / per);
    auto al = [](const void *q) { return reinterpret_cast<uintptr_t>(q) % 16 == 0; };
    const bool vec = vec_ok<real>(B.V, L, (long long)B.Kmax * B.N) && al(f.a) && al(f.s) && al(f.ux) && al(f.uy) && al(f.prev) &&
                     al(f.x) && f.astride % 4 == 0 && f.pstride % 4 == 0 && f.xstride % 4 == 0 && f.fstride % 4 == 0;
    // x: where the front leaves it (FRONT 0 without prev leaves it where it is)
    const real *x = front == 0 && !f.prev ? f.a : f.x;
    const long long xs = front == 0 && !f.prev ? f.astride : f.xstride;
#define GK(F)                                                                                                                     \
    if (vec) k_gk_dots<real, F, sizeof(real) == 4><<<dim3(nc, B.B), KT, 0, st>>>(B.V, B.N, B.Kmax, B.K, B.act, f, partial, nc, coef, done); \
    else k_gk_dots<real, F, false><<<dim3(nc, B.B), KT, 0, st>>>(B.V, B.N, B.Kmax, B.K, B.act, f, partial, nc, coef, done);
    ::mof::count_launch();
    if (front == 0) {
        GK(0)
    } else if (front == 1) {
        GK(1)
    } else {
        GK(2)
    }
#undef GK
    const int nb = (int)((B.N + 4LL * CT - 1) / (4LL * CT));
    int *slot = reinterpret_cast<int *>(aux);
    real *inv = reinterpret_cast<real *>(aux + B.B);
    ::mof::count_launch();
    if (vec)
        k_gk_sub<real, sizeof(real) == 4><<<dim3(nb, B.B), CT, 0, st>>>(B.V, B.N, B.Kmax, Kmut, B.act, coef, x, xs, partial, nb, nrm2_out,
                                                                        scale, tol, grow, slot, inv, sq1, sq2, done);
    else
        k_gk_sub<real, false><<<dim3(nb, B.B), CT, 0, st>>>(B.V, B.N, B.Kmax, Kmut, B.act, coef, x, xs, partial, nb, nrm2_out, scale, tol,
                                                            grow, slot, inv, sq1, sq2, done);
    if (scaled) ::mof::count_launch(), k_gk_scale<real><<<dim3(nb, B.B), KT, 0, st>>>(B.V, B.N, B.Kmax, slot, inv);
}

template <typename real>
void Krylov<real>::reorth_second(const BasisRef<real> &B, real *x, long long xstride, const double *c1, double *coef,
                                 double *nrm2_out, cudaStream_t st) const {
    // the first projection's coefficients are given, the second are taken by dot products, fused
    // with the first update where the layout allows
    if (!sub_dot(B, c1, B.Kmax, x, xstride, coef, st)) {
        subtract(B, c1, B.Kmax, x, xstride, x, xstride, nullptr, st);
        dots(B, x, xstride, coef, B.Kmax, 1.0, st);
    }
    subtract(B, coef, B.Kmax, x, xstride, x, xstride, nrm2_out, st);
}

template <typename real>
void Krylov<real>::append_parts(const BasisRef<real> &B, int *Kmut, const real *x, long long xstride, int nparts,
                                double *nrm2_out, const double *scale, double tol, int *grow, int *appended, real *stage,
                                double *sq1, double *sq2, cudaStream_t st, const double *parts) const {
    int *slot = reinterpret_cast<int *>(aux);
    real *inv = reinterpret_cast<real *>(aux + B.B);
    ::mof::count_launch(), k_append_prep_sum<real><<<(B.B + 1) / 2, 64, 0, st>>>(Kmut, B.Kmax, parts ? parts : partial, nparts,
                                                                                nrm2_out, scale, tol, grow, B.B, slot, inv,
                                                                                appended, sq1, sq2);
    const int blocks = (int)std::min<long long>(1024, (B.N + KT - 1) / KT);
    ::mof::count_launch(), k_append<real><<<dim3(blocks, B.B), KT, 0, st>>>(B.V, B.N, B.Kmax, slot, inv, x, xstride, stage);
}

template <typename real>
void Krylov<real>::append(const BasisRef<real> &B, int *Kmut, const real *x, long long xstride, const double *nrm2,
                          const double *scale, double tol, int *grow, int *appended, real *stage, cudaStream_t st) const {
    int *slot = reinterpret_cast<int *>(aux);
    real *inv = reinterpret_cast<real *>(aux + B.B);
    ::mof::count_launch(), k_append_prep<real><<<(B.B + 63) / 64, 64, 0, st>>>(Kmut, B.Kmax, nrm2, scale, tol, grow, B.B, slot, inv,
                                                                              appended);
    const int blocks = (int)std::min<long long>(1024, (B.N + KT - 1) / KT);
    ::mof::count_launch(), k_append<real><<<dim3(blocks, B.B), KT, 0, st>>>(B.V, B.N, B.Kmax, slot, inv, x, xstride, stage);
}

// The totals of k_of_proj_gram_pass (one per warp and output) summed in FP64 (one warp per output, lanes over its
// contiguous chunks, fixed order): res[b][0..3 Kmax + 4). The last CTA of a pair to finish
// (counter done[b], left at zero) takes the append decision on ||x'|| (as k_append_prep) and
// writes, for an appended vector v = x' / ||x'||, its Gram columns G_A, G_L, g, its Euclidean
// overlaps Mg, and its slot and scale for k_of_combine (see k_of_proj_gram_pass for the formulas).
constexpr int PF_T = 256;
template <typename real>
__global__ void __launch_bounds__(PF_T) k_of_pass_finish(const double *__restrict__ partial, int nchunk, double *res,
                                                         const double *__restrict__ d, int Kmax, int *__restrict__ K,
                                                         const int *__restrict__ act, const double *__restrict__ scale, double tol,
                                                         int *__restrict__ grow, double *GA, double *GL, double *g, double *Mg,
                                                         double *__restrict__ nrm2_out, int *__restrict__ appended,
                                                         int *__restrict__ slot, real *__restrict__ inv, int *done) {
    __shared__ double s_gd[64], s_sum[2];
    __shared__ int s_last;
    const int b = blockIdx.y, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (act && !act[b]) {
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            slot[b] = -1;
            if (appended) appended[b] = 0;
        }
        return;
    }
    const int stride = 3 * Kmax + 4, Kb = min(K[b], Kmax);
    double *rs = res + (long long)b * stride;
    const int o = blockIdx.x * (PF_T / 32) + w;
    if (o < stride && (o >= 3 * Kmax || o % Kmax < Kb)) {
        const double *src = partial + ((long long)b * stride + o) * nchunk;
        double sum = 0.0;
#pragma unroll 8
        for (int c = lane; c < nchunk; c += 32) sum += src[c];
        sum = warp_sum(sum);
        if (lane == 0) rs[o] = sum;
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        s_last = atomicAdd(done + b, 1) == (int)gridDim.x - 1;
        if (s_last) done[b] = 0;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    const volatile double *c2 = rs, *ay = rs + Kmax, *aq = rs + 2 * Kmax, *sc = rs + 3 * Kmax;
    const double *db = d + (long long)b * Kmax;
    const long long KK = (long long)Kmax * Kmax;
    double *A = GA + b * KK, *L = GL + b * KK, *M = Mg + b * KK;
    const double nr2 = sc[0];
    const bool ok = append_ok(grow[b], Kb, Kmax, nr2, scale, b, tol);
    // (G_L d)_i (one warp per row), then d^T (V^T q) and d^T G_L d for the new column of G_L
    for (int i = w; i < Kb; i += PF_T / 32) {
        double gd = 0.0;
        for (int k = lane; k < Kb; k += 32) gd += L[(long long)i * Kmax + k] * db[k];
        gd = warp_sum(gd);
        if (lane == 0) s_gd[i] = gd;
    }
    __syncthreads();
    if (w < 2) {
        double t = 0.0;
        for (int i = lane; i < Kb; i += 32) t += db[i] * (w == 0 ? aq[i] : s_gd[i]);
        t = warp_sum(t);
        if (lane == 0) s_sum[w] = t;
    }
    __syncthreads();
    const double ib = 1.0 / sqrt(nr2), ib2 = 1.0 / nr2;
    if (ok) {
        for (int i = threadIdx.x; i < Kb; i += PF_T) {
            const double va = ay[i] * ib, vl = (aq[i] - s_gd[i]) * ib, vm = c2[i] * ib;
            A[(long long)i * Kmax + Kb] = va;
            A[(long long)Kb * Kmax + i] = va;
            L[(long long)i * Kmax + Kb] = vl;
            L[(long long)Kb * Kmax + i] = vl;
            M[(long long)i * Kmax + Kb] = vm;
            M[(long long)Kb * Kmax + i] = vm;
        }
        if (threadIdx.x == 0) {
            A[(long long)Kb * Kmax + Kb] = sc[1] * ib2;
            L[(long long)Kb * Kmax + Kb] = (sc[2] - s_sum[0] + s_sum[1]) * ib2;
            M[(long long)Kb * Kmax + Kb] = 1.0;
            g[(long long)b * Kmax + Kb] = sc[3] * ib;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        nrm2_out[b] = nr2;
        slot[b] = ok ? Kb : -1;
        inv[b] = ok ? (real)ib : (real)0;
        if (ok) K[b] = Kb + 1;
        else grow[b] = 0;
        if (appended) appended[b] = ok;
    }
}

// s[b] = sum_j V[b][j] z[b][j] for Solve-OF, with the scale of a vector appended by
// k_of_pass_finish: slot[b] (-1: none) holds x' still, which becomes x' inv[b] here on its way
// through (one pass over the vector less than a separate append). 16 bytes per thread; VEC: s on a
// 16-byte boundary, else (a caller's own array in the plain form and in timed calls) it is stored value
// by value.
template <typename real, bool VEC>
__global__ void __launch_bounds__(CT) k_of_combine(real *__restrict__ V, long long N, int Kmax, const int *__restrict__ K,
                                                   const double *__restrict__ z, const int *__restrict__ slot,
                                                   const real *__restrict__ inv, real *__restrict__ out) {
    using vec_t = typename std::conditional<sizeof(real) == 4, float4, double2>::type;
    constexpr int EPT = 16 / sizeof(real);
    __shared__ real sc[64];
    const int b = blockIdx.y, Kb = min(K[b], Kmax), sl = slot[b];
    for (int j = threadIdx.x; j < Kb; j += CT) sc[j] = (real)z[(long long)b * Kmax + j];
    __syncthreads();
    const long long i = ((long long)blockIdx.x * CT + threadIdx.x) * EPT;
    if (i >= N) return;
    real *Vb = V + (long long)b * Kmax * N + i;
    __align__(16) real acc[EPT];
#pragma unroll
    for (int e = 0; e < EPT; ++e) acc[e] = 0;
    const int Kd = sl >= 0 ? Kb - 1 : Kb;  // a new vector is the last one
    int j = 0;
    for (; j + 3 < Kd; j += 4) {
        vec_t q[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) q[c] = __ldcs(reinterpret_cast<const vec_t *>(Vb + (long long)(j + c) * N));
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int e = 0; e < EPT; ++e) acc[e] += reinterpret_cast<const real *>(&q[c])[e] * sc[j + c];
    }
    for (; j < Kd; ++j) {
        const vec_t q = __ldcs(reinterpret_cast<const vec_t *>(Vb + (long long)j * N));
#pragma unroll
        for (int e = 0; e < EPT; ++e) acc[e] += reinterpret_cast<const real *>(&q)[e] * sc[j];
    }
    if (sl >= 0) {
        const real iv = inv[b];
        vec_t q = *reinterpret_cast<const vec_t *>(Vb + (long long)Kd * N);
#pragma unroll
        for (int e = 0; e < EPT; ++e) {
            real &v = reinterpret_cast<real *>(&q)[e];
            v *= iv;
            acc[e] += v * sc[Kd];
        }
        *reinterpret_cast<vec_t *>(Vb + (long long)Kd * N) = q;
    }
    real *o = out + (long long)b * N + i;
    if (VEC) {
        *reinterpret_cast<vec_t *>(o) = *reinterpret_cast<vec_t *>(acc);
    } else {
#pragma unroll
        for (int e = 0; e < EPT; ++e) o[e] = acc[e];
    }
}

template <typename real>
mof_status launch_of_combine(const BasisRef<real> &B, const double *z, double *aux, real *out, cudaStream_t st) {
    const int *slot = reinterpret_cast<const int *>(aux);
    const real *inv = reinterpret_cast<const real *>(aux + B.B);
    const long long per = CT * (16 / (int)sizeof(real));
    const dim3 grid((unsigned)((B.N + per - 1) / per), B.B);
    ::mof::count_launch();
    if (reinterpret_cast<uintptr_t>(out) % 16 == 0) k_of_combine<real, true><<<grid, CT, 0, st>>>(B.V, B.N, B.Kmax, B.K, z, slot, inv, out);
    else k_of_combine<real, false><<<grid, CT, 0, st>>>(B.V, B.N, B.Kmax, B.K, z, slot, inv, out);
    MOF_LAUNCH_CHECK();
    return MOF_OK;
}

// r = Ups^T Ups s - Ups^T b + gamma (L(+)L)^T (L(+)L) s (the normal-equation residual of Alg. 2)
// and q = L^T L r on both components (graph Laplacians with free boundary) in one pass, on 32 x 8
// tiles with the borders of s and r in shared memory, one thread per pixel. FP64: bound by the FP64
// pipe (1024^2 x 7 pairs 640 us; the marching form below 633, 256^2 x 31 184 against 254 us).
template <typename real>
__device__ __forceinline__ real lap5(real c, bool l, real fl, bool r, real fr, bool u, real fu, bool d, real fd) {
    real v = 0;
    if (l) v += c - fl;
    if (r) v += c - fr;
    if (u) v += c - fu;
    if (d) v += c - fd;
    return v;
}
template <typename real>
__global__ void __launch_bounds__(256) k_of_resid_lap_tile(const real *__restrict__ ux, const real *__restrict__ uy,
                                                           const real *__restrict__ AtB, const real *__restrict__ s,
                                                           const double *__restrict__ gam, real *__restrict__ r, real *__restrict__ q,
                                                           int nx, int ny, const int *__restrict__ act) {
    constexpr int W = 32, H = 8;
    __shared__ real S[2][H + 4][W + 4], R[2][H + 2][W + 2];
    __shared__ real s_g;
    const int b = blockIdx.z;
    if (!act[b]) return;
    const int x0 = blockIdx.x * W, y0 = blockIdx.y * H, tid = threadIdx.y * W + threadIdx.x;
    const long long ns = (long long)nx * ny;
    const real *sb = s + b * 2 * ns;
    if (tid == 0) s_g = (real)gam[b];
    for (int e = tid; e < 2 * (H + 4) * (W + 4); e += 256) {
        const int c = e / ((H + 4) * (W + 4)), m = e - c * (H + 4) * (W + 4), ly = m / (W + 4), lx = m - ly * (W + 4);
        const int x = x0 + lx - 2, y = y0 + ly - 2;
        S[c][ly][lx] = (x >= 0 && x < nx && y >= 0 && y < ny) ? sb[c * ns + y * nx + x] : (real)0;
    }
    __syncthreads();
    const real g = s_g;
    for (int e = tid; e < (H + 2) * (W + 2); e += 256) {
        const int ly = e / (W + 2), lx = e - ly * (W + 2), x = x0 + lx - 1, y = y0 + ly - 1;
        if (x < 0 || x >= nx || y < 0 || y >= ny) continue;
        const int i = y * nx + x;
        const real ax = ux[b * ns + i], ay = uy[b * ns + i];
        const real v0 = S[0][ly + 1][lx + 1], v1 = S[1][ly + 1][lx + 1], a = ax * v0 + ay * v1;
        const bool l = x > 0, rr = x < nx - 1, u = y > 0, d = y < ny - 1;
        const real q0 = lap5(v0, l, S[0][ly + 1][lx], rr, S[0][ly + 1][lx + 2], u, S[0][ly][lx + 1], d, S[0][ly + 2][lx + 1]);
        const real q1 = lap5(v1, l, S[1][ly + 1][lx], rr, S[1][ly + 1][lx + 2], u, S[1][ly][lx + 1], d, S[1][ly + 2][lx + 1]);
        R[0][ly][lx] = ax * a - AtB[b * 2 * ns + i] + g * q0;
        R[1][ly][lx] = ay * a - AtB[b * 2 * ns + ns + i] + g * q1;
    }
    __syncthreads();
    const int x = x0 + threadIdx.x, y = y0 + threadIdx.y, lx = threadIdx.x + 1, ly = threadIdx.y + 1;
    if (x >= nx || y >= ny) return;
    const long long i = b * 2 * ns + y * nx + x;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        const real v = R[c][ly][lx];
        r[i + c * ns] = v;
        q[i + c * ns] = lap5(v, x > 0, R[c][ly][lx - 1], x < nx - 1, R[c][ly][lx + 1], y > 0, R[c][ly - 1][lx], y < ny - 1, R[c][ly + 1][lx]);
    }
}

// The same for FP32 rows of a multiple of 4 pixels. A lane takes V = 4 columns and marches down
// `rows` rows with three rows of s and of r in registers; the neighbours come from the adjacent lanes,
// so the first and last lane of a warp only serve the others (except at the image's edge). The next
// row is loaded before the present one is used. Bound by HBM: six values read and four written per
// pixel. 63 pairs of 1024^2: 0.45 ms (0.86 of the copy rate) against 1.15 for the tiles; 31 pairs of
// 256^2: 22 against 37 us.
constexpr int RL_W = 4;  // warps per CTA
template <typename real>
__global__ void __launch_bounds__(32 * RL_W) k_of_resid_lap(const real *__restrict__ ux, const real *__restrict__ uy,
                                                            const real *__restrict__ AtB, const real *__restrict__ s,
                                                            const double *__restrict__ gam, real *__restrict__ r,
                                                            real *__restrict__ q, int nx, int ny, int rows,
                                                            const int *__restrict__ act) {
    constexpr int V = 16 / (int)sizeof(real), HL = 1, OUT = 32 - 2 * HL;  // HL: serving lanes on each side
    const int b = blockIdx.z, lane = threadIdx.x, y0 = (blockIdx.y * RL_W + threadIdx.y) * rows;
    if (y0 >= ny || !act[b]) return;  // whole warps
    const int C = nx / V, c = blockIdx.x * OUT + lane;
    const bool out = c < C && (lane >= HL || blockIdx.x == 0) && (lane < 32 - HL || blockIdx.x == gridDim.x - 1);
    const int x = min(c, C - 1) * V, ye = min(y0 + rows, ny);
    const long long ns = (long long)nx * ny;
    ux += b * ns + x;
    uy += b * ns + x;
    AtB += b * 2 * ns + x;
    s += b * 2 * ns + x;
    r += b * 2 * ns + x;
    q += b * 2 * ns + x;
    const real g = (real)gam[b];
    struct __align__(V * sizeof(real)) Vec {
        real v[V];
    };
    auto row = [&](const real *f, int y) { return *reinterpret_cast<const Vec *>(f + (long long)min(max(y, 0), ny - 1) * nx); };
    Vec sm[2], sc[2], sp[2], rm[2], rc[2], f[4];
    auto fetch = [&](int y, Vec (&sn)[2], Vec (&fn)[4]) {  // s of row y + 1, the fields of row y
        sn[0] = row(s, y + 1);
        sn[1] = row(s + ns, y + 1);
        fn[0] = row(ux, y);
        fn[1] = row(uy, y);
        fn[2] = row(AtB, y);
        fn[3] = row(AtB + ns, y);
    };
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        sm[k] = row(s + k * ns, y0 - 2);
        sc[k] = row(s + k * ns, y0 - 1);
#pragma unroll
        for (int e = 0; e < V; ++e) rm[k].v[e] = rc[k].v[e] = 0;
    }
    fetch(y0 - 1, sp, f);
    // a row's five-point sums; m, n: the rows above and below
    auto lap = [&](const Vec &m, const Vec &w, const Vec &n, int y, Vec &o) {
        const real lf = __shfl_up_sync(0xffffffffu, w.v[V - 1], 1), rt = __shfl_down_sync(0xffffffffu, w.v[0], 1);
#pragma unroll
        for (int e = 0; e < V; ++e)
            o.v[e] = lap5(w.v[e], x + e > 0, e ? w.v[e ? e - 1 : 0] : lf, x + e < nx - 1, e < V - 1 ? w.v[e < V - 1 ? e + 1 : e] : rt, y > 0,
                          m.v[e], y < ny - 1, n.v[e]);
    };
    for (int y = y0 - 1; y <= ye; ++y) {
        Vec sn[2], fn[4], rp[2];
        if (y < ye) fetch(y + 1, sn, fn);
        Vec l0, l1;
        lap(sm[0], sc[0], sp[0], y, l0);
        lap(sm[1], sc[1], sp[1], y, l1);
#pragma unroll
        for (int e = 0; e < V; ++e) {
            const real ax = f[0].v[e], ay = f[1].v[e], a = ax * sc[0].v[e] + ay * sc[1].v[e];
            rp[0].v[e] = ax * a - f[2].v[e] + g * l0.v[e];
            rp[1].v[e] = ay * a - f[3].v[e] + g * l1.v[e];
        }
        if (out && y >= y0 && y < ye) {
            *reinterpret_cast<Vec *>(r + (long long)y * nx) = rp[0];
            *reinterpret_cast<Vec *>(r + ns + (long long)y * nx) = rp[1];
        }
        if (y > y0) {
            lap(rm[0], rc[0], rp[0], y - 1, l0);
            lap(rm[1], rc[1], rp[1], y - 1, l1);
            if (out) {
                *reinterpret_cast<Vec *>(q + (long long)(y - 1) * nx) = l0;
                *reinterpret_cast<Vec *>(q + ns + (long long)(y - 1) * nx) = l1;
            }
        }
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            rm[k] = rc[k];
            rc[k] = rp[k];
            sm[k] = sc[k];
            sc[k] = sp[k];
            sp[k] = sn[k];
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) f[k] = fn[k];
    }
}

template <typename real>
mof_status launch_of_resid_lap(int nb, int pairs, int nx, int ny, const real *ux, const real *uy, const real *AtB, const real *s,
                               const double *gam, real *r, real *q, const int *act, cudaStream_t st) {
    auto al = [](const void *p) { return reinterpret_cast<uintptr_t>(p) % 16 == 0; };
    const int gx = std::max(1, (nx / 4 - 2 + 29) / 30);
    ::mof::count_launch();
    // marching where strips of 4 rows give every SM four warps (256^2 x 7 pairs, 1344 strips: 10 against
    // 13 us; 128^2 x 7, 224 strips: 8.8 both)
    if (sizeof(real) == 4 && nx % 4 == 0 && al(ux) && al(uy) && al(AtB) && al(s) && al(r) && al(q) &&
        (long long)gx * pairs * ((ny + 3) / 4) >= 152LL * 4) {
        // strips of 16 rows (four rows of s and two of the rest are read twice) where they give every SM
        // 16 warps, else of 8 or 4
        int rows = 16;
        while (rows > 4 && (long long)gx * pairs * ((ny + rows - 1) / rows) < 152LL * 16) rows /= 2;
        k_of_resid_lap<float><<<dim3(gx, (ny + RL_W * rows - 1) / (RL_W * rows), nb), dim3(32, RL_W), 0, st>>>(
            (const float *)ux, (const float *)uy, (const float *)AtB, (const float *)s, gam, (float *)r, (float *)q, nx, ny, rows, act);
    } else {
        k_of_resid_lap_tile<real><<<dim3((nx + 31) / 32, (ny + 7) / 8, nb), dim3(32, 8), 0, st>>>(ux, uy, AtB, s, gam, r, q, nx, ny, act);
    }
    MOF_LAUNCH_CHECK();
    return MOF_OK;
}

template <typename real>
bool of_pass_applicable(long long ns, const void *V, const void *x) {
    const long long es = sizeof(real);
    return (ns * es) % 16 == 0 && (reinterpret_cast<uintptr_t>(V) % 16) == 0 && (reinterpret_cast<uintptr_t>(x) % 16) == 0;
}

template <typename real>
mof_status launch_of_proj_gram_pass(const BasisRef<real> &B, int *Kmut, long long ns, int pairs, const double *d, const real *x, const real *q,
                                    const real *AtB, const real *ux, const real *uy, double *partial, double *res, int *err,
                                    int kcap, const double *scale, double tol, int *grow, double *GA, double *GL, double *g,
                                    double *Mg, double *nrm2_out, int *appended, double *aux, int *done, cudaStream_t st) {
    static std::atomic<bool> configured{false};
    if (!configured.load()) {
        if (cudaFuncSetAttribute(k_of_proj_gram_pass<real>, cudaFuncAttributeMaxDynamicSharedMemorySize, 140 * 1024) !=
            cudaSuccess)
            return fail(MOF_ECUDA, "shared-memory attribute of the Solve-OF pass");
        configured.store(true);
    }
    const int nc = of_pass_parts_of(ns, pairs, (int)sizeof(real));
    const int kc = kcap > 0 ? std::min(kcap, B.Kmax) : B.Kmax;
    const size_t smem = (size_t)(kc + 4) * 1024;
    ::mof::count_launch(), k_of_proj_gram_pass<real><<<dim3(nc, B.B), 32, smem, st>>>(B.V, ns, B.Kmax, B.K, B.act, d, x, q, B.V, AtB,
                                                                                     ux, uy, partial, nc, err, kc);
    const int stride = of_pass_stride(B.Kmax);
    int *slot = reinterpret_cast<int *>(aux);
    real *inv = reinterpret_cast<real *>(aux + B.B);
    ::mof::count_launch(), k_of_pass_finish<real><<<dim3((stride + PF_T / 32 - 1) / (PF_T / 32), B.B), PF_T, 0, st>>>(
        partial, nc, res, d, B.Kmax, Kmut, B.act, scale, tol, grow, GA, GL, g, Mg, nrm2_out, appended, slot, inv, done);
    MOF_LAUNCH_CHECK();
    return MOF_OK;
}

template bool of_pass_applicable<float>(long long, const void *, const void *);
template bool of_pass_applicable<double>(long long, const void *, const void *);
#define MOF_INST_OF(real)                                                                                                      \
    template mof_status launch_of_proj_gram_pass<real>(const BasisRef<real> &, int *, long long, int, const double *, const real *, \
                                                       const real *, const real *, const real *, const real *, double *,      \
                                                       double *, int *, int, const double *, double, int *, double *,         \
                                                       double *, double *, double *, double *, int *, double *, int *,        \
                                                       cudaStream_t);                                                          \
    template mof_status launch_of_combine<real>(const BasisRef<real> &, const double *, double *, real *, cudaStream_t);       \
    template mof_status launch_of_resid_lap<real>(int, int, int, int, const real *, const real *, const real *, const real *,       \
                                                  const double *, real *, real *, const int *, cudaStream_t);
MOF_INST_OF(float)
MOF_INST_OF(double)

template struct Krylov<float>;
template struct Krylov<double>;

}  // namespace mof

// K11: the small projected problem of MMGKS / GKS, in FP64, one block per
// problem (Sec. 4.1.1 eq. (QR)-(minKryov2), Sec. 4.1.3 DP and GCV).
//
// Given the Gram matrices G_A = (A V)^T (A V), G_L = (L V)^T (L V) and
// g = (A V)^T b of the current basis (R_A^T R_A = G_A and R_L^T R_L = G_L for
// the R factors of eq. (QR)), the block
//   1. factors M = G_A + rho G_L = R^T R (Cholesky, FP64), rho = tr G_A / tr G_L,
//      and forms C = R^-T G_A R^-1 and h = R^-T g by two triangular solves;
//   2. diagonalises C: cyclic one-sided Jacobi sweeps in FP32 (four warps,
//      each holding a quarter of every column) give approximate
//      eigenvectors W; one third-order Newton-Schulz step makes them
//      orthonormal in FP64 (W <- W (I - E/2 + 3E^2/8), E = W^T W - I), and
//      cyclic Jacobi sweeps in FP64 on W^T C W, which start near diagonal,
//      finish the decomposition (usually in one sweep: the sweeps stop once no
//      off-diagonal entry exceeds 1e-12 max|c_ii|) while rotating the one vector
//      W^T h they need; with the eigenvalues theta_i in [0, 1] and the
//      eigenvectors, X = R^-1 W satisfies X^T G_A X = diag(theta),
//      X^T G_L X = diag(1 - theta)/rho (the generalized singular values of
//      (R_A, R_L));
//   3. with ghat = X^T g, chat_i^2 = ghat_i^2 / theta_i and the filter factors
//      f_i = theta_i / (theta_i + mu (1 - theta_i)), mu = lam / rho, has
//      ||R_A z - Q_A^T b||^2 = sum chat_i^2 (1 - f_i)^2 and
//      trace(I - S) = sum (1 - f_i), with closed-form derivatives in lam;
//   4. picks lam on the bracket 10^[log10 rho - 12, log10 rho + 12]:
//      GCV: the first minimum of a 200-point log grid (ties to the smaller
//      lam): an FP32 scan leaves the points that can be it, FP64 decides among
//      those; then refined between its two grid neighbours by
//      safeguarded Newton steps on dG/dlog10(lam) = 0 (FP32 steps, then FP64
//      steps, which stop after a Newton step below 1e-6 -- the next would be
//      below ~1e-12 -- or once the derivative is at its rounding level), kept
//      only if it improves on the grid value; where the five FP64 values agree
//      to 1e-13 the neighbourhood is flat to rounding (the plateau G takes
//      as lam -> 0 when every theta_i > 0) and the grid point stands;
//      DP: the root of ||A V z - b||^2 = (eta delta)^2 (monotone in lam); the
//      bracket ends decide the no-root flags in FP64, an FP32 grid locates the
//      sign change (its cell is confirmed in FP64), and safeguarded Newton
//      steps in log10 lam (FP32, then FP64) converge to the root;
//   5. returns z = R^-1 (C + mu (I - C))^-1 h, the solution of
//      (G_A + lam G_L) z = g, by an FP64 Cholesky solve in the R basis.
//
// GB300 executes FP64 at about 2 fused multiply-adds per clock per SM, and a
// warp's FP64 instruction costs the same with one lane active as with 32, so
// the block does its FP64 arithmetic with full warps wherever the work is
// parallel (triangular updates over all threads, symmetric products over the
// upper triangle), keeps the serial parts (pivots, rotation angles,
// substitutions, Newton steps) in one warp, and evaluates in FP32 what a
// later FP64 step corrects (the Jacobi warm start, the lambda grids).
//
// The solves of one Solve-OF (p = q = 2) differ by one basis vector each: from the second on steps 1
// and 2 are replaced by the update of the bordered eigenproblem below (rho that of the first), and z
// comes from X with one step of refinement. All blocks of a call run side by side, one per SM, so a
// call lasts as long as one block; 31 pairs at 256^2, basis 10 to 29, mean of 20 calls: 190 us when
// every call factored anew and scanned the grid in FP64, 80 us now (of about 61 + 42 + 34 thousand
// clocks for update, lambda and the rest at K = 20, the FP64 pipe is busy or waited for in all).
#include "solver.cuh"

#include <atomic>
#include <cfloat>
#include <cmath>

namespace mof {

namespace {

constexpr int ST = 256;
constexpr int NW = ST / 32;
constexpr int GRID_POINTS = 200;
constexpr int NEWTON_MAX = 60;
constexpr int NEWTON32_MAX = 30;
constexpr int NREF = 5;  // grid points around the minimum that decide whether it is flat
constexpr double BRACKET_DECADES = 12.0;
constexpr double THETA_TINY = 1e-14;
constexpr int JACOBI32_MAX_SWEEPS = 12;
constexpr int JACOBI64_MAX_SWEEPS = 10;
constexpr int JW = 4;  // warps of the FP32 one-sided Jacobi
constexpr int RW = 32 / JW;
constexpr double LN10 = 2.302585092994045684;

// ------------------------------------------------------------ index helpers
// The n(n+1)/2 pairs (r, c), r <= c < n, of an upper triangle enumerated as a
// ceil(n/2) x (n+1) rectangle whose row q holds triangle rows q and n-1-q.
__device__ __forceinline__ int tri_count(int n) { return ((n + 1) / 2) * (n + 1); }
__device__ __forceinline__ bool tri_pair(int e, int n, int &r, int &c) {
    const int q = e / (n + 1), x = e - q * (n + 1);
    if (x < n - q) {
        r = q;
        c = q + x;
        return true;
    }
    r = n - 1 - q;
    if (r == q) return false;  // middle row of an odd n: already enumerated
    c = r + (x - (n - q));
    return true;
}

// round-robin tournament: player at position j in round r (positions 0..Kp-1)
__device__ __forceinline__ int rr_player(int j, int r, int Kp) {
    int v = j - 1 + r;
    if (v >= Kp - 1) v -= Kp - 1;
    return j == 0 ? 0 : 1 + v;
}

// ------------------------------------------------------------ reductions
// Sums over the warp of two values, each returned to every lane; 5 FP64
// additions per lane instead of 10.
__device__ __forceinline__ void warp_sum2(double &a, double &b) {
    const bool hi = (threadIdx.x & 16) != 0;
    double y = (hi ? b : a) + __shfl_xor_sync(0xffffffffu, hi ? a : b, 16);
    for (int o = 8; o > 0; o >>= 1) y += __shfl_xor_sync(0xffffffffu, y, o);
    a = __shfl_sync(0xffffffffu, y, 0);
    b = __shfl_sync(0xffffffffu, y, 16);
}
// Sums over the warp of six values with 8 FP64 additions per lane instead of
// 30: each shuffle level halves the number of distinct partial sums a lane
// carries; the totals end in lanes 0, 16, 8, 24, 4, 20 and are broadcast.
__device__ __forceinline__ void warp_sum6(double s[6]) {
    const int lane = threadIdx.x & 31;
    const bool h = (lane & 16) != 0, g = (lane & 8) != 0, f = (lane & 4) != 0;
    const double r0 = __shfl_xor_sync(0xffffffffu, h ? s[0] : s[1], 16);
    const double r1 = __shfl_xor_sync(0xffffffffu, h ? s[2] : s[3], 16);
    const double r2 = __shfl_xor_sync(0xffffffffu, h ? s[4] : s[5], 16);
    const double a = (h ? s[1] : s[0]) + r0, b = (h ? s[3] : s[2]) + r1;
    double c = (h ? s[5] : s[4]) + r2;
    const double x = (g ? b : a) + __shfl_xor_sync(0xffffffffu, g ? a : b, 8);
    c += __shfl_xor_sync(0xffffffffu, c, 8);
    double y = (f ? c : x) + __shfl_xor_sync(0xffffffffu, f ? x : c, 4);
    y += __shfl_xor_sync(0xffffffffu, y, 2);
    y += __shfl_xor_sync(0xffffffffu, y, 1);
    s[0] = __shfl_sync(0xffffffffu, y, 0);
    s[1] = __shfl_sync(0xffffffffu, y, 16);
    s[2] = __shfl_sync(0xffffffffu, y, 8);
    s[3] = __shfl_sync(0xffffffffu, y, 24);
    s[4] = __shfl_sync(0xffffffffu, y, 4);
    s[5] = __shfl_sync(0xffffffffu, y, 20);
}

// 1 / x from the FP32 reciprocal by two Newton steps, |x| within the normal FP32 range
__device__ __forceinline__ double rcp_newton(double x) {
    double r = (double)__frcp_rn((float)x);
    r = fma(r, fma(-x, r, 1.0), r);
    return fma(r, fma(-x, r, 1.0), r);
}
// Sums over k < m of f(i, k) (and of f2) for the rows i < n <= 64: the rows over the lanes, k over
// the CTA's warps, the warps' partial sums in part (2 ST doubles). A reduction over lanes would
// take five dependent FP64 additions per row, the costly part on a pipe that a warp holds for
// 64 cycles per instruction. out(i, sum, sum2) is called by one thread per row. All threads
// call; ends with a barrier.
template <typename F, typename O>
__device__ __forceinline__ void row_sums2(int n, int m, double *part, F &&f, O &&out) {
    const int tid = threadIdx.x, RS = n <= 32 ? 32 : 64, parts = ST / RS, i = tid & (RS - 1);
    double x = 0.0, y = 0.0;
    if (i < n)
        for (int k = tid / RS; k < m; k += parts) f(i, k, x, y);
    part[tid] = x;
    part[ST + tid] = y;
    __syncthreads();
    if (tid < n) {
        for (int q = 1; q < parts; ++q) {
            x += part[q * RS + tid];
            y += part[ST + q * RS + tid];
        }
        out(tid, x, y);
    }
    __syncthreads();
}
template <typename F, typename O>
__device__ __forceinline__ void row_sums(int n, int m, double *part, F &&f, O &&out) {
    const int tid = threadIdx.x, RS = n <= 32 ? 32 : 64, parts = ST / RS, i = tid & (RS - 1);
    double x = 0.0;
    if (i < n)
        for (int k = tid / RS; k < m; k += parts) x += f(i, k);
    part[tid] = x;
    __syncthreads();
    if (tid < n) {
        for (int q = 1; q < parts; ++q) x += part[q * RS + tid];
        out(tid, x);
    }
    __syncthreads();
}

// ------------------------------------------------------------ dense kernels
// Upper Cholesky in place: on return row j of A holds R[j][j..K) with
// A = R^T R (only the upper triangle of A is referenced) and
// invd[j] = 1 / R[j][j]. One barrier per column: warp 0 factors the pivot
// row, which it brought up to date itself in the previous column, while the
// other warps finish the previous column's trailing update. A non-positive or
// non-finite pivot sets *fail. All threads call; ends with a barrier.
__device__ void chol_upper(double *A, int lds, int K, double *invd, int *fail) {
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    for (int j = 0; j < K; ++j) {
        if (wid == 0) {
            const double d = A[j * lds + j];
            const bool ok = d > 0.0 && isfinite(d);
            const double rs = ok ? rsqrt(d) : 1.0;
            for (int k = j + lane; k < K; k += 32) A[j * lds + k] = (k == j) ? d * rs : A[j * lds + k] * rs;
            if (lane == 0) {
                invd[j] = rs;
                if (!ok) *fail = 1;
            }
        }
        __syncthreads();
        if (wid == 0) {
            const int k = j + 1;
            if (k < K) {
                const double ajk = A[j * lds + k];
                for (int l = k + lane; l < K; l += 32) A[k * lds + l] -= ajk * A[j * lds + l];
            }
            __syncwarp();
        } else {
            const int n = K - j - 2;  // rows j+2 .. K-1
            if (n > 0) {
                const int cnt = tri_count(n);
                for (int e = tid - 32; e < cnt; e += ST - 32) {
                    int r, c;
                    if (!tri_pair(e, n, r, c)) continue;
                    const int k = j + 2 + r, l = j + 2 + c;
                    A[k * lds + l] -= A[j * lds + k] * A[j * lds + l];
                }
            }
        }
    }
    __syncthreads();
}

// Y <- R^-T Y for the K x nc block Y (row stride ldy): forward substitution
// in column-oriented form with the division by R[i][i] deferred to the end,
// so the update by row i needs U[i][k] = R[i][k] / R[i][i] (k > i) only. One
// barrier per row; all threads call; ends with a barrier.
__device__ void trsm_rt(const double *U, int ldu, const double *invd, double *Y, int ldy, int K, int nc) {
    const int tid = threadIdx.x;
    for (int i = 0; i + 1 < K; ++i) {
        const int cnt = (K - 1 - i) * nc;
        for (int e = tid; e < cnt; e += ST) {
            const int k = i + 1 + e / nc, j = e - (e / nc) * nc;
            Y[k * ldy + j] -= U[i * ldu + k] * Y[i * ldy + j];
        }
        __syncthreads();
    }
    for (int e = tid; e < K * nc; e += ST) {
        const int i = e / nc, j = e - (e / nc) * nc;
        Y[i * ldy + j] *= invd[i];
    }
    __syncthreads();
}

// Y <- Y R^-1 for the nr x K block Y: column-oriented solve of Z R = Y with
// deferred scaling. One barrier per column; all threads call.
__device__ void trsm_r(const double *U, int ldu, const double *invd, double *Y, int ldy, int nr, int K) {
    const int tid = threadIdx.x;
    for (int j = 0; j + 1 < K; ++j) {
        const int w = K - 1 - j, cnt = nr * w;
        for (int e = tid; e < cnt; e += ST) {
            const int r = e / w, l = j + 1 + (e - (e / w) * w);
            Y[r * ldy + l] -= Y[r * ldy + j] * U[j * ldu + l];
        }
        __syncthreads();
    }
    for (int e = tid; e < nr * K; e += ST) {
        const int r = e / K, j = e - (e / K) * K;
        Y[r * ldy + j] *= invd[j];
    }
    __syncthreads();
}

// O = op(A) op(B) for K x K operands (op = transpose when the flag is set).
// With sym, only the upper triangle is computed and mirrored. Ends with a barrier.
__device__ void gemm_kk(double *O, const double *A, bool tA, const double *B, bool tB, int K, int lds, bool sym) {
    const int tid = threadIdx.x;
    const int cnt = sym ? tri_count(K) : K * K;
    for (int e = tid; e < cnt; e += ST) {
        int i, j;
        if (sym) {
            if (!tri_pair(e, K, i, j)) continue;
        } else {
            i = e / K;
            j = e - i * K;
        }
        double s = 0.0;
        for (int k = 0; k < K; ++k) s += (tA ? A[k * lds + i] : A[i * lds + k]) * (tB ? B[j * lds + k] : B[k * lds + j]);
        O[i * lds + j] = s;
        if (sym) O[j * lds + i] = s;
    }
    __syncthreads();
}

// Triangular solve in one warp, column-oriented; lane k holds entries k and
// k + 32 of the right-hand side (K <= 64). R is upper, given by its rows, and
// invd = 1 / diag(R). forward = true solves R^T x = x, else R x = x.
__device__ void warp_trsv(const double *R, int lds, const double *invd, double &x0, double &x1, int K, bool forward) {
    const int lane = threadIdx.x & 31;
    for (int s = 0; s < K; ++s) {
        const int i = forward ? s : K - 1 - s;
        const double own = (i >> 5) ? x1 : x0;
        const double xi = __shfl_sync(0xffffffffu, own, i & 31) * invd[i];
        if (lane == (i & 31)) {
            if (i >> 5) x1 = xi;
            else x0 = xi;
        }
        if (forward) {  // x_k -= R[i][k] x_i for k > i
            if (lane > i && lane < K) x0 -= R[i * lds + lane] * xi;
            if (lane + 32 > i && lane + 32 < K) x1 -= R[i * lds + lane + 32] * xi;
        } else {  // x_k -= R[k][i] x_i for k < i
            if (lane < i) x0 -= R[lane * lds + i] * xi;
            if (lane + 32 < i) x1 -= R[(lane + 32) * lds + i] * xi;
        }
    }
}

// ------------------------------------------------------------ Jacobi
// Rotation (c, s) that zeroes a_pq of [[a_pp, a_pq], [a_pq, a_qq]]: tan(phi)
// by the classical formula in FP32, from the FP64 difference a_qq - a_pp.
// For the FP64 sweeps the FP32 pair is renormalised in FP64 with the series
// 1/sqrt(1 + d) = 1 - d/2 + 3d^2/8 (|d| < 1e-6), so the rotation is orthogonal
// to FP64 accuracy; an angle accurate to FP32 still shrinks a_pq by ~1e-7 per
// visit, which is what the FP64 sweeps (started near diagonal) need.
__device__ __forceinline__ void rot_from(float th, float &c0, float &s0) {
    const float t = (th >= 0.0f ? 1.0f : -1.0f) / (fabsf(th) + sqrtf(fmaf(th, th, 1.0f)));
    c0 = rsqrtf(fmaf(t, t, 1.0f));
    s0 = t * c0;
}
__device__ __forceinline__ void rot_angle(float app, float aqq, float apq, float &c, float &s) {
    rot_from((aqq - app) / (2.0f * apq), c, s);
}
__device__ __forceinline__ void rot_angle(double app, double aqq, double apq, double &c, double &s) {
    float c0, s0;
    rot_from((float)(aqq - app) / (2.0f * (float)apq), c0, s0);
    const double cd = c0, sd = s0;
    const double dl = fma(cd, cd, sd * sd) - 1.0;
    const double r = fma(dl, fma(0.375, dl, -0.5), 1.0);
    c = cd * r;
    s = sd * r;
}

template <typename T>
struct JacobiShared {
    T c[2][32], s[2][32];
    int any[2];
};

// Cyclic two-sided Jacobi on the symmetric Kp x Kp matrix A (rows/columns
// beyond K are zero padding) with eigenvector accumulation W <- W J (W may be
// null) and the rotations applied to one vector v <- J^T v (v may be null).
// Each round of the round-robin ordering rotates Kp/2 disjoint pairs: warp 0
// decides and computes the rotations and rotates v, then all threads update
// the 2x2 blocks (pair i rows, pair j columns) of the upper block triangle
// from their old values and mirror them, and the rows of W. A pair rotates
// while |a_pq| > rel sqrt(|a_pp a_qq|) and |a_pq| > rel_abs max_i |a_ii|; the
// sweeps stop when a parallel scan after a sweep finds no such pair, or after
// max_sweeps. The rotation buffers alternate between rounds, so a round costs
// one barrier when it rotates nothing and two otherwise. All threads call.
template <typename T>
__device__ void jacobi(T *A, int lda, T *W, int ldw, T *v, int K, int Kp, int max_sweeps, float rel, float rel_abs,
                       JacobiShared<T> &sh, float *redf) {
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int half = Kp / 2;
    float dm = 0.0f;
    for (int i = tid; i < K; i += ST) dm = fmaxf(dm, fabsf((float)A[i * lda + i]));
    dm = warp_maxf(dm);
    if (lane == 0) redf[wid] = dm;
    __syncthreads();
    dm = 0.0f;
    for (int w = 0; w < NW; ++w) dm = fmaxf(dm, redf[w]);
    const float floor_abs = rel_abs * dm;
    int buf = 0;
    const int nblk = tri_count(half);
    for (int sweep = 0; sweep < max_sweeps; ++sweep) {
        for (int round = 0; round < Kp - 1; ++round, buf ^= 1) {
            if (wid == 0) {
                T c = 1, s = 0;
                bool rot = false;
                if (lane < half) {
                    const int pl = rr_player(lane, round, Kp), ql = rr_player(Kp - 1 - lane, round, Kp);
                    if (pl < K && ql < K) {
                        const T apq = A[pl * lda + ql], app = A[pl * lda + pl], aqq = A[ql * lda + ql];
                        const float fpq = fabsf((float)apq);
                        rot = fpq > rel * sqrtf(fabsf((float)app * (float)aqq)) && fpq > floor_abs && fpq > 1e-35f;
                        if (rot) rot_angle(app, aqq, apq, c, s);
                        if (rot && v) {
                            const T vp = v[pl], vq = v[ql];
                            v[pl] = c * vp - s * vq;
                            v[ql] = s * vp + c * vq;
                        }
                    }
                    sh.c[buf][lane] = c;
                    sh.s[buf][lane] = rot ? s : (T)0;
                }
                const int any = __any_sync(0xffffffffu, rot);
                if (lane == 0) sh.any[buf] = any;
            }
            __syncthreads();
            if (!sh.any[buf]) continue;
            for (int e = tid; e < nblk; e += ST) {
                int bi, bj;
                if (!tri_pair(e, half, bi, bj)) continue;
                const T ci = sh.c[buf][bi], si = sh.s[buf][bi], cj = sh.c[buf][bj], sj = sh.s[buf][bj];
                if (si == (T)0 && sj == (T)0) continue;
                const int pi = rr_player(bi, round, Kp), qi = rr_player(Kp - 1 - bi, round, Kp);
                const int pj = rr_player(bj, round, Kp), qj = rr_player(Kp - 1 - bj, round, Kp);
                const T a = A[pi * lda + pj], b = A[pi * lda + qj], cc = A[qi * lda + pj], d = A[qi * lda + qj];
                const T a1 = ci * a - si * cc, b1 = ci * b - si * d, c1 = si * a + ci * cc, d1 = si * b + ci * d;
                const T na = cj * a1 - sj * b1, nb = sj * a1 + cj * b1, nd = sj * c1 + cj * d1;
                const T nc = (bi == bj) ? nb : cj * c1 - sj * d1;  // exact symmetry of a diagonal block
                A[pi * lda + pj] = na;
                A[pi * lda + qj] = nb;
                A[qi * lda + pj] = nc;
                A[qi * lda + qj] = nd;
                if (bi != bj) {
                    A[pj * lda + pi] = na;
                    A[qj * lda + pi] = nb;
                    A[pj * lda + qi] = nc;
                    A[qj * lda + qi] = nd;
                }
            }
            if (W) {
                for (int e = tid; e < Kp * half; e += ST) {  // W <- W J on the columns of each pair
                    const int r = e / half, j = e - (e / half) * half;
                    const T s = sh.s[buf][j];
                    if (s == (T)0) continue;
                    const T c = sh.c[buf][j];
                    const int pl = rr_player(j, round, Kp), ql = rr_player(Kp - 1 - j, round, Kp);
                    const T wp = W[r * ldw + pl], wq = W[r * ldw + ql];
                    W[r * ldw + pl] = c * wp - s * wq;
                    W[r * ldw + ql] = s * wp + c * wq;
                }
            }
            __syncthreads();
        }
        // does any pair still exceed the rotation threshold?
        int more = 0;
        for (int e = tid; e < K * K; e += ST) {
            const int p = e / K, q = e - (e / K) * K;
            if (q <= p) continue;
            const float fpq = fabsf((float)A[p * lda + q]);
            if (fpq > rel * sqrtf(fabsf((float)A[p * lda + p] * (float)A[q * lda + q])) && fpq > floor_abs &&
                fpq > 1e-35f)
                more = 1;
        }
        if (!__syncthreads_or(more)) break;
    }
}

__device__ __forceinline__ void jw_bar() { asm volatile("bar.sync 1, %0;" ::"r"(JW * 32) : "memory"); }

// The partner of column l in round r of the round-robin ordering of Kp
// (even, <= 32) columns; columns l >= Kp pair with themselves.
__device__ __forceinline__ int rr_partner(int l, int r, int Kp) {
    if (l >= Kp) return l;
    int pos = 0;
    if (l > 0) {
        pos = (l - 1 - r) % (Kp - 1);
        if (pos < 0) pos += Kp - 1;
        pos += 1;
    }
    return rr_player(Kp - 1 - pos, r, Kp);
}

// FP32 one-sided (Hestenes) Jacobi in registers, K <= 32, by warps 0..JW-1:
// lane i of every warp holds column i of the symmetric positive semi-definite
// C and of the accumulated rotation V, warp w the rows [w RW, (w + 1) RW). In
// each round of the round-robin ordering (partners from the table ptab) a lane
// takes its partner's entries by shuffles; the warps' partial dot products and
// squared norms are summed through shared memory in a fixed order (one named
// barrier per round, the buffer alternating between rounds), so every warp,
// and both lanes of a pair, take the same rotation from the same numbers, and
// each lane updates its own column (lower index p: c x_p - s x_q, higher q:
// s x_p + c x_q). At convergence the columns of C V are orthogonal, so V
// diagonalises C^2 and therefore C. The warm start needs eigenvectors to FP32
// accuracy only; V is written to X (FP64, K x K).
__device__ void jacobi1_warps(const double *C, int lds, int K, double *X, int max_sweeps, float tol,
                              float2 (*xch)[JW][32], const unsigned char (*ptab)[32]) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    float a[RW], v[RW];
#pragma unroll
    for (int r = 0; r < RW; ++r) {
        const int k = w * RW + r;
        a[r] = (lane < K && k < K) ? (float)C[k * lds + lane] : 0.0f;
        v[r] = (k == lane && lane < K) ? 1.0f : 0.0f;
    }
    const int Kp = K + (K & 1);
    // pairs whose dot product is below floor_g (set by ||C||_F^2, invariant under the
    // rotations) are left alone: their directions carry eigenvalues too small for FP32
    // to resolve, and the FP64 stage handles them
    float f2 = 0.0f;
#pragma unroll
    for (int r = 0; r < RW; ++r) f2 = fmaf(a[r], a[r], f2);
    f2 = warp_sumf(f2);
    xch[1][w][lane] = make_float2(f2, 0.0f);
    jw_bar();
    float f2t = 0.0f;
    for (int u = 0; u < JW; ++u) f2t += xch[1][u][lane].x;
    const float floor_g = 1e-14f * f2t, tol2 = tol * tol;
    int buf = 0;
    for (int sweep = 0; sweep < max_sweeps; ++sweep) {
        bool any = false;
        for (int round = 0; round < Kp - 1; ++round, buf ^= 1) {
            const int partner = ptab[round][lane];
            const int src = partner < 32 ? partner : lane;
            float pa[RW];
            float g = 0.0f, nrm = 0.0f;
#pragma unroll
            for (int r = 0; r < RW; ++r) {
                pa[r] = __shfl_sync(0xffffffffu, a[r], src);
                g = fmaf(a[r], pa[r], g);
                nrm = fmaf(a[r], a[r], nrm);
            }
            xch[buf][w][lane] = make_float2(g, nrm);
            jw_bar();
            g = 0.0f;
            nrm = 0.0f;
#pragma unroll
            for (int u = 0; u < JW; ++u) {
                const float2 t = xch[buf][u][lane];
                g += t.x;
                nrm += t.y;
            }
            const float pn = __shfl_sync(0xffffffffu, nrm, src);
            const bool low = lane < partner;
            const float alpha = low ? nrm : pn, beta = low ? pn : nrm;  // norms^2 of the lower, higher column
            const bool rot = lane < K && partner < K && g * g > tol2 * (alpha * beta) && fabsf(g) > floor_g &&
                             fabsf(g) > 1e-30f;
            float c = 1.0f, sp = 0.0f;  // own' = c own + sp partner
            if (rot) {
                // tangent of the rotation angle: 2 g sign(d) / (|d| + sqrt(d^2 + 4 g^2)), d = beta - alpha
                const float dd = beta - alpha, g2 = 2.0f * g;
                const float r2 = fmaf(dd, dd, g2 * g2);
                const float t = __fdividef(dd >= 0.0f ? g2 : -g2, fabsf(dd) + r2 * rsqrtf(r2));
                c = rsqrtf(fmaf(t, t, 1.0f));
                sp = low ? -t * c : t * c;
                any = true;
            }
#pragma unroll
            for (int r = 0; r < RW; ++r) {
                const float pv = __shfl_sync(0xffffffffu, v[r], src);
                a[r] = fmaf(sp, pa[r], c * a[r]);
                v[r] = fmaf(sp, pv, c * v[r]);
            }
        }
        if (!__any_sync(0xffffffffu, any)) break;  // the same decision in every warp
    }
#pragma unroll
    for (int r = 0; r < RW; ++r) {
        const int k = w * RW + r;
        if (lane < K && k < K) X[k * lds + lane] = (double)v[r];
    }
}

// ------------------------------------------------------------ lambda functions
struct Spec {
    int K;
    double rho, rho0sq;
    const double *theta, *c2;
};
// FP32 copies of theta, 1 - theta and c2 (scaled by 1 / sum c2) for the scans
struct SpecF {
    int K;
    const float *th, *a, *c2;
};

// per-lane terms (lanes stride over i) of the lam-functions and their
// mu-derivatives: s[0] = N = sum c2 g^2, s[1] = N', s[2] = N'', s[3] = D = sum g,
// s[4] = D', s[5] = D'' with g_i = mu a_i / d_i = 1 - f_i, a_i = 1 - theta_i,
// d_i = theta_i + mu a_i.
template <typename R, typename SP>
__device__ __forceinline__ void lam_terms6(const SP &S, R mu, R s[6]) {
    for (int k = 0; k < 6; ++k) s[k] = R(0);
    for (int i = threadIdx.x & 31; i < S.K; i += 32) {
        R th, a, c;
        if constexpr (sizeof(R) == 8) {
            th = S.theta[i];
            a = 1.0 - th;
            c = S.c2[i];
        } else {
            th = S.th[i];
            a = S.a[i];
            c = S.c2[i];
        }
        const R d = th + mu * a;
        if (!(d > R(0))) {
            s[3] += R(1);
            continue;
        }
        R inv;
        if constexpr (sizeof(R) == 8) inv = rcp_newton(d);  // d within [1e-13, 1e13]
        else inv = R(1) / d;
        const R g = mu * a * inv, g1 = a * th * inv * inv, g2 = R(-2) * a * g1 * inv;
        s[0] += c * g * g;
        s[1] += R(2) * c * g * g1;
        s[2] += R(2) * c * (g1 * g1 + g * g2);
        s[3] += g;
        s[4] += g1;
        s[5] += g2;
    }
}
// N and N' only (DP)
template <typename R, typename SP>
__device__ __forceinline__ void lam_terms_n(const SP &S, R mu, R &N, R &N1) {
    N = R(0);
    N1 = R(0);
    for (int i = threadIdx.x & 31; i < S.K; i += 32) {
        R th, a, c;
        if constexpr (sizeof(R) == 8) {
            th = S.theta[i];
            a = 1.0 - th;
            c = S.c2[i];
        } else {
            th = S.th[i];
            a = S.a[i];
            c = S.c2[i];
        }
        const R d = th + mu * a;
        if (!(d > R(0))) continue;
        const R inv = R(1) / d;
        const R g = mu * a * inv, g1 = a * th * inv * inv;
        N += c * g * g;
        N1 += R(2) * c * g * g1;
    }
}
// N and D only (GCV values)
__device__ __forceinline__ void lam_terms_nd(const Spec &S, double mu, double &N, double &D) {
    N = 0.0;
    D = 0.0;
    for (int i = threadIdx.x & 31; i < S.K; i += 32) {
        const double th = S.theta[i], a = 1.0 - th, d = th + mu * a;
        const double g = d > 0.0 ? mu * a * rcp_newton(d) : 1.0;
        N += S.c2[i] * g * g;
        D += g;
    }
}
__device__ __forceinline__ double gcv_value(double N, double D) {
    const double g = N / (D * D);
    return g == g ? g : DBL_MAX;
}
// one thread's FP32 grid value: GCV (N / D^2) or the DP function N - delta
__device__ __forceinline__ void grid_nd(const SpecF &S, float mu, float &N, float &D) {
    N = 0.0f;
    D = 0.0f;
    for (int i = 0; i < S.K; ++i) {
        const float ai = S.a[i], d = fmaf(mu, ai, S.th[i]);
        const float gg = d > 0.0f ? __fdividef(mu * ai, d) : 1.0f;
        N = fmaf(S.c2[i] * gg, gg, N);
        D += gg;
    }
}
template <typename R>
__device__ __forceinline__ R warp_sum_t(R v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// first and second derivative of G = N / D^2 with respect to t = log10(lam)
template <typename R>
__device__ __forceinline__ void gcv_dt(const R s[6], R mu, R &d1, R &d2) {
    const R N = s[0], N1 = s[1], N2 = s[2], D = s[3], D1 = s[4], D2 = s[5];
    const R iD = R(1) / D, iD2 = iD * iD;
    const R G1 = N1 * iD2 - R(2) * N * D1 * iD2 * iD;
    const R G2 = N2 * iD2 - R(4) * N1 * D1 * iD2 * iD - R(2) * N * D2 * iD2 * iD + R(6) * N * D1 * D1 * iD2 * iD2;
    const R ln10 = R(LN10);
    d1 = G1 * mu * ln10;
    d2 = (G2 * mu * mu + G1 * mu) * ln10 * ln10;
}

// size of the two terms whose difference is dG/dt: |dG/dt| below a small
// multiple of it is rounding noise
template <typename R>
__device__ __forceinline__ R gcv_dt_scale(const R s[6], R mu) {
    const R iD = R(1) / s[3];
    return (fabs(s[1]) + fabs(R(2) * s[0] * s[4] * iD)) * iD * iD * mu * R(LN10);
}

// safeguarded Newton step for a root of an increasing function f (f1 = f')
// inside [A, B], which the sign of f shrinks
template <typename R>
__device__ __forceinline__ R newton_step(R t, R f, R f1, R &A, R &B) {
    if (f > R(0)) B = t;
    else if (f < R(0)) A = t;
    R tn = (f1 > R(0)) ? t - f / f1 : R(0.5) * (A + B);
    if (!(tn > A && tn < B)) tn = R(0.5) * (A + B);
    return tn;
}

// mu 10^dt for a small dt (|dt ln 10| < 3e-3: the series to x^5 is exact to 1e-18), else exp10
__device__ __forceinline__ double scale_pow10(double mu, double dt) {
    const double x = dt * LN10;
    if (fabs(x) > 3e-3) return mu * exp10(dt);
    return mu * fma(x, fma(x, fma(x, fma(x, fma(x, 1.0 / 120.0, 1.0 / 24.0), 1.0 / 6.0), 0.5), 1.0), 1.0);
}

// Choice of lam by GCV on rho 10^[-12, 12], mu = lam / rho_mu (theta and c2 belong to the scaling
// rho_mu; ratio = rho / rho_mu). The first minimum of the grid (ties to the smaller lam) is that of
// the FP64 values: an FP32 scan, whose values are exact to 1e-5 (sums of at most 64 positive terms
// with a few roundings each), leaves the points within 1e-4 of its minimum, and those are compared
// in FP64, one warp per point with the terms over the lanes; many such points (a plateau) take one
// thread each. Then safeguarded Newton steps on dG/dt = 0 between the neighbours, t = log10 mu:
// FP32 steps to a starting point, then FP64 steps that carry mu itself (an FP64 exponential per step
// would cost as much as the step); where the five FP64 values around the minimum agree to 1e-13
// the grid point stands. The result is sh.mu. All threads call; ends with a barrier.
struct GcvShared {
    float val[GRID_POINTS];   // FP32 grid (0: not usable)
    double grid[GRID_POINTS]; // FP64 values of the candidates, else DBL_MAX
    int cand[GRID_POINTS];
    float wmin[NW];
    int count, ig, check;
    double mu;
};
// the grid 10^(-12 + 24 i / 199), passed to the kernel as a parameter
struct GcvGrid {
    double v[GRID_POINTS];
};

__device__ void gcv_lambda(const Spec &S, const SpecF &SF, const GcvGrid &grid, double ratio, GcvShared &sh) {
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    constexpr float stepf = (float)(2.0 * BRACKET_DECADES / (GRID_POINTS - 1)), lof = (float)-BRACKET_DECADES;
    const float ratiof = (float)ratio;
    float v = 3.4e38f;
    if (tid < GRID_POINTS) {
        float N, D;
        grid_nd(SF, exp10f(fmaf((float)tid, stepf, lof)) * ratiof, N, D);
        const float g = N / (D * D);
        const bool ok = N > 1e-36f && D * D > 1e-36f && g < 3e38f;
        sh.val[tid] = ok ? g : 0.0f;
        if (ok) v = g;
        sh.grid[tid] = DBL_MAX;
    }
    for (int o = 16; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(0xffffffffu, v, o));
    if (lane == 0) sh.wmin[wid] = v;
    if (tid == 0) sh.count = 0;
    __syncthreads();
    v = sh.wmin[0];
    for (int w = 1; w < NW; ++w) v = fminf(v, sh.wmin[w]);
    if (tid < GRID_POINTS && sh.val[tid] <= v * 1.0001f) sh.cand[atomicAdd(&sh.count, 1)] = tid;
    __syncthreads();
    auto value = [&](int gi) {  // by a warp, the terms over its lanes
        double N, D;
        lam_terms_nd(S, grid.v[gi] * ratio, N, D);
        warp_sum2(N, D);
        return gcv_value(N, D);
    };
    if (sh.count <= 4 * NW) {
        for (int c = wid; c < sh.count; c += NW) {
            const double g = value(sh.cand[c]);
            if (lane == 0) sh.grid[sh.cand[c]] = g;
        }
    } else if (tid < sh.count) {
        const int gi = sh.cand[tid];
        const double mu = grid.v[gi] * ratio;
        double N = 0.0, D = 0.0;
        for (int i = 0; i < S.K; ++i) {
            const double th = S.theta[i], am = 1.0 - th, d = th + mu * am;
            const double g = d > 0.0 ? mu * am / d : 1.0;
            N += S.c2[i] * g * g;
            D += g;
        }
        sh.grid[gi] = gcv_value(N, D);
    }
    __syncthreads();
    if (wid == 0) {
        double bv = DBL_MAX;
        int ig = GRID_POINTS;
        for (int gi = lane; gi < GRID_POINTS; gi += 32)
            if (sh.grid[gi] < bv) {
                bv = sh.grid[gi];
                ig = gi;
            }
        for (int o = 16; o > 0; o >>= 1) {
            const double bo = __shfl_xor_sync(0xffffffffu, bv, o);
            const int io = __shfl_xor_sync(0xffffffffu, ig, o);
            if (bo < bv || (bo == bv && io < ig)) {
                bv = bo;
                ig = io;
            }
        }
        if (ig >= GRID_POINTS) ig = 0;
        // flat to rounding only if the FP32 neighbours are within their error of it
        bool check = true;
        for (int w = -(NREF / 2); w <= NREF / 2; ++w) {
            const float q = sh.val[min(max(ig + w, 0), GRID_POINTS - 1)];
            if (q > v * 1.0001f) check = false;
        }
        if (lane == 0) {
            sh.ig = ig;
            sh.check = check;
        }
    }
    __syncthreads();
    const int ig = sh.ig;
    if (sh.check) {
        for (int w = wid; w < NREF; w += NW) {
            const int gi = min(max(ig + w - NREF / 2, 0), GRID_POINTS - 1);
            if (sh.grid[gi] != DBL_MAX) continue;
            const double g = value(gi);
            __syncwarp();
            if (lane == 0) sh.grid[gi] = g;
        }
        __syncthreads();
    }
    if (wid == 0) {
        const double bv = sh.grid[ig];
        bool flat = false;
        if (sh.check) {
            double vmax = bv;
            for (int w = -(NREF / 2); w <= NREF / 2; ++w) vmax = fmax(vmax, sh.grid[min(max(ig + w, 0), GRID_POINTS - 1)]);
            flat = vmax - bv <= 1e-13 * bv;
        }
        const double mu0 = grid.v[ig] * ratio;
        double mu = mu0;
        if (!flat) {
            // t is relative to the grid point, the bracket its neighbours
            const float Af = ig > 0 ? -stepf : 0.f, Bf = ig < GRID_POINTS - 1 ? stepf : 0.f, muf = (float)mu0;
            float tf = 0.f, Af0 = Af, Bf0 = Bf;
            for (int it = 0; it < NEWTON32_MAX; ++it) {
                float s[6], d1, d2;
                const float m = exp10f(tf) * muf;
                lam_terms6<float>(SF, m, s);
                for (int k = 0; k < 6; ++k) s[k] = warp_sum_t(s[k]);
                gcv_dt<float>(s, m, d1, d2);
                if (d1 == 0.0f || !(d1 == d1)) break;
                if (fabsf(d1) <= 1e-5f * gcv_dt_scale<float>(s, m)) break;  // at the rounding level
                const float tn = newton_step<float>(tf, d1, d2, Af0, Bf0);
                const float dt = fabsf(tn - tf);
                tf = tn;
                if (dt <= 1e-6f || Bf0 - Af0 <= 1e-6f) break;
            }
            double t = (double)tf, A1 = (double)Af, B1 = (double)Bf;
            if (!(t > A1 && t < B1)) t = 0.0;
            mu = mu0 * (t == 0.0 ? 1.0 : (double)exp10f(tf));  // t follows mu to FP32 accuracy: it only brackets
            for (int it = 0; it < NEWTON_MAX; ++it) {
                double s6[6];
                lam_terms6<double>(S, mu, s6);
                warp_sum6(s6);
                // derivatives of G in mu times D^2: G1 D^2 = N1 - 2 N D1 / D, G2 D^2 = N2 - 4 N1 D1 / D -
                // 2 N D2 / D + 6 N (D1 / D)^2, and in t: d1 = G1 mu ln10, d2 = (G2 mu + G1) mu ln10^2
                const double iD = rcp_newton(s6[3]), u = s6[4] * iD, w = s6[0] * u;
                const double g1 = s6[1] - 2.0 * w;
                if (g1 == 0.0 || !(g1 == g1) || fabs(g1) <= 1e-12 * (fabs(s6[1]) + fabs(2.0 * w))) break;  // at the rounding level
                const double g2 = s6[2] - u * (4.0 * s6[1] - 6.0 * w) - 2.0 * s6[0] * s6[5] * iD, q = fma(g2, mu, g1) * LN10;
                if (g1 > 0.0) B1 = t;
                else A1 = t;
                double tn = t - g1 / q;
                const bool pure = q > 0.0 && tn > A1 && tn < B1;
                if (!pure) tn = 0.5 * (A1 + B1);
                const double dt = fabs(tn - t);
                mu = scale_pow10(mu, tn - t);
                t = tn;
                if (dt <= 1e-10 || B1 - A1 <= 1e-10) break;
                if (pure && dt <= 1e-6) break;  // quadratic: the next step is ~1e-12
            }
            double N, D;
            lam_terms_nd(S, mu, N, D);
            warp_sum2(N, D);
            if (!(gcv_value(N, D) <= bv)) mu = mu0;
        }
        if (lane == 0) sh.mu = mu;
    }
    __syncthreads();
}

// ------------------------------------------------------------ bordered eigenproblem
// A GKS iteration appends one vector, so its Grams are the previous ones with one more row and
// column. With Y the generalised eigenvectors of the previous pair scaled to Y^T (G_A + rho G_L) Y
// = I (rho that of the first, full solve), Y^T G_A Y = diag(d), the new problem in the basis
// [Y, w / nu], w = e_n - Y m, m = Y^T (new column of G_A + rho G_L), nu^2 = its new diagonal entry
// - ||m||^2, is the bordered diagonal matrix [diag(d) c; c^T gam], whose eigenvalues are the
// roots of the secular equation F(x) = x - gam - sum c_i^2 / (x - d_i) = 0, one between any two
// neighbouring poles and one beyond each end. A root is held as its distance mu from the nearest
// pole, found in FP32 by interpolation with two poles (four threads per root) and then by FP64
// Newton steps on mu F. The borders c that have exactly the computed roots follow from
// c_i^2 = prod_j (x_j - d_i) / prod_{j != i} (d_j - d_i) (Loewner; Gu and Eisenstat 1995), so
// the eigenvectors c_i / (x_j - d_i) are orthogonal to rounding however close the roots are.
// One product of n x n matrices updates Y; all else is O(n^2). Entries with |c_i| at the rounding
// level of the matrix are eigenpairs already. Poles closer than that, a nearly dependent new
// vector or a root that did not converge leave the call to the full solve.
constexpr int BE_NV = 14;        // vectors of the bordered solve in shared memory
constexpr int BE_PART = 2 * ST;  // doubles of its partial sums
struct BorderShared {
    double gam, eta, inu, tol;
    int p, bad;
};

// One interpolation step of a root in FP32 by four adjacent lanes (sub = 0..3, all of the warp
// call): poles de[i] (relative to the origin pole o), squared borders z2[i], the first k poles left
// of the root; e = origin - gam. Returns F, the proposal in x and the size of F's terms.
__device__ float be_step32(const float *de, const float *z2, int p, int k, int o, float e, float m, int sub, float &x, float &size) {
    float P = 0.f, Pp = 0.f, R = 0.f, Rp = 0.f;
#pragma unroll 4
    for (int i = sub; i < p; i += 4) {
        const float q = __fdividef(1.0f, m - de[i]), t = z2[i] * q, t2 = t * q;
        const bool left = i < k;
        P -= left ? t : 0.f;
        Pp += left ? t2 : 0.f;
        R -= left ? 0.f : t;
        Rp += left ? 0.f : t2;
    }
#pragma unroll
    for (int w = 1; w < 4; w <<= 1) {
        P += __shfl_xor_sync(0xffffffffu, P, w);
        Pp += __shfl_xor_sync(0xffffffffu, Pp, w);
        R += __shfl_xor_sync(0xffffffffu, R, w);
        Rp += __shfl_xor_sync(0xffffffffu, Rp, w);
    }
    const float F = e + m + P + R;
    size = fabsf(e) + fabsf(m) + fabsf(P) + fabsf(R);
    if (k == 0 || k == p) {  // one pole, at the origin: x^2 + C x = a
        const float a = (k == 0 ? Rp : Pp) * m * m, C = e + (k == 0 ? R : P) + a / m;
        const float ds = sqrtf(fmaf(C, C, 4.0f * a));
        if (k == 0) x = C >= 0.f ? -0.5f * (C + ds) : 2.0f * a / (C - ds);
        else x = C <= 0.f ? 0.5f * (ds - C) : 2.0f * a / (C + ds);
        return F;
    }
    const float dL = de[k - 1], dR = de[k];
    const float a = Pp * (m - dL) * (m - dL), pc = P + a / (m - dL);
    const float b = (1.0f + Rp) * (dR - m) * (dR - m), qc = m + R - b / (dR - m);
    const float C = e + pc + qc, W = o == k - 1 ? dR : dL, t = o == k - 1 ? a : b;
    const float B = fmaf(C, W, a + b), ds = sqrtf(fmaxf(fmaf(B, B, -4.0f * C * t * W), 0.f));
    x = B > 0.f ? 2.0f * t * W / (B + ds) : (B - ds) / (2.0f * C);
    return F;
}

// Updates Y (K - 1 x K - 1 in Ym, the result K x K in Yo; row stride lds) with its eigenvalues d
// and the components gh = Y^T g to K, for the new last row and column of G_A, G_L and entry of g.
// Q: K x K scratch; v: BE_NV vectors of lds; part: BE_PART doubles. False: not possible (d, gh, Ym are
// as they were).
__device__ bool be_update(const double *GA, const double *GL, const double *g, int ld, int K, double rho, double *Ym, double *Yo,
                          double *Q, int lds, double *d, double *gh, double *v, double *part, BorderShared &sh) {
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, n = K - 1;
    double *av = v, *mv = v + lds, *ah = v + 2 * lds, *mh = v + 3 * lds, *c = v + 4 * lds, *yw = v + 5 * lds;
    double *D = v + 6 * lds, *Z = v + 7 * lds, *Z2 = av, *mu = v + 8 * lds, *ct = v + 9 * lds, *nrm = v + 10 * lds, *nd = v + 11 * lds;
    int *map = reinterpret_cast<int *>(v + 12 * lds), *org = map + lds;
    float *zf = reinterpret_cast<float *>(v + 13 * lds);
    float *df = reinterpret_cast<float *>(Q);  // [root][pole], free until Q is formed
    for (int i = tid; i < n; i += ST) {
        const double x = GA[i * ld + n];
        av[i] = x;
        mv[i] = fma(rho, GL[i * ld + n], x);
    }
    if (tid == 0) sh.bad = 0;
    __syncthreads();
    row_sums2(n, n, part,  // Y^T (new columns)
              [&](int j, int r, double &x, double &y) {
                  const double q = Ym[r * lds + j];
                  x += q * av[r];
                  y += q * mv[r];
              },
              [&](int j, double x, double y) {
                  ah[j] = x;
                  mh[j] = y;
              });
    row_sums(n, n, part, [&](int r, int j) { return Ym[r * lds + j] * mh[j]; }, [&](int r, double x) { yw[r] = x; });  // Y m
    if (wid == 0) {
        double mm = 0.0, ma = 0.0, tm = 0.0, mg = 0.0;
        for (int i = lane; i < n; i += 32) {
            const double m = mh[i];
            mm += m * m;
            ma += m * ah[i];
            tm += d[i] * m * m;
            mg += m * gh[i];
        }
        warp_sum2(mm, ma);
        warp_sum2(tm, mg);
        const double al = GA[n * ld + n], mnn = fma(rho, GL[n * ld + n], al), nu2 = mnn - mm;
        const bool ok = nu2 > 1e-8 * mnn && isfinite(nu2);
        const double inu = ok ? rsqrt(nu2) : 0.0, gam = (al - 2.0 * ma + tm) * inu * inu;
        float big = fabsf((float)gam);
        for (int i = lane; i < n; i += 32) {
            const double x = (ah[i] - d[i] * mh[i]) * inu;
            c[i] = x;
            big = fmaxf(big, fmaxf(fabsf((float)x), fabsf((float)d[i])));
        }
        big = warp_maxf(big);
        if (lane == 0) {
            sh.gam = gam;
            sh.inu = inu;
            sh.eta = (g[n] - mg) * inu;
            sh.tol = 16.0 * 2.22e-16 * (double)big;
            if (!ok || !(big < 1e6f)) sh.bad = 1;
        }
    }
    __syncthreads();
    const double gam = sh.gam, tol = sh.tol, inu = sh.inu, eta = sh.eta;
    // the poles that take part, in ascending order
    if (tid == 0) sh.p = 0;
    __syncthreads();
    // (as integers in the order of the doubles: an FP64 comparison holds the pipe like an addition)
    long long *key = reinterpret_cast<long long *>(mu);
    if (tid < n) {
        const long long q = __double_as_longlong(d[tid]);
        key[tid] = fabs(c[tid]) > tol ? (q ^ ((q >> 63) & 0x7fffffffffffffffll)) : 0x7fffffffffffffffll;
    }
    __syncthreads();
    if (tid < n && key[tid] != 0x7fffffffffffffffll) {
        int rank = 0;
        const double x = d[tid];
        const long long kt = key[tid];
        for (int j = 0; j < n; ++j) rank += key[j] < kt || (key[j] == kt && j < tid);
        D[rank] = x;
        Z[rank] = c[tid];
        map[rank] = tid;
        atomicAdd(&sh.p, 1);
    }
    __syncthreads();
    const int p = sh.p;
    if (tid + 1 < p && D[tid + 1] - D[tid] <= 4.0 * tol) sh.bad = 1;
    if (tid < p) {
        Z2[tid] = Z[tid] * Z[tid];
        zf[tid] = (float)Z2[tid];
    }
    if (tid <= p) org[tid] = max(tid - 1, 0);
    if (p == 0 && tid == 0) sh.bad = 1;
    __syncthreads();
    if (sh.bad) return false;
    // roots in FP32, four threads each: first the pole it is nearer to
    for (int pass = 0; pass < 2; ++pass) {
        for (int e = tid; e < (p + 1) * p; e += ST) {
            const int k = e / p, i = e - k * p;
            df[e] = (float)(D[i] - D[org[k]]);
        }
        __syncthreads();
        if (pass == 0) {
            const int k = min(max(tid >> 2, 1), p);  // (threads of no interior root repeat another's)
            const float *de = df + k * p;
            float x, size;
            const float gap = k < p ? de[k] : 1.f;
            const float F = be_step32(de, zf, p, k, k - 1, (float)(D[k - 1] - gam), 0.5f * gap, tid & 3, x, size);
            __syncthreads();
            if ((tid & 3) == 0 && (tid >> 2) == k && k < p && !(F >= 0.f)) org[k] = k;
        }
        __syncthreads();
    }
    {
        const int k = min(tid >> 2, p), o = org[k];
        const float *de = df + k * p, e = (float)(D[o] - gam);
        float A, B;
        if (k == 0 || k == p) {  // |x - pole| <= |pole - gam| + ||c||
            float z = 0.f;
            for (int i = 0; i < p; ++i) z += zf[i];
            const float w = fabsf(e) + sqrtf(z) * 1.0001f + 1e-30f;
            A = k == 0 ? -w : 0.f;
            B = k == 0 ? 0.f : w;
        } else {
            A = o == k ? 0.5f * de[k - 1] : 0.f;
            B = o == k ? 0.f : 0.5f * de[k];
        }
        float m = 0.5f * (A + B);
        bool on = true;
        for (int it = 0; it < 32 && __any_sync(0xffffffffu, on); ++it) {
            float x, size;
            const float F = be_step32(de, zf, p, k, o, e, m, tid & 3, x, size);
            if (!on) continue;
            if (fabsf(F) <= 2.4e-7f * size) {
                on = false;
                continue;
            }
            if (F > 0.f) B = m;
            else A = m;
            if (!(x > A && x < B)) x = 0.5f * (A + B);
            on = fabsf(x - m) > 1e-6f * fabsf(x);
            m = x;
        }
        if ((tid & 3) == 0 && (tid >> 2) <= p) mu[k] = (double)m;
    }
    __syncthreads();
    // FP64: Newton steps on mu F(mu) = mu (origin - gam + mu - S1) - c_o^2, S1 and S2 the sums over
    // the other poles; the terms of a root spread over the threads of its column of parts
    const int RS = p + 1 <= 32 ? 32 : 64, parts = ST / RS, root = tid & (RS - 1), pt = tid / RS;
    for (int it = 0; it < 8; ++it) {
        double S1 = 0.0, S2 = 0.0;
        const bool on = root <= p;
        const int o = on ? org[root] : 0;
        const double m = on ? mu[root] : 1.0, Do = D[o];
        if (on)
            for (int i = pt; i < p; i += parts) {
                if (i == o) continue;
                const double q = rcp_newton(m - (D[i] - Do)), t = Z2[i] * q;
                S1 += t;
                S2 += t * q;
            }
        part[tid] = S1;
        part[ST + tid] = S2;
        __syncthreads();
        int more = 0;
        if (tid <= p) {  // (the first p + 1 threads are part 0 of every root)
            for (int q = 1; q < parts; ++q) {
                S1 += part[q * RS + tid];
                S2 += part[ST + q * RS + tid];
            }
            const double r = (Do - gam) + m - S1, z = Z2[o], h = m * r - z, hp = r + m + m * S2;
            const double x = m - h / hp;
            // the root stays on its side of the pole and short of the next one: a step that leads away from
            // there started on the wrong side of the root (an FP32 search among terms that cancel)
            const double lim = root == 0 || root == p ? 1e30 : 0.75 * (D[root] - D[root - 1]);
            if (!(x * m > 0.0 && fabs(x) < lim)) sh.bad = 1;  // (the step from m is the same in every round)
            const double dx = fabs(x - m);
            mu[tid] = x;
            more = dx > 1e-9 * fabs(x);  // quadratic: the next step would be at the rounding level
            if (it == 7 && more) sh.bad = 1;
        }
        if (!__syncthreads_or(more)) break;
    }
    if (sh.bad) return false;
    // Loewner borders: products over the roots in parts, each factor a quotient near 1
    {
        const int i = root;
        double pr = 1.0;
        if (i < p)
            for (int j = pt; j < p; j += parts) {
                const double f = (D[org[j]] - D[i]) + mu[j];
                pr *= j == i ? f : f * rcp_newton(D[j] - D[i]);
            }
        part[tid] = pr;
        __syncthreads();
        if (tid < p) {
            for (int q = 1; q < parts; ++q) pr *= part[q * RS + tid];
            pr *= (D[org[p]] - D[tid]) + mu[p];
            const double x = sqrt(fabs(pr));
            ct[tid] = Z[tid] < 0.0 ? -x : x;
        }
        __syncthreads();
    }
    // eigenvectors c_i / (x_j - d_i) (the last component 1) and their norms
    for (int e = tid; e < p * (p + 1); e += ST) {
        const int i = e / (p + 1), j = e - i * (p + 1);
        Q[i * lds + j] = ct[i] * rcp_newton((D[org[j]] - D[i]) + mu[j]);
    }
    __syncthreads();
    row_sums2(p + 1, p, part,
              [&](int j, int i, double &x, double &y) {
                  const double q = Q[i * lds + j];
                  x += q * q;
                  y += q * gh[map[i]];
              },
              [&](int j, double x, double y) {
                  const double f = rsqrt(1.0 + x);
                  nrm[j] = f;
                  ah[j] = (y + eta) * f;  // component of g
                  nd[j] = D[org[j]] + mu[j];
              });
    // Yo = [Y, w / nu] Q: rows 0..n-1, then the last row (0, ..., 0, 1 / nu)
    for (int e = tid; e < n * (p + 1); e += ST) {
        const int r = e / (p + 1), j = e - r * (p + 1);
        double x = -yw[r] * inu;
        for (int i = 0; i < p; ++i) x += Ym[r * lds + map[i]] * Q[i * lds + j];
        Yo[r * lds + j] = x * nrm[j];
    }
    for (int j = tid; j <= p; j += ST) Yo[n * lds + j] = inu * nrm[j];
    // eigenpairs that the border leaves alone, behind the others
    if (wid == 0) {
        int at = p + 1;
        for (int i0 = 0; i0 < n; i0 += 32) {
            const int i = i0 + lane;
            const bool still = i < n && !(fabs(c[i]) > tol);
            const unsigned m = __ballot_sync(0xffffffffu, still);
            if (still) {
                const int j = at + __popc(m & ((1u << lane) - 1u));
                nd[j] = d[i];
                ah[j] = gh[i];
                for (int r = 0; r < n; ++r) Yo[r * lds + j] = Ym[r * lds + i];
                Yo[n * lds + j] = 0.0;
            }
            at += __popc(m);
        }
    }
    __syncthreads();
    for (int j = tid; j < K; j += ST) {
        d[j] = nd[j];
        gh[j] = ah[j];
    }
    __syncthreads();
    return true;
}

}  // namespace

__global__ void __launch_bounds__(ST, 1) k_small_solve(SmallArgs a, const __grid_constant__ GcvGrid grid) {
    extern __shared__ double sm[];
    __shared__ double s_rho, s_rho0sq, s_t, s_scale, s_lam;
    __shared__ GcvShared s_gcv;
    __shared__ BorderShared s_be;
    __shared__ float s_redf[NW];
    __shared__ int s_fail, s_flag, s_idx[NW], s_end[4];
    __shared__ JacobiShared<float> jf;
    __shared__ JacobiShared<double> jd;
    __shared__ float2 s_xch[2][JW][32];
    __shared__ unsigned char s_ptab[31][32];
    const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int ld = a.ld;
    const int K = min(a.K[b], ld);
    double *z = a.z + (long long)b * ld;
    for (int i = tid; i < ld; i += ST) z[i] = 0.0;
    if (K <= 0 || (a.active && !a.active[b])) {
        if (tid == 0) {
            a.lam[b] = 0.0;
            a.flag[b] = 0;
        }
        return;
    }
    const int Kp = K + (K & 1);
    if (Kp <= 32)  // partners of the FP32 Jacobi rounds
        for (int e = tid; e < (Kp - 1) * 32; e += ST) s_ptab[e >> 5][e & 31] = (unsigned char)rr_partner(e & 31, e >> 5, Kp);
    const int lds = (ld + 1) | 1;  // FP64 leading dimension: odd, >= Kp and >= K + 1
    const int ldf = ld + 3;        // FP32 leading dimension
    double *Rm = sm;               // Cholesky rows of M = G_A + rho G_L (kept for z)
    double *Cm = Rm + lds * lds;   // [G_A | g] -> [R^-T G_A | h] -> C = R^-T G_A R^-1 (kept for z)
    double *Um = Cm + lds * lds;   // R rows over their diagonal; then X^T C X; then C + mu (I - C)
    double *Xm = Um + lds * lds;   // eigenvector estimate
    double *Tm = Xm + lds * lds;   // scratch (FP32 Jacobi matrix first)
    double *Em = Tm + lds * lds;   // scratch (FP32 eigenvectors first)
    double *vec = Em + lds * lds;
    double *theta = vec, *gh = vec + lds, *c2 = vec + 2 * lds, *invd = vec + 3 * lds, *hv = vec + 4 * lds;
    float *fvec = reinterpret_cast<float *>(vec + 5 * lds);  // 3 x lds floats within 2 x lds doubles
    double *bv = vec + 7 * lds;                              // bordered solve: BE_NV vectors, partial sums
    double *bpart = bv + BE_NV * lds;
    float *thf = fvec, *af = fvec + lds, *c2f = fvec + 2 * lds;
    float *Af = reinterpret_cast<float *>(Tm);
    float *Wf = reinterpret_cast<float *>(Em);
    const double *GA = a.GA + (long long)b * ld * ld;
    const double *GL = a.GL + (long long)b * ld * ld;
    const double *g = a.g + (long long)b * ld;
#define AT(P, i, j) P[(i) * lds + (j)]
#define AF(P, i, j) P[(i) * ldf + (j)]

    // ---------------------------------------------- 1. Cholesky of M, C and h (FP64)
    if (wid == 0) {
        double tA = 0.0, tL = 0.0;
        for (int i = lane; i < K; i += 32) {
            tA += GA[i * ld + i];
            tL += GL[i * ld + i];
        }
        warp_sum2(tA, tL);
        if (lane == 0) {
            s_rho = (tA > 0.0 && tL > 0.0) ? tA / tL : 1.0;
            s_fail = 0;
            s_flag = 0;
        }
    }
    __syncthreads();
    const double rho = s_rho;
    // lambda by GCV for theta = clamped eigenvalues raw[] in the scaling rho_mu and components gh
    auto choose_gcv = [&](const double *raw, double rho_mu) {
        for (int i = tid; i < K; i += ST) {
            const double x = fmin(fmax(raw[i], 0.0), 1.0);
            theta[i] = x;
            c2[i] = x > THETA_TINY ? gh[i] * gh[i] / x : 0.0;
        }
        __syncthreads();
        if (wid == 0) {
            double kept = 0.0, unused = 0.0;
            for (int i = lane; i < K; i += 32) kept += c2[i];
            warp_sum2(kept, unused);
            if (lane == 0) {
                s_rho0sq = a.bb[b] - kept;
                s_scale = kept > 0.0 ? 1.0 / kept : 1.0;
            }
        }
        __syncthreads();
        for (int i = tid; i < K; i += ST) {
            thf[i] = (float)theta[i];
            af[i] = (float)(1.0 - theta[i]);
            c2f[i] = (float)(c2[i] * s_scale);
        }
        __syncthreads();
        if (a.rule != MOF_RULE_GCV) return;
        if (tid == 0) s_t = rho / rho_mu;
        __syncthreads();
        gcv_lambda(Spec{K, rho, s_rho0sq, theta, c2}, SpecF{K, thf, af, c2f}, grid, s_t, s_gcv);
        if (tid == 0) s_lam = s_gcv.mu * rho_mu;
        __syncthreads();
    };
    // ---------------------------------------------- 0. from the previous call's eigenvectors
    bool bordered = false;
    double lam = a.lam_fixed;
    if (a.Y) {
        double *Yg = a.Y + (long long)b * ld * ld, *dg = a.Yd + (long long)b * ld, *hg = a.Yh + (long long)b * ld;
        const int nY = a.nY[b];
        const double rho0 = a.Yrho[b];
        if (nY > 0 && (nY == K || nY == K - 1)) {
            for (int e = tid; e < nY * nY; e += ST) {
                const int i = e / nY, j = e - i * nY;
                AT(Cm, i, j) = Yg[i * ld + j];
            }
            for (int i = tid; i < nY; i += ST) {
                hv[i] = dg[i];
                gh[i] = hg[i];
            }
            __syncthreads();
            double *Ym = Cm;
            bordered = nY == K;
            if (!bordered) {
                bordered = be_update(GA, GL, g, ld, K, rho0, Cm, Tm, Um, lds, hv, gh, bv, bpart, s_be);
                Ym = Tm;
            }
            if (bordered) {
                if (nY != K) {
                    for (int e = tid; e < K * K; e += ST) {
                        const int i = e / K, j = e - i * K;
                        Yg[i * ld + j] = AT(Tm, i, j);
                    }
                    for (int i = tid; i < K; i += ST) {
                        dg[i] = hv[i];
                        hg[i] = gh[i];
                    }
                    if (tid == 0) a.nY[b] = K;
                }
                choose_gcv(hv, rho0);
                lam = s_lam;
                const double mu = lam / rho0;
                // z = Y diag(1 / (theta + mu (1 - theta))) Y^T g, and one step of refinement with the
                // residual of (G_A + lam G_L) z = g
                double *w = bv, *zz = bv + lds, *rr = bv + 2 * lds;
                for (int i = tid; i < K; i += ST) w[i] = gh[i] / (theta[i] + mu * (1.0 - theta[i]));
                __syncthreads();
                row_sums(K, K, bpart, [&](int i, int k) { return AT(Ym, i, k) * w[k]; }, [&](int i, double t) { zz[i] = t; });
                row_sums2(K, K, bpart,
                          [&](int i, int k, double &x, double &y) {  // (the Grams are stored symmetric)
                              x += GA[k * ld + i] * zz[k];
                              y += GL[k * ld + i] * zz[k];
                          },
                          [&](int i, double x, double y) { rr[i] = g[i] - (x + lam * y); });
                row_sums(K, K, bpart, [&](int j, int r) { return AT(Ym, r, j) * rr[r]; },
                         [&](int j, double t) { w[j] = t / (theta[j] + mu * (1.0 - theta[j])); });
                row_sums(K, K, bpart, [&](int i, int k) { return AT(Ym, i, k) * w[k]; }, [&](int i, double t) { zz[i] += t; });
                int bad = 0;
                for (int i = tid; i < K; i += ST) {
                    z[i] = gh[i] = zz[i];
                    bad |= !isfinite(zz[i]);
                }
                if (__syncthreads_or(bad) && tid == 0) atomicOr(a.err, 2);
                if (tid == 0) {
                    a.lam[b] = lam;
                    a.flag[b] = 0;
                }
            }
        }
    }
    if (!bordered) {
    __syncthreads();
    for (int e = tid; e < K * K; e += ST) {
        const int i = e / K, j = e - (e / K) * K;
        const double ga = GA[i * ld + j];
        AT(Cm, i, j) = ga;
        AT(Rm, i, j) = ga + rho * GL[i * ld + j];
    }
    for (int i = tid; i < K; i += ST) AT(Cm, i, K) = g[i];
    __syncthreads();
    chol_upper(Rm, lds, K, invd, &s_fail);
    if (s_fail) {
        if (tid == 0) {
            atomicOr(a.err, 1);
            a.lam[b] = 0.0;
            a.flag[b] = 0;
        }
        return;
    }
    for (int e = tid; e < K * K; e += ST) {
        const int i = e / K, k = e - (e / K) * K;
        if (k > i) AT(Um, i, k) = AT(Rm, i, k) * invd[i];
    }
    __syncthreads();
    trsm_rt(Um, lds, invd, Cm, lds, K, K + 1);  // [G_A | g] <- R^-T [G_A | g]
    for (int i = tid; i < K; i += ST) hv[i] = AT(Cm, i, K);
    trsm_r(Um, lds, invd, Cm, lds, K, K);  // C = (R^-T G_A) R^-1
    for (int e = tid; e < K * K; e += ST) {  // exact symmetry
        const int i = e / K, j = e - (e / K) * K;
        if (j > i) {
            const double s = 0.5 * (AT(Cm, i, j) + AT(Cm, j, i));
            AT(Cm, i, j) = s;
            AT(Cm, j, i) = s;
        }
    }
    __syncthreads();

    if (a.rule != MOF_RULE_FIXED) {
        // ------------------------------------------ 2a. FP32 Jacobi on C
        if (K <= 32) {  // registers only
            if (wid < JW) jacobi1_warps(Cm, lds, K, Xm, JACOBI32_MAX_SWEEPS, 1e-6f, s_xch, s_ptab);
            __syncthreads();
        } else {
            for (int e = tid; e < Kp * Kp; e += ST) {
                const int i = e / Kp, j = e - (e / Kp) * Kp;
                AF(Af, i, j) = (i < K && j < K) ? (float)AT(Cm, i, j) : 0.0f;
                AF(Wf, i, j) = i == j ? 1.0f : 0.0f;
            }
            __syncthreads();
            jacobi<float>(Af, ldf, Wf, ldf, (float *)nullptr, K, Kp, JACOBI32_MAX_SWEEPS, 1e-6f, 1e-7f, jf, s_redf);
            for (int e = tid; e < K * K; e += ST) {
                const int i = e / K, j = e - (e / K) * K;
                AT(Xm, i, j) = (double)AF(Wf, i, j);
            }
            __syncthreads();
        }

        // ------------------------------------------ 2b. FP64: orthonormalise, congruence
        gemm_kk(Tm, Xm, true, Xm, false, K, lds, true);  // X0^T X0 (the FP32 matrix is done with)
        for (int i = tid; i < K; i += ST) AT(Tm, i, i) -= 1.0;  // E = X0^T X0 - I
        __syncthreads();
        gemm_kk(Em, Tm, false, Tm, false, K, lds, true);  // E^2 (the FP32 eigenvectors are in Xm)
        for (int e = tid; e < K * K; e += ST) {           // P = I - E/2 + 3 E^2/8
            const int i = e / K, j = e - (e / K) * K;
            AT(Em, i, j) = (i == j ? 1.0 : 0.0) - 0.5 * AT(Tm, i, j) + 0.375 * AT(Em, i, j);
        }
        __syncthreads();
        gemm_kk(Tm, Xm, false, Em, false, K, lds, false);  // X = X0 P
        for (int e = tid; e < K * K; e += ST) {
            const int i = e / K, j = e - (e / K) * K;
            AT(Xm, i, j) = AT(Tm, i, j);
        }
        __syncthreads();
        gemm_kk(Tm, Cm, false, Xm, false, K, lds, false);  // T = C X
        gemm_kk(Um, Xm, true, Tm, false, K, lds, true);    // X^T C X
        for (int i = tid; i < Kp; i += ST) {               // gh = X^T h; zero padding of an odd size
            double s = 0.0;
            if (i < K)
                for (int k = 0; k < K; ++k) s += AT(Xm, k, i) * hv[k];
            gh[i] = s;
            if (K & 1) {
                AT(Um, i, K) = 0.0;
                AT(Um, K, i) = 0.0;
            }
        }
        __syncthreads();

        // ------------------------------------------ 2c. FP64 Jacobi polish
        jacobi<double>(Um, lds, a.Y ? Xm : (double *)nullptr, lds, gh, K, Kp, JACOBI64_MAX_SWEEPS, 1e-16f, 1e-12f, jd, s_redf);
        for (int i = tid; i < K; i += ST) {
            bv[i] = AT(Um, i, i);
            if (a.Y) {
                a.Yd[(long long)b * ld + i] = bv[i];
                a.Yh[(long long)b * ld + i] = gh[i];
            }
        }
        __syncthreads();

        // ------------------------------------------ 3-4. lambda
        choose_gcv(bv, rho);
        const Spec S{K, rho, s_rho0sq, theta, c2};
        const SpecF SF{K, thf, af, c2f};
        const double lrho = log10(rho);
        const double lo = lrho - BRACKET_DECADES, hi = lrho + BRACKET_DECADES;
        const double step = (hi - lo) / (GRID_POINTS - 1);
        if (a.rule != MOF_RULE_GCV) {  // DP on F(t) = N(mu(t)) + rho0^2 - (eta delta)^2, increasing in t
            if (wid < 2) {  // the bracket ends, in FP64
                double N, N1;
                lam_terms_n<double>(S, exp10(wid ? hi : lo) / rho, N, N1);
                warp_sum2(N, N1);
                const double F = N + S.rho0sq - a.target2;
                if (lane == 0) s_end[wid] = wid ? (F <= 0.0) : (F >= 0.0);
            }
            __syncthreads();
            const int flag = s_end[0] ? 1 : (s_end[1] ? 2 : 0);
            if (flag == 0) {
                const float delta = (float)((a.target2 - S.rho0sq) * s_scale);
                // FP32 grid: the first point with F >= 0
                int first = GRID_POINTS;
                if (tid < GRID_POINTS) {
                    float N, D;
                    grid_nd(SF, exp10f((float)(-BRACKET_DECADES + tid * step)), N, D);
                    if (N - delta >= 0.0f) first = tid;
                }
                for (int o = 16; o > 0; o >>= 1) first = min(first, __shfl_xor_sync(0xffffffffu, first, o));
                if (lane == 0) s_idx[wid] = first;
                __syncthreads();
                int k = GRID_POINTS;
                for (int w = 0; w < NW; ++w) k = min(k, s_idx[w]);
                // the sign change within (t_{k-2}, t_{k+1}), confirmed in FP64
                const double A1 = lo + max(k - 2, 0) * step, B1 = lo + min(k + 1, GRID_POINTS - 1) * step;
                if (wid < 2) {
                    double N, N1;
                    lam_terms_n<double>(S, exp10(wid ? B1 : A1) / rho, N, N1);
                    warp_sum2(N, N1);
                    const double F = N + S.rho0sq - a.target2;
                    if (lane == 0) s_end[2 + wid] = wid ? (F > 0.0) : (F < 0.0);
                }
                __syncthreads();
                if (wid == 0) {
                    const bool cell = s_end[2] && s_end[3];
                    double A0 = cell ? A1 : lo, B0 = cell ? B1 : hi;
                    float tf = (float)(0.5 * (A0 + B0) - lrho), Af0 = (float)(A0 - lrho), Bf0 = (float)(B0 - lrho);
                    for (int it = 0; it < NEWTON32_MAX; ++it) {
                        float N, N1;
                        const float mu = exp10f(tf);
                        lam_terms_n<float>(SF, mu, N, N1);
                        N = warp_sum_t(N);
                        N1 = warp_sum_t(N1);
                        const float tn = newton_step<float>(tf, N - delta, N1 * mu * (float)LN10, Af0, Bf0);
                        const float dt = fabsf(tn - tf);
                        tf = tn;
                        if (dt <= 1e-6f || Bf0 - Af0 <= 1e-6f) break;
                    }
                    double t = lrho + (double)tf;
                    if (!(t > A0 && t < B0)) t = 0.5 * (A0 + B0);
                    for (int it = 0; it < NEWTON_MAX; ++it) {
                        const double mu = exp10(t) / rho;
                        double N, N1;
                        lam_terms_n<double>(S, mu, N, N1);
                        warp_sum2(N, N1);
                        const double tn = newton_step<double>(t, N + S.rho0sq - a.target2, N1 * mu * LN10, A0, B0);
                        const double dt = fabs(tn - t);
                        t = tn;
                        if (dt <= 1e-15 * fmax(1.0, fabs(t)) || B0 - A0 <= 1e-15 * fmax(1.0, fabs(t))) break;
                    }
                    if (lane == 0) s_t = t;
                }
            } else if (tid == 0) {
                s_t = flag == 1 ? lo : hi;
            }
            if (tid == 0) {
                s_flag = flag;
                s_lam = exp10(s_t);
            }
            __syncthreads();
        }
        lam = s_lam;
    }
    const double mu = lam / rho;

    // ---------------------------------------------- 5. z = R^-1 (C + mu (I - C))^-1 h
    // (G_A + lam G_L = R^T (C + mu (I - C)) R and g = R^T h)
    for (int e = tid; e < K * K; e += ST) {
        const int i = e / K, j = e - (e / K) * K;
        if (j >= i) AT(Um, i, j) = (1.0 - mu) * AT(Cm, i, j) + (i == j ? mu : 0.0);
    }
    __syncthreads();
    double *invs = gh;  // 1 / diagonal of the Cholesky factor of C + mu (I - C)
    chol_upper(Um, lds, K, invs, &s_fail);
    if (wid == 0) {
        double x0 = lane < K ? hv[lane] : 0.0, x1 = lane + 32 < K ? hv[lane + 32] : 0.0;
        warp_trsv(Um, lds, invs, x0, x1, K, true);   // Rs^T w = h
        warp_trsv(Um, lds, invs, x0, x1, K, false);  // Rs y = w
        warp_trsv(Rm, lds, invd, x0, x1, K, false);  // R z = y
        const bool bad = (lane < K && !isfinite(x0)) || (lane + 32 < K && !isfinite(x1));
        if (lane < K) z[lane] = gh[lane] = x0;
        if (lane + 32 < K) z[lane + 32] = gh[lane + 32] = x1;
        if (__any_sync(0xffffffffu, bad) || s_fail) {
            if (lane == 0) atomicOr(a.err, 2);
        }
        if (lane == 0) {
            a.lam[b] = lam;
            a.flag[b] = s_flag;
        }
    }
    if (a.Y) {  // Y = R^-1 X for the next call: rows from the last on, one barrier each
        __syncthreads();
        for (int i = K - 1; i >= 0; --i) {
            for (int j = tid; j < K; j += ST) AT(Xm, i, j) *= invd[i];
            __syncthreads();
            for (int e = tid; e < i * K; e += ST) {
                const int k = e / K, j = e - k * K;
                AT(Xm, k, j) -= AT(Rm, k, i) * AT(Xm, i, j);
            }
            __syncthreads();
        }
        double *Yg = a.Y + (long long)b * ld * ld;
        for (int e = tid; e < K * K; e += ST) {
            const int i = e / K, j = e - i * K;
            Yg[i * ld + j] = AT(Xm, i, j);
        }
        if (tid == 0) {
            a.Yrho[b] = rho;
            a.nY[b] = K;
        }
    }
    }  // !bordered
    if (!a.proj) return;

    // ---------------------------------------------- 6. proj = Mg^-1 ((G_A + lam G_L) z - g)
    // by the inverse Cholesky factor of Mg: matrix-vector products instead of two triangular
    // solves (each a chain of K dependent FP64 steps); a new vector adds one row
    double *Li = a.Linv + (long long)b * ld * ld, *zs = gh, *cv = theta, *lv = c2;
    const double *Mg = a.Mg + (long long)b * ld * ld;
    const int n0 = a.nL[b];
    for (int e = tid; e < K * K; e += ST) {
        const int i = e / K, j = e - (e / K) * K;
        AT(Tm, i, j) = (j <= i && i < n0) ? Li[i * ld + j] : 0.0;
    }
    __syncthreads();
    for (int r = n0; r < K; ++r) {  // Linv of [L 0; l^T d]: the row [-(l^T Linv) / d, 1 / d], l = Linv Mg[:, r]
        row_sums(r, r, bpart, [&](int i, int k) { return k <= i ? AT(Tm, i, k) * Mg[k * ld + r] : 0.0; }, [&](int i, double t) { lv[i] = t; });
        row_sums(r, r, bpart, [&](int i, int k) { return k >= i ? AT(Tm, k, i) * lv[k] : 0.0; }, [&](int i, double t) { cv[i] = t; });
        if (wid == 0) {
            double t = 0.0;
            for (int k = lane; k < r; k += 32) t += lv[k] * lv[k];
            t = warp_sum(t);
            const double id = rsqrt(fmax(Mg[r * ld + r] - t, 1e-300));
            for (int k = lane; k < r; k += 32) Li[r * ld + k] = AT(Tm, r, k) = -cv[k] * id;
            if (lane == 0) Li[r * ld + r] = AT(Tm, r, r) = id;
        }
        __syncthreads();
    }
    row_sums2(K, K, bpart,
              [&](int i, int k, double &x, double &y) {  // (the Grams are stored symmetric)
                  x += GA[k * ld + i] * zs[k];
                  y += GL[k * ld + i] * zs[k];
              },
              [&](int i, double x, double y) { cv[i] = x + lam * y - g[i]; });
    row_sums(K, K, bpart, [&](int i, int k) { return k <= i ? AT(Tm, i, k) * cv[k] : 0.0; }, [&](int i, double t) { lv[i] = t; });
    row_sums(K, K, bpart, [&](int i, int k) { return k >= i ? AT(Tm, k, i) * lv[k] : 0.0; }, [&](int i, double t) { zs[i] = t; });
    for (int i = tid; i < K; i += ST) a.proj[(long long)b * ld + i] = zs[i];
    if (tid == 0) a.nL[b] = K;
#undef AT
#undef AF
}

static size_t small_smem(int ld) {
    const size_t lds = (size_t)((ld + 1) | 1);
    return sizeof(double) * (6 * lds * lds + (7 + BE_NV) * lds + BE_PART);
}

mof_status prepare_small_solve(int ld) {
    // the limit only ever grows: smaller problems launched later still fit (set
    // from the first call on: static and dynamic shared memory together exceed
    // the default 48 KB before the dynamic part alone does)
    static std::atomic<size_t> configured{0};
    const size_t smem = small_smem(ld);
    size_t cur = configured.load();
    while (smem > cur) {
        MOF_CUDA(cudaFuncSetAttribute(k_small_solve, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        if (configured.compare_exchange_weak(cur, smem)) break;
    }
    return MOF_OK;
}

mof_status launch_small_solve(const SmallArgs &a, cudaStream_t st) {
    // (DP and fixed lambda leave the eigenvectors unformed)
    if (a.Y && a.rule != MOF_RULE_GCV) return fail(MOF_EINVAL, "the small solve keeps eigenvectors between calls for GCV only");
    static const GcvGrid grid = [] {
        GcvGrid g;
        for (int i = 0; i < GRID_POINTS; ++i) g.v[i] = std::pow(10.0, -BRACKET_DECADES + i * (2.0 * BRACKET_DECADES / (GRID_POINTS - 1)));
        return g;
    }();
    const size_t smem = small_smem(a.ld);
    ::mof::count_launch(), k_small_solve<<<a.B, ST, smem, st>>>(a, grid);
    MOF_LAUNCH_CHECK();
    return MOF_OK;
}

}  // namespace mof

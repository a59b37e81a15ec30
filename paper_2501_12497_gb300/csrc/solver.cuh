// Internal interfaces of the Krylov layer and the solver (krylov.cu,
// small.cu, solver.cu).
#pragma once

#include "common.cuh"

namespace mof {

// ------------------------------------------------------ per-problem scratch
// Small buffers of the stand-alone operator entry points, allocated on first
// use and kept until mof_problem_destroy.
enum ScratchKind { SCR_IMAGE = 0, SCR_RADIUS = 1, SCR_DEST = 2, SCR_FLOWROWS = 3, SCR_COUNT = 4 };
mof_status apply_scratch(mof_problem *p, ScratchKind kind, void **out);
void free_workspace(mof_problem *p);

// ------------------------------------------------------------ Krylov bases
template <typename real>
struct BasisRef {
    real *V;          // [B][Kmax][N]
    long long N;      // vector length
    int Kmax;
    int B;            // number of independent problems
    const int *K;     // device [B]: current basis size
    const int *act;   // device [B] or null: problems with act[b] == 0 are skipped
};

// Up to three right-hand vectors of one batched multi-dot.
template <typename real>
struct DotVecs {
    const real *x[3];
    long long stride[3];  // between problems
};
// Output addressing of one dot result i (i < K[b]) of problem b:
//   out[b*bstride + i*istride + col*jstride], col = K[b]-1 if last_col else 0.
struct DotOut {
    double *out;
    long long bstride;
    int istride;
    int jstride;
    int last_col;
    double sign;
};
struct DotOuts {
    DotOut o[3];
};

// What a Golub-Kahan half-step starts from (k_gk_dots): a (front 0), or s and the velocity gradients
// ux, uy (fronts 1 and 2, s scaled in place by inv when given); coef, prev: the recurrence term
// (prev null: none); x receives the vector.
template <typename real>
struct GkFront {
    const real *a;
    real *s;
    long long astride;  // of a or s
    const real *ux, *uy;
    long long fstride;
    const real *inv;
    const double *coef;
    const real *prev;
    long long pstride;
    real *x;
    long long xstride;
};

long long krylov_chunks(long long N);
// doubles of Krylov::partial needed per problem of length N and basis capacity Kmax
long long krylov_partial_doubles(long long N, int Kmax);

template <typename real>
struct Krylov {
    double *partial = nullptr;  // scratch [B][chunks][Kmax] (sized by the owner: krylov_partial_doubles)
    int *err = nullptr;         // device error word (|= 4: a bounded wait ran out), may be null
    double *aux = nullptr;      // scratch [2][B] of append (slot, 1/||x||), sized by the owner
    // out[b][j] = sign * <V[b][j], x[b]>, j < K[b]
    void dots(const BasisRef<real> &B, const real *x, long long xstride, double *out, long long ostride, double sign,
              cudaStream_t st) const;
    // dots of every basis vector with nv (1..3) vectors in one pass over V; exact: error-free
    // accumulation of FP32 products (for Grams whose projected residual cancels)
    void multidot(const BasisRef<real> &B, int nv, const DotVecs<real> &xs, const DotOuts &outs, cudaStream_t st,
                  bool exact = false) const;
    // out[b] = sum_j V[b][j] c[b][j]
    void combine(const BasisRef<real> &B, const double *c, long long cstride, real *out, long long ostride,
                 cudaStream_t st) const;
    // out[b] = sum_j V[b][j] c[b][j] - x[b]; optionally ||out[b]||^2 -> nrm2_out[b]
    void combine_minus(const BasisRef<real> &B, const double *c, long long cstride, const real *x, long long xstride,
                       real *out, long long ostride, double *nrm2_out, cudaStream_t st) const;
    // out[b] = x[b] - sum_j V[b][j] c[b][j]; optionally ||out[b]||^2 -> nrm2_out[b]
    void subtract(const BasisRef<real> &B, const double *c, long long cstride, const real *x, long long xstride, real *out,
                  long long ostride, double *nrm2_out, cudaStream_t st) const;
    void norm2(const real *x, long long N, long long xstride, int nb, double *out, cudaStream_t st,
               bool exact = false) const;
    // One Golub-Kahan half-step: x from the front, x - V V^T x, its norm (||x||^2 in nrm2_out,
    // ||x|| in sq1 / sq2, which may be null, for problems still growing) and the append (as
    // append_parts). scaled: the new vector is normalised here; else it stays x' until the next
    // half-step's front scales it by inv = aux[B..2B) (as real). done: [B] ints, zero between calls.
    void gk_half_step(const BasisRef<real> &B, int *Kmut, int front, const GkFront<real> &f, double *coef, double *nrm2_out,
                      const double *scale, double tol, int *grow, double *sq1, double *sq2, int *done, bool scaled,
                      cudaStream_t st) const;
    // x[b] <- (I - V V^T)^2 x[b] (classical Gram-Schmidt twice; coef [B][Kmax] scratch), ||x||^2 -> nrm2_out,
    // with the first projection's coefficients V^T x supplied by the caller from an exact identity
    // (c1 [B][Kmax]), so that only the second projection streams V for its dot products
    void reorth_second(const BasisRef<real> &B, real *x, long long xstride, const double *c1, double *coef,
                       double *nrm2_out, cudaStream_t st) const;
    // x[b] <- x[b] - V[b] c[b] and out[b] = V[b]^T x[b] in one pass over V (false: not
    // applicable to this layout, nothing enqueued)
    // kcap (> 0): a bound on every K[b] known to the caller, which sizes the pass's shared-memory
    // tile (a larger K[b] sets bit 8 of err)
    // nparts (may be null): also the chunk partials of ||x'[b]||^2, after the dot partials in
    // partial (at partial + B.B * nparts * Kmax), their number per problem in *nparts
    bool sub_dot(const BasisRef<real> &B, const double *c, long long cstride, real *x, long long xstride, double *out,
                 cudaStream_t st, int kcap = 0, int *nparts = nullptr) const;
    // append with ||x||^2 summed from the nparts partials of the preceding update (written to
    // nrm2_out), and sqrt(||x||^2) written to sq1 / sq2 (may be null) for problems still growing
    // (parts: where the partials are, default the start of partial)
    void append_parts(const BasisRef<real> &B, int *Kmut, const real *x, long long xstride, int nparts, double *nrm2_out,
                      const double *scale, double tol, int *grow, int *appended, real *stage, double *sq1, double *sq2,
                      cudaStream_t st, const double *parts = nullptr) const;
    // V[b][K[b]] = x[b]/||x[b]||, K[b]++ unless ||x[b]|| <= tol*scale[b] (then grow[b] = 0);
    // scale may be null (only ||x|| > 0 required); stage[b] (may be null) receives the new vector
    void append(const BasisRef<real> &B, int *Kmut, const real *x, long long xstride, const double *nrm2,
                const double *scale, double tol, int *grow, int *appended, real *stage, cudaStream_t st) const;
};

// Solve-OF (p = q = 2) GKS step. launch_of_resid_lap: the residual r at s and its graph
// Laplacian q. launch_of_proj_gram_pass, after the projection coefficients d: one pass over the
// basis forming x' = r - V d (into the slot behind the basis) with the dot products that give the
// new vector's Gram columns, then the append decision and the new columns of G_A, G_L, g and Mg.
// launch_of_combine: s = V z, scaling a vector appended since the last call to x' / ||x'||.
// partial: [B][3 Kmax + 4][of_pass_parts] doubles; res: [B][3 Kmax + 4]; aux: 2 B doubles (the slot and
// scale between an append and the next combine); done: [B] ints, zero between calls.
long long of_pass_parts(long long ns, int pairs);
int of_pass_stride(int Kmax);
template <typename real> bool of_pass_applicable(long long ns, const void *V, const void *x);
template <typename real>
mof_status launch_of_resid_lap(int nb, int pairs, int nx, int ny, const real *ux, const real *uy, const real *AtB, const real *s,
                               const double *gam, real *r, real *q, const int *act, cudaStream_t st);
template <typename real>
mof_status launch_of_proj_gram_pass(const BasisRef<real> &B, int *Kmut, long long ns, int pairs, const double *d, const real *x, const real *q,
                                    const real *AtB, const real *ux, const real *uy, double *partial, double *res, int *err,
                                    int kcap, const double *scale, double tol, int *grow, double *GA, double *GL, double *g,
                                    double *Mg, double *nrm2_out, int *appended, double *aux, int *done, cudaStream_t st);
template <typename real>
mof_status launch_of_combine(const BasisRef<real> &B, const double *z, double *aux, real *out, cudaStream_t st);

// Bound of the device waits on tile copies for the current device (polls; < 0: the
// default); used by mof_debug_set_wait_limit.
mof_status set_wait_polls(long long polls);

// ------------------------------------------------------ small FP64 solver
// One projected problem per block: min ||A V z - b||^2 + lam ||L V z||^2
// given G_A = (AV)^T(AV), G_L = (LV)^T(LV), g = (AV)^T b, bb = ||b||^2.
struct SmallArgs {
    const double *GA;      // [B][ld][ld]
    const double *GL;      // [B][ld][ld]
    const double *g;       // [B][ld]
    const double *bb;      // [B]
    const int *K;          // [B] problem dimension
    const int *active;     // [B] (null = all active); inactive -> z = 0, lam = 0
    int ld;                // leading dimension (Kmax)
    int B;
    int rule;              // MOF_RULE_*
    double target2;        // DP: (eta delta)^2
    double lam_fixed;
    double *lam;           // [B] out
    double *z;             // [B][ld] out
    int *flag;             // [B] out: DP flag
    int *err;              // error word (|= 1: factorisation failed, 2: non-finite)
    // Projection of the residual at z onto the stored basis (null: none). With r the residual of
    // the normal equations at V z, V^T r = (G_A + lam G_L) z - g exactly, so the coefficients
    // proj = Mg^-1 V^T r of its orthogonal projection need no pass over V. Mg [B][ld][ld] is the
    // basis's Euclidean Gram, Linv the inverse of its Cholesky factor over the first nL[b]
    // vectors, which the call brings up to K[b].
    const double *Mg;
    double *Linv;
    int *nL;
    double *proj;          // [B][ld] out
    // State between the calls of one basis that grows by at most a vector per call while its Grams
    // stay as they are (null: none): generalised eigenvectors Y [B][ld][ld], their eigenvalues Yd,
    // Yh = Y^T g, the scaling Yrho and their number nY (zero before the first call). GCV only.
    double *Y, *Yd, *Yh, *Yrho;
    int *nY;
};
mof_status launch_small_solve(const SmallArgs &a, cudaStream_t st);
// Raise the kernel's dynamic shared-memory limit for leading dimension ld
// (done before any graph capture).
mof_status prepare_small_solve(int ld);

}  // namespace mof

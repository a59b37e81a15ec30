// K1 ray-driven Joseph projector b = H u and K2 pixel-driven exact transpose
// u = H^T b (Sec. 2.1: H = blockdiag(H^1..H^nt), 2D parallel beam).
//
// Both evaluate the same matrix entry
//     a(theta, k; i, j) = (h/mu) * max(0, 1 - |sigma_k - p_ij| / (mu h)),
//     p_ij = x_i cos(theta) + y_j sin(theta),  mu = max(|cos|, |sin|),
// K1 from the ray side (march over the axis the ray is least inclined to,
// two linear-interpolation taps per step, weight h/mu), K2 from the pixel
// side (the <= 2 bins within mu*h of p_ij), so <H u, b> = <u, H^T b> holds to
// rounding.
//
// Fan beam (flat detector, the geometry of the paper's experiments, Sec. 5.1):
// every ray is the line from the source through its bin, integrated by the
// same Joseph rule with its own direction (k_project_fan); the transpose
// (k_backproject_fan) visits, per pixel and view, the bins whose rays can
// cross the pixel's two Joseph segments and re-evaluates the forward entry.
#include "common.cuh"

#include <algorithm>

namespace mof {

// ------------------------------------------------------------------ helpers
constexpr float FLOOR_MAGIC = 12582912.0f;      // 1.5 2^23: x + FLOOR_MAGIC rounded down is floor(x) + FLOOR_MAGIC
constexpr int FLOOR_BITS = 0x4B400000;          // its bit pattern: an integer n adds n to it
constexpr float INV32 = 2.3283064365386963e-10f;  // 2^-32

// floor and fraction of both values: the bits of floor + FLOOR_MAGIC in n0, n1
__device__ __forceinline__ F2 floor2(F2 f, int &n0, int &n1) {
    const F2 t = add2_rd(f, both(FLOOR_MAGIC));
    float t0, t1;
    unpack2(t, t0, t1);
    n0 = __float_as_int(t0);
    n1 = __float_as_int(t1);
    return sub2(f, sub2(t, both(FLOOR_MAGIC)));
}

// v as a float, within 2^-23 of it (a 64-bit conversion holds the FP64 pipe)
__device__ __forceinline__ float near_float(long long v) {
    const unsigned long long a = v < 0 ? -(unsigned long long)v : (unsigned long long)v;
    const float f = fmaf((float)(unsigned)(a >> 32), 4294967296.0f, (float)(unsigned)a);
    return v < 0 ? -f : f;
}

// --------------------------------------------------------------- transpose
// uT[t][x][y] = u[t][y][x], 32x32 tiles through shared memory.
template <typename real>
__global__ void k_transpose(const real *__restrict__ u, real *__restrict__ uT, int nx, int ny) {
    __shared__ real tile[32][33];
    const long long off = (long long)blockIdx.z * nx * ny;
    const int x0 = blockIdx.x * 32, y0 = blockIdx.y * 32;
    for (int dy = threadIdx.y; dy < 32; dy += blockDim.y) {
        const int x = x0 + threadIdx.x, y = y0 + dy;
        if (x < nx && y < ny) tile[dy][threadIdx.x] = u[off + (long long)y * nx + x];
    }
    __syncthreads();
    for (int dx = threadIdx.y; dx < 32; dx += blockDim.y) {
        const int y = y0 + threadIdx.x, x = x0 + dx;
        if (x < nx && y < ny) uT[off + (long long)x * ny + y] = tile[threadIdx.x][dx];
    }
}

// -------------------------------------------------------------- K1 project
// FP32: one lane per ray, the 32 rays of a warp at the same step j, so that every load of
// the warp falls into one row of the frame (of the transposed frame for steep rays).
// The crossing f(j) = f0 + j df runs in fixed point (2^-40 pixels, 64-bit integers) from block
// to block of MARCH steps; within a block it is f = fc + (e - MARCH / 2) df in FP32 about the
// block's middle, fc in [0, 1), so it is exact to 2^-22 pixels. The floor comes from an
// addition that rounds down to the integers (1.5 2^23): one FMA and three additions a step, no
// conversion and no integer arithmetic but the address.
// A block in which every lane's two taps lie inside the row is taken without bounds checks;
// only the blocks where a ray of the warp enters or leaves the frame test each tap.
// The sums of the blocks are compensated (Kahan): a ray's rounding stays at a few units of
// FP32 however long it is.
// What bounds it: the two 4-byte loads a step, each of which touches two to three 128-byte
// lines of L1 (32 adjacent rays cross 32 to 46 pixels of a row; 65 % of the L1 data pipe), and
// instruction issue (63 %, 13 instructions a step). 1024x1024x64, 90 views: 3.02 ms against 7.21
// for the march with a conversion pair per coordinate and per-ray step ranges, whose lanes read
// different rows; 256x256x32, 30 views: 62 against 130 us. Fan beam 256x256x32: 68 against 119 us.
// Few rays leave the chip idle and the march's load latency exposed, so the warps of a CTA
// share rays of small problems: each takes a segment of the steps (ProjSplit).
constexpr int MARCH = 8;  // steps per block
constexpr int PW = 8;     // warps per CTA
// The warps of a CTA as (32-bin groups) x (adjacent views) x (segments of the steps), all
// powers of two with product PW. Adjacent views cross the same rows together, so they share
// L1 lines.
struct ProjSplit {
    int views, segs, bins;  // bins in groups of 32
};

// The sum of one ray's taps, as the compensated pair (sum, correction to subtract). img: the
// frame in the march's orientation; F, D: f0 and df in 2^-40 pixels, |f0| < 2^22 pixels,
// |df| <= 1; off lanes (on = false) take part in the warp's votes only; segment seg of nseg of
// the warp's steps. All lanes call. INF: a sum that is not finite is that of plain additions, so that
// an infinity stays one (its correction would be NaN).
constexpr float FLT_LARGEST = 3.402823466e+38f;
template <bool INF>
__device__ __forceinline__ float2 ray_march(const float *__restrict__ img, int nfast, int nstep, long long F, long long D,
                                            bool on, int seg, int nseg) {
    const unsigned lanes = __ballot_sync(0xffffffffu, on);
    if (!lanes) return make_float2(0.f, 0.f);
    const int src = __ffs(lanes) - 1;  // off lanes follow a ray that is marched
    const long long Fs = __shfl_sync(0xffffffffu, F, src), Ds = __shfl_sync(0xffffffffu, D, src);
    if (!on) {
        F = Fs;
        D = Ds;
    }
    // steps whose crossing can lie in (-1, nfast), with two steps of margin each side (the
    // checked taps beyond add nothing), over the warp's rays. The distances to both edges are exact in
    // fixed point, so what is rounded is their quotients: a few 2^-24 of a step number of at most
    // 4096 (f0 in FP32 would be off by up to 2e-4 pixels: hundreds of steps of a ray along the edge)
    int jlo = 0, jhi = nstep - 1;
    {
        const long long to_lo = -(1LL << 40) - F, to_hi = ((long long)nfast << 40) - F;
        if (D != 0) {
            const float d = (float)D, ja = near_float(to_lo) / d, jb = near_float(to_hi) / d;
            const float lo = fmaxf(fminf(ja, jb), -1.0f), hi = fminf(fmaxf(ja, jb), (float)nstep);
            jlo = max(0, (int)floorf(lo) - 2);
            jhi = min(nstep - 1, (int)ceilf(hi) + 2);
        } else if (!(to_lo < 0 && to_hi > 0)) {
            jhi = -1;
        }
    }
    jlo = __reduce_min_sync(0xffffffffu, jlo);
    jhi = __reduce_max_sync(0xffffffffu, jhi);
    if (nseg > 1) {  // whole blocks
        const int nblk = (jhi - jlo + MARCH) / MARCH;
        const int b0 = seg * nblk / nseg, b1 = (seg + 1) * nblk / nseg;
        jhi = min(jhi, jlo + b1 * MARCH - 1);
        jlo += b0 * MARCH;
    }
    float acc = 0.f, cmp = 0.f, raw = 0.f;
    const unsigned last = (unsigned)(nfast - 1);
    const float df = (float)D * 9.094947017729282e-13f;
    F += (jlo + MARCH / 2) * D;  // the crossing at the middle of the block
    const F2 df2 = both(df), one = both(1.0f);
    for (int j = jlo; j <= jhi; j += MARCH) {
        const int ic = (int)(F >> 40);
        const float fc = (float)(unsigned)((unsigned long long)F >> 8) * INV32;
        const F2 fc2 = both(fc);
        int n[MARCH];
        F2 w[MARCH / 2];
#pragma unroll
        for (int e = 0; e < MARCH; e += 2)
            w[e / 2] = floor2(fma2(pack2((float)(e - MARCH / 2), (float)(e + 1 - MARCH / 2)), df2, fc2), n[e], n[e + 1]);
        const int c0 = ic - FLOOR_BITS;
        const bool inside = j + MARCH <= nstep && (unsigned)(n[0] + c0) < last && (unsigned)(n[MARCH - 1] + c0) < last;
        float a[MARCH], c[MARCH];
        if (__all_sync(0xffffffffu, inside)) {
            const unsigned long long base = (unsigned long long)(uintptr_t)(img + (j * nfast + ic)) - 4ull * (unsigned)FLOOR_BITS;
#pragma unroll
            for (int e = 0; e < MARCH; ++e) {
                const float *t = reinterpret_cast<const float *>((uintptr_t)(base + 4ull * ((unsigned)n[e] + (unsigned)(e * nfast))));
                a[e] = ldg(t);
                c[e] = ldg(t + 1);
            }
        } else {
#pragma unroll
            for (int e = 0; e < MARCH; ++e) {
                const int i0 = n[e] + c0;
                const float *t = img + ((j + e) * nfast + i0);
                const bool row = j + e <= jhi;
                a[e] = (row && (unsigned)i0 <= last) ? ldg(t) : 0.f;
                c[e] = (row && (unsigned)(i0 + 1) <= last) ? ldg(t + 1) : 0.f;
            }
        }
        F2 s2 = both(0.f);
#pragma unroll
        for (int e = 0; e < MARCH; e += 2)
            s2 = fma2(w[e / 2], pack2(c[e], c[e + 1]), fma2(sub2(one, w[e / 2]), pack2(a[e], a[e + 1]), s2));
        float s, so;
        unpack2(s2, s, so);
        s += so;
        if (INF) raw += s;
        F += MARCH * D;
        const float y = __fsub_rn(s, cmp), t = __fadd_rn(acc, y);
        cmp = __fsub_rn(__fsub_rn(t, acc), y);
        acc = t;
    }
    if (INF && !(fabsf(acc) <= FLT_LARGEST)) return make_float2(raw, 0.f);
    return make_float2(acc, cmp);
}

// The segments' sums of the CTA's rays, added in segment order by the first segment's warps
// (true there; the others are done). All threads call.
__device__ __forceinline__ bool join_segments(float2 &r, const ProjSplit &sp) {
    __shared__ float2 part[32 * PW];
    if (sp.segs == 1) return true;
    part[threadIdx.x] = r;
    __syncthreads();
    const int w = threadIdx.x >> 5, per = PW / sp.segs;
    if (w >= per) return false;
    for (int g = 1; g < sp.segs; ++g) {
        const float2 o = part[threadIdx.x + g * per * 32];
        const float y = __fsub_rn(o.x, __fadd_rn(r.y, o.y)), t = __fadd_rn(r.x, y);
        r.y = fabsf(t) <= FLT_LARGEST ? __fsub_rn(__fsub_rn(t, r.x), y) : 0.f;
        r.x = t;
    }
    return true;
}

// (sum - correction) * w with w = wh + wl, rounded once
__device__ __forceinline__ float scale_sum(float2 a, float wh, float wl) {
    const float p = __fmul_rn(a.x, wh);
    const float e = fmaf(-a.y, wh, fmaf(a.x, wl, __fmaf_rn(a.x, wh, -p)));
    return isfinite(p) ? p + e : p;
}

__global__ void __launch_bounds__(32 * PW) k_project32(const float *__restrict__ u, const float *__restrict__ uT,
                                                       float *__restrict__ b, const AngleParams *__restrict__ ang, int nang,
                                                       int nx, int ny, int nb, ProjSplit sp) {
    const int w = threadIdx.x >> 5, per = PW / sp.segs, seg = w / per, wr = w - seg * per;
    const int a = blockIdx.y * sp.views + wr % sp.views;
    const int k = (blockIdx.x * sp.bins + wr / sp.views) * 32 + (threadIdx.x & 31);
    const AngleParams &P = ang[min(a, nang - 1)];
    const int kk = min(k, nb - 1);
    long long F;
    if (!P.wide) {
        F = P.f0cQ + kk * P.f0kQ;
    } else {  // rays so far apart that 2^-40 pixels do not fit: the ray's own f0, held off the frame
        const double f0 = fmin(fmax((double)kk * P.f0_k + P.f0_c, -F0_LIMIT), F0_LIMIT);
        F = __double2ll_rn(f0 * 1099511627776.0);
    }
    const long long ns = (long long)nx * ny;
    const int rows = P.rows;
    const bool on = a < nang && k < nb;
    float2 r = ray_march<false>((rows ? u : uT) + P.frame * ns, rows ? nx : ny, rows ? ny : nx, F, P.dfQ, on, seg, sp.segs);
    if (join_segments(r, sp) && on) b[(long long)a * nb + k] = scale_sum(r, P.wstep, P.wstep_lo);
}

// FP64 coordinates in 64-bit fixed point, units of 2^-51: the integer part is a shift, and the
// fraction becomes a double in [1, 2) by its bits. (An FP64 instruction holds its pipe for 64 clocks
// a warp; floor and the conversions are such instructions too.) |coordinate| < FIX64_LIMIT.
constexpr int FIX64 = 51;
__device__ __forceinline__ long long fix64(double f) { return __double2ll_rn(f * 2251799813685248.0); }
__device__ __forceinline__ double one_plus_frac(long long F) {
    return __longlong_as_double(((F << 1) & 0x000fffffffffffffLL) | 0x3ff0000000000000LL);
}

// FP64: one ray per lane (angle a = blockIdx.y, bin k); the four warps of a CTA take a quarter of the
// steps of the same 32 rays each. The coordinate starts from its FP64 value every 32 steps and the
// step has 32 bits more, so the steps round less than the FP64 sums they replace. Bound by the FP64 pipe, four
// instructions a step. With the transposition before it: 64 x 64 x 8, 16 views of 64 bins: 19 us against
// 31 with the whole ray in one thread and floor, conversions and weights in FP64 (eight instructions a
// step, 256 warps); 256 x 256 x 8, 30 views: 177 against 347 us.
constexpr int P64_W = 4;
__global__ void __launch_bounds__(32 * P64_W) k_project64_fix(const double *__restrict__ u, const double *__restrict__ uT,
                                                              double *__restrict__ b, const AngleParams *__restrict__ ang, int nx,
                                                              int ny, int nb) {
    __shared__ double part[P64_W][32];
    const int a = blockIdx.y, lane = threadIdx.x & 31, w = threadIdx.x >> 5, k = blockIdx.x * 32 + lane;
    const AngleParams &P = ang[a];
    const int rows = P.rows, nfast = rows ? nx : ny, nstep = rows ? ny : nx;
    const double *img = (rows ? u : uT) + P.frame * ((long long)nx * ny);
    const double df = P.df, f0 = (double)min(k, nb - 1) * P.f0_k + P.f0_c;
    // the steps that can touch the frame, a little widened (each tap is checked anyway): FP32 with its
    // rounding errors as a margin
    const float ff = (float)f0, d = (float)df, nf = (float)nfast;
    int jlo = 0, jhi = nstep - 1;
    if (fabsf(d) > 1e-30f) {
        const float ja = (-1.0f - ff) / d, jb = (nf - ff) / d;
        const float err = 1.0f + 4e-7f * ((fabsf(ff) + nf) / fabsf(d));
        jlo = (int)floorf(fminf(fmaxf(fminf(ja, jb) - err, 0.0f), (float)nstep));
        jhi = (int)ceilf(fmaxf(fminf(fmaxf(ja, jb) + err, (float)(nstep - 1)), -1.0f));
    } else if (!(f0 > -1.0 && f0 < (double)nfast)) {
        jhi = -1;
    }
    if (!(fabsf(ff) < 1048576.0f)) jhi = -1;  // no step of at most one pixel leads from there to the frame
    const int per = (nstep + P64_W - 1) / P64_W;
    jlo = max(jlo, w * per);
    jhi = min(jhi, min((w + 1) * per, nstep) - 1);
    if (k >= nb) jhi = -1;
    const long long D = P.df51;
    const unsigned Dl = P.df51_lo;
    double acc = 0;
    for (int j0 = jlo; j0 <= jhi; j0 += 32) {
        long long F = fix64(fma((double)j0, df, f0));
        unsigned Fl = 0;
        const int j1 = min(j0 + 31, jhi);
        const double *row = img + (long long)j0 * nfast;
#pragma unroll 4
        for (int j = j0; j <= j1; ++j) {
            const int i0 = (int)(F >> FIX64);
            const double o = one_plus_frac(F);
            const double v0 = (unsigned)i0 < (unsigned)nfast ? ldg(row + i0) : 0.0;
            const double v1 = (unsigned)(i0 + 1) < (unsigned)nfast ? ldg(row + i0 + 1) : 0.0;
            acc = fma(2.0 - o, v0, acc);
            acc = fma(o - 1.0, v1, acc);
            Fl += Dl;
            F += D + (Fl < Dl);
            row += nfast;
        }
    }
    part[w][lane] = acc;
    __syncthreads();
    if (w == 0 && k < nb) b[(long long)a * nb + k] = ((part[0][lane] + part[1][lane]) + (part[2][lane] + part[3][lane])) * P.wstep_d;
}

// The same for frames, detectors or distances beyond FIX64_LIMIT: one thread per ray.
__global__ void __launch_bounds__(128) k_project64(const double *__restrict__ u, const double *__restrict__ uT,
                                                   double *__restrict__ b, const AngleParams *__restrict__ ang, int nx,
                                                   int ny, int nb) {
    const int a = blockIdx.y;
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nb) return;
    const AngleParams &P = ang[a];
    const long long ns = (long long)nx * ny;
    const int rows = P.rows;
    const double *img = rows ? u + P.frame * ns : uT + P.frame * ns;
    const int nfast = rows ? nx : ny, nstep = rows ? ny : nx;
    double acc = 0;
    const double f0 = (double)k * P.f0_k + P.f0_c;  // fractional fast index at step 0
    int jlo = 0, jhi = nstep - 1;
    if (P.df != 0.0) {
        double ja = (-1.0 - f0) / P.df, jb = ((double)nfast - f0) / P.df;
        double lo = fmin(ja, jb), hi = fmax(ja, jb);
        lo = fmax(lo, -1.0);
        hi = fmin(hi, (double)nstep);
        jlo = max(0, (int)floor(lo) - 1);
        jhi = min(nstep - 1, (int)ceil(hi) + 1);
    } else if (!(f0 > -1.0 && f0 < (double)nfast)) {
        jhi = -1;
    }
    for (int j = jlo; j <= jhi; ++j) {
        const double f = fma((double)j, P.df, f0);
        const double fl = floor(f);
        const int i0 = (int)fl;
        const double w1 = f - fl;
        const double *row = img + (long long)j * nfast;
        if (i0 >= 0 && i0 < nfast) acc = fma(1.0 - w1, ldg(row + i0), acc);
        if (i0 + 1 >= 0 && i0 + 1 < nfast) acc = fma(w1, ldg(row + i0 + 1), acc);
    }
    b[(long long)a * nb + k] = acc * P.wstep_d;
}

// ---------------------------------------------------------- K1 fan beam
// FP32: the march of the parallel kernel with each ray's own start and step from the ray
// table; the rays of a warp that step over rows, then those that step over columns (both
// only where a fan straddles 45 degrees).
__global__ void __launch_bounds__(32 * PW) k_project_fan32(const float *__restrict__ u, const float *__restrict__ uT,
                                                           float *__restrict__ b, const FanRay<float> *__restrict__ rays,
                                                           const AngleParams *__restrict__ ang, int nang, int nx, int ny,
                                                           int nb, float h, ProjSplit sp) {
    const int w = threadIdx.x >> 5, per = PW / sp.segs, seg = w / per, wr = w - seg * per;
    const int a = blockIdx.y * sp.views + wr % sp.views, ac = min(a, nang - 1);
    const int k = (blockIdx.x * sp.bins + wr / sp.views) * 32 + (threadIdx.x & 31);
    const bool on = a < nang && k < nb;
    const long long ns = (long long)nx * ny;
    const FanRay<float> R = rays[(long long)ac * nb + min(k, nb - 1)];
    const int rows = (int)(R.f0q & 1);
    const long long F = R.f0q >> 1, D = R.dq, fr = ang[ac].frame * ns;
    float2 r = ray_march<true>(u + fr, nx, ny, F, D, on && rows, seg, sp.segs);
    const float2 rc = ray_march<true>(uT + fr, ny, nx, F, D, on && !rows, seg, sp.segs);
    if (!rows) r = rc;
    if (!join_segments(r, sp) || !on) return;
    // length per step h sqrt(1 + df^2), its rounding kept: r = sqrt(x) + e, e = (x - s^2) / (2 s)
    const float df = (float)D * 9.094947017729282e-13f, dl = (float)(D - __float2ll_rn(df * 1099511627776.0f)) * 9.094947017729282e-13f;
    const float d2 = __fmul_rn(df, df), x = 1.0f + d2;
    const float xl = fmaf(2.0f * df, dl, fmaf(df, df, -d2)) + (d2 - (x - 1.0f));
    const float s = sqrtf(x), sl = (fmaf(-s, s, x) + xl) / (2.0f * s);
    const float wh = h * s, wl = fmaf(h, s, -wh) + h * sl;
    b[(long long)a * nb + k] = scale_sum(r, wh, wl);
}

__global__ void __launch_bounds__(128) k_project_fan64(const double *__restrict__ u, const double *__restrict__ uT,
                                                       double *__restrict__ b, const FanRay<double> *__restrict__ rays,
                                                       const AngleParams *__restrict__ ang, int nx, int ny, int nb) {
    const int a = blockIdx.y;
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nb) return;
    const long long ns = (long long)nx * ny;
    const FanRay<double> R = rays[(long long)a * nb + k];
    const int frame = ang[a].frame;
    double acc = 0;
    const double *img = R.rows ? u + frame * ns : uT + frame * ns;
    const int nfast = R.rows ? nx : ny;
    for (int j = R.jlo; j <= R.jhi; ++j) {
        const double f = fma((double)j, R.df, R.f0), fl = floor(f);
        const int i0 = (int)fl;
        const double w1 = f - fl;
        const double *row = img + (long long)j * nfast;
        if (i0 >= 0 && i0 < nfast) acc = fma(1.0 - w1, ldg(row + i0), acc);
        if (i0 + 1 >= 0 && i0 + 1 < nfast) acc = fma(w1, ldg(row + i0 + 1), acc);
    }
    b[(long long)a * nb + k] = acc * R.wstep;
}

// Segments per ray: doubled while the launch has fewer warps than two rounds of full SMs
// (152 x 64) and a segment keeps four blocks of steps; the other warps of a CTA take up to four
// adjacent views. Measured: 256x256x32 (30 views) 97 us with one segment, 87 with this rule, 89
// with twice the warps; 181x149x9 (23 views) 44 and 26 us; 1024x1024x64 is above the line. One
// view per CTA: 1024x1024x64 3.94 against 3.79 ms for four and 3.81 for eight (all with the
// march before its packed form).
constexpr long long PROJ_WARPS = 2LL * 152 * 64;
constexpr int PROJ_VIEWS = 4;
static ProjSplit proj_split(const mof_problem *p, int nang) {
    const long long warps = (long long)nang * ((p->nb + 31) / 32);
    const int blocks = std::max(p->nx, p->ny) / MARCH;
    ProjSplit sp{1, 1, 1};
    while (sp.segs < PW && warps * sp.segs < PROJ_WARPS && blocks >= 8 * sp.segs) sp.segs *= 2;
    sp.views = std::min(PW / sp.segs, PROJ_VIEWS);
    sp.bins = PW / (sp.segs * sp.views);
    return sp;
}

// the rays of `nang` views from a0 on; b from the first of them on
static void project_views(const mof_problem *p, const float *u, const float *uT, float *b, int a0, int nang, cudaStream_t st) {
    const ProjSplit sp = proj_split(p, nang);
    const dim3 grid((p->nb + 32 * sp.bins - 1) / (32 * sp.bins), (nang + sp.views - 1) / sp.views);
    if (p->fan)
        ::mof::count_launch(), k_project_fan32<<<grid, 32 * PW, 0, st>>>(
            u, uT, b, static_cast<const FanRay<float> *>(p->d_fanray) + (long long)a0 * p->nb, p->d_ang + a0, nang, p->nx,
            p->ny, p->nb, (float)p->h, sp);
    else
        ::mof::count_launch(), k_project32<<<grid, 32 * PW, 0, st>>>(u, uT, b, p->d_ang + a0, nang, p->nx, p->ny, p->nb, sp);
}
static void project_views(const mof_problem *p, const double *u, const double *uT, double *b, int a0, int nang, cudaStream_t st) {
    const dim3 grid((p->nb + 127) / 128, nang);
    if (p->fan)
        ::mof::count_launch(), k_project_fan64<<<grid, 128, 0, st>>>(
            u, uT, b, static_cast<const FanRay<double> *>(p->d_fanray) + (long long)a0 * p->nb, p->d_ang + a0, p->nx, p->ny,
            p->nb);
    else if (p->fix64)
        ::mof::count_launch(), k_project64_fix<<<dim3((p->nb + 31) / 32, nang), 32 * P64_W, 0, st>>>(u, uT, b, p->d_ang + a0, p->nx,
                                                                                                  p->ny, p->nb);
    else
        ::mof::count_launch(), k_project64<<<grid, 128, 0, st>>>(u, uT, b, p->d_ang + a0, p->nx, p->ny, p->nb);
}

template <typename real>
mof_status launch_project(const mof_problem *p, const real *u, real *uT, real *b, cudaStream_t st, bool per_frame) {
    dim3 tb(32, 8), tg((p->nx + 31) / 32, (p->ny + 31) / 32, p->nt);
    if (per_frame && !p->fan) {  // the plain form: frame by frame (the angles' tables hold their frame)
        const long long ns = (long long)p->nx * p->ny;
        for (int t = 0; t < p->nt; ++t) {
            dim3 tg1((p->nx + 31) / 32, (p->ny + 31) / 32, 1);
            ::mof::count_launch(), k_transpose<real><<<tg1, tb, 0, st>>>(u + t * ns, uT + t * ns, p->nx, p->ny);
            project_views(p, u, uT, b + (long long)p->aoff[t] * p->nb, p->aoff[t], p->aoff[t + 1] - p->aoff[t], st);
        }
        MOF_LAUNCH_CHECK();
        return MOF_OK;
    }
    ::mof::count_launch(), k_transpose<real><<<tg, tb, 0, st>>>(u, uT, p->nx, p->ny);
    project_views(p, u, uT, b, 0, p->A, st);
    MOF_LAUNCH_CHECK();
    return MOF_OK;
}

// ---------------------------------------------------------- K2 backproject
// FP64: one thread per pixel (tile 32 x 8 per block), looping over the angles of its frame. Per
// angle the bin coordinate at the tile origin is computed once (shared memory).
constexpr int BP_TX = 32, BP_TY = 8, BP_CHUNK = 64;

// For footprints of at most RT (1, 2) bins each side and coordinates within FIX64_LIMIT: those of the
// tile's pixels in fixed point about its origin, the tent weights 1 - (fr + m) / r and
// 1 - (1 + m - fr) / r by the reciprocal of r, taken as zero (with their bins, whatever they hold)
// where not positive. Six (RT = 1) or ten FP64 instructions a pixel and view, which bound it, against 35
// with divisions. 64 x 64 x 8, 16 views: 19 us against 50; 256 x 256 x 8, 30 views: 183 against 1045 us.
struct Bt64 {
    long long t, a, b;  // coordinate of the tile's first pixel, its steps in x and y in units of 2^-55
    double ir, c1, wf;  // 1 / r, 1 - 1 / r, the footprint's height
};
template <int RT>
__global__ void __launch_bounds__(BP_TX *BP_TY) k_backproject64_fix(const double *__restrict__ b, double *__restrict__ u,
                                                                    const AngleParams *__restrict__ ang,
                                                                    const int *__restrict__ aoff, int nx, int ny, int nb, int t0) {
    __shared__ Bt64 s_v[BP_CHUNK];
    const int t = t0 + blockIdx.z, x0 = blockIdx.x * BP_TX, y0 = blockIdx.y * BP_TY;
    const int di = threadIdx.x, dj = threadIdx.y, x = x0 + di, y = y0 + dj, tid = threadIdx.y * BP_TX + threadIdx.x;
    const int a_begin = aoff[t], a_end = aoff[t + 1];
    const bool on = x < nx && y < ny;
    double acc = 0;
    for (int ac = a_begin; ac < a_end; ac += BP_CHUNK) {
        const int cn = min(BP_CHUNK, a_end - ac);
        __syncthreads();
        if (tid < cn) {
            const AngleParams &P = ang[ac + tid];
            Bt64 &v = s_v[tid];
            v.t = fix64(P.t0 + (double)x0 * P.tA + (double)y0 * P.tB);
            v.a = P.tA55;
            v.b = P.tB55;
            v.ir = P.inv_rfoot_d;
            v.c1 = 1.0 - P.inv_rfoot_d;
            v.wf = P.wfoot_d;
        }
        __syncthreads();
        if (!on) continue;
#pragma unroll 4
        for (int q = 0; q < cn; ++q) {
            const Bt64 &A = s_v[q];
            const double *row = b + (long long)(ac + q) * nb;
            const long long F = A.t + ((di * A.a + dj * A.b) >> 4);
            const int ib = (int)(F >> FIX64);
            const double fr = one_plus_frac(F) - 1.0;
            double w0 = fma(-fr, A.ir, 1.0), w1 = fma(fr, A.ir, A.c1), s = 0.0;
#pragma unroll
            for (int m = 0; m < RT; ++m) {
                const int k0 = ib - m, k1 = ib + 1 + m;
                // (a weight of zero is common: a whole coordinate where r is whole. Positive by the upper half's bits:
                // one comparison, and no weight but zero has them all clear, as fr and 1 / r are multiples of 2^-53)
                const bool p0 = __double2hiint(w0) > 0, p1 = __double2hiint(w1) > 0;
                const double v0 = p0 && (unsigned)k0 < (unsigned)nb ? ldg(row + k0) : 0.0;
                const double v1 = p1 && (unsigned)k1 < (unsigned)nb ? ldg(row + k1) : 0.0;
                s = m ? fma(p0 ? w0 : 0.0, v0, s) : (p0 ? w0 : 0.0) * v0;
                s = fma(p1 ? w1 : 0.0, v1, s);
                w0 -= A.ir;
                w1 -= A.ir;
            }
            acc = fma(A.wf, s, acc);
        }
    }
    if (on) u[(long long)t * nx * ny + (long long)y * nx + x] = acc;
}

// Any footprint and coordinate.

__global__ void __launch_bounds__(BP_TX *BP_TY) k_backproject64(const double *__restrict__ b, double *__restrict__ u,
                                                                const AngleParams *__restrict__ ang,
                                                                const int *__restrict__ aoff, int nx, int ny, int nb, int t0) {
    __shared__ double s_tb[BP_CHUNK];
    const int t = t0 + blockIdx.z;
    const int x0 = blockIdx.x * BP_TX, y0 = blockIdx.y * BP_TY;
    const int di = threadIdx.x, dj = threadIdx.y;
    const int x = x0 + di, y = y0 + dj;
    const int tid = threadIdx.y * BP_TX + threadIdx.x;
    const int a_begin = aoff[t], a_end = aoff[t + 1];
    double acc = 0;
    for (int ac = a_begin; ac < a_end; ac += BP_CHUNK) {
        const int cn = min(BP_CHUNK, a_end - ac);
        __syncthreads();
        if (tid < cn) {
            const AngleParams &P = ang[ac + tid];
            s_tb[tid] = P.t0 + (double)x0 * P.tA + (double)y0 * P.tB;
        }
        __syncthreads();
        if (x < nx && y < ny) {
            for (int q = 0; q < cn; ++q) {
                const double *row = b + (long long)(ac + q) * nb;
                const AngleParams &P = ang[ac + q];
                const double tt = s_tb[q] + (double)di * P.tA + (double)dj * P.tB;
                const double ff = floor(tt);
                const int ib = (int)ff;
                const double fr = tt - ff;
                const double rd = P.rfoot_d, wf = P.wfoot_d;
                for (int m = 0; (double)m < rd; ++m) {
                    const double d0 = fr + m, d1 = 1.0 - fr + m;
                    const int k0 = ib - m, k1 = ib + 1 + m;
                    if (d0 < rd && k0 >= 0 && k0 < nb) acc = fma(wf * (1.0 - d0 / rd), ldg(row + k0), acc);
                    if (d1 < rd && k1 >= 0 && k1 < nb) acc = fma(wf * (1.0 - d1 / rd), ldg(row + k1), acc);
                }
            }
        }
    }
    if (x < nx && y < ny) u[(long long)t * nx * ny + (long long)y * nx + x] = acc;
}

// FP32, footprints of at most 2 RT bins (mu h <= RT db for every view; RT = 1 for a detector
// no finer than the pixels, RT = 2 for one up to twice as fine). A CTA owns a tile of
// 32 x 32 pixels of a frame; per view it stages the bins that the tile's pixels can reach,
// times the footprint height (zero beyond the detector), in shared memory, so that the pixels
// need no bounds checks and adjacent lanes read adjacent words. A thread owns a column of
// eight pixels; the bin coordinate at the column's middle comes from 64-bit fixed point, the
// pixels' from one FMA each about it (exact to 2^-22 bins), the floor by the addition of
// ray_march. The tent weights sat(1 - (fr + m) / r) and sat(1 - (1 + m - fr) / r) are saturating
// FMAs: they vanish by themselves outside the footprint. The sum over the views is compensated
// (Kahan).
// A segment with a non-finite value takes the weights that are zero out of the sum (careful),
// so that the value reaches exactly the pixels whose footprint holds it.
// What bounds it: instruction issue (about 74 %, 17 instructions a pixel and view), with the
// FP32 pipe, which a packed pair occupies twice, and the shared loads close behind. 1024x1024x64,
// 90 views: 3.29 ms against 9.48 for one thread per four pixels of a row with global loads and
// three floors a coordinate; 256x256x32, 30 views: 46 against 130 us. Two columns per thread
// (64 x 32 tiles): 3.31 ms, no gain. Kahan steps every 2 and 4 views: 10 and 15 % faster, but
// 3 and 7 % further from the exact sum.
constexpr int BT_X = 32, BT_Y = 4, BT_E = 8;  // threads, pixels per thread down a column
constexpr int BT_CH = 32;                     // views staged at a time (one lane each sets them up)
struct __align__(16) BtAngle {
    long long t;    // bin coordinate of the tile's first pixel in the segment, units of 2^-FB
    int a, b;       // its steps in x and y, units of 2^-FB
    float df;       // step in y
    float ir, c1;   // 1 / r, 1 - 1 / r
    unsigned seg;   // shared address of the segment
};

__device__ __forceinline__ float lds(unsigned addr) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
    return v;
}

template <int RT, bool CAREFUL>
__device__ __forceinline__ void bt_view(const BtAngle &A, F2 (&acc)[BT_E / 2], F2 (&cmp)[BT_E / 2]) {
    constexpr int FB = 31 - RT;
    const float ir = A.ir, c1 = A.c1;
    const F2 df2 = both(A.df);
    const long long P = A.t + (long long)(int)threadIdx.x * A.a + (long long)(int)(threadIdx.y * BT_E + BT_E / 2) * A.b;
    const F2 fc2 = both((float)((unsigned)P & ((1u << FB) - 1u)) * (1.0f / (float)(1u << FB)));
    const unsigned base = A.seg + 4u * ((unsigned)(int)(P >> FB) - (unsigned)FLOOR_BITS);
#pragma unroll
    for (int e = 0; e < BT_E; e += 2) {
        int n0, n1;
        const F2 fr2 = floor2(fma2(pack2((float)(e - BT_E / 2), (float)(e + 1 - BT_E / 2)), df2, fc2), n0, n1);
        float f0, f1;
        unpack2(fr2, f0, f1);
        const unsigned at0 = base + 4u * (unsigned)n0, at1 = base + 4u * (unsigned)n1;
        F2 tap = both(0.f);
#pragma unroll
        for (int m = 0; m < RT; ++m) {  // bins i - m and i + 1 + m
            const float o0 = m == 0 ? 1.0f : c1, o1 = m == 0 ? c1 : c1 - ir;
            const float w00 = __saturatef(fmaf(-f0, ir, o0)), w10 = __saturatef(fmaf(-f1, ir, o0));
            const float w01 = __saturatef(fmaf(f0, ir, o1)), w11 = __saturatef(fmaf(f1, ir, o1));
            float b00 = lds(at0 + 4 * (RT - 1 - m)), b10 = lds(at1 + 4 * (RT - 1 - m));
            float b01 = lds(at0 + 4 * (RT + m)), b11 = lds(at1 + 4 * (RT + m));
            if (CAREFUL) {  // a bin outside the footprint is no part of the sum
                b00 = w00 > 0.f ? b00 : 0.f;
                b10 = w10 > 0.f ? b10 : 0.f;
                b01 = w01 > 0.f ? b01 : 0.f;
                b11 = w11 > 0.f ? b11 : 0.f;
            }
            const F2 w0 = pack2(w00, w10), w1 = pack2(w01, w11);
            tap = m == 0 ? mul2(w0, pack2(b00, b10)) : fma2(w0, pack2(b00, b10), tap);
            tap = fma2(w1, pack2(b01, b11), tap);
        }
        const F2 y = sub2(tap, cmp[e / 2]), t = add2(acc[e / 2], y);
        cmp[e / 2] = sub2(sub2(t, acc[e / 2]), y);
        acc[e / 2] = t;
    }
}

template <int RT>
__global__ void __launch_bounds__(BT_X *BT_Y) k_backproject_tile(const float *__restrict__ b, float *__restrict__ u,
                                                                 const AngleParams *__restrict__ ang,
                                                                 const int *__restrict__ aoff, int nx, int ny, int nb, int t0) {
    constexpr int W = 64 * RT;  // words of a segment
    constexpr int FB = 31 - RT;
    __shared__ float s_seg[BT_CH][W];
    __shared__ BtAngle s_a[BT_CH];
    __shared__ int2 s_k[BT_CH];  // first and last bin of the segment
    __shared__ float s_w[BT_CH];
    const int t = t0 + blockIdx.z;
    const int x0 = blockIdx.x * BT_X, y0 = blockIdx.y * BT_Y * BT_E;
    const int lane = threadIdx.x, w = threadIdx.y;
    const int a_begin = aoff[t], a_end = aoff[t + 1];
    F2 acc[BT_E / 2], cmp[BT_E / 2];
#pragma unroll
    for (int e = 0; e < BT_E / 2; ++e) acc[e] = cmp[e] = both(0.f);
    for (int ac = a_begin; ac < a_end; ac += BT_CH) {
        const int cn = min(BT_CH, a_end - ac);
        __syncthreads();
        if (w == 0 && lane < cn) {
            const AngleParams &P = ang[ac + lane];
            const long long a = P.tAQ, bb = P.tBQ, tt = P.t0Q + x0 * a + y0 * bb;
            const long long ex = (BT_X - 1) * a, ey = (BT_Y * BT_E - 1) * bb;
            // the segment starts RT bins before the smallest bin coordinate of the tile (one more
            // than the footprint needs: the fixed-point steps may round below it)
            const int k0 = (int)((tt + min(0LL, ex) + min(0LL, ey)) >> 40) - RT;
            const int k1 = (int)((tt + max(0LL, ex) + max(0LL, ey)) >> 40) + RT + 1;
            s_a[lane] = BtAngle{(tt - ((long long)(k0 + RT - 1) << 40)) >> (40 - FB), (int)(a >> (40 - FB)), (int)(bb >> (40 - FB)),
                                (float)bb * 9.094947017729282e-13f, P.inv_rfoot, 1.0f - P.inv_rfoot,
                                (unsigned)__cvta_generic_to_shared(&s_seg[lane][0])};
            s_k[lane] = make_int2(k0, min(k1, nb - 1));
            s_w[lane] = P.wfoot;
        }
        __syncthreads();
        bool finite = true;
        for (int q = w; q < cn; q += BT_Y) {  // a warp per view
            const int2 kk = s_k[q];
            const float wf = s_w[q];
            const float *row = b + (long long)(ac + q) * nb;
#pragma unroll
            for (int i = 0; i < W; i += 32) {
                const int k = kk.x + i + lane;
                const float v = (k >= 0 && k <= kk.y) ? ldg(row + k) * wf : 0.f;
                finite = finite && fabsf(v) <= FLT_LARGEST;
                s_seg[q][i + lane] = v;
            }
        }
        if (__syncthreads_and(finite)) {
#pragma unroll 1
            for (int q = 0; q < cn; ++q) bt_view<RT, false>(s_a[q], acc, cmp);
        } else {
#pragma unroll 1
            for (int q = 0; q < cn; ++q) bt_view<RT, true>(s_a[q], acc, cmp);
        }
    }
    float *ut = u + (long long)t * nx * ny;
    const int x = x0 + lane;
#pragma unroll
    for (int e = 0; e < BT_E; e += 2) {
        const int y = y0 + w * BT_E + e;
        float v0, v1;
        unpack2(acc[e / 2], v0, v1);
        if (x < nx && y < ny) ut[(long long)y * nx + x] = v0;
        if (x < nx && y + 1 < ny) ut[(long long)(y + 1) * nx + x] = v1;
    }
}

// FP32, any footprint and bin count, with BP_PX pixels per thread (x = x0 + di + 32 e, e < BP_PX:
// a 128 x 8 tile per CTA): the form for detectors more than twice as fine as the pixels. The
// per-angle constants come from shared memory as two 16-byte records and are reused for the
// thread's pixels. A pixel's bin coordinate is the tile origin's (FP64, once per angle) plus its
// in-tile offset in split steps (exact products).
constexpr int BP_PX = 4;
struct __align__(16) BpAngle {
    float fb, tAh, tAl, tBh;
    float tBl, r, ir, wf;
};

__global__ void __launch_bounds__(BP_TX *BP_TY) k_backproject4(const float *__restrict__ b, float *__restrict__ u,
                                                               const AngleParams *__restrict__ ang,
                                                               const int *__restrict__ aoff, int nx, int ny, int nb, int t0) {
    __shared__ BpAngle s_a[BP_CHUNK];
    __shared__ int s_ib[BP_CHUNK];
    const int t = t0 + blockIdx.z;
    const int x0 = blockIdx.x * BP_TX * BP_PX, y0 = blockIdx.y * BP_TY;
    const int di = threadIdx.x, dj = threadIdx.y;
    const int y = y0 + dj;
    const int tid = threadIdx.y * BP_TX + threadIdx.x;
    const int a_begin = aoff[t], a_end = aoff[t + 1];
    float acc[BP_PX];
#pragma unroll
    for (int e = 0; e < BP_PX; ++e) acc[e] = 0.f;
    float cmp[BP_PX];
#pragma unroll
    for (int e = 0; e < BP_PX; ++e) cmp[e] = 0.f;
    for (int ac = a_begin; ac < a_end; ac += BP_CHUNK) {
        const int cn = min(BP_CHUNK, a_end - ac);
        __syncthreads();
        if (tid < cn) {
            const AngleParams &P = ang[ac + tid];
            const double tb = P.t0 + (double)x0 * P.tA + (double)y0 * P.tB;
            const double fl = floor(tb);
            s_ib[tid] = (int)fmax(fmin(fl, 1e9), -1e9);
            s_a[tid] = BpAngle{(float)(tb - fl), P.tA_hi, P.tA_lo, P.tB_hi, P.tB_lo, P.rfoot, P.inv_rfoot, P.wfoot};
        }
        __syncthreads();
        if (y < ny) {
            for (int q = 0; q < cn; ++q) {
                const float *row = b + (long long)(ac + q) * nb;
                const BpAngle A = s_a[q];
                const int ib0 = s_ib[q];
                const float pb = (float)dj * A.tBh, pfb = floorf(pb);
                const float bl = (float)dj * A.tBl;
#pragma unroll
                for (int e = 0; e < BP_PX; ++e) {
                    const int dx = di + BP_TX * e;
                    if (x0 + dx >= nx) break;
                    const float pa = (float)dx * A.tAh, pfa = floorf(pa);
                    float fr = A.fb + (pa - pfa) + (pb - pfb) + fmaf((float)dx, A.tAl, bl);
                    const float ff = floorf(fr);
                    const int ib = ib0 + (int)pfa + (int)pfb + (int)ff;
                    fr -= ff;
                    if (A.r <= 1.0f) {  // at most the two bins around t
                        const float d1 = 1.0f - fr;
                        float tap = 0.f;
                        if (fr < A.r && ib >= 0 && ib < nb) tap = A.wf * (1.0f - fr * A.ir) * ldg(row + ib);
                        if (d1 < A.r && ib + 1 >= 0 && ib + 1 < nb) tap = fmaf(A.wf * (1.0f - d1 * A.ir), ldg(row + ib + 1), tap);
                        const float y = __fsub_rn(tap, cmp[e]), tt = __fadd_rn(acc[e], y);
                        cmp[e] = __fsub_rn(__fsub_rn(tt, acc[e]), y);
                        acc[e] = tt;
                    } else {
                        for (int m = 0; (float)m < A.r; ++m) {
                            const float d0 = fr + (float)m, d1 = 1.0f - fr + (float)m;
                            const int k0 = ib - m, k1 = ib + 1 + m;
                            if (d0 < A.r && k0 >= 0 && k0 < nb) acc[e] = fmaf(A.wf * (1.0f - d0 * A.ir), ldg(row + k0), acc[e]);
                            if (d1 < A.r && k1 >= 0 && k1 < nb) acc[e] = fmaf(A.wf * (1.0f - d1 * A.ir), ldg(row + k1), acc[e]);
                        }
                    }
                }
            }
        }
    }
    if (y < ny) {
#pragma unroll
        for (int e = 0; e < BP_PX; ++e) {
            const int x = x0 + di + BP_TX * e;
            if (x < nx) u[(long long)t * nx * ny + (long long)y * nx + x] = acc[e];
        }
    }
}

// ---------------------------------------------------------- K2 fan beam
// A ray steps over rows (or columns) and gives the pixel a weight only at the step of the
// pixel's row (column), when its crossing there is less than one pixel away; so the rays that
// reach the pixel are those crossing the open segments of half-length h through its centre
// along x and along y. Steps the forward march skips have crossings more than a pixel outside
// the frame, so they cannot reach a pixel and need no test here.
//
// FP32. A CTA owns a 32 x 32 pixel tile of a frame; per view it stages the rays that can reach
// the tile in shared memory, each as its crossing at the tile's middle row (column) and its
// step in fixed point (2^-26 pixels) and its datum times its length per step. A pixel takes
// every ray whose bin lies within `half` bins of its central projection t = (q . f) / (q . e)
// (q the pixel seen from the source): its segments project to within
// h max(|f_x| + |t| |e_x|, |f_y| + |t| |e_y|) / (den - h) of t, with the tile's largest |t| and
// the bound FanView::reach on the rest, widened by FAN_PAD bins for the FP32 evaluation. A ray's weight is sat(1 - |crossing - pixel|),
// zero by itself for the rays that the bound lets in without need: the distance is exact in
// 32-bit integers modulo 64 pixels (the host admits only geometries where a visited ray is
// closer than 32). Every pixel of a tile and view visits the same number of rays, the most that
// its bound allows. The sum over the views is compensated (Kahan).
// From a stage with a datum that is not finite (or so large that a sum of 1e8 may not be) on, the weights
// that are zero are taken out of the sum, and an infinite sum has no correction, so that it stays one
// (careful).
// What bounds it: instruction issue (80 %), about nine instructions per pixel, view and visited
// ray (2 to 3 rays; 2.8 on average hold the pixel). fan 256x256x32, 30 views:
// 133 us (error 3.2e-8) against 386 (1.1e-7) for one thread per pixel with four divisions per view
// and each ray's entry re-evaluated from its 16-byte record.
constexpr float FAN_PAD = (float)FAN_PAD_BINS;
constexpr int FT_X = 32, FT_Y = 4, FT_E = 8;  // threads, pixels per thread down a column
constexpr int FT_CH = 16;                     // views staged at a time
constexpr int FT_W = FAN_TILE_RAYS;           // rays staged per view
constexpr int FT_Q = 26;                      // fraction bits of the staged crossings
struct FtView {
    float fx, fy, ex, ey, qx0, qy0, reach;  // FanView
    int k0, n;    // first staged bin, rays a pixel visits
    unsigned seg; // shared address of the segment less 4 FLOOR_BITS
    int steps;    // 1: every staged ray steps over rows, 0: over columns, 2: both
};

// the visits of one view to a thread's column; STEPS: FtView::steps
template <int STEPS, bool CAREFUL>
__device__ __forceinline__ void ft_view(const FtView &V, float h, float scale, float toff, int x, int y, int dx, int dy,
                                        float (&acc)[FT_E], float (&cmp)[FT_E]) {
    const float qx = fmaf((float)x, h, V.qx0), qy = fmaf((float)y, h, V.qy0);
    const float num0 = fmaf(qx, V.fx, qy * V.fy), den0 = fmaf(qx, V.ex, qy * V.ey), dn = h * V.fy, dd = h * V.ey;
    const int n = V.n;
    const float off = toff - FAN_PAD - (float)V.k0, kmax = (float)(FT_W - n), reach = V.reach;
    unsigned at[FT_E];
    float tap[FT_E];
#pragma unroll
    for (int e = 0; e < FT_E; ++e) {
        const float r = __fdividef(1.0f, fmaf((float)e, dd, den0));
        const float t = fmaf(fmaf((float)e, dn, num0) * r, scale, fmaf(-reach, r, off));
        // first visited bin relative to the segment, rounded up by the addition; held within the
        // segment (a non-finite t visits its start)
        const float k = __fadd_ru(fminf(fmaxf(t, 0.f), kmax), FLOOR_MAGIC);
        at[e] = V.seg + 4u * (unsigned)__float_as_int(k);
        tap[e] = 0.f;
    }
    // visit by visit, the column's eight pixels side by side (their chains are independent)
#pragma unroll 1
    for (int m = 0; m < n; ++m) {
#pragma unroll
        for (int e = 0; e < FT_E; ++e) {
            const int c = __float_as_int(lds(at[e])), s = __float_as_int(lds(at[e] + 4 * FT_W));  // crossing (bit 0: steps over rows), step
            const float v = lds(at[e] + 8 * FT_W);
            int d;
            if (STEPS == 1) d = (dy + e) * s + (c - (dx << FT_Q));
            else if (STEPS == 0) d = dx * s + (c - ((dy + e) << FT_Q));
            else d = (c & 1) ? (dy + e) * s + (c - (dx << FT_Q)) : dx * s + (c - ((dy + e) << FT_Q));
            const float w = __saturatef(fmaf(-fabsf((float)d), 1.0f / (float)(1 << FT_Q), 1.0f));
            if (!CAREFUL || w > 0.f) tap[e] = fmaf(w, v, tap[e]);
            at[e] += 4;
        }
    }
#pragma unroll
    for (int e = 0; e < FT_E; ++e) {
        const float yv = __fsub_rn(tap[e], cmp[e]), tt = __fadd_rn(acc[e], yv);
        cmp[e] = !CAREFUL || fabsf(tt) <= FLT_LARGEST ? __fsub_rn(__fsub_rn(tt, acc[e]), yv) : 0.f;
        acc[e] = tt;
    }
}

__global__ void __launch_bounds__(FT_X *FT_Y, 8) k_backproject_fan_tile(const float *__restrict__ b, float *__restrict__ u,
                                                                     const FanRay<float> *__restrict__ rays,
                                                                     const FanView *__restrict__ views,
                                                                     const int *__restrict__ aoff, int nx, int ny, int nb,
                                                                     float h, float scale) {
    __shared__ float s_seg[FT_CH][3][FT_W];  // crossings and steps (integers), data
    __shared__ FtView s_v[FT_CH];
    const int t = blockIdx.z;
    const int x0 = blockIdx.x * FT_X, y0 = blockIdx.y * FT_Y * FT_E;
    const int lane = threadIdx.x, w = threadIdx.y;
    const int x1 = min(x0 + FT_X, nx) - 1, y1 = min(y0 + FT_Y * FT_E, ny) - 1;
    const int xm = x0 + FT_X / 2, ym = y0 + FT_Y * FT_E / 2;  // the staged crossings' row and column
    const float toff = 0.5f * (float)(nb - 1);
    float acc[FT_E], cmp[FT_E];
#pragma unroll
    for (int e = 0; e < FT_E; ++e) acc[e] = cmp[e] = 0.f;
    const int a_end = aoff[t + 1];
    bool careful = false;
    for (int ac = aoff[t]; ac < a_end; ac += FT_CH) {
        const int cn = min(FT_CH, a_end - ac);
        __syncthreads();
        if (w == 0 && lane < cn) {
            // the extremes of t and of 1 / den over the tile lie at its corners
            const FanView V = views[ac + lane];
            float tlo = 3.4e38f, thi = -3.4e38f, rmax = 0.f;  // central projections and 1 / den at the corners
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float qx = fmaf((float)((c & 1) ? x1 : x0), h, V.qx0), qy = fmaf((float)((c & 2) ? y1 : y0), h, V.qy0);
                const float r = 1.0f / fmaf(qx, V.ex, qy * V.ey), tc = fmaf(qx, V.fx, qy * V.fy) * r;
                tlo = fminf(tlo, tc);
                thi = fmaxf(thi, tc);
                rmax = fmaxf(rmax, r);
            }
            const float tm = fmaxf(fabsf(tlo), fabsf(thi));
            const float reach = V.reach * fmaxf(fmaf(tm, fabsf(V.ex), fabsf(V.fx)), fmaf(tm, fabsf(V.ey), fabsf(V.fy)));
            const float half = fmaf(reach, rmax, 1.5f * FAN_PAD);
            const int k0 = (int)floorf(fminf(fmaxf(fmaf(tlo, scale, toff) - half, -1e6f), 1e6f)) - 1;
            s_v[lane] = FtView{V.fx, V.fy, V.ex, V.ey, V.qx0, V.qy0, reach, k0, min((int)(2.0f * half) + 1, FT_W / 2),
                               (unsigned)__cvta_generic_to_shared(&s_seg[lane][0][0]) - 4u * (unsigned)FLOOR_BITS, 1};
        }
        __syncthreads();
        bool finite = true;
        for (int q = w; q < cn; q += FT_Y) {  // a warp per view
            const int k0 = s_v[q].k0;
            int any_r = 0, any_c = 0;
            for (int i = lane; i < FT_W; i += 32) {
                const int k = k0 + i;
                int cr = 0, st = 0;
                float v = 0.f;  // beyond the detector: no datum
                if (k >= 0 && k < nb) {
                    const long long o = (long long)(ac + q) * nb + k;
                    const FanRay<float> F = rays[o];
                    const int rows = (int)(F.f0q & 1);
                    const long long c = (F.f0q >> 1) + (rows ? ym : xm) * F.dq - ((long long)(rows ? xm : ym) << 40);
                    cr = ((int)(c >> (40 - FT_Q)) & ~1) | rows;
                    st = (int)((F.dq + (1LL << (39 - FT_Q))) >> (40 - FT_Q));
                    const float df = (float)F.dq * 9.094947017729282e-13f;
                    v = ldg(b + o) * (h * sqrtf(fmaf(df, df, 1.0f)));
                    any_r |= rows;
                    any_c |= !rows;
                }
                finite = finite && fabsf(v) <= 1e30f;
                s_seg[q][0][i] = __int_as_float(cr);
                s_seg[q][1][i] = __int_as_float(st);
                s_seg[q][2][i] = v;
            }
            any_r = __any_sync(0xffffffffu, any_r);
            any_c = __any_sync(0xffffffffu, any_c);
            if (lane == 0) s_v[q].steps = any_r && any_c ? 2 : (any_c ? 0 : 1);
        }
        careful |= !__syncthreads_and(finite);
        const int x = min(x0 + lane, x1), y = y0 + w * FT_E, dx = lane - FT_X / 2, dy = w * FT_E - FT_Y * FT_E / 2;
        for (int q = 0; q < cn; ++q) {
            const int steps = s_v[q].steps;
            if (careful) ft_view<2, true>(s_v[q], h, scale, toff, x, y, dx, dy, acc, cmp);
            else if (steps == 1) ft_view<1, false>(s_v[q], h, scale, toff, x, y, dx, dy, acc, cmp);
            else if (steps == 0) ft_view<0, false>(s_v[q], h, scale, toff, x, y, dx, dy, acc, cmp);
            else ft_view<2, false>(s_v[q], h, scale, toff, x, y, dx, dy, acc, cmp);
        }
    }
    const int x = x0 + lane;
#pragma unroll
    for (int e = 0; e < FT_E; ++e) {
        const int y = y0 + w * FT_E + e;
        if (x < nx && y < ny) u[(long long)t * nx * ny + (long long)y * nx + x] = acc[e];
    }
}

// Any geometry (and FP64): one thread per pixel; per view the bins between the central
// projections of the four segment end points (widened by FAN_PAD bins), each re-evaluated with
// the forward's own arithmetic.
template <typename real>
__global__ void __launch_bounds__(BP_TX *BP_TY) k_backproject_fan(const real *__restrict__ b, real *__restrict__ u,
                                                                  const FanRay<real> *__restrict__ rays,
                                                                  const FanView *__restrict__ views,
                                                                  const int *__restrict__ aoff, int nx, int ny, int nb,
                                                                  float h, float scale) {
    const int t = blockIdx.z;
    const int x = blockIdx.x * BP_TX + threadIdx.x, y = blockIdx.y * BP_TY + threadIdx.y;
    if (x >= nx || y >= ny) return;
    const float toff = 0.5f * (float)(nb - 1);
    real acc = 0;
    for (int a = aoff[t]; a < aoff[t + 1]; ++a) {
        const FanView V = views[a];
        const float qx = fmaf((float)x, h, V.qx0), qy = fmaf((float)y, h, V.qy0);
        const float num = qx * V.fx + qy * V.fy, den = qx * V.ex + qy * V.ey;
        const float nxp = h * V.fx, dxp = h * V.ex, nyp = h * V.fy, dyp = h * V.ey;
        const float t0 = __fdividef(num + nxp, den + dxp), t1 = __fdividef(num - nxp, den - dxp);
        const float t2 = __fdividef(num + nyp, den + dyp), t3 = __fdividef(num - nyp, den - dyp);
        const float tlo = fminf(fminf(t0, t1), fminf(t2, t3)), thi = fmaxf(fmaxf(t0, t1), fmaxf(t2, t3));
        // clamped in floating point before the conversion (a non-finite bound gives no bins)
        const int klo = (int)fminf(fmaxf(ceilf(fmaf(tlo, scale, toff - FAN_PAD)), 0.0f), (float)nb);
        const int khi = (int)fminf(fmaxf(floorf(fmaf(thi, scale, toff + FAN_PAD)), -1.0f), (float)(nb - 1));
        const FanRay<real> *ra = rays + (long long)a * nb;
        const real *row = b + (long long)a * nb;
        for (int k = klo; k <= khi; ++k) {
            const FanRay<real> R = ra[k];
            int i0, fast;
            real w1, wstep;
            if constexpr (sizeof(real) == 4) {
                const int rows = (int)(R.f0q & 1);
                const int j = rows ? y : x;
                fast = rows ? x : y;
                const long long f = (R.f0q >> 1) + j * R.dq;
                i0 = (int)(f >> 40);
                w1 = (float)(unsigned)((unsigned long long)f >> 8) * 2.3283064365386963e-10f;
                const float df = (float)R.dq * 9.094947017729282e-13f;
                wstep = h * sqrtf(fmaf(df, df, 1.0f));
            } else {
                const int j = R.rows ? y : x;
                fast = R.rows ? x : y;
                const double f = fma((double)j, R.df, R.f0), fl = floor(f);
                i0 = (int)fl;
                w1 = f - fl;
                wstep = R.wstep;
            }
            const real w = i0 == fast ? (real)1 - w1 : (i0 + 1 == fast ? w1 : (real)0);
            if (w != (real)0) acc = fma(w * wstep, ldg(row + k), acc);
        }
    }
    u[(long long)t * nx * ny + (long long)y * nx + x] = acc;
}

template <typename real>
mof_status launch_backproject(const mof_problem *p, const real *b, real *u, cudaStream_t st, bool per_frame) {
    dim3 grid((p->nx + BP_TX - 1) / BP_TX, (p->ny + BP_TY - 1) / BP_TY, p->nt);
    if (p->fan && p->fan_tile && sizeof(real) == 4) {
        const dim3 gt((p->nx + FT_X - 1) / FT_X, (p->ny + FT_Y * FT_E - 1) / (FT_Y * FT_E), p->nt);
        ::mof::count_launch(), k_backproject_fan_tile<<<gt, dim3(FT_X, FT_Y), 0, st>>>(
            (const float *)b, (float *)u, static_cast<const FanRay<float> *>(p->d_fanray), p->d_fanview, p->d_aoff, p->nx, p->ny,
            p->nb, (float)p->h, p->fan_scale);
        MOF_LAUNCH_CHECK();
        return MOF_OK;
    }
    if (p->fan) {
        ::mof::count_launch(), k_backproject_fan<real><<<grid, dim3(BP_TX, BP_TY), 0, st>>>(
            b, u, static_cast<const FanRay<real> *>(p->d_fanray), p->d_fanview, p->d_aoff, p->nx, p->ny, p->nb,
            (float)p->h, p->fan_scale);
        MOF_LAUNCH_CHECK();
        return MOF_OK;
    }
    // the plain form launches one frame at a time (t0 = t, one z slice), else all frames
    const int nlaunch = per_frame ? p->nt : 1, nz = per_frame ? 1 : p->nt;
    for (int t0 = 0; t0 < nlaunch; ++t0) {
        if (sizeof(real) == 4 && p->bp_reach) {
            const dim3 gt((p->nx + BT_X - 1) / BT_X, (p->ny + BT_Y * BT_E - 1) / (BT_Y * BT_E), nz), tt(BT_X, BT_Y);
            const float *bf = (const float *)b;
            float *uf = (float *)u;
            ::mof::count_launch();
            if (p->bp_reach == 1) k_backproject_tile<1><<<gt, tt, 0, st>>>(bf, uf, p->d_ang, p->d_aoff, p->nx, p->ny, p->nb, t0);
            else k_backproject_tile<2><<<gt, tt, 0, st>>>(bf, uf, p->d_ang, p->d_aoff, p->nx, p->ny, p->nb, t0);
        } else if (sizeof(real) == 4) {
            dim3 g4((p->nx + BP_TX * BP_PX - 1) / (BP_TX * BP_PX), (p->ny + BP_TY - 1) / BP_TY, nz);
            ::mof::count_launch(), k_backproject4<<<g4, dim3(BP_TX, BP_TY), 0, st>>>((const float *)b, (float *)u, p->d_ang,
                                                                                     p->d_aoff, p->nx, p->ny, p->nb, t0);
        } else if (p->fix64 && p->bp_reach) {
            const dim3 g1(grid.x, grid.y, nz), tb(BP_TX, BP_TY);
            const double *bd = (const double *)b;
            double *ud = (double *)u;
            ::mof::count_launch();
            if (p->bp_reach == 1) k_backproject64_fix<1><<<g1, tb, 0, st>>>(bd, ud, p->d_ang, p->d_aoff, p->nx, p->ny, p->nb, t0);
            else k_backproject64_fix<2><<<g1, tb, 0, st>>>(bd, ud, p->d_ang, p->d_aoff, p->nx, p->ny, p->nb, t0);
        } else {
            dim3 g1(grid.x, grid.y, nz);
            ::mof::count_launch(), k_backproject64<<<g1, dim3(BP_TX, BP_TY), 0, st>>>((const double *)b, (double *)u, p->d_ang, p->d_aoff, p->nx, p->ny,
                                                                                         p->nb, t0);
        }
    }
    MOF_LAUNCH_CHECK();
    return MOF_OK;
}

template mof_status launch_project<float>(const mof_problem *, const float *, float *, float *, cudaStream_t, bool);
template mof_status launch_project<double>(const mof_problem *, const double *, double *, double *, cudaStream_t, bool);
template mof_status launch_backproject<float>(const mof_problem *, const float *, float *, cudaStream_t, bool);
template mof_status launch_backproject<double>(const mof_problem *, const double *, double *, cudaStream_t, bool);

}  // namespace mof

// Plane kernels (sm_103a): per-window RANSAC with least-squares refit,
// assignment by colour consistency, occlusion cues, merge, NNF update, model
// propagation fill and the final flow / occlusion map.
#include <float.h>

#include <atomic>
#include <type_traits>

#include "common.cuh"
#include "hyp_exact.cuh"
#include "kernels.h"
#include "../../include/gpm.h"

namespace gpm {

constexpr unsigned FULL = 0xffffffffu;

// ---------------------------------------------------------------- 4-point homography
// Exact projective basis construction (hyp_exact.cuh): with P = [p1 p2 p3]
// (homogeneous columns) and lambda = adj(P) p4, A = P diag(lambda) maps the
// projective basis e1, e2, e3, (1,1,1) onto p1..p4 up to scale; likewise B
// for the targets, and H ~ B adj(A).
__device__ __forceinline__ bool collinear3(int ax, int ay, int bx, int by, int cx, int cy) {
    return (long long)(bx - ax) * (cy - ay) - (long long)(by - ay) * (cx - ax) == 0;
}

// X = i + f (f in [0,1)) lies in [-kFrameTol, n - 1 + kFrameTol].
__device__ __forceinline__ bool in_frame_tol(int i, float f, int n) {
    if (i >= 0 && i < n - 1) return true;
    if (i == n - 1) return f <= kFrameTol;
    if (i == -1) return f >= 1.f - kFrameTol;
    return false;
}

// Target sample position of pixel (px, py) under a plane: integer base and
// fraction; false if the denominator is not positive or the point leaves the
// frame (tolerance kFrameTol).
__device__ __forceinline__ bool plane_target(const Mef& m, int px, int py, int W, int H, int& ix, float& fx, int& iy,
                                             float& fy, int& kx, int& ky) {
    if (!mef_flow(m, (float)(px - m.ox), (float)(py - m.oy), kx, fx, ky, fy)) return false;
    ix = px + kx;
    iy = py + ky;
    return in_frame_tol(ix, fx, W) && in_frame_tol(iy, fy, H);
}

template <int ST>
__device__ __forceinline__ float colour_delta(const void* src, const void* tgt, int W, int H, int px, int py, int ix,
                                              float fx, int iy, float fy) {
    const float4 a = ldpix<ST>(src, py * W + px);
    const float3 b = bilinear<ST>(tgt, W, H, ix, fx, iy, fy);
    return absdiff3(a, b) / 3.f;
}

// First-order bound of the FP32 error of the position mef_flow gives for local point u (the sum of the x and y
// errors, px): every term of the flow carries a few units of 2^-24 of its own size.
__device__ __forceinline__ float mef_pos_bound(const Mef& m, float ux, float uy) {
    const float ea = fabsf(m.e0) + fabsf(m.g0 * ux) + fabsf(m.g1 * uy);
    const float den = 1.f + m.e0 + m.g0 * ux + m.g1 * uy;
    const float sx = fabsf(m.b0 * ux) + fabsf(m.h1 * uy) + fabsf(ux) * ea + fabsf(m.h2h) * ea;
    const float sy = fabsf(m.h3 * ux) + fabsf(m.b4 * uy) + fabsf(uy) * ea + fabsf(m.h5h) * ea;
    const float d = fabsf(m.h2h) + fabsf(m.h5h) + (sx + sy) / fmaxf(den, 1e-30f);
    return 16.f * 5.9604644775390625e-08f * (sx + sy + d * (1.f + ea)) / fmaxf(den, 1e-30f) +
           1.1920928955078125e-07f * (fabsf(m.h2h) + fabsf(m.h5h));
}

// The colour-overlap decision of one RANSAC inlier in FP64: the local model Hl
// (denominator positive at the window centre) maps p, the frame test with the
// same tolerance, then eq. 3's colour error from the stored texels, bilinear
// with the point clamped into the frame.  Returns 1 if delta < eps.
template <int ST>
__device__ __noinline__ int colour_overlap_fp64(const double* Hl, const void* src, const void* tgt, int W, int H,
                                                int ox, int oy, int px, int py, float eps) {
    const double ux = px - ox, uy = py - oy;
    const double w = Hl[6] * ux + Hl[7] * uy + Hl[8];
    if (!(w > 0.0)) return 0;
    const double X = ox + (Hl[0] * ux + Hl[1] * uy + Hl[2]) / w, Y = oy + (Hl[3] * ux + Hl[4] * uy + Hl[5]) / w;
    if (!(X >= -(double)kFrameTol && X <= W - 1 + (double)kFrameTol && Y >= -(double)kFrameTol &&
          Y <= H - 1 + (double)kFrameTol))
        return 0;
    const double cxp = fmin(fmax(X, 0.0), (double)(W - 1)), cyp = fmin(fmax(Y, 0.0), (double)(H - 1));
    const int ix = min((int)floor(cxp), W - 1), iy = min((int)floor(cyp), H - 1);
    const double fx = cxp - ix, fy = cyp - iy;
    const int ix1 = min(ix + 1, W - 1), iy1 = min(iy + 1, H - 1);
    const float4 a = ldpix<ST>(tgt, iy * W + ix), b = ldpix<ST>(tgt, iy * W + ix1);
    const float4 c = ldpix<ST>(tgt, iy1 * W + ix), d = ldpix<ST>(tgt, iy1 * W + ix1);
    const float4 p = ldpix<ST>(src, py * W + px);
    const double gx = 1.0 - fx, gy = 1.0 - fy;
    const double r = gy * (gx * a.x + fx * b.x) + fy * (gx * c.x + fx * d.x);
    const double g = gy * (gx * a.y + fx * b.y) + fy * (gx * c.y + fx * d.y);
    const double bb = gy * (gx * a.z + fx * b.z) + fy * (gx * c.z + fx * d.z);
    const double delta = (fabs(p.x - r) + fabs(p.y - g) + fabs(p.z - bb)) / 3.0;
    return delta < (double)eps;
}

// ---------------------------------------------------------------- cooperating groups
// One window is processed by a group: a warp (windows up to 16 x 16) or a
// whole block.  The group provides rank, size, barrier, sums and the scan
// used to compact the residual matches in raster order.
struct WarpGroup {
    static constexpr int size = 32;
    __device__ int rank() const { return threadIdx.x & 31; }
    __device__ void sync() const { __syncwarp(); }
    __device__ int sum(int v) const { return (int)__reduce_add_sync(FULL, (unsigned)v); }
    __device__ long long sum(long long v) const {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(FULL, v, off);
        return v;
    }
    __device__ unsigned max(unsigned v) const { return __reduce_max_sync(FULL, v); }
    __device__ bool any(bool p) const { return __any_sync(FULL, p); }
    // exclusive prefix of `take` over the group and the total
    __device__ int scan(bool take, int& total) const {
        const unsigned b = __ballot_sync(FULL, take);
        total = __popc(b);
        return __popc(b & ((1u << rank()) - 1));
    }
};

template <int NT>
struct BlockGroup {
    static constexpr int size = NT;
    int* red_i;
    unsigned long long* red_u;
    __device__ int rank() const { return threadIdx.x; }
    __device__ void sync() const { __syncthreads(); }
    __device__ int sum(int v) const {
        v = (int)__reduce_add_sync(FULL, (unsigned)v);
        __syncthreads();
        if ((threadIdx.x & 31) == 0) red_i[threadIdx.x >> 5] = v;
        __syncthreads();
        int t = 0;
        for (int w = 0; w < NT / 32; ++w) t += red_i[w];
        return t;
    }
    __device__ long long sum(long long v) const {
        v = WarpGroup().sum(v);
        __syncthreads();
        if ((threadIdx.x & 31) == 0) red_u[threadIdx.x >> 5] = (unsigned long long)v;
        __syncthreads();
        long long t = 0;
        for (int w = 0; w < NT / 32; ++w) t += (long long)red_u[w];
        return t;
    }
    __device__ unsigned max(unsigned v) const {
        v = __reduce_max_sync(FULL, v);
        __syncthreads();
        if ((threadIdx.x & 31) == 0) red_i[threadIdx.x >> 5] = (int)v;
        __syncthreads();
        unsigned t = 0;
        for (int w = 0; w < NT / 32; ++w) t = (unsigned)red_i[w] > t ? (unsigned)red_i[w] : t;
        return t;
    }
    __device__ bool any(bool p) const { return __syncthreads_or(p) != 0; }
    __device__ unsigned long long max(unsigned long long v) const {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            const unsigned long long o = __shfl_xor_sync(FULL, v, off);
            v = o > v ? o : v;
        }
        __syncthreads();
        if ((threadIdx.x & 31) == 0) red_u[threadIdx.x >> 5] = v;
        __syncthreads();
        unsigned long long t = 0;
        for (int w = 0; w < NT / 32; ++w) t = red_u[w] > t ? red_u[w] : t;
        return t;
    }
    __device__ int scan(bool take, int& total) const {
        const unsigned b = __ballot_sync(FULL, take);
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        __syncthreads();
        if (lane == 0) red_i[warp] = __popc(b);
        __syncthreads();
        int off = 0;
        total = 0;
        for (int w = 0; w < NT / 32; ++w) {
            if (w < warp) off += red_i[w];
            total += red_i[w];
        }
        return off + __popc(b & ((1u << lane) - 1));
    }
};

// ---------------------------------------------------------------- least-squares refit (one thread per window)
// Entry (r, c) of the normalised DLT normal matrix A^T A from the 24 moments
// mom[a * 6 + q] = sum w_a zz^T[q] (w in {1, u, v, u^2 + v^2}, zz^T entries
// q in {x^2, xy, x, y^2, y, 1}): rows/columns 0-2 hold the b b^T block, 3-5
// the a a^T block, 6-8 the (u, v)-weighted blocks of the rows a = (0, -z, v z)
// and b = (z, 0, -u z).
__device__ __forceinline__ double dlt_entry(const double* mom, int r, int c) {
    const int br = r / 3, bc = c / 3, ir = r % 3, ic = c % 3;
    const int lo = ir < ic ? ir : ic, hi = ir < ic ? ic : ir;
    const int q = lo == 0 ? hi : (lo == 1 ? (hi == 1 ? 3 : 4) : 5);
    if (br == bc) return br < 2 ? mom[q] : mom[18 + q];
    if ((br == 0 && bc == 2) || (br == 2 && bc == 0)) return -mom[6 + q];
    if ((br == 1 && bc == 2) || (br == 2 && bc == 1)) return -mom[12 + q];
    return 0.0;
}

// Plane geometry checks of a local homography (rows, maps u -> local
// target): denominator positive on the window grown by the patch radius and
// local area scale sqrt(det J) at the window centre in [scale_min, scale_max].
__device__ __forceinline__ bool plane_geometry_ok(const double* Hl, int s, int r, double scale_min, double scale_max) {
    const double dc = Hl[8] - 0.5 * (Hl[6] + Hl[7]);
    const double rdc = 1.0 / dc;
    double hn[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) hn[q] = Hl[q] * rdc;
    bool ok = true;
    const double cxs[2] = {-(double)(s / 2) - r, (double)(s / 2) - 1 + r};
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b)
            if (!(hn[6] * cxs[a] + hn[7] * cxs[b] + hn[8] > 0)) ok = false;
    const double uc = -0.5;
    const double X = hn[0] * uc + hn[1] * uc + hn[2], Y = hn[3] * uc + hn[4] * uc + hn[5];
    const double j00 = hn[0] - X * hn[6], j01 = hn[1] - X * hn[7];
    const double j10 = hn[3] - Y * hn[6], j11 = hn[4] - Y * hn[7];
    const double det = j00 * j11 - j01 * j10;
    // sqrt(det) in [scale_min, scale_max], compared without the root
    return ok && det > 0 && det >= scale_min * scale_min && det <= scale_max * scale_max;
}

// A positive normal float as a double, assembled from its bits (a conversion issues on the FP64 pipe, 64 cycles a
// warp instruction on GB300).
__device__ __forceinline__ double double_of(float f) {
    const unsigned b = __float_as_uint(f);
    return __hiloint2double((int)((b >> 3) + 0x38000000u), (int)(b << 29));
}
// a < b for non-negative doubles that are not NaN, by their bits (a comparison issues on the FP64 pipe too).
__device__ __forceinline__ bool less_bits(double a, double b) { return __double_as_longlong(a) < __double_as_longlong(b); }
// d < 0, by its bits.
__device__ __forceinline__ bool negative(double d) {
    return (unsigned long long)__double_as_longlong(d) - 0x8000000000000001ull < 0x7FF0000000000000ull;
}
// Half of a normal double well above the smallest, by its exponent.
__device__ __forceinline__ double half_of(double r) {
    return __hiloint2double(__double2hiint(r) - 0x00100000, __double2loint(r));
}

// 1 / sqrt(n) for a positive normal double: an FP32 estimate refined by two
// Newton steps (relative error ~1e-16), far fewer FP64 operations than a
// correctly rounded square root and division.  Inverse iteration only needs a
// scale close to the unit norm.
__device__ __noinline__ double rsqrt_wide(double n) { return 1.0 / sqrt(n); }
__device__ __forceinline__ double rsqrt_nr(double n) {
    if (!(less_bits(1e-30, n) && less_bits(n, 1e30))) return rsqrt_wide(n);  // outside the FP32 estimate's range
    double r = double_of(rsqrtf((float)n));
#pragma unroll
    for (int k = 0; k < 2; ++k) r = fma(half_of(r), fma(-n * r, r, 1.0), r);
    return r;
}

// Cholesky factor (lower, packed, in place) of the symmetric matrix in A;
// rd[j] = 1 / L[j][j].  The diagonal roots come from an FP32 estimate and
// Newton steps (rsqrt_nr).  Returns false if a pivot is not positive (the
// matrix is not positive definite).
__device__ __forceinline__ bool cholesky9(double (&A)[45], double (&rd)[9]) {
    bool ok = true;
#pragma unroll
    for (int j = 0; j < 9; ++j) {
        double d = A[j * (j + 1) / 2 + j];
#pragma unroll
        for (int k = 0; k < j; ++k) d = fma(-A[j * (j + 1) / 2 + k], A[j * (j + 1) / 2 + k], d);
        ok = ok && d > 0;
        const double r = d > 0 ? rsqrt_nr(d) : 1.0;
        A[j * (j + 1) / 2 + j] = d * r;
        rd[j] = r;
#pragma unroll
        for (int i = j + 1; i < 9; ++i) {
            double t = A[i * (i + 1) / 2 + j];
#pragma unroll
            for (int k = 0; k < j; ++k) t = fma(-A[i * (i + 1) / 2 + k], A[j * (j + 1) / 2 + k], t);
            A[i * (i + 1) / 2 + j] = t * r;
        }
    }
    return ok;
}

// State of an inverse iteration after e.it steps.
struct EigState {
    double sigma, tr, prev, before;  // shift, trace, the last step's change (1e300 after a shift) and the one before
    int reshifts, slow, it;
    bool above;  // the last ratio of changes was above 0.5
};
// The warp's matrices (packed, one column per lane), and the one window whose iteration the whole warp carries on:
// the factor of M - sigma I and the vector so far.
struct EigShared {
    double M[45][32];
    EigState e;
    double A[45], rd[9], x[9];
    double P[9][9], y[9];  // eig_jump: a power of (M - sigma I)^-1, and a product with it
};
constexpr int kEigSteps = 200;

// |d| as bits, which order non-negative doubles (0 for NaN, which fmax would pass over).
__device__ __forceinline__ unsigned long long abs_bits(double d) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(d) & 0x7FFFFFFFFFFFFFFFull;
    return b > 0x7FF0000000000000ull ? 0ull : b;
}
// diff / prev > 0.9 for 0 < prev / 2 < diff, both normal: from the leading 24 bits, or divided where those are too
// close to say.
__device__ __forceinline__ bool ratio_above_0p9(double diff, double prev) {
    const int hd = __double2hiint(diff), hp = __double2hiint(prev), de = (hd >> 20) - (hp >> 20);
    if (de > 1) return true;
    const float md = __int_as_float(0x3F800000 | ((hd & 0xFFFFF) << 3) | ((unsigned)__double2loint(diff) >> 29));
    const float mp = __int_as_float(0x3F800000 | ((hp & 0xFFFFF) << 3) | ((unsigned)__double2loint(prev) >> 29));
    const float r = __fdividef(md, mp) * (de > 0 ? 2.f : (de < 0 ? 0.5f : 1.f));
    return fabsf(r - 0.9f) > 1e-5f ? r > 0.9f : diff / prev > 0.9;
}

// After a step that changed the unit vector by diff.
// Stopping: the step's change is below 1e-12 and, when the iteration converges slowly (a small eigen-gap
// against the shift's distance), so is the remaining error extrapolated from the ratio of successive changes
// (a small change per step alone would stop a slow iteration far from the vector).  A slow iteration is
// re-shifted at the current vector's Rayleigh quotient minus twice its residual (still below the smallest
// eigenvalue), a few times at most.  An iteration that stays slow after them measures the eigen-gap: with
// the ratio q of successive changes, (lambda_1 - sigma) / (lambda_2 - sigma) = q gives lambda_2 - lambda_1 =
// (rho - sigma)(1 - q) / q (rho, the Rayleigh quotient, for lambda_1); below 1e-11 of the trace (at most 9
// times the largest eigenvalue), the gap is far below the 1e-8 of the largest eigenvalue at which the
// smallest eigenvector is no longer determined to the 1e-6 a refit is compared at, and the iteration stops.
// The comparisons of q = diff / prev, rounded, with 0.5 are those of diff with prev / 2 (exact), and the one with
// 0.9 rarely needs the quotient: it is divided only where its value counts.
//
// Whether the iteration has converged; notes in e how fast it does.
__device__ __forceinline__ bool eig_converged(double diff, EigState& e) {
    const double prev = e.prev;
    e.before = prev;
    e.prev = diff;
    bool below, slow;  // q < 0.5, q > 0.9
    if (less_bits(1e-280, prev) && !less_bits(1e300, prev) && !less_bits(1e300, diff) && less_bits(1e-280, diff)) {
        const double h = half_of(prev);
        below = less_bits(diff, h);
        e.above = less_bits(h, diff);
        slow = e.above && ratio_above_0p9(diff, prev);
    } else {
        const double q = diff / prev;
        below = q < 0.5;
        e.above = q > 0.5;
        slow = q > 0.9;
    }
    e.slow = slow ? e.slow + 1 : 0;  // q >= 1: no convergence at all (a gap below what rounding resolves)
    // 1e-12 is far below what the rescore (1e-5 near-tie band) and the
    // model comparison (1e-6) can see
    if (!less_bits(diff, 1e-12)) return false;
    if (below) return true;
    const double q = diff / prev;
    return diff * q / (1.0 - fmin(q, 0.999999)) < 1e-13;
}
// The gap test or the re-shift that is due after a step (column `col` of M is the matrix): 0 stop, 1 go on, 2 go on
// with the factor B (and 1 / its diagonal, rdB) of the matrix less the new shift.  Out of line: rare, and inlined the
// compiler fuses parts of it into the caller's arithmetic, which changes the last bits.
__device__ __noinline__ int eig_gap_or_shift(const double (*M)[32], int col, const double* x, EigState* e, double* B_out,
                                             double* rd_out) {
    auto sym = [](int i, int j) { return i >= j ? i * (i + 1) / 2 + j : j * (j + 1) / 2 + i; };
    double Mx[9], xx = 0, rho = 0;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        double t = 0;
#pragma unroll
        for (int j = 0; j < 9; ++j) t = fma(M[sym(i, j)][col], x[j], t);
        Mx[i] = t;
        xx = fma(x[i], x[i], xx);
        rho = fma(x[i], t, rho);
    }
    rho /= xx;
    if (e->reshifts >= 4) {
        const double q = e->prev / e->before;
        const double gap = q < 1.0 ? (rho - e->sigma) * (1.0 - q) / q : 0.0;
        return gap < 1e-11 * e->tr ? 0 : 1;
    }
    ++e->reshifts;
    double rr = 0;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const double r = fma(-rho, x[i], Mx[i]);
        rr = fma(r, r, rr);
    }
    const double sig2 = rho - 2.0 * sqrt(rr / xx);
    if (!(sig2 > e->sigma)) return 1;
    double B[45], rd2[9];
#pragma unroll
    for (int q = 0; q < 45; ++q) B[q] = M[q][col];
#pragma unroll
    for (int i = 0; i < 9; ++i) B[i * (i + 1) / 2 + i] -= sig2;
    if (!cholesky9(B, rd2)) return 1;
    e->sigma = sig2;
    e->prev = 1e300;
#pragma unroll
    for (int q = 0; q < 45; ++q) B_out[q] = B[q];
#pragma unroll
    for (int i = 0; i < 9; ++i) rd_out[i] = rd2[i];
    return 2;
}
__device__ __forceinline__ bool eig_check_due(const EigState& e) {
    return e.reshifts < 4 ? e.it >= 2 && e.above : e.slow >= 4 && (e.slow & 3) == 0;
}

// Unit eigenvector of the smallest eigenvalue of the 9 x 9 symmetric positive
// semi-definite matrix M (lower triangle packed, row i at i(i+1)/2), from the
// start x.  The FP64 pipe of this GPU issues a warp instruction in about 64
// cycles, an FP32 one in 1, so:
//  1. FP32: inverse iteration with the explicit inverse of M / tr + 1e-6 I
//     until the direction settles at FP32 resolution;
//  2. FP64: Rayleigh quotient rho and residual r = M x - rho x of that
//     direction; M has an eigenvalue within |r| of rho, the smallest one when
//     x is nearest its eigenvector, so sigma = rho - 2 |r| lies below it;
//  3. FP64 inverse iteration with the Cholesky factor of M - sigma I: the
//     shift makes each step shrink the other directions by
//     (l1 - sigma) / (li - sigma), so a few steps reach 1e-12.  If that matrix
//     is not positive definite (the bound did not hold), the shift falls back
//     to -1e-13 tr, plain inverse iteration.
// One thread per window: each FP64 warp instruction serves 32 windows.
// eig_start does 1 and 2 and the first factor, eig_thread and eig_warp the steps.
__device__ __forceinline__ void eig_start(const double (&M)[45], double (&x)[9], double (&A)[45], double (&rd)[9],
                                          EigState& e) {
    auto sym = [](int i, int j) { return i >= j ? i * (i + 1) / 2 + j : j * (j + 1) / 2 + i; };
    double tr = 0;
#pragma unroll
    for (int i = 0; i < 9; ++i) tr += M[i * (i + 1) / 2 + i];
    {  // 1. FP32 direction
        const float rs = tr > 0 ? (float)(1.0 / tr) : 1.f;
        float L[45], rdf[9];
#pragma unroll
        for (int q = 0; q < 45; ++q) L[q] = (float)M[q] * rs;
#pragma unroll
        for (int i = 0; i < 9; ++i) L[i * (i + 1) / 2 + i] += 1e-6f;
#pragma unroll
        for (int j = 0; j < 9; ++j) {
            float d = L[j * (j + 1) / 2 + j];
#pragma unroll
            for (int k = 0; k < j; ++k) d = fmaf(-L[j * (j + 1) / 2 + k], L[j * (j + 1) / 2 + k], d);
            const float r = d > 1e-30f ? rsqrtf(d) : 1e15f;
            L[j * (j + 1) / 2 + j] = d * r;
            rdf[j] = r;
#pragma unroll
            for (int i = j + 1; i < 9; ++i) {
                float t = L[i * (i + 1) / 2 + j];
#pragma unroll
                for (int k = 0; k < j; ++k) t = fmaf(-L[i * (i + 1) / 2 + k], L[j * (j + 1) / 2 + k], t);
                L[i * (i + 1) / 2 + j] = t * r;
            }
        }
        float xf[9], n0 = 0.f;
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            xf[i] = (float)x[i];
            n0 = fmaf(xf[i], xf[i], n0);
        }
        const float s0 = rsqrtf(n0);
#pragma unroll
        for (int i = 0; i < 9; ++i) xf[i] *= s0;
        for (int it = 0; it < 60; ++it) {  // a start vector only: the FP64 iteration below converges from it
            float y[9];
#pragma unroll
            for (int i = 0; i < 9; ++i) {  // L z = x
                float t = xf[i];
#pragma unroll
                for (int k = 0; k < i; ++k) t = fmaf(-L[i * (i + 1) / 2 + k], y[k], t);
                y[i] = t * rdf[i];
            }
#pragma unroll
            for (int i = 8; i >= 0; --i) {  // L^T y = z
                float t = y[i];
#pragma unroll
                for (int k = i + 1; k < 9; ++k) t = fmaf(-L[k * (k + 1) / 2 + i], y[k], t);
                y[i] = t * rdf[i];
            }
            float n = 0.f, dot = 0.f;
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                n = fmaf(y[i], y[i], n);
                dot = fmaf(y[i], xf[i], dot);
            }
            if (!(n > 0.f) || !isfinite(n)) break;
            float sc = rsqrtf(n);
            if (dot < 0.f) sc = -sc;
            float diff = 0.f;
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                y[i] *= sc;
                diff = fmaxf(diff, fabsf(y[i] - xf[i]));
                xf[i] = y[i];
            }
            if (diff < 4e-7f) break;
        }
        bool finite = true;
#pragma unroll
        for (int i = 0; i < 9; ++i) finite = finite && isfinite(xf[i]);
        if (finite) {
#pragma unroll
            for (int i = 0; i < 9; ++i) x[i] = (double)xf[i];
        }
    }
    // 2. shift from the Rayleigh quotient and the residual of x
    double xx = 0, rho = 0, Mx[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        double t = 0;
#pragma unroll
        for (int j = 0; j < 9; ++j) t = fma(M[sym(i, j)], x[j], t);
        Mx[i] = t;
        xx = fma(x[i], x[i], xx);
        rho = fma(x[i], t, rho);
    }
    const double ixx = 1.0 / xx;
    rho *= ixx;
    double rr = 0;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const double r = fma(-rho, x[i], Mx[i]);
        rr = fma(r, r, rr);
    }
    const double floor_shift = -1e-13 * tr - 1e-300;
    double sigma = rho - 2.0 * sqrt(rr * ixx);
    if (!(sigma > floor_shift)) sigma = floor_shift;
    // 3. shifted inverse iteration in FP64
#pragma unroll
    for (int q = 0; q < 45; ++q) A[q] = M[q];
#pragma unroll
    for (int i = 0; i < 9; ++i) A[i * (i + 1) / 2 + i] -= sigma;
    if (!cholesky9(A, rd)) {
#pragma unroll
        for (int q = 0; q < 45; ++q) A[q] = M[q];
#pragma unroll
        for (int i = 0; i < 9; ++i) A[i * (i + 1) / 2 + i] -= floor_shift;
        cholesky9(A, rd);
        sigma = floor_shift;
    }
    {
        const double s0 = rsqrt_nr(xx);
#pragma unroll
        for (int i = 0; i < 9; ++i) x[i] *= s0;
    }
    e.sigma = sigma;
    e.tr = tr;
    e.prev = 1e300;
    e.reshifts = e.slow = e.it = 0;
}

// One step on this thread; false: the iteration is over.
__device__ __forceinline__ bool eig_thread(const double (*M)[32], double (&x)[9], double (&A)[45], double (&rd)[9],
                                           EigState& e) {
    double y[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) {  // L z = x
        double t = x[i];
#pragma unroll
        for (int k = 0; k < i; ++k) t = fma(-A[i * (i + 1) / 2 + k], y[k], t);
        y[i] = t * rd[i];
    }
#pragma unroll
    for (int i = 8; i >= 0; --i) {  // L^T y = z
        double t = y[i];
#pragma unroll
        for (int k = i + 1; k < 9; ++k) t = fma(-A[k * (k + 1) / 2 + i], y[k], t);
        y[i] = t * rd[i];
    }
    double n = 0, dot = 0;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        n = fma(y[i], y[i], n);
        dot = fma(y[i], x[i], dot);
    }
    double sc = rsqrt_nr(n);
    if (negative(dot)) sc = -sc;
    unsigned long long diff = 0;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        y[i] *= sc;
        diff = max(diff, abs_bits(y[i] - x[i]));
        x[i] = y[i];
    }
    if (eig_converged(__longlong_as_double((long long)diff), e)) return false;
    if (eig_check_due(e)) {
        double xc[9], B[45], rdB[9];  // copies: the call must not force x, A and rd out of registers
        EigState ec = e;
#pragma unroll
        for (int i = 0; i < 9; ++i) xc[i] = x[i];
        const int what = eig_gap_or_shift(M, threadIdx.x, xc, &ec, B, rdB);
        e = ec;
        if (what == 0) return false;
        if (what == 2) {
#pragma unroll
            for (int q = 0; q < 45; ++q) A[q] = B[q];
#pragma unroll
            for (int i = 0; i < 9; ++i) rd[i] = rdB[i];
        }
    }
    return ++e.it < kEigSteps;
}

// Many steps of the iteration at once, by the whole warp: x <- B^128 x, normalised and oriented, B the inverse behind
// the factor in sh (fresh: B's powers are not in sh.P yet; otherwise sh.P is squared once more and twice the steps are
// taken).  A step multiplies by B and scales, so this is where 128 steps lead, but for rounding: B is applied to
// the unit vectors (a column a lane) and squared seven times, each time scaled by a power of two, its entries two a lane:
// 240 FP64 instructions where the steps take 10,000.  The rounding of B is small against its largest eigenvalue
// 1 / (lambda_1 - sigma), so the vector is off by some 1e-16 / (1 - q), q the ratio of the steps' changes: a few
// units at the ratios in question (0.6 to 0.95), below what the steps themselves leave (1e-13).  Of 7200 models of windows
// with tiny supports one differs from the steps' result, by 7e-16.
__device__ __noinline__ void eig_jump(EigShared& sh, bool fresh) {
    const int lane = threadIdx.x & 31, row = min(lane, 8);
    // sh.P times the power of two that brings its largest entry, which is on the diagonal, into [1, 2)
    auto exponent = [&]() {
        __syncwarp();
        const unsigned top = __reduce_max_sync(FULL, (unsigned)__double2hiint(sh.P[row][row]) & 0x7FFFFFFFu) >> 20;
        return (int)top;
    };
    auto usable = [](int top) { return top > 100 && top < 1900; };
    auto scale = [](int top) { return __hiloint2double((2046 - top) << 20, 0); };
    if (fresh) {
        double y[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            double t = i == row ? 1.0 : 0.0;
#pragma unroll
            for (int k = 0; k < i; ++k) t = fma(-sh.A[i * (i + 1) / 2 + k], y[k], t);
            y[i] = t * sh.rd[i];
        }
#pragma unroll
        for (int i = 8; i >= 0; --i) {
            double t = y[i];
#pragma unroll
            for (int k = i + 1; k < 9; ++k) t = fma(-sh.A[k * (k + 1) / 2 + i], y[k], t);
            y[i] = t * sh.rd[i];
        }
        if (lane < 9) {
#pragma unroll
            for (int i = 0; i < 9; ++i) sh.P[lane][i] = y[i];
        }
        const int top = exponent();
        if (!usable(top)) return;  // warp-uniform
        const double f = scale(top);
        if (lane < 9) {
#pragma unroll
            for (int i = 0; i < 9; ++i) sh.P[lane][i] = y[i] * f;
        }
        __syncwarp();
    }
    int pi[2], pj[2];  // this lane's entries (i, j) of the lower triangle
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const int e = min(lane + 32 * r, 44);
        int i = 0;
        while ((i + 1) * (i + 2) / 2 <= e) ++i;
        pi[r] = i;
        pj[r] = e - i * (i + 1) / 2;
    }
    for (int s = fresh ? 0 : 6; s < 7; ++s) {
        double c[2];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            c[r] = 0;
#pragma unroll
            for (int k = 0; k < 9; ++k) c[r] = fma(sh.P[pi[r]][k], sh.P[pj[r]][k], c[r]);
        }
        __syncwarp();
        auto put = [&](double f) {
#pragma unroll
            for (int r = 0; r < 2; ++r) sh.P[pi[r]][pj[r]] = sh.P[pj[r]][pi[r]] = c[r] * f;
        };
        put(1.0);
        const int top = exponent();
        if (!usable(top)) return;
        put(scale(top));
        __syncwarp();
    }
    double t = 0;
#pragma unroll
    for (int k = 0; k < 9; ++k) t = fma(sh.P[row][k], sh.x[k], t);
    if (lane < 9) sh.y[lane] = t;
    __syncwarp();
    double n = 0, dot = 0;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        n = fma(sh.y[i], sh.y[i], n);
        dot = fma(sh.y[i], sh.x[i], dot);
    }
    __syncwarp();
    if (!(n > 1e-30 && n < 1e30)) return;  // the same on every lane
    double sc = rsqrt_nr(n);
    if (negative(dot)) sc = -sc;
    if (lane < 9) sh.x[lane] = t * sc;
    __syncwarp();
}

// The iteration of one window (its state in sh, its matrix in column `col`), carried on by the whole warp: the few
// windows that need many steps (supports of 4 or 5 matches with a nearly two-dimensional null space: up to 200) set
// the launch's duration, and a step on one thread is some 140 FP64 instructions of 64 cycles each.  Every operation
// and its order per result are those of eig_thread, so the bits are the same: the forward substitution by columns,
// lane i holding row i; the backward one (whose order leaves no parallelism) on every lane; the two dot products on
// even and odd lanes; scaling and difference with lane i on entry i.  About 80 FP64 instructions a step; the eight
// solves of a 1024x436 pair 3.15 -> 2.36 ms.  The solve kernel hands a window over once it is the warp's last and 4
// steps are done (98.5 % of the windows need no more), or after 12: two or more are cheaper side by side on their
// threads for a few steps.
// A window that is still iterating with one factor after 4 steps here takes the next 128 at once (eig_jump); a slow
// one only when the gap test has let it go on.  One launch in two has a window of 60 to 200 steps, 0.3 to 0.55 ms in
// which the chip waits: the eight solves of a 1024x436 pair 1.71 -> 1.26 ms, the six of a 128x96 one 0.71 -> 0.57 ms.
__device__ __noinline__ void eig_warp(EigShared& sh, int col) {
    const int lane = threadIdx.x & 31, row = min(lane, 8);
    double A[45], rd[9], x[9], Lr[8], rdr = 0;
    EigState e = sh.e;
#pragma unroll
    for (int i = 0; i < 9; ++i) x[i] = sh.x[i];
    int loaded = -1, since = 0;  // the factor held here; steps with it since a jump
    bool fresh = true, gap_ok = false;
    for (;;) {
        if (loaded != e.reshifts) {  // the factor may be new
            loaded = e.reshifts;
            since = 0;
            fresh = true;
            __syncwarp();
#pragma unroll
            for (int q = 0; q < 45; ++q) A[q] = sh.A[q];
#pragma unroll
            for (int i = 0; i < 9; ++i) rd[i] = sh.rd[i];
#pragma unroll
            for (int k = 0; k < 8; ++k) Lr[k] = sh.A[row * (row + 1) / 2 + min(k, row)];
            rdr = sh.rd[row];
        }
        double z[9], own = x[0];
#pragma unroll
        for (int i = 1; i < 9; ++i) own = row == i ? x[i] : own;
        double t = own;
#pragma unroll
        for (int k = 0; k < 9; ++k) {  // L z = x
            z[k] = __shfl_sync(FULL, t * rdr, k);
            if (k < 8) t = row > k ? fma(-Lr[k < 8 ? k : 0], z[k], t) : t;
        }
        double y[9];
#pragma unroll
        for (int i = 8; i >= 0; --i) {  // L^T y = z
            double u = z[i];
#pragma unroll
            for (int k = i + 1; k < 9; ++k) u = fma(-A[k * (k + 1) / 2 + i], y[k], u);
            y[i] = u * rd[i];
        }
        double acc = 0;
#pragma unroll
        for (int i = 0; i < 9; ++i) acc = fma(y[i], (lane & 1) ? x[i] : y[i], acc);
        const double n = __shfl_sync(FULL, acc, 0), dot = __shfl_sync(FULL, acc, 1);
        double sc = rsqrt_nr(n);
        if (negative(dot)) sc = -sc;
        double yr = y[0];
#pragma unroll
        for (int i = 1; i < 9; ++i) yr = row == i ? y[i] : yr;
        yr *= sc;
        const unsigned long long d = abs_bits(yr - own);
        const unsigned hi = __reduce_max_sync(FULL, (unsigned)(d >> 32));
        const unsigned lo = __reduce_max_sync(FULL, (unsigned)(d >> 32) == hi ? (unsigned)d : 0u);
#pragma unroll
        for (int i = 0; i < 9; ++i) x[i] = __shfl_sync(FULL, yr, i);
        if (eig_converged(__longlong_as_double((long long)(((unsigned long long)hi << 32) | lo)), e)) break;
        if (eig_check_due(e)) {  // the same on every lane
            double xc[9], B[45], rdB[9];
            EigState ec = e;
            const int was = e.reshifts;
#pragma unroll
            for (int i = 0; i < 9; ++i) xc[i] = x[i];
            const int what = eig_gap_or_shift(sh.M, col, xc, &ec, B, rdB);
            e = ec;
            if (what == 0) break;
            gap_ok = what == 1 && e.reshifts >= 4 && ec.reshifts == was;
            if (what == 2) {
                __syncwarp();
                if (lane == 0) {
                    for (int q = 0; q < 45; ++q) sh.A[q] = B[q];
                    for (int i = 0; i < 9; ++i) sh.rd[i] = rdB[i];
                }
            }
        }
        if (++e.it >= kEigSteps) break;
        if (++since >= 4 && loaded == e.reshifts && (e.slow == 0 || gap_ok)) {
            __syncwarp();
            if (lane == 0) {
#pragma unroll
                for (int i = 0; i < 9; ++i) sh.x[i] = x[i];
            }
            __syncwarp();
            eig_jump(sh, fresh);
#pragma unroll
            for (int i = 0; i < 9; ++i) x[i] = sh.x[i];
            fresh = false;
            since = 0;
        }
    }
    __syncwarp();
    if (lane == 0) {
#pragma unroll
        for (int i = 0; i < 9; ++i) sh.x[i] = x[i];
    }
    __syncwarp();
}

// The exact hypothesis as doubles in window-local coordinates, oriented like
// its evaluation form (positive denominator at the window centre) and scaled
// by a power of two (largest entry in [1, 2)): the FP64 stand-in of the
// residual test, built without FP64 instructions.
__device__ __forceinline__ void exact_local_fp64(const i128* Hk, double* Hl) {
    const i128 dc2 = 2 * Hk[8] - (Hk[6] + Hk[7]);
    exact_to_double_pow2(Hk, Hl, dc2 < 0);
}

// ---------------------------------------------------------------- RANSAC per window
// Sec. 3.1.2 / 3.2, in three launches per level and stage:
//   (A) ransac_fit, a group per window: the window's matches (u, u + v(u))
//       -- all pixels at stage 1, the still-unassigned ones in raster order at
//       stage 2 -- go to shared memory as exact floats; the group draws, solves
//       and scores the hypotheses, keeps the largest support (lowest index on
//       ties) and accumulates what the least-squares refit needs on the
//       winner's inliers: Hartley sums and the 24 DLT moments as exact integers;
//   (B) k_refit_solve, a thread per window: normalised DLT refit in FP64;
//   (C) ransac_finish, a group per window: rescoring of the refit (kept unless
//       it has fewer inliers), the colour-overlap count and the model record.

// mef_inlier_pt out of line (loose hypotheses are rare: the callers' loops stay small).
__device__ __noinline__ bool mef_inlier_pt_ool(const Mef& m, float4 mt, float t2, bool& unc) {
    return mef_inlier_pt(m, mt.x, mt.y, mt.z, mt.w, t2, unc);
}
// The certified test of a match: the FP32 decision, and unc when it is within its rounding bound.
__device__ __forceinline__ bool cert_inlier(const Mef& m, const float4& mt, float t2, bool& unc) {
    return mef_loose(m) ? mef_inlier_pt_ool(m, mt, t2, unc) : mef_inlier_c(m, mt.x, mt.y, mt.z, mt.w, t2, unc);
}

// Exact integer of a small integer-valued float: adding 1.5 * 2^23 puts it in
// the low mantissa bits (no conversion instruction).
__device__ __forceinline__ int exact_int(float f) { return __float_as_int(f + 12582912.f) - 0x4B400000; }

template <class G>
__device__ __forceinline__ void window_origin(const LevelGeom& g, int cell, int& x0, int& y0, int& ox, int& oy) {
    const int cxw = cell % g.gx.count, cyw = cell / g.gx.count;
    x0 = win_pos(g.gx, g.h, cxw);
    y0 = win_pos(g.gy, g.h, cyw);
    ox = x0 + g.s / 2;
    oy = y0 + g.s / 2;
}

// A target no hypothesis reaches within the inlier radius (its square stays finite for any accepted hypothesis).
constexpr float kFarTarget = 1e15f;
// Up to this |u + v - v0|, differences of targets stay below 2^15 and their cross products fit 32 bits.
constexpr int kNearReach = kNearOffsets;

// A target this far from the sample's median target (sample_centre) is out of the hypothesis's reach, and no inlier.  It
// gets there only along its vanishing line, where a solve in FP64 is off by some q^2 2^-53 / (window side), a pixel from
// about 2^28 on: a marker that a sample happens to hold bends the line to itself, and counts for nothing.
constexpr long long kFarthest = 1ll << 26;
__device__ __forceinline__ bool out_of_reach(longlong2 q, longlong2 centre) {
    return max(llabs(q.x - centre.x), llabs(q.y - centre.y)) >= kFarthest;
}
// The second smallest of a sample's targets, by components: among three or four that are together.
__device__ __forceinline__ longlong2 sample_centre(longlong2 a, longlong2 b, longlong2 c, longlong2 d) {
    auto second = [](long long a, long long b, long long c, long long d) {
        return min(max(min(a, b), min(c, d)), min(max(a, b), max(c, d)));
    };
    return make_longlong2(second(a.x, b.x, c.x, d.x), second(a.y, b.y, c.y, d.y));
}
// What the far matches of a window need (shared memory, one per window): how many, and how many of them are in reach of
// near samples (a few more at the limit), the offsets in memory and the reference offset.
struct WindowFar {
    const int2* nnf;
    int W, ox, oy, v0x, v0y, n, n_reach;
};
// A far match's target relative to v0 (components below 2^33), from its pixel.  Out of line (rare).
__device__ __noinline__ longlong2 far_target(const WindowFar* far, float x, float y) {
    const int ux = exact_int(x), uy = exact_int(y);
    const int2 v = far->nnf[(far->oy + uy) * far->W + far->ox + ux];
    return make_longlong2((long long)v.x - far->v0x + ux, (long long)v.y - far->v0y + uy);
}
// The window's matches in raster order, in shared memory, as planes of floats holding exact integers (so a lane
// loads four consecutive matches with one 16-byte load per plane): the pixel u in window coordinates, and its
// target u + v relative to the window's reference offset v0.  An imported offset may be any integer: a match whose
// target is beyond kNearReach of v0 is far, its target in the planes is kFarTarget (no hypothesis counts it), and
// far_target reads its offset again.  A window with far matches is left to the FAR instances of the kernels and functions
// below, so that the others keep their registers and code (with both in one kernel 512x384 planes took 3.86 ms, with a
// launch each 3.64; without any far matches to serve 3.54).
// Entries past N, up to the next multiple of `pad`, are no match's inlier.
struct Window {
    float *x, *y, *qx, *qy;
    const WindowFar* far;
    int N;
    float U;     // half the window side: bounds |u|
    float vq;    // largest component of |u + v - v0| among the near matches
    float vmax;  // largest component of |v|
    __device__ __forceinline__ bool is_far(int j) const { return qx[j] == kFarTarget; }
    // a near match, its offset relative to v0
    __device__ __forceinline__ float4 match(int j) const {
        const float a = x[j], b = y[j];
        return make_float4(a, b, qx[j] - a, qy[j] - b);
    }
    __device__ __forceinline__ longlong2 far_target(int j) const { return gpm::far_target(far, x[j], y[j]); }
    // any match's target relative to v0
    __device__ __forceinline__ longlong2 target(int j) const {
        return is_far(j) ? far_target(j) : make_longlong2(exact_int(qx[j]), exact_int(qy[j]));
    }
};

// For a window with far matches: the reference is moved to one of the eight matches (offset mx, my of the lane) if more are
// near that one (planes still in integers).  Samples that mix places are bounded by how many matches are far: with at most
// half of them, most are dropped by the bound.
template <class G>
__device__ __forceinline__ void choose_reference(const G& grp, const Window& w, int mx, int my, int& v0x, int& v0y) {
    auto near = [&](int x, int y) {
        int n = 0;
        for (int j = grp.rank(); j < w.N; j += G::size)
            n += max(llabs((long long)__float_as_int(w.qx[j]) - x), llabs((long long)__float_as_int(w.qy[j]) - y)) < kNearReach / 2;
        return grp.sum(n);
    };
    int most = near(v0x, v0y);
    for (int l = 0; l < 8 && 2 * most < w.N; ++l) {  // uniform over the window
        const int x = __shfl_sync(FULL, mx, l), y = __shfl_sync(FULL, my, l), n = near(x, y);
        if (n > most) most = n, v0x = x, v0y = y;
    }
}

// Which windows an instance of the fit kernels serves: of a field whose matches cannot be far from each other; of any
// field, leaving those with far matches (kFarPending); the windows left.  (Pairs through FIT_ANY: 1024x436 15.14 -> 15.32
// ms against the code without far matches, 1.2 %; through FIT_NEAR 0.8 %, 0.5 of it the shared bound's broadcast.)
enum FitMode { FIT_NEAR, FIT_ANY, FIT_FAR };

// Gathers the window's matches (stage 1: every pixel; stage 2: the residual ones) into planes of `cap` floats.
template <int MODE, class G>
__device__ __forceinline__ void gather_window(const G& grp, const PairView& pv, const LevelGeom& g, int stage, int dir,
                                              int cell, float* planes, int cap, int pad, WindowFar* far, Window& w) {
    const int tid = grp.rank(), s = g.s, W = pv.W;
    int x0, y0, ox, oy;
    window_origin<G>(g, cell, x0, y0, ox, oy);
    const int2* nnf = pv.nnf[dir];
    const uint8_t* resid = pv.resid[dir];
    w.x = planes;
    w.y = planes + cap;
    w.qx = planes + 2 * cap;
    w.qy = planes + 3 * cap;
    w.far = far;
    int N = 0;
    for (int base = 0; base < s * s; base += G::size) {
        const int j = base + tid;
        bool take = j < s * s;
        const int yl = j / s, xl = j - yl * s, i = (y0 + yl) * W + x0 + xl;
        int at = j, total = min(G::size, s * s - base);
        if (stage != 1) {
            take = take && resid[i];
            at = N + grp.scan(take, total);
        }
        if (take) {
            const int2 v = nnf[i];
            w.x[at] = (float)(x0 + xl - ox);
            w.y[at] = (float)(y0 + yl - oy);
            w.qx[at] = __int_as_float(v.x);  // integers until the reference is known
            w.qy[at] = __int_as_float(v.y);
        }
        N += total;
    }
    w.N = N;
    w.U = 0.5f * (float)s;
    grp.sync();
    // reference offset: the component-wise median of eight matches spread over the list (any value is correct;
    // one near the window's main motion keeps the rounding bounds of its hypotheses small and few matches far)
    int mx = 0, my = 0;
    if (N > 0) {
        const int lane = tid & 31, j = ((2 * (lane & 7) + 1) * N) >> 4;
        mx = __float_as_int(w.qx[j]);
        my = __float_as_int(w.qy[j]);
    }
    int rx = 0, ry = 0;
#pragma unroll
    for (int l = 0; l < 8; ++l) {
        const int a = __shfl_sync(FULL, mx, l), b = __shfl_sync(FULL, my, l);
        const bool before = l < (int)(threadIdx.x & 7);
        rx += a < mx || (a == mx && before);
        ry += b < my || (b == my && before);
    }
    int v0x = __shfl_sync(FULL, mx, __ffs(__ballot_sync(FULL, rx == 3)) - 1);
    int v0y = __shfl_sync(FULL, my, __ffs(__ballot_sync(FULL, ry == 3)) - 1);
    if constexpr (MODE == FIT_FAR) choose_reference(grp, w, mx, my, v0x, v0y);
    if (tid == 0) *far = WindowFar{nnf, W, ox, oy, v0x, v0y, 0, 0};
    grp.sync();
    unsigned vm = 0, vq = 0;
    int n_far = 0;  // and those in reach, times 2^16
    for (int j = tid; j < N; j += G::size) {
        const int vx = __float_as_int(w.qx[j]), vy = __float_as_int(w.qy[j]);
        const int dx = (int)((unsigned)vx - (unsigned)v0x), dy = (int)((unsigned)vy - (unsigned)v0y);
        const int bx = (int)((unsigned)dx + (unsigned)exact_int(w.x[j])), by = (int)((unsigned)dy + (unsigned)exact_int(w.y[j]));
        vm = max(vm, max((unsigned)abs(vx), (unsigned)abs(vy)));
        // in range, and the subtractions did not wrap
        const bool near = MODE == FIT_NEAR ||
                          (max((unsigned)(bx + kNearReach), (unsigned)(by + kNearReach)) <= 2u * kNearReach &&
                           (((vx ^ v0x) & (vx ^ dx)) | ((vy ^ v0y) & (vy ^ dy))) >= 0);
        if (near)
            vq = max(vq, (unsigned)max(abs(bx), abs(by)));
        else  // rounded: at the limit it may count as in reach without being so
            n_far += fmaxf(fabsf((float)vx - (float)v0x), fabsf((float)vy - (float)v0y)) > 1.02f * (float)kFarthest ? 1 : 0x10001;
        w.qx[j] = near ? (float)bx : kFarTarget;
        w.qy[j] = near ? (float)by : kFarTarget;
    }
    for (int j = N + tid; j < (N + pad - 1) / pad * pad; j += G::size) {
        w.x[j] = w.y[j] = 0.f;
        w.qx[j] = w.qy[j] = kFarTarget;
    }
    w.vmax = (float)grp.max(vm);
    unsigned reach = grp.max(n_far ? 1u << 14 : vq);  // vq is below 2^14
    if (MODE != FIT_NEAR && reach >> 14) {  // uniform over the window
        n_far = grp.sum(n_far);
        if (tid == 0) far->n = n_far & 0xFFFF, far->n_reach = n_far >> 16;
        reach = grp.max(vq);
    }
    w.vq = (float)reach;
    grp.sync();
}

// ---- hypotheses
// Four Philox indices into the N matches of a window.
__device__ __forceinline__ void draw_indices(int N, int cell, int k, uint32_t tag, uint32_t pair_id, uint32_t k0,
                                             uint32_t k1, int idx[4]) {
    const uint4 r = philox((uint32_t)cell, (uint32_t)k, tag, pair_id, k0, k1);
    idx[0] = (int)bounded_u32(r.x, (uint32_t)N);
    idx[1] = (int)bounded_u32(r.y, (uint32_t)N);
    idx[2] = (int)bounded_u32(r.z, (uint32_t)N);
    idx[3] = (int)bounded_u32(r.w, (uint32_t)N);
}

// Hypothesis k of a window, exact (128-bit integers, hyp_exact.cuh), from window coordinates to targets relative to v0;
// false if the sample is degenerate (three source or three target points collinear).
__device__ __forceinline__ bool draw_exact(const Window& w, int cell, int k, uint32_t tag, uint32_t pair_id,
                                           uint32_t k0, uint32_t k1, i128* Hk) {
    int idx[4], px[4], py[4], qx[4], qy[4];
    draw_indices(w.N, cell, k, tag, pair_id, k0, k1, idx);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        px[j] = exact_int(w.x[idx[j]]);
        py[j] = exact_int(w.y[idx[j]]);
        qx[j] = exact_int(w.qx[idx[j]]);
        qy[j] = exact_int(w.qy[idx[j]]);
    }
    bool degen = false;
    const int T3[4][3] = {{0, 1, 2}, {0, 1, 3}, {0, 2, 3}, {1, 2, 3}};
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        const int a = T3[t][0], b = T3[t][1], c = T3[t][2];
        degen |= collinear3(px[a], py[a], px[b], py[b], px[c], py[c]);
        degen |= collinear3(qx[a], qy[a], qx[b], qy[b], qx[c], qy[c]);
    }
    if (degen) return false;
    minimal_h_exact(px, py, qx, qy, Hk);
    return true;
}

// Hypothesis k of a window with far matches, whose targets are read from their own integers, as its FP64 and its evaluation
// form; false also if the targets are too far apart for the products (sample_in_range) or the denominator is 0 at the
// centre.  middle: sample_centre.  Out of line.
__device__ __noinline__ bool solve_far(const Window& w, int cell, int k, uint32_t tag, uint32_t pair_id, uint32_t k0,
                                       uint32_t k1, double* Hl, Mef& m, longlong2& middle) {
    int idx[4], px[4], py[4];
    int64_t qx[4], qy[4];
    draw_indices(w.N, cell, k, tag, pair_id, k0, k1, idx);
#pragma unroll 1
    for (int j = 0; j < 4; ++j) {
        px[j] = exact_int(w.x[idx[j]]);
        py[j] = exact_int(w.y[idx[j]]);
        const longlong2 q = w.target(idx[j]);
        qx[j] = q.x;
        qy[j] = q.y;
    }
    auto q = [&](int j) { return make_longlong2(qx[j], qy[j]); };
    middle = sample_centre(q(0), q(1), q(2), q(3));
    bool degen = false;
#pragma unroll 1
    for (int t = 0; t < 4; ++t) {
        const int a = t == 3 ? 1 : 0, b = t < 2 ? 1 : 2, c = t == 0 ? 2 : 3;
        degen |= collinear3(px[a], py[a], px[b], py[b], px[c], py[c]);
        degen |= (i128)(qx[b] - qx[a]) * (qy[c] - qy[a]) == (i128)(qy[b] - qy[a]) * (qx[c] - qx[a]);
    }
    if (degen || !sample_in_range(qx, qy, max(llabs((long long)w.far->v0x), llabs((long long)w.far->v0y)))) return false;
    i128 Hk[9];
    minimal_h_exact(px, py, qx, qy, Hk);
    if (!make_mef_exact(Hk, m)) return false;
    exact_local_fp64(Hk, Hl);
    return true;
}

// A hypothesis in FP32, for scoring: den(u) = c0 + g0 ux + g1 uy (positive at the window centre), the target
// relative to v0 times den, X(u) = xc + x0 ux + x1 uy and Y(u) likewise, and kap, a bound of everything rounding
// can do to the inlier test: with n = (X - qx den, Y - qy den), an inlier has |n| < t den, so it passes
// |n| <= t den + kap as computed, and a match that passes |n| < t den - kap as computed is an inlier.  kap is for the
// near matches.  For a far one (FAR only) it is 1.2 kap + far_kap |q|_1; away: the sample's centre is far.
struct FastHyp {
    float g0, g1, c0, kap, x0, x1, xc, far_kap, y0, y1, yc;
    int away;
};
enum { HYP_DEAD = 0, HYP_OK = 1, HYP_LOOSE = 2 };  // degenerate; scored in FP32; the FP32 form says too little
// t widened by 2^-20: covers the relative roundings of both sides of the comparison (at most 6 units of 2^-24).
__device__ __forceinline__ float t_above(float t2) { return sqrtf(t2) * (1.f + 9.5367431640625e-07f); }
__device__ __forceinline__ float t_below(float t2) { return sqrtf(t2) * (1.f - 9.5367431640625e-07f); }

// A hypothesis solved in FP32.  Relative to the fourth pair (p3, q3), with the cross products l_k, mu_k of
// hyp_exact.cuh (exact: floats below 2^24 and integers) and rho_k = mu_k / (M l_k), M = sum mu, the form's
// coefficients are sums over k of rho_k (dy_i - dy_j), rho_k (dx_j - dx_i) and their products with the target
// differences, normalised to 1 at p3.
// Rounding, in units of u = 2^-24, first order: mu, M, M l one each, the division 4 (2 ulp): rho 7; a product with
// an exact integer 8, the sums 11 (g) and 12 (h00..h11).  With e_k = |rho_k| (|dy_i - dy_j| + |dx_j - dx_i|),
// S = U sum e_k and SQ = U sum e_k (|X_k| + |Y_k|): den carries at most 28 (1 + S), X and Y together at most
// 32 (SQ + |q3|_1 (1 + S)), n in addition |q|_1 28 (1 + S).  A match that can pass has
// |q|_1 <= (|X| + |Y|) / den + 2 t, which the window's extremes of the form bound where den stays positive; else
// the window's largest |q| does.  (34 and 30 below leave the second order room.)
// FAR_SAMPLE: mu and M are within 2 units and the target differences are rounded themselves, which makes 15 of the 12
// above: the bounds are taken half as large again.
template <bool FAR, bool FAR_SAMPLE>
__device__ __forceinline__ int solve_form(const Window& w, float p3x, float p3y, float q3x, float q3y, const float (&dx)[3],
                                          const float (&dy)[3], const float (&X)[3], const float (&Y)[3],
                                          const float (&l)[3], const float (&mu)[3], float M, float t, FastHyp& h) {
    float S = 0.f, SQ = 0.f, h00 = 0.f, h01 = 0.f, h10 = 0.f, h11 = 0.f;
    h.g0 = h.g1 = 0.f;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const int a = (j + 1) % 3, b = (j + 2) % 3;
        const float rho = __fdividef(mu[j], M * l[j]);
        const float al = rho * (dy[a] - dy[b]), be = rho * (dx[b] - dx[a]);
        const float e = fabsf(al) + fabsf(be);
        S += e;
        SQ = fmaf(e, fabsf(X[j]) + fabsf(Y[j]), SQ);
        h.g0 += al;
        h.g1 += be;
        h00 = fmaf(al, X[j], h00);
        h01 = fmaf(be, X[j], h01);
        h10 = fmaf(al, Y[j], h10);
        h11 = fmaf(be, Y[j], h11);
    }
    h.c0 = fmaf(-h.g1, p3y, fmaf(-h.g0, p3x, 1.f));
    h.x0 = fmaf(q3x, h.g0, h00);
    h.x1 = fmaf(q3x, h.g1, h01);
    h.xc = fmaf(-h01, p3y, fmaf(-h00, p3x, q3x * h.c0));
    h.y0 = fmaf(q3y, h.g0, h10);
    h.y1 = fmaf(q3y, h.g1, h11);
    h.yc = fmaf(-h11, p3y, fmaf(-h10, p3x, q3y * h.c0));
    const float u = (FAR_SAMPLE ? 1.5f : 1.f) * 5.9604644775390625e-08f, U = w.U;
    const float one = fmaf(U, S, 1.f), ed = 30.f * u * one;
    const float dc = h.c0 - 0.5f * (h.g0 + h.g1);
    if (!(fabsf(dc) > 2.f * ed)) return HYP_LOOSE;  // its orientation needs the exact form
    if (dc < 0.f) {
        h.g0 = -h.g0, h.g1 = -h.g1, h.c0 = -h.c0;
        h.x0 = -h.x0, h.x1 = -h.x1, h.xc = -h.xc;
        h.y0 = -h.y0, h.y1 = -h.y1, h.yc = -h.yc;
    }
    const float dmin = h.c0 - (fabsf(h.g0) + fabsf(h.g1)) * U - 2.f * ed;
    float Q = 2.f * w.vq;
    if (dmin > 0.f) {
        const float XY = fabsf(h.xc) + fabsf(h.yc) + (fabsf(h.x0) + fabsf(h.x1) + fabsf(h.y0) + fabsf(h.y1)) * U;
        Q = fminf(Q, __fdividef(1.05f * XY + t, dmin) + 2.2f * t);
    }
    h.kap = 1.0001f * fmaf(34.f * u, fmaf(fabsf(q3x) + fabsf(q3y) + Q, one, SQ * U), t * ed);
    if (FAR) h.far_kap = 40.f * u * one;  // the target rounded itself; the rest of kap grows from 34 to 40 u
    // a wide bound still excludes most (far targets are up to 2^18 times as far); NaN: loose
    return h.kap < (FAR_SAMPLE ? 1e14f : 1e6f) ? HYP_OK : HYP_LOOSE;
}

// A sample with far targets, solved relative to a near one, so that q3 is small and the far targets' differences come with
// a small rho_k of their own: the bound is not much wider than for near samples.  With targets out of reach of each other
// it is solved relative to the one next to the centre, since three of them together make every rho_k large otherwise.
// 512x384 planes (3.67 ms without markers) with 15 and 50 % at 2^20: 42 -> 9.3 and 287 -> 76 ms; at 2^30, 50 %: 68.
__device__ __forceinline__ int far_hypothesis(const Window& w, const int (&idx)[4], float t, FastHyp& h) {
    longlong2 q[4];
    bool apart = false, any_near = false;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        q[j] = w.target(idx[j]);
        apart = apart || out_of_reach(q[j], make_longlong2(0, 0));
        any_near = any_near || !w.is_far(idx[j]);
    }
    const longlong2 c = sample_centre(q[0], q[1], q[2], q[3]);
    h.away = max(llabs(c.x), llabs(c.y)) > kNearReach;
    const longlong2 at = apart || !any_near ? c : make_longlong2(0, 0);
    int r = 0, i3 = idx[0];
    longlong2 q3 = q[0];
#pragma unroll
    for (int j = 1; j < 4; ++j)
        if (llabs(q[j].x - at.x) + llabs(q[j].y - at.y) < llabs(q3.x - at.x) + llabs(q3.y - at.y)) r = j, i3 = idx[j], q3 = q[j];
    const float p3x = w.x[i3], p3y = w.y[i3];
    float dx[3], dy[3], X[3], Y[3], l[3], mu[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const int i = j == r ? idx[3] : idx[j];
        if (j == r) q[j] = q[3];
        dx[j] = w.x[i] - p3x;
        dy[j] = w.y[i] - p3y;
        X[j] = (float)(q[j].x - q3.x);
        Y[j] = (float)(q[j].y - q3.y);
    }
    i128 M = 0;
    bool degen = false;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const int a = (j + 1) % 3, b = (j + 2) % 3;
        const i128 m = (i128)(q[a].x - q3.x) * (q[b].y - q3.y) - (i128)(q[b].x - q3.x) * (q[a].y - q3.y);
        l[j] = dx[a] * dy[b] - dx[b] * dy[a];
        M += m;
        mu[j] = i128_to_float(m);
        degen |= l[j] == 0.f || m == 0;
    }
    if (degen || l[0] + l[1] + l[2] == 0.f || M == 0) return HYP_DEAD;
    return solve_form<true, true>(w, p3x, p3y, (float)q3.x, (float)q3.y, dx, dy, X, Y, l, mu, i128_to_float(M), t, h);
}

// Draws hypothesis k and solves it in FP32.  The degeneracy test is exact: the eight triangle areas are the l_k, the mu_k
// and their sums.
template <bool FAR>
__device__ __forceinline__ int fast_hypothesis(const Window& w, int cell, int k, uint32_t tag, uint32_t pair_id,
                                               uint32_t k0, uint32_t k1, float t, FastHyp& h) {
    int idx[4];
    draw_indices(w.N, cell, k, tag, pair_id, k0, k1, idx);
    if (FAR && (w.is_far(idx[0]) || w.is_far(idx[1]) || w.is_far(idx[2]) || w.is_far(idx[3])))
        return far_hypothesis(w, idx, t, h);
    if (FAR) h.away = 0;
    const float p3x = w.x[idx[3]], p3y = w.y[idx[3]], q3x = w.qx[idx[3]], q3y = w.qy[idx[3]];
    float dx[3], dy[3], X[3], Y[3], l[3], mu[3];
    int Xi[3], Yi[3], M = 0;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        dx[j] = w.x[idx[j]] - p3x;
        dy[j] = w.y[idx[j]] - p3y;
        X[j] = w.qx[idx[j]] - q3x;
        Y[j] = w.qy[idx[j]] - q3y;
        Xi[j] = exact_int(X[j]);
        Yi[j] = exact_int(Y[j]);
    }
    bool degen = false;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const int a = (j + 1) % 3, b = (j + 2) % 3;
        l[j] = dx[a] * dy[b] - dx[b] * dy[a];
        const int m = Xi[a] * Yi[b] - Xi[b] * Yi[a];
        M = (int)((unsigned)M + (unsigned)m);
        mu[j] = (float)m;
        degen |= l[j] == 0.f || m == 0;
    }
    if (degen || l[0] + l[1] + l[2] == 0.f || M == 0) return HYP_DEAD;
    return solve_form<FAR, false>(w, p3x, p3y, q3x, q3y, dx, dy, X, Y, l, mu, (float)M, t, h);
}

// The form of a hypothesis with every coefficient in both halves of a pair, for tests of two matches per
// instruction on the packed FP32x2 pipe; the denominator negated, so that no product needs a sign change.
struct PairHyp {
    float2 g0, g1, c0, kap, x0, x1, xc, y0, y1, yc;
};
__device__ __forceinline__ float2 both(float v) { return make_float2(v, v); }
__device__ __forceinline__ PairHyp pair_hyp(const FastHyp& h) {
    PairHyp p;
    p.g0 = both(-h.g0), p.g1 = both(-h.g1), p.c0 = both(-h.c0), p.kap = both(-h.kap);
    p.x0 = both(h.x0), p.x1 = both(h.x1), p.xc = both(h.xc);
    p.y0 = both(h.y0), p.y1 = both(h.y1), p.yc = both(h.yc);
    return p;
}
// How many of two matches can be inliers: 12 FP32 operations a match (three linear forms, two residuals, the
// comparison squared with a negative radius cut to zero), the count from the sign bit of |n|^2 - radius^2.
__device__ __forceinline__ void count_pair(const PairHyp& h, float2 t, float2 ux, float2 uy, float2 qx, float2 qy,
                                           int& cnt) {
    const float2 nd = __ffma2_rn(h.g1, uy, __ffma2_rn(h.g0, ux, h.c0));  // -den
    const float2 nx = __ffma2_rn(qx, nd, __ffma2_rn(h.x1, uy, __ffma2_rn(h.x0, ux, h.xc)));
    const float2 ny = __ffma2_rn(qy, nd, __ffma2_rn(h.y1, uy, __ffma2_rn(h.y0, ux, h.yc)));
    const float2 m = __ffma2_rn(t, nd, h.kap);  // -(t den + kap)
    const float2 n2 = __ffma2_rn(nx, nx, __fmul2_rn(ny, ny));
    const float ma = fminf(m.x, 0.f), mb = fminf(m.y, 0.f);
    cnt += (int)(__float_as_uint(fmaf(-ma, ma, n2.x)) >> 31) + (int)(__float_as_uint(fmaf(-mb, mb, n2.y)) >> 31);
}
// The same for the four matches from index j (a multiple of 4).
__device__ __forceinline__ void count_quad(const Window& w, const PairHyp& h, float2 t, int j, int& cnt) {
    const float4 x = *reinterpret_cast<const float4*>(w.x + j), y = *reinterpret_cast<const float4*>(w.y + j);
    const float4 a = *reinterpret_cast<const float4*>(w.qx + j), b = *reinterpret_cast<const float4*>(w.qy + j);
    count_pair(h, t, make_float2(x.x, x.y), make_float2(y.x, y.y), make_float2(a.x, a.y), make_float2(b.x, b.y), cnt);
    count_pair(h, t, make_float2(x.z, x.w), make_float2(y.z, y.w), make_float2(a.z, a.w), make_float2(b.z, b.w), cnt);
}

// One match against a scored hypothesis: sure (an inlier whatever the rounding) and maybe (possibly one).
__device__ __forceinline__ void test_match(const Window& w, const FastHyp& h, float tl, float th, int j, bool& sure,
                                           bool& maybe) {
    const float ux = w.x[j], uy = w.y[j];
    const float den = fmaf(h.g1, uy, fmaf(h.g0, ux, h.c0));
    const float nx = fmaf(-w.qx[j], den, fmaf(h.x1, uy, fmaf(h.x0, ux, h.xc)));
    const float ny = fmaf(-w.qy[j], den, fmaf(h.y1, uy, fmaf(h.y0, ux, h.yc)));
    const float n2 = fmaf(nx, nx, ny * ny);
    const float a = fmaf(th, den, h.kap), b = fmaf(tl, den, -h.kap);
    maybe = a > 0.f && n2 < a * a;
    sure = b > 0.f && n2 < b * b;
}

// How many far matches a scored hypothesis may have as inliers: those in reach, unless its targets in the window stay near
// (the bound on them in solve_form, with kap / t for ed, which is below it).
__device__ __forceinline__ int far_allowance(const Window& w, const FastHyp& h, float t) {
    if (h.away) return w.far->n;
    const float dmin = h.c0 - (fabsf(h.g0) + fabsf(h.g1)) * w.U - 2.f * h.kap / t;
    const float XY = fabsf(h.xc) + fabsf(h.yc) + (fabsf(h.x0) + fabsf(h.x1) + fabsf(h.y0) + fabsf(h.y1)) * w.U;
    return dmin > 0.f && 1.05f * XY + t + 2.2f * t * dmin < 0.999f * (float)kNearReach * dmin ? 0 : w.far->n_reach;
}
// Whether a far match can be an inlier of a scored hypothesis.
__device__ __forceinline__ bool far_maybe(const Window& w, const FastHyp& h, float t, int j) {
    const longlong2 q = w.far_target(j);
    const float ux = w.x[j], uy = w.y[j], qx = (float)q.x, qy = (float)q.y;
    const float den = fmaf(h.g1, uy, fmaf(h.g0, ux, h.c0));
    const float nx = fmaf(-qx, den, fmaf(h.x1, uy, fmaf(h.x0, ux, h.xc)));
    const float ny = fmaf(-qy, den, fmaf(h.y1, uy, fmaf(h.y0, ux, h.yc)));
    const float a = fmaf(t, den, 1.001f * fmaf(h.far_kap, fabsf(qx) + fabsf(qy), 1.2f * h.kap));
    const bool reach = h.away || fmaxf(fabsf(qx), fabsf(qy)) < 1.01f * (float)kFarthest;
    return reach && a > 0.f && fmaf(nx, nx, ny * ny) < a * a;
}

// The order of two hypotheses: more inliers, then the lower index.  Zero is below every hypothesis.
__device__ __forceinline__ unsigned long long hyp_key(int score, int k) {
    return ((unsigned long long)(unsigned)(score + 1) << 32) | (unsigned long long)(0xFFFFFFFFu - (uint32_t)k);
}
__device__ __forceinline__ int key_score(unsigned long long key) { return (int)(key >> 32) - 1; }
__device__ __forceinline__ int key_index(unsigned long long key) {
    return (int)(0xFFFFFFFFu - (uint32_t)(key & 0xFFFFFFFFull));
}

// The certified test of a match by the exact hypothesis: its FP32 evaluation form, and FP64 (Hl) where that is
// within its rounding bound.
__device__ __forceinline__ bool exact_inlier(const Mef& m, const double* Hl, const float4& mt, float t2, int& nfp64) {
    bool unc;
    const bool in = cert_inlier(m, mt, t2, unc);
    if (!unc) return in;
    ++nfp64;
    return hyp_inlier_fp64(Hl, mt.x, mt.y, mt.z, mt.w, (double)t2);
}

// The test of any match by a hypothesis in FP64 (middle: its sample's centre), a far one from its own integers.
__device__ __forceinline__ bool inlier_fp64(const Window& w, const double* Hl, longlong2 middle, int j, float t2) {
    const longlong2 q = w.target(j);
    return !out_of_reach(q, middle) &&
           hyp_inlier_fp64(Hl, (double)w.x[j], (double)w.y[j], (double)q.x, (double)q.y, (double)t2);
}

// What a warp counts of its work (profiling counters).
struct RansacStats {
    int tests = 0, fp64 = 0, loose = 0;
};

// The exact support of hypothesis k, by one warp: -1 if its sample is degenerate, or as soon as it cannot reach
// `floor` (a key).  Out of line: for the few hypotheses that contend with uncertain tests, and the loose ones.
template <bool FAR>
__device__ __noinline__ int exact_support(const Window& w, int cell, int k, uint32_t tag, uint32_t pair_id,
                                          uint32_t k0, uint32_t k1, float t2, unsigned long long floor,
                                          RansacStats& st) {
    const int lane = threadIdx.x & 31;
    double Hl[9];
    Mef m;
    longlong2 middle = make_longlong2(0, 0);
    if constexpr (FAR) {
        if (!solve_far(w, cell, k, tag, pair_id, k0, k1, Hl, m, middle)) return -1;
    } else {
        i128 Hk[9];
        if (!draw_exact(w, cell, k, tag, pair_id, k0, k1, Hk) || !make_mef_exact(Hk, m)) return -1;
        exact_local_fp64(Hk, Hl);
    }
    mef_set_bounds(m, w.U, w.vq + w.U, t2);
    int score = 0, f = 0;
    for (int c = 0; c < w.N; c += 128) {
#pragma unroll 1
        for (int j = c + lane; j < c + 128 + lane; j += 32) {
            bool in = false;
            if (FAR && j < w.N && w.is_far(j)) {
                in = inlier_fp64(w, Hl, middle, j, t2);
                ++f;
            } else if (j < w.N && !(FAR && out_of_reach(w.target(j), middle))) {
                in = exact_inlier(m, Hl, w.match(j), t2, f);
            }
            score += __popc(__ballot_sync(FULL, in));
        }
        st.tests += min(128, w.N - c);
        if (hyp_key(score + max(w.N - c - 128, 0), k) < floor) return -1;
    }
    st.fp64 += (int)__reduce_add_sync(FULL, (unsigned)f);
    return score;
}

// The support of scored hypothesis k (its form in `form`, shared memory), by one warp: the FP32 count if no test is
// uncertain, else exact; -1 if it cannot reach `floor`.  Out of line (contenders only).
template <bool FAR>
__device__ __noinline__ int contender_support(const Window& w, const FastHyp* form, int cell, int k, uint32_t tag,
                                              uint32_t pair_id, uint32_t k0, uint32_t k1, float t2,
                                              unsigned long long floor, RansacStats& st) {
    const FastHyp h = *form;
    const float tl = t_below(t2), th = t_above(t2);
    int lo = 0, hi = 0;
    for (int j = threadIdx.x & 31; j < w.N; j += 32) {
        bool sure = false, maybe;
        if (FAR && w.is_far(j))
            maybe = far_maybe(w, h, th, j);
        else
            test_match(w, h, tl, th, j, sure, maybe);
        lo += sure && !(FAR && h.away);  // it may be out of reach
        hi += maybe;
    }
    lo = (int)__reduce_add_sync(FULL, (unsigned)lo);
    hi = (int)__reduce_add_sync(FULL, (unsigned)hi);
    st.tests += w.N;
    if (hyp_key(hi, k) < floor) return -1;
    return hi == lo ? lo : exact_support<FAR>(w, cell, k, tag, pair_id, k0, k1, t2, floor, st);
}

// The window's matches in raster order into `match`; returns their number.
template <class G>
__device__ int gather_matches(const G& grp, const PairView& pv, const LevelGeom& g, int stage, int dir, int cell,
                              float4* match) {
    const int tid = grp.rank();
    const int s = g.s;
    int x0, y0, ox, oy;
    window_origin<G>(g, cell, x0, y0, ox, oy);
    const int W = pv.W;
    const int2* nnf = pv.nnf[dir];
    const uint8_t* resid = pv.resid[dir];
    int N = 0;
    for (int base = 0; base < s * s; base += G::size) {
        const int j = base + tid;
        bool take = false;
        float4 mt = make_float4(0, 0, 0, 0);
        if (j < s * s) {
            const int yy = y0 + j / s, xx = x0 + j % s;
            const int i = yy * W + xx;
            take = stage == 1 || resid[i];
            const int2 v = nnf[i];
            mt = make_float4((float)(xx - ox), (float)(yy - oy), (float)v.x, (float)v.y);
        }
        int total;
        const int off = grp.scan(take, total);
        if (take) match[N + off] = mt;
        N += total;
    }
    grp.sync();
    return N;
}

// An integer in [1, 2^62] as a double, from its bits; above 2^53 it is converted, rounded once.
__device__ __forceinline__ double double_of(long long K) {
    const int lz = __clzll(K);
    const unsigned long long m = (unsigned long long)K << lz;
    if (m & 0x7FFull) return (double)K;
    return __longlong_as_double(((long long)(1085 - lz) << 52) + (long long)(m >> 11));
}

// Sum of |(a, b)| over a lane's points, for exact integers a, b: each root of
// the sum of squares K (exact in 64-bit integers, rounded once to FP64 above
// 2^53) to about 1e-14 relative, added in FP64.  The least-squares refit of a thin, ill-conditioned support
// moves with its Hartley normalisation, so the scale must carry far less than
// FP32 rounding (with FP32 roots, refits moved by ~1e-6).  The root: the FP32
// root s0 and reciprocal 1 / (2 s0), then one Newton step in FP64,
// s0 + (K - s0^2) / (2 s0): its error is about s0 times the square of s0's
// relative error (2^-23), for three FP64 operations.
__device__ __forceinline__ void add_dist(double& s, int a, int b) {
    const long long K = (long long)a * a + (long long)b * b;  // exact: |a|, |b| < 2^31
    const float fa = (float)a, fb = (float)b;
    const float s0 = sqrtf(fmaf(fa, fa, fb * fb));
    if (!(s0 > 0.f)) return;  // K = 0
    const double sd = double_of(s0);
    const double e = fma(-sd, sd, double_of(K));
    s += fma(e, double_of(0.5f / s0), sd);
}

// The warp's totals of the lanes' 24 moments, one on each lane whose low two index bits are below 3 (`slot`: its
// index): five exchange steps halve what a lane keeps, 24 exchanges in all instead of 120.
__device__ __forceinline__ long long warp_moments(const long long (&R)[24], int& slot) {
    const int lane = threadIdx.x & 31;
    long long a[12], b[6], c[4], d[2];
    auto step = [&](bool hi, long long lo_v, long long hi_v, int off) {
        const long long send = hi ? lo_v : hi_v;
        return (hi ? hi_v : lo_v) + __shfl_xor_sync(FULL, send, off);
    };
#pragma unroll
    for (int q = 0; q < 12; ++q) a[q] = step(lane & 16, R[q], R[q + 12], 16);
#pragma unroll
    for (int q = 0; q < 6; ++q) b[q] = step(lane & 8, a[q], a[q + 6], 8);
#pragma unroll
    for (int q = 0; q < 3; ++q) c[q] = step(lane & 4, b[q], b[q + 3], 4);
    c[3] = 0;
#pragma unroll
    for (int q = 0; q < 2; ++q) d[q] = step(lane & 2, c[q], c[q + 2], 2);
    const int low = lane & 3;
    slot = low < 3 ? ((lane & 16) ? 12 : 0) + ((lane & 8) ? 6 : 0) + ((lane & 4) ? 3 : 0) + low : -1;
    return step(lane & 1, d[0], d[1], 1);
}
// Totals of the 24 moments over the group, into out; scratch: 24 values per warp (blocks).
__device__ __forceinline__ void group_moments(const WarpGroup&, const long long (&R)[24], long long*, long long* out) {
    int q;
    const long long t = warp_moments(R, q);
    if (q >= 0) out[q] = t;
}
template <int NT>
__device__ __forceinline__ void group_moments(const BlockGroup<NT>&, const long long (&R)[24], long long* scratch,
                                              long long* out) {
    int q;
    const long long t = warp_moments(R, q);
    if (q >= 0) scratch[(threadIdx.x >> 5) * 24 + q] = t;
    __syncthreads();
    if (threadIdx.x < 24) {
        long long v = 0;
        for (int w = 0; w < NT / 32; ++w) v += scratch[w * 24 + threadIdx.x];
        out[threadIdx.x] = v;
    }
}
// The warp's sums of two doubles, each added in the order of an exchange over lane distances 16, 8, 4, 2, 1, in one
// chain of five additions: lanes 0-15 keep the first, lanes 16-31 the second.
__device__ __forceinline__ double warp_sum_pair(double first, double second) {
    const bool hi = threadIdx.x & 16;
    double v = (hi ? second : first) + __shfl_xor_sync(FULL, hi ? first : second, 16);
#pragma unroll
    for (int off = 8; off > 0; off >>= 1) v += __shfl_xor_sync(FULL, v, off);
    return v;
}
__device__ __forceinline__ void group_dists(const WarpGroup&, double s, double t, double*, RefitWork* rw) {
    const double v = warp_sum_pair(s, t);
    if ((threadIdx.x & 31) == 0) rw->ds = v;
    if ((threadIdx.x & 31) == 16) rw->dt = v;
}
template <int NT>
__device__ __forceinline__ void group_dists(const BlockGroup<NT>&, double s, double t, double* scratch, RefitWork* rw) {
    const double v = warp_sum_pair(s, t);
    const int lane = threadIdx.x & 31;
    if ((lane & 15) == 0) scratch[(threadIdx.x >> 5) * 2 + (lane >> 4)] = v;
    __syncthreads();
    if (threadIdx.x < 2) {
        double a = 0;
        for (int w = 0; w < NT / 32; ++w) a += scratch[w * 2 + threadIdx.x];  // in warp order
        (threadIdx.x ? rw->dt : rw->ds) = a;
    }
}

constexpr int kFarPending = 1;  // RefitWork::status of a window with far matches that is yet to be fitted
// The window's model record, cleared before its fit.
__device__ __forceinline__ void clear_model(const PairView& pv, int dir, int id, int N, RefitWork* rw) {
    int* mi = pv.mi[dir] + (size_t)id * kMI;
    for (int k = 0; k < kMI; ++k) mi[k] = 0;
    mi[MI_NIN] = N;
    mi[MI_BESTK] = -1;
    for (int k = 0; k < 9; ++k) pv.mh[dir][(size_t)id * 9 + k] = 0.0;
    pv.mef[dir][id] = Mef{};
    rw->status = 0;
}

// The exact hypothesis k in FP64 (shared memory), by one warp: for the winner's uncertain tests.  Out of line (rare).
__device__ __noinline__ void winner_fp64(const Window& w, int cell, int k, uint32_t tag, uint32_t pair_id, uint32_t k0,
                                         uint32_t k1, double* whl) {
    i128 Hk[9];
    draw_exact(w, cell, k, tag, pair_id, k0, k1, Hk);
    double Hl[9];
    exact_local_fp64(Hk, Hl);
    if ((threadIdx.x & 31) == 0)
        for (int q = 0; q < 9; ++q) whl[q] = Hl[q];
}

// finish_fit's first part in a window with far matches: the winner's inliers among this thread's matches, all decided in
// FP64, its sample into rw, and, if there are far inliers, the inliers' targets in the planes about another reference, the
// offset of the winner's first match, now in v0: far inliers are near it.  wide: one is not within kPlaneReach of it (within
// it an inlier is at most 3/4 of their span from their mean, and squares stay below 2^30); then nothing is moved.
template <class G>
__device__ __forceinline__ unsigned long long far_winner(const G& grp, const Window& w, int cell, int k, uint32_t tag,
                                                      uint32_t pair_id, uint32_t k0, uint32_t k1, float t2, RefitWork* rw,
                                                      int2& v0, bool& wide) {
    constexpr int kPlaneReach = 20000;
    const int tid = grp.rank();
    double Hl[9];
    Mef m;
    longlong2 middle;
    solve_far(w, cell, k, tag, pair_id, k0, k1, Hl, m, middle);
    unsigned long long inm = 0;
    bool far = false;
    for (int j = tid, c = 0; j < w.N; j += G::size, ++c)
        if (inlier_fp64(w, Hl, middle, j, t2)) {
            inm |= 1ull << c;
            far = far || w.is_far(j);
        }
    int idx[4];
    draw_indices(w.N, cell, k, tag, pair_id, k0, k1, idx);
    if (tid < 4) {
        const int j = tid == 0 ? idx[0] : (tid == 1 ? idx[1] : (tid == 2 ? idx[2] : idx[3]));
        const longlong2 q = w.target(j);
        rw->sample[tid] = exact_int(w.x[j]);
        rw->sample[4 + tid] = exact_int(w.y[j]);
        rw->target[tid] = v0.x + q.x;
        rw->target[4 + tid] = v0.y + q.y;
    }
    wide = false;
    if (!grp.any(far)) return inm;
    longlong2 shift = w.target(idx[0]);
    shift.x -= exact_int(w.x[idx[0]]);
    shift.y -= exact_int(w.y[idx[0]]);
    for (unsigned long long b = inm; b; b &= b - 1) {
        const longlong2 q = w.target(tid + (__ffsll((long long)b) - 1) * G::size);
        wide = wide || max(llabs(q.x - shift.x), llabs(q.y - shift.y)) > kPlaneReach;
    }
    wide = grp.any(wide);
    grp.sync();  // the targets are read
    if (wide) return inm;
    for (unsigned long long b = inm; b; b &= b - 1) {
        const int j = tid + (__ffsll((long long)b) - 1) * G::size;
        const longlong2 q = w.target(j);
        w.qx[j] = (float)(int)(q.x - shift.x);
        w.qy[j] = (float)(int)(q.y - shift.y);
    }
    v0 = make_int2((int)(v0.x + shift.x), (int)(v0.y + shift.y));
    return inm;
}

// The refit's inputs for inliers whose targets are too far apart for 32 bits (a plane whose vanishing line passes by some of
// them): the same sums, the moments in 128 bits and stored as doubles (RefitWork::wide).
template <class G>
__device__ __noinline__ void wide_sums(const G& grp, const Window& w, unsigned long long inm, int nw, int2 v0, double* whl,
                                       RefitWork* rw) {
    const int tid = grp.rank();
    int sx = 0, sy = 0;
    long long tx = 0, ty = 0;
    for (unsigned long long b = inm; b; b &= b - 1) {
        const int j = tid + (__ffsll((long long)b) - 1) * G::size;
        const longlong2 q = w.target(j);
        sx += exact_int(w.x[j]);
        sy += exact_int(w.y[j]);
        tx += q.x;
        ty += q.y;
    }
    sx = grp.sum(sx);
    sy = grp.sum(sy);
    tx = grp.sum(tx);
    ty = grp.sum(ty);
    const double n = nw, lim = 2147483000.0;
    const int cx = __double2int_rn(sx / n), cy = __double2int_rn(sy / n);
    const int cu = __double2int_rn(fmin(fmax(tx / n + v0.x, -lim), lim));
    const int cv = __double2int_rn(fmin(fmax(ty / n + v0.y, -lim), lim));
    double ds = 0.0, dt = 0.0;
    for (unsigned long long b = inm; b; b &= b - 1) {
        const int j = tid + (__ffsll((long long)b) - 1) * G::size;
        const longlong2 q = w.target(j);
        const double ax = n * exact_int(w.x[j]) - sx, ay = n * exact_int(w.y[j]) - sy;
        const double bx = n * (double)q.x - (double)tx, by = n * (double)q.y - (double)ty;
        ds += sqrt(fma(ax, ax, ay * ay));
        dt += sqrt(fma(bx, bx, by * by));
    }
#pragma unroll 1
    for (int k = 0; k < 24; ++k) {
        i128 m = 0;
        for (unsigned long long b = inm; b; b &= b - 1) {
            const int j = tid + (__ffsll((long long)b) - 1) * G::size;
            const longlong2 q = w.target(j);
            const int X = exact_int(w.x[j]) - cx, Y = exact_int(w.y[j]) - cy;
            const long long U = q.x + v0.x - cu, V = q.y + v0.y - cv;
            const int e = k % 6, z = e == 0 ? X * X : (e == 1 ? X * Y : (e == 2 ? X : (e == 3 ? Y * Y : (e == 4 ? Y : 1))));
            m += (k < 6 ? (i128)1 : (k < 12 ? (i128)U : (k < 18 ? (i128)V : (i128)U * U + (i128)V * V))) * z;
        }
        i128 t = 0;  // the group's, by 32-bit limbs
#pragma unroll
        for (int l = 0; l < 4; ++l) {
            const long long limb = l < 3 ? (long long)(uint32_t)(m >> (32 * l)) : (long long)(m >> 96);
            t += (i128)grp.sum(limb) * ((i128)1 << (32 * l));
        }
        const bool neg = t < 0;
        const u128 a = neg ? (u128)0 - (u128)t : (u128)t;
        const double d = (double)(unsigned long long)(a >> 64) * 18446744073709551616.0 + (double)(unsigned long long)a;
        if (tid == 0) rw->mom[k] = __double_as_longlong(neg ? -d : d);
    }
    group_dists(grp, ds, dt, whl, rw);
    if (tid == 0) {
        rw->cx = cx;
        rw->cy = cy;
        rw->cu = cu;
        rw->cv = cv;
    }
}

// What follows the search: the refit's inputs on the winner's inliers (Hartley centroids as exact integer sums,
// distances, and the DLT moments as exact integers about the rounded centroids) and the winner's sample, from which
// the solve (a thread per window) forms the exact homography.  best: the winner's key, 0 if there is none; whl: 9
// doubles of shared memory; scratch: 24 values per warp of a block.
template <int MODE, class G>
__device__ __forceinline__ void finish_fit(const G& grp, const PairView& pv, const Window& w, const PlaneParams& pp,
                                           int dir, int cell, int id, uint32_t tag, unsigned long long best,
                                           const RansacStats& st, double* whl, long long* scratch, RefitWork* rw) {
    const int tid = grp.rank(), N = w.N;
    int* mi = pv.mi[dir] + (size_t)id * kMI;
    if (pv.evals) {  // residual tests performed, those decided in FP64, loose hypotheses (profiling)
        const bool one = (tid & 31) == 0;
        const int t = grp.sum(one ? st.tests : 0), f = grp.sum(one ? st.fp64 : 0), lo = grp.sum(one ? st.loose : 0);
        if (tid == 0) {
            atomicAdd(&pv.evals[GPM_COUNT_RANSAC], (unsigned long long)t);
            atomicAdd(&pv.evals[GPM_COUNT_RANSAC_FP64], (unsigned long long)f);
            atomicAdd(&pv.evals[GPM_COUNT_RANSAC_LOOSE], (unsigned long long)lo);
        }
    }
    if (best == 0ull) {  // every sample degenerate: no winner, best score -1
        if (tid == 0) mi[MI_BESTSCORE] = -1;
        return;
    }
    const int nw = key_score(best), wk = key_index(best);
    if (tid == 0) {
        mi[MI_BESTK] = wk;
        mi[MI_BESTSCORE] = nw;
    }
    if (nw < 4) return;
    // the winner's inliers among this thread's matches (bit c: match tid + c G::size; N <= 64 G::size for every
    // group: 256 matches per warp window, 96 x 96 per block window), uncertain ones decided in FP64
    static_assert(kMaxCell * kMaxCell <= 64 * 256 && 16 * 16 <= 64 * 32, "inlier mask too small");
    unsigned long long inm = 0;
    int2 v0 = make_int2(w.far->v0x, w.far->v0y);
    bool wide = false;
    if constexpr (MODE == FIT_FAR) {
        inm = far_winner(grp, w, cell, wk, tag, pv.pair_id, pp.k0, pp.k1, pp.t2, rw, v0, wide);
    } else {
        unsigned long long um = 0;
        {
            FastHyp h;
            const float tl = t_below(pp.t2), th = t_above(pp.t2);
            const bool scored = fast_hypothesis<false>(w, cell, wk, tag, pv.pair_id, pp.k0, pp.k1, th, h) == HYP_OK;
            for (int j = tid, c = 0; j < N; j += G::size, ++c) {
                bool sure = false, maybe = true;
                if (scored) test_match(w, h, tl, th, j, sure, maybe);
                if (sure)
                    inm |= 1ull << c;
                else if (maybe)
                    um |= 1ull << c;
            }
        }
        if (grp.any(um != 0)) {
            if (tid < 32) winner_fp64(w, cell, wk, tag, pv.pair_id, pp.k0, pp.k1, whl);
            grp.sync();
            for (; um; um &= um - 1) {
                const int c = __ffsll((long long)um) - 1;
                const float4 mt = w.match(tid + c * G::size);
                if (hyp_inlier_fp64(whl, mt.x, mt.y, mt.z, mt.w, (double)pp.t2)) inm |= 1ull << c;
            }
        }
        if (tid < 4) {
            int idx[4];
            draw_indices(N, cell, wk, tag, pv.pair_id, pp.k0, pp.k1, idx);
            const int j = tid == 0 ? idx[0] : (tid == 1 ? idx[1] : (tid == 2 ? idx[2] : idx[3]));
            rw->sample[tid] = exact_int(w.x[j]);
            rw->sample[4 + tid] = exact_int(w.y[j]);
            rw->target[tid] = (long long)v0.x + exact_int(w.qx[j]);
            rw->target[4 + tid] = (long long)v0.y + exact_int(w.qy[j]);
        }
    }
    if (tid == 0) {
        rw->nin = nw;
        rw->vmax = w.vmax;
        rw->wide = wide;
        rw->status = 2;
    }
    if (MODE == FIT_FAR && wide) return wide_sums(grp, w, inm, nw, v0, whl, rw);
    int sx = 0, sy = 0, tx = 0, ty = 0;  // target sums about v0
    for (unsigned long long m = inm; m; m &= m - 1) {
        const int j = tid + (__ffsll((long long)m) - 1) * G::size;
        sx += exact_int(w.x[j]);
        sy += exact_int(w.y[j]);
        tx += exact_int(w.qx[j]);
        ty += exact_int(w.qy[j]);
    }
    sx = grp.sum(sx);
    sy = grp.sum(sy);
    tx = grp.sum(tx);
    ty = grp.sum(ty);
    const float fn = (float)nw;
    const int cx = __float2int_rn(__fdiv_rn((float)sx, fn)), cy = __float2int_rn(__fdiv_rn((float)sy, fn));
    using Sum = std::conditional_t<MODE == FIT_NEAR, int, long long>;  // near a frame, 32 bits hold n times an offset
    const int cu = __float2int_rn(__fdiv_rn((float)((Sum)nw * v0.x + tx), fn));
    const int cv = __float2int_rn(__fdiv_rn((float)((Sum)nw * v0.y + ty), fn));
    const int du = (int)((Sum)v0.x - cu), dv = (int)((Sum)v0.y - cv);  // small: cu is v0 and a mean about it
    // Hartley scales: distances to the exact centroids, as n |p - mean| = |n p - sum| from exact integers
    // (the least-squares refit of a noisy support moves with its normalisation, so the scale must carry no
    // more than float rounding); windows up to 96 px: n |coordinate about v0| < 2^31
    double ds = 0.0, dt = 0.0;
    long long R[24];
#pragma unroll
    for (int q = 0; q < 24; ++q) R[q] = 0;
    for (; inm; inm &= inm - 1) {
        const int j = tid + (__ffsll((long long)inm) - 1) * G::size;
        const int ax = exact_int(w.x[j]), ay = exact_int(w.y[j]);
        const int bx = exact_int(w.qx[j]), by = exact_int(w.qy[j]);
        add_dist(ds, nw * ax - sx, nw * ay - sy);
        add_dist(dt, nw * bx - tx, nw * by - ty);
        const int X = ax - cx, Y = ay - cy, U = bx + du, V = by + dv;
        const int zz[6] = {X * X, X * Y, X, Y * Y, Y, 1};
        const int w3 = U * U + V * V;
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            R[q] += zz[q];
            R[6 + q] += (long long)U * zz[q];
            R[12 + q] += (long long)V * zz[q];
            R[18 + q] += (long long)w3 * zz[q];
        }
    }
    group_dists(grp, ds, dt, reinterpret_cast<double*>(whl), rw);
    group_moments(grp, R, scratch, rw->mom);
    if (tid == 0) {
        rw->cx = cx;
        rw->cy = cy;
        rw->cu = cu;
        rw->cv = cv;
    }
}

// The search keeps the hypothesis with the most inliers (lowest index on ties).  Every hypothesis is bounded, not
// counted: `maybe` tests give the most inliers it can have, whatever the rounding of its FP32 form, and it is
// dropped as soon as those and the matches not yet tested leave it below the best support known.  Only contenders
// are counted exactly, their uncertain tests decided in FP64 with the exact hypothesis; hypotheses whose FP32 form
// says too little (ill-conditioned samples, windows with far-flung imported offsets) are counted exactly at once.
// The outcome is that of counting every hypothesis exactly.  Once one has every match as an inlier, later ones can
// at most tie and are not drawn.

// Windows up to 16 x 16, one warp each: 32 hypotheses at a time, one per lane, each lane testing its own against
// the matches four at a time (every lane reads the same ones: broadcasts).  The quads go in four interleaved
// passes spread over the window; after each, lanes that cannot win drop out, and once few are left the warp counts
// those one by one with its lanes over the matches.
// What bounds it: instruction fetch, then the FP32 pipe in the tests (12 operations a match).  1024x436, stage 1:
// the 16 px windows 1.44 -> 0.41 ms, the 8 px windows 1.73 -> 0.53 ms, against scoring exact 128-bit hypotheses
// (0.64 and 1.12 ms of these gains while the winner was still solved here, in 180 KB of code, not 97; an integer
// reference offset has since cost 5 %: 8 px 0.67 -> 0.70 ms, a capture each).
template <bool FAR>
__device__ __forceinline__ unsigned long long search_warp(const Window& w, const PlaneParams& pp, int cell,
                                                          uint32_t tag, uint32_t pair_id, FastHyp* slot,
                                                          RansacStats& st) {
    const int lane = threadIdx.x & 31, N = w.N, nq = (N + 3) >> 2;
    const float t = t_above(pp.t2);
    const float2 tt = both(t);
    unsigned long long best = 0ull;
    for (int b = 0; b < pp.num_hyp; b += 32) {
        if (key_score(best) >= N) break;
        const int k = b + lane;
        FastHyp h;
        const int status =
            k < pp.num_hyp ? fast_hypothesis<FAR>(w, cell, k, tag, pair_id, pp.k0, pp.k1, t, h) : (int)HYP_DEAD;
        st.loose += __popc(__ballot_sync(FULL, status == HYP_LOOSE));
        unsigned alive = __ballot_sync(FULL, status == HYP_OK);
        int cnt = 0, left = 4 * nq;  // maybe tests passed; matches not yet tested
        if (FAR && status == HYP_OK) cnt = far_allowance(w, h, t);  // taken as passed
        if (alive) {
            const PairHyp ph = pair_hyp(h);
            for (int pass = 0; pass < 4; ++pass) {
                int done = 0;
#pragma unroll 2
                for (int q = pass; q < nq; q = (q | 3) + 1 + ((q + 1) & 3)) {  // 4 i + ((i + pass) & 3)
                    count_quad(w, ph, tt, 4 * q, cnt);
                    done += 4;
                }
                left -= done;
                st.tests += done * __popc(alive);
                alive = __ballot_sync(FULL, status == HYP_OK && hyp_key(cnt + min(left, N), k) >= best);
                if (__popc(alive) <= 2 * (3 - pass)) break;
            }
        }
        // contenders, the most promising first
        const int reach = status == HYP_OK ? cnt + max(min(left, N), 0) : (status == HYP_LOOSE ? N : -1);
        alive |= __ballot_sync(FULL, status == HYP_LOOSE);
        while (alive) {
            const bool in = (alive >> lane) & 1u;
            const int top = (int)__reduce_max_sync(FULL, (unsigned)(in ? reach + 1 : 0)) - 1;
            const unsigned ok = __ballot_sync(FULL, in && reach == top && status == HYP_OK);
            const int l = __ffs(ok ? ok : __ballot_sync(FULL, in && reach == top)) - 1;
            if (lane == l) *slot = h;
            __syncwarp();
            const int score =
                ok ? contender_support<FAR>(w, slot, cell, b + l, tag, pair_id, pp.k0, pp.k1, pp.t2, best, st)
                   : exact_support<FAR>(w, cell, b + l, tag, pair_id, pp.k0, pp.k1, pp.t2, best, st);
            __syncwarp();
            if (score >= 0) best = max(best, hyp_key(score, b + l));
            alive &= ~(1u << l);
            alive &= __ballot_sync(FULL, hyp_key(reach, k) >= best);
        }
    }
    return best;
}

// Larger windows, one block of 256 or 512 threads each: 256 hypotheses a round, solved one per thread into shared memory.
// The warps first test every hypothesis on an eighth of the matches (chunks of 128, spread over the window); the
// one with the most is counted from below on all of them, by the whole block, which gives the bound the others have
// to reach from the start; then the warps take the hypotheses that still can, one at a time, chunk by chunk.
// What bounds it: the FP32 pipe and the shared loads of the tests.  1024x436, stage 1: the 64 px windows 1.99 ->
// 0.77 ms, the 32 px windows 1.03 -> 0.47 ms, against scoring in index order from exact 128-bit hypotheses (reading the
// bound once a warp has since cost 7 %: 64 px 0.73 -> 0.79 ms, a capture each; reading it every fourth chunk gained nothing).
constexpr int kHypRound = 256;
struct BlockSearch {
    FastHyp form[kHypRound];
    short cnt[kHypRound];           // maybe tests passed in the first chunks; -1: not scored
    short todo[kHypRound];          // the hypotheses to finish, loose ones from the back
    unsigned long long best;        // a lower bound of the best key; the winner's at the end
    int next, n_ok, n_loose;
};
// A key in shared memory that other warps may raise meanwhile, the same value on every lane: what it decides holds
// collectives of the whole warp, and the lanes' own loads may fall on either side of a change.  A stale bound only drops less.
__device__ __forceinline__ unsigned long long shared_key(const volatile unsigned long long* key) {
    return __shfl_sync(FULL, (threadIdx.x & 31) == 0 ? *key : 0ull, 0);
}
template <bool FAR, int NT>
__device__ __forceinline__ unsigned long long search_block(const BlockGroup<NT>& grp, const Window& w,
                                                           const PlaneParams& pp, int cell, uint32_t tag,
                                                           uint32_t pair_id, BlockSearch& bs, RansacStats& st) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, N = w.N;
    const float t = t_above(pp.t2), tl = t_below(pp.t2);
    const float2 tt = both(t);
    const int nch = (N + 127) >> 7, nfirst = max(1, nch >> 3);
    // visiting order of the chunks: i -> i * step mod nch, step coprime to nch
    int step = max(1, (3 * nch) >> 3);
    for (;; ++step) {
        int a = step, b = nch;
        while (b) {
            const int r = a % b;
            a = b;
            b = r;
        }
        if (a == 1) break;
    }
    volatile unsigned long long* vbest = &bs.best;
    if (tid == 0) bs.best = 0ull;
    __syncthreads();
    for (int b = 0; b < pp.num_hyp; b += kHypRound) {
        if (key_score(*vbest) >= N) break;  // block-uniform: the barrier below has passed since it was written
        const int k = b + tid;
        int status = HYP_DEAD;
        {
            FastHyp h;
            if (tid < kHypRound && k < pp.num_hyp)
                status = fast_hypothesis<FAR>(w, cell, k, tag, pair_id, pp.k0, pp.k1, t, h);
            if (status == HYP_OK) bs.form[tid] = h;
        }
        if (tid < kHypRound) bs.cnt[tid] = status == HYP_OK ? 0 : -1;
        if (tid == 0) bs.next = bs.n_ok = bs.n_loose = 0;
        __syncthreads();
        for (int e = warp; e < kHypRound; e += NT / 32) {
            if (bs.cnt[e] < 0) continue;  // warp-uniform
            const PairHyp ph = pair_hyp(bs.form[e]);
            int c = 0, ch = 0;
            for (int i = 0; i < nfirst; ++i) {
                count_quad(w, ph, tt, 128 * ch + 4 * lane, c);
                ch += step;
                if (ch >= nch) ch -= nch;
            }
            c = (int)__reduce_add_sync(FULL, (unsigned)c);
            if (FAR) c += far_allowance(w, bs.form[e], t);  // taken as passed
            if (lane == 0) bs.cnt[e] = (short)c;
            st.tests += 128 * nfirst;
        }
        __syncthreads();
        const int rest = 128 * (nch - nfirst);
        {
            const int mine = tid < kHypRound ? bs.cnt[tid] : -1;
            const unsigned long long lead = grp.max(mine >= 0 ? hyp_key(mine, k) : 0ull);
            if (lead && hyp_key(min(key_score(lead) + rest, N), key_index(lead)) >= *vbest) {  // block-uniform
                const FastHyp h = bs.form[key_index(lead) - b];
                int lo = 0;
                for (int j = tid; j < N; j += NT) {
                    bool sure, maybe;
                    test_match(w, h, tl, t, j, sure, maybe);
                    lo += sure && !(FAR && h.away);
                }
                lo = grp.sum(lo);
                if (tid == 0) bs.best = max(bs.best, hyp_key(lo, key_index(lead)));
                st.tests += lane == 0 ? N / (NT / 32) : 0;
                __syncthreads();
            }
            const bool go = mine >= 0 && hyp_key(min(mine + rest, N), k) >= *vbest;
            if (go) bs.todo[atomicAdd(&bs.n_ok, 1)] = (short)tid;
            if (status == HYP_LOOSE) bs.todo[kHypRound - 1 - atomicAdd(&bs.n_loose, 1)] = (short)tid;
        }
        __syncthreads();
        const int n_ok = bs.n_ok, n_all = n_ok + bs.n_loose;
        for (;;) {
            int at = 0;
            if (lane == 0) at = atomicAdd(&bs.next, 1);
            at = __shfl_sync(FULL, at, 0);
            if (at >= n_all) break;
            const bool loose = at >= n_ok;
            const int e = bs.todo[loose ? kHypRound - 1 - (at - n_ok) : at];
            int score = -1;
            unsigned long long floor = shared_key(vbest);
            if (loose) {
                ++st.loose;
                if (hyp_key(N, b + e) >= floor)
                    score = exact_support<FAR>(w, cell, b + e, tag, pair_id, pp.k0, pp.k1, pp.t2, floor, st);
            } else {
                const PairHyp ph = pair_hyp(bs.form[e]);
                int have = bs.cnt[e], left = rest, ch = (int)((long long)nfirst * step % nch);
                bool alive = hyp_key(min(have + left, N), b + e) >= floor;
                while (alive && left > 0) {
                    int c = 0;
                    count_quad(w, ph, tt, 128 * ch + 4 * lane, c);
                    ch += step;
                    if (ch >= nch) ch -= nch;
                    left -= 128;
                    have += (int)__reduce_add_sync(FULL, (unsigned)c);
                    st.tests += 128;
                    floor = shared_key(vbest);
                    alive = hyp_key(min(have + left, N), b + e) >= floor;
                }
                if (alive)
                    score = contender_support<FAR>(w, &bs.form[e], cell, b + e, tag, pair_id, pp.k0, pp.k1, pp.t2, floor, st);
            }
            if (score >= 0 && lane == 0) atomicMax(&bs.best, hyp_key(score, b + e));
            __syncwarp();
        }
        __syncthreads();
    }
    return *vbest;
}

// The frames a refit is normalised in, for its way back.
struct RefitFrame {
    double ss, isq, mx, my, mqx, mqy;
};
// One window's normalised DLT matrix M and start x; false if the support has no extent.
__device__ __forceinline__ bool refit_system(RefitWork* rw, const LevelGeom& g, const PlaneParams& pp, int cell,
                                             double (&A)[45], double (&x)[9], RefitFrame& f) {
    int x0, y0, ox, oy;
    window_origin<WarpGroup>(g, cell, x0, y0, ox, oy);
    // the winner, exact, from its sample: its evaluation form with test bounds, its FP64 form for uncertain tests,
    // and itself normalised by its largest entry (a thread per window: the 128-bit solve serves 32 windows an
    // instruction here; by the fit's warp per window it took a third of the 8 px level's instructions)
    double Hw[9];
    {
        i128 hx[9];
        minimal_h_exact(rw->sample, rw->sample + 4, rw->target, rw->target + 4, hx);
        Mef m0;
        make_mef_exact(hx, m0);
        mef_set_bounds(m0, 0.5f * (float)g.s, rw->vmax, pp.t2);
        rw->mef0 = m0;
        exact_local_fp64(hx, rw->hl_w);
        exact_to_double(hx, Hw, 9);
    }
    double big = 0;
#pragma unroll
    for (int q = 0; q < 9; ++q) big = fmax(big, fabs(Hw[q]));
    const double rf = 1.0 / big;
#pragma unroll
    for (int q = 0; q < 9; ++q) Hw[q] *= rf;
    rw->geo_w = plane_geometry_ok(Hw, g.s, pp.radius, pp.scale_min, pp.scale_max) ? 1 : 0;
    local_to_abs(Hw, ox, oy, rw->ha_w);
    rw->refit_ok = 0;
    rw->geo_r = 0;

    // centroids and Hartley scales
    double R[24];
#pragma unroll
    for (int q = 0; q < 24; ++q) R[q] = (double)rw->mom[q];  // exact: |moment| < 2^53
    if (rw->wide) {
#pragma unroll
        for (int q = 0; q < 24; ++q) R[q] = __longlong_as_double(rw->mom[q]);
    }
    const double inv_n = 1.0 / (double)rw->nin;
    const double dx = R[2] * inv_n, dy = R[4] * inv_n, du = R[11] * inv_n, dv = R[17] * inv_n;
    const double mx = rw->cx + dx, my = rw->cy + dy, mqx = rw->cu + du, mqy = rw->cv + dv;
    const double n_in = (double)rw->nin, ds = rw->ds / n_in * inv_n, dt = rw->dt / n_in * inv_n;  // mean distances
    if (!(ds > 1e-12 && dt > 1e-12)) return false;
    const double ss = sqrt(2.0) / ds, sq = sqrt(2.0) / dt;
    const double iss = ds * 0.70710678118654752440, isq = dt * 0.70710678118654752440;  // 1 / ss, 1 / sq
    // centre the source terms (per raw weight 1, U, V, U^2 + V^2), then the weights
    double P[24];
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        const double* r = R + 6 * a;
        P[6 * a + 0] = r[0] - 2.0 * dx * r[2] + dx * dx * r[5];
        P[6 * a + 1] = r[1] - dy * r[2] - dx * r[4] + dx * dy * r[5];
        P[6 * a + 2] = r[2] - dx * r[5];
        P[6 * a + 3] = r[3] - 2.0 * dy * r[4] + dy * dy * r[5];
        P[6 * a + 4] = r[4] - dy * r[5];
        P[6 * a + 5] = r[5];
    }
    double mom[24];
    const double sz[6] = {ss * ss, ss * ss, ss, ss * ss, ss, 1.0};
#pragma unroll
    for (int q = 0; q < 6; ++q) {
        const double c0 = P[q];
        const double c1 = P[6 + q] - du * P[q];
        const double c2 = P[12 + q] - dv * P[q];
        const double c3 = P[18 + q] - 2.0 * du * P[6 + q] - 2.0 * dv * P[12 + q] + (du * du + dv * dv) * P[q];
        mom[q] = sz[q] * c0;
        mom[6 + q] = sq * sz[q] * c1;
        mom[12 + q] = sq * sz[q] * c2;
        mom[18 + q] = sq * sq * sz[q] * c3;
    }
#pragma unroll
    for (int i = 0; i < 9; ++i)
#pragma unroll
        for (int j = 0; j <= i; ++j) A[i * (i + 1) / 2 + j] = dlt_entry(mom, i, j);
    // start: the winner in the normalised frames, h0 = Tq Hw Tp^-1
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            double b[3];
#pragma unroll
            for (int k = 0; k < 3; ++k)
                b[k] = c == 0 ? Hw[k * 3] * iss
                              : (c == 1 ? Hw[k * 3 + 1] * iss : Hw[k * 3] * mx + Hw[k * 3 + 1] * my + Hw[k * 3 + 2]);
            x[r * 3 + c] = r == 0 ? sq * (b[0] - mqx * b[2]) : (r == 1 ? sq * (b[1] - mqy * b[2]) : b[2]);
        }
    f = RefitFrame{ss, isq, mx, my, mqx, mqy};
    return true;
}

// The refit from the eigenvector x: denormalised, its evaluation and FP64 forms, the geometry checks.
__device__ __forceinline__ void refit_record(RefitWork* rw, const LevelGeom& g, const PlaneParams& pp, int cell,
                                             const double (&x)[9], const RefitFrame& f) {
    int x0, y0, ox, oy;
    window_origin<WarpGroup>(g, cell, x0, y0, ox, oy);
    const double ss = f.ss, isq = f.isq, mx = f.mx, my = f.my, mqx = f.mqx, mqy = f.mqy;
    // Hr = Tq^-1 h Tp
    double Hr[9];
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            double b[3];
#pragma unroll
            for (int k = 0; k < 3; ++k)
                b[k] = c == 0 ? x[k * 3] * ss
                              : (c == 1 ? x[k * 3 + 1] * ss : x[k * 3 + 2] - ss * (mx * x[k * 3] + my * x[k * 3 + 1]));
            Hr[r * 3 + c] = r == 0 ? b[0] * isq + mqx * b[2] : (r == 1 ? b[1] * isq + mqy * b[2] : b[2]);
        }
    Mef m1;
    if (!make_mef(Hr, 0, 0, m1)) return;
    mef_set_bounds(m1, 0.5f * (float)g.s, rw->vmax, pp.t2);
    rw->mef1 = m1;
    {
        // the refit for FP64 tests: denominator 1 at the window centre (-0.5, -0.5), as its evaluation form
        const double k = 1.0 / (Hr[8] - 0.5 * (Hr[6] + Hr[7]));
#pragma unroll
        for (int q = 0; q < 9; ++q) rw->hl_r[q] = Hr[q] * k;
    }
    rw->geo_r = plane_geometry_ok(Hr, g.s, pp.radius, pp.scale_min, pp.scale_max) ? 1 : 0;
    local_to_abs(Hr, ox, oy, rw->ha_r);
    rw->refit_ok = 1;
}

// (B) Normalised DLT refit of each window whose fit is pending, one thread
// per window and direction: centred, Hartley-scaled moments from the exact
// integer ones, the smallest eigenvector of A^T A started from the winner,
// denormalisation, and the geometry checks of the winner and of the refit.
__global__ void __launch_bounds__(32) k_refit_solve(const __grid_constant__ Batch bt, int level, PlaneParams pp) {
    begin_kernel();
    const PairView& pv = bt.view(blockIdx.z);
    const LevelGeom g = bt.geom(blockIdx.z, level);
    __shared__ EigShared sh;
    const int nc = g.ncells(), lane = threadIdx.x;
    const int t = blockIdx.x * 32 + lane;
    const int dir = min(t / max(nc, 1), 1), cell = t - dir * nc;
    RefitWork* rw = pv.rw[dir] + cell;
    RefitFrame f;
    double x[9], A[45], rd[9];
    EigState e;
    const bool todo = t < 2 * nc && rw->status == 2;
    bool act = todo;
    if (act) {
        double M[45];
        act = refit_system(rw, g, pp, cell, M, x, f);
        if (act) {
#pragma unroll
            for (int q = 0; q < 45; ++q) sh.M[q][lane] = M[q];
            eig_start(M, x, A, rd, e);
        }
    }
    const bool refit = act;
    unsigned left;
    for (int step = 0;; ++step) {
        left = __ballot_sync(FULL, act);
        if (!left || (step >= 4 && __popc(left) == 1) || step >= 12) break;
        if (act) act = eig_thread(sh.M, x, A, rd, e);
    }
    for (; left; left &= left - 1) {  // a window's iteration goes on
        const bool mine = lane == __ffs(left) - 1;
        if (mine) {
            sh.e = e;
#pragma unroll
            for (int q = 0; q < 45; ++q) sh.A[q] = A[q];
#pragma unroll
            for (int i = 0; i < 9; ++i) sh.rd[i] = rd[i], sh.x[i] = x[i];
        }
        __syncwarp();
        eig_warp(sh, __ffs(left) - 1);
        if (mine) {
#pragma unroll
            for (int i = 0; i < 9; ++i) x[i] = sh.x[i];
        }
        __syncwarp();
    }
    if (!refit) return;
    refit_record(rw, g, pp, cell, x, f);
}

// (C) Rescore the refit on the window's matches, choose, count colour
// inliers among the RANSAC inliers (|S_R n S_C|, Sec. 3.4 third cue) and
// write the model: valid iff the support is at least max(min_inliers, N / 5)
// and the chosen homography passed the geometry checks.
template <class G, int ST>
__device__ void ransac_finish(const G& grp, const PairView& pv, const LevelGeom& g, int stage, const PlaneParams& pp,
                              int dir, int cell, float4* match) {
    const RefitWork* rw = pv.rw[dir] + cell;
    if (rw->status != 2) return;
    const int tid = grp.rank();
    const int id = (g.base + cell) * 2 + (stage - 1);
    int* mi = pv.mi[dir] + (size_t)id * kMI;
    const int N = gather_matches<G>(grp, pv, g, stage, dir, cell, match);
    int x0, y0, ox, oy;
    window_origin<G>(g, cell, x0, y0, ox, oy);
    const int W = pv.W, H = pv.H;
    const float t2 = pp.t2;
    const int2* nnf = pv.nnf[dir];
    // a match's test, certified: FP64 where the FP32 form cannot tell, or its offset is no exact float
    auto inlier = [&](const Mef& m, const double* Hl, const float4& mt) {
        bool unc;
        const bool in = cert_inlier(m, mt, t2, unc), far = fmaxf(fabsf(mt.z), fabsf(mt.w)) >= 16777216.f;
        if (!(unc || far)) return in;
        int2 v = make_int2(0, 0);
        if (far) v = nnf[(oy + (int)mt.y) * W + ox + (int)mt.x];
        return hyp_inlier_fp64(Hl, (double)mt.x, (double)mt.y, (double)mt.x + (far ? (double)v.x : (double)mt.z),
                               (double)mt.y + (far ? (double)v.y : (double)mt.w), (double)t2);
    };
    const int wscore = rw->nin;
    const bool have_refit = rw->refit_ok != 0;
    int rcount = 0;
    if (have_refit) {
        const Mef rm = rw->mef1;
        for (int j = tid; j < N; j += G::size) {
            rcount += inlier(rm, rw->hl_r, match[j]);
        }
    }
    rcount = grp.sum(rcount);
    const bool use_refit = have_refit && rcount >= wscore;
    Mef fm = use_refit ? rw->mef1 : rw->mef0;
    // the chosen model in FP64 (local coordinates), for decisions the FP32 form cannot certify
    const double* Hl = use_refit ? rw->hl_r : rw->hl_w;
    const int count = use_refit ? rcount : wscore;
    const void* src = pv.img[dir];
    const void* tgt = pv.img[1 - dir];
    fm.ox = ox;
    fm.oy = oy;
    int nrc = 0;
    for (int j = tid; j < N; j += G::size) {
        const float4 mt = match[j];
        if (!inlier(fm, Hl, mt)) continue;
        const int px = ox + (int)mt.x, py = oy + (int)mt.y;
        int ix, iy, kx, ky;
        float fx, fy;
        // certified: a frame test or colour decision within the FP32 position error (times the largest
        // texel difference, 2) is taken again in FP64
        const float dp = mef_pos_bound(fm, mt.x, mt.y);
        bool sure = mef_flow(fm, mt.x, mt.y, kx, fx, ky, fy);
        int dec = 0;
        if (sure) {
            ix = px + kx;
            iy = py + ky;
            const float X = (float)ix + fx, Y = (float)iy + fy;
            const float e0 = -kFrameTol, ex = (float)(W - 1) + kFrameTol, ey = (float)(H - 1) + kFrameTol;
            sure = fabsf(X - e0) > dp && fabsf(X - ex) > dp && fabsf(Y - e0) > dp && fabsf(Y - ey) > dp;
            if (sure) {
                if (in_frame_tol(ix, fx, W) && in_frame_tol(iy, fy, H)) {
                    const float dl = colour_delta<ST>(src, tgt, W, H, px, py, ix, fx, iy, fy);
                    sure = fabsf(dl - pp.eps) > 2.f * dp + 1e-6f;
                    dec = dl < pp.eps;
                }
            }
        } else {
            // the FP32 denominator is not positive: certain unless it is within its rounding of zero
            const float den = 1.f + fm.e0 + fm.g0 * mt.x + fm.g1 * mt.y;
            sure = fabsf(den) > __int_as_float(fm.eden);
        }
        nrc += sure ? dec : colour_overlap_fp64<ST>(Hl, src, tgt, W, H, ox, oy, px, py, pp.eps);
    }
    nrc = grp.sum(nrc);
    if (tid == 0) {
        const bool valid = count >= pp.min_inliers && 5 * count >= N && (use_refit ? rw->geo_r : rw->geo_w) != 0;
        const double* Ha = use_refit ? rw->ha_r : rw->ha_w;
        for (int q = 0; q < 9; ++q) pv.mh[dir][(size_t)id * 9 + q] = Ha[q];
        fm.valid = valid ? 1 : 0;
        pv.mef[dir][id] = fm;
        mi[MI_VALID] = valid ? 1 : 0;
        mi[MI_COUNT] = count;
        mi[MI_FLAGS] = F_FITTED | (use_refit ? F_REFIT : 0) | (valid ? 0 : F_BAD_GEOM);
        mi[MI_NRC] = nrc;
    }
}

// (A) Windows up to 16 x 16: one warp per window, kRansacWarps windows per block.  CAP: the most matches a window
// has (64 for sides up to 8, else 256).
constexpr int kRansacWarps = 4;
template <int CAP, int MODE>
__global__ void __launch_bounds__(32 * kRansacWarps, 24 / kRansacWarps)
    k_ransac_warp(const __grid_constant__ Batch bt, int level, int stage, PlaneParams pp) {
    begin_kernel();
    const PairView& pv = bt.view(blockIdx.z);
    const LevelGeom g = bt.geom(blockIdx.z, level);
    __shared__ __align__(16) float planes[kRansacWarps][4 * CAP];
    __shared__ FastHyp slot[kRansacWarps];
    __shared__ WindowFar far[kRansacWarps];
    __shared__ double whl[kRansacWarps][9];
    const int warp = threadIdx.x >> 5, dir = blockIdx.y;
    const int cell = blockIdx.x * kRansacWarps + warp;
    if (cell >= g.ncells()) return;
    const WarpGroup grp;
    const int id = (g.base + cell) * 2 + (stage - 1);
    RefitWork* rw = pv.rw[dir] + cell;
    if (MODE == FIT_FAR && rw->status != kFarPending) return;
    Window w;
    gather_window<MODE>(grp, pv, g, stage, dir, cell, planes[warp], CAP, 4, &far[warp], w);
    if (grp.rank() == 0) clear_model(pv, dir, id, w.N, rw);
    if (w.N < pp.min_inliers || w.N < 4) return;
    if (MODE == FIT_ANY && w.far->n) {
        if (grp.rank() == 0) rw->status = kFarPending;
        return;
    }
    const uint32_t tag = stream_tag(RNG_RANSAC, dir, level, stage);
    RansacStats st;
    const unsigned long long best = search_warp<MODE == FIT_FAR>(w, pp, cell, tag, pv.pair_id, &slot[warp], st);
    finish_fit<MODE>(grp, pv, w, pp, dir, cell, id, tag, best, st, whl[warp], nullptr, rw);
}
template <int ST>
__global__ void __launch_bounds__(256) k_ransac_finish_warp(const __grid_constant__ Batch bt, int level, int stage, PlaneParams pp) {
    begin_kernel();
    const PairView& pv = bt.view(blockIdx.z);
    const LevelGeom g = bt.geom(blockIdx.z, level);
    __shared__ float4 match[8][256];
    const int warp = threadIdx.x >> 5;
    const int cell = blockIdx.x * 8 + warp;
    if (cell >= g.ncells()) return;
    WarpGroup grp;
    ransac_finish<WarpGroup, ST>(grp, pv, g, stage, pp, blockIdx.y, cell, match[warp]);
}

// Larger windows: one block per window (matches in dynamic shared memory: four planes of block_cap(s)).
__host__ __device__ constexpr int block_cap(int s) { return (s * s + 127) / 128 * 128; }
// 512 threads a window instead of 256: where the matches leave an SM room for two blocks only (s > 60: 3 blocks' 16 s^2 +
// 14 KB are above its 228 KB), and where all windows are resident at once, so that the launch lasts as one window (three
// 256-thread blocks on each of 152 SMs).  First stage: 64 px windows of 1024x436 0.81 -> 0.72 ms, of 512x384 0.49 -> 0.37,
// of 253x187 0.30 -> 0.24; 80 px of 1024x436 1.05 -> 0.82; 330 32 px windows 0.12 -> 0.12, their second stage 0.10 -> 0.08.
// Elsewhere 256 is faster: 3300 32 px windows 0.51 against 0.56 ms, 2000 40 px ones 0.52 against 0.54.
static bool ransac_wide(int s, int windows) { return s > 60 || windows <= 3 * 152; }
template <int NT, int MODE>
__global__ void __launch_bounds__(NT, NT > 256 ? 2 : 3) k_ransac_block(const __grid_constant__ Batch bt, int level, int stage, PlaneParams pp) {
    begin_kernel();
    const PairView& pv = bt.view(blockIdx.z);
    const LevelGeom g = bt.geom(blockIdx.z, level);
    const int cell = blockIdx.x, dir = blockIdx.y;
    if (cell >= g.ncells()) return;  // past this pair's windows (block-uniform)
    extern __shared__ __align__(16) float planes_dyn[];
    __shared__ int red_i[NT / 32];
    __shared__ unsigned long long red_u[NT / 32];
    __shared__ __align__(16) BlockSearch bs;
    __shared__ double whl[16];  // also two sums per warp
    __shared__ WindowFar far;
    const BlockGroup<NT> grp{red_i, red_u};
    const int id = (g.base + cell) * 2 + (stage - 1);
    RefitWork* rw = pv.rw[dir] + cell;
    if (MODE == FIT_FAR && rw->status != kFarPending) return;  // block-uniform: cleared behind the barriers of gather_window
    Window w;
    gather_window<MODE>(grp, pv, g, stage, dir, cell, planes_dyn, block_cap(g.s), 128, &far, w);
    if (threadIdx.x == 0) clear_model(pv, dir, id, w.N, rw);
    if (w.N < pp.min_inliers || w.N < 4) return;
    if (MODE == FIT_ANY && w.far->n) {
        if (threadIdx.x == 0) rw->status = kFarPending;
        return;
    }
    const uint32_t tag = stream_tag(RNG_RANSAC, dir, level, stage);
    RansacStats st;
    const unsigned long long best = search_block<MODE == FIT_FAR>(grp, w, pp, cell, tag, pv.pair_id, bs, st);
    // the winner's sums by 256 threads, whatever the block: their FP64 ones are in one order (barriers wait for the
    // threads that are left)
    if (NT > 256 && threadIdx.x >= 256) {
        if (pv.evals && (threadIdx.x & 31) == 0) {
            atomicAdd(&pv.evals[GPM_COUNT_RANSAC], (unsigned long long)st.tests);
            atomicAdd(&pv.evals[GPM_COUNT_RANSAC_FP64], (unsigned long long)st.fp64);
            atomicAdd(&pv.evals[GPM_COUNT_RANSAC_LOOSE], (unsigned long long)st.loose);
        }
        return;
    }
    finish_fit<MODE>(BlockGroup<256>{red_i, red_u}, pv, w, pp, dir, cell, id, tag, best, st, whl,
                    reinterpret_cast<long long*>(bs.form), rw);
}
template <int ST>
__global__ void __launch_bounds__(256) k_ransac_finish_block(const __grid_constant__ Batch bt, int level, int stage, PlaneParams pp) {
    begin_kernel();
    const PairView& pv = bt.view(blockIdx.z);
    const LevelGeom g = bt.geom(blockIdx.z, level);
    if ((int)blockIdx.x >= g.ncells()) return;  // past this pair's windows (block-uniform)
    extern __shared__ float4 match_dyn[];
    __shared__ int red_i[8];
    __shared__ unsigned long long red_u[8];
    BlockGroup<256> grp{red_i, red_u};
    ransac_finish<BlockGroup<256>, ST>(grp, pv, g, stage, pp, blockIdx.y, blockIdx.x, match_dyn);
}

// ---------------------------------------------------------------- assignment (eq. 3-4)
// For each pixel, over the windows of the level that cover it (window
// order), the valid plane of the given stage maps p to H p; delta is the mean
// absolute RGB difference between I_src(p) and the bilinear I_tgt(H p); the
// pixel is an inlier iff delta < eps, and takes the inlier plane with the
// smallest L = delta (first window on ties), with flow H p - p.
//
// A level assigns four times: the first stage's planes into tent, again into st1 once the cues have discarded some, then the
// residual stage's on the pixels without one into lvl (the others copied from st1), and again there.  The second
// assignment of a stage differs from its first only where a window that covers the pixel lost its plane in between,
// so it is computed there and taken over elsewhere (the winner alone does not tell: without a discarded plane a
// near tie between two others may fall the other way).
// What bounds it: the gathers of up to nine windows' models and four texels each.  1024x436, sixteen launches: 0.46 -> 0.38 ms.
enum AssignMode { ASSIGN_TENT, ASSIGN_ST1, ASSIGN_LVL, ASSIGN_LVL_AGAIN };
template <int ST, int MODE>
__global__ void k_assign(const __grid_constant__ Batch bt, int level, PlaneParams pp) {
    begin_kernel();
    constexpr int stage = MODE <= ASSIGN_ST1 ? 1 : 2;
    const PairView& pv = bt.view(blockIdx.z);
    const LevelGeom g = bt.geom(blockIdx.z, level);
    const int dir = blockIdx.y;
    const int W = pv.W, H = pv.H, n = pv.n;
    const Labels out = MODE == ASSIGN_TENT ? pv.tent[dir] : (MODE == ASSIGN_ST1 ? pv.st1[dir] : pv.lvl[dir]);
    const void* src = pv.img[dir];
    const void* tgt = pv.img[1 - dir];
    const Mef* mef = pv.mef[dir];
    const int* mi = pv.mi[dir];
    uint8_t* resid = pv.resid[dir];
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        if (MODE == ASSIGN_LVL_AGAIN) pv.m2o_key[dir][i] = ~0ull;  // for the many-to-one test that follows
        if (MODE == ASSIGN_LVL && !resid[i]) {
            const Labels in = pv.st1[dir];
            out.m[i] = in.m[i];
            out.L[i] = in.L[i];
            out.v[i] = in.v[i];
            out.r[i] = in.r[i];
            continue;
        }
        if (MODE == ASSIGN_LVL_AGAIN && !resid[i]) continue;
        const int y = i / W, x = i - y * W;
        int ix3[3], iy3[3];
        const int nxw = covering(g.gx, g.s, g.h, x, ix3), nyw = covering(g.gy, g.s, g.h, y, iy3);
        if (MODE == ASSIGN_ST1 || MODE == ASSIGN_LVL_AGAIN) {
            bool lost = false;
            for (int a = 0; a < nyw; ++a)
                for (int b = 0; b < nxw; ++b) {
                    const int id = (g.base + iy3[a] * g.gx.count + ix3[b]) * 2 + (stage - 1);
                    lost = lost || (mi[(size_t)id * kMI + MI_FLAGS] & (F_BAD_FB | F_BAD_KAPPA)) != 0;
                }
            if (!lost) {
                if (MODE == ASSIGN_ST1) {
                    const Labels in = pv.tent[dir];
                    const int m = in.m[i];
                    out.m[i] = m;
                    out.L[i] = in.L[i];
                    out.v[i] = in.v[i];
                    out.r[i] = in.r[i];
                    resid[i] = m < 0;
                }
                continue;
            }
        }
        int bm = -1, bkx = 0, bky = 0;
        float bL = FLT_MAX, bfx = 0.f, bfy = 0.f;
        for (int a = 0; a < nyw; ++a)
            for (int b = 0; b < nxw; ++b) {
                const int cell = iy3[a] * g.gx.count + ix3[b];
                const int id = (g.base + cell) * 2 + (stage - 1);
                const Mef m = mef[id];
                if (!m.valid) continue;
                int ix, iy, kx, ky;
                float fx, fy;
                if (!plane_target(m, x, y, W, H, ix, fx, iy, fy, kx, ky)) continue;
                const float d = colour_delta<ST>(src, tgt, W, H, x, y, ix, fx, iy, fy);
                if (!(d < pp.eps)) continue;
                if (d < bL - kLTie) {
                    bL = d;
                    bm = id;
                    bkx = kx;
                    bky = ky;
                    bfx = fx;
                    bfy = fy;
                }
            }
        int vx = 0, vy = 0;
        float rx = 0.f, ry = 0.f;
        if (bm >= 0) {
            round_split(bkx, bfx, vx, rx);
            round_split(bky, bfy, vy, ry);
        }
        out.m[i] = bm;
        out.L[i] = bm >= 0 ? bL : pp.eps;
        out.v[i] = make_int2(vx, vy);
        out.r[i] = make_float2(rx, ry);
        if (MODE == ASSIGN_ST1) resid[i] = bm < 0;
    }
}

// ---------------------------------------------------------------- occlusion cues (Sec. 3.4)
// Forward-backward plane projection symmetry: a pixel assigned to a plane of
// this level and stage with flow f is symmetric iff q = round(p + f) holds an
// assigned pixel of the other direction with flow g, |f + g| < t_fb.
__global__ void k_cue_counts(const __grid_constant__ Batch bt, int level, int stage, int which, PlaneParams pp) {
    begin_kernel();
    const PairView& pv = bt.view(blockIdx.z);
    const LevelGeom g = bt.geom(blockIdx.z, level);
    const int dir = blockIdx.y;
    const int W = pv.W, H = pv.H, n = pv.n;
    const Labels lab = which == 0 ? pv.tent[dir] : pv.lvl[dir];
    const Labels oth = which == 0 ? pv.tent[1 - dir] : pv.lvl[1 - dir];
    const int lo = g.base * 2, hi = (g.base + g.ncells()) * 2, lane = threadIdx.x & 31;
    int* mi = pv.mi[dir];
    // a warp's pixels of one plane count together: neighbours mostly share theirs, and one by one their additions queue at
    // its counters (1024x436: the cues' sixteen launches 0.16 ms with one addition a pixel and eight more launches, 0.11 now)
    for (int i0 = blockIdx.x * blockDim.x + threadIdx.x - lane; i0 < n; i0 += gridDim.x * blockDim.x) {
        const int i = i0 + lane;
        const int m = i < n ? lab.m[i] : -1;
        const bool counts = m >= lo && m < hi && (m & 1) == stage - 1;
        const unsigned some = __ballot_sync(0xffffffffu, counts);
        if (!counts) continue;
        bool symmetric = false;
        const int y = i / W, x = i - y * W;
        const int2 v = lab.v[i];
        const int qx = x + v.x, qy = y + v.y;
        if (qx >= 0 && qx < W && qy >= 0 && qy < H) {
            const int j = qy * W + qx;
            if (oth.m[j] >= 0) {
                const int2 w = oth.v[j];
                const float2 r = lab.r[i], s = oth.r[j];
                const float ex = (float)(v.x + w.x) + (r.x + s.x);
                const float ey = (float)(v.y + w.y) + (r.y + s.y);
                symmetric = ex * ex + ey * ey < pp.fb2;
            }
        }
        const unsigned same = __match_any_sync(some, m), sym = __ballot_sync(some, symmetric) & same;
        if (lane == __ffs(same) - 1) {
            atomicAdd(&mi[(size_t)m * kMI + MI_NASSIGN], __popc(same));
            if (sym) atomicAdd(&mi[(size_t)m * kMI + MI_NSYM], __popc(sym));
        }
    }
}

// Discard planes failing the symmetry cue (eta) or the RANSAC/colour overlap cue (kappa).
__global__ void k_cue_invalidate(const __grid_constant__ Batch bt, int level, int stage, PlaneParams pp) {
    begin_kernel();
    const PairView& pv = bt.view(blockIdx.z);
    const LevelGeom g = bt.geom(blockIdx.z, level);
    const int dir = blockIdx.y;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < g.ncells(); c += gridDim.x * blockDim.x) {
        const int id = (g.base + c) * 2 + stage - 1;
        int* f = pv.mi[dir] + (size_t)id * kMI;
        if (!f[MI_VALID]) continue;
        bool bad = false;
        if (f[MI_NASSIGN] > 0 && (float)f[MI_NSYM] < pp.eta * (float)f[MI_NASSIGN]) {
            f[MI_FLAGS] |= F_BAD_FB;
            bad = true;
        }
        if ((float)f[MI_NRC] < pp.kappa * (float)f[MI_COUNT]) {
            f[MI_FLAGS] |= F_BAD_KAPPA;
            bad = true;
        }
        if (bad) {
            f[MI_VALID] = 0;
            pv.mef[dir][id].valid = 0;
        }
    }
}

// Many-to-one: per target q = round(p + f), the lowest (L, index) keeps it;
// a loser whose flow differs from the winner's by t_fb or more is occluded.  (The level's last assignment clears the keys.)
__global__ void k_m2o_claim(const __grid_constant__ Batch bt) {
    begin_kernel();
    const PairView& pv = bt.view(blockIdx.z);
    const int dir = blockIdx.y;
    const int W = pv.W, n = pv.n;
    const Labels lab = pv.lvl[dir];
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        if (lab.m[i] < 0) continue;
        const int y = i / W, x = i - y * W;
        const int2 v = lab.v[i];
        if (x + v.x < 0 || x + v.x >= W || y + v.y < 0 || y + v.y >= pv.H) continue;
        const int q = (y + v.y) * W + (x + v.x);
        const unsigned long long key = ((unsigned long long)__float_as_uint(lab.L[i]) << 32) | (unsigned)i;
        atomicMin(&pv.m2o_key[dir][q], key);
    }
}
__global__ void k_m2o_resolve(const __grid_constant__ Batch bt, PlaneParams pp) {
    begin_kernel();
    const PairView& pv = bt.view(blockIdx.z);
    const int dir = blockIdx.y;
    const int W = pv.W, n = pv.n;
    const Labels lab = pv.lvl[dir];
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        if (lab.m[i] < 0) continue;
        const int y = i / W, x = i - y * W;
        const int2 v = lab.v[i];
        if (x + v.x < 0 || x + v.x >= W || y + v.y < 0 || y + v.y >= pv.H) continue;
        const int q = (y + v.y) * W + (x + v.x);
        const int w = (int)(pv.m2o_key[dir][q] & 0xFFFFFFFFull);
        if (w == i) continue;
        const int2 vw = lab.v[w];
        const float2 r = lab.r[i], rw = lab.r[w];
        const float ex = (float)(v.x - vw.x) + (r.x - rw.x);
        const float ey = (float)(v.y - vw.y) + (r.y - rw.y);
        if (!(ex * ex + ey * ey < pp.fb2)) {
            lab.m[i] = -1;
            pv.cue[dir][i] |= CUE_M2O;
        }
    }
}

// Sec. 3.3 merge with coarse priority, then the NNF update of Sec. 3.3.1.
__global__ void k_merge_update(const __grid_constant__ Batch bt, PlaneParams pp) {
    begin_kernel();
    const PairView& pv = bt.view(blockIdx.z);
    const int dir = blockIdx.y;
    const int n = pv.n;
    const Labels lab = pv.lvl[dir], acc = pv.acc[dir];
    if (blockIdx.x == 0 && threadIdx.x < 2) pv.list_count[dir * 2 + threadIdx.x] = 0;  // for the lists that follow
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int m = lab.m[i];
        int am = acc.m[i];
        if (m >= 0 && (am < 0 || lab.L[i] < acc.L[i] - pp.beta)) {
            acc.m[i] = m;
            acc.L[i] = lab.L[i];
            acc.v[i] = lab.v[i];
            acc.r[i] = lab.r[i];
            am = m;
        }
        pv.frozen[dir][i] = am >= 0;
        if (am >= 0) pv.nnf[dir][i] = acc.v[i];
    }
}

// ---------------------------------------------------------------- fill and final map (Sec. 3.4.1)
// One Jacobi iteration: labels from acc into tent (flip = 0) or from tent into acc (flip = 1).  After the first one the two
// differ only in pixels filled by the iteration before, so a label that both hold, or that stays unfilled, is not copied
// again: an iteration reads 8 bytes of most pixels where it moved 48 (1920x1080, eight iterations: 0.42 -> 0.22 ms).
template <int ST>
__global__ void k_fill(const __grid_constant__ Batch bt, int flip, int first, PlaneParams pp) {
    begin_kernel();
    const PairView& pv = bt.view(blockIdx.z);
    const int dir = blockIdx.y;
    const int W = pv.W, H = pv.H, n = pv.n;
    const Labels cur = flip ? pv.tent[dir] : pv.acc[dir], nxt = flip ? pv.acc[dir] : pv.tent[dir];
    const void* src = pv.img[dir];
    const void* tgt = pv.img[1 - dir];
    const Mef* mef = pv.mef[dir];
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int cm = cur.m[i];
        if (!first && cm >= 0 && nxt.m[i] == cm) continue;
        int bm = cm, bkx = 0, bky = 0;
        float bL = cur.L[i], bfx = 0.f, bfy = 0.f;
        bool filled = false;
        if (cm < 0 && !(pv.cue[dir][i] & CUE_M2O)) {
            const int y = i / W, x = i - y * W;
            bm = -1;
            bL = FLT_MAX;
            for (int k = 0; k < 4; ++k) {
                const int xx = x + (k == 0 ? -1 : (k == 1 ? 1 : 0));
                const int yy = y + (k == 2 ? -1 : (k == 3 ? 1 : 0));
                if (xx < 0 || xx >= W || yy < 0 || yy >= H) continue;
                const int m = cur.m[yy * W + xx];
                if (m < 0 || m >= pv.m_models) continue;
                const Mef mm = mef[m];
                int ix, iy, kx, ky;
                float fx, fy;
                if (!plane_target(mm, x, y, W, H, ix, fx, iy, fy, kx, ky)) continue;
                const float d = colour_delta<ST>(src, tgt, W, H, x, y, ix, fx, iy, fy);
                if (!(d < pp.eps)) continue;
                if (d < bL - kLTie || (fabsf(d - bL) <= kLTie && m < bm)) {
                    bL = d;
                    bm = m;
                    bkx = kx;
                    bky = ky;
                    bfx = fx;
                    bfy = fy;
                }
            }
            filled = bm >= 0;
            if (!filled) bL = cur.L[i];
        }
        if (!first && cm < 0 && !filled) continue;
        nxt.m[i] = bm;
        nxt.L[i] = bL;
        if (filled) {
            int vx, vy;
            float rx, ry;
            round_split(bkx, bfx, vx, rx);
            round_split(bky, bfy, vy, ry);
            nxt.v[i] = make_int2(vx, vy);
            nxt.r[i] = make_float2(rx, ry);
        } else {
            nxt.v[i] = cur.v[i];
            nxt.r[i] = cur.r[i];
        }
    }
}

// ---------------------------------------------------------------- edge-aware fill of unassigned pixels
// Each pixel left without a plane takes the plane of the assigned pixel
// nearest in geodesic distance (steps 256 + |q_i - q_j| between
// 4-neighbours, q = floor(1024 (R + G + B)) of frame 1 as given).  Integer
// distances by fast sweeping: rounds of four in-place scans in the order rows
// left to right, rows right to left, columns top to bottom, columns bottom to
// top; an offer wins with a lower distance, or an equal one from a lower seed
// index.
// Scratch of the edge-aware fill (the many-to-one keys and the pixel lists are idle by then): distances and seeds.
__device__ __forceinline__ long long* seed_dist(const PairView& pv) { return reinterpret_cast<long long*>(pv.m2o_key[0]); }
__device__ __forceinline__ int* seed_of(const PairView& pv) { return pv.list[0]; }
__global__ void k_seed_init(const __grid_constant__ Batch bt) {
    begin_kernel();
    const PairView& pv = bt.view(blockIdx.z);
    const int* am = pv.acc[0].m;
    const int n = pv.n;
    long long* dist = seed_dist(pv);
    int* seed = seed_of(pv);
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        dist[i] = am[i] >= 0 ? 0 : (1ll << 62);
        seed[i] = am[i] >= 0 ? i : -1;
    }
}
// One scan relaxes each pixel of a line from the one before it: the pixel takes (distance before + step, seed before) if
// that is less than its own pair, by distance, then seed.  A step adds the same to every offer that passes it, so
// after the scan a pixel holds the least of the offers of all pixels before it and its own, and that minimum is
// associative: offers are compared in any grouping, as (distance less the steps' sum from the line's start), and the
// distances are integers, so the result is that of the pixel-by-pixel walk.  A pixel without a seed has distance 2^62
// and seed -1, above every offer (line sums stay below 2^47), and changes nothing by being compared.
// What bounds these: latency.  1280x720, four rounds: 1.72 ms while a thread walked a line, 0.34 now.
struct Offer {
    long long d;
    int seed;
};
__device__ __forceinline__ Offer lesser(Offer a, Offer b) { return b.d < a.d || (b.d == a.d && b.seed < a.seed) ? b : a; }
__device__ __forceinline__ long long seed_step(int q, int before) { return 256 + (long long)abs(q - before); }

// Rows, a warp each: left to right, then right to left, 32 pixels at a time (their steps' prefix sums, then the
// offers' prefix minima, by shuffles; the last pixel's offer goes on to the next 32).
__global__ void __launch_bounds__(128) k_seed_rows(const __grid_constant__ Batch bt) {
    begin_kernel();
    const PairView& pv = bt.view(blockIdx.z);
    const int W = pv.W, y = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (y >= pv.H) return;
    const int* q = pv.gq + (size_t)y * W;
    long long* dist = seed_dist(pv) + (size_t)y * W;
    int* seed = seed_of(pv) + (size_t)y * W;
    for (int way = 0; way < 2; ++way) {
        Offer carry{1ll << 62, -1};
        int before = 0;  // the grey before the chunk
        auto at = [&](int i) { return way ? W - 1 - i : i; };
        Offer next{1ll << 62, -1};
        int qn = 0;
        if (lane < W) next = Offer{dist[at(lane)], seed[at(lane)]}, qn = q[at(lane)];
        for (int i0 = 0; i0 < W; i0 += 32) {
            const int i = i0 + lane;
            const bool in = i < W;
            const Offer own = next;
            const int qi = qn;
            if (i + 32 < W) next = Offer{dist[at(i + 32)], seed[at(i + 32)]}, qn = q[at(i + 32)];
            int qb = __shfl_up_sync(FULL, qi, 1);
            if (lane == 0) qb = before;
            long long sum = i == 0 || !in ? 0 : seed_step(qi, qb);
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const long long t = __shfl_up_sync(FULL, sum, o);
                if (lane >= o) sum += t;
            }
            Offer best{in ? own.d - sum : 1ll << 62, in ? own.seed : -1};
            if (lane == 0) best = lesser(best, carry);
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const Offer t{__shfl_up_sync(FULL, best.d, o), __shfl_up_sync(FULL, best.seed, o)};
                if (lane >= o) best = lesser(best, t);
            }
            best.d += sum;
            if (in && best.seed >= 0 && (best.d != own.d || best.seed != own.seed)) {
                dist[at(i)] = best.d;
                seed[at(i)] = best.seed;
            }
            carry = best.seed >= 0 ? best : Offer{1ll << 62, -1};
            carry = Offer{__shfl_sync(FULL, carry.d, 31), __shfl_sync(FULL, carry.seed, 31)};
            before = __shfl_sync(FULL, qi, 31);
        }
        __syncwarp();
    }
}

// Columns, 32 a block: top to bottom, then bottom to top.  Each of the block's 32 warps takes a section of the rows, a
// lane a column: it walks its section for the steps' sum and the offer at its end, adds up the sections before it, and walks
// it again with that offer.
__global__ void __launch_bounds__(1024) k_seed_columns(const __grid_constant__ Batch bt) {
    begin_kernel();
    constexpr int U = 8;  // rows loaded together
    const PairView& pv = bt.view(blockIdx.z);
    const int W = pv.W, H = pv.H, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if ((int)blockIdx.x * 32 >= W) return;  // past this pair's columns (block-uniform)
    const int x = blockIdx.x * 32 + lane;
    const bool in = x < W;
    const int* q = pv.gq + (in ? x : 0);
    long long* dist = seed_dist(pv) + (in ? x : 0);
    int* seed = seed_of(pv) + (in ? x : 0);
    __shared__ long long sum[32][32], end_d[32][32];
    __shared__ int end_s[32][32];
    const int len = (H + 31) >> 5, lo = warp * len, hi = min(lo + len, H);
    for (int way = 0; way < 2; ++way) {
        // row r of the scan; the section [lo, hi) of the scan's order is this warp's
        auto at = [&](int r) { return (size_t)(way ? H - 1 - r : r) * W; };
        const int first = lo < hi && lo > 0 ? q[at(lo - 1)] : 0;
        auto walk = [&](Offer o, bool store, long long& total) {
            int before = first;
            total = 0;
            for (int r0 = lo; r0 < hi; r0 += U) {
                Offer own[U];
                int qr[U];
#pragma unroll
                for (int k = 0; k < U; ++k) {
                    const size_t p = at(min(r0 + k, hi - 1));
                    own[k] = Offer{dist[p], seed[p]};
                    qr[k] = q[p];
                }
#pragma unroll
                for (int k = 0; k < U; ++k) {
                    if (r0 + k >= hi) break;
                    const long long step = r0 + k ? seed_step(qr[k], before) : 0;
                    before = qr[k];
                    total += step;
                    if (o.seed >= 0) o.d += step;
                    const Offer best = lesser(own[k], o);
                    if (store && in && best.seed >= 0 && (best.d != own[k].d || best.seed != own[k].seed)) {
                        dist[at(r0 + k)] = best.d;
                        seed[at(r0 + k)] = best.seed;
                    }
                    o = best;
                }
            }
            return o;
        };
        long long total;
        const Offer none{1ll << 62, -1};
        const Offer end = walk(none, false, total);
        sum[warp][lane] = total;
        end_d[warp][lane] = end.d;
        end_s[warp][lane] = end.seed;
        __syncthreads();
        Offer carry = none;
        for (int k = 0; k < warp; ++k) {
            if (carry.seed >= 0) carry.d += sum[k][lane];
            carry = lesser(carry, Offer{end_d[k][lane], end_s[k][lane]});
        }
        walk(carry, true, total);
        __syncthreads();  // before the sections change hands: upwards a warp's rows are another's
    }
}

// Final flow (plane flow, else the NNF offset, else with a seed the seed's
// plane at this pixel) and occlusion: no plane, a cue flag, or colour error
// after warping by the final flow >= occ_thresh.
template <int ST>
__global__ void k_final(const __grid_constant__ Batch bt, PlaneParams pp, int interp, const __grid_constant__ FinalOut out) {
    begin_kernel();
    const PairView& pv = bt.view(blockIdx.z);
    const int dir = 0;
    const int* seed = interp ? seed_of(pv) : nullptr;
    float* flow = out.flow[blockIdx.z];
    uint8_t* occ = out.occ[blockIdx.z];
    const int W = pv.W, H = pv.H, n = pv.n;
    const Labels acc = pv.acc[dir];
    const void* src = pv.img[dir];
    const void* tgt = pv.img[1 - dir];
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int y = i / W, x = i - y * W;
        int bx, by;
        float fx, fy;
        const bool as = acc.m[i] >= 0;
        if (as) {
            const int2 v = acc.v[i];
            const float2 r = acc.r[i];
            flow[2 * i] = (float)v.x + r.x;
            flow[2 * i + 1] = (float)v.y + r.y;
            bx = x + v.x + (r.x < 0.f ? -1 : 0);
            fx = r.x < 0.f ? r.x + 1.f : r.x;
            by = y + v.y + (r.y < 0.f ? -1 : 0);
            fy = r.y < 0.f ? r.y + 1.f : r.y;
        } else {
            const int2 v = pv.nnf[dir][i];
            flow[2 * i] = (float)v.x;
            flow[2 * i + 1] = (float)v.y;
            bx = x + v.x;
            by = y + v.y;
            fx = fy = 0.f;
            const int sd = seed ? seed[i] : -1;
            if (sd >= 0) {  // edge-aware fill: the seed's plane here, or the seed's flow
                const Mef m = pv.mef[dir][acc.m[sd]];
                int kx, ky;
                float gx, gy;
                if (mef_flow(m, (float)(x - m.ox), (float)(y - m.oy), kx, gx, ky, gy)) {
                    flow[2 * i] = (float)kx + gx;
                    flow[2 * i + 1] = (float)ky + gy;
                } else {
                    const int2 vs = acc.v[sd];
                    const float2 rs = acc.r[sd];
                    flow[2 * i] = (float)vs.x + rs.x;
                    flow[2 * i + 1] = (float)vs.y + rs.y;
                }
            }
        }
        bool o = !as || (pv.cue[dir][i] & CUE_M2O);
        if (!in_frame_tol(bx, fx, W) || !in_frame_tol(by, fy, H))
            o = true;
        else if (!(colour_delta<ST>(src, tgt, W, H, x, y, bx, fx, by, fy) < pp.occ_thresh))
            o = true;
        occ[i] = o ? 1 : 0;
    }
}

// ---------------------------------------------------------------- state import / export helpers
// Evaluation forms of imported absolute homographies.
__global__ void k_import_models(const __grid_constant__ Batch bt, int nlev, int m) {
    begin_kernel();
    const PairView& pv = bt.view(blockIdx.z);
    const LevelGeom* geoms = bt.geo[blockIdx.z];
    const int dir = blockIdx.y;
    for (int id = blockIdx.x * blockDim.x + threadIdx.x; id < m; id += gridDim.x * blockDim.x) {
        const int cell_all = id >> 1;
        int l = 0;
        while (l + 1 < nlev && geoms[l + 1].base <= cell_all) ++l;
        const LevelGeom g = geoms[l];
        const int cell = cell_all - g.base;
        const int cx = cell % g.gx.count, cy = cell / g.gx.count;
        const int ox = win_pos(g.gx, g.h, cx) + g.s / 2, oy = win_pos(g.gy, g.h, cy) + g.s / 2;
        double Hl[9];
        abs_to_local(pv.mh[dir] + (size_t)id * 9, ox, oy, Hl);
        Mef f = {};
        const bool ok = make_mef(Hl, ox, oy, f);
        f.valid = ok && pv.mi[dir][(size_t)id * kMI + MI_VALID] ? 1 : 0;
        pv.mef[dir][id] = f;
    }
}

// labels <-> (model, L, flow) with flow = v + r in double
__global__ void k_labels_export(Labels l, int n, int* om, float* oL, double* of) {
    begin_kernel();
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        om[i] = l.m[i];
        oL[i] = l.L[i];
        of[2 * i] = (double)l.v[i].x + (double)l.r[i].x;
        of[2 * i + 1] = (double)l.v[i].y + (double)l.r[i].y;
    }
}
__global__ void k_labels_import(Labels l, int n, int m, const int* im, const float* iL, const double* iF,
                                int* flag) {
    begin_kernel();
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        int id = im[i];
        const double fx = iF[2 * i], fy = iF[2 * i + 1];
        // |flow| < 2^30 (and finite): the rounded offset fits an int
        const bool flow_ok = fabs(fx) < 1073741824.0 && fabs(fy) < 1073741824.0;
        if (id < -1 || id >= m || (id >= 0 && !flow_ok)) {
            *flag = 1;
            id = -1;
        }
        l.m[i] = id;
        l.L[i] = iL[i];
        if (flow_ok) {
            const double vx = floor(fx + 0.5), vy = floor(fy + 0.5);
            l.v[i] = make_int2((int)vx, (int)vy);
            l.r[i] = make_float2((float)(fx - vx), (float)(fy - vy));
        } else {
            l.v[i] = make_int2(0, 0);
            l.r[i] = make_float2(0.f, 0.f);
        }
    }
}

// ---------------------------------------------------------------- launchers
// Every launch covers np pairs (blockIdx.z); grids are sized for the largest pair, and each block past its own
// pair's pixels or windows does nothing.
// Launches a kernel whose windows' matches are in dynamic shared memory.  Its limit is raised before the first launch on each
// device, by whichever thread comes first.
template <auto KERNEL>
static void launch_windows(dim3 grid, unsigned threads, size_t shared, cudaStream_t st, const Batch& bt, int level, int stage,
                           const PlaneParams& pp) {
    static std::atomic<unsigned long long> raised{0};  // bit d: on device d
    int dev = 0;
    cudaGetDevice(&dev);
    const unsigned long long bit = dev < 64 ? 1ull << dev : 0ull;
    if (!(raised.load(std::memory_order_acquire) & bit)) {
        const int largest = kMaxCell * kMaxCell * (int)sizeof(float4);
        if (cudaFuncSetAttribute(KERNEL, cudaFuncAttributeMaxDynamicSharedMemorySize, largest) == cudaSuccess)
            raised.fetch_or(bit, std::memory_order_release);
    }
    launch_kernel(KERNEL, grid, threads, shared, st, bt, level, stage, pp);
}
template <int ST>
static void launch_ransac_st(const Batch& bt, int np, int level, int s, int max_cells, int stage, bool any_offsets,
                             const PlaneParams& pp, cudaStream_t st) {
    const int nc = max_cells;
    const dim3 solve((2 * nc + 31) / 32, 1, np);
    if (s <= 16) {
        const dim3 fgrid((nc + kRansacWarps - 1) / kRansacWarps, 2, np), grid((nc + 7) / 8, 2, np);
        auto fit = [&](auto kernel) { launch_kernel(kernel, fgrid, 32 * kRansacWarps, 0, st, bt, level, stage, pp); };
        if (any_offsets) {
            fit(s <= 8 ? k_ransac_warp<64, FIT_ANY> : k_ransac_warp<256, FIT_ANY>);
            fit(s <= 8 ? k_ransac_warp<64, FIT_FAR> : k_ransac_warp<256, FIT_FAR>);
        } else {
            fit(s <= 8 ? k_ransac_warp<64, FIT_NEAR> : k_ransac_warp<256, FIT_NEAR>);
        }
        launch_kernel(k_refit_solve, solve, 32, 0, st, bt, level, pp);
        launch_kernel(k_ransac_finish_warp<ST>, grid, 256, 0, st, bt, level, stage, pp);
        return;
    }
    const size_t smem = (size_t)s * s * sizeof(float4), fit_smem = (size_t)block_cap(s) * sizeof(float4);
    const dim3 grid(nc, 2, np);
    auto fit = [&](auto narrow, auto broad) {
        if (ransac_wide(s, 2 * nc * np))
            launch_windows<broad()>(grid, 512, fit_smem, st, bt, level, stage, pp);
        else
            launch_windows<narrow()>(grid, 256, fit_smem, st, bt, level, stage, pp);
    };
    if (any_offsets) {
        fit([] { return k_ransac_block<256, FIT_ANY>; }, [] { return k_ransac_block<512, FIT_ANY>; });
        fit([] { return k_ransac_block<256, FIT_FAR>; }, [] { return k_ransac_block<512, FIT_FAR>; });
    } else {
        fit([] { return k_ransac_block<256, FIT_NEAR>; }, [] { return k_ransac_block<512, FIT_NEAR>; });
    }
    launch_kernel(k_refit_solve, solve, 32, 0, st, bt, level, pp);
    launch_windows<k_ransac_finish_block<ST>>(grid, 256, smem, st, bt, level, stage, pp);
}
void launch_ransac(const Batch& bt, int np, int level, int s, int max_cells, int stage, bool any_offsets,
                   const PlaneParams& pp, cudaStream_t st) {
    switch (pp.storage) {
        case 0: launch_ransac_st<0>(bt, np, level, s, max_cells, stage, any_offsets, pp, st); break;
        case 1: launch_ransac_st<1>(bt, np, level, s, max_cells, stage, any_offsets, pp, st); break;
        case 2: launch_ransac_st<2>(bt, np, level, s, max_cells, stage, any_offsets, pp, st); break;
    }
}

template <int ST>
static void launch_assign_st(const Batch& bt, dim3 grid, int level, int stage, int again, const PlaneParams& pp, cudaStream_t st) {
    if (stage == 1 && !again)
        launch_kernel(k_assign<ST, ASSIGN_TENT>, grid, 256, 0, st, bt, level, pp);
    else if (stage == 1)
        launch_kernel(k_assign<ST, ASSIGN_ST1>, grid, 256, 0, st, bt, level, pp);
    else if (!again)
        launch_kernel(k_assign<ST, ASSIGN_LVL>, grid, 256, 0, st, bt, level, pp);
    else
        launch_kernel(k_assign<ST, ASSIGN_LVL_AGAIN>, grid, 256, 0, st, bt, level, pp);
}
void launch_assign(const Batch& bt, int np, int level, int stage, int again, const PlaneParams& pp, int grid_blocks,
                   cudaStream_t st) {
    const dim3 grid(grid_blocks, 2, np);
    switch (pp.storage) {
        case 0: launch_assign_st<0>(bt, grid, level, stage, again, pp, st); break;
        case 1: launch_assign_st<1>(bt, grid, level, stage, again, pp, st); break;
        case 2: launch_assign_st<2>(bt, grid, level, stage, again, pp, st); break;
    }
}

void launch_cues(const Batch& bt, int np, int level, int max_cells, int stage, int which, const PlaneParams& pp,
                 int grid_blocks, cudaStream_t st) {
    const int cb = (max_cells + 255) / 256;
    launch_kernel(k_cue_counts, dim3(grid_blocks, 2, np), 256, 0, st, bt, level, stage, which, pp);
    launch_kernel(k_cue_invalidate, dim3(cb, 2, np), 256, 0, st, bt, level, stage, pp);
}

void launch_many_to_one(const Batch& bt, int np, const PlaneParams& pp, int grid_blocks, cudaStream_t st) {
    launch_kernel(k_m2o_claim, dim3(grid_blocks, 2, np), 256, 0, st, bt);
    launch_kernel(k_m2o_resolve, dim3(grid_blocks, 2, np), 256, 0, st, bt, pp);
}

void launch_merge_update(const Batch& bt, int np, const PlaneParams& pp, int grid_blocks, cudaStream_t st) {
    launch_kernel(k_merge_update, dim3(grid_blocks, 2, np), 256, 0, st, bt, pp);
}

// Label sets of a pair: 0 acc, 1 tent, 2 st1, 3 lvl.
__device__ __forceinline__ Labels label_set(const PairView& pv, int set, int dir) {
    return set == 0 ? pv.acc[dir] : (set == 1 ? pv.tent[dir] : (set == 2 ? pv.st1[dir] : pv.lvl[dir]));
}
__global__ void k_copy_labels(const __grid_constant__ Batch bt, int from, int to) {
    begin_kernel();
    const PairView& pv = bt.view(blockIdx.z);
    const int dir = blockIdx.y;
    const Labels a = label_set(pv, from, dir), b = label_set(pv, to, dir);
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < pv.n; i += gridDim.x * blockDim.x) {
        b.m[i] = a.m[i];
        b.L[i] = a.L[i];
        b.v[i] = a.v[i];
        b.r[i] = a.r[i];
    }
}
void launch_copy_labels(const Batch& bt, int np, int from, int to, int grid_blocks, cudaStream_t st) {
    launch_kernel(k_copy_labels, dim3(grid_blocks, 2, np), 256, 0, st, bt, from, to);
}

void launch_fill(const Batch& bt, int np, const PlaneParams& pp, int iters, int grid_blocks, cudaStream_t st) {
    // ping-pong between acc and tent (tent is free after the last level)
    const dim3 grid(grid_blocks, 2, np);
    for (int it = 0; it < iters; ++it) {
        switch (pp.storage) {
            case 0: launch_kernel(k_fill<0>, grid, 256, 0, st, bt, it & 1, it == 0, pp); break;
            case 1: launch_kernel(k_fill<1>, grid, 256, 0, st, bt, it & 1, it == 0, pp); break;
            case 2: launch_kernel(k_fill<2>, grid, 256, 0, st, bt, it & 1, it == 0, pp); break;
        }
    }
    if (iters & 1) launch_copy_labels(bt, np, 1, 0, grid_blocks, st);  // the result sits in tent
}

void launch_fill_seeds(const Batch& bt, int np, int max_w, int max_h, int rounds, int grid_blocks, cudaStream_t st) {
    launch_kernel(k_seed_init, dim3(grid_blocks, 1, np), 256, 0, st, bt);
    for (int r = 0; r < rounds; ++r) {
        launch_kernel(k_seed_rows, dim3((max_h + 3) / 4, 1, np), 128, 0, st, bt);
        launch_kernel(k_seed_columns, dim3((max_w + 31) / 32, 1, np), 1024, 0, st, bt);
    }
}

void launch_final(const Batch& bt, int np, const PlaneParams& pp, int interp, const FinalOut& out, int grid_blocks,
                  cudaStream_t st) {
    const dim3 grid(grid_blocks, 1, np);
    switch (pp.storage) {
        case 0: launch_kernel(k_final<0>, grid, 256, 0, st, bt, pp, interp, out); break;
        case 1: launch_kernel(k_final<1>, grid, 256, 0, st, bt, pp, interp, out); break;
        case 2: launch_kernel(k_final<2>, grid, 256, 0, st, bt, pp, interp, out); break;
    }
}

// Clears the models of every window of every level (model ids below m_models).
__global__ void k_reset_models(const __grid_constant__ Batch bt) {
    begin_kernel();
    const PairView& pv = bt.view(blockIdx.z);
    const int dir = blockIdx.y;
    for (int id = blockIdx.x * blockDim.x + threadIdx.x; id < pv.m_models; id += gridDim.x * blockDim.x) {
#pragma unroll
        for (int q = 0; q < 9; ++q) pv.mh[dir][(size_t)id * 9 + q] = 0.0;
        pv.mef[dir][id] = Mef{};
#pragma unroll
        for (int q = 0; q < kMI; ++q) pv.mi[dir][(size_t)id * kMI + q] = 0;
    }
}
void launch_reset_models(const Batch& bt, int np, int max_models, cudaStream_t st) {
    if (max_models <= 0) return;  // no plane levels: no model table (an empty grid is not a launch)
    launch_kernel(k_reset_models, dim3((max_models + 255) / 256, 2, np), 256, 0, st, bt);
}

__global__ void k_reset_labels(const __grid_constant__ Batch bt, float eps) {
    begin_kernel();
    const PairView& pv = bt.view(blockIdx.z);
    const int dir = blockIdx.y;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < pv.n; i += gridDim.x * blockDim.x) {
        pv.acc[dir].m[i] = -1;
        pv.acc[dir].L[i] = eps;
        pv.acc[dir].v[i] = make_int2(0, 0);
        pv.acc[dir].r[i] = make_float2(0.f, 0.f);
        pv.cue[dir][i] = 0;
        pv.frozen[dir][i] = 0;
    }
}
__global__ void k_frozen_from_labels(const __grid_constant__ Batch bt) {
    begin_kernel();
    const PairView& pv = bt.view(blockIdx.z);
    const int dir = blockIdx.y;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < pv.n; i += gridDim.x * blockDim.x)
        pv.frozen[dir][i] = pv.acc[dir].m[i] >= 0;
}
void launch_frozen_from_labels(const Batch& bt, int np, int grid_blocks, cudaStream_t st) {
    launch_kernel(k_frozen_from_labels, dim3(grid_blocks, 2, np), 256, 0, st, bt);
}

void launch_reset_labels(const Batch& bt, int np, float eps, int grid_blocks, cudaStream_t st) {
    launch_kernel(k_reset_labels, dim3(grid_blocks, 2, np), 256, 0, st, bt, eps);
}

template <int ST>
__global__ void k_frames_export(const __grid_constant__ Batch bt, float* dst) {
    begin_kernel();
    const PairView& pv = bt.view(blockIdx.z);
    const int dir = blockIdx.y;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < pv.n; i += gridDim.x * blockDim.x) {
        const float4 a = ldpix<ST>(pv.img[dir], i);
        reinterpret_cast<float4*>(dst)[(size_t)dir * pv.n + i] = a;
    }
}
void launch_frames_export(const Batch& bt, int n, int storage, float* dst, cudaStream_t st) {
    const dim3 grid((n + 255) / 256, 2);
    switch (storage) {
        case 0: launch_kernel(k_frames_export<0>, grid, 256, 0, st, bt, dst); break;
        case 1: launch_kernel(k_frames_export<1>, grid, 256, 0, st, bt, dst); break;
        case 2: launch_kernel(k_frames_export<2>, grid, 256, 0, st, bt, dst); break;
    }
}

void launch_import_models(const Batch& bt, int nlev, int m, cudaStream_t st) {
    if (m <= 0) return;  // no model table
    launch_kernel(k_import_models, dim3((m + 255) / 256, 2), 256, 0, st, bt, nlev, m);
}

void launch_labels_export(const Labels& l, int n, int* om, float* oL, double* of, cudaStream_t st) {
    launch_kernel(k_labels_export, (n + 255) / 256, 256, 0, st, l, n, om, oL, of);
}
void launch_labels_import(const Labels& l, int n, int m, const int* im, const float* iL, const double* iF, int* flag,
                          cudaStream_t st) {
    launch_kernel(k_labels_import, (n + 255) / 256, 256, 0, st, l, n, m, im, iL, iF, flag);
}

}  // namespace gpm

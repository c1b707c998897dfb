// Frame ingest and PatchMatch kernels (sm_103a).
//
// PatchMatch (Sec. 3.1; Barnes et al. 2009) with red-black scheduling: one
// launch per half-iteration updates every pixel of one colour from the state
// before the launch (its four neighbours all have the other colour).  One
// warp evaluates one pixel: each lane owns ceil(T/32) taps of the (2r+1)^2
// patch, keeps their source texels in registers for all candidates, and the
// per-candidate cost is one integer reduction of the lanes' sums (rounded to
// 2^-24), identical on every lane, so the accept/reject decision is
// warp-uniform.  At levels >= 1 the patch is
// distorted by the pixel's home-window plane (Sec. 3.3.2 with the plane
// distortion compensation of Sec. 3.1.3): tap d samples the target frame at
// p + v + G(s) - G(p), s = clamp(p + d).
#include "common.cuh"
#include "kernels.h"
#include "../../include/gpm.h"

namespace gpm {

constexpr unsigned FULL = 0xffffffffu;

// ---------------------------------------------------------------- ingest
// Optional HSV histogram equalisation (Sec. 4.2): V = max(R, G, B) of each
// frame is equalised over 256 bins of [0, 1] (bin = min(255, floor(256 V)),
// V' = (cdf(bin) - cdf_min) / (n - cdf_min), cdf_min the count of the lowest
// occupied bin) with H and S kept.  At fixed H and S the hexcone RGB is
// proportional to V, so the equalised pixel is RGB * V' / V (V' grey for
// black pixels).  A frame with a single occupied bin is left unchanged
// (its table holds -1).
// Element k of an input frame as a float: FP32, FP16 or BF16 (gpm_dtype), each converted exactly.
__device__ __forceinline__ float in_elem(const void* f, int dtype, int64_t k) {
    if (dtype == GPM_F16) return __half2float(reinterpret_cast<const __half*>(f)[k]);
    if (dtype == GPM_BF16) return __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(f)[k]);
    return reinterpret_cast<const float*>(f)[k];
}

__device__ __forceinline__ int v_bin(float v) {
    float x = floorf(v * 256.f);
    if (!(x >= 0.f)) x = 0.f;
    return (int)fminf(x, 255.f);
}

// Up to four pixels of a row from element e (a multiple of 12 from the row's start), as 12 floats; `wide`: FP32 rows on
// 16-byte boundaries, so that four whole pixels are three loads.  Elements past `cnt` pixels are 0.
__device__ __forceinline__ bool wide_rows(const void* f, int dtype, int64_t stride) {
    return dtype == GPM_F32 && (stride & 3) == 0 && (reinterpret_cast<uintptr_t>(f) & 15) == 0;
}
__device__ __forceinline__ void load_px4(const void* f, int dtype, int64_t e, int cnt, bool wide, float (&v)[12]) {
    if (wide && cnt == 4) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float4 a = __ldg(reinterpret_cast<const float4*>(reinterpret_cast<const float*>(f) + e) + k);
            v[4 * k] = a.x, v[4 * k + 1] = a.y, v[4 * k + 2] = a.z, v[4 * k + 3] = a.w;
        }
        return;
    }
#pragma unroll
    for (int k = 0; k < 12; ++k) v[k] = k < 3 * cnt ? in_elem(f, dtype, e + k) : 0.f;
}

// Clears the V histograms of the jobs that equalise (blockIdx.z = job).
__global__ void k_vhist_zero(const __grid_constant__ IngestJobs J) {
    begin_kernel();
    const IngestJob& j = J.j[blockIdx.z];
    if (j.hist)
        for (int k = threadIdx.x; k < 2 * 256; k += blockDim.x) j.hist[k] = 0;
}

// V histogram of each frame (blockIdx.y = frame, blockIdx.z = job); hist holds 2 x 256 zeroed counts.
__global__ void __launch_bounds__(512) k_vhist(const __grid_constant__ IngestJobs J) {
    begin_kernel();
    const IngestJob& j = J.j[blockIdx.z];
    if (!j.hist) return;  // block-uniform
    const int W = j.W, H = j.H;
    __shared__ int h[256];
    for (int k = threadIdx.x; k < 256; k += blockDim.x) h[k] = 0;
    __syncthreads();
    const void* f = blockIdx.y ? j.f2 : j.f1;
    const bool wide = wide_rows(f, j.dtype, j.stride);
    const int Q = (W + 3) >> 2, n = Q * H;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int y = i / Q, x = 4 * (i - y * Q), cnt = min(4, W - x);
        float v[12];
        load_px4(f, j.dtype, (int64_t)y * j.stride + 3 * x, cnt, wide, v);
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (q < cnt) atomicAdd(&h[v_bin(fmaxf(v[3 * q], fmaxf(v[3 * q + 1], v[3 * q + 2])))], 1);
    }
    __syncthreads();
    for (int k = threadIdx.x; k < 256; k += blockDim.x)
        if (h[k]) atomicAdd(&j.hist[blockIdx.y * 256 + k], h[k]);
}

// Equalised V per bin of both frames, into lut (shared memory), from their counts: an inclusive scan, a frame by 256
// threads each.  Every thread of the block must call it (at least 512); it ends with a barrier.
__device__ __forceinline__ void equalized_v(const int* hist, int n, float* lut) {
    __shared__ int total[16], lowest[16];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    int own = 0, sum = 0;
    if (t < 512) {  // warp-uniform
        own = sum = hist[t];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(FULL, sum, o);
            if (lane >= o) sum += v;
        }
        const unsigned occupied = __ballot_sync(FULL, own > 0);
        const int low = __shfl_sync(FULL, own, occupied ? __ffs(occupied) - 1 : 0);  // 0 if none
        if (lane == 31) total[warp] = sum, lowest[warp] = low;
    }
    __syncthreads();
    if (t < 512) {
        int cmin = 0;  // the count of the lowest occupied bin
        for (int b = (warp & 8) + 7; b >= (warp & 8); --b) {
            if (b < warp) sum += total[b];
            if (lowest[b] > 0) cmin = lowest[b];
        }
        // counts below 2^24 are exact floats, so this is the correctly rounded quotient
        lut[t] = cmin == 0 || cmin == n ? -1.f : (float)(sum - cmin) / (float)(n - cmin);
    }
    __syncthreads();
}

__device__ __forceinline__ float3 equalize_px(float r, float g, float b, const float* lut) {
    const float v = fmaxf(r, fmaxf(g, b));
    const float l = lut[v_bin(v)];
    if (l < 0.f) return make_float3(r, g, b);
    if (v > 0.f) {
        const float k = l / v;
        return make_float3(r * k, g * k, b * k);
    }
    return make_float3(l, l, l);
}

// ---------------------------------------------------------------- census codes (Sec. 6)
// Grey = R + G + B in FP64 (the same additions as the FP64 oracle, so the
// same values), stored as an orderable integer key: the bits of a
// non-negative double increase with it, negative ones are mirrored; + 0.0
// turns -0 into +0.  The 24 comparisons per pixel then run on the integer
// pipe with exactly the outcomes of comparing the doubles.
__global__ void k_grey_keys(const __grid_constant__ IngestJobs J) {
    begin_kernel();
    const IngestJob& j = J.j[blockIdx.z];
    if (!j.k1) return;  // block-uniform
    const int W = j.W, n = j.W * j.H;
    const int64_t stride = j.stride;
    const void* f = blockIdx.y ? j.f2 : j.f1;
    long long* k = blockIdx.y ? j.k2 : j.k1;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int y = i / W, x = i - y * W;
        const int64_t e = (int64_t)y * stride + 3 * x;
        const double g = (((double)in_elem(f, j.dtype, e) + (double)in_elem(f, j.dtype, e + 1)) +
                          (double)in_elem(f, j.dtype, e + 2)) + 0.0;
        const long long b = __double_as_longlong(g);
        k[i] = b >= 0 ? b : (long long)(0x8000000000000000ull - (unsigned long long)b) - 1;
    }
}

// 5x5 census code per pixel: bit k (raster order without the centre, neighbours clamped into the frame) set iff
// the neighbour's grey is below the centre's.
__global__ void k_census(const __grid_constant__ IngestJobs J) {
    begin_kernel();
    const IngestJob& j = J.j[blockIdx.z];
    if (!j.k1) return;  // block-uniform
    const int W = j.W, H = j.H, n = j.W * j.H;
    const long long* k = blockIdx.y ? j.k2 : j.k1;
    uint32_t* c = blockIdx.y ? j.c2 : j.c1;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int y = i / W, x = i - y * W;
        const long long kc = k[i];
        uint32_t code = 0;
        int bit = 0;
#pragma unroll
        for (int dy = -2; dy <= 2; ++dy)
#pragma unroll
            for (int dx = -2; dx <= 2; ++dx) {
                if (dx == 0 && dy == 0) continue;
                const int nx = min(max(x + dx, 0), W - 1), ny = min(max(y + dy, 0), H - 1);
                code |= (k[ny * W + nx] < kc ? 1u : 0u) << bit;
                ++bit;
            }
        c[i] = code;
    }
}

template <int ST>
__device__ __forceinline__ void store_pix(void* base, int i, float r, float g, float b) {
    if constexpr (ST == 0) {
        reinterpret_cast<float4*>(base)[i] = make_float4(r, g, b, 0.f);
    } else if constexpr (ST == 1) {
        __half2 lo = __floats2half2_rn(r, g), hi = __floats2half2_rn(b, 0.f);
        uint2 u;
        u.x = *reinterpret_cast<uint32_t*>(&lo);
        u.y = *reinterpret_cast<uint32_t*>(&hi);
        reinterpret_cast<uint2*>(base)[i] = u;
    } else {
        __nv_bfloat162 lo = __floats2bfloat162_rn(r, g), hi = __floats2bfloat162_rn(b, 0.f);
        uint2 u;
        u.x = *reinterpret_cast<uint32_t*>(&lo);
        u.y = *reinterpret_cast<uint32_t*>(&hi);
        reinterpret_cast<uint2*>(base)[i] = u;
    }
}

// A sum of floats: those in [2^-16, 2) as exact integers of 2^-40 (a block adds at most 2^21 of them, below 2^62), the
// others in FP64.  An FP64 addition and the conversion before it take the FP64 pipe, 64 cycles each a warp instruction on
// GB300; the integers take ten of one cycle.
struct FrameSum {
    long long fix = 0;
    double rest = 0;
    __device__ __forceinline__ void add(float v) {
        const unsigned u = __float_as_uint(v);
        if (u - 0x37800000u < 0x40000000u - 0x37800000u)
            fix += (long long)((u & 0x7FFFFFu) | 0x800000u) << ((u >> 23) - 110);
        else if (v != 0.f)
            rest += (double)v;
    }
    // The block's total (of 1024 threads), on thread 0: a fixed tree, so the same bits at every run.
    __device__ __forceinline__ double total(long long* sf, double* sr) {
        const bool any = __syncthreads_or(rest != 0.0);  // also true for NaN
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            fix += __shfl_xor_sync(FULL, fix, o);
            if (any) rest += __shfl_xor_sync(FULL, rest, o);
        }
        if ((threadIdx.x & 31) == 0) sf[threadIdx.x >> 5] = fix, sr[threadIdx.x >> 5] = rest;
        __syncthreads();
        if (threadIdx.x >= 32) return 0;
        fix = sf[threadIdx.x];
        rest = sr[threadIdx.x];
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            fix += __shfl_xor_sync(FULL, fix, o);
            if (any) rest += __shfl_xor_sync(FULL, rest, o);
        }
        return (double)fix * 9.094947017729282379150390625e-13 + rest;  // 2^-40
    }
};

// Sums of both frames (equalised where the job asks for it) per block, over rows blockIdx.x, + gridDim.x, ...
// (blockIdx.z = job), and frame 1 stored, which needs no gain.  What bounds it: the FP32 and integer pipes (a pixel pair with
// equalisation takes 150 instructions).  1280x720 with equalisation: sums and table 60 us with FP64 additions, 25 with
// integers and the table in a launch of its own, 17 now with frame 1's half of k_pack besides.
template <int ST>
__global__ void __launch_bounds__(1024) k_frame_sums(const __grid_constant__ IngestJobs J) {
    begin_kernel();
    const IngestJob& j = J.j[blockIdx.z];
    const int W = j.W, H = j.H;
    __shared__ long long sf[2][32];
    __shared__ double sr[2][32];
    __shared__ float lut[512];
    if (j.hist) {  // block-uniform
        equalized_v(j.hist, W * H, lut);
        if (blockIdx.x == 0 && threadIdx.x < 512) j.lut[threadIdx.x] = lut[threadIdx.x];
    }
    FrameSum sum[2];
    // the block's rows as one sequence of four-pixel groups, so that short rows leave no thread idle
    const int rows = (H - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;  // at most 0 past the last row
    const int Q = (W + 3) >> 2;
    const bool wide = wide_rows(j.f1, j.dtype, j.stride) && wide_rows(j.f2, j.dtype, j.stride);
    for (int i = threadIdx.x; i < rows * Q; i += blockDim.x) {
        const int r = i / Q, x = 4 * (i - r * Q), y = blockIdx.x + r * gridDim.x, cnt = min(4, W - x);
        const int64_t e = (int64_t)y * j.stride + 3 * x;
        float v[2][12];
        load_px4(j.f1, j.dtype, e, cnt, wide, v[0]);
        load_px4(j.f2, j.dtype, e, cnt, wide, v[1]);
#pragma unroll
        for (int f = 0; f < 2; ++f)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if (q >= cnt) break;
                float3 p = make_float3(v[f][3 * q], v[f][3 * q + 1], v[f][3 * q + 2]);
                if (j.hist) p = equalize_px(p.x, p.y, p.z, lut + 256 * f);
                sum[f].add(p.x), sum[f].add(p.y), sum[f].add(p.z);
                if (f == 0) store_pix<ST>(j.o1, y * W + x + q, p.x, p.y, p.z);
            }
    }
    const double ta = sum[0].total(sf[0], sr[0]), tb = sum[1].total(sf[1], sr[1]);
    if (threadIdx.x == 0) {
        j.partial[2 * blockIdx.x] = ta;
        j.partial[2 * blockIdx.x + 1] = tb;
    }
}

// The gain of frame 2, mean(I1) / mean(I2), or 1: every block of k_pack adds the partial sums itself, in one order
// (a launch of its own took 15 us, all of it one thread's 256 dependent FP64 additions).
__device__ __forceinline__ double frame_gain(const double* partial, int enable) {
    __shared__ double sg;
    static_assert(kIngestPartialBlocks == 128, "four partial sums a lane");
    if (threadIdx.x < 32) {
        double a = 0, b = 0;
        if (enable) {
            double2 v[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) v[k] = reinterpret_cast<const double2*>(partial)[threadIdx.x + 32 * k];
            a = (v[0].x + v[1].x) + (v[2].x + v[3].x);
            b = (v[0].y + v[1].y) + (v[2].y + v[3].y);
#pragma unroll
            for (int o = 16; o; o >>= 1) {
                a += __shfl_xor_sync(FULL, a, o);
                b += __shfl_xor_sync(FULL, b, o);
            }
        }
        if (threadIdx.x == 0) sg = (enable && b > 0) ? a / b : 1.0;
    }
    __syncthreads();
    return sg;
}

// (float)((double)q * g), mostly without the FP64 pipe: gh + gl holds g to 2^-48, the product's high part and its
// error are exact, and the rest is within 2^-46 of the product, so the sum s rounds as the FP64 product does unless a
// change of 2^-44 moves it (one product in 2^18); those, and products far from 1, are taken in FP64.  `wide`: g itself
// is far from 1.  k_pack at 1280x720: 21 -> 14 us.
struct Gain {
    double g;
    float gh, gl;
    bool wide;
    __device__ __forceinline__ explicit Gain(double v) : g(v), gh((float)v), gl((float)(v - (double)(float)v)) {
        wide = !(v > 9.0949470177292824e-13 && v < 1099511627776.0);  // 2^-40, 2^40
    }
    __device__ __noinline__ static float wide_product(float q, double g) { return (float)((double)q * g); }
    __device__ __forceinline__ float times(float q) const {
        const float p = __fmul_rn(q, gh), e = __fmaf_rn(q, gh, -p), t = __fmaf_rn(q, gl, e);
        const float d = __fmul_rn(fabsf(p), 5.6843418860808015e-14f);  // 2^-44
        const float s = __fadd_rn(p, t);
        const bool sure = s == __fadd_rn(p, __fadd_rn(t, d)) && s == __fadd_rn(p, __fsub_rn(t, d)) &&
                          fabsf(p) > 8.67361738e-19f && fabsf(p) < 1.15292150e18f;  // 2^-60, 2^60
        if (!wide && (sure || q == 0.f)) return q == 0.f ? q : s;
        return wide_product(q, g);
    }
};

// Frame 2 stored, equalised where the job asks for it and times the gain (blockIdx.z = job).
template <int ST>
__global__ void k_pack(const __grid_constant__ IngestJobs J, int gain_enable) {
    begin_kernel();
    const IngestJob& j = J.j[blockIdx.z];
    const int W = j.W, H = j.H;
    const float* lut = j.hist ? j.lut + 256 : nullptr;
    const Gain g(frame_gain(j.partial, gain_enable));
    const int n = W * H;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int y = i / W, x = i - y * W;
        const int64_t e = (int64_t)y * j.stride + 3 * x;
        float3 q = make_float3(in_elem(j.f2, j.dtype, e), in_elem(j.f2, j.dtype, e + 1), in_elem(j.f2, j.dtype, e + 2));
        if (lut) q = equalize_px(q.x, q.y, q.z, lut);
        store_pix<ST>(j.o2, i, g.times(q.x), g.times(q.y), g.times(q.z));
    }
}

// ---------------------------------------------------------------- patch machinery
template <int R>
struct Patch {
    static constexpr int D = 2 * R + 1;
    static constexpr int T = D * D;
    static constexpr int NT = (T + 31) / 32;
};

// Per-lane patch state of one pixel.  Tap j of the lane reads the target at
// (tx + cx, ty + cy) for candidate offset c -- the clamped source pixel for a
// square patch, or the integer part of p + G(s) - G(p) with fraction (fx, fy)
// for a plane-distorted one -- and tidx = ty * W + tx.  [xlo, xhi] x [ylo, yhi]
// bounds every texel the patch touches at offset 0 (including the +1 column
// and row of bilinear taps), so a candidate whose shifted bounds stay inside
// the frame needs no clamping: one add per tap gives the texel index.
template <int R>
struct LanePatch {
    float4 a[Patch<R>::NT];   // source texels of the lane's taps
    uint32_t code[Patch<R>::NT];  // census data term: source codes of the lane's taps
    int tx[Patch<R>::NT], ty[Patch<R>::NT], tidx[Patch<R>::NT];
    float fx[Patch<R>::NT], fy[Patch<R>::NT];
    // offsets c with oxlo <= c.x < oxlo + oxnum and oylo <= c.y < oylo + oynum keep every texel of the patch
    // inside the frame (the unclamped, one-add indexing path)
    int oxlo, oxnum, oylo, oynum;
    bool warped;
};

// The patch touches texels [xlo, xhi] x [ylo, yhi] at offset 0; offsets keep them inside the frame iff
// -xlo <= c.x <= W-1-xhi (likewise y).  A patch wider than the frame has no such offset (an incumbent may be any
// imported value, so a start that no offset reaches would not do).
template <int R>
__device__ __forceinline__ void set_interior_box(LanePatch<R>& lp, int xlo, int xhi, int ylo, int yhi, int W, int H) {
    lp.oxlo = -xlo;
    lp.oxnum = max((W - xhi) + xlo, 0);
    lp.oylo = -ylo;
    lp.oynum = max((H - yhi) + ylo, 0);
}

// CENSUS: src holds the frame's census codes (uint32 per pixel) instead of texels.
// Wp > 0: src is a padded copy (row length Wp, border kPad) and the target
// is read from the other frame's copy: tidx then indexes the clamped tap
// there, and a candidate whose target pixel is in the frame needs no clamping
// for any tap (the interior box, in unpadded terms, is then not consulted).
template <int R, int ST, bool CENSUS = false>
__device__ __forceinline__ void load_patch(LanePatch<R>& lp, const void* src, int W, int H, int px, int py,
                                           int lane, int Wp = 0) {
#pragma unroll
    for (int j = 0; j < Patch<R>::NT; ++j) {
        const int t = lane + 32 * j;
        const int tt = t < Patch<R>::T ? t : 0;
        const int dy = tt / Patch<R>::D - R, dx = tt % Patch<R>::D - R;
        lp.tx[j] = min(max(px + dx, 0), W - 1);
        lp.ty[j] = min(max(py + dy, 0), H - 1);
        const int si = lp.ty[j] * W + lp.tx[j];
        lp.tidx[j] = Wp > 0 ? (lp.ty[j] + kPad) * Wp + lp.tx[j] + kPad : si;
        if (CENSUS)
            lp.code[j] = __ldg(reinterpret_cast<const uint32_t*>(src) + si);
        else
            lp.a[j] = ldpix<ST>(src, Wp > 0 ? lp.tidx[j] : si);
        lp.fx[j] = 0.f;
        lp.fy[j] = 0.f;
    }
    set_interior_box(lp, max(px - R, 0), min(px + R, W - 1), max(py - R, 0), min(py + R, H - 1), W, H);
    lp.warped = false;
}

// Tap displacements G(s) - G(p) for the plane m at pixel p, from the local
// Jacobian form: with J the derivative of G at p and c = (g0, g1) / den(p),
// G(p + d) - G(p) = J d / (1 + c . d) exactly.
// Returns whether every tap moves less than one pixel from its square place (warp-uniform).
template <int R>
__device__ __forceinline__ bool warp_taps(LanePatch<R>& lp, const Mef& m, int px, int py, int W, int H, int lane) {
    const float ux = (float)(px - m.ox), uy = (float)(py - m.oy);
    const float e = m.e0 + m.g0 * ux + m.g1 * uy;
    const float den = 1.f + e;
    const float Sx = m.b0 * ux + m.h1 * uy - ux * e;
    const float Sy = m.h3 * ux + m.b4 * uy - uy * e;
    // local target of p: X = u + D(u)
    const float rden = __frcp_rn(den);
    const float X = ux + (m.h2h + (m.h2l + (Sx - m.h2h * e) * rden));
    const float Y = uy + (m.h5h + (m.h5l + (Sy - m.h5h * e) * rden));
    const float j00 = (1.f + m.b0 - X * m.g0) * rden, j01 = (m.h1 - X * m.g1) * rden;
    const float j10 = (m.h3 - Y * m.g0) * rden, j11 = (1.f + m.b4 - Y * m.g1) * rden;
    const float c0 = m.g0 * rden, c1 = m.g1 * rden;
    int xlo = 1 << 30, xhi = -(1 << 30), ylo = 1 << 30, yhi = -(1 << 30);
    bool near = true;
#pragma unroll
    for (int j = 0; j < Patch<R>::NT; ++j) {
        const float dx = (float)(lp.tx[j] - px), dy = (float)(lp.ty[j] - py);
        const float rq = __frcp_rn(1.f + c0 * dx + c1 * dy);
        const float ex = (j00 * dx + j01 * dy) * rq;
        const float ey = (j10 * dx + j11 * dy) * rq;
        const float fx = floorf(ex), fy = floorf(ey);
        near = near && fabsf(ex - dx) < 0.99f && fabsf(ey - dy) < 0.99f;
        lp.tx[j] = px + (int)fx;
        lp.ty[j] = py + (int)fy;
        lp.tidx[j] = lp.ty[j] * W + lp.tx[j];
        lp.fx[j] = ex - fx;
        lp.fy[j] = ey - fy;
        if (lane + 32 * j < Patch<R>::T) {
            xlo = min(xlo, lp.tx[j]);
            xhi = max(xhi, lp.tx[j] + 1);
            ylo = min(ylo, lp.ty[j]);
            yhi = max(yhi, lp.ty[j] + 1);
        }
    }
    set_interior_box(lp, __reduce_min_sync(FULL, xlo), __reduce_max_sync(FULL, xhi), __reduce_min_sync(FULL, ylo),
                     __reduce_max_sync(FULL, yhi), W, H);
    lp.warped = true;
    return __all_sync(FULL, near);
}

// Target sample of tap j for candidate offset c (off = c.y * W + c.x).  IN:
// the offset keeps every texel of the patch inside the frame (one add gives
// the index); otherwise the coordinates are clamped.  The caller makes this
// warp-uniform choice once per candidate, outside the tap loop.
template <int R, int ST, bool IN>
__device__ __forceinline__ float3 tap_sample(const LanePatch<R>& lp, const void* tgt, int W, int H, int j, int2 c,
                                             int off) {
    if (!lp.warped) {
        const int idx = IN ? lp.tidx[j] + off
                           : min(max(lp.ty[j] + c.y, 0), H - 1) * W + min(max(lp.tx[j] + c.x, 0), W - 1);
        const float4 v = ldpix<ST>(tgt, idx);
        return make_float3(v.x, v.y, v.z);
    }
    if (IN) {
        const int i0 = lp.tidx[j] + off;
        return blend4(ldpix<ST>(tgt, i0), ldpix<ST>(tgt, i0 + 1), ldpix<ST>(tgt, i0 + W), ldpix<ST>(tgt, i0 + W + 1),
                      lp.fx[j], lp.fy[j]);
    }
    return bilinear<ST>(tgt, W, H, lp.tx[j] + c.x, lp.fx[j], lp.ty[j] + c.y, lp.fy[j]);
}

template <int R>
__device__ __forceinline__ bool interior_of(const LanePatch<R>& lp, int2 c) {
    return (unsigned)(c.x - lp.oxlo) < (unsigned)lp.oxnum && (unsigned)(c.y - lp.oylo) < (unsigned)lp.oynum;
}

// Raw patch cost of offset (vx, vy): the sum over taps and channels of
// |difference|.  The NNF cost buffer holds these sums (strict-less decisions
// compare them directly); the exported cost is the sum divided by 3T.
// The warp's total of the lanes' tap sums: each lane's sum rounded to a
// multiple of 2^-23 and the integers added exactly by one redux, so every
// lane gets the same bits.  A lane's sum is at most 18 (three taps of three
// channels, each |difference| at most 2: frames in [0, 1], a gain below 2),
// so the total of at most 243 channel terms stays below 2^32; it is within
// 32 * 2^-24 = 2^-19 of the exact total of the lane sums, and costs one
// reduction instead of five dependent shuffles and additions.
__device__ __forceinline__ float warp_sum_q23(float s) {
    const unsigned q = __float2uint_rn(s * 8388608.f);
    return (float)__reduce_add_sync(FULL, q) * 1.1920928955078125e-07f;
}

template <int R, int ST, bool IN>
__device__ __forceinline__ float patch_sum_in(const LanePatch<R>& lp, const void* tgt, int W, int H, int2 c, int lane) {
    const int off = c.y * W + c.x;
    float s = 0.f;
#pragma unroll
    for (int j = 0; j < Patch<R>::NT; ++j) {
        const int t = lane + 32 * j;
        if (t < Patch<R>::T) s += absdiff3(lp.a[j], tap_sample<R, ST, IN>(lp, tgt, W, H, j, c, off));
    }
    return warp_sum_q23(s);
}
template <int R, int ST>
__device__ __forceinline__ float patch_sum(const LanePatch<R>& lp, const void* tgt, int W, int H, int px, int py,
                                           int vx, int vy, int lane) {
    const int2 c = make_int2(vx, vy);
    return interior_of<R>(lp, c) ? patch_sum_in<R, ST, true>(lp, tgt, W, H, c, lane)
                                 : patch_sum_in<R, ST, false>(lp, tgt, W, H, c, lane);
}

// ---------------------------------------------------------------- census data term (Sec. 6)
// Square patches only (level 0).  The cost is the sum over taps of the
// Hamming distance of the source and target census codes: an exact integer,
// summed across the warp by one redux, so decisions are exact and the
// abandon test needs no margin (a partial sum at or above the best cannot
// become strictly lower).  Returns false when abandoned; best < 0 never
// abandons.
template <int R, bool IN>
__device__ __forceinline__ bool census_sum_in(const LanePatch<R>& lp, const uint32_t* tgt, int W, int H, int2 c,
                                              int best, int& sum, int lane) {
    const int off = c.y * W + c.x;
    int s = 0;
#pragma unroll
    for (int j = 0; j < Patch<R>::NT; ++j) {
        const int t = lane + 32 * j;
        if (t < Patch<R>::T) {
            const int idx = IN ? lp.tidx[j] + off
                               : min(max(lp.ty[j] + c.y, 0), H - 1) * W + min(max(lp.tx[j] + c.x, 0), W - 1);
            s += __popc(lp.code[j] ^ __ldg(tgt + idx));
        }
        const int tot = (int)__reduce_add_sync(FULL, (unsigned)s);
        if (j + 1 < Patch<R>::NT) {
            if (best >= 0 && tot >= best) return false;
        } else {
            sum = tot;
        }
    }
    return true;
}
template <int R>
__device__ __forceinline__ bool census_sum(const LanePatch<R>& lp, const uint32_t* tgt, int W, int H, int2 c,
                                           int best, int& sum, int lane) {
    return interior_of<R>(lp, c) ? census_sum_in<R, true>(lp, tgt, W, H, c, best, sum, lane)
                                 : census_sum_in<R, false>(lp, tgt, W, H, c, best, sum, lane);
}

// Integer threshold for the abandon test of tap_sum: with thr the best raw
// sum so far, returns ceil(thr * 2^19 * (1 + 2^-21)) + 1.  A partial bound at
// or above it means the exact total of the lane sums is at least
// thr (1 + 2^-21) + 2^-19; the final sum (warp_sum_q23) is within 2^-19 of
// that total and then rounded to a float, so it stays above thr.
__device__ __forceinline__ int abandon_threshold(float thr) {
    return __float2int_ru(__fmul_ru(thr * 524288.f, 1.f + 4.76837158203125e-07f)) + 1;
}

// Raw tap sum of candidate offset c (over taps and channels of |difference|,
// before the division by 3T), abandoned once it cannot win.  After a tested
// 32-tap chunk every lane floors its partial sum to a multiple of 2^-19 and
// the warp adds those integers exactly (one redux): a lower bound of the
// exact partial sum.  The terms are non-negative and FP32 addition is
// monotonic, so a lane's final sum is at least its partial sum; a bound at
// or above `ithr` (abandon_threshold) therefore means the full cost is above
// the best, and the strict-less test would reject the candidate anyway: the
// function returns false.  Each lane accumulates its taps in the same order
// as patch_sum and the total is warp_sum_q24's, so a full sum is bitwise the
// same as patch_sum's.
template <int R, int ST, bool IN>
__device__ __forceinline__ bool tap_sum_in(const LanePatch<R>& lp, const void* tgt, int W, int H, int2 c, int ithr,
                                        float& sum, int& nch, int lane) {
    const int off = c.y * W + c.x;
    float s = 0.f;
#pragma unroll
    for (int j = 0; j < Patch<R>::NT; ++j) {
        const int t = lane + 32 * j;
        if (t < Patch<R>::T) s += absdiff3(lp.a[j], tap_sample<R, ST, IN>(lp, tgt, W, H, j, c, off));
        if (j + 1 < Patch<R>::NT) {
            // floor(min(s * 2^19, 2^23 - 1)): exact scaling, clamp (keeps a lower bound), truncation in the
            // mantissa of 2^23
            const unsigned q =
                (unsigned)(__float_as_int(__fadd_rz(fminf(s * 524288.f, 8388607.f), 8388608.f)) - 0x4B000000);
            if ((int)__reduce_add_sync(FULL, q) >= ithr) {
                nch = j + 1;
                return false;
            }
        }
        if (j + 1 == Patch<R>::NT) sum = warp_sum_q23(s);
    }
    nch = Patch<R>::NT;
    return true;
}
// For the plane levels, where a chunk costs four gathers per tap (level 0 sums in full: the patch-sum bound has
// already removed most losing candidates there).
template <int R, int ST>
__device__ __forceinline__ bool tap_sum(const LanePatch<R>& lp, const void* tgt, int W, int H, int2 c, int ithr,
                                        float& sum, int& nch, int lane) {
    return interior_of<R>(lp, c) ? tap_sum_in<R, ST, true>(lp, tgt, W, H, c, ithr, sum, nch, lane)
                                 : tap_sum_in<R, ST, false>(lp, tgt, W, H, c, ithr, sum, nch, lane);
}

// A candidate offset in one word (|c.x|, |c.y| < 2^15 for frames below 2^15 pixels a side).
__device__ __forceinline__ uint32_t pack_off(int2 c) { return (uint32_t)(uint16_t)c.x | ((uint32_t)c.y << 16); }
__device__ __forceinline__ int2 unpack_off(uint32_t k) { return make_int2((int)(int16_t)(k & 0xFFFFu), (int)k >> 16); }

__device__ __forceinline__ unsigned lanemask_lt(int lane) { return (1u << lane) - 1u; }

// Lanes whose candidate is to be evaluated: valid, not the incumbent and not
// a repeat of a lower lane's candidate.  Skipping those changes nothing: the
// cost of an offset is a deterministic function of it, and a repeat can never
// be strictly cheaper than the best so far, which is at most its first cost.  The offsets are matched as one word: a
// match of 64-bit keys takes the warp as long as an evaluation (plane sweeps of a 1024x436 pair 5.45 -> 5.02 ms, the
// census sweeps of a 512x384 one 5.55 -> 4.97).
__device__ __forceinline__ unsigned fresh_lanes(bool ok, int2 c, int2 inc, int lane) {
    ok = ok && !(c.x == inc.x && c.y == inc.y);
    const unsigned some = __ballot_sync(FULL, ok);
    bool keep = false;
    if (ok) keep = (__match_any_sync(some, pack_off(c)) & lanemask_lt(lane)) == 0;
    return __ballot_sync(FULL, keep);
}

// Home-window plane of p at a level (residual-stage model first), or nullptr.
__device__ __forceinline__ const Mef* home_plane(const LevelGeom& g, const Mef* mef, int x, int y) {
    const int cx = home_index(g.gx, g.s, g.h, x), cy = home_index(g.gy, g.s, g.h, y);
    const int cell = cy * g.gx.count + cx;
    const Mef* m2 = mef + (g.base + cell) * 2 + 1;
    if (m2->valid) return m2;
    const Mef* m1 = mef + (g.base + cell) * 2;
    if (m1->valid) return m1;
    return nullptr;
}

// ---------------------------------------------------------------- init
// The costs of two pixels' candidates at once (patches l1, l2, interior offsets
// c1, c2 into the padded target copy of row length Wp): the same arithmetic per
// pixel as patch_sum_in, with the two pixels' gathers in flight together.
template <int R, int ST>
__device__ __forceinline__ void patch_sum_pair_in(const LanePatch<R>& l1, const LanePatch<R>& l2, const void* tgt,
                                                  int Wp, int H, int2 c1, int2 c2, float& sum1, float& sum2) {
    const int o1 = c1.y * Wp + c1.x, o2 = c2.y * Wp + c2.x;
    float s1 = 0.f, s2 = 0.f;
#pragma unroll
    for (int j = 0; j < Patch<R>::NT; ++j) {
        const int t = (int)(threadIdx.x & 31) + 32 * j;
        if (t < Patch<R>::T) {
            const float3 v1 = tap_sample<R, ST, true>(l1, tgt, Wp, H, j, c1, o1);
            const float3 v2 = tap_sample<R, ST, true>(l2, tgt, Wp, H, j, c2, o2);
            s1 += absdiff3(l1.a[j], v1);
            s2 += absdiff3(l2.a[j], v2);
        }
    }
    sum1 = warp_sum_q23(s1);
    sum2 = warp_sum_q23(s2);
}

template <int R, int ST, bool CENSUS>
__global__ void __launch_bounds__(256) k_pm_init(const __grid_constant__ Batch bt, uint32_t k0, uint32_t k1) {
    begin_kernel();
    const PairView& pv = bt.view(blockIdx.z);
    const int dir = blockIdx.y;
    const int lane = threadIdx.x & 31;
    const int W = pv.W, H = pv.H, n = pv.n;
    const void* src = CENSUS ? (const void*)pv.code[dir] : pv.img[dir];
    const void* tgt = CENSUS ? (const void*)pv.code[1 - dir] : pv.img[1 - dir];
    const int nw = gridDim.x * (blockDim.x >> 5);
    const int first = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if constexpr (!CENSUS) {
        // two pixels per warp and round (i and i + nw): their gathers share the latency
        for (int i = first; i < n; i += 2 * nw) {
            const int i2 = i + nw < n ? i + nw : i;  // warp-uniform; the last odd pixel is computed twice
            const int y1 = i / W, x1 = i - y1 * W, y2 = i2 / W, x2 = i2 - y2 * W;
            const uint32_t tag = stream_tag(RNG_INIT, dir, 0, 0);
            const uint4 w1 = philox((uint32_t)i, 0u, tag, pv.pair_id, k0, k1);
            const uint4 w2 = philox((uint32_t)i2, 0u, tag, pv.pair_id, k0, k1);
            const int2 c1 = make_int2((int)(w1.x % (uint32_t)W) - x1, (int)(w1.y % (uint32_t)H) - y1);
            const int2 c2 = make_int2((int)(w2.x % (uint32_t)W) - x2, (int)(w2.y % (uint32_t)H) - y2);
            LanePatch<R> l1, l2;
            load_patch<R, ST>(l1, pv.imgp[dir], W, H, x1, y1, lane, pv.Wp);
            load_patch<R, ST>(l2, pv.imgp[dir], W, H, x2, y2, lane, pv.Wp);
            float s1, s2;
            patch_sum_pair_in<R, ST>(l1, l2, pv.imgp[1 - dir], pv.Wp, H, c1, c2, s1, s2);
            if (lane == 0) {
                pv.nnf[dir][i] = c1;
                pv.cost[dir][i] = s1;
                pv.nnf[dir][i2] = c2;
                pv.cost[dir][i2] = s2;
                if (pv.evals) atomicAdd(&pv.evals[GPM_COUNT_INIT], i2 != i ? 2ull : 1ull);
            }
        }
        return;
    }
    for (int i = first; i < n; i += nw) {
        const int y = i / W, x = i - y * W;
        const uint4 w = philox((uint32_t)i, 0u, stream_tag(RNG_INIT, dir, 0, 0), pv.pair_id, k0, k1);
        const int vx = (int)(w.x % (uint32_t)W) - x, vy = (int)(w.y % (uint32_t)H) - y;
        LanePatch<R> lp;
        float c;
        if constexpr (CENSUS) {
            load_patch<R, ST, CENSUS>(lp, src, W, H, x, y, lane);
            int sum = 0;
            census_sum<R>(lp, reinterpret_cast<const uint32_t*>(tgt), W, H, make_int2(vx, vy), -1, sum, lane);
            c = (float)sum;
        } else {
            load_patch<R, ST>(lp, pv.imgp[dir], W, H, x, y, lane, pv.Wp);
            c = patch_sum_in<R, ST, true>(lp, pv.imgp[1 - dir], pv.Wp, H, make_int2(vx, vy), lane);
        }
        if (lane == 0) {
            pv.nnf[dir][i] = make_int2(vx, vy);
            pv.cost[dir][i] = c;
            if (pv.evals) atomicAdd(&pv.evals[GPM_COUNT_INIT], 1ull);
        }
    }
}

// ---------------------------------------------------------------- recost (level >= 1)
template <int R, int ST>
__global__ void __launch_bounds__(256) k_pm_recost(const __grid_constant__ Batch bt, int level) {
    begin_kernel();
    const PairView& pv = bt.view(blockIdx.z);
    const LevelGeom g = bt.geom(blockIdx.z, level);
    const int dir = blockIdx.y;
    const int lane = threadIdx.x & 31;
    const int W = pv.W, H = pv.H;
    const void* src = pv.img[dir];
    const void* tgt = pv.img[1 - dir];
    const int nw = gridDim.x * (blockDim.x >> 5);
    const int half = pv.n;  // list capacity per colour
    for (int col = 0; col < 2; ++col) {
        const int cnt = pv.list_count[dir * 2 + col];
        const int* list = pv.list[dir] + col * half;
        for (int w = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); w < cnt; w += nw) {
            const int i = list[w];
            const int y = i / W, x = i - y * W;
            LanePatch<R> lp;
            // an imported offset may be any integer: past 2^30 on either side every tap is off the frame on that side,
            // and sums of coordinates stay in range
            int2 v = pv.nnf[dir][i];
            v.x = min(max(v.x, -(1 << 30)), 1 << 30);
            v.y = min(max(v.y, -(1 << 30)), 1 << 30);
            float c;
            // the padded copy serves square patches whose target pixel is in the frame (an imported offset
            // need not be)
            if (level > 0 || (unsigned)(x + v.x) >= (unsigned)W || (unsigned)(y + v.y) >= (unsigned)H) {
                load_patch<R, ST>(lp, src, W, H, x, y, lane);
                if (level > 0) {
                    const Mef* G = home_plane(g, pv.mef[dir], x, y);
                    if (G) warp_taps<R>(lp, *G, x, y, W, H, lane);
                }
                c = patch_sum<R, ST>(lp, tgt, W, H, x, y, v.x, v.y, lane);
            } else {
                load_patch<R, ST>(lp, pv.imgp[dir], W, H, x, y, lane, pv.Wp);
                c = patch_sum_in<R, ST, true>(lp, pv.imgp[1 - dir], pv.Wp, H, v, lane);
            }
            if (lane == 0) {
                pv.cost[dir][i] = c;
                if (pv.evals) atomicAdd(&pv.evals[GPM_COUNT_INIT], 1ull);
            }
        }
    }
}

// ---------------------------------------------------------------- patch-sum lower bound (level 0)
// For a pixel p whose patch stays inside the frame and an offset c whose
// target pixel is in the frame, the raw cost is
// sum_t sum_ch |a - b| >= sum_ch |sum_t a - sum_t b| = LB, the sums read from
// the frames' box images (k_box_sums).  A candidate is dropped, without a
// tap, when LB_f - m >= bc (1 + 2^-16) + 2^-18, which allows for rounding on
// both sides: the computed cost C_f is at least C (1 - 2^-18) - 2^-19 (FP32
// sums of at most 9 terms per lane, the 2^-23 rounding of 32 lane sums, one
// conversion), and the exact LB is at least the computed one minus
// m = 2^-19 (sum of both boxes' channels) (each box sum carries at most 16
// FP32 roundings of its own size, then six FP32 operations), so the test
// implies C_f >= bc: the candidate could not be strictly cheaper.
__device__ __forceinline__ float box_lb(float4 b1, float4 b2) {
    const float lb = fabsf(b1.x - b2.x) + fabsf(b1.y - b2.y) + fabsf(b1.z - b2.z);
    const float m = 1.9073486328125e-06f * (((b1.x + b1.y) + b1.z) + ((b2.x + b2.y) + b2.z));
    return lb - m;
}
__device__ __forceinline__ float box_threshold(float bc) {
    return fmaf(bc, 1.52587890625e-05f, bc) + 3.814697265625e-06f;
}

// A second, tighter bound for the random candidates that pass the first, at r = 4 with 16-byte texels: the patch is nine
// regions of 3 x 3 texels, and the raw cost is at least the sum over them of sum_ch |region sum of a - region sum of b|,
// the region sums from k_box_sums (in the many-to-one keys' buffer, idle at level 0).  Half of those candidates go;
// a test costs a lane 100 instructions and 9 gathers of 8 bytes, an evaluation the warp as many and 81 gathers of 16.
// 1024x436: the 16 sweeps 5.20 -> 4.73 ms.  Where it does not pay: 8-byte texels (half the gathers' cost: 1920x1080 FP16
// 17.7 -> 17.8 ms), r = 3 (49 texels, four 3 x 3 corners and the cross between them: 511x383 1.17 -> 1.19 ms), and
// propagated candidates (mostly good ones: with them tested 4.87 ms).
// A sum is held as 16-bit multiples of 2^-11 per channel (.x = r | g << 16, .y = b; at most 9 * 2), off by at most
// 2^-12 and eight FP32 roundings, 2.54e-4 in all; bit 31 of .y marks a texel out of the domain of in_domain, for which
// nothing is dropped.  The margin: 54 such values, 0.0138 = 28.2 units.
template <int R, int ST>
constexpr bool kRegionBound = R == 4 && ST == 0;
struct RegionSums {
    uint2 a[9];  // the source patch's
    __device__ __forceinline__ static int at(int k, int W) { return (k / 3 - 1) * 3 * W + (k % 3 - 1) * 3; }
    __device__ __forceinline__ void load(const uint2* s1, int W) {
#pragma unroll
        for (int k = 0; k < 9; ++k) a[k] = __ldg(s1 + at(k, W));
    }
    // Whether a candidate cannot cost less than thr (box_threshold's); s2: the sums at its target pixel.
    __device__ __forceinline__ bool excludes(const uint2* s2, int W, float thr) const {
        unsigned flags = 0, lb = 0;
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            const uint2 b = __ldg(s2 + at(k, W));
            flags |= a[k].y | b.y;
            lb = __dp2a_lo(__vmaxu2(a[k].x, b.x) - __vminu2(a[k].x, b.x), 0x0101u, lb);
            lb = __dp2a_lo(__vmaxu2(a[k].y, b.y) - __vminu2(a[k].y, b.y), 0x0001u, lb);
        }
        return !(flags >> 31) && (float)lb - 29.f >= thr * 2048.f;
    }
};

// ---------------------------------------------------------------- interval lower bound (levels >= 1)
// A warped tap samples between pixels, so the patch sums above do not apply; but a bilinear sample less than one pixel
// from a place lies between the least and the greatest texel of the 3 x 3 around it.  k_interval_sums replaces
// the box images, idle after level 0, by the sums over each pixel's patch of those minima and maxima, as
// FP16 rounded outwards (6 values in 12 of 16 bytes: one load a candidate).  For a pixel whose patch stays in the frame
// and whose taps move less than one pixel (any plane of local scale within a quarter of 1 at r = 4; no plane: not at
// all), and an offset c whose target pixel is in the frame, the raw cost is at least
// LB = sum_ch max(sum a - sum max, sum min - sum a, 0).  The candidate is dropped when LB - 3e-4 reaches
// box_threshold(bc): 3e-4 covers sum a (2^-16 and two roundings a channel) and the blends' rounding (81 taps,
// 4 units of 2^-24 of at most 2, a channel); the sums' own rounding is in the widening before FP16.
__device__ __forceinline__ float interval_lb(uint4 iv, float ar, float ag, float ab) {
    const float2 u = __half22float2(*reinterpret_cast<const __half2*>(&iv.x));  // min r, g
    const float2 v = __half22float2(*reinterpret_cast<const __half2*>(&iv.y));  // min b, max r
    const float2 w = __half22float2(*reinterpret_cast<const __half2*>(&iv.z));  // max g, b
    return (fmaxf(fmaxf(ar - v.y, u.x - ar), 0.f) + fmaxf(fmaxf(ag - w.x, u.y - ag), 0.f)) +
           (fmaxf(fmaxf(ab - w.y, v.x - ab), 0.f) - 3e-4f);
}
// Texels the bound is for: frames in [0, 1] and a gain below 2 (others may overflow warp_sum_q23's total).
__device__ __forceinline__ bool in_domain(float r, float g, float b) {
    return fminf(fminf(r, g), b) >= 0.f && fmaxf(fmaxf(r, g), b) <= 2.f && r + g + b >= 0.f;  // false for NaN
}
// The warp's sums of the patch's source texels, per channel, to 2^-16; false if one is out of the bound's domain.
template <int R>
__device__ __forceinline__ bool patch_sums(const LanePatch<R>& lp, int lane, float& ar, float& ag, float& ab) {
    float r = 0.f, g = 0.f, b = 0.f;
    bool ok = true;
#pragma unroll
    for (int j = 0; j < Patch<R>::NT; ++j)
        if (lane + 32 * j < Patch<R>::T) {
            ok = ok && in_domain(lp.a[j].x, lp.a[j].y, lp.a[j].z);
            r += lp.a[j].x;
            g += lp.a[j].y;
            b += lp.a[j].z;
        }
    auto total = [](float v) {  // at most 6 a lane
        return (float)__reduce_add_sync(FULL, __float2uint_rn(v * 1048576.f)) * 9.5367431640625e-07f;
    };
    ar = total(r);
    ag = total(g);
    ab = total(b);
    return __all_sync(FULL, ok);
}

// ---------------------------------------------------------------- sweep
// PLANES: levels >= 1 (restricted pixel list, plane-distorted patches, plane
// candidates); otherwise level 0 with the census data term (level 0 with
// colour patches runs k_pm_sweep0).
//
// Candidates come in two lists, one candidate per lane, in the fixed order:
// (A) propagation from the left, right, upper and lower neighbours (lanes
// 0-3), then at levels >= 1 the models of the windows covering p in window
// order, first stage then residual stage (lanes 4..21); (B) random search
// around the best offset after A, radius R0 >> k on lane k.  The warp walks
// each list in lane order through one evaluation site (a small kernel body
// keeps the instruction cache warm) and accepts with the strict-less rule.
// After the first iteration only the offsets of neighbours that moved in
// their last half-iteration are candidates of list A, and no window's model:
// the others were candidates at this pixel's visit one iteration ago, so
// their cost is at least the best of then, and the best never rises (an
// offset that became the best is repeated by it).  pv.resid is free during
// the sweeps and holds which pixels moved.
// CENSUS (level 0 only): the census data term on the frames' code images.
template <int R, int ST, bool PLANES, bool CENSUS>
__global__ void __launch_bounds__(256, 4) k_pm_sweep(const __grid_constant__ Batch bt, int level, int it, int phase, uint32_t k0,
                                                  uint32_t k1) {
    begin_kernel();
    static_assert(!(PLANES && CENSUS), "the census data term is for square patches");
    static_assert(PLANES || CENSUS, "level 0 with colour patches runs k_pm_sweep0");
    __shared__ PairView spv;
    const PairView& pv = shared_view(bt, spv);
    const LevelGeom g = bt.geom(blockIdx.z, level);
    const int dir = blockIdx.y;
    const int lane = threadIdx.x & 31;
    const int W = pv.W, H = pv.H;
    const void* src = CENSUS ? (const void*)pv.code[dir] : pv.img[dir];
    const void* tgt = CENSUS ? (const void*)pv.code[1 - dir] : pv.img[1 - dir];
    int2* __restrict__ nnf = pv.nnf[dir];
    uint8_t* __restrict__ moved = pv.resid[dir];
    const int nw = gridDim.x * (blockDim.x >> 5);
    const int hw = (W + 1) >> 1;
    const int total = !PLANES ? H * hw : pv.list_count[dir * 2 + phase];
    const int* list = !PLANES ? nullptr : pv.list[dir] + phase * pv.n;
    const int R0 = max(W, H);
    int nrad = 0;  // search radii R0 >> k >= 1
    while ((R0 >> nrad) >= 1) ++nrad;
    const uint32_t tag = stream_tag(RNG_SEARCH, dir, level, 0);
    // Level 0: a block takes tiles of 8 x 8 pixels of this colour (16 x 8 image pixels), its eight warps one
    // row of the tile per round, so that successive rounds reuse the target region already in the SM's L1.
    // Plane levels: the compacted pixel list, grid-strided.
    const int wid = threadIdx.x >> 5;
    const int ntx = (hw + 7) >> 3, ntiles = ntx * ((H + 7) >> 3);
    int w = blockIdx.x * (blockDim.x >> 5) + wid;
    int next = PLANES && w < total ? list[w] : 0;  // the warp's next listed pixel, loaded a visit ahead (128x96 pair
                                                       // 1.59 -> 1.53 ms, 80/40 px levels of 1024x436 10.04 -> 9.74)
    for (int rnd = 0;; ++rnd) {
        int x, y, i;
        if (!PLANES) {
            const int tile = blockIdx.x + (rnd >> 3) * gridDim.x;
            if (tile >= ntiles) break;  // block-uniform
            const int ty = tile / ntx, tx = tile - ty * ntx;
            y = 8 * ty + (rnd & 7);
            const int xh = 8 * tx + wid;
            if (y >= H || xh >= hw) continue;
            x = 2 * xh + ((y + phase) & 1);
            if (x >= W) continue;
            i = y * W + x;
        } else {
            if (w >= total) break;
            i = next;
            w += nw;
            if (w < total) next = list[w];
            y = i / W;
            x = i - y * W;
        }
        LanePatch<R> lp;
        load_patch<R, ST, CENSUS>(lp, src, W, H, x, y, lane);
        bool bounded = false;  // the interval bound applies
        float ar = 0.f, ag = 0.f, ab = 0.f;
        if (PLANES) {
            const Mef* G = home_plane(g, pv.mef[dir], x, y);
            const bool near = G ? warp_taps<R>(lp, *G, x, y, W, H, lane) : true;
            bounded = near && x >= R && y >= R && x < W - R && y < H - R && patch_sums<R>(lp, lane, ar, ag, ab);
        }
        const int2 before = nnf[i];
        int2 best = before;
        float bc = pv.cost[dir][i];  // raw sum of the incumbent
        int ithr = CENSUS ? 0 : abandon_threshold(bc);
        int nev = 0, ntap = 0;
        // list A
        int2 cand = make_int2(0, 0);
        bool ok = false;
        if (lane < 4) {
            const int nx = x + (lane == 0 ? -1 : (lane == 1 ? 1 : 0));
            const int ny = y + (lane == 2 ? -1 : (lane == 3 ? 1 : 0));
            if (nx >= 0 && nx < W && ny >= 0 && ny < H && (it == 0 || moved[ny * W + nx])) {
                cand = nnf[ny * W + nx];
                const int tx = x + cand.x, ty = y + cand.y;
                ok = tx >= 0 && tx < W && ty >= 0 && ty < H;
            }
        } else if (PLANES && it == 0 && lane < 4 + 18) {
            int fx0, nrx, fy0, nry;
            const int nxw = covering_range(g.gx, g.s, g.h, x, fx0, nrx);
            const int nyw = covering_range(g.gy, g.s, g.h, y, fy0, nry);
            const int j = lane - 4, st = j & 1, wk = j >> 1;       // window wk of at most 3 x 3, stage st
            const int a = nxw == 1 ? wk : (nxw == 2 ? wk >> 1 : (wk * 11) >> 5);  // wk / nxw for wk < 9
            const int b = wk - a * nxw;
            if (nxw > 0 && a < nyw) {
                const int cell = covering_at(g.gy, fy0, nry, a) * g.gx.count + covering_at(g.gx, fx0, nrx, b);
                const Mef m = pv.mef[dir][(g.base + cell) * 2 + st];
                int kx, ky;
                float fx, fy;
                if (m.valid && mef_flow(m, (float)(x - m.ox), (float)(y - m.oy), kx, fx, ky, fy)) {
                    float rx, ry;
                    round_split(kx, fx, cand.x, rx);
                    round_split(ky, fy, cand.y, ry);
                    const int tx = x + cand.x, ty = y + cand.y;
                    ok = tx >= 0 && tx < W && ty >= 0 && ty < H;
                }
            }
        }
        // candidates that the bound rules out against the best so far
        const uint4* iv = reinterpret_cast<const uint4*>(pv.box[1 - dir]) + i;
        auto excluded = [&](bool in, int2 c) {
            return PLANES && bounded && in && interval_lb(__ldg(iv + c.y * W + c.x), ar, ag, ab) >= box_threshold(bc);
        };
        unsigned todo = fresh_lanes(ok && !excluded(ok, cand), cand, best, lane);
#pragma unroll 1
        for (int list_b = 0; list_b < 2; ++list_b) {
            if (list_b) {
                // list B: random search around v0, the best offset after list A
                const int2 v0 = best;
                // random words for the search radii, two radii per Philox call, one call per lane
                uint4 rw = make_uint4(0, 0, 0, 0);
                if (lane < (nrad + 1) / 2)
                    rw = philox((uint32_t)i, ((uint32_t)it << 8) | (uint32_t)lane, tag, pv.pair_id, k0, k1);
                const int src_lane = lane >> 1;
                uint32_t wx = __shfl_sync(FULL, rw.x, src_lane), wy = __shfl_sync(FULL, rw.y, src_lane);
                const uint32_t wz = __shfl_sync(FULL, rw.z, src_lane), ww = __shfl_sync(FULL, rw.w, src_lane);
                if (lane & 1) {
                    wx = wz;
                    wy = ww;
                }
                const int Rk = R0 >> lane;
                const int ox = (int)bounded_u32(wx, (uint32_t)(2 * Rk + 1)) - Rk;
                const int oy = (int)bounded_u32(wy, (uint32_t)(2 * Rk + 1)) - Rk;
                const int tx = min(max(x + v0.x + ox, 0), W - 1), ty = min(max(y + v0.y + oy, 0), H - 1);
                cand = make_int2(tx - x, ty - y);
                ok = lane < nrad;
                todo = fresh_lanes(ok && !excluded(ok, cand), cand, v0, lane);
            }
            while (todo) {
                const int l = __ffs(todo) - 1;
                todo &= todo - 1;
                const int2 c = make_int2(__shfl_sync(FULL, cand.x, l), __shfl_sync(FULL, cand.y, l));
                if constexpr (CENSUS) {
                    int sum;  // exact integer costs: the incumbent's sum is an integer held in a float
                    if (census_sum<R>(lp, reinterpret_cast<const uint32_t*>(tgt), W, H, c, (int)bc, sum, lane) &&
                        sum < (int)bc) {
                        bc = (float)sum;
                        best = c;
                    }
                } else {
                    float sum;
                    int nch;
                    const bool done = tap_sum<R, ST>(lp, tgt, W, H, c, ithr, sum, nch, lane);
                    ntap += min(32 * nch, Patch<R>::T);
                    if (done && sum < bc) {
                        bc = sum;
                        best = c;
                        ithr = abandon_threshold(bc);
                    }
                }
                ++nev;
            }
        }
        if (lane == 0) {
            const bool m = best.x != before.x || best.y != before.y;
            moved[i] = m;
            if (m) {
                nnf[i] = best;
                pv.cost[dir][i] = bc;
            }
            if (pv.evals) {
                atomicAdd(&pv.evals[PLANES ? GPM_COUNT_SWEEP_PLANE : GPM_COUNT_SWEEP0], (unsigned long long)nev);
                atomicAdd(&pv.evals[PLANES ? GPM_COUNT_SWEEP_PLANE_TAPS : GPM_COUNT_SWEEP0_TAPS],
                          (unsigned long long)(CENSUS ? nev * Patch<R>::T : ntap));
            }
        }
    }
}

// ---------------------------------------------------------------- level-0 sweep, two layouts
// Tiles of the level-0 sweep: 16 pixels of one colour by `rows` rows (32 x rows image pixels), the block's four
// warps owning 4 rows pixels each, one pixel per lane: rows = 8 fills the lanes and shares the staging best; small
// frames take 4, 2 or 1, so that the launch still covers the chip (sweep0_rows).  The staged source region is the
// tile grown by r, in rows of TW texels (TW congruent to 2r + 1 modulo 8, so that eight consecutive taps of a patch
// row fall on eight distinct 16-byte bank groups).
template <int R>
struct Tile0L {
    static constexpr int TXC = 16, TYMAX = 8, TX = 2 * TXC, WARPS = 4;
    static constexpr int TW0 = TX + 2 * R;
    static constexpr int TW = TW0 + ((2 * R + 1 - TW0) % 8 + 8) % 8;
    static constexpr int TH = TYMAX + 2 * R;
};
// Search radii R0 >> k >= 1 for frames below 2^15 pixels a side: at most 15.
constexpr int kMaxRadii = 16;

int sweep0_tiles(int W, int H, int rows) {
    const int hw = (W + 1) >> 1;
    return ((hw + Tile0L<1>::TXC - 1) / Tile0L<1>::TXC) * ((H + rows - 1) / rows);
}
// The most rows a tile may have with at least four blocks per SM in the launch (a block's warps walk their pixels
// one after another, so a launch of fewer blocks lasts as long as one of that many): 128x96 takes 1 row, 253x187
// four, from 512x384 on 8.
int sweep0_rows(int W, int H, int pairs, int nsm) {
    int rows = Tile0L<1>::TYMAX;
    while (rows > 1 && (int64_t)sweep0_tiles(W, H, rows) * 2 * pairs < 4 * nsm) rows >>= 1;
    return rows;
}

// Appends candidate c to a pixel's list (column `lane` of list[k][32]) unless an earlier entry holds it.
__device__ __forceinline__ void list_push(uint32_t (*list)[32], int& n, int2 c, int lane) {
    const uint32_t key = pack_off(c);
    bool dup = false;
    for (int k = 0; k < n; ++k) dup |= list[k][lane] == key;
    if (!dup) list[n++][lane] = key;
}

// One pixel's patch, one tap per lane and chunk: the source texels, and the taps' byte offsets into the padded target
// copy at offset 0 (frames hold at most 2^26 texels of 16 bytes, so 32 bits address the copy).
template <int R>
struct SquarePatch {
    float4 a[Patch<R>::NT];
    unsigned at[Patch<R>::NT];
};
// What a lane's taps add to a pixel whose patch stays inside the frame: its texels in the staged tile and in the
// padded copy (constants of the lane, so that such a pixel's patch takes two additions a tap; clamping every tap's
// coordinates took eleven instructions).
template <int R>
struct TapOffsets {
    int tile[Patch<R>::NT];
    unsigned at[Patch<R>::NT];
};
template <int R, int ST, int TW>
__device__ __forceinline__ void load_square(SquarePatch<R>& sp, const TapOffsets<R>& to, const void* tile, int x0, int y0,
                                            int W, int H, int px, int py, bool inside, int lane, int Wp) {
    constexpr unsigned B = sizeof(typename TexelOf<ST>::type);
    if (inside) {  // warp-uniform
        const int tp = (py - y0) * TW + (px - x0);
        const unsigned ap = (unsigned)((py + kPad) * Wp + px + kPad) * B;
#pragma unroll
        for (int j = 0; j < Patch<R>::NT; ++j) {
            sp.a[j] = ldpix_shared<ST>(tile, tp + to.tile[j]);
            sp.at[j] = ap + to.at[j];
        }
        return;
    }
#pragma unroll
    for (int j = 0; j < Patch<R>::NT; ++j) {
        const int t = lane + 32 * j;
        const int tt = t < Patch<R>::T ? t : 0;
        const int dy = tt / Patch<R>::D - R, dx = tt % Patch<R>::D - R;
        const int tx = min(max(px + dx, 0), W - 1), ty = min(max(py + dy, 0), H - 1);
        sp.at[j] = (unsigned)((ty + kPad) * Wp + tx + kPad) * B;
        sp.a[j] = ldpix_shared<ST>(tile, (ty - y0 + R) * TW + tx - x0 + R);
    }
}

// Maximum number of one pixel's candidates whose costs are summed together.
constexpr int kSweep0Group = 3;

// N listed candidates of one square patch, from the k-th: their raw tap sums, all in full, each lane accumulating its
// taps in the order of tap_sum_in and the totals warp_sum_q23's times 2^23 (an exact scaling, so they compare
// alike; best costs are held scaled too); the N candidates' gathers of a chunk are in flight together.  Then the
// strict-less updates in list order.
template <int R, int ST, int N>
__device__ __forceinline__ void eval_group(const SquarePatch<R>& sp, const void* tgtp, int Wp,
                                           const uint32_t (*list)[32], int p, int k, int lane, int2& best, float& bc) {
    constexpr unsigned B = sizeof(typename TexelOf<ST>::type);
    int2 c[N];
    unsigned off[N];
    float s[N];
#pragma unroll
    for (int q = 0; q < N; ++q) {
        c[q] = unpack_off(list[k + q][p]);
        off[q] = (unsigned)(c[q].y * Wp + c[q].x) * B;
        s[q] = 0.f;
    }
#pragma unroll
    for (int j = 0; j < Patch<R>::NT; ++j) {
        if (lane + 32 * j < Patch<R>::T) {
            float4 v[N];
#pragma unroll
            for (int q = 0; q < N; ++q) v[q] = ldpix<ST>(static_cast<const char*>(tgtp) + (sp.at[j] + off[q]), 0);
#pragma unroll
            for (int q = 0; q < N; ++q) s[q] += absdiff3(sp.a[j], make_float3(v[q].x, v[q].y, v[q].z));
        }
    }
#pragma unroll
    for (int q = 0; q < N; ++q) {
        const float sum = (float)__reduce_add_sync(FULL, __float2uint_rn(s[q] * 8388608.f));
        if (sum < bc) {
            bc = sum;
            best = c[q];
        }
    }
}

// The warp (one tap per lane) evaluates the n listed candidates of one pixel in list order, up to kSweep0Group
// at a time, with the strict-less rule (every cost summed in full, then the updates in list order): best / bc
// are warp-uniform on entry and on return.
template <int R, int ST>
__device__ __forceinline__ void eval_listed(const SquarePatch<R>& sp, const void* tgtp, int Wp,
                                            const uint32_t (*list)[32], int p, int n, int lane, int2& best, float& bc) {
    for (int k = 0; k < n;) {
        const int g = min(n - k, kSweep0Group);
        if (g == 3)
            eval_group<R, ST, 3>(sp, tgtp, Wp, list, p, k, lane, best, bc);
        else if (g == 2)
            eval_group<R, ST, 2>(sp, tgtp, Wp, list, p, k, lane, best, bc);
        else
            eval_group<R, ST, 1>(sp, tgtp, Wp, list, p, k, lane, best, bc);
        k += g;
    }
}

// Level-0 sweep with square colour patches (Sec. 3.1), one colour of the red-black schedule per launch.  Each
// pixel's candidates come in two lists: (A) propagation, the offsets of its left, right, upper and lower
// neighbours; (B) random search around the best offset after A, radius R0 >> k for k = 0, 1, ... (Philox words,
// two radii per call).  A candidate replaces the best only if its raw tap sum is strictly lower, in list order;
// candidates that repeat the best or an earlier entry, or that the patch-sum bound rules out, cannot win and are
// not listed, nor are, after the first iteration, the offsets of neighbours that did not move (see k_pm_sweep).
// The per-pixel scalar work runs with one pixel per lane: the neighbours' offsets, the Philox words
// and the search candidates, the bound and the removal of repeats, into a list per pixel in shared memory.  The
// patch costs run with one tap per lane, the warp walking its pixels' lists in turn; list B is built once
// list A is evaluated for all of them.
template <int R, int ST>
__global__ void __launch_bounds__(128, 6) k_pm_sweep0(const __grid_constant__ Batch bt, int it, int phase, int rows,
                                                      uint32_t k0, uint32_t k1) {
    begin_kernel();
    using TL = Tile0L<R>;
    using Tex = typename TexelOf<ST>::type;
    __shared__ Tex stile[TL::TH * TL::TW];
    __shared__ uint32_t slist[TL::WARPS][kMaxRadii][32];
    const PairView& pv = bt.view(blockIdx.z);
    const int dir = blockIdx.y;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int W = pv.W, H = pv.H, Wp = pv.Wp;
    const int hw = (W + 1) >> 1;
    const int ntx = (hw + TL::TXC - 1) / TL::TXC, nty = (H + rows - 1) / rows;
    if ((int)blockIdx.x >= ntx * nty) return;  // block-uniform: the grid covers the largest pair of the batch
    const int tyi = blockIdx.x / ntx, txi = blockIdx.x - tyi * ntx;
    const int x0 = TL::TX * txi, y0 = rows * tyi;
    {
        // the tile's source region, from the padded copy (entries past its edge are clamped and unused)
        const Tex* sp = reinterpret_cast<const Tex*>(pv.imgp[dir]);
        const int Hp = H + 2 * kPad;
        for (int e = threadIdx.x; e < (rows + 2 * R) * TL::TW; e += blockDim.x) {
            const int ly = e / TL::TW, lx = e - ly * TL::TW;
            const int gx = min(x0 - R + lx + kPad, Wp - 1), gy = min(y0 - R + ly + kPad, Hp - 1);
            stile[e] = sp[gy * Wp + gx];
        }
    }
    TapOffsets<R> to;
#pragma unroll
    for (int j = 0; j < Patch<R>::NT; ++j) {
        const int t = lane + 32 * j, tt = t < Patch<R>::T ? t : 0;
        const int dy = tt / Patch<R>::D - R, dx = tt % Patch<R>::D - R;
        to.tile[j] = (dy + R) * TL::TW + dx + R;
        to.at[j] = (unsigned)(dy * Wp + dx) * (unsigned)sizeof(Tex);
    }
    __syncthreads();
    const void* tgtp = pv.imgp[1 - dir];
    uint32_t(*list)[32] = slist[wid];
    int2* __restrict__ nnf = pv.nnf[dir];
    uint8_t* __restrict__ moved = pv.resid[dir];
    const float4* __restrict__ boxt = pv.box[1 - dir];
    // the lane's pixel: the wid * npix + lane-th of the tile, 16 a row
    const int npix = 4 * rows;
    const int yq = y0 + ((wid * npix + lane) >> 4);
    const int xq = 2 * (TL::TXC * txi + ((wid * npix + lane) & 15)) + ((yq + phase) & 1);
    const bool mine = lane < npix && yq < H && xq < W;
    const int iq = mine ? yq * W + xq : 0;
    int2 best = make_int2(0, 0);
    float bc = 0.f;  // times 2^23
    if (mine) {
        best = nnf[iq];
        bc = pv.cost[dir][iq] * 8388608.f;
    }
    const float before = bc;
    // interior pixels: the patch-sum bound applies
    const bool prune = mine && xq >= R && yq >= R && xq < W - R && yq < H - R;
    const unsigned inside = __ballot_sync(FULL, prune);
    const float4 b1 = prune ? pv.box[dir][iq] : make_float4(0.f, 0.f, 0.f, 0.f);
    const uint2* __restrict__ region1 = reinterpret_cast<const uint2*>(pv.m2o_key[dir]) + iq;
    const uint2* __restrict__ region2 = reinterpret_cast<const uint2*>(pv.m2o_key[1 - dir]) + iq;
    unsigned npr = 0, nev = 0;
    // list A, one pixel per lane: the four neighbours' offsets whose target is in the frame, neither the
    // incumbent nor a repeat, and not excluded by the bound
    int n = 0;
    if (mine) {
        const float thr = box_threshold(bc * 1.1920928955078125e-07f);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int nx = xq + (k == 0 ? -1 : (k == 1 ? 1 : 0));
            const int ny = yq + (k == 2 ? -1 : (k == 3 ? 1 : 0));
            if (nx < 0 || nx >= W || ny < 0 || ny >= H || (it > 0 && !moved[ny * W + nx])) continue;
            const int2 c = nnf[ny * W + nx];
            const int tx = xq + c.x, ty = yq + c.y;
            if (tx < 0 || tx >= W || ty < 0 || ty >= H || (c.x == best.x && c.y == best.y)) continue;
            if (prune && box_lb(b1, boxt[iq + c.y * W + c.x]) >= thr) {
                ++npr;
                continue;
            }
            list_push(list, n, c, lane);
        }
    }
    for (int part = 0;; ++part) {
        if constexpr (kRegionBound<R, ST>) {
            // list B by the regions' bound, one pixel per lane (targets whose patch stays in the frame, as the regions must)
            if (part && prune && n > 0) {
                RegionSums regions;
                regions.load(region1, W);
                const float thr = box_threshold(bc * 1.1920928955078125e-07f);
                int kept = 0;
                for (int k = 0; k < n; ++k) {
                    const uint32_t key = list[k][lane];
                    const int2 c = unpack_off(key);
                    if ((unsigned)(xq + c.x - R) < (unsigned)(W - 2 * R) && (unsigned)(yq + c.y - R) < (unsigned)(H - 2 * R) &&
                        regions.excludes(region2 + c.y * W + c.x, W, thr))
                        ++npr;
                    else
                        list[kept++][lane] = key;
                }
                n = kept;
            }
        }
        __syncwarp();
        // the list's costs, one tap per lane, pixel by pixel
        nev += n;
        for (unsigned todo = __ballot_sync(FULL, n > 0); todo; todo &= todo - 1) {
            const int p = __ffs(todo) - 1, np_ = __shfl_sync(FULL, n, p);
            const int yp = y0 + ((wid * npix + p) >> 4);
            const int xp = 2 * (TL::TXC * txi + ((wid * npix + p) & 15)) + ((yp + phase) & 1);
            SquarePatch<R> sp;
            load_square<R, ST, TL::TW>(sp, to, stile, x0, y0, W, H, xp, yp, (inside >> p) & 1u, lane, Wp);
            int2 b = make_int2(__shfl_sync(FULL, best.x, p), __shfl_sync(FULL, best.y, p));
            float c = __shfl_sync(FULL, bc, p);
            eval_listed<R, ST>(sp, tgtp, Wp, list, p, np_, lane, b, c);
            if (lane == p) {
                best = b;
                bc = c;
            }
        }
        if (part) break;
        __syncwarp();
        // list B, one pixel per lane: random search around v0, the best offset after list A (Philox words two radii
        // per call, as in k_pm_sweep)
        n = 0;
        if (mine) {
            const int2 v0 = best;
            const int R0 = max(W, H);
            int nrad = 0;
            while ((R0 >> nrad) >= 1) ++nrad;
            const uint32_t tag = stream_tag(RNG_SEARCH, dir, 0, 0);
            const float thr = box_threshold(bc * 1.1920928955078125e-07f);
            for (int call = 0; 2 * call < nrad; ++call) {
                const uint4 rw = philox((uint32_t)iq, ((uint32_t)it << 8) | (uint32_t)call, tag, pv.pair_id, k0, k1);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int k = 2 * call + h;
                    if (k >= nrad) break;
                    const uint32_t wx = h ? rw.z : rw.x, wy = h ? rw.w : rw.y;
                    const int Rk = R0 >> k;
                    const int ox = (int)bounded_u32(wx, (uint32_t)(2 * Rk + 1)) - Rk;
                    const int oy = (int)bounded_u32(wy, (uint32_t)(2 * Rk + 1)) - Rk;
                    const int tx = min(max(xq + v0.x + ox, 0), W - 1), ty = min(max(yq + v0.y + oy, 0), H - 1);
                    const int2 c = make_int2(tx - xq, ty - yq);
                    if (c.x == v0.x && c.y == v0.y) continue;
                    if (prune && box_lb(b1, boxt[iq + c.y * W + c.x]) >= thr) {
                        ++npr;
                        continue;
                    }
                    list_push(list, n, c, lane);
                }
            }
        }
    }
    if (mine) {
        // a candidate is only taken at a lower cost; the offsets packed would not tell, as an imported one may be any integer
        const bool m = bc < before;
        moved[iq] = m;
        if (m) {
            nnf[iq] = best;
            pv.cost[dir][iq] = bc * 1.1920928955078125e-07f;
        }
    }
    if (pv.evals) {
        const unsigned npw = __reduce_add_sync(FULL, npr), nevw = __reduce_add_sync(FULL, nev);
        if (lane == 0) {
            atomicAdd(&pv.evals[GPM_COUNT_SWEEP0], (unsigned long long)nevw);
            atomicAdd(&pv.evals[GPM_COUNT_SWEEP0_TAPS], (unsigned long long)nevw * Patch<R>::T);
            if (npw) atomicAdd(&pv.evals[GPM_COUNT_SWEEP0_PRUNED], (unsigned long long)npw);
        }
    }
}

// Unfrozen pixels of each colour, for the restricted sweeps (order is free:
// pixels of one colour are independent within a half-iteration).
__global__ void k_lists_zero(const __grid_constant__ Batch bt) {
    begin_kernel();
    if (threadIdx.x < 4) bt.view(blockIdx.z).list_count[threadIdx.x] = 0;
}
__global__ void k_build_lists(const __grid_constant__ Batch bt) {
    begin_kernel();
    const PairView& pv = bt.view(blockIdx.z);
    const int dir = blockIdx.y;
    const int n = pv.n, W = pv.W;
    const int lane = threadIdx.x & 31;
    for (int base = blockIdx.x * blockDim.x; base < n; base += gridDim.x * blockDim.x) {
        const int i = base + threadIdx.x;
        bool ok = false;
        int col = 0;
        if (i < n) {
            ok = !pv.frozen[dir][i];
            if (!ok) pv.resid[dir][i] = 0;  // a frozen pixel never moves in the sweeps
            const int y = i / W, x = i - y * W;
            col = (x + y) & 1;
        }
        for (int c = 0; c < 2; ++c) {
            const unsigned mask = __ballot_sync(FULL, ok && col == c);
            if (!mask) continue;
            int off = 0;
            if (lane == 0) off = atomicAdd(&pv.list_count[dir * 2 + c], __popc(mask));
            off = __shfl_sync(FULL, off, 0);
            if (ok && col == c) pv.list[dir][c * n + off + __popc(mask & ((1u << lane) - 1))] = i;
        }
    }
}

// ---------------------------------------------------------------- launchers
template <int R, int ST>
static void launch_pm_r(const PmLaunch& L, cudaStream_t st) {
    const dim3 grid(L.grid_blocks, 2, L.np), block(256);
    switch (L.op) {
        case PmLaunch::INIT:  // census codes do not depend on the texel storage: one instance serves all
            if (L.census)
                launch_kernel(k_pm_init<R, 0, true>, grid, block, 0, st, L.bt, L.k0, L.k1);
            else
                launch_kernel(k_pm_init<R, ST, false>, grid, block, 0, st, L.bt, L.k0, L.k1);
            break;
        case PmLaunch::RECOST:
            launch_kernel(k_pm_recost<R, ST>, grid, block, 0, st, L.bt, L.level);
            break;
        case PmLaunch::SWEEP:
            if (L.level == 0 && L.census)
                launch_kernel(k_pm_sweep<R, 0, false, true>, grid, block, 0, st, L.bt, 0, L.it, L.phase, L.k0, L.k1);
            else if (L.level == 0)
                launch_kernel(k_pm_sweep0<R, ST>, dim3(L.tiles0, 2, L.np), dim3(32 * Tile0L<R>::WARPS), 0, st, L.bt, L.it, L.phase, L.rows0,
                                                                                                  L.k0, L.k1);
            else
                launch_kernel(k_pm_sweep<R, ST, true, false>, grid, block, 0, st, L.bt, L.level, L.it, L.phase, L.k0, L.k1);
            break;
    }
}

template <int ST>
static void launch_pm_st(const PmLaunch& L, cudaStream_t st) {
    switch (L.radius) {
        case 1: launch_pm_r<1, ST>(L, st); break;
        case 2: launch_pm_r<2, ST>(L, st); break;
        case 3: launch_pm_r<3, ST>(L, st); break;
        case 4: launch_pm_r<4, ST>(L, st); break;
        default: break;
    }
}

void launch_pm(const PmLaunch& L, cudaStream_t st) {
    switch (L.storage) {
        case 0: launch_pm_st<0>(L, st); break;
        case 1: launch_pm_st<1>(L, st); break;
        case 2: launch_pm_st<2>(L, st); break;
    }
}

// Greys of frame 1 as given, for the edge-aware fill (the jobs that ask for them).
__global__ void k_grey_q(const __grid_constant__ IngestJobs J) {
    begin_kernel();
    const IngestJob& j = J.j[blockIdx.z];
    if (!j.gq) return;
    const int W = j.W, n = j.W * j.H;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int y = i / W, x = i - y * W;
        const int64_t e = (int64_t)y * j.stride + 3 * x;
        j.gq[i] = (int)floor(1024.0 * (((double)in_elem(j.f1, j.dtype, e) + (double)in_elem(j.f1, j.dtype, e + 1)) +
                                       (double)in_elem(j.f1, j.dtype, e + 2)));
    }
}

// The ingest of nj pairs, each kernel one launch over the jobs (blockIdx.z).  Per job the grid and the order
// of every reduction are those of a single pair's ingest, so each result is the same alone and in a batch.
void launch_ingest_jobs(const IngestJobs& J, int nj, int max_n, int max_h, int gain_enable, int storage,
                        cudaStream_t st) {
    (void)max_n;
    (void)max_h;
    const int blocks = 152 * 4;
    bool eq = false, census = false, grey = false;
    for (int k = 0; k < nj; ++k) {
        eq |= J.j[k].hist != nullptr;
        census |= J.j[k].k1 != nullptr;
        grey |= J.j[k].gq != nullptr;
    }
    if (census) {
        launch_kernel(k_grey_keys, dim3(blocks, 2, nj), 256, 0, st, J);
        launch_kernel(k_census, dim3(blocks, 2, nj), 256, 0, st, J);
    }
    if (grey) launch_kernel(k_grey_q, dim3(blocks, 1, nj), 256, 0, st, J);
    if (eq) {
        launch_kernel(k_vhist_zero, dim3(1, 1, nj), 256, 0, st, J);
        launch_kernel(k_vhist, dim3(152, 2, nj), 512, 0, st, J);
    }
    const dim3 sums(kIngestPartialBlocks, 1, nj), pack(blocks, 1, nj);
    switch (storage) {
        case 0:
            launch_kernel(k_frame_sums<0>, sums, 1024, 0, st, J);
            launch_kernel(k_pack<0>, pack, 256, 0, st, J, gain_enable);
            break;
        case 1:
            launch_kernel(k_frame_sums<1>, sums, 1024, 0, st, J);
            launch_kernel(k_pack<1>, pack, 256, 0, st, J, gain_enable);
            break;
        case 2:
            launch_kernel(k_frame_sums<2>, sums, 1024, 0, st, J);
            launch_kernel(k_pack<2>, pack, 256, 0, st, J, gain_enable);
            break;
    }
}

void launch_ingest(const float* f1, const float* f2, int W, int H, int64_t stride, int gain_enable, int storage,
                   double* partial, void* o1, void* o2, int* eq_hist, float* eq_lut, cudaStream_t st) {
    IngestJobs J{};
    J.j[0] = IngestJob{f1, f2, GPM_F32, W, H, stride, partial, o1, o2, eq_lut ? eq_hist : nullptr, eq_lut,
                       nullptr, nullptr, nullptr, nullptr, nullptr};
    launch_ingest_jobs(J, 1, W * H, H, gain_enable, storage, st);
}

// Padded copy of each ingested frame: texel (x, y) of the copy, for x in
// [-kPad, W + kPad) and y in [-kPad, H + kPad), is the frame's texel at the
// clamped coordinates (T: one texel, 16 or 8 bytes).
template <typename T>
__global__ void k_pad_frames(const __grid_constant__ Batch bt) {
    begin_kernel();
    const PairView& pv = bt.view(blockIdx.z);
    const int dir = blockIdx.y;
    const T* src = reinterpret_cast<const T*>(pv.img[dir]);
    T* dst = reinterpret_cast<T*>(const_cast<void*>(pv.imgp[dir]));
    const int W = pv.W, H = pv.H, Wp = pv.Wp, np = Wp * (H + 2 * kPad);
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < np; i += gridDim.x * blockDim.x) {
        const int yp = i / Wp, xp = i - yp * Wp;
        const int x = min(max(xp - kPad, 0), W - 1), y = min(max(yp - kPad, 0), H - 1);
        dst[i] = src[y * W + x];
    }
}
// Patch sums of each ingested frame: box[q] = the RGB sums over the (2r+1)^2 taps of q's patch, taps clamped
// into the frame (read from the padded copy).  For a pixel p whose patch stays inside the frame and an offset c
// whose target pixel is in the frame, the level-0 cost's taps are exactly these patches' texels, so
// sum_ch |box1(p)_ch - box2(p + c)_ch| bounds the raw cost from below.  Separable, in FP32: a block stages a
// 32 x 8 tile and its r-halo, sums each row's 2r + 1 texels, then each column's 2r + 1 row sums, in a fixed order
// (at most 16 FP32 roundings per sum, which the sweep's test allows for).
template <int R, int ST>
__global__ void __launch_bounds__(256) k_box_sums(const __grid_constant__ Batch bt) {
    begin_kernel();
    constexpr int BX = 32, BY = 8, TWB = BX + 2 * R, THB = BY + 2 * R;
    __shared__ float3 tex[THB][TWB];
    __shared__ float3 hs[THB][BX];
    const PairView& pv = bt.view(blockIdx.z >> 1);  // blockIdx.z = 2 pair + direction
    const int dir = blockIdx.z & 1;
    const int W = pv.W, H = pv.H, Wp = pv.Wp, Hp = H + 2 * kPad;
    const int x0 = blockIdx.x * BX, y0 = blockIdx.y * BY;
    if (x0 >= W || y0 >= H) return;  // past this pair's frame (block-uniform)
    for (int e = threadIdx.x; e < THB * TWB; e += blockDim.x) {
        const int ly = e / TWB, lx = e - ly * TWB;
        const int gx = min(x0 - R + lx + kPad, Wp - 1), gy = min(y0 - R + ly + kPad, Hp - 1);
        const float4 v = ldpix<ST>(pv.imgp[dir], gy * Wp + gx);
        tex[ly][lx] = make_float3(v.x, v.y, v.z);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < THB * BX; e += blockDim.x) {
        const int ly = e / BX, lx = e - ly * BX;
        float3 a = tex[ly][lx];
#pragma unroll
        for (int d = 1; d <= 2 * R; ++d) {
            const float3 v = tex[ly][lx + d];
            a.x += v.x;
            a.y += v.y;
            a.z += v.z;
        }
        hs[ly][lx] = a;
    }
    __syncthreads();
    const int lx = threadIdx.x & (BX - 1), ly = threadIdx.x / BX;
    const int x = x0 + lx, y = y0 + ly;
    if (x < W && y < H) {
        float3 a = hs[ly][lx];
#pragma unroll
        for (int d = 1; d <= 2 * R; ++d) {
            const float3 v = hs[ly + d][lx];
            a.x += v.x;
            a.y += v.y;
            a.z += v.z;
        }
        pv.box[dir][y * W + x] = make_float4(a.x, a.y, a.z, 0.f);
        if constexpr (kRegionBound<R, ST>) {  // the 3 x 3 sums
            float3 t = make_float3(0.f, 0.f, 0.f);
            bool ok = true;
#pragma unroll
            for (int d = 0; d < 9; ++d) {
                const float3 v = tex[ly + R - 1 + d / 3][lx + R - 1 + d % 3];
                ok = ok && in_domain(v.x, v.y, v.z);
                t = make_float3(t.x + v.x, t.y + v.y, t.z + v.z);
            }
            const unsigned r = __float2uint_rn(t.x * 2048.f), g = __float2uint_rn(t.y * 2048.f), b = __float2uint_rn(t.z * 2048.f);
            reinterpret_cast<uint2*>(pv.m2o_key[dir])[y * W + x] = ok ? make_uint2(r | g << 16, b) : make_uint2(0u, 0x80000000u);
        }
    }
}
template <int ST>
static void launch_box_st(const Batch& bt, dim3 grid, int radius, cudaStream_t st) {
    switch (radius) {
        case 1: launch_kernel(k_box_sums<1, ST>, grid, 256, 0, st, bt); break;
        case 2: launch_kernel(k_box_sums<2, ST>, grid, 256, 0, st, bt); break;
        case 3: launch_kernel(k_box_sums<3, ST>, grid, 256, 0, st, bt); break;
        case 4: launch_kernel(k_box_sums<4, ST>, grid, 256, 0, st, bt); break;
    }
}
void launch_box_sums(const Batch& bt, int np, int max_w, int max_h, int radius, int storage, cudaStream_t st) {
    const dim3 grid((max_w + 31) / 32, (max_h + 7) / 8, 2 * np);
    switch (storage) {
        case 0: launch_box_st<0>(bt, grid, radius, st); break;
        case 1: launch_box_st<1>(bt, grid, radius, st); break;
        case 2: launch_box_st<2>(bt, grid, radius, st); break;
    }
}

// The sums over each pixel's patch (taps clamped into the frame) of the channels' minima and maxima over 3 x 3 texels
// (clamped too), into pv.box (see interval_lb).  A sample the sweeps clamp into the frame touches texels of the
// clamped 3 x 3 around its unclamped place, so the bound holds at borders.  A texel out of the bound's domain opens
// its intervals.  Separable, a 32 x 8 tile a block: 3 x 3 extremes of the tile grown by r, row sums, column sums.
// 1024x436, both frames: 0.04 ms, for 60 % of the plane sweeps' evaluations.
template <int R, int ST>
__global__ void __launch_bounds__(256) k_interval_sums(const __grid_constant__ Batch bt) {
    begin_kernel();
    constexpr int BX = 32, BY = 8, MW = BX + 2 * R, MH = BY + 2 * R, TWI = MW + 2, THI = MH + 2;
    __shared__ float3 tex[THI][TWI];
    __shared__ float3 mn[MH][MW], mx[MH][MW];
    const PairView& pv = bt.view(blockIdx.z >> 1);  // blockIdx.z = 2 pair + direction
    const int dir = blockIdx.z & 1;
    const int W = pv.W, H = pv.H;
    const int x0 = blockIdx.x * BX, y0 = blockIdx.y * BY;
    if (x0 >= W || y0 >= H) return;  // past this pair's frame (block-uniform)
    for (int e = threadIdx.x; e < THI * TWI; e += blockDim.x) {
        const int ly = e / TWI, lx = e - ly * TWI;
        const int gx = min(max(x0 - R - 1 + lx, 0), W - 1), gy = min(max(y0 - R - 1 + ly, 0), H - 1);
        const float4 v = ldpix<ST>(pv.img[dir], gy * W + gx);
        tex[ly][lx] = make_float3(v.x, v.y, v.z);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < MH * MW; e += blockDim.x) {
        const int ly = e / MW, lx = e - ly * MW;
        float3 a = tex[ly][lx], b = a;
        bool ok = true;
#pragma unroll
        for (int d = 0; d < 9; ++d) {
            const float3 v = tex[ly + d / 3][lx + d % 3];
            ok = ok && in_domain(v.x, v.y, v.z);
            a = make_float3(fminf(a.x, v.x), fminf(a.y, v.y), fminf(a.z, v.z));
            b = make_float3(fmaxf(b.x, v.x), fmaxf(b.y, v.y), fmaxf(b.z, v.z));
        }
        mn[ly][lx] = ok ? a : make_float3(-INFINITY, -INFINITY, -INFINITY);
        mx[ly][lx] = ok ? b : make_float3(INFINITY, INFINITY, INFINITY);
    }
    __syncthreads();
    // row sums, through registers back into the same arrays
    float3 rn[(MH * BX + 255) / 256], rx[(MH * BX + 255) / 256];
#pragma unroll
    for (int k = 0; k < (MH * BX + 255) / 256; ++k) {
        const int e = threadIdx.x + 256 * k, ly = e / BX, lx = e - ly * BX;
        if (e >= MH * BX) break;
        float3 a = mn[ly][lx], b = mx[ly][lx];
#pragma unroll
        for (int d = 1; d <= 2 * R; ++d) {
            const float3 v = mn[ly][lx + d], w = mx[ly][lx + d];
            a = make_float3(a.x + v.x, a.y + v.y, a.z + v.z);
            b = make_float3(b.x + w.x, b.y + w.y, b.z + w.z);
        }
        rn[k] = a;
        rx[k] = b;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < (MH * BX + 255) / 256; ++k) {
        const int e = threadIdx.x + 256 * k, ly = e / BX, lx = e - ly * BX;
        if (e >= MH * BX) break;
        mn[ly][lx] = rn[k];
        mx[ly][lx] = rx[k];
    }
    __syncthreads();
    const int lx = threadIdx.x & (BX - 1), ly = threadIdx.x / BX;
    const int x = x0 + lx, y = y0 + ly;
    if (x < W && y < H) {
        float3 a = mn[ly][lx], b = mx[ly][lx];
#pragma unroll
        for (int d = 1; d <= 2 * R; ++d) {
            const float3 v = mn[ly + d][lx], w = mx[ly + d][lx];
            a = make_float3(a.x + v.x, a.y + v.y, a.z + v.z);
            b = make_float3(b.x + w.x, b.y + w.y, b.z + w.z);
        }
        // widened by more than the 16 roundings of a sum, then rounded outwards
        auto lo = [](float v) { return __float2half_rd(v - (2e-6f * fabsf(v) + 1e-6f)); };
        auto hi = [](float v) { return __float2half_ru(v + (2e-6f * fabsf(v) + 1e-6f)); };
        const __half2 p = __halves2half2(lo(a.x), lo(a.y)), q = __halves2half2(lo(a.z), hi(b.x)),
                      r = __halves2half2(hi(b.y), hi(b.z));
        uint4 o;
        o.x = *reinterpret_cast<const unsigned*>(&p);
        o.y = *reinterpret_cast<const unsigned*>(&q);
        o.z = *reinterpret_cast<const unsigned*>(&r);
        o.w = 0u;
        reinterpret_cast<uint4*>(pv.box[dir])[y * W + x] = o;
    }
}
template <int ST>
static void launch_interval_st(const Batch& bt, dim3 grid, int radius, cudaStream_t st) {
    switch (radius) {
        case 1: launch_kernel(k_interval_sums<1, ST>, grid, 256, 0, st, bt); break;
        case 2: launch_kernel(k_interval_sums<2, ST>, grid, 256, 0, st, bt); break;
        case 3: launch_kernel(k_interval_sums<3, ST>, grid, 256, 0, st, bt); break;
        case 4: launch_kernel(k_interval_sums<4, ST>, grid, 256, 0, st, bt); break;
    }
}
void launch_interval_sums(const Batch& bt, int np, int max_w, int max_h, int radius, int storage, cudaStream_t st) {
    const dim3 grid((max_w + 31) / 32, (max_h + 7) / 8, 2 * np);
    switch (storage) {
        case 0: launch_interval_st<0>(bt, grid, radius, st); break;
        case 1: launch_interval_st<1>(bt, grid, radius, st); break;
        case 2: launch_interval_st<2>(bt, grid, radius, st); break;
    }
}

void launch_pad_frames(const Batch& bt, int np, int storage, int grid_blocks, cudaStream_t st) {
    if (storage == 0)
        launch_kernel(k_pad_frames<uint4>, dim3(grid_blocks, 2, np), 256, 0, st, bt);
    else
        launch_kernel(k_pad_frames<uint2>, dim3(grid_blocks, 2, np), 256, 0, st, bt);
}

void launch_build_lists(const Batch& bt, int np, bool cleared, int grid_blocks, cudaStream_t st) {
    if (!cleared) launch_kernel(k_lists_zero, dim3(1, 1, np), 32, 0, st, bt);
    launch_kernel(k_build_lists, dim3(grid_blocks, 2, np), 256, 0, st, bt);
}

// Exported patch costs: the raw sums divided by 3T (the same division, so the same bits, as a mean taken
// at evaluation time).
__global__ void k_cost_export(const float* src, float* dst, int n, float scale) {
    begin_kernel();
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) dst[i] = src[i] / scale;
}
void launch_cost_export(const float* src, float* dst, int n, int radius, int census, cudaStream_t st) {
    const int d = 2 * radius + 1;
    launch_kernel(k_cost_export, (n + 255) / 256, 256, 0, st, src, dst, n, (float)((census ? 24 : 3) * d * d));
}



}  // namespace gpm

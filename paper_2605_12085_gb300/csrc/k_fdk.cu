// FDK reconstruction (the analytic baseline of Sec. 3) on sm_103a: cosine
// weighting and Ram-Lak ramp filtering of every detector row, then a
// weighted gather backprojection.  Everything is written on the virtual
// detector through the rotation axis (scale m = SOD/SDD):
//
//   q(a_i, b) = t * sum_n h(a_i - a_n) p(a_n, b) SOD / sqrt(SOD^2 + a_n^2 + b^2),
//       t = du m, h(0) = 1/(4 t^2), h(k t) = -1/(pi^2 k^2 t^2) for odd k, 0 else;
//   f(x) = sum_views (dtheta/2) q(eta/U, z/U) / U^2,
//       U = (SOD - xi)/SOD, xi = x cos + y sin, eta = -x sin + y cos.
//
// k_fdk_filter: a block takes FDK_ROWS consecutive detector rows of one view
// and stages the weighted rows in shared memory; each thread forms 8 filtered
// values of one row (same parity, two columns apart) from a sliding window of
// coefficients in registers, so one shared-memory read feeds 8 FMAs.  It
// writes q transposed, as column pairs:
// entry (s, c, e) = (q(c - 1, e - 2), q(c, e - 2)) for c = 0 .. nu and rows of
// fdk_row_stride(nv) entries, zero outside the detector, so the
// backprojection reads the four taps of a voxel as two aligned float2 loads of
// consecutive entries along z and needs no bounds test at the edges.  The
// block restages its results in shared memory and stores them as float4s.
// k_fdk_bp (one launch per 32 views; each adds into the volume but the very
// first, which writes it): a block owns 8 x 4 voxel columns, a warp 2 x 2 of them
// and 32 * KPL voxels along z (lane l: k0 + l + 32 q).  The geometry of a (column,
// view) pair -- detector column and weight, the row coordinate of voxel k0 and the
// rows per voxel in Q.32 -- is formed by one thread in FP64 (slow on this part: one
// reciprocal by an FP32 estimate and a Newton step) and kept in shared memory for the
// warp.  Per voxel and view: a 64-bit add and a funnel shift for the row, two 8-byte
// loads, the interpolation along the rows as one packed subtraction and FMA, along
// the columns and into the sum as three operations.  The four voxel columns of a
// warp and the 32 of a block read the same few detector columns of a view from L1.
// Output in [j][i][k] order.
#include <math.h>

#include "fbl_internal.cuh"

namespace fbl {
namespace {

constexpr int FDK_ROWS = 8;    // detector rows per filter block
constexpr int FDK_FT = 256;    // filter block threads
constexpr int FDK_WARPS = 8;   // warps per backprojection block: 4 x 2, each 2 x 2 voxel columns
constexpr int FDK_VB = 16;     // views whose pair geometry a block forms at once

// float2 entries per detector column of the filtered projections: row v at
// entry v + 2, two zero entries below row 0 and at least two above row nv - 1,
// even so that every column starts on a 16-byte boundary
__host__ __device__ inline int fdk_row_stride(int nv) { return (nv + 5) & ~1; }

// The filter's row staging: FR_PAD zero columns on each side of a row and a
// row stride of 2 (mod 32) words, so that the 32 lanes of a warp (8 rows x 2
// column groups 16 apart x 2 parities) read 32 different shared-memory banks.
constexpr int FR_PAD = 32;
constexpr int FR_E = 8;  // outputs per thread: columns i0, i0 + 2, .., i0 + 14
__host__ __device__ inline int fr_row_len(int nu) { return ((nu + 2 * FR_PAD + 29) & ~31) + 2; }
__host__ __device__ inline int fr_kh(int nu) { return (nu + FR_PAD + 2 * FR_E - 1) | 1; }  // odd

template <typename TY>
__global__ void __launch_bounds__(FDK_FT) k_fdk_filter(const TY *__restrict__ y, int nu, int nv,
                                                       double sod, double du_m, double dv_m, double cu,
                                                       double cv, float *__restrict__ qt) {
    extern __shared__ float fsm[];
    const int lp = nu + 2 * FR_PAD, rl = fr_row_len(nu), KH = fr_kh(nu);
    float *P = fsm;                      // [FDK_ROWS][rl] weighted rows, zero-padded
    float *Q = fsm + FDK_ROWS * rl;      // [FDK_ROWS][nu] filtered rows
    float *H = Q + FDK_ROWS * nu;        // t h(k t) for odd k in [-KH, KH], at (k + KH) / 2
    const int s = blockIdx.y, r0 = blockIdx.x * FDK_ROWS;
    const double t = du_m;
    // the odd taps in FP32 (k^2 is exact, one rounded division): FP64
    // divisions per block would cost more than the filtering
    const float ct = (float)(-1.0 / (M_PI * M_PI * t));
    for (int j = threadIdx.x; j <= KH; j += FDK_FT) {
        const float k = (float)(2 * j - KH);
        H[j] = ct / (k * k);
    }
    // cosine weight in FP32 (relative error below 1e-6): FP64 arithmetic is
    // slow on this part
    const float sodf = (float)sod, sod2 = (float)(sod * sod), duf = (float)du_m, dvf = (float)dv_m;
    const float cuf = (float)cu, cvf = (float)cv;
    for (int e = threadIdx.x; e < FDK_ROWS * lp; e += FDK_FT) {
        const int r = e / lp, c = e - r * lp, iu = c - FR_PAD, iv = r0 + r;
        float val = 0.f;
        if (iv < nv && iu >= 0 && iu < nu) {
            const float a = ((float)iu - cuf) * duf, b = ((float)iv - cvf) * dvf;
            const float w = sodf * rsqrtf(fmaf(a, a, fmaf(b, b, sod2)));
            val = w * to_f32(y[((size_t)s * nv + iv) * nu + iu]);
        }
        P[r * rl + c] = val;
    }
    __syncthreads();
    // A warp takes the 8 rows and 32 columns [Iw, Iw + 32): lane l the row
    // l / 4 and the 8 outputs i0 + 2e, i0 = Iw + 16 ((l / 2) % 2) + l % 2.
    // Output i sums t h(n - i) P(n) over the odd offsets n - i (the even ones
    // other than 0 vanish); with d = n - i0 the coefficient of output e is
    // t h(d - 2e), so as d steps by 2 the 8 coefficients shift by one place and
    // one new one is read (the same for the whole warp).  d runs over
    // [-Iw - 31, nu - 1 - Iw], which covers n = 0 .. nu - 1 for every lane; the
    // zero padding supplies the rest.
    const float c0 = (float)(1.0 / (4.0 * t));
    const int nseg = (nu + 31) / 32;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int r = lane >> 2;
    const float *Pr = P + r * rl + FR_PAD;
    for (int seg = warp; seg < nseg; seg += FDK_FT / 32) {
        const int Iw = seg * 32;
        const int i0 = Iw + 16 * ((lane >> 1) & 1) + (lane & 1);
        float acc[FR_E], hw[FR_E];
        const int dmin = -Iw - 31, dmax = nu - 1 - Iw;
#pragma unroll
        for (int e = 0; e < FR_E; ++e) {
            acc[e] = c0 * Pr[i0 + 2 * e];
            hw[e] = H[(dmin - 2 * e + KH) >> 1];
        }
        const float *pp = Pr + i0;
        const float *hh = H + ((dmin + 2 + KH) >> 1);
#pragma unroll 8
        for (int d = dmin; d <= dmax; d += 2, ++hh) {
            const float p = pp[d];
#pragma unroll
            for (int e = 0; e < FR_E; ++e) acc[e] = fmaf(hw[e], p, acc[e]);
#pragma unroll
            for (int e = FR_E - 1; e > 0; --e) hw[e] = hw[e - 1];
            hw[0] = *hh;
        }
#pragma unroll
        for (int e = 0; e < FR_E; ++e)
            if (i0 + 2 * e < nu) Q[r * nu + i0 + 2 * e] = acc[e];
    }
    __syncthreads();
    // column pairs (c - 1, c) of row pairs (r0 + 2p, r0 + 2p + 1) as one float4;
    // rows at or past nv keep the zeros of the cleared buffer
    const int rs = fdk_row_stride(nv);
    float2 *out2 = reinterpret_cast<float2 *>(qt) + (size_t)s * (nu + 1) * rs + r0 + 2;
    for (int e = threadIdx.x; e < (nu + 1) * (FDK_ROWS / 2); e += FDK_FT) {
        const int c = e / (FDK_ROWS / 2), p = e - c * (FDK_ROWS / 2), r = 2 * p;
        if (r0 + r >= nv) continue;
        float4 v;
        v.x = c > 0 ? Q[r * nu + c - 1] : 0.f;
        v.y = c < nu ? Q[r * nu + c] : 0.f;
        v.z = c > 0 ? Q[(r + 1) * nu + c - 1] : 0.f;
        v.w = c < nu ? Q[(r + 1) * nu + c] : 0.f;
        *reinterpret_cast<float4 *>(out2 + (size_t)c * rs + r) = v;
    }
}

struct FdkView {
    double c, s, w;  // cos, sin, dtheta / 2
};

struct __align__(16) FdkPair {
    const float2 *col;  // row 0 of the column pair
    long long t;        // Q.32 detector row of voxel k0
    long long dv;       // Q.32 rows per voxel
    float tu, w;        // horizontal weight; (dtheta/2) / U^2, 0 where the column is off the detector
};

// Interpolation between two rows of a column pair: a + f (b - a) on both halves
// (packed FP32x2, the roundings of two scalar operations).
__device__ __forceinline__ float2 fdk_lerp2(float f, float2 a, float2 b) {
    float2 d;
    asm("{\n\t.reg .b64 a, b, f, d;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tmov.b64 f, {%6, %6};\n\t"
        "sub.rn.f32x2 b, b, a;\n\tfma.rn.f32x2 d, f, b, a;\n\tmov.b64 {%0, %1}, d;\n\t}"
        : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(f));
    return d;
}

// One (column, view) pair added to the lane's voxels.  CLAMP: some voxel's row
// lies outside [-2, nv]; it is clamped to rows that are zero, with zero followers.
template <int KPL, bool CLAMP>
__device__ __forceinline__ void fdk_add(const FdkPair &p, int nv, float (&acc)[KPL]) {
    const int lane = threadIdx.x;
    const float2 *col = p.col;
    const long long dv = p.dv, dv32 = dv << 5;
    long long t = p.t + (long long)lane * dv;
    const float tu = p.tu, w = p.w;
#pragma unroll
    for (int q = 0; q < KPL; ++q) {
        int r = fx32_floor(t);
        if (CLAMP) r = min(max(r, -2), nv);
        const float2 A = __ldg(col + r), B = __ldg(col + r + 1);
        const float2 v = fdk_lerp2(fx32_frac(t), A, B);
        acc[q] = fmaf(w, fmaf(tu, v.y - v.x, v.x), acc[q]);
        t += dv32;
    }
}

template <int KPL>
__global__ void __launch_bounds__(32 * FDK_WARPS, 3) k_fdk_bp(const float2 *__restrict__ qt, const FdkView *views, int n_sel,
                                                           int nx, int ny, int nz, int nu, int nv, double vx, double vy,
                                                           double sod, double inv_du_m, double rows_per_voxel, double cu,
                                                           double cv, int accumulate, float *__restrict__ gzi) {
    __shared__ FdkPair pairs[FDK_WARPS][FDK_VB][4];
    const int lane = threadIdx.x, wi = threadIdx.y;
    const int i0 = blockIdx.x * 8 + 2 * (wi & 3), j0 = blockIdx.y * 4 + 2 * (wi >> 2);
    const int k0 = blockIdx.z * 32 * KPL;
    const int rs = fdk_row_stride(nv);
    const size_t vstride = (size_t)(nu + 1) * rs;
    float acc[4][KPL];
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int q = 0; q < KPL; ++q) acc[c][q] = 0.f;
    for (int s0 = 0; s0 < n_sel; s0 += FDK_VB) {
        const int nb = min(FDK_VB, n_sel - s0);
        __syncwarp();
        // half a warp per voxel column, a view per lane
        for (int h = 0; h < 2; ++h) {
            const int c = 2 * h + (lane >> 4), sv = lane & 15;
            if (sv >= nb) continue;
            const FdkView v = views[s0 + sv];
            const double x = (i0 + (c & 1) - 0.5 * (nx - 1)) * vx, y = (j0 + (c >> 1) - 0.5 * (ny - 1)) * vy;
            const double D = sod - fma(x, v.c, y * v.s);
            // 1 / D: an FP32 estimate and one Newton step (relative error 2^-45)
            const double e0 = (double)__frcp_rn((float)D), inv = fma(e0, fma(-D, e0, 1.0), e0);
            const double invU = sod * inv;
            const double fu = fma(fma(y, v.c, -x * v.s) * invU, inv_du_m, cu);
            const double dfv = rows_per_voxel * invU;
            FdkPair p;
            p.col = qt;
            p.t = p.dv = 0;
            p.tu = p.w = 0.f;
            const bool in = i0 + (c & 1) < nx && j0 + (c >> 1) < ny;
            if (in && fu > -1.0 && fu < (double)nu) {
                const long long F = __double2ll_rd(fu * 4294967296.0);
                p.col = qt + (size_t)(s0 + sv) * vstride + (size_t)(fx32_floor(F) + 1) * rs + 2;
                p.tu = fx32_frac(F);
                p.w = (float)(v.w * invU * invU);
                p.dv = __double2ll_rn(dfv * 4294967296.0);
                p.t = __double2ll_rn(fma(k0 - 0.5 * (nz - 1), dfv, cv) * 4294967296.0);
            }
            pairs[wi][sv][c] = p;
        }
        __syncwarp();
        for (int t = 0; t < nb; ++t) {
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const FdkPair &p = pairs[wi][t][c];
                if (p.w == 0.f) continue;  // uniform over the warp
                if (fx32_floor(p.t) >= -2 && fx32_floor(p.t + (32 * KPL - 1) * p.dv) <= nv) fdk_add<KPL, false>(p, nv, acc[c]);
                else fdk_add<KPL, true>(p, nv, acc[c]);
            }
        }
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const int i = i0 + (c & 1), j = j0 + (c >> 1);
        if (i >= nx || j >= ny) continue;
        float *out = gzi + ((size_t)j * nx + i) * nz;
#pragma unroll
        for (int q = 0; q < KPL; ++q) {
            const int k = k0 + lane + 32 * q;
            if (k < nz) out[k] = accumulate ? out[k] + acc[c][q] : acc[c][q];
        }
    }
}

}  // namespace

size_t fdk_filtered_elems(int n_sel, int nu, int nv) { return (size_t)n_sel * (nu + 1) * fdk_row_stride(nv) * 2; }

cudaError_t launch_fdk_filter(const void *y, int y_dtype, int n_sel, int nu, int nv, double sod, double sdd,
                              double du, double dv, float *qt, cudaStream_t st) {
    if (n_sel <= 0) return cudaSuccess;
    const double m = sod / sdd;
    const size_t smem = ((size_t)FDK_ROWS * fr_row_len(nu) + (size_t)FDK_ROWS * nu + fr_kh(nu) + 1) * sizeof(float);
    dim3 grid((nv + FDK_ROWS - 1) / FDK_ROWS, n_sel);
    const double cu = 0.5 * (nu - 1), cv = 0.5 * (nv - 1);
    cudaError_t e = cudaSuccess;
    switch (y_dtype) {
        case FBL_BF16:
            e = cudaFuncSetAttribute(k_fdk_filter<__nv_bfloat16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)smem);
            if (e == cudaSuccess)
                k_fdk_filter<<<grid, FDK_FT, smem, st>>>((const __nv_bfloat16 *)y, nu, nv, sod, du * m, dv * m,
                                                         cu, cv, qt);
            break;
        case FBL_F16:
            e = cudaFuncSetAttribute(k_fdk_filter<__half>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e == cudaSuccess)
                k_fdk_filter<<<grid, FDK_FT, smem, st>>>((const __half *)y, nu, nv, sod, du * m, dv * m, cu, cv,
                                                         qt);
            break;
        default:
            e = cudaFuncSetAttribute(k_fdk_filter<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e == cudaSuccess)
                k_fdk_filter<<<grid, FDK_FT, smem, st>>>((const float *)y, nu, nv, sod, du * m, dv * m, cu, cv,
                                                         qt);
            break;
    }
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

// One launch per FDK_SUB views (accumulating into the volume): every block of a
// launch reads the same few views, whose filtered rows then stay in L2 for
// the blocks of neighbouring voxel rows (a launch over all views of a chunk
// let blocks drift apart by up to the whole chunk and re-read from DRAM).
constexpr int FDK_SUB = 32;

cudaError_t launch_fdk_bp(const float *qt, const double *view_csw, int n_sel, int nx, int ny, int nz, int nu,
                          int nv, double vx, double vy, double vz, double sod, double sdd, double du, double dv,
                          int accumulate, float *gzi, cudaStream_t st) {
    const double m = sod / sdd;
    // voxels per lane: the least work over the spans of 32 KPL voxels
    int kpl = 8;
    const auto cost = [nz](int k) { return ((nz + 32 * k - 1) / (32 * k)) * (k + 1); };
    for (int k : {6, 4, 2})
        if (cost(k) < cost(kpl)) kpl = k;
    dim3 block(32, FDK_WARPS);
    dim3 grid((nx + 7) / 8, (ny + 3) / 4, (nz + 32 * kpl - 1) / (32 * kpl));
    const size_t vstride = (size_t)(nu + 1) * fdk_row_stride(nv);  // float2 entries per view
    auto kernel = kpl == 8 ? k_fdk_bp<8> : kpl == 6 ? k_fdk_bp<6> : kpl == 4 ? k_fdk_bp<4> : k_fdk_bp<2>;
    for (int s0 = 0; s0 < n_sel; s0 += FDK_SUB) {
        const int ns = n_sel - s0 < FDK_SUB ? n_sel - s0 : FDK_SUB;
        kernel<<<grid, block, 0, st>>>((const float2 *)qt + (size_t)s0 * vstride, (const FdkView *)view_csw + s0, ns, nx,
                                       ny, nz, nu, nv, vx, vy, sod, 1.0 / (du * m), vz / (dv * m), 0.5 * (nu - 1),
                                       0.5 * (nv - 1), (accumulate || s0 > 0) ? 1 : 0, gzi);
    }
    return cudaGetLastError();
}

}  // namespace fbl

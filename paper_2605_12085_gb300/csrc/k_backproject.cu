// K2 -- exact transpose A_N^T of the mini-batch projector (Step 2b's
// grad f_N = (n_theta/N_t) A_N^T (A_N x - b_N), eq. (2.5)) on sm_103a, in
// gather form: every voxel collects the taps that K1 gives it.  No atomics.
//
// A ray of family f touches voxel (i, j, k) only on the plane m of its
// dominant axis that contains the voxel (m = i for x-planes, m = j for
// y-planes), with weight wb * wz: wb from the in-plane crossing q_b(m) of its
// detector column, wz from the vertical crossing q_z(m) of its row.
//
// Two forms.  Volumes large enough to fill the GPU run in strips (k_strips.cu) where
// the detector rows are at most STRIP_MAX_STEP voxels apart in them.
// The others run here, one voxel column per warp: many more and shorter warps
// (64^3, 10 views: 23.9 against 36 us).  A batch runs each volume in its own
// geometry's form, so that its results are the single-volume solver's, although
// a batch of small volumes fills the GPU and strips would be a little faster there
// (16 volumes of 24^3..80^3: 0.95 against 1.01 ms per iteration).
//
// A warp owns 32*VPL voxels of one (i, j) column along z (lane l holds the VPL
// consecutive voxels k0 + VPL*l ..; VPL = 2 or 4).  Everything that depends only on (i, j)
// and the view -- the candidate columns within hwu of the voxel column's
// projection, each column's family, plane m, exact in-plane weight wb (from
// the same Q.40 crossing K1 uses) and vertical step -- is uniform over the
// warp.  Along z the kernel forms the column's z-profile, the transpose of
// K1's linear interpolation: the rows of the column cross plane m at q_z =
// q_z(first) + t*step, and a row whose crossing lies in the unit cell
// [k, k + 1) at fraction f gives (1 - f) r to voxel k and f r to voxel k + 1.
// A lane walks the cells kfirst - 1 .. kfirst + VPL - 1 in order, taking each
// row once (at most C = ceil(1 / step) rows per cell, a warp-uniform template
// choice); the offset of the lane's first row is exact from the Q.40
// crossing and the next ones follow by the per-row step, so the weights are
// accurate to about 1e-6.  Columns whose cells all stay inside the zero pads
// skip the clamp (a warp vote).  The residual arrives transposed and
// zero-padded (rt[s][iu][RT_PAD + iv], already multiplied by K1's row weight
// W), so the lanes' row reads are contiguous and need no bounds test.  The
// gradient is written in z-innermost order [j][i][k], coalesced.
#include "fbl_internal.cuh"
#include "fbl_reduce.cuh"

namespace fbl {
namespace {

constexpr int K2_LANES = 32;

// Launch configuration of the backprojector: k2_vpl 2 and 4 (24 the same) are
// one voxel column per warp with that many consecutive voxels per lane; 8 and 28
// are strips with 4 or 8 voxels per lane, 16 strips with 6 (all three run as 4
// where the geometry's rows are too far apart for strips).
__host__ __device__ __forceinline__ int k2_vpl_of(const DevGeom &g) { return g.k2_vpl == 2 && g.wide_rows < 2 ? 2 : 4; }
constexpr int K2_WARPS = 8;   // consecutive i per block

// Packed FP32x2 arithmetic (sm_100 family): the same IEEE operation on each
// half, so results equal two scalar operations bit for bit.
__device__ __forceinline__ void pk_mul(float ax, float ay, float bx, float by, float &dx, float &dy) {
    asm("{\n\t.reg .b64 a, b, d;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\t"
        "mul.rn.f32x2 d, a, b;\n\tmov.b64 {%0, %1}, d;\n\t}"
        : "=f"(dx), "=f"(dy) : "f"(ax), "f"(ay), "f"(bx), "f"(by));
}
__device__ __forceinline__ void pk_add(float ax, float ay, float bx, float by, float &dx, float &dy) {
    asm("{\n\t.reg .b64 a, b, d;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\t"
        "add.rn.f32x2 d, a, b;\n\tmov.b64 {%0, %1}, d;\n\t}"
        : "=f"(dx), "=f"(dy) : "f"(ax), "f"(ay), "f"(bx), "f"(by));
}
__device__ __forceinline__ void pk_sub(float ax, float ay, float bx, float by, float &dx, float &dy) {
    asm("{\n\t.reg .b64 a, b, d;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\t"
        "sub.rn.f32x2 d, a, b;\n\tmov.b64 {%0, %1}, d;\n\t}"
        : "=f"(dx), "=f"(dy) : "f"(ax), "f"(ay), "f"(bx), "f"(by));
}
__device__ __forceinline__ void pk_fma(float ax, float ay, float bx, float by, float cx, float cy, float &dx,
                                       float &dy) {
    asm("{\n\t.reg .b64 a, b, c, d;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\t"
        "mov.b64 c, {%6, %7};\n\tfma.rn.f32x2 d, a, b, c;\n\tmov.b64 {%0, %1}, d;\n\t}"
        : "=f"(dx), "=f"(dy) : "f"(ax), "f"(ay), "f"(bx), "f"(by), "f"(cx), "f"(cy));
}

// One cell's rows: r[t] the row values already masked (0 where the row is not
// in the cell), et[t] their offsets from the cell's bottom; then the walk
// moves to the next cell.
template <int C, bool CLAMP>
struct CellRows {
    float r[C], et[C];
    __device__ __forceinline__ void load(const float *__restrict__ rcol, int &lo, float &e, float step, int lo_max) {
        // a 32-bit row index, the address formed per cell (cheaper than stepping
        // a 64-bit pointer by the data-dependent row count)
        const float *w = rcol + (CLAMP ? min(max(lo, -RT_PAD), lo_max) : lo);
        bool v[C];
        et[0] = e;
        v[0] = C > 1 ? true : e < 1.f;
        {
            const float r0 = __ldg(w);
            r[0] = v[0] ? r0 : 0.f;
        }
#pragma unroll
        for (int t = 1; t < C; ++t) {
            et[t] = fmaf((float)t, step, e);
            v[t] = et[t] < 1.f;
            r[t] = v[t] ? __ldg(w + t) : 0.f;
        }
        // next cell: e of the first row not taken, minus one
        float en = fmaf((float)C, step, e);
#pragma unroll
        for (int t = C - 1; t >= 0; --t) en = v[t] ? en : fmaf((float)t, step, e);
        e = en - 1.f;
        int n = 0;
#pragma unroll
        for (int t = 0; t < C; ++t) n += v[t] ? 1 : 0;
        lo += n;
    }
};

// The z-profile of one candidate column over the lane's VPL voxels, by unit
// cells: cell c = [k, k + 1) of the z axis holds the rows whose crossing q_z
// lies in it; a row at fraction f = q_z - k gives (1 - f) r to voxel k and
// f r to voxel k + 1 (the transpose of K1's linear interpolation along z).
// The lane walks cells kfirst - 1 .. kfirst + VPL - 1 (VPL + 1 cells) with
// e = q_z(first row not yet taken) - k, in [0, step] (a row on a cell
// boundary may be taken by either cell: f = 1 in the lower cell gives the
// same two weights as f = 0 in the upper one).  C = 1: rows more than one
// voxel apart, at most one per cell, tested.  C >= 2: rows at most one voxel
// apart (step <= 1), so the first row is always in the cell, and at most C
// rows per cell, the others tested.  The cells of voxels q and q + 1 are
// loaded one after the other and their sums formed with packed FP32x2
// operations; add2(q, P_q, P_q+1) receives the two voxels' profile values.
// CLAMP as for the windows: a window outside [-RT_PAD, lo_max] holds only
// zero rows.
template <int C, int VPL, bool CLAMP, class Add2>
__device__ __forceinline__ void column_cells(Add2 add2, const float *__restrict__ rcol, int lo, float e,
                                             float step, int lo_max) {
    float carry;
    {  // cell kfirst - 1: only its f part, to voxel 0
        CellRows<C, CLAMP> a;
        a.load(rcol, lo, e, step, lo_max);
        float s1 = a.et[0] * a.r[0];
#pragma unroll
        for (int t = 1; t < C; ++t) s1 = fmaf(a.et[t], a.r[t], s1);
        carry = s1;
    }
#pragma unroll
    for (int q = 0; q < VPL; q += 2) {  // the cells of voxels q and q + 1, two at a time
        CellRows<C, CLAMP> a, b;
        a.load(rcol, lo, e, step, lo_max);
        b.load(rcol, lo, e, step, lo_max);
        float s0a = a.r[0], s0b = b.r[0], s1a, s1b;
        pk_mul(a.et[0], b.et[0], a.r[0], b.r[0], s1a, s1b);
#pragma unroll
        for (int t = 1; t < C; ++t) {
            pk_add(s0a, s0b, a.r[t], b.r[t], s0a, s0b);
            pk_fma(a.et[t], b.et[t], a.r[t], b.r[t], s1a, s1b, s1a, s1b);
        }
        float da, db, Pa, Pb;
        pk_sub(s0a, s0b, s1a, s1b, da, db);
        pk_add(carry, s1a, da, db, Pa, Pb);
        add2(q, Pa, Pb);
        carry = s1b;
    }
}

// Dispatch on the column's row spacing: one row per cell at most (step > 1),
// else the geometry's largest rows-per-cell bound or one less.
template <int NTAP, int VPL, bool CLAMP, class Add>
__device__ __forceinline__ void column_cells_c(int cc, float step, Add add, const float *__restrict__ rcol, int lo,
                                               float e, int lo_max) {
    constexpr int CM = (NTAP + 1) / 2;
    constexpr int CM1 = CM > 2 ? CM - 1 : 2;
    if (CM < 2 || step > 1.f) column_cells<1, VPL, CLAMP>(add, rcol, lo, e, step, lo_max);
    else if (CM > 2 && cc <= CM1) column_cells<CM1, VPL, CLAMP>(add, rcol, lo, e, step, lo_max);
    else column_cells<(CM < 2 ? 2 : CM), VPL, CLAMP>(add, rcol, lo, e, step, lo_max);
}

// Rows per cell of a column (an upper bound: the geometry's ntap is
// floor(2 x) + 1 and this floor(x) + 1 with the same x).
__device__ __forceinline__ int cells_rows(float inv) { return (int)(inv * 1.0001f + 0.001f) + 1; }

// One candidate column's z-profile over the lane's VPL voxels, added to acc
// with the in-plane weight wb; lo and d0 = q_z(lo) - kfirst in (-1, -1 + step]
// locate the lane's first row.
template <int NTAP, int VPL>
__device__ __forceinline__ void column_profile(float (&acc)[VPL], float wb, const float *__restrict__ rcol,
                                                int lo, float d0, float step, float inv, int lo_max) {
    const int cc = cells_rows(inv);
    const bool inside = lo >= -RT_PAD && lo + (int)((float)VPL * inv) + 2 <= lo_max;
    auto add = [&](int q, float Pa, float Pb) { pk_fma(wb, wb, Pa, Pb, acc[q], acc[q + 1], acc[q], acc[q + 1]); };
    if (__all_sync(0xffffffffu, inside))
        column_cells_c<NTAP, VPL, false>(cc, step, add, rcol, lo, d0 + 1.f, lo_max);
    else
        column_cells_c<NTAP, VPL, true>(cc, step, add, rcol, lo, d0 + 1.f, lo_max);
}

// One block's work: voxel columns i = bx*8 .. bx*8+7 of row j, z-span bz;
// the block's sum of squared gradient values goes to *g2_partial (if not NULL).
// WIDE: rows too far apart for 32-bit conversions.  Called by every thread.
template <int NTAP, int K2_VPL, bool WIDE = false>
__device__ __forceinline__ void k2_tile(const BpArgs &a, int bx, int j, int bz, double *g2_partial) {
    constexpr int K2_KSPAN = K2_LANES * K2_VPL;
    const DevGeom &g = a.g;
    const int lane = threadIdx.x;
    const int i = bx * K2_WARPS + threadIdx.y;  // uniform over the warp
    const int kfirst = bz * K2_KSPAN + K2_VPL * lane;  // this lane: kfirst .. kfirst+VPL-1
    float acc[K2_VPL];
#pragma unroll
    for (int q = 0; q < K2_VPL; ++q) acc[q] = 0.f;
    const float xc = ((float)i - g.cx) * g.vx;
    const float yc = ((float)j - g.cy) * g.vy;
    const int rp = rt_pitch(g.nv);
    const int nsel = i < g.nx ? a.n_sel : 0;  // a warp past the volume edge only joins the block sum
    const int lo_max = g.nv + RT_PAD - NTAP;  // last first-row whose taps stay in the pad
    const long long kfirst_fx = (long long)kfirst << FX_BITS;
    constexpr float kInv24 = 1.0f / 16777216.0f;  // 2^-24 (Q.40 >> 16)
    for (int s = 0; s < nsel; ++s) {
        const int v = a.views[s];
        const float2 cs = g.trig[v];
        const float xi = xc * cs.x + yc * cs.y;
        const float eta = -xc * cs.y + yc * cs.x;
        // the voxel column's projection: an estimate only (the window hwu keeps a
        // slack of 2% + 0.05 columns; the fast division errs by ~1e-4 column)
        const float iuc = eta * __fdividef(g.sdd, g.sod - xi) * g.inv_du + g.cu;
        const int iu_lo = max(0, (int)ceilf(iuc - g.hwu));
        const int iu_hi = min(g.nu - 1, (int)floorf(iuc + g.hwu));
        for (int iu = iu_lo; iu <= iu_hi; ++iu) {
            const size_t col = (size_t)v * g.nu + iu;
            const FxCol cF = g.colF[col];
            const bool famY = g.colB[col].z != 0.f;
            const int m = famY ? j : i;
            const int bb = famY ? i : j;
            const long long qb = cF.qb0 + (long long)m * cF.qb1;
            const int b0 = fx_floor(qb);
            const float fb = fx_frac(qb);
            const float wb = (b0 == bb) ? 1.f - fb : ((b0 + 1 == bb) ? fb : 0.f);
            if (wb == 0.f) continue;
            // row iv crosses plane m at q_z = 2*iv*Z + zoff (Q.40), 0 < Z < 2^40
            const long long Z = cF.h0 + (long long)m * cF.h1;
            const long long zoff = g.cz_fx - (long long)(g.nv - 1) * Z;
            // dq_z per row = 2Z (32-bit path)
            const float step = WIDE ? (float)(Z >> 15) * kInv24 : (float)(int)(Z >> 15) * kInv24;
            const float inv = __fdividef(1.f, step);            // rows per voxel (estimate)
            const float zoff_f = g.cz - (float)(g.nv - 1) * 0.5f * step;
            // first row whose crossing lies above kfirst - 1: estimate, then one exact correction
            int lo = (int)ceilf(((float)kfirst - zoff_f) * inv - inv);
            const long long d_fx = 2LL * lo * Z + zoff - kfirst_fx;
            // q_z(lo) - kfirst (|.| < 2 + step)
            float d0 = WIDE ? (float)(d_fx >> 16) * kInv24 : (float)(int)(d_fx >> 16) * kInv24;
            if (d0 <= -1.f) {
                ++lo;
                d0 += step;
            } else if (d0 - step > -1.f) {
                --lo;
                d0 -= step;
            }
            const float *rcol = a.rt + ((size_t)s * g.nu + iu) * rp + RT_PAD;
            column_profile<NTAP, K2_VPL>(acc, wb, rcol, lo, d0, step, inv, lo_max);
        }
    }
    float g2 = 0.f;
    if (i < g.nx) {
        float *out = a.gzi + ((size_t)j * g.nx + i) * g.nz;
#pragma unroll
        for (int q = 0; q < K2_VPL; ++q) {
            const int k = kfirst + q;
            if (k < g.nz) {
                const float val = a.scale * acc[q];
                out[k] = val;
                g2 = fmaf(val, val, g2);
            }
        }
    }
    if (g2_partial) {
        float vv[1] = {g2};
        double o[1];
        block_sum_f64<K2_LANES * K2_WARPS, 1>(vv, o);
        if (threadIdx.x == 0 && threadIdx.y == 0) *g2_partial = o[0];
    }
}

template <int NTAP, int K2_VPL>
// At most 48 registers (5 blocks per SM); with the per-voxel tap loop this
// kernel had before the cell walk, that cap measured 14.47 ms per 40-view
// launch at 512^3 (8 voxels per lane) against 14.68 and 18.9 ms with the
// compiler's own choices (40 registers, and 92-168 with one block per SM).
__global__ void __launch_bounds__(K2_LANES *K2_WARPS, 5) k2_backproject(const BpArgs a) {
    const size_t blk = ((size_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
    k2_tile<NTAP, K2_VPL>(a, blockIdx.x, blockIdx.y, blockIdx.z, a.g2_partials ? a.g2_partials + blk : nullptr);
}

// Rows more than COLUMN_MAX_STEP voxels apart: one form for all such geometries (a larger
// NTAP only adds tested rows), a call of its own in the batch, so that the usual tiles
// keep their registers (as a flag in them: 1.7 % of small batches).
__device__ __noinline__ void k2_tile_wide(const BpArgs &a, int bx, int j, int bz, double *g2_partial) {
    k2_tile<RT_PAD, 4, true>(a, bx, j, bz, g2_partial);
}
__global__ void __launch_bounds__(K2_LANES *K2_WARPS) k2_backproject_wide(const __grid_constant__ BpArgs a) {
    const size_t blk = ((size_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
    k2_tile_wide(a, blockIdx.x, blockIdx.y, blockIdx.z, a.g2_partials ? a.g2_partials + blk : nullptr);
}

// Persistent batched backprojector: the blocks of k2_backproject of every volume
// that does not run in strips (the tiles from hdr->strip_tiles on), taken from an
// atomic counter.  Each volume keeps its own voxels per lane (its geometry's
// k2_vpl, a warp-uniform switch).  At most 64 registers (4 blocks per SM): with the
// single-volume kernel's 48 it spills, 12 iterations of 4 volumes of 20^3..41^3 took
// 2.42 instead of 2.35 ms (4 voxels per lane; BF16), 16 of 96^3..320^3 in columns 42.2
// instead of 41.6 ms per iteration (learned first step).
template <int NTAP>
__global__ void __launch_bounds__(K2_LANES *K2_WARPS, 4) kb_backproject(const BatchHdr *hdr,
                                                                        const BatchVol *vols, int *ctr) {
    __shared__ int s_tile;
    __shared__ BpArgs sa;
    const int tid = threadIdx.x + K2_LANES * threadIdx.y;
    const int total = hdr->total[1];
    for (;;) {
        if (tid == 0) s_tile = hdr->strip_tiles + atomicAdd(ctr, 1);
        __syncthreads();
        const int t = s_tile;
        __syncthreads();
        if (t >= total) break;
        const int vi = batch_find(*hdr, vols, 1, t);
        const BatchVol &bv = vols[vi];
        // the volume's arguments, staged in shared memory for the whole block
        stage_words(&sa.g, &bv.g, sizeof(DevGeom), tid, K2_LANES * K2_WARPS);
        if (tid == 0) {
            sa.rt = bv.rt;
            sa.views = bv.views;
            sa.n_sel = bv.N_t;
            sa.scale = bv.scale;
            sa.gzi = bv.grad;
            sa.g2_partials = bv.partials;
        }
        __syncthreads();
        const BpArgs &a = sa;
        const int local = t - bv.first[1];
        const int gx = (bv.g.nx + K2_WARPS - 1) / K2_WARPS;
        const int bx = local % gx;
        const int rest = local / gx;
        const int j = rest % bv.g.ny;
        const int bz = rest / bv.g.ny;
        double *part = bv.partials + local;
        if (bv.g.wide_rows > 1) k2_tile_wide(a, bx, j, bz, part);
        else if (k2_vpl_of(bv.g) == 2) k2_tile<NTAP, 2>(a, bx, j, bz, part);
        else k2_tile<NTAP, 4>(a, bx, j, bz, part);
    }
    batch_leave(ctr);
}

}  // namespace

static dim3 k2_grid(const DevGeom &g) {
    if (k2_is_strips(g)) {
        const unsigned span = 32 * strip_zp(g.k2_vpl, g.nz);
        return dim3((g.nx + STRIP_EDGE - 1) / STRIP_EDGE, (g.ny + STRIP_EDGE - 1) / STRIP_EDGE, (g.nz + span - 1) / span);
    }
    const int vpl = k2_vpl_of(g);
    return dim3((g.nx + K2_WARPS - 1) / K2_WARPS, g.ny, (g.nz + K2_LANES * vpl - 1) / (K2_LANES * vpl));
}

int backproject_num_partials(const DevGeom &g) {
    const dim3 gr = k2_grid(g);
    return (int)(gr.x * gr.y * gr.z);
}

int backproject_default_config(const DevGeom &g) {
    const int nx = g.nx, ny = g.ny, nz = g.nz;
    // fewer than 100 patches of 8 x 8 x 128 (80^3) leave SMs idle: one voxel column
    // per warp, 64 voxels high where that is enough (64^3, 10 views: 23.9 us with 2
    // voxels per lane, 28.0 with 4, 36 in strips; 96^3: 48.5 with 4, 37 in strips)
    const int64_t patches = (int64_t)((nx + 7) / 8) * ((ny + 7) / 8) * ((nz + 127) / 128);
    if (patches <= 100) return nz <= 64 ? 2 : 4;
    if (g.wide_rows) return 4;
    return strip_cost(nz, 6) < strip_cost(nz, strip_zp(28, nz)) ? 16 : 28;
}

bool backproject_same_launch(const DevGeom &a, const DevGeom &b) {
    if (k2_is_strips(a) != k2_is_strips(b)) return false;
    return k2_is_strips(a) ? strip_zp(a.k2_vpl, a.nz) == strip_zp(b.k2_vpl, b.nz) : k2_vpl_of(a) == k2_vpl_of(b);
}

template <int NT>
static void launch_k2(int vpl, dim3 grid, dim3 block, cudaStream_t st, const BpArgs &a) {
    if (vpl == 2) k2_backproject<NT, 2><<<grid, block, 0, st>>>(a);
    else k2_backproject<NT, 4><<<grid, block, 0, st>>>(a);
}

template <class K>
static int k2_persistent_grid(K kernel) {
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, K2_LANES * K2_WARPS, 0);
    return (sms > 0 ? sms : 1) * (per_sm > 0 ? per_sm : 1);
}

template <int NT>
static cudaError_t launch_kb2(const BatchHdr *hdr, BatchVol *vols, int *ctr, cudaStream_t st) {
    auto k = kb_backproject<NT>;
    static const int grid = k2_persistent_grid(k);
    k<<<grid, dim3(K2_LANES, K2_WARPS), 0, st>>>(hdr, vols, ctr);
    return cudaGetLastError();
}

cudaError_t launch_batch_backproject(const BatchHdr *hdr, BatchVol *vols, int ntap, int *ctr,
                                     cudaStream_t st) {
    switch (ntap) {
        case 1: return launch_kb2<1>(hdr, vols, ctr, st);
        case 2: return launch_kb2<2>(hdr, vols, ctr, st);
        case 3: return launch_kb2<3>(hdr, vols, ctr, st);
        case 4: return launch_kb2<4>(hdr, vols, ctr, st);
        case 5: return launch_kb2<5>(hdr, vols, ctr, st);
        case 6: return launch_kb2<6>(hdr, vols, ctr, st);
        case 7: return launch_kb2<7>(hdr, vols, ctr, st);
        default: return launch_kb2<8>(hdr, vols, ctr, st);
    }
}

cudaError_t launch_backproject(const DevGeom &g, const float *rt, const int32_t *views,
                               int n_sel, float scale, float *gzi, cudaStream_t st,
                               double *g2_partials, const int *nonfinite) {
    BpArgs a;
    a.g2_partials = g2_partials;
    a.nonfinite = nonfinite;
    a.g = g;
    a.rt = rt;
    a.views = views;
    a.n_sel = n_sel;
    a.scale = scale;
    a.gzi = gzi;
    dim3 block(K2_LANES, K2_WARPS);
    const dim3 grid = k2_grid(g);
    if (k2_is_strips(g)) return launch_strips(a, grid, strip_zp(g.k2_vpl, g.nz), st);
    if (g.wide_rows > 1) {
        k2_backproject_wide<<<grid, block, 0, st>>>(a);
        return cudaGetLastError();
    }
    const int vpl = k2_vpl_of(g);
    switch (g.ntap) {  // rows per voxel and column, fixed per geometry (<= RT_PAD)
        case 1: launch_k2<1>(vpl, grid, block, st, a); break;
        case 2: launch_k2<2>(vpl, grid, block, st, a); break;
        case 3: launch_k2<3>(vpl, grid, block, st, a); break;
        case 4: launch_k2<4>(vpl, grid, block, st, a); break;
        case 5: launch_k2<5>(vpl, grid, block, st, a); break;
        case 6: launch_k2<6>(vpl, grid, block, st, a); break;
        case 7: launch_k2<7>(vpl, grid, block, st, a); break;
        default: launch_k2<8>(vpl, grid, block, st, a); break;
    }
    return cudaGetLastError();
}

}  // namespace fbl

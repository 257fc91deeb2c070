// K2 in strips -- the exact transpose A_N^T of k_backproject.cu for volumes large
// enough to fill the GPU: the same gather of the same taps, organised so that a
// column's z-profile is formed once for many voxels.
//
// A ray of family f touches voxel (i, j, k) only on the plane m of its dominant
// axis that contains the voxel, with weight wb * wz: wb from the in-plane
// crossing q_b(m) of its detector column, wz from the vertical crossing q_z(m)
// of its row.  The sum over a column's rows, the column's z-profile
// P(k) = sum_iv wz(iv, k) r(iv), is the same for the two in-plane voxels
// b0, b0 + 1 the column crosses between; only wb differs.
//
// Work decomposition.  A block owns an 8 x 8 patch of voxel columns and
// 32 * ZP voxels along z.  For the rays of one family a warp owns one plane of
// the patch and its strip of 8 in-plane voxels, 32 * ZP voxels high (lane l:
// k = kb + l + 32 q); it forms every z-profile that reaches the strip once and
// adds it to the profile's two voxel columns: about 9 profiles per 8 voxel
// columns and view (2.35 per voxel column with one column per warp, 1.5 with the
// 2 x 2 groups this replaced).  The families own different strips of the same
// patch: the y-planes' sums go to the gradient first, the x-planes' are added.
//
// A profile's constants -- the in-plane crossing, the rows per voxel to 32
// fractional bits, the row coordinate of the strip's first voxel -- depend only on
// the view, the column and the plane.  The lanes of a warp form them in parallel,
// one lane per candidate column of two views, into a list in shared memory.
// When the list is full the warp orders it by in-plane voxel (votes) and walks it
// voxel by voxel: the sums of the current voxel column and of the next one are in
// registers, and a finished column's is added to the strip's accumulators, which
// live in tensor memory (8 ZP columns of the warp's 32 lanes: 64 registers' worth
// per thread that would halve the resident warps).
//
// Per voxel a profile costs one 32 x 32 + 64 bit multiply-add and a funnel shift
// for the position of the voxel's first row, one FMA per weight (saturated
// where the weight may end), and one coalesced load and half a packed FMA per
// row: two rows where rows are more than a voxel apart, three down to 2/3 of a
// voxel, four down to 1/2 (uniform over the warp), with no chain from one voxel
// to the next.  The position is a fraction of a row, so rows are at most
// STRIP_MAX_STEP voxels apart here.  The rows taken in beside a voxel have weight
// 0; where some residual is infinite or NaN, an instantiation that leaves them out
// runs instead (launch_weight's flag).
//
// Measured (40 views at 512^3, 768^2; CUDA events): 8.23 ms for the 2 x 2 groups
// at 44.5 warp instructions per 32 voxel-views; 7.58 with strips and their sums in
// registers (36.3); 5.76 with one FMA per weight and 8 voxels per lane (23.1);
// 5.06 with the sums in tensor memory and 4 blocks per SM; 4.83 with the
// multiply-add position and the views of the other family dropped by a vote
// (21.0).  All 720 views through backproject(): 165.6 -> 111.0 ms, 91 in several
// launches (see launch_strips).  What bounds it now: instruction issue is
// active 56 % of cycles, L1 throughput 61 % (three loads per voxel), the rest
// are load and fixed latencies of 24 to 32 warps per SM.  Not kept: prefetching
// the next profile's rows or constants (5.1 to 5.5 ms), partial sums ended at
// the same views for every strip so that results do not depend on the
// configuration (5.3 ms).
#include <algorithm>

#include "fbl_internal.cuh"
#include "fbl_reduce.cuh"

namespace fbl {
namespace {

// Two FP32 values with packed arithmetic (sm_100 family FP32x2: the same
// roundings as two scalar operations).
struct F2 {
    float x, y;
};
__device__ __forceinline__ F2 pk_mul(F2 a, F2 b) {
    F2 d;
    asm("{\n\t.reg .b64 a, b, d;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\t"
        "mul.rn.f32x2 d, a, b;\n\tmov.b64 {%0, %1}, d;\n\t}"
        : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ F2 pk_fma(F2 a, F2 b, F2 c) {
    F2 d;
    asm("{\n\t.reg .b64 a, b, c, d;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tmov.b64 c, {%6, %7};\n\t"
        "fma.rn.f32x2 d, a, b, c;\n\tmov.b64 {%0, %1}, d;\n\t}"
        : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return d;
}
__device__ __forceinline__ F2 pk_fma(F2 a, float b, float c) { return pk_fma(a, F2{b, b}, F2{c, c}); }

// Tensor memory as the strips' accumulators: a warp's strip is EDGE * ZP
// columns of its 32 lanes (warp w of a block: lanes 32 (w % 4) on, columns
// (w / 4) EDGE ZP on).  Only this warp touches them.
__device__ __forceinline__ void tm_alloc(unsigned *slot, int cols) {  // one warp
    const unsigned a = (unsigned)__cvta_generic_to_shared(slot);
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(a), "r"(cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tm_free(unsigned addr, int cols) {  // the same warp
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(addr), "r"(cols) : "memory");
}
__device__ __forceinline__ void tm_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tm_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void tm_ld(unsigned addr, float *v) {
    if constexpr (N == 2)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];" : "=f"(v[0]), "=f"(v[1]) : "r"(addr) : "memory");
    else if constexpr (N == 4)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                     : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]) : "r"(addr) : "memory");
    else if constexpr (N == 8)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
                     : "r"(addr) : "memory");
    else {  // 6
        tm_ld<4>(addr, v);
        tm_ld<2>(addr + 4, v + 4);
    }
}
template <int N>
__device__ __forceinline__ void tm_st(unsigned addr, const float *v) {
    if constexpr (N == 2)
        asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%0], {%1, %2};" ::"r"(addr), "f"(v[0]), "f"(v[1]) : "memory");
    else if constexpr (N == 4)
        asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(v[0]), "f"(v[1]),
                     "f"(v[2]), "f"(v[3]) : "memory");
    else if constexpr (N == 8)
        asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(addr), "f"(v[0]),
                     "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]) : "memory");
    else {
        tm_st<4>(addr, v);
        tm_st<2>(addr + 4, v + 4);
    }
}
// Columns a block of `warps` warps holds (a power of two, at least 32).
__host__ __device__ constexpr int tm_cols(int warps, int edge, int zp) {
    int c = 32;
    while (c < (warps + 3) / 4 * edge * zp) c *= 2;
    return c;
}

// One z-profile of a strip.
struct __align__(16) K2Entry {
    const float *row;      // rt at the column's row 0, plus the kind's offset
    long long t;           // Q.32 row coordinate of the strip's first voxel
    unsigned inv;          // fraction of the rows per voxel, Q.32
    float step;            // voxels per row
    float w1;              // in-plane weight of voxel rel + 1 (1 - w1: of voxel rel)
    int info;              // rel + 1 | kind << 8 | whole rows per voxel << 16
};
static_assert(sizeof(K2Entry) == 32, "two 16-byte loads");

// Kinds of profile, by the rows per voxel and so the rows that can reach a
// voxel: two below 1 (rows more than a voxel apart), three in [1, 3/2], four in
// (3/2, 2), RT_PAD otherwise; +4 where some rows of the strip lie outside the
// pads.
enum K2Kind { K2_TWO = 0, K2_THREE = 1, K2_FOUR = 2, K2_MANY = 3, K2_CLAMP = 4 };
template <int KIND> struct K2Taps {
    static constexpr int kind = KIND & 3;
    static constexpr int taps = kind == K2_MANY ? RT_PAD : kind + 2;
    static constexpr int whole = kind == K2_TWO ? 0 : 1;  // whole rows per voxel (K2_MANY: the entry's)
    // The profile of voxel k starts at row floor(t) + off: two and four rows
    // bracket k (t its row coordinate, off = 0 and -1); three and more start at
    // the first row above k - 1 (t the row coordinate of k - 1, off = 1).
    static constexpr int off = kind == K2_TWO ? 0 : (kind == K2_FOUR ? -1 : 1);
};

// The constants of column iu of batch slot s in plane m, for the strip of
// voxels [bs, bs + edge) x [kb, kb + span); false if it does not reach the strip.
// MASKED: some residual is infinite or NaN, every profile is of the kind that
// leaves rows of weight 0 out.
template <bool MASKED>
__device__ __forceinline__ bool k2_entry(const BpArgs &a, int fam, int m, int bs, int edge, int kb, int span, int s,
                                         int v, int iu, K2Entry &e) {
    const DevGeom &g = a.g;
    const size_t col = (size_t)v * g.nu + iu;
    const float cfam = __ldg(&g.colB[col].z);
    const longlong2 q = __ldg((const longlong2 *)(g.colF + col)), h = __ldg((const longlong2 *)(g.colF + col) + 1);
    const long long qb = q.x + (long long)m * q.y;
    const int b0 = fx_floor(qb), rel = b0 - bs;
    // (a crossing in (-1, Nb) is within a voxel of the volume, in front of the source: Z > 0 below)
    if ((cfam != 0.f) != (fam != 0) || rel < -1 || rel >= edge || b0 >= (fam ? g.nx : g.ny)) return false;
    // row iv crosses the plane at q_z = iv S + zoff (Q.40)
    const long long Z = h.x + (long long)m * h.y, S = 2 * Z, zoff = g.cz_fx - (long long)(g.nv - 1) * Z;
    constexpr float k2m40 = 9.094947017729282e-13f;  // 2^-40
    const float step = fmaf((float)(int)(S >> 20), 1048576.f, (float)(int)(S & 0xfffff)) * k2m40;
    // rows per voxel in Q.32: an FP32 reciprocal X and one correction by its
    // exact remainder 2^72 - S X (below 2^51 for rows up to 8 voxels apart, so exact
    // modulo 2^64 and its top bits in 32; geometries here have at most STRIP_MAX_STEP)
    const float x0 = __fdividef(1.f, step);
    const unsigned long long X = (unsigned long long)__float2uint_rz(x0 * 16777216.f) << 8;
    const int R = (int)((long long)(0ull - (unsigned long long)S * X) >> 20);
    const long long inv = (long long)X + __float2int_rn((float)R * x0 * (1.f / 1048576.f));
    const int whole = (int)(inv >> 32);
    const unsigned invf = (unsigned)inv;
    const int kind = MASKED ? K2_MANY : whole == 0 ? K2_TWO : (whole == 1 ? (invf <= 0x80000000u ? K2_THREE : K2_FOUR) : K2_MANY);
    const int taps = kind == K2_MANY ? RT_PAD : kind + 2;
    const bool bracket = kind == K2_TWO || kind == K2_FOUR;
    const int off = kind == K2_TWO ? 0 : (kind == K2_FOUR ? -1 : 1);
    const int kt = kb - (bracket ? 0 : 1);
    // row coordinate of z = kt: an FP32 estimate, then the exact offset from that row
    const float zoff_f = g.cz - (float)(g.nv - 1) * 0.5f * step;
    const int r0 = (int)floorf(((float)kt - zoff_f) * x0);
    const long long d = ((long long)kt << FX_BITS) - zoff - (long long)r0 * S;  // about [0, S)
    // (and half a unit of the 23 bits its fraction is cut to: rounded, not cut)
    const long long t = ((long long)r0 << 32) + (((d >> 12) * inv) >> 28) + 256;
    // first rows of the strip's first and last voxel
    const int lo0 = fx32_floor(t) + off, lo1 = fx32_floor(t + (long long)(span - 1) * inv) + off;
    if (lo1 + taps <= 0 || lo0 >= g.nv) return false;  // only rows outside the detector
    const bool clamp = lo0 < -RT_PAD || lo1 + taps > g.nv + RT_PAD;
    e.row = a.rt + ((size_t)s * g.nu + iu) * rt_pitch(g.nv) + RT_PAD + off;
    e.t = t;
    e.inv = invf;
    e.step = step;
    e.w1 = fx_frac(qb);
    e.info = (rel + 1) | ((kind | (clamp ? K2_CLAMP : 0)) << 8) | (whole << 16);
    return true;
}

// Weights of a kind's rows at two voxels whose row coordinates have the
// fractions f1 - 1 (f1 in [1, 2)).  Bracketing kinds: with d = frac step the
// rows lie d + step and d below, step - d and 2 step - d above the voxel; the
// others: row j lies u + j step above k - 1, u = (1 - frac) step.  The weight
// is 1 - distance where positive, each one FMA on f1.
template <int KIND>
__device__ __forceinline__ void k2_weights(F2 f1, float step, F2 (&w)[K2Taps<KIND>::taps]) {
    constexpr int kind = K2Taps<KIND>::kind;
    auto sat = [](F2 f, float b, float c) { return F2{__saturatef(fmaf(f.x, b, c)), __saturatef(fmaf(f.y, b, c))}; };
    if constexpr (kind == K2_TWO) {
        w[0] = sat(f1, -step, 1.f + step);
        w[1] = sat(f1, step, fmaf(-2.f, step, 1.f));
    } else if constexpr (kind == K2_THREE) {
        w[0] = pk_fma(f1, -step, 2.f * step);
        const F2 x = pk_fma(f1, -step, fmaf(3.f, step, -1.f));
        w[1] = F2{1.f - fabsf(x.x), 1.f - fabsf(x.y)};
        w[2] = sat(f1, step, fmaf(-4.f, step, 2.f));
    } else if constexpr (kind == K2_FOUR) {
        w[0] = sat(f1, -step, 1.f);
        w[1] = pk_fma(f1, -step, 1.f + step);
        w[2] = pk_fma(f1, step, fmaf(-2.f, step, 1.f));
        w[3] = sat(f1, step, fmaf(-3.f, step, 1.f));
    } else {
        const F2 u = pk_fma(f1, -step, 2.f * step);
#pragma unroll
        for (int j = 0; j < RT_PAD; ++j) {
            const float c = fmaf((float)j, step, -1.f);
            w[j] = F2{__saturatef(1.f - fabsf(u.x + c)), __saturatef(1.f - fabsf(u.y + c))};
        }
    }
}

// The z-profile at the lane's voxels, k = lane + 32 q from the strip's first
// (row coordinate t).  The whole rows per voxel go into the row pointer (0 or
// 1, known from the kind), the fraction times k into t with one 32 x 32 + 64
// bit multiply-add.
template <int KIND, int ZP, bool MASKED = false>
__device__ __forceinline__ void k2_profile(float (&P)[ZP], const float *__restrict__ row, unsigned long long t,
                                           unsigned invf, int whole, float step, int nv) {
    constexpr int taps = K2Taps<KIND>::taps, off = K2Taps<KIND>::off;
    constexpr bool many = K2Taps<KIND>::kind == K2_MANY;
    const unsigned lane = threadIdx.x & 31;
    const int wl = many ? whole : K2Taps<KIND>::whole;
    t += (unsigned long long)lane * invf;
    row += lane * wl;
    // 1 + the fraction of t, to 23 bits
    auto frac1 = [](unsigned long long v) { return __uint_as_float(__funnelshift_r((unsigned)v, 0x7Fu, 9)); };
    // rows outside [-RT_PAD, nv] are clamped to rows whose followers are all pads (zero)
    auto rows = [&](unsigned long long v, int q) {
        const int lo = (int)(v >> 32);
        if (KIND & K2_CLAMP) {
            const int k = ((int)lane + 32 * q) * wl;
            return row - (int)lane * wl + min(max(lo + k, -RT_PAD - off), nv - off);
        }
        return row + lo + 32 * q * wl;
    };
#pragma unroll
    for (int q = 0; q < ZP; q += 2) {
        const unsigned long long ta = t + (unsigned long long)invf * (32u * q);
        const unsigned long long tb = t + (unsigned long long)invf * (32u * (q + 1));
        F2 w[taps];
        k2_weights<KIND>(F2{frac1(ta), frac1(tb)}, step, w);
        const float *ra = rows(ta, q), *rb = rows(tb, q + 1);
        F2 p{0.f, 0.f};
        if constexpr (MASKED) {  // a row that does not reach the voxel may hold an infinity or NaN
#pragma unroll
            for (int j = 0; j < taps; ++j) {
                const float xa = __ldg(ra + j), xb = __ldg(rb + j);
                if (w[j].x > 0.f) p.x = fmaf(w[j].x, xa, p.x);
                if (w[j].y > 0.f) p.y = fmaf(w[j].y, xb, p.y);
            }
        } else {
            p = pk_mul(w[0], F2{__ldg(ra), __ldg(rb)});
#pragma unroll
            for (int j = 1; j < taps; ++j) p = pk_fma(w[j], F2{__ldg(ra + j), __ldg(rb + j)}, p);
        }
        P[q] = p.x;
        P[q + 1] = p.y;
    }
}

template <int ZP>
__device__ __forceinline__ void k2_axpy(float w, const float (&P)[ZP], float (&acc)[ZP]) {
#pragma unroll
    for (int q = 0; q < ZP; q += 2) {
        const F2 r = pk_fma(F2{P[q], P[q + 1]}, F2{w, w}, F2{acc[q], acc[q + 1]});
        acc[q] = r.x;
        acc[q + 1] = r.y;
    }
}

// A warp's list of profiles, their order by strip voxel and each voxel's end in it.
constexpr int K2_CAP = 112;  // a round appends up to 32 entries
struct K2List {
    K2Entry e[K2_CAP];
    unsigned char order[K2_CAP];
    unsigned char end[16];
};

// One entry: its profile P times 1 - w1 into A (the strip's voxel rel) and w1 into B (rel + 1).
template <int ZP, bool MASKED>
__device__ __forceinline__ void k2_add(const K2Entry *e, int nv, float (&A)[ZP], float (&B)[ZP]) {
    const int4 wa = reinterpret_cast<const int4 *>(e)[0], wb = reinterpret_cast<const int4 *>(e)[1];
    const unsigned long long t = ((unsigned long long)(unsigned)wa.w << 32) | (unsigned)wa.z;
    const float *row = (const float *)(((unsigned long long)(unsigned)wa.y << 32) | (unsigned)wa.x);
    const unsigned invf = (unsigned)wb.x;
    const float step = __int_as_float(wb.y), w1 = __int_as_float(wb.z), w0 = 1.f - w1;
    float P[ZP];
    if constexpr (MASKED) {  // (w1 may be 0 and P infinite or NaN)
        k2_profile<K2_MANY | K2_CLAMP, ZP, true>(P, row, t, invf, wb.w >> 16, step, nv);
        k2_axpy<ZP>(w0, P, A);
        if (w1 != 0.f) k2_axpy<ZP>(w1, P, B);
        return;
    }
    const int kind = (wb.w >> 8) & 7;
    if (kind == K2_TWO) k2_profile<K2_TWO, ZP>(P, row, t, invf, 0, step, nv);
    else if (kind == K2_THREE) k2_profile<K2_THREE, ZP>(P, row, t, invf, 0, step, nv);
    else if (kind == (K2_TWO | K2_CLAMP)) k2_profile<K2_TWO | K2_CLAMP, ZP>(P, row, t, invf, 0, step, nv);
    else if (kind == (K2_THREE | K2_CLAMP)) k2_profile<K2_THREE | K2_CLAMP, ZP>(P, row, t, invf, 0, step, nv);
    else if (kind == K2_FOUR) k2_profile<K2_FOUR, ZP>(P, row, t, invf, 0, step, nv);
    else if (kind == (K2_FOUR | K2_CLAMP)) k2_profile<K2_FOUR | K2_CLAMP, ZP>(P, row, t, invf, 0, step, nv);
    else k2_profile<K2_MANY | K2_CLAMP, ZP>(P, row, t, invf, wb.w >> 16, step, nv);
    k2_axpy<ZP>(w0, P, A);
    k2_axpy<ZP>(w1, P, B);
}

// The n listed profiles into the strip's voxels (voxel b at tensor-memory column
// strip + b ZP): ordered by rel with warp votes, then summed voxel by voxel
// in registers, each voxel's sum added to tensor memory once.
template <int EDGE, int ZP, bool MASKED>
__device__ __forceinline__ void k2_sum(K2List &L, int n, int nv, unsigned strip) {
    const int lane = threadIdx.x & 31;
    constexpr int G = (K2_CAP + 31) / 32;
    int key[G];
#pragma unroll
    for (int q = 0; q < G; ++q) key[q] = lane + 32 * q < n ? (L.e[lane + 32 * q].info & 15) : 15;
    int base = 0;
#pragma unroll 1
    for (int b = 0; b <= EDGE; ++b) {
#pragma unroll
        for (int q = 0; q < G; ++q) {
            const unsigned m = __ballot_sync(0xffffffffu, key[q] == b);
            if (key[q] == b) L.order[base + __popc(m & ((1u << lane) - 1u))] = (unsigned char)(lane + 32 * q);
            base += __popc(m);
        }
        if (lane == 0) L.end[b] = (unsigned char)base;
    }
    __syncwarp();
    float A[ZP], B[ZP];
#pragma unroll
    for (int q = 0; q < ZP; ++q) B[q] = 0.f;
    int p = 0;
#pragma unroll 1
    for (int b = 0; b <= EDGE; ++b) {  // the columns between voxels b - 1 and b
#pragma unroll
        for (int q = 0; q < ZP; ++q) {
            A[q] = B[q];
            B[q] = 0.f;
        }
        const int end = L.end[b];
#pragma unroll 1
        for (; p < end; ++p) k2_add<ZP, MASKED>(&L.e[L.order[p]], nv, A, B);
        if (b > 0) {
            float C[ZP];
            __syncwarp();
            tm_wait_st();
            tm_ld<ZP>(strip + (b - 1) * ZP, C);
            tm_wait_ld();
#pragma unroll
            for (int q = 0; q < ZP; ++q) C[q] += A[q];
            tm_st<ZP>(strip + (b - 1) * ZP, C);
        }
    }
    __syncwarp();
}

// One warp's strip: the profiles of family fam from all batch slots.
template <int EDGE, int ZP, bool MASKED>
__device__ __forceinline__ void k2_strip(const BpArgs &a, int fam, int m, int bs, int kb, K2List &L,
                                         unsigned strip) {
    const DevGeom &g = a.g;
    const int lane = threadIdx.x & 31;
    const int Na = fam ? g.ny : g.nx, Nb = fam ? g.nx : g.ny;
    if (m >= Na || bs >= Nb) return;
    const int be = min(bs + EDGE - 1, Nb - 1);
    const float xa = ((float)(fam ? bs : m) - g.cx) * g.vx, xb = ((float)(fam ? be : m) - g.cx) * g.vx;
    const float ya = ((float)(fam ? m : bs) - g.cy) * g.vy, yb = ((float)(fam ? m : be) - g.cy) * g.vy;
    // the strip, a little longer at either end: a view whose rays to both ends
    // are dominated by the other family's axis, on the same side of the source,
    // has no column of this family here (that cone is convex)
    const float ex = fam ? 1.1f * g.vx : 0.f, ey = fam ? 0.f : 1.1f * g.vy, eps = 1e-4f * g.sod;
    int n = 0;
#pragma unroll 1
    for (int s0 = 0; s0 < a.n_sel; s0 += 32) {
        // lane l looks at view s0 + l: its columns within hwu of the projections of
        // the strip's end voxels (the projection is monotone along the strip; an
        // estimate, the window keeps a slack of 2 % + 0.05 columns)
        const int sv = min(s0 + lane, a.n_sel - 1);
        const int v = a.views[sv];
        const float2 cs = __ldg(&g.trig[v]);
        const float ua = (ya * cs.x - xa * cs.y) * __fdividef(g.sdd, g.sod - (xa * cs.x + ya * cs.y)) * g.inv_du + g.cu;
        const float ub = (yb * cs.x - xb * cs.y) * __fdividef(g.sdd, g.sod - (xb * cs.x + yb * cs.y)) * g.inv_du + g.cu;
        const int lo = max(0, (int)ceilf(fminf(ua, ub) - g.hwu));
        const int hi = min(g.nu - 1, (int)floorf(fmaxf(ua, ub) + g.hwu));
        const float dxa = xa - ex - g.sod * cs.x, dxb = xb + ex - g.sod * cs.x;
        const float dya = ya - ey - g.sod * cs.y, dyb = yb + ey - g.sod * cs.y;
        const float pa = fam ? dxa : dya, pb = fam ? dxb : dyb;  // along the other family's axis
        const float oa = fabsf(fam ? dya : dxa) + eps, ob = fabsf(fam ? dyb : dxb) + eps;
        const bool other = (pa > oa && pb > ob) || (-pa > oa && -pb > ob);
        unsigned todo = __ballot_sync(0xffffffffu, s0 + lane < a.n_sel && lo <= hi && !other);
        while (todo) {  // two views at a time, half a warp each
            const int v0 = __ffs(todo) - 1;
            todo &= todo - 1;
            const int v1 = todo ? __ffs(todo) - 1 : -1;
            todo &= todo - 1;
            const int src = lane < 16 ? v0 : v1;
            const int vv = __shfl_sync(0xffffffffu, v, src & 31), l = __shfl_sync(0xffffffffu, lo, src & 31);
            const int hs = __shfl_sync(0xffffffffu, hi, src & 31), h = src < 0 ? -1 : hs;  // (l >= 0)
            const int rounds = __reduce_max_sync(0xffffffffu, (h - l + 16) >> 4);
#pragma unroll 1
            for (int r = 0; r < rounds; ++r) {
                const int iu = l + (lane & 15) + 16 * r;
                K2Entry e;
                const bool on = iu <= h && k2_entry<MASKED>(a, fam, m, bs, EDGE, kb, 32 * ZP, s0 + src, vv, iu, e);
                const unsigned mask = __ballot_sync(0xffffffffu, on);
                if (on) L.e[n + __popc(mask & ((1u << lane) - 1u))] = e;
                __syncwarp();
                n += __popc(mask);
                if (n > K2_CAP - 32) {
                    k2_sum<EDGE, ZP, MASKED>(L, n, g.nv, strip);
                    n = 0;
                }
            }
        }
    }
    if (n > 0) k2_sum<EDGE, ZP, MASKED>(L, n, g.nv, strip);
}

// One block's patch: voxel columns [EDGE bx, ..) x [EDGE by, ..), z-span bz;
// the block's sum of squared gradient values goes to *g2_partial (if not
// NULL).  The y-planes' strips are summed into gzi first, then the x-planes' are
// added and the sum scaled (the patch stays in L2 between).  Warp w takes the
// planes w, w + WARPS, ..; sm.tmem holds tm_cols columns.  Called by every
// thread.
template <int WARPS>
struct K2Smem {
    K2List lists[WARPS];
    unsigned tmem;
    float g2[STRIP_EDGE];  // a block of fewer warps than planes: each plane's sum of squares
};
template <int EDGE, int ZP, int WARPS, bool MASKED = false>
__device__ __forceinline__ void k2_tile(const BpArgs &a, K2Smem<WARPS> &sm, int bx, int by, int bz, double *g2_partial) {
    const DevGeom &g = a.g;
    const int lane = threadIdx.x & 31, w0 = threadIdx.x >> 5;
    const int i0 = bx * EDGE, j0 = by * EDGE, kb = bz * 32 * ZP;
    const unsigned strip = sm.tmem + ((unsigned)(w0 & 3) << 21) + (w0 >> 2) * EDGE * ZP;
    float g2 = 0.f;
#pragma unroll 1
    for (int fam = 1; fam >= 0; --fam) {
#pragma unroll 1
        for (int w = w0; w < EDGE; w += WARPS) {
            float C[ZP];
#pragma unroll
            for (int q = 0; q < ZP; ++q) C[q] = 0.f;
            __syncwarp();
#pragma unroll 1
            for (int b = 0; b < EDGE; ++b) tm_st<ZP>(strip + b * ZP, C);
            k2_strip<EDGE, ZP, MASKED>(a, fam, (fam ? j0 : i0) + w, fam ? i0 : j0, kb, sm.lists[w0], strip);
            if (!fam && w == w0) __syncthreads();  // every y-plane's sums are in gzi
            __syncwarp();
            tm_wait_st();
#pragma unroll 1
            for (int b = 0; b < EDGE; ++b) {
                const int i = i0 + (fam ? b : w), j = j0 + (fam ? w : b);
                __syncwarp();
                tm_ld<ZP>(strip + b * ZP, C);
                tm_wait_ld();
                if (i >= g.nx || j >= g.ny) continue;
                float *out = a.gzi + ((size_t)j * g.nx + i) * g.nz;
#pragma unroll
                for (int q = 0; q < ZP; ++q) {
                    const int k = kb + lane + 32 * q;
                    if (k < g.nz) {
                        float val = fam && !a.more ? C[q] : out[k] + C[q];
                        if (!fam && a.last) {
                            val *= a.scale;
                            g2 = fmaf(val, val, g2);
                        }
                        out[k] = val;
                    }
                }
            }
            if (WARPS < EDGE && !fam) {
                g2 = warp_sum_f32(g2);
                if (lane == 0) sm.g2[w] = g2;
                g2 = 0.f;
            }
        }
    }
    if (WARPS < EDGE) {
        // the planes' sums in the order that a block of one plane per warp adds them in,
        // so that a batch reports the single-volume solver's ||g||^2
        __syncthreads();
        if (g2_partial && threadIdx.x == 0) {
            double o = 0.0;
#pragma unroll 1
            for (int w = 0; w < EDGE; ++w) o += (double)sm.g2[w];
            *g2_partial = o;
        }
    } else if (g2_partial) {
        float vv[1] = {g2};
        double o[1];
        block_sum_f64<32 * WARPS, 1>(vv, o);
        if (threadIdx.x == 0) *g2_partial = o[0];
    }
}

// The patch with infinities or NaN among the residuals: a call of its own, so that
// the usual path keeps its registers (the mask as a flag inside it: 406 -> 431 us for
// 20 views at 256^3).
template <int ZP>
__device__ __noinline__ void k2_tile_masked(const BpArgs &a, K2Smem<STRIP_EDGE> &sm) {
    k2_tile<STRIP_EDGE, ZP, STRIP_EDGE, true>(a, sm, blockIdx.x, blockIdx.y, blockIdx.z, nullptr);
}

// At most 64 registers (4 blocks per SM, 32 warps): 4.79 against 4.84 ms per
// 40-view launch at 512^3 with 80 registers and 3 blocks, 1.14 against 1.20 ms at
// 384^3 with 6 voxels per lane; the few spilled values lie outside the inner loops.
template <int ZP>
__global__ void __launch_bounds__(32 * STRIP_EDGE, 4) k2_strips(const __grid_constant__ BpArgs a) {
    const size_t blk = ((size_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
    __shared__ K2Smem<STRIP_EDGE> sm;
    constexpr int cols = tm_cols(STRIP_EDGE, STRIP_EDGE, ZP);
    if (threadIdx.x < 32) tm_alloc(&sm.tmem, cols);
    __syncthreads();
    if (a.nonfinite && __ldcg(a.nonfinite)) k2_tile_masked<ZP>(a, sm);
    else
        k2_tile<STRIP_EDGE, ZP, STRIP_EDGE>(a, sm, blockIdx.x, blockIdx.y, blockIdx.z,
                                            a.g2_partials ? a.g2_partials + blk : nullptr);
    __syncthreads();
    if (threadIdx.x < 32) tm_free(sm.tmem, cols);
}

// Views a launch takes at most: 512 MiB of residual rows.  The blocks of a launch
// walk its views in order but drift apart; over 1.7 GB of rows (720 views at 512^3)
// the re-reads from DRAM cost more than adding into the gradient again (107 ms in one
// launch, 91 in four), up to 0.5 GB they do not (720 views at 256^3: 12.3 ms in one
// launch, 13.4 in five; 200 at 512^3: 24.7 and 24.8).
constexpr size_t STRIP_BYTES = size_t(512) << 20;
__host__ __device__ __forceinline__ int strip_parts(const DevGeom &g, int n_sel) {
    const size_t bytes = (size_t)n_sel * g.nu * rt_pitch(g.nv) * sizeof(float);
    const size_t parts = (bytes + STRIP_BYTES - 1) / STRIP_BYTES;
    return (int)(parts < (size_t)n_sel ? parts : (size_t)n_sel);
}
// The rows and views of part p of n_sel (g apart from a: a block's copy of it is still
// being staged when its first part is set).
__host__ __device__ __forceinline__ void strip_part(BpArgs &a, const DevGeom &g, const float *rt, const int32_t *views,
                                                    int n_sel, int p, int parts) {
    const int s0 = (int)((int64_t)n_sel * p / parts), s1 = (int)((int64_t)n_sel * (p + 1) / parts);
    a.rt = rt + (size_t)s0 * g.nu * rt_pitch(g.nv);
    a.views = views + s0;
    a.n_sel = s1 - s0;
    a.more = p > 0;
    a.last = p + 1 == parts;
}

// Persistent batched strips: the patches of the volumes that run in strips (the
// first `total` tiles of the phase), taken from an atomic counter.  Each volume
// keeps its own voxels per lane (a block-uniform switch) and the parts that its
// views run in (launch_strips), so its sums are those of its single-volume
// launches; a block is 4 warps, which take two planes each.
constexpr int KBS_WARPS = 4, KBS_BLOCKS = 5;
static_assert(KBS_BLOCKS * tm_cols(KBS_WARPS, STRIP_EDGE, 8) <= 512, "tensor memory of an SM");
__global__ void __launch_bounds__(32 * KBS_WARPS, KBS_BLOCKS) kb_strips(const BatchHdr *hdr, const BatchVol *vols, int *ctr) {
    __shared__ int s_tile;
    __shared__ BpArgs sa;
    __shared__ K2Smem<KBS_WARPS> sm;
    constexpr int cols = tm_cols(KBS_WARPS, STRIP_EDGE, 8);
    const int tid = threadIdx.x;
    const int total = hdr->strip_tiles;
    if (tid < 32) tm_alloc(&sm.tmem, cols);
    for (;;) {
        if (tid == 0) s_tile = atomicAdd(ctr, 1);
        __syncthreads();
        const int t = s_tile;
        __syncthreads();
        if (t >= total) break;
        const int vi = batch_find(*hdr, vols, 1, t);
        const BatchVol &bv = vols[vi];
        // the volume's arguments, staged in shared memory for the whole block
        stage_words(&sa.g, &bv.g, sizeof(DevGeom), tid, 32 * KBS_WARPS);
        if (tid == 0) {
            sa.scale = bv.scale;
            sa.gzi = bv.grad;
            sa.g2_partials = bv.partials;
            sa.nonfinite = nullptr;  // (a solver's step fails where a residual is not finite)
        }
        const BpArgs &a = sa;
        const int local = t - bv.first[1];
        const int gx = (bv.g.nx + STRIP_EDGE - 1) / STRIP_EDGE, gy = (bv.g.ny + STRIP_EDGE - 1) / STRIP_EDGE;
        const int bx = local % gx, rest = local / gx, by = rest % gy, bz = rest / gy;
        const int parts = strip_parts(bv.g, bv.N_t);
#pragma unroll 1
        for (int p = 0; p < parts; ++p) {
            if (p > 0) __syncthreads();  // the last part's arguments and sums
            if (tid == 0) strip_part(sa, bv.g, bv.rt, bv.views, bv.N_t, p, parts);
            __syncthreads();
            double *part = a.last ? bv.partials + local : nullptr;
            switch (strip_zp(bv.g.k2_vpl, bv.g.nz)) {
                case 4: k2_tile<STRIP_EDGE, 4, KBS_WARPS>(a, sm, bx, by, bz, part); break;
                case 6: k2_tile<STRIP_EDGE, 6, KBS_WARPS>(a, sm, bx, by, bz, part); break;
                default: k2_tile<STRIP_EDGE, 8, KBS_WARPS>(a, sm, bx, by, bz, part); break;
            }
        }
    }
    __syncthreads();
    if (tid < 32) tm_free(sm.tmem, cols);
    batch_leave(ctr);
}

}  // namespace

// As many blocks per SM as the launch bound admits (registers, shared memory and
// 64 of the 512 tensor-memory columns each).  The occupancy query is no guide: it
// answers 1 for a kernel that allocates tensor memory, and one block per SM took
// 51.6 ms per iteration of 16 volumes of 96^3 .. 320^3 (learned steps), three
// 30.5, five 26.5.  No block waits for another, so fewer resident ones are safe.
cudaError_t launch_batch_strips(const BatchHdr *hdr, BatchVol *vols, int *ctr, cudaStream_t st) {
    static const int grid = [] {
        int dev = 0, sms = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        return (sms > 0 ? sms : 1) * KBS_BLOCKS;
    }();
    kb_strips<<<grid, 32 * KBS_WARPS, 0, st>>>(hdr, vols, ctr);
    return cudaGetLastError();
}

cudaError_t launch_strips(const BpArgs &a, dim3 grid, int zp, cudaStream_t st) {
    auto k = zp == 4 ? k2_strips<4> : zp == 6 ? k2_strips<6> : k2_strips<8>;
    const int parts = strip_parts(a.g, a.n_sel);
    for (int p = 0; p < parts; ++p) {
        BpArgs b = a;
        strip_part(b, a.g, a.rt, a.views, a.n_sel, p, parts);
        if (!b.last) b.g2_partials = nullptr;
        k<<<grid, 32 * STRIP_EDGE, 0, st>>>(b);
    }
    return cudaGetLastError();
}

}  // namespace fbl

// K4: harmonic sums and the thresholded peak list (Sec. 2.1: a pulsar shows as peaks at
// integer multiples of f and fdot, and the summed power of the harmonics is the detection
// statistic).
//
// For level H (1, 2, 4, 8, 16): S_H(r, i) = sum_{h=1..H} P(h r, i_h), z_{i_h} = h z_i,
// summed in FP32 in the order h = 1..H (BF16 planes are widened by placing the 16 stored
// bits in the top half of a float, the paper's quick cast of Sec. 3.1), defined where
// |H z_i| <= zmax and H r < Nb.  Peak: S_H > thr and a 3x3 local maximum (strictly above
// earlier neighbours in row-major (i, r) order, >= later ones, undefined neighbours ignored).
//
// The defined regions nest (level 2H's lies inside level H's), so one pass builds every level:
// a warp owns one (row i, chunk of CB = 512 bins) of the plane and the running sums S_H of its
// bins stay in registers; S_2H = S_H + sum_{h = H+1 .. 2H} P(h r, i_h) adds the new harmonics in
// order, so every S_H is bit-identical to the direct sum.  Level 1 (a stream over the whole plane,
// or over the units the plane kernel marked) gives lane l the 16 consecutive bins r0 + 16 l ..
// r0 + 16 l + 15, read as 16-byte vectors.  Levels 2 .. 16 interleave instead -- lane l holds
// r0 + l + 32 e, e < 16 -- so that one warp-wide load of harmonic h reads 32 elements h apart,
// a span of whole sectors, where consecutive bins per lane would touch 32 sectors per load.  A
// lane tests its 16 values against the threshold through their maximum; only cells above it (a
// handful per plane, thousands with low thresholds) recompute their 3x3 neighbourhood's sums to
// decide the peak.  Level 1, whose sums are plane values, decides its own (level1_many), and on BF16
// planes so do the plain sums' levels (IN_PLACE: what each way costs); the others leave the mask of such
// cells to k4_verify, nine lanes of a warp to a cell or, where they are many, a lane to a bin.
//
// Output order (H, i, r): a "unit" is (level, row, chunk of CB bins), units are numbered in
// that order, and
//   pass A (k4_level1 over the plane, k4_levels over level 2's region, then k4_verify where cells
//     were left to it) writes each unit's peak count and CB-bit mask, and lists the units (in no
//     order) that hold peaks, or whose cells were left to k4_verify;
//   pass B (k4_emit_listed): when the list holds all of them (PEAK_LIST_CAP; the usual case) each
//     listed unit goes to a warp, which sums the counts of the units before it and writes its
//     records; otherwise every unit's count is scanned in order.  Either way a record's power is
//     S_H recomputed at its cell, at offset + rank.
// Listed calls with thousands of peaks (FP32 plane, N = 2^21, 85 templates, low thresholds, some 3000
// units): 243-260 us with each lane testing its own cells and one block writing all records, 134 now.
#include <algorithm>
#include <cmath>
#include <vector>

#include "fdas_internal.cuh"

namespace fdas {

namespace {

constexpr int CB = PEAK_CHUNK;           // bins per unit (a warp's chunk)
constexpr int LB = CB / 32;              // bins per lane (16)
constexpr int WORDS = CB / 32;           // mask words per unit
constexpr int DETECT_WARPS = 4;          // warps per k4_level1 / k4_levels block
#ifndef FDAS_K4_CPW
#define FDAS_K4_CPW 1                    // chunks per k4_levels warp
#endif
constexpr int CPW = FDAS_K4_CPW;
static_assert((CPW & (CPW - 1)) == 0 && CPW <= 2, "chunks per warp: 1 or 2 (chunks1 >= 2 is a power of two)");
#ifndef FDAS_K4_L1_MIN_BLOCKS
#define FDAS_K4_L1_MIN_BLOCKS 8          // resident k4_level1 blocks per SM the registers must allow
#endif
#ifndef FDAS_K4_RAY_BF16
#define FDAS_K4_RAY_BF16 1               // 1: the BF16 plane's levels in ray order too (the FP32 plane's always are)
#endif
#ifndef FDAS_K4_MIN_BLOCKS
#define FDAS_K4_MIN_BLOCKS 4             // resident k4_levels blocks per SM the registers must allow
#endif

static_assert(LB == 16, "a lane owns 16 bins: two BF16 or four FP32 16-byte vectors");

__device__ __forceinline__ float ld_plane(const float *p, int64_t i) { return __ldg(p + i); }
__device__ __forceinline__ float ld_plane(const __nv_bfloat16 *p, int64_t i) {
    const unsigned short bits = __ldg(reinterpret_cast<const unsigned short *>(p) + i);
    return __uint_as_float(((unsigned)bits) << 16);
}

// Plane element formats: elements per 16-byte vector, widening of one vector, and the maximum of
// a lane's 16 values (BF16 compares packed pairs; widening is exact, so the order is the same).
template <typename E>
struct Fmt;
template <>
struct Fmt<float> {
    static constexpr int EPV = 4;
    struct Raw {
        float4 v[LB / 4];
    };
    __device__ __forceinline__ static void load_raw(const float *p, Raw &r) {
#pragma unroll
        for (int k = 0; k < LB / 4; k++) r.v[k] = __ldg(reinterpret_cast<const float4 *>(p) + k);
    }
    __device__ __forceinline__ static void widen(const Raw &r, float (&s)[LB]) {
#pragma unroll
        for (int k = 0; k < LB / 4; k++) {
            s[4 * k] = r.v[k].x; s[4 * k + 1] = r.v[k].y; s[4 * k + 2] = r.v[k].z; s[4 * k + 3] = r.v[k].w;
        }
    }
    __device__ __forceinline__ static float max16(const Raw &r) {
        float m = -INFINITY;
#pragma unroll
        for (int k = 0; k < LB / 4; k++) m = fmaxf(fmaxf(m, fmaxf(r.v[k].x, r.v[k].y)), fmaxf(r.v[k].z, r.v[k].w));
        return m;
    }
};
template <>
struct Fmt<__nv_bfloat16> {
    static constexpr int EPV = 8;
    struct Raw {
        uint4 v[LB / 8];
    };
    __device__ __forceinline__ static void load_raw(const __nv_bfloat16 *p, Raw &r) {
#pragma unroll
        for (int k = 0; k < LB / 8; k++) r.v[k] = __ldg(reinterpret_cast<const uint4 *>(p) + k);
    }
    __device__ __forceinline__ static void widen(const Raw &r, float (&s)[LB]) {
        const uint32_t w[8] = {r.v[0].x, r.v[0].y, r.v[0].z, r.v[0].w, r.v[1].x, r.v[1].y, r.v[1].z, r.v[1].w};
#pragma unroll
        for (int k = 0; k < 8; k++) {
            s[2 * k] = __uint_as_float(w[k] << 16);
            s[2 * k + 1] = __uint_as_float(w[k] & 0xFFFF0000u);
        }
    }
    // packed BF16 maximum (exact: widening preserves the order)
    __device__ __forceinline__ static float max16(const Raw &r) {
        const uint32_t w[8] = {r.v[0].x, r.v[0].y, r.v[0].z, r.v[0].w, r.v[1].x, r.v[1].y, r.v[1].z, r.v[1].w};
        __nv_bfloat162 m = *reinterpret_cast<const __nv_bfloat162 *>(&w[0]);
#pragma unroll
        for (int k = 1; k < 8; k++) m = __hmax2(m, *reinterpret_cast<const __nv_bfloat162 *>(&w[k]));
        return fmaxf(__low2float(m), __high2float(m));
    }
};

template <typename E>
__device__ __forceinline__ float harm_sum(const E *plane, int64_t nb, int zmax, int H, int i, int64_t r) {
    const int z = -zmax + 2 * i;
    float s = 0.0f;
    float v[16];                                         // all the gathers in flight together
#pragma unroll
    for (int h = 1; h <= 16; h++)
        if (h <= H) v[h - 1] = ld_plane(plane, (int64_t)((h * z + zmax) >> 1) * nb + (int64_t)h * r);
#pragma unroll
    for (int h = 1; h <= 16; h++)
        if (h <= H) s = __fadd_rn(s, v[h - 1]);
    return s;
}

// Highest-harmonic-anchored sum with rounding (harm_mode 1): the cell (r, i) is harmonic H; the
// harmonic j of level L sits at r_j = floor((2 j r + L) / (2 L)) (j r / L rounded, halves up) and
// row floor((j z + L zmax + L) / (2 L)) (the grid row nearest j z / L, halves up).  Level 2L's
// even fractions are level L's with the same rounding, so S_2L = S_L + the odd j < 2L in
// increasing j, S_1 = P; FP32 adds in that order.
template <typename E>
__device__ float harm_sum_anch(const E *plane, int64_t nb, int zmax, int H, int i, int64_t r) {
    const int z = -zmax + 2 * i;
    float s = ld_plane(plane, (int64_t)i * nb + r);
#pragma unroll
    for (int l = 1; l <= 4; l++) {                       // a level's loads (at most 8) in flight together
        const int L = 1 << l;
        if (L > H) break;
        float v[8];
#pragma unroll
        for (int j = 1; j < L; j += 2) {
            const int ij = (j * z + L * zmax + L) >> (l + 1);
            v[j >> 1] = ld_plane(plane, (int64_t)ij * nb + ((2 * (int64_t)j * r + L) >> (l + 1)));
        }
#pragma unroll
        for (int j = 1; j < L; j += 2) s = __fadd_rn(s, v[j >> 1]);
    }
    return s;
}

__device__ __forceinline__ bool row_in_level(int i, int K, int zmax, int H) {
    const int z = -zmax + 2 * i;
    return i >= 0 && i < K && abs(H * z) <= zmax;
}

// Levels 2 .. 16 interleave the bins: lane l of a warp owns bins r0 + l + 32 e (e < 16) of its
// 512-bin chunk, so one load of harmonic h for the whole warp reads the 32 elements h (r0 + l +
// 32 e), l < 32 -- a span of 32 h elements, whole sectors -- instead of 32 lanes each touching
// their own sectors.  s[e] += P(h r, i_h) for the lane's bins r = rb + 32 e with r <= rmax (then
// h r <= H rmax < Nb); the sums keep the order h = 1..H.
// S_H from S_{H/2}: the new harmonics h = H/2 + 1 .. H in order, the loads of FDAS_K4_HBATCH
// harmonics in flight together (16 per harmonic and lane; the adds keep the order h = 1..H).
#ifndef FDAS_K4_HBATCH
#define FDAS_K4_HBATCH 1                 // 2 measured 0.210 ms against 0.180 ms for 1 (BF16, N = 2^23)
#endif
template <typename E, int H>
__device__ __forceinline__ void add_level(const E *__restrict__ plane, int64_t nb, int zmax, int z, int64_t rb,
                                          int64_t rmax, float (&s)[LB]) {
    constexpr int NB = FDAS_K4_HBATCH < H / 2 ? FDAS_K4_HBATCH : H / 2;
#pragma unroll
    for (int q0 = 0; q0 < H / 2; q0 += NB) {
        float v[NB][LB];
#pragma unroll
        for (int q = 0; q < NB; q++) {
            const int h = H / 2 + 1 + q0 + q;
            const E *row = plane + (int64_t)((h * z + zmax) >> 1) * nb;
#pragma unroll
            for (int e = 0; e < LB; e++) {
                const int64_t r = rb + 32 * e;
                v[q][e] = r <= rmax ? ld_plane(row, (int64_t)h * r) : 0.0f;
            }
        }
#pragma unroll
        for (int q = 0; q < NB; q++)
#pragma unroll
            for (int e = 0; e < LB; e++) s[e] = __fadd_rn(s[e], v[q][e]);
        // bound the loads in flight (the registers of levels 8, 16)
        asm volatile("" ::: "memory");
    }
}

// harm_sum with U gathers in flight.
template <typename E, int U = 2>
__device__ __forceinline__ float harm_sum_inorder(const E *plane, int64_t nb, int zmax, int H, int i, int64_t r) {
    const int z = -zmax + 2 * i;
    float s = 0.0f;
#pragma unroll U
    for (int h = 1; h <= H; h++)
        s = __fadd_rn(s, ld_plane(plane, (int64_t)((h * z + zmax) >> 1) * nb + (int64_t)h * r));
    return s;
}

// The 3x3 rule for a cell of level H holding S_H = v, by one lane inside the level search: strictly
// above the defined neighbours that come earlier in row-major (i, r) order, at least equal to the
// later ones.  The registers it asks for are the caller's loss: with its sums' gathers unrolled by
// the compiler's choice the search spilled, and N = 2^23, BF16, took 207 us instead of 191 (all 16 in
// flight: 275).
template <typename E>
__device__ __noinline__ bool local_max(const E *plane, int64_t nb, int zmax, int K, int H, int64_t rmax, int i, int64_t r, float v) {
    for (int di = -1; di <= 1; di++) {
        const int ii = i + di;
        if (!row_in_level(ii, K, zmax, H)) continue;
        for (int dr = -1; dr <= 1; dr++) {
            if (di == 0 && dr == 0) continue;
            const int64_t rr = r + dr;
            if (rr < 0 || rr > rmax) continue;
            const float w = harm_sum_inorder(plane, nb, zmax, H, ii, rr);
            const bool earlier = di < 0 || (di == 0 && dr < 0);
            if (earlier ? !(v > w) : !(v >= w)) return false;
        }
    }
    return true;
}

// The unit list of the step: PEAK_LIST_WORDS words directly before the counts (word 0 the number of
// units listed, words 4 .. the first PEAK_LIST_CAP unit numbers, in no order).
__device__ __forceinline__ unsigned int *unit_list(int32_t *unit_count) {
    return reinterpret_cast<unsigned int *>(unit_count) - PEAK_LIST_WORDS;
}
__device__ __forceinline__ const unsigned int *unit_list(const int32_t *unit_count) {
    return reinterpret_cast<const unsigned int *>(unit_count) - PEAK_LIST_WORDS;
}
// The unit on the list (one thread per unit; out of line, a handful of times per plane, so that it
// costs the callers no registers).
__device__ __noinline__ void list_unit(int32_t *unit_count, int64_t u) {
    unsigned int *list = unit_list(unit_count);
    const unsigned int slot = atomicAdd(list, 1u);
    if (slot < (unsigned int)PEAK_LIST_CAP) list[4 + slot] = (unsigned int)u;
}

// A unit's count, and the unit on the list when it holds peaks (one thread per unit).
__device__ __forceinline__ void count_unit(int32_t *__restrict__ unit_count, int64_t u, int cnt) {
    unit_count[u] = cnt;
    if (cnt > 0) list_unit(unit_count, u);
}

// Whether the plain sums' level search (k4_levels*) tests its cells in place instead of leaving them to
// k4_verify.  N = 2^23, 85 templates, the whole region: BF16 planes 191 us in place, 253 us leaving
// them; FP32 planes 229 us in place, 209 us leaving them (the compiler schedules the kernels' loads
// differently).  FP32, N = 2^21 with low thresholds, thousands of cells to test: 130 us in place, 63 us.
template <typename E>
constexpr bool IN_PLACE = sizeof(E) == 2;

// What the level kernels leave of one unit u to be tested: a zero count, or, when a cell is above the
// threshold, the mask of those cells, the unit on the list and a count of -1.  word: lane w < 16 holds
// word w of the mask, bins 32 w .. 32 w + 31.
__device__ __forceinline__ void leave_unit(uint32_t word, int u, int32_t *__restrict__ unit_count,
                                           uint32_t *__restrict__ unit_mask) {
    const int lane = threadIdx.x & 31;
    if (lane < WORDS) unit_mask[(int64_t)u * WORDS + lane] = word;
    if (lane == 0) {
        unit_count[u] = -1;
        list_unit(unit_count, u);
    }
}

// The same from a warp's sums: s[e] of bin lane + 32 e, bins defined up to rest.
__device__ __forceinline__ void leave_sums(const float (&s)[LB], float thr, int rest, int u, int32_t *__restrict__ unit_count,
                                           uint32_t *__restrict__ unit_mask) {
    const int lane = threadIdx.x & 31;
    float vmax = -INFINITY;
#pragma unroll
    for (int e = 0; e < LB; e++)
        if (lane + 32 * e <= rest) vmax = fmaxf(vmax, s[e]);
    if (__any_sync(0xffffffffu, vmax > thr)) {
        uint32_t word = 0;
#pragma unroll
        for (int e = 0; e < LB; e++) {
            const uint32_t b = __ballot_sync(0xffffffffu, lane + 32 * e <= rest && s[e] > thr);
            if (lane == e) word = b;
        }
        leave_unit(word, u, unit_count, unit_mask);
    } else if (lane == 0) {
        unit_count[u] = 0;
    }
}

// One level H > 1 of one (row, chunk), lane bins rb + 32 e: S_H from S_{H/2}, then the unit's peaks or
// its cells above the threshold (word e of the mask, bins 32 e .. 32 e + 31 of the chunk, is the
// warp's ballot of bit e).  Returns false when the chunk lies outside level H's region (the regions
// nest: stop there).
template <typename E, int H, bool ADD = true>
__device__ __forceinline__ bool level_step(const E *__restrict__ plane, int64_t nb, int zmax, int K,
                                           const LevelDesc &d, int i, int z, int chunk, int64_t rb, float (&s)[LB],
                                           int32_t *__restrict__ unit_count, uint32_t *__restrict__ unit_mask) {
    if (!row_in_level(i, K, zmax, H) || (int64_t)chunk * CB > d.rmax) return false;   // warp-uniform
    if (ADD) add_level<E, H>(plane, nb, zmax, z, rb, d.rmax, s);
    // unit indices fit 32 bits (at most 1023 rows x 2^17 chunks per level, five levels)
    const int u = (int)d.unit0 + (i - d.i_lo) * (int)d.chunks + chunk;
    if constexpr (IN_PLACE<E>) {
        const int lane = threadIdx.x & 31;
        float vmax = -INFINITY;
#pragma unroll
        for (int e = 0; e < LB; e++)
            if (rb + 32 * e <= d.rmax) vmax = fmaxf(vmax, s[e]);
        if (__any_sync(0xffffffffu, vmax > d.thr)) {
            uint32_t pk = 0;
            if (vmax > d.thr) {
#pragma unroll
                for (int e = 0; e < LB; e++) {
                    const int64_t r = rb + 32 * e;
                    if (r <= d.rmax && s[e] > d.thr && local_max(plane, nb, zmax, K, H, d.rmax, i, r, s[e])) pk |= 1u << e;
                }
            }
            int cnt = __popc(pk);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
            if (lane == 0) count_unit(unit_count, u, cnt);
            if (cnt > 0) {
                uint32_t word = 0;
#pragma unroll
                for (int e = 0; e < LB; e++) {
                    const uint32_t b = __ballot_sync(0xffffffffu, (pk >> e) & 1u);
                    if (lane == e) word = b;
                }
                if (lane < WORDS) unit_mask[(int64_t)u * WORDS + lane] = word;
            }
        } else if (lane == 0) {
            unit_count[u] = 0;
        }
    } else {
        leave_sums(s, d.thr, (int)min(d.rmax - (int64_t)chunk * CB, (int64_t)CB), u, unit_count, unit_mask);
    }
    return true;
}

// Levels 4, 8 and 16 (under 10 % of the cells): out of line, so that their gathers do not set
// the register budget of the common path (level 2).
template <typename E>
__device__ __noinline__ void high_levels(const E *__restrict__ plane, int64_t nb, int zmax, int K,
                                         const LevelTable *lt, int i, int z, int chunk, int64_t rb,
                                         const float *s_in, int32_t *__restrict__ unit_count,
                                         uint32_t *__restrict__ unit_mask) {
    float s[LB];
#pragma unroll
    for (int e = 0; e < LB; e++) s[e] = s_in[e];
    const int n = lt->n_levels;
    if (!level_step<E, 4>(plane, nb, zmax, K, lt->lev[2], i, z, chunk, rb, s, unit_count, unit_mask)) return;
    if (n < 4 || !level_step<E, 8>(plane, nb, zmax, K, lt->lev[3], i, z, chunk, rb, s, unit_count, unit_mask))
        return;
    if (n > 4) level_step<E, 16>(plane, nb, zmax, K, lt->lev[4], i, z, chunk, rb, s, unit_count, unit_mask);
}

// Levels 2 .. of one (row, chunk) inside level 2's region; s holds S_2 of the lane's bins on entry
// (the caller reads S_1 and the second harmonic together).
template <typename E>
__device__ __forceinline__ void detect_chunk(const E *__restrict__ plane, int64_t nb, int zmax, int K,
                                             const LevelTable &lt, int i, int z, int chunk, int64_t rb,
                                             float (&s)[LB], int32_t *__restrict__ unit_count,
                                             uint32_t *__restrict__ unit_mask) {
    if (!level_step<E, 2, false>(plane, nb, zmax, K, lt.lev[1], i, z, chunk, rb, s, unit_count, unit_mask)) return;
    if (lt.n_levels > 2 && row_in_level(i, K, zmax, 4) && (int64_t)chunk * CB <= lt.lev[2].rmax) {
        float t[LB];                                 // the out-of-line call's copy (S_2 stays in registers)
#pragma unroll
        for (int e = 0; e < LB; e++) t[e] = s[e];
        high_levels<E>(plane, nb, zmax, K, &lt, i, z, chunk, rb, t, unit_count, unit_mask);
    }
}

struct UnitRef {
    int H, row;
    int64_t chunk, rmax;
};

// Level, row and chunk of unit u (selects, not an indexed table: that would sit in local memory).
__device__ __forceinline__ UnitRef unit_of(const LevelTable &lt, int64_t u) {
    UnitRef ref;
    ref.H = 1;
    ref.rmax = lt.lev[0].rmax;
    int i_lo = lt.lev[0].i_lo;
    int64_t local = u, chunks = lt.lev[0].chunks;
#pragma unroll
    for (int k = 1; k < 5; k++)
        if (k < lt.n_levels && u >= lt.lev[k].unit0) {
            ref.H = lt.lev[k].H;
            ref.rmax = lt.lev[k].rmax;
            i_lo = lt.lev[k].i_lo;
            local = u - lt.lev[k].unit0;
            chunks = lt.lev[k].chunks;
        }
    // unit numbers and chunk counts fit 32 bits
    const uint32_t q = (uint32_t)local / (uint32_t)chunks;
    ref.row = i_lo + (int)q;
    ref.chunk = (uint32_t)local - q * (uint32_t)chunks;
    return ref;
}

// The mask of a unit's peaks (lane w < 16: word w) among its cells when they are many: a lane to a bin,
// 32 consecutive bins at a time, so that the gathers of a warp share their sectors.  Every lane's own
// sum serves its row neighbours through shuffles; then the cells still standing look at the rows
// before and after, each lane up to the first neighbour that beats its cell.
template <typename E>
__device__ __noinline__ uint32_t verify_dense(const E *__restrict__ plane, int64_t nb, int zmax, int K, bool anchored, int H,
                                              int row, int64_t r0, int64_t rmax, uint32_t cells) {
    const int lane = threadIdx.x & 31;
    uint32_t word = 0;
    for (int e = 0; e < WORDS; e++) {
        const uint32_t bits = __shfl_sync(0xffffffffu, cells, e);
        if (bits == 0) continue;                     // warp-uniform
        const int64_t r = r0 + 32 * e + lane;
        bool ok = (bits >> lane) & 1u;
        float v = 0.0f, edge = 0.0f;                 // S(row, r); lanes 0 and 31: S of the bin before and after
        // k = 0: the own sums, 1: the edges', 2 .. 7: the other rows' (one copy of the sums' code)
#pragma unroll 1
        for (int k = 0; k < 8; k++) {
            const int a = k < 2 ? 0 : k < 5 ? -1 : 1, d = k == 0 ? 0 : k == 1 ? (lane == 0 ? -1 : 1) : (k - 2) % 3 - 1;
            const int ii = row + a;
            const int64_t rr = r + d;
            const bool defined = (anchored ? (ii >= 0 && ii < K) : row_in_level(ii, K, zmax, H)) && rr >= 0 && rr <= rmax;
            const bool want = defined && (k == 0 || (ok && (k > 1 || lane == 0 || lane == 31)));
            float w = 0.0f;
            if (want) w = anchored ? harm_sum_anch(plane, nb, zmax, H, ii, rr) : harm_sum_inorder<E, 4>(plane, nb, zmax, H, ii, rr);
            if (k == 0) {
                v = w;
            } else if (k == 1) {
                edge = w;
                const float before = __shfl_up_sync(0xffffffffu, v, 1), after = __shfl_down_sync(0xffffffffu, v, 1);
                if (r > 0 && !(v > (lane == 0 ? edge : before))) ok = false;
                if (r < rmax && !(v >= (lane == 31 ? edge : after))) ok = false;
                if (!__any_sync(0xffffffffu, ok)) break;
            } else if (want) {
                ok = a < 0 ? v > w : v >= w;
            }
        }
        const uint32_t b = __ballot_sync(0xffffffffu, ok);
        if (lane == e) word = b;
    }
    return word;
}

// The peaks of one unit u among the cells its mask holds: its count and the mask of the peaks.  The
// 3x3 rule for a cell: strictly above the defined neighbours that come earlier in row-major (i, r)
// order, at least equal to the later ones.
// One warp, nine lanes to a cell, three cells at a time, each lane one of the nine sums with its
// gathers in flight together: one or two round trips to L2 per three cells.  (One lane per cell, its
// neighbours one after another, cost up to 8 H dependent round trips for each cell of a lane, and the
// cells along a strong signal were often all in one lane.)  From DENSE_CELLS cells on the
// gathers' sectors cost more than their latency: verify_dense (FP32, N = 2^23, whole call, 11 million peaks, mostly
// units of 30 to 200 cells: 6.1 ms with the line at 32, 4.8 at 128, 4.6 at 256; 54 million: 10.7, and 28.5 without
// verify_dense).
constexpr int DENSE_CELLS = 256;
template <typename E>
__device__ __forceinline__ void verify_unit(const E *__restrict__ plane, int64_t nb, int zmax, int K, bool anchored,
                                            const UnitRef &ref, int64_t u, int32_t *unit_count,
                                            uint32_t *unit_mask) {
    const int lane = threadIdx.x & 31, H = ref.H;
    const uint32_t cells = lane < WORDS ? unit_mask[u * WORDS + lane] : 0u;
    int incl = __popc(cells);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    const int total = __shfl_sync(0xffffffffu, incl, 31);
    const int g = lane / 9, q = lane - 9 * g, a = q / 3 - 1, d = q % 3 - 1;          // cell of three, neighbour
    const int ii = ref.row + a;
    const bool row_ok = anchored ? (ii >= 0 && ii < K) : row_in_level(ii, K, zmax, H);
    uint32_t word = 0;                               // lane w < 16: word w of the peaks' mask
    const int listed = total < DENSE_CELLS ? total : 0;
    if (listed < total) word = verify_dense<E>(plane, nb, zmax, K, anchored, H, ref.row, ref.chunk * CB, ref.rmax, cells);
    for (int k0 = 0; k0 < listed; k0 += 3) {         // warp-uniform
        const int k = k0 + g;                        // the group's cell: the first word with incl > k holds it
        int w = 0;
#pragma unroll
        for (int o = 8; o > 0; o >>= 1)
            if (__shfl_sync(0xffffffffu, incl, w + o - 1) <= k) w += o;
        const int last = __shfl_sync(0xffffffffu, incl, w);
        uint32_t bits = __shfl_sync(0xffffffffu, cells, w);
        const bool live = g < 3 && k < total;
        int bin = 0;
        bool ok = false;
        float sum = 0.0f;
        if (live) {
            for (int skip = k - (last - __popc(bits)); skip > 0; skip--) bits &= bits - 1;
            bin = 32 * w + __ffs(bits) - 1;
            const int64_t r = ref.chunk * CB + bin + d;
            ok = row_ok && r >= 0 && r <= ref.rmax;
            if (ok) sum = anchored ? harm_sum_anch(plane, nb, zmax, H, ii, r) : harm_sum(plane, nb, zmax, H, ii, r);
        }
        const float v = __shfl_sync(0xffffffffu, sum, (9 * g + 4) & 31);
        const uint32_t beaten = __ballot_sync(0xffffffffu, ok && q != 4 && !(q < 4 ? v > sum : v >= sum));
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const int b = __shfl_sync(0xffffffffu, bin, 9 * c + 4);
            if (k0 + c < total && !(beaten & (0x1ffu << (9 * c))) && lane == (b >> 5)) word |= 1u << (b & 31);
        }
    }
    int cnt = __popc(word);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    if (lane == 0) unit_count[u] = cnt;
    if (lane < WORDS) unit_mask[u * WORDS + lane] = word;
}

// max(a, b, c), NaN when any of them is (a cell beside a NaN is no peak); three-input max.f32: sm_100 and later.
__device__ __forceinline__ float max3_nan(float a, float b, float c) {
    float d;
    asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// The peaks of one level-1 unit u of row i, bins r0 .. r0 + 511, that holds a value above the threshold.  At
// level 1 a neighbour's sum is a plane value.  Two forms, both out of line and reading the own row again, so that
// the callers' streams keep their registers:
//  * level1_many: a lane reads its 16 bins of the three rows as vectors (one round trip for the whole unit,
//    however many cells are above) and the bins beside them come by shuffles.  FP32, N = 2^23, 85 templates, 54
//    million peaks at all levels: 18.8 -> 10.7 ms with this in place of nine lanes to a cell (below 256 cells a
//    unit) or a lane to a bin.
//  * level1_few, after a marking plane kernel: only the words of 32 bins with cells, at most LEVEL1_FEW, a lane to
//    a bin, in a short loop.  A search with a few strong cells waits longer for level1_many's unrolled code than for
//    its loads (N = 2^18, BF16, 4 pulse trains: k4_level1_marked 15.0 -> 9.4 us with cold caches, the search
//    62.8 -> 60.7).
constexpr int LEVEL1_FEW = 4;
template <typename E>
__device__ __noinline__ void level1_many(const E *__restrict__ plane, int64_t nb, int K, const LevelDesc &d, int i, int64_t r0,
                                         int u, int32_t *__restrict__ unit_count, uint32_t *__restrict__ unit_mask) {
    const int lane = threadIdx.x & 31;
    const int64_t rl = r0 + LB * lane;
    const E *own = plane + (int64_t)i * nb + rl;
    typename Fmt<E>::Raw raw[3];                         // rows i, i - 1, i + 1
    float edge[3];                                       // lane 0: the bin before the unit, lane 31: the bin after
#pragma unroll
    for (int k = 0; k < 3; k++) {
        const int a = (k == 2) - (k == 1);
        edge[k] = -INFINITY;                             // an undefined neighbour: beaten by any cell above the threshold
        if (i + a < 0 || i + a >= K) continue;
        Fmt<E>::load_raw(own + a * nb, raw[k]);
        if (lane == 0 && r0 > 0) edge[k] = ld_plane(own + a * nb, -1);
        if (lane == 31 && rl + LB <= d.rmax) edge[k] = ld_plane(own + a * nb, LB);
    }
    float v[LB];
    Fmt<E>::widen(raw[0], v);
    uint32_t pk = 0;
#pragma unroll
    for (int e = 0; e < LB; e++)
        if (v[e] > d.thr) pk |= 1u << e;
#pragma unroll
    for (int k = 0; k < 3; k++) {
        const int a = (k == 2) - (k == 1);
        if (i + a < 0 || i + a >= K) continue;           // warp-uniform
        float w[LB];
        Fmt<E>::widen(raw[k], w);
        float before = __shfl_up_sync(0xffffffffu, w[LB - 1], 1), after = __shfl_down_sync(0xffffffffu, w[0], 1);
        if (lane == 0) before = edge[k];
        if (lane == 31) after = edge[k];
#pragma unroll
        for (int e = 0; e < LB; e++) {
            const float b = e == 0 ? before : w[e == 0 ? 0 : e - 1], c = e == LB - 1 ? after : w[e == LB - 1 ? e : e + 1];
            if (k == 0 ? !(v[e] > b && v[e] >= c) : k == 1 ? !(v[e] > max3_nan(b, w[e], c)) : !(v[e] >= max3_nan(b, w[e], c)))
                pk &= ~(1u << e);
        }
    }
    int cnt = __popc(pk);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    const uint32_t hi = __shfl_down_sync(0xffffffffu, pk, 1);
    if (lane == 0) count_unit(unit_count, u, cnt);
    if (cnt > 0 && !(lane & 1)) unit_mask[(int64_t)u * WORDS + (lane >> 1)] = pk | (hi << 16);
}

template <typename E>
__device__ __noinline__ bool level1_few(const E *__restrict__ plane, int64_t nb, int K, const LevelDesc &d, int i, int64_t r0,
                                        int u, int32_t *__restrict__ unit_count, uint32_t *__restrict__ unit_mask) {
    const int lane = threadIdx.x & 31;
    uint32_t above = 0;                                  // the lane's 16 bins
    {
        typename Fmt<E>::Raw raw;
        Fmt<E>::load_raw(plane + (int64_t)i * nb + r0 + LB * lane, raw);
        float v[LB];
        Fmt<E>::widen(raw, v);
#pragma unroll
        for (int e = 0; e < LB; e++)
            if (v[e] > d.thr) above |= 1u << e;
    }
    // word w of the unit in lane w < 16
    const uint32_t cells = __shfl_sync(0xffffffffu, above, (2 * lane) & 31) | __shfl_sync(0xffffffffu, above, (2 * lane + 1) & 31) << 16;
    uint32_t live = __ballot_sync(0xffffffffu, lane < WORDS && cells != 0);
    if (__popc(live) > LEVEL1_FEW) return false;
    uint32_t word = 0;
#pragma unroll 1
    for (; live; live &= live - 1) {
        const int w = __ffs(live) - 1;
        const int64_t r = r0 + 32 * w + lane;
        const E *p = plane + (int64_t)i * nb + r;
        const int side = lane == 0 ? -1 : 1;             // lanes 0 and 31 read the bin beside the word, too
        const bool edge = (lane == 0 && r > 0) || (lane == 31 && r < d.rmax);
        float v[3], o[3];                                // rows i - 1, i, i + 1; an undefined neighbour loses
#pragma unroll
        for (int a = 0; a < 3; a++) {
            const bool row = i + a > 0 && i + a <= K;
            v[a] = row ? ld_plane(p, (a - 1) * nb) : -INFINITY;
            o[a] = row && edge ? ld_plane(p, (a - 1) * nb + side) : -INFINITY;
        }
        bool ok = (__shfl_sync(0xffffffffu, cells, w) >> lane) & 1u;
#pragma unroll
        for (int a = 0; a < 3; a++) {
            float b = __shfl_up_sync(0xffffffffu, v[a], 1), c = __shfl_down_sync(0xffffffffu, v[a], 1);
            if (lane == 0) b = o[a];
            if (lane == 31) c = o[a];
            if (a == 0) ok = ok && v[1] > b && v[1] > v[0] && v[1] > c;
            if (a == 1) ok = ok && v[1] > b && v[1] >= c;
            if (a == 2) ok = ok && v[1] >= b && v[1] >= v[2] && v[1] >= c;
        }
        const uint32_t m = __ballot_sync(0xffffffffu, ok);
        if (lane == w) word = m;
    }
    const int cnt = (int)__reduce_add_sync(0xffffffffu, __popc(word));
    if (lane == 0) count_unit(unit_count, u, cnt);
    if (cnt > 0 && lane < WORDS) unit_mask[(int64_t)u * WORDS + lane] = word;
    return true;
}

// Level 1 over the whole plane: a pure stream.  Grid (ceil(chunks1 / (DETECT_WARPS * CPW1)), K);
// each warp takes CPW1 consecutive chunks of row blockIdx.y, all loads issued first; a lane tests
// its 16 values through their maximum (BF16: packed) and widens them only when it holds a
// candidate.  Few registers, so many warps keep the loads in flight.
template <typename E>
__global__ void __launch_bounds__(DETECT_WARPS * 32, FDAS_K4_L1_MIN_BLOCKS) k4_level1(const E *__restrict__ plane, int64_t nb, int K,
                                                              LevelDesc d, int chunks1,
                                                              int32_t *__restrict__ unit_count,
                                                              uint32_t *__restrict__ unit_mask) {
    constexpr int CPW1 = Fmt<E>::EPV == 8 ? 4 : 2;
    const int lane = threadIdx.x & 31;
    const int i = blockIdx.y;
    const int c0 = (blockIdx.x * DETECT_WARPS + (threadIdx.x >> 5)) * CPW1;
    if (c0 >= chunks1) return;                       // warp-uniform
    const E *row = plane + (int64_t)i * nb;
    typename Fmt<E>::Raw raw[CPW1];
#pragma unroll
    for (int c = 0; c < CPW1; c++)
        if (c0 + c < chunks1) Fmt<E>::load_raw(row + (int64_t)(c0 + c) * CB + LB * lane, raw[c]);
    uint32_t hot = 0;                                // the chunks with a value above the threshold
#pragma unroll
    for (int c = 0; c < CPW1; c++) {
        if (c0 + c >= chunks1) break;
        const int u = (int)d.unit0 + i * (int)d.chunks + c0 + c;
        if (__any_sync(0xffffffffu, Fmt<E>::max16(raw[c]) > d.thr)) hot |= 1u << c;
        else if (lane == 0) unit_count[u] = 0;
    }
    for (; hot; hot &= hot - 1) {
        const int c = c0 + __ffs(hot) - 1;
        level1_many<E>(plane, nb, K, d, i, (int64_t)c * CB, (int)d.unit0 + i * (int)d.chunks + c, unit_count, unit_mask);
    }
}

// Whether chunk c of row i (in level 2's region) can hold a level-2 .. peak given the plane
// kernel's unit marks: always inside level 4's region; outside it only when its unit or one of the
// two units of its second harmonic is marked (see levels_group).
__device__ __forceinline__ bool chunk_needs_search(const uint8_t *__restrict__ marks, int64_t chunks1, int zmax, int K,
                                                   const LevelTable &lt, int i, int c) {
    if (lt.n_levels >= 3 && row_in_level(i, K, zmax, 4) && (int64_t)c * CB <= lt.lev[2].rmax) return true;
    const int i2 = (2 * (-zmax + 2 * i) + zmax) >> 1;
    return __ldg(marks + (int64_t)i * chunks1 + c) | __ldg(marks + (int64_t)i2 * chunks1 + 2 * c) |
           __ldg(marks + (int64_t)i2 * chunks1 + 2 * c + 1);
}

// The level search's work list: one thread per entry k of the block order (row << 16 | 4-chunk
// group); an entry is kept when any of its chunks needs the search (chunk_needs_search), else its
// chunks' level-2 units count zero here.  Whole warps call it.  Short orders: kept entries are appended
// per warp (ballot prefix, one atomic; *count, word 1 of the unit list's header, was cleared before the
// peak search), in whatever order the warps come by.  Long ones (keep != nullptr): the warp leaves its
// ballot, and k4_compact writes the list in the order's order, on which the search's locality rests.
__device__ __noinline__ void select_entry(int64_t k, const uint32_t *__restrict__ order, int64_t n_order,
                                             const uint8_t *__restrict__ marks, int zmax, int K, const LevelTable &lt,
                                             int chunks2, uint32_t *__restrict__ work, unsigned int *__restrict__ count,
                                             uint32_t *__restrict__ keep_words, int32_t *__restrict__ unit_count) {
    const int lane = threadIdx.x & 31;
    bool keep = false;
    uint32_t o = 0;
    if (k < n_order) {
        o = __ldg(order + k);
        const int a = (int)(o >> 16);
        if (a < lt.lev[1].rows) {
            const int i = lt.lev[1].i_lo + a;
            const int64_t chunks1 = lt.lev[0].chunks;
            const int c0 = (int)(o & 0xffffu) * DETECT_WARPS * CPW;
            for (int w = 0; w < DETECT_WARPS * CPW && c0 + w < chunks2; w++)
                keep |= chunk_needs_search(marks, chunks1, zmax, K, lt, i, c0 + w);
            if (!keep)
                for (int w = 0; w < DETECT_WARPS * CPW && c0 + w < chunks2; w++)
                    unit_count[(int)lt.lev[1].unit0 + a * (int)lt.lev[1].chunks + c0 + w] = 0;
        }
    }
    const uint32_t b = __ballot_sync(0xffffffffu, keep);
    if (keep_words != nullptr) {
        if (lane == 0 && k < n_order) keep_words[k >> 5] = b;
        return;
    }
    unsigned int base = 0;
    if (lane == 0 && b) base = atomicAdd(count, (unsigned int)__popc(b));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (keep) work[base + __popc(b & ((1u << lane) - 1u))] = o;
}

// The work list of a long order from the warps' ballots (keep, one word per 32 entries): a block takes
// eight words, counts the entries kept before them (a few KB from L2) and writes its own in order.
// Appended as the warps came by, the list was in random order (mean displacement 4000 of 13887) and
// the search had lost the ray order's locality: N = 2^23, 85 templates, BF16.
__global__ void __launch_bounds__(256) k4_compact(const uint32_t *keep, const uint32_t *__restrict__ order,
                                                  int64_t n_order, uint32_t *__restrict__ work, unsigned int *__restrict__ count) {
    __shared__ unsigned int before[8], own[8];
    grid_wait();
    grid_release();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t n_words = (n_order + 31) / 32, w0 = 8 * (int64_t)blockIdx.x, w = w0 + warp;
    unsigned int sum = 0;
    for (int64_t i = threadIdx.x; i < w0; i += 256) sum += __popc(keep[i]);
    sum = __reduce_add_sync(0xffffffffu, sum);
    const uint32_t bits = w < n_words ? keep[w] : 0u;
    if (lane == 0) {
        before[warp] = sum;
        own[warp] = __popc(bits);
    }
    __syncthreads();
    unsigned int base = 0, total = 0;
#pragma unroll
    for (int i = 0; i < 8; i++) {
        base += before[i] + (i < warp ? own[i] : 0u);
        total += before[i] + own[i];
    }
    if ((bits >> lane) & 1u) work[base + __popc(bits & ((1u << lane) - 1u))] = order[32 * w + lane];
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *count = total;
}

// Level 1 after a plane kernel that marked its units (flags[u] != 0: the unit u = i chunks + c holds
// a stored value above the threshold): a warp takes 32 units, writes a zero count for the unmarked
// ones and runs the level-1 test of k4_level1 on each marked one (a handful per plane).  The
// plane is not streamed; the result is the same as k4_level1's.
// The blocks from l1_blocks on build the level search's work list instead (select_entry, one
// thread per entry of the block order; n_order = 0: none): the list depends only on the marks.
template <typename E>
__global__ void __launch_bounds__(DETECT_WARPS * 32) k4_level1_marked(const E *__restrict__ plane, int64_t nb, int zmax,
                                                                    int K, LevelDesc d, int64_t n_units1,
                                                                    const uint8_t *__restrict__ flags,
                                                                    int32_t *__restrict__ unit_count,
                                                                    uint32_t *__restrict__ unit_mask,
                                                                    int64_t l1_blocks,
                                                                    const uint32_t *__restrict__ order, int64_t n_order,
                                                                    LevelTable lt, int chunks2, uint32_t *__restrict__ work,
                                                                    uint32_t *__restrict__ keep) {
    grid_release();
    const int lane = threadIdx.x & 31;
    if (blockIdx.x >= l1_blocks) {                   // block-uniform
        select_entry((int64_t)(blockIdx.x - l1_blocks) * blockDim.x + threadIdx.x, order, n_order, flags, zmax, K, lt,
                     chunks2, work, unit_list(unit_count) + 1, keep, unit_count);
        return;
    }
    const int64_t u0 = ((int64_t)blockIdx.x * DETECT_WARPS + (threadIdx.x >> 5)) * 32;
    if (u0 >= n_units1) return;                      // warp-uniform
    const int64_t u = u0 + lane;
    const bool marked = u < n_units1 && flags[u] != 0;
    if (u < n_units1 && !marked) unit_count[d.unit0 + u] = 0;
    uint32_t todo = __ballot_sync(0xffffffffu, marked);
    while (todo) {
        const int64_t uu = u0 + (__ffs(todo) - 1);
        todo &= todo - 1;
        const int i = (int)(uu / d.chunks), unit = (int)(d.unit0 + uu);
        const int64_t r0 = (uu - (int64_t)i * d.chunks) * CB;
        typename Fmt<E>::Raw raw;                    // most are marked for level 2's sake (mark_threshold)
        Fmt<E>::load_raw(plane + (int64_t)i * nb + r0 + LB * lane, raw);
        if (__any_sync(0xffffffffu, Fmt<E>::max16(raw) > d.thr)) {
            if (!level1_few<E>(plane, nb, K, d, i, r0, unit, unit_count, unit_mask))
                level1_many<E>(plane, nb, K, d, i, r0, unit, unit_count, unit_mask);
        } else if (lane == 0) {
            unit_count[unit] = 0;
        }
    }
}

// Levels 2 .. 16 of one (row i, CPW chunks from c0) of level 2's region: each warp re-reads S_1
// of its chunks (interleaved bins, see add_level) and carries the running sums through the
// levels in registers.
//   With the plane kernel's unit marks (l2mark: the units holding a stored value above
// mark_threshold <= thr[1] / 2), a chunk outside level 4's region whose unit and the two units of
// its second harmonic are all unmarked is skipped: every P(r) and P(2 r) there is at most
// thr[1] / 2, so S_2 = P(r) + P(2 r) rounds to at most thr[1] (rounded addition is monotone and
// 2 (thr[1] / 2) is exact) and no cell can be a level-2 peak; its unit counts zero without reading
// the plane.  On a noise plane (mean 2) about one 512-bin unit in a hundred holds a value above
// thr[1] / 2 for the thresholds of the searches here, so most of these chunks are skipped.
template <typename E>
__device__ __forceinline__ void levels_group(const E *__restrict__ plane, int64_t nb, int zmax, int K,
                                             const LevelTable &lt, int chunks2, int i, int c0,
                                             int32_t *__restrict__ unit_count, uint32_t *__restrict__ unit_mask,
                                             const uint8_t *__restrict__ l2mark) {
    const int lane = threadIdx.x & 31;
    const int z = -zmax + 2 * i;
    if (l2mark != nullptr && CPW == 1 &&
        (lt.n_levels < 3 || !row_in_level(i, K, zmax, 4) || (int64_t)c0 * CB > lt.lev[2].rmax)) {
        const int64_t chunks1 = lt.lev[0].chunks;
        const int i2 = (2 * z + zmax) >> 1;
        const int64_t mu = lane == 0 ? (int64_t)i * chunks1 + c0 : (int64_t)i2 * chunks1 + 2 * c0 + (lane - 1);
        const bool marked = lane < 3 && __ldg(l2mark + mu) != 0;
        if (!__any_sync(0xffffffffu, marked)) {
            if (lane == 0) unit_count[(int)lt.lev[1].unit0 + (i - lt.lev[1].i_lo) * (int)lt.lev[1].chunks + c0] = 0;
            return;
        }
    }
    const E *row = plane + (int64_t)i * nb;
    const E *row2 = plane + (int64_t)((2 * z + zmax) >> 1) * nb;      // harmonic 2
    const int64_t rmax2 = lt.lev[1].rmax;
    float s2[CPW][LB];                               // S_2 of the lane's bins r0 + lane + 32 e
#pragma unroll
    for (int c = 0; c < CPW; c++)
        if (c0 + c < chunks2) {
            float v[LB];
#pragma unroll
            for (int e = 0; e < LB; e++) {           // S_1 and the second harmonic, all loads at once
                const int64_t r = (int64_t)(c0 + c) * CB + lane + 32 * e;
                s2[c][e] = ld_plane(row, r);
                v[e] = r <= rmax2 ? ld_plane(row2, 2 * r) : 0.0f;
            }
#pragma unroll
            for (int e = 0; e < LB; e++) s2[c][e] = __fadd_rn(s2[c][e], v[e]);
        }
#pragma unroll
    for (int c = 0; c < CPW; c++) {
        if (c0 + c >= chunks2) break;
        detect_chunk<E>(plane, nb, zmax, K, lt, i, z, c0 + c, (int64_t)(c0 + c) * CB + lane, s2[c], unit_count,
                        unit_mask);
    }
}

// Level 2's region row by row: grid (ceil(chunks2 / (DETECT_WARPS * CPW)), rows2), blocks of
// DETECT_WARPS warps on consecutive chunks of one row.
template <typename E>
__global__ void __launch_bounds__(DETECT_WARPS * 32, FDAS_K4_MIN_BLOCKS) k4_levels(const E *__restrict__ plane, int64_t nb, int zmax, int K,
                                                              LevelTable lt, int chunks2,
                                                              int32_t *__restrict__ unit_count,
                                                              uint32_t *__restrict__ unit_mask,
                                                              const uint8_t *__restrict__ l2mark) {
    const int c0 = (blockIdx.x * DETECT_WARPS + (threadIdx.x >> 5)) * CPW;
    if (c0 >= chunks2) return;                       // warp-uniform
    levels_group<E>(plane, nb, zmax, K, lt, chunks2, lt.lev[1].i_lo + blockIdx.y, c0, unit_count, unit_mask, l2mark);
}

// A word written by the kernel before a launch_after(early) one.
__device__ __forceinline__ uint32_t ld_call(const uint32_t *p) {
    uint32_t v;
    asm volatile("ld.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Whether k4_levels_ordered may be launched early.
template <typename E>
constexpr bool EARLY_LEVELS = sizeof(E) == 2;

// Level 2's region in the ray order of upload_levels_order, each entry a (row << 16 | chunk
// group): block b takes the entries b, b + gridDim.x, ... (so the blocks in flight keep to a short
// stretch of the order); with a persistent grid the next entry's code is loaded while the current
// one runs, which keeps the table's latency (about 1 us under load) off the critical path.  Any
// grid size covers every entry once; a grid of one block per entry runs the loop once.
template <typename E>
__global__ void __launch_bounds__(DETECT_WARPS * 32, FDAS_K4_MIN_BLOCKS) k4_levels_ordered(const E *__restrict__ plane, int64_t nb, int zmax, int K,
                                                                      LevelTable lt, int chunks2,
                                                                      const uint32_t *__restrict__ order, int64_t n_order,
                                                                      const unsigned int *__restrict__ d_count,
                                                                      int32_t *__restrict__ unit_count,
                                                                      uint32_t *__restrict__ unit_mask,
                                                                      const uint8_t *__restrict__ l2mark) {
    // BF16 planes: launched early, the list read past the read-only path (ld_call).  FP32 planes' search
    // stays as it was: with the wait it took 185 us instead of 170 (N = 2^23), wherever it was launched.
    constexpr bool EARLY = EARLY_LEVELS<E>;
    auto entry = [&](int64_t k) { return EARLY ? ld_call(order + k) : __ldg(order + k); };
    if constexpr (EARLY) {
        grid_wait();
        grid_release();
    }
    if (d_count != nullptr) n_order = EARLY ? ld_call(d_count) : *d_count;   // a work list (the level-1 pass's selection blocks)
    int64_t idx = blockIdx.x;
    uint32_t next = idx < n_order ? entry(idx) : 0u;
    for (; idx < n_order; idx += gridDim.x) {
        const uint32_t o = next;
        if (idx + gridDim.x < n_order) next = entry(idx + gridDim.x);
        if ((int)(o >> 16) >= lt.lev[1].rows) continue;                       // block-uniform
        const int c0 = ((int)(o & 0xffffu) * DETECT_WARPS + (threadIdx.x >> 5)) * CPW;
        if (c0 >= chunks2) continue;                                          // warp-uniform
        levels_group<E>(plane, nb, zmax, K, lt, chunks2, lt.lev[1].i_lo + (int)(o >> 16), c0, unit_count, unit_mask,
                        l2mark);
    }
}

// Levels 2 .. 16 of the highest-harmonic-anchored sums (harm_mode 1) over the whole plane: grid
// (K rows, ceil(chunks / DETECT_WARPS)), so the blocks in flight share chunk positions across rows
// and the rows they gather from stay in L2.  A warp owns one (row, 512-bin chunk) with the lane
// bins interleaved (lane l holds r0 + l + 32 e) and carries the running sums through the levels.
// For each new harmonic j of level L, the terms r_j = floor((2 j r + L) / (2 L)) of 32
// consecutive r are at most 32 consecutive elements of row i_j, so each warp-wide load reads one
// or two sectors; a harmonic's 16 loads per lane are issued together.
#ifndef FDAS_K4A_BATCH
#define FDAS_K4A_BATCH 2                 // anchored harmonics whose loads are issued together
#endif
// S_L from S_{L/2} for the anchored sums: the odd harmonics j < L in increasing order, the loads
// of FDAS_K4A_BATCH harmonics in flight together (16 per harmonic and lane).  2 j r + L < 2^31 (r < Nb <= 2^26, j < 16),
// so the index arithmetic is 32-bit.  Lane bin r = rb + 32 e gathers at (2 j r + L) >> (LOG + 1) =
// ((2 j rb + L) >> (LOG + 1)) + 32 j e / L exactly (64 j e is a multiple of 2 L for L <= 32), so one
// index per harmonic and lane serves all 16 loads, which then differ by compile-time offsets.
template <typename E, int LOG>
__device__ __forceinline__ void anch_add_level(const E *__restrict__ plane, int64_t nb, int zmax, int z, uint32_t rb,
                                               float (&s)[LB]) {
    constexpr int L = 1 << LOG;
    constexpr int NB = FDAS_K4A_BATCH;
#pragma unroll
    for (int j0 = 1; j0 < L; j0 += 2 * NB) {
        float v[NB][LB];
#pragma unroll
        for (int q = 0; q < NB; q++) {
            const int j = j0 + 2 * q;
            if (j < L) {
                const int ij = (j * z + L * zmax + L) >> (LOG + 1);
                const uint32_t b = (2u * (uint32_t)j * rb + (uint32_t)L) >> (LOG + 1);
                const E *rowj = plane + (int64_t)ij * nb + b;
                static_assert(LOG + 1 <= 6, "the e-offsets are exact while 2 L divides 64");
#pragma unroll
                for (int e = 0; e < LB; e++) v[q][e] = ld_plane(rowj, (int64_t)((64 * j * e) >> (LOG + 1)));
            }
        }
#pragma unroll
        for (int q = 0; q < NB; q++)
            if (j0 + 2 * q < L) {
#pragma unroll
                for (int e = 0; e < LB; e++) s[e] = __fadd_rn(s[e], v[q][e]);
            }
        asm volatile("" ::: "memory");
    }
}

// Levels 2 .. 16 of the anchored sums for one (row i, chunk c), lane bins rb + 32 e.
template <typename E>
__device__ __forceinline__ void anch_chunk(const E *__restrict__ plane, int64_t nb, int zmax, int K, const LevelTable &lt,
                                           int i, int c, int32_t *__restrict__ unit_count,
                                           uint32_t *__restrict__ unit_mask) {
    const int lane = threadIdx.x & 31;
    const int z = -zmax + 2 * i;
    const int64_t rb = (int64_t)c * CB + lane;
    float s[LB];
    {
        const E *row = plane + (int64_t)i * nb;
#pragma unroll
        for (int e = 0; e < LB; e++) s[e] = ld_plane(row, rb + 32 * e);
    }
    auto leave = [&](int l) {                        // the anchored levels cover whole chunks of every row
        leave_sums(s, lt.lev[l].thr, CB - 1, (int)lt.lev[l].unit0 + i * (int)lt.lev[l].chunks + c, unit_count, unit_mask);
    };
    anch_add_level<E, 1>(plane, nb, zmax, z, (uint32_t)rb, s);
    leave(1);
    if (lt.n_levels < 3) return;
    anch_add_level<E, 2>(plane, nb, zmax, z, (uint32_t)rb, s);
    leave(2);
    if (lt.n_levels < 4) return;
    anch_add_level<E, 3>(plane, nb, zmax, z, (uint32_t)rb, s);
    leave(3);
    if (lt.n_levels < 5) return;
    anch_add_level<E, 4>(plane, nb, zmax, z, (uint32_t)rb, s);
    leave(4);
}

template <typename E>
__global__ void __launch_bounds__(DETECT_WARPS * 32, FDAS_K4_MIN_BLOCKS) k4a_levels(const E *__restrict__ plane, int64_t nb,
                                                                               int zmax, int K, LevelTable lt,
                                                                               int chunks,
                                                                               int32_t *__restrict__ unit_count,
                                                                               uint32_t *__restrict__ unit_mask) {
    const int c = blockIdx.y * DETECT_WARPS + (threadIdx.x >> 5);
    if (c >= chunks) return;                         // warp-uniform
    anch_chunk<E>(plane, nb, zmax, K, lt, blockIdx.x, c, unit_count, unit_mask);
}

// The anchored levels in the ray order of upload_levels_order (whole plane, entries
// row << 16 | chunk group): the gathers of cell (r, z) lie on the segment from the origin to
// (r, z), so blocks taken by increasing z / r read each plane sector within a short stretch of
// the kernel's progress (from DRAM about once, where the row-major grid re-fetches the sectors of
// each fraction j / L of the chunk positions).  One block per entry.
template <typename E>
__global__ void __launch_bounds__(DETECT_WARPS * 32, FDAS_K4_MIN_BLOCKS) k4a_levels_ordered(
    const E *__restrict__ plane, int64_t nb, int zmax, int K, LevelTable lt, int chunks,
    const uint32_t *__restrict__ order, int32_t *__restrict__ unit_count, uint32_t *__restrict__ unit_mask) {
    const uint32_t o = __ldg(order + blockIdx.x);
    const int c = (int)(o & 0xffffu) * DETECT_WARPS + (threadIdx.x >> 5);
    if (c >= chunks) return;                         // warp-uniform
    anch_chunk<E>(plane, nb, zmax, K, lt, (int)(o >> 16), c, unit_count, unit_mask);
}

// The units left to be tested (count -1), one warp each: those on the list, or, when it did not hold all
// units, every one in the order of the level search (order: entries row << 16 | chunk group, rows from
// lt.lev[1].i_lo; nullptr: column by column), so that the sums around a unit's cells find their sectors in
// L2 (FP32, N = 2^23, 42 million peaks, when level 1 was tested here too: 37 ms in the units' order, 20 in the
// search's).  Four blocks to an SM at 64 registers, which spill some (404 bytes of stores on FP32 planes, 724 on
// BF16): the gathers' latency is hidden by warps (anchored sums, N = 2^21, 19 million peaks: 13.0 ms with two blocks,
// 11.4; plain sums on short planes, N = 2^18, 333943 peaks: 0.27 ms with two, 0.36).
constexpr int VERIFY_WARPS = 8;
template <typename E>
__global__ void __launch_bounds__(VERIFY_WARPS * 32, 4) k4_verify(const E *__restrict__ plane, int64_t nb, int zmax, int K,
                                                               LevelTable lt, const uint32_t *__restrict__ order,
                                                               int64_t n_order, int32_t *unit_count,
                                                               uint32_t *unit_mask) {
    grid_wait();
    grid_release();
    const unsigned int *list = unit_list(unit_count);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int n = (int)*list;
    const bool anchored = lt.anchored != 0;
    if (n <= PEAK_LIST_CAP) {
        for (int k = (int)blockIdx.x + wid * (int)gridDim.x; k < n; k += VERIFY_WARPS * (int)gridDim.x) {
            const int64_t u = list[4 + k];
            if (unit_count[u] >= 0) continue;            // level 1: tested already
            verify_unit<E>(plane, nb, zmax, K, anchored, unit_of(lt, u), u, unit_count, unit_mask);
        }
        return;
    }
    const int group = anchored ? DETECT_WARPS : DETECT_WARPS * CPW;             // chunks of an order's entry
    const int64_t total = n_order * group;
    for (int64_t k = (int64_t)blockIdx.x * VERIFY_WARPS + wid; k < total; k += (int64_t)gridDim.x * VERIFY_WARPS) {
        int64_t u = -1;                              // lanes 1 .. 4: the chunk's unit of that level
        if (lane > 0 && lane < lt.n_levels) {
            const int64_t o = k / group;
            const uint32_t code = order ? __ldg(order + o) : (uint32_t)(o % lt.lev[1].rows) << 16 | (uint32_t)(o / lt.lev[1].rows);
            const int i = lt.lev[1].i_lo + (int)(code >> 16), c = (int)(code & 0xffffu) * group + (int)(k % group);
            int i_lo = 0, rows = 0;
            int64_t unit0 = 0, chunks = 0;
#pragma unroll
            for (int l = 1; l < 5; l++)
                if (l == lane) {
                    i_lo = lt.lev[l].i_lo;
                    rows = lt.lev[l].rows;
                    unit0 = lt.lev[l].unit0;
                    chunks = lt.lev[l].chunks;
                }
            if (i >= i_lo && i < i_lo + rows && c < chunks) u = unit0 + (int64_t)(i - i_lo) * chunks + c;
        }
        uint32_t todo = __ballot_sync(0xffffffffu, u >= 0 && unit_count[u < 0 ? 0 : u] < 0);
        for (; todo; todo &= todo - 1) {
            const int64_t uu = __shfl_sync(0xffffffffu, u, __ffs(todo) - 1);
            verify_unit<E>(plane, nb, zmax, K, anchored, unit_of(lt, uu), uu, unit_count, unit_mask);
        }
    }
}

// The records of one non-empty unit u, the first at out[base]: one warp, the unit's mask words one
// per lane, the peaks dealt to the lanes in bin order (the order of the output within a unit).
template <typename E>
__device__ __noinline__ void emit_unit(const E *__restrict__ plane, int64_t nb, int zmax, bool anchored, UnitRef ref,
                                       int64_t u, int64_t base, const uint32_t *unit_mask,
                                       fdas_peak *__restrict__ out, int max_peaks, uint32_t series) {
    const int lane = threadIdx.x & 31;
    const int H = ref.H;
    const uint32_t w = lane < WORDS ? unit_mask[u * WORDS + lane] : 0u;
    int incl = __popc(w);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    const int total = __shfl_sync(0xffffffffu, incl, 31);
    for (int k0 = 0; k0 < total; k0 += 32) {                 // warp-uniform
        const int k = k0 + lane;                             // this lane's peak of the unit
        int word = 0, before = 0;
#pragma unroll
        for (int j = 0; j < WORDS; j++) {                    // the word holding it: the first with incl > k
            const int ij = __shfl_sync(0xffffffffu, incl, j);
            if (ij <= k) {
                word = j + 1;
                before = ij;
            }
        }
        uint32_t bits = __shfl_sync(0xffffffffu, w, word & 31);
        if (k < total && base + k < max_peaks) {
            for (int skip = k - before; skip > 0; skip--) bits &= bits - 1;
            const int64_t r = ref.chunk * CB + word * 32 + (__ffs(bits) - 1);
            fdas_peak pk;
            pk.series = series;
            pk.r = (uint32_t)r;
            pk.zi = (int16_t)ref.row;
            pk.harm = (uint8_t)H;
            pk.pad = 0;
            pk.power = anchored ? harm_sum_anch(plane, nb, zmax, H, ref.row, r)
                                   : harm_sum(plane, nb, zmax, H, ref.row, r);
            out[base + k] = pk;
        }
    }
}

// Exclusive scan of one value per thread over a block of 1024 threads; *total = the block's sum.
// warp_tot: 32 ints of shared memory.  Every thread calls it (two barriers).
__device__ __forceinline__ int32_t block_excl_scan(int32_t c, int32_t *warp_tot, int32_t *total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int32_t incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) warp_tot[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        const int32_t wt = warp_tot[lane];
        int32_t wi = wt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += y;
        }
        warp_tot[lane] = wi - wt;                        // exclusive warp offsets
        if (lane == 31) warp_tot[32] = wi;
    }
    __syncthreads();
    *total = warp_tot[32];
    return warp_tot[warp] + incl - c;
}

// The step's peaks, blocks of 1024 threads.  Usually the unit list holds every
// non-empty unit (a handful to a few thousand of ~10^6): unit k of the list goes to warp k / grid of
// block k mod grid, which sums the counts of the listed units with smaller numbers (its output
// offset; the list and its counts in shared memory, 32 a step) and emits the unit's records.
// Units are numbered in (level, row, chunk) order, so the records come out in (H, i, r) order.
// One block that sorted the list and emitted all units itself took 51 us for some 600 units of
// anchored sums, this 6 us.
// When more than PEAK_LIST_CAP units hold peaks (low thresholds, up to millions of peaks), every
// block takes an equal share of the units: it sums the counts before its range (its first output
// offset; a few MB read from L2 per block, no communication between blocks), then scans its
// range, 4096 units a round at most, and deals the round's non-empty units to its warps.  Shares of
// whole rounds left a plane of 10^4 units to two or three blocks (level 1 alone, FP32, N = 2^18, 27296 peaks:
// 395 -> 55 us for the call; N = 2^16, 312797 peaks: 886 -> 35 us).  1024 threads leave 64 registers: emit_unit's
// 16 gathers in flight spill some 130 bytes.  The last block (or block 0
// on the listed path) writes the total and the overflow flag.
static_assert(PEAK_LIST_CAP == 4 * 1024, "a round of the scan: four units a thread");
template <typename E>
__global__ void __launch_bounds__(1024, 1) k4_emit_listed(const E *__restrict__ plane, int64_t nb, int zmax, LevelTable lt,
                                                       int64_t n_units, const int32_t *unit_count,
                                                       const uint32_t *unit_mask,
                                                       fdas_peak *__restrict__ out, int max_peaks, uint32_t series,
                                                       int32_t *__restrict__ npeaks, int32_t *__restrict__ status) {
    __shared__ uint32_t key[PEAK_LIST_CAP];
    __shared__ int32_t cnt[PEAK_LIST_CAP];
    __shared__ int32_t warp_tot[33];
    grid_wait();
    grid_release();
    const int t = threadIdx.x, warp = t >> 5;
    const unsigned int *list = unit_list(unit_count);
    const int n = (int)*list;
    int64_t total = 0;
    bool writer = false;                                 // the block that writes the total
    if (n <= PEAK_LIST_CAP) {                            // grid-uniform
        if (blockIdx.x != 0 && (int)blockIdx.x >= n) return;
        writer = blockIdx.x == 0;
        for (int k = t; k < n; k += 1024) {
            key[k] = list[4 + k];
            cnt[k] = unit_count[key[k]];
        }
        __syncthreads();
        // at most 4096 units x 512 peaks: 32-bit offsets
        const int lane = t & 31;
        for (int k = (int)blockIdx.x + warp * (int)gridDim.x; k < n; k += 32 * (int)gridDim.x) {
            const uint32_t mine = key[k];
            int before = 0;
            for (int j = lane; j < n; j += 32) before += key[j] < mine ? cnt[j] : 0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) before += __shfl_xor_sync(0xffffffffu, before, o);
            emit_unit<E>(plane, nb, zmax, lt.anchored != 0, unit_of(lt, mine), (int64_t)mine, before, unit_mask, out, max_peaks,
                         series);
        }
        if (writer && warp == 31) {
            int all = 0;
            for (int j = lane; j < n; j += 32) all += cnt[j];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) all += __shfl_xor_sync(0xffffffffu, all, o);
            total = all;
        }
        writer = writer && warp == 31;
    } else {
        // this block's units [ub, ue), an equal share to every block, and the count before them
        const int64_t per = (n_units + gridDim.x - 1) / gridDim.x;
        const int64_t ub = min(n_units, (int64_t)blockIdx.x * per);
        const int64_t ue = min(n_units, ub + per);
        writer = blockIdx.x == gridDim.x - 1 && warp == 0;
        {
            __shared__ unsigned long long pre_tot;       // counts are non-negative
            if (t == 0) pre_tot = 0ull;
            __syncthreads();
            unsigned long long acc = 0ull;
            for (int64_t u = t; u < ub; u += 1024) acc += (unsigned long long)unit_count[u];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if ((t & 31) == 0) atomicAdd(&pre_tot, acc);
            __syncthreads();
            total = (int64_t)pre_tot;
        }
        for (int64_t u0 = ub; u0 < ue; u0 += PEAK_LIST_CAP) {
            const int n_round = (int)min((int64_t)PEAK_LIST_CAP, ue - u0);
            int32_t v[4];                                // this thread's 4 units: counts, then offsets in the round
#pragma unroll
            for (int k = 0; k < 4; k++) v[k] = 4 * t + k < n_round ? unit_count[u0 + 4 * t + k] : 0;
            int32_t tot;
            int32_t run = block_excl_scan(v[0] + v[1] + v[2] + v[3], warp_tot, &tot);
#pragma unroll
            for (int k = 0; k < 4; k++) {
                cnt[4 * t + k] = v[k];
                key[4 * t + k] = (uint32_t)run;
                run += v[k];
            }
            __syncthreads();
            // unit j to warp (j - j / 32) mod 32: neighbours to different warps, a warp's 32 counts on 32 banks
            const int lane = t & 31;
            for (int j0 = 0; j0 < n_round; j0 += 1024) {
                uint32_t busy = __ballot_sync(0xffffffffu, cnt[j0 + 32 * lane + ((warp + lane) & 31)] != 0);
                for (; busy; busy &= busy - 1) {         // warp-uniform
                    const int l = __ffs(busy) - 1, j = j0 + 32 * l + ((warp + l) & 31);
                    emit_unit<E>(plane, nb, zmax, lt.anchored != 0, unit_of(lt, u0 + j), u0 + j, total + key[j], unit_mask, out,
                                 max_peaks, series);
                }
            }
            total += tot;
            __syncthreads();                             // the arrays are reused by the next round
        }
    }
    if (writer && (t & 31) == 0) {
        *npeaks = (int32_t)(total < 0x7fffffff ? total : 0x7fffffff);
        if (total > max_peaks) atomicOr(status, FDAS_DEV_PEAK_OVERFLOW);
    }
}

template <typename E>
cudaError_t run_peaks(const Plan &p, const E *plane, char *ws, fdas_peak *peaks, int32_t *npeaks, uint32_t series,
                      cudaStream_t st, const uint8_t *l1flag, bool list_cleared, bool early, bool early_tail) {
    const LevelTable lt = make_levels(p);
    int32_t *unit_count = reinterpret_cast<int32_t *>(ws + p.ws_ucount);
    uint32_t *unit_mask = reinterpret_cast<uint32_t *>(ws + p.ws_umask);
    const int64_t chunks1 = lt.lev[0].chunks;
    constexpr int CPW1 = Fmt<E>::EPV == 8 ? 4 : 2;
    const dim3 level1_grid((unsigned)((chunks1 + DETECT_WARPS * CPW1 - 1) / (DETECT_WARPS * CPW1)), (unsigned)p.K);
    const int64_t chunks2 = lt.n_levels > 1 ? lt.lev[1].chunks : 0;
    const dim3 levels_grid((unsigned)((chunks2 + DETECT_WARPS * CPW - 1) / (DETECT_WARPS * CPW)),
                           (unsigned)(lt.n_levels > 1 ? lt.lev[1].rows : 0));
    if (lt.n_levels > 1 && !lt.anchored &&
        (!p.d_k4order || p.k4order_n != (int64_t)lt.lev[1].rows * ((chunks2 + DETECT_WARPS * CPW - 1) / (DETECT_WARPS * CPW))))
        return cudaErrorInvalidValue;                // the block order was not built for this region
    const int64_t n_units = p.n_units;
    // the plane kernel's unit marks (mark_threshold) bound the level-2 sums too
    const uint8_t *l2mark = l1flag && lt.n_levels > 1 ? l1flag : nullptr;
    p.prof.begin(FDAS_STAGE_PEAKS, st);
    // the unit list starts empty (its counter: the word PEAK_LIST_WORDS before the counts)
    // and so does the level search's work count (the next word); a search's long FFT has cleared
    // both already (list_cleared)
    uint32_t *list_hdr = reinterpret_cast<uint32_t *>(unit_count) - PEAK_LIST_WORDS;
    cudaError_t e = cudaSuccess;
    if (!list_cleared) {
        e = cudaMemsetAsync(list_hdr, 0, 2 * sizeof(uint32_t), st);
        if (e != cudaSuccess) return e;
    }
    p.prof.launches += lt.n_levels > 1 ? 3 : 2;
    // whether some level kernel leaves cells above the threshold to k4_verify
    const bool verify = lt.n_levels > 1 && (lt.anchored || !IN_PLACE<E>);
    // with the marks, the level search's work list is built by extra blocks of the level-1 pass
    const bool select_list = l2mark != nullptr && lt.n_levels > 1 && !lt.anchored && (sizeof(E) == 4 || FDAS_K4_RAY_BF16);
    uint32_t *work = reinterpret_cast<uint32_t *>(ws + p.ws_k4work);
    unsigned int *wcount = select_list ? list_hdr + 1 : nullptr;
    // from 4096 entries on the list is put in order (one more launch, 4 us; below, the whole region is
    // a few MB of plane and any order will do): the level search of N = 2^23, 85 templates takes 132 us
    // instead of 148 (BF16), 170 instead of 190 (FP32); N = 2^21, BF16, 3500 entries of 4 chunks:
    // 43 instead of 49
    uint32_t *keep = select_list && p.k4order_n >= 4096 ? work + p.k4order_n : nullptr;
    p.prof.begin(PROF_PEAKS_LEVEL1, st);
    if (l1flag) {
        const int64_t n1 = (int64_t)p.K * chunks1;
        const int64_t blocks = (n1 + DETECT_WARPS * 32 - 1) / (DETECT_WARPS * 32);
        const int64_t n_sel = select_list ? p.k4order_n : 0;
        const int64_t sel_blocks = (n_sel + DETECT_WARPS * 32 - 1) / (DETECT_WARPS * 32);
        k4_level1_marked<E><<<(unsigned)(blocks + sel_blocks), DETECT_WARPS * 32, 0, st>>>(
            plane, p.nb, p.cfg.zmax, p.K, lt.lev[0], n1, l1flag, unit_count, unit_mask, blocks, p.d_k4order, n_sel,
            lt, (int)chunks2, work, keep);
        if (keep) {
            e = launch_after(early_tail, k4_compact, (unsigned)((p.k4order_n + 255) / 256), 256, 0, st, keep, p.d_k4order, p.k4order_n, work, wcount);
            if (e != cudaSuccess) return e;
            p.prof.launches++;
        }
        p.prof.level1_fused++;
    } else {
        k4_level1<E><<<level1_grid, DETECT_WARPS * 32, 0, st>>>(plane, p.nb, p.K, lt.lev[0], (int)chunks1, unit_count, unit_mask);
    }
    p.prof.end(PROF_PEAKS_LEVEL1, st);
    if (lt.n_levels > 1 && lt.anchored) {
        p.prof.begin(PROF_PEAKS_LEVELS, st);
        const int64_t agroups = (chunks1 + DETECT_WARPS - 1) / DETECT_WARPS;
        if (p.d_k4order_a && p.k4order_a_n == (int64_t)p.K * agroups) {
            k4a_levels_ordered<E><<<(unsigned)p.k4order_a_n, DETECT_WARPS * 32, 0, st>>>(
                plane, p.nb, p.cfg.zmax, p.K, lt, (int)chunks1, p.d_k4order_a, unit_count, unit_mask);
        } else {
            const dim3 agrid((unsigned)p.K, (unsigned)agroups);
            k4a_levels<E><<<agrid, DETECT_WARPS * 32, 0, st>>>(plane, p.nb, p.cfg.zmax, p.K, lt, (int)chunks1,
                                                               unit_count, unit_mask);
        }
        p.prof.end(PROF_PEAKS_LEVELS, st);
    } else if (lt.n_levels > 1) {
        p.prof.begin(PROF_PEAKS_LEVELS, st);
        if (sizeof(E) == 4 || FDAS_K4_RAY_BF16) {
            // BF16 plane: a persistent grid (whole region, N = 2^23, 85 templates: 0.191 ms, one block
            // per entry 0.26; entries drawn from a counter 0.22).  FP32 plane: one block per entry
            // (with the marks' list 0.170 ms, persistent 0.268: its entries carry twice the bytes and
            // the static stride balances worse; drawn from a counter 0.188)
            int sms = 0;
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, p.device >= 0 ? p.device : 0);
            const int64_t blocks = sizeof(E) == 4 ? p.k4order_n
                                                  : std::min<int64_t>(p.k4order_n, (int64_t)std::max(sms, 1) * FDAS_K4_MIN_BLOCKS);
            // with the marks: select the entries to search first (a list in the workspace), so that the
            // skipped chunks cost one thread each instead of a warp's round trip in the search
            // (the work list from the level-1 pass's extra blocks, when the marks exist)
            const uint32_t *order = select_list ? work : p.d_k4order;
            // (the plane and the marks were complete when the kernel before, which waited or was launched
            // plainly, let this one in; the work list is the last kernel's)
            e = launch_after(early && EARLY_LEVELS<E>, k4_levels_ordered<E>, (unsigned)blocks, DETECT_WARPS * 32, 0, st, plane, p.nb, p.cfg.zmax, p.K, lt,
                             (int)chunks2, order, p.k4order_n, wcount, unit_count, unit_mask, l2mark);
            if (e != cudaSuccess) return e;
        } else {
            k4_levels<E><<<levels_grid, DETECT_WARPS * 32, 0, st>>>(plane, p.nb, p.cfg.zmax, p.K, lt, (int)chunks2,
                                                                     unit_count, unit_mask, l2mark);
        }
        p.prof.end(PROF_PEAKS_LEVELS, st);
    }
    int sms_out = 152;
    cudaDeviceGetAttribute(&sms_out, cudaDevAttrMultiProcessorCount, p.device >= 0 ? p.device : 0);
    if (verify) {
        const int64_t group = lt.anchored ? DETECT_WARPS : DETECT_WARPS * CPW;
        const int64_t n_order = (int64_t)lt.lev[1].rows * ((lt.lev[1].chunks + group - 1) / group);
        const uint32_t *order = !lt.anchored ? p.d_k4order : p.k4order_a_n == n_order ? p.d_k4order_a : nullptr;
        e = launch_after(early_tail, k4_verify<E>, (unsigned)std::max(1, 4 * sms_out), VERIFY_WARPS * 32, 0, st, plane, p.nb, p.cfg.zmax, p.K, lt,
                         order, n_order, unit_count, unit_mask);
        if (e != cudaSuccess) return e;
        p.prof.launches++;
    }
    // one block per SM: a listed unit per block and warp in the usual case, a range of all units each else
    e = launch_after(early_tail, k4_emit_listed<E>, (unsigned)std::max(1, sms_out), 1024, 0, st, plane, p.nb, p.cfg.zmax, lt, n_units, unit_count,
                     unit_mask, peaks, p.cfg.max_peaks, series, npeaks, p.d_status);
    p.prof.end(FDAS_STAGE_PEAKS, st);
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace

// Level H's region: rows [i_lo, i_lo + rows) and bins r <= rmax.  Plain sums: the rows with
// |H z| <= zmax and H r < Nb; anchored sums: the whole plane.
static void level_region(const Plan &p, int H, bool anchored, LevelDesc &d) {
    int zl = p.cfg.zmax / H;
    zl -= zl & 1;                                   // largest even z with |H z| <= zmax
    if (anchored) zl = p.cfg.zmax;
    d.H = H;
    d.i_lo = (p.cfg.zmax - zl) / 2;
    d.rows = zl + 1;
    d.rmax = anchored ? p.nb - 1 : (p.nb - 1) / H;
    d.chunks = (d.rmax + 1 + PEAK_CHUNK - 1) / PEAK_CHUNK;
}

LevelTable make_levels(const Plan &p) {
    LevelTable lt{};
    int64_t unit0 = 0;
    int n = 0;
    for (int l = 0; l < 5; l++) {
        const int H = 1 << l;
        if (H > p.cfg.max_harm) break;
        LevelDesc &d = lt.lev[n];
        level_region(p, H, p.cfg.harm_mode == 1, d);
        d.unit0 = unit0;
        d.thr = p.cfg.thr[l];
        unit0 += (int64_t)d.rows * d.chunks;
        n++;
    }
    lt.n_levels = n;
    lt.anchored = p.cfg.harm_mode == 1;
    return lt;
}

// The order in which k4_levels_ordered takes the (row, chunk group) blocks of level 2's region.
// Cell (r, z) gathers its harmonics at (h r, h z), on the ray from the origin through (r, z),
// where every other cell of that ray gathers too, and the rest of each gathered sector belongs
// to neighbouring rays.  Taking the blocks by increasing z / r (of the group's middle bin; ties
// by row, then group) brings all reads of a plane sector into a short stretch of the kernel's
// progress, so it comes from DRAM about once; row by row (k4_levels) the harmonic rows of rows
// far apart are fetched again, about twice the bytes.  Built for level 2's region whatever
// max_harm and harm_mode say, so that plans of one shape can share it.
bool levels_order(const Plan &p, std::vector<uint32_t> &order, bool anchored) {
    LevelDesc d{};
    level_region(p, 2, anchored, d);                  // anchored: the whole plane
    const int64_t per = DETECT_WARPS * (anchored ? 1 : CPW);   // chunks per block
    const int64_t groups = (d.chunks + per - 1) / per;
    if (d.rows >= (1 << 16) || groups >= (1 << 16)) return false;
    struct Item {
        double key;
        uint32_t code;
    };
    std::vector<Item> items;
    items.reserve((size_t)(d.rows * groups));
    for (int a = 0; a < d.rows; a++) {
        const int z = -p.cfg.zmax + 2 * (d.i_lo + a);
        for (int64_t g = 0; g < groups; g++)
            items.push_back({(double)z / ((double)(g * per) + 0.5 * (double)per), ((uint32_t)a << 16) | (uint32_t)g});
    }
    std::sort(items.begin(), items.end(),
              [](const Item &x, const Item &y) { return x.key < y.key || (x.key == y.key && x.code < y.code); });
    order.resize(items.size());
    for (size_t k = 0; k < items.size(); k++) order[k] = items[k].code;
    return true;
}

int64_t levels_order_size(const Plan &p) {
    LevelDesc d{};
    level_region(p, 2, false, d);
    const int64_t per = DETECT_WARPS * CPW;
    return (int64_t)d.rows * ((d.chunks + per - 1) / per);
}

cudaError_t upload_levels_order(Plan &p) {
    std::vector<uint32_t> order;
    if (!levels_order(p, order, false)) return cudaErrorInvalidValue;
    p.k4order_n = (int64_t)order.size();
    cudaError_t e = cudaMalloc((void **)&p.d_k4order, sizeof(uint32_t) * order.size());
    if (e == cudaSuccess)
        e = cudaMemcpy(p.d_k4order, order.data(), sizeof(uint32_t) * order.size(), cudaMemcpyHostToDevice);
    // the anchored sums' whole-plane order, for plans that use them
    if (e == cudaSuccess && p.cfg.harm_mode == 1 && levels_order(p, order, true)) {
        p.k4order_a_n = (int64_t)order.size();
        e = cudaMalloc((void **)&p.d_k4order_a, sizeof(uint32_t) * order.size());
        if (e == cudaSuccess)
            e = cudaMemcpy(p.d_k4order_a, order.data(), sizeof(uint32_t) * order.size(), cudaMemcpyHostToDevice);
    }
    return e;
}

cudaError_t launch_peaks(const Plan &p, const void *d_plane, bool bf16, char *ws, fdas_peak *d_peaks,
                         int32_t *d_npeaks, uint32_t series, cudaStream_t st, const uint8_t *l1flag, bool list_cleared, bool early, bool early_tail) {
    if (bf16)
        return run_peaks<__nv_bfloat16>(p, reinterpret_cast<const __nv_bfloat16 *>(d_plane), ws, d_peaks, d_npeaks,
                                        series, st, l1flag, list_cleared, early, early_tail);
    return run_peaks<float>(p, reinterpret_cast<const float *>(d_plane), ws, d_peaks, d_npeaks, series, st, l1flag,
                            list_cleared, early, early_tail);
}

}  // namespace fdas

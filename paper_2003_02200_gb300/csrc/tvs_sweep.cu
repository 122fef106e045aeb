// tvs_sweep.cu -- the sweep of the sDEM total viewshed (Kernel-2, Alg. 7 and
// 8) with the relocation of Kernel-1 (Alg. 6) fused into its row staging.
//
// A work item is one skewed row and one walk direction; a warp takes one, both
// directions of several short rows, or a share of a long one.  The row's
// samples are gathered straight from the DEM (section 4.1 step 1(a): sample j of
// line b blends view rows a = b + dest(j) and a + 1 with weights 1 - r(j) and
// r(j)), so the skewed DEM never reaches HBM, then every usable sample of the
// row walks it (forward items walk the row, backward items its reverse).
//
// Two decision modes:
//
//  * FP32 decisions (the paper's kernel precision: "float" heights and
//    slopes in Alg. 6-8): the staged height is (1-r)*a + r*b in single
//    precision and a target is visible iff fl(fl(z - h) * fl(1/d)) is
//    strictly above the running maximum.
//
//  * Certified decisions (the default): every visibility decision is the one
//    exact arithmetic takes on the exact blended heights, which is what the
//    FP64 definition decides (it rounds some 10^-16 away from exact).  The
//    row is staged as a double-float (hi + lo) pair per sample.  The fast
//    path still decides in FP32, on height differences formed against a
//    per-group reference, and proves each decision with a margin derived
//    below; a decision inside its margin leaves its block of the walk to an
//    exact pass (double-float slopes with their own margin, and the FP64
//    definition itself for what that margin cannot settle).
//
// Pruned launches (the default) evaluate only the blocks of a walk that can
// hold a visible target; unpruned ones evaluate every target.
#include "tvs.h"
#include "tvs_internal.h"
#include "tvs_df.cuh"

#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

namespace tvs {

// Index checks of the sweep.  The indices of the staging, of the blocks and
// tests (once per row or group) and of the exact walks are checked against
// their buffers (not the inner step loop, whose indices follow): a
// violation records the first offending index in g_sweep_check (code, index,
// bound, CTA) and skips the access instead of faulting.  Read and cleared by
// tvs_debug_sweep_check.
__device__ int g_sweep_check[4];
// Event counts of the certified sweep: blocks (or rests of walks, or whole walks) decided again
// exactly, of them in FP64, SM clock cycles warps spent in the exact pass, and
// cycles warps spent in the certified sweep kernels.
__device__ unsigned long long g_sweep_stats[4];

__device__ __forceinline__ bool in_range(long long idx, long long bound, int code)
{
    if (idx >= 0 && idx < bound) return true;
    if (atomicCAS(&g_sweep_check[0], 0, code) == 0) {
        g_sweep_check[1] = (int)idx;
        g_sweep_check[2] = (int)bound;
        g_sweep_check[3] = (int)blockIdx.x;
    }
    return false;
}

namespace {

__device__ __forceinline__ float neg_inf() { return __int_as_float(0xff800000); }
__device__ __forceinline__ float pos_inf() { return __int_as_float(0x7f800000); }

struct SweepParams {
    const DirDev* dirs;
    const JobDev* jobs;
    const int* item_start;
    const int* rowlo;
    const int* rowhi;
    int* cv_fwd;       // forward measure of every sample (slab layout)
    int* cv_bwd;       // backward measure of every sample (slab layout)
    unsigned* counter;
    int4* flag_buf;    // certified: flagged walks for the exact pass
    unsigned* flag_count;   // its fill, one unused, and whether a flag found it full
    int flag_cap;
    int ndir;
    int total_items;
    int scan_blocks;   // 32-sample blocks of the longest row
    int inv_len;       // entries of the per-distance table
    int tab_floats;    // floats it takes (a multiple of 4)
    int istart_len;    // ints of the item-start table (multiple of 4)
    int half;          // floats of one staged row array (multiple of 4)
    int padr;          // of them after the row's samples
    int lgna;          // packed kernel: log2 of the staged rows per warp
    int per_row;       // packed kernel: floats of a staged row's arrays
    int lgw;           // log2 of the warps that share a row (certified, long rows)
    int per_pair;      // floats of their shared area
    int zs_len;        // floats of the row's suffix maxima (0 without pruning)
    int wm_len;        // floats of the row's window maxima (0 without pruning)
    int per_warp;      // floats of a warp's shared area
};

// ------------------------------------------------------ row geometry --
// DEM index of view cell (a, j) of direction d and the index step from view
// row a to view row a + 1 (the four D4 views of section 4.1 / Alg. 6).
__device__ __forceinline__ long long view_index(const DirDev& d, int cols, int a, int j, int* step)
{
    switch (d.frame) {
    case 0:  *step = cols;  return (long long)a * cols + j;
    case 1:  *step = 1;     return (long long)j * cols + a;
    case 2:  *step = 1;     return (long long)(d.W - 1 - j) * cols + a;
    default: *step = -cols; return (long long)(d.H - 1 - a) * cols + j;
    }
}

// The paper's single-precision blend of Kernel-1: r = float(fr) 2^-32,
// (1 - r) a + r b with every operation rounded.
__device__ __forceinline__ float blend32(float va, float vb, unsigned fr)
{
    if (fr == 0u) return va;
    const float r = __fmul_rn(__uint2float_rn(fr), 0x1p-32f);
    const float wa = __fsub_rn(1.0f, r);
    return __fadd_rn(__fmul_rn(wa, va), __fmul_rn(r, vb));
}

// A sweep work item: (direction, skewed row, walk direction).
struct ItemRow {
    long long rowbase;   // slab offset of the row's first usable sample
    int dir, p, jlo;
    int L, K, pov;
    float h0;
    bool rev;
};

// Skewed row p of direction `dir`, walked forward or backward; false when the
// row is empty.
__device__ __forceinline__ bool decode_row(const SweepParams& sp, int dir, int p, bool rev, ItemRow* it)
{
    const DirDev& d = sp.dirs[dir];
    it->rev = rev;
    const int jlo = sp.rowlo[d.row_off + p], jhi = sp.rowhi[d.row_off + p];
    it->dir = dir;
    it->p = p;
    it->jlo = jlo;
    it->L = jhi - jlo + 1;
    it->K = d.K;
    it->h0 = d.h0;
    it->pov = row_pov(it->L, d.K, d.pov, d.p4_pct);
    it->rowbase = d.slab + (long long)p * d.Wp + jlo;
    return it->L > 0;
}

// Decodes item into its row; false when the row is empty.
__device__ __forceinline__ bool decode_item(const SweepParams& sp, const int* istart, int item, ItemRow* it)
{
    int lo = 0, hi = sp.ndir - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (istart[mid] <= item) lo = mid; else hi = mid - 1;
    }
    const int rem = item - istart[lo];
    return decode_row(sp, lo, rem >> 1, (rem & 1) != 0, it);
}

// Stages the item's row from the DEM: FP32 heights into Fh, or with CERT hi
// parts into Fh and lo parts into Fl, reversed for backward items unless
// rev_ok is false (rows that both walk directions share stay in row order);
// with mirror arrays also reversed into those.  The last sample and sp.padr samples after
// it hold -inf (lo 0): the last target of a walk never adds area, so it may be
// a sentinel that is never visible.  With CERT the first sample and the
// ROW_PADL samples before it are sentinels too (the last target of a backward
// walk), and the real hi and lo parts of the two end samples, which are POVs,
// go to ends[0..3] (first hi, first lo, last hi, last lo).  Returns (with CERT)
// the row's largest |elevation| read, for the error bounds.
template <bool CERT>
__device__ __forceinline__ float stage_row(const SweepParams& sp, const ItemRow& it, float* Fh, float* Fl,
                                           float* ends, int lane, int part = 0, int parts = 1, bool rev_ok = true,
                                           float* mirror_h = nullptr, float* mirror_l = nullptr)
{
    const DirDev& d = sp.dirs[it.dir];
    const float* __restrict__ dem = sp.jobs[d.job].dem;
    const int cols = sp.jobs[d.job].cols;
    const long long cells = (long long)sp.jobs[d.job].rows * cols;
    const int b = it.p - d.D;
    const unsigned long long t_fx = d.t_fx;
    const bool rev = rev_ok && it.rev;
    const float NEG = neg_inf();
    float zmax = 0.f;
    constexpr int B = 4;
    for (int x0 = lane + 32 * B * part; x0 < it.L; x0 += 32 * B * parts) {
        float va[B], vb[B];
        unsigned fr[B];
#pragma unroll
        for (int k = 0; k < B; ++k) {
            const int x = x0 + 32 * k;
            va[k] = 0.f; vb[k] = 0.f; fr[k] = 0u;
            if (x < it.L) {
                const int j = it.jlo + (rev ? it.L - 1 - x : x);
                const unsigned long long y = (unsigned long long)j * t_fx;
                const int a = b + (int)(y >> 32);
                fr[k] = (unsigned)y;
                int st;
                const long long idx = view_index(d, cols, a, j, &st);
                va[k] = in_range(idx, cells, 1) ? dem[idx] : 0.f;
                vb[k] = fr[k] != 0u ? (in_range(idx + st, cells, 2) ? dem[idx + st] : 0.f) : va[k];
            }
        }
#pragma unroll
        for (int k = 0; k < B; ++k) {
            const int x = x0 + 32 * k;
            if (x >= it.L || !in_range(ROW_PADL + x, sp.half, 3)) continue;
            if (CERT) {
                float zh, zl;
                df::df_blend(va[k], vb[k], fr[k], zh, zl);
                const bool end = x == 0 || x == it.L - 1;
                if (x == 0) { ends[0] = zh; ends[1] = zl; }
                if (x == it.L - 1) { ends[2] = zh; ends[3] = zl; }
                Fh[ROW_PADL + x] = end ? NEG : zh;
                Fl[ROW_PADL + x] = end ? 0.f : zl;
                if (mirror_h) {
                    mirror_h[ROW_PADL + it.L - 1 - x] = end ? NEG : zh;
                    mirror_l[ROW_PADL + it.L - 1 - x] = end ? 0.f : zl;
                }
                zmax = fmaxf(zmax, fmaxf(fabsf(va[k]), fabsf(vb[k])));
            } else {
                Fh[ROW_PADL + x] = x == it.L - 1 ? NEG : blend32(va[k], vb[k], fr[k]);
            }
        }
    }
    for (int m = lane; part == 0 && m < sp.padr; m += 32) {
        if (!in_range(ROW_PADL + it.L + m, sp.half, 4)) continue;
        Fh[ROW_PADL + it.L + m] = NEG;
        if (CERT) Fl[ROW_PADL + it.L + m] = 0.f;
        if (CERT && mirror_h) { mirror_h[ROW_PADL + it.L + m] = NEG; mirror_l[ROW_PADL + it.L + m] = 0.f; }
    }
    if (CERT) {
        if (part == 0 && lane < ROW_PADL) { Fh[lane] = NEG; Fl[lane] = 0.f; }
        if (part == 0 && mirror_h && lane < ROW_PADL) { mirror_h[lane] = NEG; mirror_l[lane] = 0.f; }
    } else if (lane < ROW_PADL) {
        Fh[lane] = NEG;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) zmax = fmaxf(zmax, __shfl_xor_sync(0xffffffffu, zmax, o));
    return zmax;
}

// ------------------------------------------------ FP32-decision sweep --
__device__ __forceinline__ float fset_gt(float a, float b)
{
    // 1.0f if a > b (strict; false for NaN), else 0.0f
    float v;
    asm("set.gt.f32.f32 %0, %1, %2;" : "=f"(v) : "f"(a), "f"(b));
    return v;
}

// Distance entry (1/d, 1/d, 2d + 1, 2d + 1) as the table holds it.
__device__ __forceinline__ float4 dist_entry(int d)
{
    const float r = __frcp_rn((float)d);
    const float c = (float)(2 * d + 1);
    return make_float4(r, r, c, c);
}

// (1/d, 1/d) and (2d + 1, 2d + 1) of step u of a block that starts at step e
// (d = e + 1 + u), tab at the block's first entry.  Unpruned walks keep both in
// the table (float4).  Pruned walks keep (1/d, 1/d) alone: their lanes stand at
// 32 different steps, so an entry of 16 bytes costs four passes over the
// shared-memory banks per step, the largest part of a pipe that was 68 % busy;
// 2d + 1 is then one packed add.  That alone measured the same (2000^2 92.8 and
// 92.1 ms); the room it frees holds more warps and packed rows.
template <bool FAR>
__device__ __forceinline__ void dist_pair(const float4* __restrict__ tab, int e, int u, float2& iv, float2& c)
{
    const float4 t = FAR ? dist_entry(e + u + 1) : tab[u];
    iv = make_float2(t.x, t.y);
    c = make_float2(t.z, t.w);
}
template <bool FAR>
__device__ __forceinline__ void dist_pair(const float2* __restrict__ tab, int e, int u, float2& iv, float2& c)
{
    if (FAR) {
        const float r = __frcp_rn((float)(e + u + 1));
        iv = make_float2(r, r);
    } else {
        // two entries per 16-byte load (the compiler keeps one of the two)
        const float4 t = *reinterpret_cast<const float4*>(tab + (u & ~1));
        iv = u % 2 ? make_float2(t.z, t.w) : make_float2(t.x, t.y);
    }
    const float b = (float)(2 * e + 3);
    c = __fadd2_rn(make_float2(b, b), make_float2((float)(2 * u), (float)(2 * u)));
}

// U steps of one lane's P POVs.  POV q at step u (distance d = e + 1 + u)
// sees target w[q + u + 1]; its slope is (target - h_q) * (1/d) in single
// precision, it is visible iff that slope is strictly above the running
// maximum M_q, and a visible target adds 2d + 1 to the POV's measure.  Two
// POVs share one packed multiply and one packed accumulate; the comparison and
// the maximum are scalar.  tab[u] holds (1/d, 1/d, 2d + 1, 2d + 1); a
// range-limited walk's last block counts only its first `nvalid` steps.
// With FAR the block's entries are computed (distances e + 1 .. e + U, past
// the end of a capped table) instead of read from tab[0 .. U).  T is the
// table's entry type (see dist_pair).
template <int P, int U, bool MASKED, bool FAR, class T>
__device__ __forceinline__ void sweep_block(const float* w, const T* __restrict__ tab, int e, const float* h,
                                            float* M, float2* acc2, int nvalid)
{
#pragma unroll
    for (int u = 0; u < U; ++u) {
        float2 iv, cpair;
        dist_pair<FAR>(tab, e, u, iv, cpair);
        if (MASKED && u >= nvalid) cpair = make_float2(0.f, 0.f);
#pragma unroll
        for (int q = 0; q < P; q += 2) {
            const float2 d = make_float2(__fsub_rn(w[q + u + 1], h[q]), __fsub_rn(w[q + u + 2], h[q + 1]));
            const float2 t = __fmul2_rn(d, iv);
            const float2 v = make_float2(fset_gt(t.x, M[q]), fset_gt(t.y, M[q + 1]));
            acc2[q / 2] = __ffma2_rn(v, cpair, acc2[q / 2]);
            M[q] = fmaxf(M[q], t.x);
            M[q + 1] = fmaxf(M[q + 1], t.y);
        }
    }
}

// Walks of more than LONG_WALK steps (rows longer than the constant, with a
// range beyond it) move their FP32 partial measures into integers every
// FLUSH_STEPS steps: a measure is a sum of odd integers 2d + 1 and stays exact
// in FP32 only below 2^24 (a walk of D steps sums to at most D^2 + 2D, and
// FLUSH_STEPS steps at d < 16384 add at most 1.1e7).  Shorter walks never
// flush (the LONG = false instantiation).
constexpr int LONG_WALK = 4000;
constexpr int FLUSH_STEPS = 336;   // a multiple of SMALL_UNROLL, LARGE_UNROLL and 24
// The maxima of a staged row that pruned walks test are kept at every
// ZS_STRIDE-th sample.
constexpr int ZS_STRIDE = 4;

// A warp item is one skewed row and one walk direction.  Its G groups of P
// consecutive POVs are taken in order (longest walks first) from a warp-local
// queue by whichever lane is free, so lanes stay busy whatever the walk
// lengths (and wherever pruning ends a walk early).  F holds the row (or the
// reversed row for backward walks) with -inf at its last sample and after it:
// the last target of a walk never adds area (its segment closes there), so it
// may be a sentinel that is never visible.  A walk's measure is
// cv = 1 + sum_{d=1}^{n-1} v_d (2d + 1) for n >= 1 targets, which is Alg. 8's
// sum of d^2 - open^2 over its closed segments plus the segment still open at
// the end (closed at the last target).
// Every target is walked; pruned launches take sweep_row_skip32.
//
// With LONG, `spill` is the lane's column (stride 32) of P integers.
template <int P, int U, bool LONG>
__device__ __forceinline__ void sweep_row(const float* __restrict__ F, const float4* __restrict__ tab, int tabn, int* __restrict__ cvrow,
                                          int* __restrict__ spill, int L, int K, float h0, bool rev, int lane)
{
    // the window is read as float4 from F + ROW_PADL + x0 + e (x0 = g P, e a
    // multiple of U): both must keep it 16-byte aligned
    static_assert(P % 4 == 0 && U % 4 == 0, "window loads must stay 16-byte aligned");
    const unsigned FULL = 0xffffffffu;
    const unsigned below = (1u << lane) - 1u;
    const float NEG = neg_inf();
    const int G = (L + P - 1) / P;
    const int klim = K - 1;          // last target distance that still adds area
    float h[P], M[P];
    float2 acc2[P / 2];
    int g = lane, next = 32;         // the lane's group; the first group nobody has taken
    int x0 = 0, e = 0, dlim = -1, seg = FLUSH_STEPS;
    bool klimited = false;

    auto start = [&]() {
        x0 = g * P;
        const int rowlim = L - 2 - x0;   // last target adding area, POV q = 0
        dlim = min(klim, rowlim);
        klimited = klim < rowlim;
        e = 0;
        seg = FLUSH_STEPS;
#pragma unroll
        for (int q = 0; q < P; ++q) { h[q] = __fadd_rn(F[ROW_PADL + x0 + q], h0); M[q] = NEG; }
#pragma unroll
        for (int q = 0; q < P / 2; ++q) acc2[q] = make_float2(0.f, 0.f);
        if (LONG) {
#pragma unroll
            for (int q = 0; q < P; ++q) spill[32 * q] = 0;
        }
    };
    if (g < G) start();
    for (;;) {
        const bool fin = g < G && e >= dlim;
        const unsigned need = __ballot_sync(FULL, fin);
        if (need) {
            if (fin) {
#pragma unroll
                for (int q = 0; q < P; ++q) {
                    const int x = x0 + q;
                    if (x < L) {
                        const int n = min(L - 1 - x, K);
                        const float s = q % 2 ? acc2[q / 2].y : acc2[q / 2].x;
                        cvrow[rev ? L - 1 - x : x] = n >= 1 ? 1 + (int)s + (LONG ? spill[32 * q] : 0) : 0;
                    }
                }
            }
            if (fin) {
                g = next + __popc(need & below);
                if (g < G) start(); else g = G;
            }
            next += __popc(need);
            if (!__any_sync(FULL, g < G)) break;
            continue;
        }
        if (g < G) {
            if (LONG && e >= seg) {
                seg += FLUSH_STEPS;
#pragma unroll
                for (int q = 0; q < P; q += 2) {
                    spill[32 * q] += __float2int_rz(acc2[q / 2].x);
                    spill[32 * (q + 1)] += __float2int_rz(acc2[q / 2].y);
                    acc2[q / 2] = make_float2(0.f, 0.f);
                }
            }
            const float* base = F + ROW_PADL + x0 + e;
            float w[P + U];
#pragma unroll
            for (int m = 0; m < P + U; m += 4) {
                const float4 v = *reinterpret_cast<const float4*>(base + m);
                w[m] = v.x; w[m + 1] = v.y; w[m + 2] = v.z; w[m + 3] = v.w;
            }
            // long walks may run past a capped distance table (LONG only)
            const bool far = LONG && e + U > tabn;
            if (klimited && e + U > dlim) {
                if (far) sweep_block<P, U, true, true>(w, tab, e, h, M, acc2, dlim - e);
                else sweep_block<P, U, true, false>(w, tab + e, e, h, M, acc2, dlim - e);
            } else {
                if (far) sweep_block<P, U, false, true>(w, tab, e, h, M, acc2, U);
                else sweep_block<P, U, false, false>(w, tab + e, e, h, M, acc2, U);
            }
            e += U;
        }
    }
}

// Maximum of the four samples 4 q .. 4 q + 3 of the staged row (ROW_PADL
// keeps them 16-byte aligned).
__device__ __forceinline__ float quad_max(const float* __restrict__ F, int q)
{
    const float4 v = *reinterpret_cast<const float4*>(F + ROW_PADL + 4 * q);
    return fmaxf(fmaxf(v.x, v.y), fmaxf(v.z, v.w));
}

// A maximum as the tests of a pruned walk take it: raised by 2^-20 of itself, for
// the roundings of the line it is compared with and the lo parts of the samples
// (-inf, of windows without samples, as the lowest float).
__device__ __forceinline__ float raised(float m)
{
    m = fmaxf(m, -3.4028234663852886e38f);
    return __fmaf_rn(0x1p-20f, fabsf(m), m);
}

// The maxima a pruned walk tests its blocks against (raised), one entry per
// ZS_STRIDE samples of the staged row F (L samples, -inf beyond them).
// warp-scans of 32 quads at a time: consecutive lanes read consecutive quads.
//
// Suffix maxima ZS[q] = max F[x >= 4 q], or prefix maxima ZS[q] = max
// F[x <= 4 q + 3] (PREFIX, backward walks), q <= (L - 1) / 4.
template <bool PREFIX>
__device__ __forceinline__ void end_max(const float* __restrict__ F, float* __restrict__ ZS, int L, int lane)
{
    static_assert(ZS_STRIDE == 4, "quads");
    const unsigned FULL = 0xffffffffu;
    const int nq = (L + 3) / 4;
    float carry = neg_inf();
    const int chunks = (nq + 31) / 32;
    for (int c = 0; c < chunks; ++c) {
        const int q = (PREFIX ? c : chunks - 1 - c) * 32 + lane;
        float m = q < nq ? quad_max(F, q) : neg_inf();
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const float t = PREFIX ? __shfl_up_sync(FULL, m, o) : __shfl_down_sync(FULL, m, o);
            if (PREFIX ? lane >= o : lane + o < 32) m = fmaxf(m, t);
        }
        m = fmaxf(m, carry);
        if (q < nq) ZS[q] = raised(m);
        carry = __shfl_sync(FULL, m, PREFIX ? 31 : 0);
    }
}

// Window maxima WM[j] = max F[x] over the P + U samples from 4 j - U on, the
// window of one block of a pruned walk that starts at sample 4 j - U, for
// j < (L + U + 3) / 4 (backward windows start up to U samples before the
// row).  `part` of `parts` warps each fill their share.
template <int P, int U>
__device__ __forceinline__ void window_max(const float* __restrict__ F, float* __restrict__ WM, int L, int lane,
                                           int part = 0, int parts = 1)
{
    static_assert(P % 4 == 0 && U % 4 == 0 && U <= ROW_PADL, "quads");
    const int n = (L + U + 3) / 4;
    for (int j = lane + 32 * part; j < n; j += 32 * parts) {
        float m = quad_max(F, j - U / 4);
#pragma unroll
        for (int k = 1; k < (P + U) / 4; ++k) m = fmaxf(m, quad_max(F, j - U / 4 + k));
        WM[j] = raised(m);
    }
}

// ------------------------------------------------ certified decisions --
//
// The fast path of a group of P POVs x0 .. x0 + P - 1 works on differences
// against the group's reference R = zh(x0) (the hi part of its first
// sample, a float): per block it forms, for every target t of its window,
// y_t = fl(fl(zh_t - R) + zl_t), and per POV q once g_q = fl(fl(fl(zh_q -
// R) + zl_q) + h0).  Then, for POV q and target t at distance d,
//     diff = fl(y_t - g_q),  x = fl(diff * fl(1/d)),  s = fl(x - M_q),
// visible iff s > 0 (the sign of s is exact), M_q = max(M_q, x).
//
// Error bound (u = 2^-24; D = z_t - h_q exact, theta = D / d, G = h_q - R):
//   |y_t - (z_t - R)| <= 2u |z_t - R| + 2 eta (eta: the staged heights'
//   error, which also covers the u |zl_t| <= 2^-48 |z_t| of adding zl_t
//   after the subtraction), |g_q - G| <= 3.01u |G| + 2.01u |h0| + |h0 -
//   float(h0)| + 2 eta, so |diff - D| <= 3.01u |D| + Eg with Eg = 5.02u |G|
//   + 2.01u |h0| + |h0 - float(h0)| + 4 eta, and |x - theta| <= 5.04u
//   |theta| + 1.01 Eg / d.
// M_q is the x of the last visible target a (the maximum is exact), so with
// every earlier decision right, comparing x_t with M_q errs by at most
//   5.04u (|theta_t| + |theta_a|) + 1.01 Eg (1/d_t + 1/d_a).
// When |s| >= delta the decision is right as soon as
//   delta (1 - u)(1 - 5.05u) >= 10.1u |M| + 1.02 Eg (1/d_t + 1/d_a)
// (|theta| <= |x| (1 + 5.1u) + Eg / d, |x_t| <= |M| + |x_t - M|).  Per block
// and POV the kernel takes
//   delta = CERT_REL * Mb + CERT_ABS * Eg' * (1/(e+1) + ia) + CERT_FLOOR,
// with Mb >= |M| over the whole block (the test runs after the block's
// steps, and M only rises within it, so Mb = max(|M| at its start, |M| at
// its end)), 1/(e+1) >= 1/d_t, ia >= 1/d_a (1/(e'+1) of the last block e' in
// which M rose; 1 at first), Eg' >= Eg from the group's largest |g_q|.
// Induction over the targets then makes every unflagged decision the exact
// one.  A POV with a step inside its margin leaves the block to the exact pass
// (flag_block); its M, the largest x whatever was decided, goes on.
constexpr float CERT_REL = 10.2f * 0x1p-24f * 1.01f;
constexpr float CERT_ABS = 1.03f * 1.01f;
constexpr float CERT_FLOOR = 0x1p-99f;
// Group size and steps per unrolled block of every certified walk.  A
// certified step takes about 40 % more instructions than an FP32 one and its
// state per POV twice the registers: groups of 4 POVs, and blocks short
// enough that the margin of a block (which grows with its window) stays
// tight.
#ifndef TVS_CERT_UNROLL
#define TVS_CERT_UNROLL 16
#endif
// The one-row-per-warp kernel (shorter rows, every walk staged forward)
// takes longer blocks: its lanes keep one margin per window block, and 24
// steps spread that block's overhead further (1000^2: 3 % faster); on the
// paired kernel's 2000-sample rows 24-step blocks were 4 % slower.
#ifndef TVS_CERT_UNROLL_SINGLE
#define TVS_CERT_UNROLL_SINGLE 24
#endif
constexpr int CERT_UNROLL = TVS_CERT_UNROLL;                 // paired-warp kernel
constexpr int CERT_UNROLL_SINGLE = TVS_CERT_UNROLL_SINGLE;   // one-row-per-warp kernel
#ifndef TVS_CERT_POV
#define TVS_CERT_POV SMALL_POV
#endif
constexpr int CERT_POV = TVS_CERT_POV;
static_assert(CERT_POV + CERT_UNROLL <= ROW_PADR && CERT_POV + CERT_UNROLL_SINGLE <= ROW_PADR,
              "a forward block's window reads up to P + U samples on");
#ifndef TVS_SKIP_READY
#define TVS_SKIP_READY 22
#endif
constexpr int SKIP_READY = TVS_SKIP_READY;   // lanes with a block before a pruned walk evaluates
#ifndef TVS_SKIP_RESTART
#define TVS_SKIP_RESTART 4
#endif
constexpr int SKIP_RESTART = TVS_SKIP_RESTART;   // finished lanes before a pruned walk replaces groups
// Blocks a searching lane tests at a time: on long rows most tests pass and
// their latency is shared by more of them, on packed short rows few blocks
// are left (2000^2 89.1 ms with 4, 88.0 with 6; 60 small tiles 14.7 with 3,
// 15.0 with 4, 15.3 with 6).
#ifndef TVS_SKIP_TESTS
#define TVS_SKIP_TESTS 6
#endif
#ifndef TVS_PACK_TESTS
#define TVS_PACK_TESTS 3
#endif
constexpr int SKIP_TESTS = TVS_SKIP_TESTS;
constexpr int PACK_TESTS = TVS_PACK_TESTS;
// Steps per pass of a block's evaluation loop: whole blocks save the loop where
// registers allow (rows of a warp's own, 1000^2: 19.3 ms with 8, 18.3 with 16);
// the kernel of shared rows, which has code for both walk directions, spills
// (2000^2: 87.2 and 97.4 ms).
#ifndef TVS_SKIP_CHUNK
#define TVS_SKIP_CHUNK 8
#endif
#ifndef TVS_SINGLE_CHUNK
#define TVS_SINGLE_CHUNK 16
#endif
#ifndef TVS_PACK_CHUNK
#define TVS_PACK_CHUNK 8
#endif
#ifndef TVS_FP32_CHUNK
#define TVS_FP32_CHUNK 16
#endif
constexpr int SKIP_CHUNK = TVS_SKIP_CHUNK, SINGLE_CHUNK = TVS_SINGLE_CHUNK, PACK_CHUNK = TVS_PACK_CHUNK;
constexpr int FP32_CHUNK = TVS_FP32_CHUNK;
#ifndef TVS_SKIP_UNROLL
#define TVS_SKIP_UNROLL 16
#endif
// Samples after a staged row that a pruned walk's windows read.
constexpr int SKIP_PADR = CERT_POV + TVS_SKIP_UNROLL + 8;
#ifndef TVS_SKIP_WARPS
#define TVS_SKIP_WARPS 16
#endif
constexpr int SKIP_WARPS = TVS_SKIP_WARPS;       // most warps of a pruned certified CTA of warp pairs
// and of rows of a warp's own: 20 when each warp holds one (1000^2 20.5 ms with
// 16), 16 when that leaves room for two or more (60 small tiles 15.0 ms with
// 20 warps, 14.5 with 16 and more rows in each).
#ifndef TVS_SINGLE_WARPS
#define TVS_SINGLE_WARPS 20
#endif
#ifndef TVS_PACK_WARPS
#define TVS_PACK_WARPS 16
#endif
constexpr int SINGLE_WARPS = TVS_SINGLE_WARPS, PACK_WARPS = TVS_PACK_WARPS;
#ifndef TVS_FP32_WARPS
#define TVS_FP32_WARPS 20
#endif
// Pruned FP32 decisions (1201 x 777: 12.5 ms with 16 warps, 11.8 with 20).
constexpr int FP32_WARPS = TVS_FP32_WARPS;
constexpr int SKIP_UNROLL = TVS_SKIP_UNROLL;   // steps per block of a pruned walk
static_assert(SKIP_UNROLL <= ROW_PADL && CERT_POV + SKIP_UNROLL <= ROW_PADR && FLUSH_STEPS % SKIP_UNROLL == 0,
              "pads and flushes of a pruned walk");
static_assert(CERT_UNROLL <= ROW_PADL, "a backward block's window starts up to U samples before the row");
static_assert(FLUSH_STEPS % CERT_UNROLL == 0, "long walks flush on block boundaries");
// A certified kernel with U-step blocks stores distance entry m at slot m +
// m / U.  A lane reads entries e .. e + U - 1 of its own block start e (a
// multiple of U); groups of different lengths leave the lanes of a warp at
// different e, and unskewed such reads would fall on a few of the eight
// 16-byte bank groups.  Skewed, entry u of block k sits in bank group
// ((U + 1) k + u) mod 8 (U a multiple of 8), which spreads blocks k over all
// eight.  Tables are sized for the shorter block, which needs the most slots.
static_assert(SKIP_UNROLL % 8 == 0 && CERT_UNROLL % 8 == 0 && CERT_UNROLL_SINGLE % 8 == 0,
              "skewed blocks cover the eight bank groups");
// A pruned kernel's 8-byte entry m sits at slot m + 2 (m / SKIP_UNROLL) (two
// slots: the blocks stay 16-byte aligned), which spreads the blocks alike.
constexpr int TAB_SKEW_MIN = std::min(CERT_UNROLL, CERT_UNROLL_SINGLE);
// Floats of a table of `entries` distances, a multiple of 4, and the most
// entries that fit `floats`.
int tab_floats_for(int entries, bool prune, bool cert)
{
    if (prune) return 2 * ((entries + 2 * (entries / SKIP_UNROLL) + 2 + 1) & ~1);
    return 4 * (cert ? (entries + entries / TAB_SKEW_MIN + 1 + 1) & ~1 : entries);
}
size_t tab_entries_fit(size_t floats, bool prune, bool cert)
{
    if (prune) return floats / 2 < 4 ? 0 : (floats / 2 - 4) * SKIP_UNROLL / (SKIP_UNROLL + 2);
    return cert ? (floats / 4 < 2 ? 0 : (floats / 4 - 2) * TAB_SKEW_MIN / (TAB_SKEW_MIN + 1)) : floats / 4;
}
// Far from the POV one margin serves several window blocks: from step
// CERT_NEAR on a margin block is 2 window blocks long, from CERT_FAR on 4
// (while the group's walks have that many steps left), so that the finish
// vote, the margins and the last-rise update are taken once per 32 or 64
// steps.  Near the POV, where the margin's 1/(e+1) terms
// fall fastest, every window block takes its own.  The lanes of a warp run
// as many window blocks as the longest of their margin blocks (the others
// wait), which pays only on long rows: the paired-warp kernel takes these
// tiers, the one-row-per-warp kernel (shorter rows) one window block per
// margin.  A pruned walk checks its stopping bound once per margin block and
// most pruned walks are short, so pruned launches keep one window block per
// margin too.
#ifndef TVS_CERT_NEAR
#define TVS_CERT_NEAR 64
#endif
#ifndef TVS_CERT_FAR
#define TVS_CERT_FAR 256
#endif
#ifndef TVS_CERT_PACKADD
#define TVS_CERT_PACKADD 1
#endif
constexpr int CERT_NEAR = TVS_CERT_NEAR;
constexpr int CERT_FAR = TVS_CERT_FAR;

// Targets per lane per chunk of an exact walk.
constexpr int XW_KPL = 8;

// 1.0f if s >= 2^-100 (s > 0 and outside every margin, which is at least
// CERT_FLOOR), 0.0f if s <= 0, a fraction only inside the margin.
__device__ __forceinline__ float sat_pos(float s)
{
    float v;
    asm("fma.rn.sat.f32 %0, %1, %2, %3;" : "=f"(v) : "f"(s), "f"(0x1p100f), "f"(0.0f));
    return v;
}

// Whether a flagged POV's whole walk will be flagged: its group's error bound
// (c2e, a height at distance 1, at least a millimetre) exceeds the running
// maximum.  That is so beside a cell kilometres and more above or below the
// ground (-1e9), which spoils its group's reference; on even ground the bound is
// some 10^-10 m.  Such a walk's rest is handed over at its first flag, not at
// its second.
__device__ __forceinline__ bool beside_outlier(float c2e, float M) { return c2e > fmaxf(fabsf(M), 0x1p-10f); }

// What names a walk's row in the flag buffer: direction (< 4096), skewed row
// (< 32768) and walk direction.
__device__ __forceinline__ int row_key(int dir, int p, bool back) { return dir << 16 | p << 1 | (back ? 1 : 0); }

// The measure the sweep writes for a flagged walk that found the flag buffer
// full: the scan after the exact pass looks for negative measures.
constexpr int CV_FLAGGED = (int)0x80000000;

// A staged row as its certified walks see it.
struct CertRow {
    const float* H;      // staged hi parts (index 0 = first sample)
    const float* Lo;     // staged lo parts
    int L, K;
    float h0;
    float eh0, el0;      // hi and lo parts of the first sample (a sentinel in H, Lo)
    float ehL, elL;      // and of the last one
    float eg0;           // 2.01u |h0| + |h0 - float(h0)| + 4 eta: the parts of Eg common to the row's groups
    float zmax;          // the row's largest |elevation|
    int* cvrow;
    int key;             // row_key of the row's walks
    bool rev_staged;     // the staged row is reversed: staged x is row sample L - 1 - x
};

// The certified row of a staged item.  eta bounds the staged heights' error,
// plus h0's split (h0 = float(h0) + h0_lo to 2^-48).
__device__ __forceinline__ CertRow cert_row(const SweepParams& sp, const ItemRow& it, const float* Fh,
                                            const float* Fl, const float* ends, float zmax, int* cv, bool rev_staged)
{
    const float eta = 0x1p-42f * (zmax + fabsf(it.h0)) + 0x1p-126f;
    CertRow r;
    r.H = Fh + ROW_PADL;
    r.Lo = Fl + ROW_PADL;
    r.L = it.L;
    r.K = it.K;
    r.h0 = it.h0;
    r.eh0 = ends[0];
    r.el0 = ends[1];
    r.ehL = ends[2];
    r.elL = ends[3];
    r.eg0 = 2.01f * 0x1p-24f * fabsf(it.h0) + fabsf(sp.dirs[it.dir].h0_lo) * 1.0001f + 4.04f * eta;
    r.zmax = zmax;
    r.cvrow = cv + it.rowbase;
    r.key = row_key(it.dir, it.p, it.rev);
    r.rev_staged = rev_staged;
    return r;
}

// Hi and lo parts of POV x's ground height (the end samples are sentinels in
// the staged arrays; their real parts are kept aside).
__device__ __forceinline__ void pov_hl(const CertRow& r, int x, float& hi, float& lo)
{
    if (x == 0) { hi = r.eh0; lo = r.el0; }
    else if (x == r.L - 1) { hi = r.ehL; lo = r.elL; }
    else { hi = r.H[x]; lo = r.Lo[x]; }
}

// The sample field of a flag entry holds the entry's kind above bit 16: the
// block's running maximum before its first step e0 lies in the block p0 in
// which the walk's maximum last rose for certain, or (FLAG_PREFIX, when a block
// after it was flagged) anywhere from there on; above that the lengths of both
// blocks in eighths.  The fourth field holds e0 and p0.  A FLAG_PREFIX entry
// is all that is left of its walk from e0 on, not one block: where a walk is
// flagged all along (ties) each of its entries would walk again from p0 (400^2,
// 36 directions: level ground seen from its own height 247 ms block by block,
// 242 so; steps of whole metres 39.2 and 37.0).  Rare elsewhere (90 of 7.3
// million entries of 12 mixed tiles), where it costs a little (4000^2, 10 km:
// 204.9 and 206.9 ms; 100 x 16384: 27.8 and 28.8).
// FLAG_WALK is a whole walk, decided in FP64 (hand_over_row).
constexpr int FLAG_BLOCK = 1, FLAG_PREFIX = 2, FLAG_WALK = 3;
static_assert(2 * 14 < 32, "e0 and p0 (< 16384) share a word");

// A staged row as the pruned certified walks see it (in shared memory, so that
// the lanes of a warp may be on different rows).
struct __align__(16) SkipRow {
    int L, K;
    int key;             // row_key of its walks
    int rev;             // staged x is row sample L - 1 - x
    float ends[4];       // hi and lo parts of the first and of the last sample (sentinels when staged)
    float h0;
    float eg0;           // as CertRow
    float zmax;          // the row's largest |elevation|
    int pad;
    int* cv;             // the row's measures
    long long pad2;
};
static_assert(sizeof(SkipRow) == 64, "16 floats");
constexpr int SKIP_ROW_FLOATS = 16;
#ifndef TVS_PACK_MAX_LG
#define TVS_PACK_MAX_LG 3
#endif
constexpr int PACK_MAX_LG = TVS_PACK_MAX_LG;           // at most 8 staged rows per warp
#ifndef TVS_PACK_MIN_CLAIMS
#define TVS_PACK_MIN_CLAIMS 3
#endif
constexpr int PACK_MIN_CLAIMS = TVS_PACK_MIN_CLAIMS;   // packs per warp that packing must leave

// The staged lo array's first word, before the samples that any window reads:
// zero when a row is staged, and set once the row's walks found the flag buffer
// full.  (Warps that share a row may set it together; volatile, as nothing
// orders them.)
__device__ __forceinline__ volatile int* full_mark(const float* lo)
{
    static_assert(CERT_UNROLL < ROW_PADL && SKIP_UNROLL < ROW_PADL, "the pad is longer than a window");
    return reinterpret_cast<volatile int*>(const_cast<float*>(lo) - ROW_PADL);
}

// Reserves `count` entries of the flag buffer; returns the first, past its end
// (and says in the third counter that a flag found it full) when there are none.
__device__ __forceinline__ unsigned reserve_flags(const SweepParams& sp, int count)
{
    const unsigned cap = (unsigned)sp.flag_cap;
    // (a full buffer's counter stays where it is)
    unsigned at = *reinterpret_cast<volatile unsigned*>(sp.flag_count);
    if (at < cap) at = atomicAdd(sp.flag_count, (unsigned)count);
    if (at + (unsigned)count > cap) sp.flag_count[2] = 1u;
    return at;
}

// The same for a pruned walk, by its row's mark.  Each flag used to ask the
// counter, also once the buffer was full, and where many walks are flagged they
// queued on its address (100 x 100 with 1 % cells of -1e9, 60 directions: sweep 706
// us with as many instructions as level ground's 64; the call 1.35 -> 0.76 ms so,
// 220 x 310 4.25 -> 2.08).  One reservation for all lanes of a warp was no better
// (0.85, 2.16) and cost the other walks more (4000^2, 10 km: 205.5 before, 208.2
// so, 213.5).  Unpruned walks go by whether their group has lost a flag: the mark
// costs them more (2000^2, 48 directions: 87.5 before, 88.3 so, 90.1 with it).
__device__ __forceinline__ unsigned flag_slots(const SweepParams& sp, int count, volatile int* full)
{
    const unsigned cap = (unsigned)sp.flag_cap;
    if (*full) return cap;
    const unsigned at = reserve_flags(sp, count);
    if (at + (unsigned)count > cap) *full = 1;
    return at;
}

// Hands the len-step block at e0 of row sample x's walk to the exact pass in
// entry `at`, p0 (plen steps) the block of its last rise; false when that is
// past the buffer.
__device__ __forceinline__ bool flag_block(const SweepParams& sp, unsigned at, int key, float zmax, int x, int e0,
                                           int len, int p0, int plen, int kind)
{
    if (at >= (unsigned)sp.flag_cap) return false;
    sp.flag_buf[at] = make_int4(key, x | kind << 16 | (len >> 3) << 18 | (plen >> 3) << 22, __float_as_int(zmax),
                                e0 | p0 << 14);
    return true;
}

// Hands every walk of a row to the exact pass, which walks it in FP64: rows
// that hold a height beyond what the margins cover (df::beyond).  Flagged block
// by block such a row's walks were wrong where differences overflowed, and
// walked in single precision, double-float and twice in FP64 (220 x 310, 24
// directions, one cell of -3.4e38: 0.97 ms, 0.45 so; 0.58 when every flag sent
// its whole walk to the exact pass).  Lanes take samples first, first + step, ...
__device__ __forceinline__ void hand_over_row(const SweepParams& sp, const ItemRow& it, bool back, float zmax, int* cv,
                                              int first, int step, const float* lo)
{
    int* cvrow = cv + it.rowbase;
    const int key = row_key(it.dir, it.p, back);
#pragma unroll 1
    for (int x = first; x < it.L; x += step) {
        const int n = min(back ? x : it.L - 1 - x, it.K);
        int m = n >= 1 ? 1 : 0;
        if (n >= 2 && !flag_block(sp, flag_slots(sp, 1, full_mark(lo)), key, zmax, x, 0, 0, 0, 0, FLAG_WALK))
            m = CV_FLAGGED;
        cvrow[x] = m;
    }
}

// Fills a staged row's SkipRow (the ends are there already), walked backward
// with `back`, staged reversed with `rev`; false when a walk of
// the row could leave its arrays or the distance table (windows start at most
// SKIP_UNROLL samples before the row and end before sample L + P + U).
__device__ __forceinline__ bool skip_row(const SweepParams& sp, const ItemRow& it, bool back, float zmax, int* cv,
                                         bool rev, bool longw, SkipRow* r)
{
    const float eta = 0x1p-42f * (zmax + fabsf(it.h0)) + 0x1p-126f;
    r->L = it.L;
    r->K = it.K;
    r->key = row_key(it.dir, it.p, back);
    r->rev = rev;
    r->h0 = it.h0;
    r->eg0 = 2.01f * 0x1p-24f * fabsf(it.h0) + fabsf(sp.dirs[it.dir].h0_lo) * 1.0001f + 4.04f * eta;
    r->zmax = zmax;
    r->cv = cv + it.rowbase;
    return in_range(ROW_PADL + it.L + CERT_POV + SKIP_UNROLL, sp.half, 19) &&
           in_range((it.L - 1) / ZS_STRIDE, sp.zs_len, 9) &&
           in_range((it.L + SKIP_UNROLL + 3) / ZS_STRIDE - 1, sp.wm_len, 10) &&
           (longw || in_range(min(it.K, it.L) + SKIP_UNROLL - 1, sp.inv_len, 11));
}

// Writes the measures of a finished group of P POVs (pov_x(q): staged sample
// of POV q; lost: POVs whose walk is taken again whole).
template <int P, bool LONG, class X, class N, class S>
__device__ __forceinline__ void finish_group(const SweepParams& sp, const CertRow& r, unsigned lost, X pov_x, N walk_n,
                                             S measure, const int* spill)
{
#pragma unroll
    for (int q = 0; q < P; ++q) {
        const int x = pov_x(q);
        if (x >= r.L) continue;
        const int cv = walk_n(x) >= 1 ? 1 + (int)measure(q) + (LONG ? spill[32 * q] : 0) : 0;
        r.cvrow[r.rev_staged ? r.L - 1 - x : x] = (lost >> q) & 1u ? CV_FLAGGED : cv;
    }
}

// What the exact walk of a sample needs.
struct ExactCtx {
    int L, K;
    float h0h, h0l;      // h0 = h0h + h0l (to 2^-48)
    float eta;           // bound of the blended heights' error, plus h0's split
    int* cvrow;
    bool bwd;            // walks go toward lower sample indices
    const DirDev* dir;
    const JobDev* job;
    int p, jlo;
};

__device__ __forceinline__ ExactCtx exact_ctx(const SweepParams& sp, const ItemRow& it, float zmax)
{
    ExactCtx c;
    c.dir = sp.dirs + it.dir;
    c.job = sp.jobs + c.dir->job;
    c.L = it.L;
    c.K = it.K;
    c.h0h = it.h0;
    c.h0l = c.dir->h0_lo;
    c.eta = 0x1p-42f * (zmax + fabsf(it.h0)) + 0x1p-126f;
    c.cvrow = (it.rev ? sp.cv_bwd : sp.cv_fwd) + it.rowbase;
    c.bwd = it.rev;
    c.p = it.p;
    c.jlo = it.jlo;
    return c;
}

// Elevations that sample xs of the row blends (row a, row a + 1) and the
// weight's fraction.
__device__ __forceinline__ void dem_pair(const ExactCtx& c, int xs, float& va, float& vb, unsigned& fr)
{
    const DirDev& d = *c.dir;
    const int j = c.jlo + xs;
    const unsigned long long y = (unsigned long long)j * d.t_fx;
    const int a = c.p - d.D + (int)(y >> 32);
    fr = (unsigned)y;
    int st;
    const long long idx = view_index(d, c.job->cols, a, j, &st);
    const long long cells = (long long)c.job->rows * c.job->cols;
    va = in_range(idx, cells, 16) ? c.job->dem[idx] : 0.f;
    vb = fr != 0u ? (in_range(idx + st, cells, 17) ? c.job->dem[idx + st] : 0.f) : va;
}

// Hi and lo parts of sample xs, as the staging forms them.
__device__ __forceinline__ void dem_hl(const ExactCtx& c, int xs, float& hi, float& lo)
{
    float va, vb;
    unsigned fr;
    dem_pair(c, xs, va, vb, fr);
    df::df_blend(va, vb, fr, hi, lo);
}

// FP64 height of sample xs exactly as the FP64 definition forms it:
// (1 - r) * a + r * b with r = fr / 2^32, every operation rounded.
__device__ __forceinline__ double z64_at(const ExactCtx& c, int xs)
{
    float va, vb;
    unsigned fr;
    dem_pair(c, xs, va, vb, fr);
    if (fr == 0u) return (double)va;
    const double r = __dmul_rn((double)fr, 0x1p-32);
    return __dadd_rn(__dmul_rn(__dsub_rn(1.0, r), (double)va), __dmul_rn(r, (double)vb));
}

__device__ __forceinline__ int warp_sum(int v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Targets per lane of an exact walk's next chunk, `left` targets before its end.
template <int KPL>
__device__ __forceinline__ int chunk_targets(int left) { return min(KPL, (left + 31) / 32); }

// The FP64 walk of POV x (Alg. 8 in double precision: theta = (z - h) / d
// rounded once, strict comparison with the running maximum): sum of 2d + 1
// over the visible targets d = from + 1 .. last.  Warp-cooperative: up to 32 x
// XW_KPL targets per chunk, a warp max-scan gives each lane the running maximum
// before its first target.  Bound by the FP64 pipe (a warp's instruction holds it
// 16 cycles), so a chunk of fewer targets gives each lane fewer instead of
// leaving lanes idle (100 x 100 level ground seen from its own height, 60
// directions, whose walks have 50 targets: 21.8 -> 7.3 ms).
__device__ __noinline__ int fp64_walk(const ExactCtx& c, int x, int from, int last, int lane)
{
    const double h = __dadd_rn(z64_at(c, x), c.job->h0);
    const int dir = c.bwd ? -1 : 1;
    double run = -__longlong_as_double(0x7ff0000000000000LL);
    int acc = 0;
    for (int base = 1; base <= last; ) {
        const int kpl = chunk_targets<XW_KPL>(last - base + 1);
        double th[XW_KPL];
        double m = run;
        const int d0 = base + lane * kpl, dl = min(d0 + kpl - 1, last);   // the lane's targets
#pragma unroll
        for (int k = 0; k < XW_KPL; ++k) {
            const int d = d0 + k;
            th[k] = d <= dl ? __ddiv_rn(__dsub_rn(z64_at(c, x + dir * d), h), (double)d) : run;
            m = fmax(m, th[k]);
        }
        double incl = m;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl = fmax(incl, t);
        }
        double cur = __shfl_up_sync(0xffffffffu, incl, 1);
        if (lane == 0) cur = run;
        cur = fmax(cur, run);
#pragma unroll
        for (int k = 0; k < XW_KPL; ++k) {
            const int d = d0 + k;
            if (d > dl) break;
            if (th[k] > cur) { acc += d > from ? 2 * d + 1 : 0; cur = th[k]; }
        }
        run = fmax(run, __shfl_sync(0xffffffffu, incl, 31));
        base += 32 * kpl;
    }
    return warp_sum(acc);
}

// The double-float walk of POV x over the targets a0 < d <= a1 and then
// b0 < d <= b1: the sum of 2d + 1 over the second span's visible targets,
// given that the largest slope before it lies in the first (a1 == a0: no
// earlier target).  32 x KPL targets per chunk.  Every comparison is proved by
// a margin (slope error <= 2^-45 |theta| + eta / d each); one inside its
// margin sets *esc and the FP64 walk decides instead.
template <int KPL>
__device__ __forceinline__ int df_walk(const ExactCtx& c, int x, int a0, int a1, int b0, int b1, int lane,
                                       bool* esc_out)
{
    const float NEG = neg_inf();
    const int dir = c.bwd ? -1 : 1;
    const int na = a1 - a0, total = na + b1 - b0;
    float hh, hl;
    {
        float zh, zl;
        dem_hl(c, x, zh, zl);
        float s, e;
        df::two_sum(zh, c.h0h, s, e);
        e = __fadd_rn(e, __fadd_rn(zl, c.h0l));
        df::two_sum(s, e, hh, hl);
    }
    float rh = NEG, rl = 0.f;
    int rd = 1;
    int acc = 0;
    bool esc = false;
    for (int base = 0; base < total; ) {
        const int kpl = chunk_targets<KPL>(total - base);
        float th[KPL], tl[KPL], iv[KPL];
        float mh = NEG, ml = 0.f;
        int md = 1;
        const int i0 = base + lane * kpl, il = min(i0 + kpl, total);   // the lane's targets
        auto dist = [&](int i) { return i < na ? a0 + 1 + i : b0 + 1 + i - na; };
#pragma unroll
        for (int k = 0; k < KPL; ++k) {
            const int i = i0 + k, d = dist(i);
            th[k] = NEG; tl[k] = 0.f; iv[k] = 1.f;
            if (i < il) {
                iv[k] = __frcp_rn((float)d);
                float zh, zl;
                dem_hl(c, x + dir * d, zh, zl);
                df::df_slope_iv(zh, zl, hh, hl, d, iv[k], th[k], tl[k]);
                if (df::df_gt(th[k], tl[k], mh, ml)) { mh = th[k]; ml = tl[k]; md = d; }
            }
        }
        // inclusive max-scan over the lanes
        float ph = mh, pl = ml;
        int pd = md;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const float qh = __shfl_up_sync(0xffffffffu, ph, o);
            const float ql = __shfl_up_sync(0xffffffffu, pl, o);
            const int qd = __shfl_up_sync(0xffffffffu, pd, o);
            if (lane >= o && df::df_gt(qh, ql, ph, pl)) { ph = qh; pl = ql; pd = qd; }
        }
        float ch = __shfl_up_sync(0xffffffffu, ph, 1);
        float cl = __shfl_up_sync(0xffffffffu, pl, 1);
        int cd = __shfl_up_sync(0xffffffffu, pd, 1);
        if (lane == 0 || df::df_gt(rh, rl, ch, cl)) { ch = rh; cl = rl; cd = rd; }
        float icd = __frcp_rn((float)cd);
#pragma unroll
        for (int k = 0; k < KPL; ++k) {
            const int i = i0 + k, d = dist(i);
            if (i >= il) break;
            bool v = true;                           // the first target (no earlier one) is visible
            if (ch > NEG) {
                float s, e;
                df::two_sum(th[k], -ch, s, e);
                const float dh = __fadd_rn(s, __fadd_rn(e, __fsub_rn(tl[k], cl)));
                const float marg = __fmaf_rn(0x1p-40f, fabsf(th[k]) + fabsf(ch), 4.04f * c.eta * (iv[k] + icd)) +
                                   0x1p-120f;
                if (!(fabsf(dh) > marg)) esc = true;
                v = dh > 0.f;
            }
            if (v && i >= na) acc += 2 * d + 1;
            if (df::df_gt(th[k], tl[k], ch, cl)) { ch = th[k]; cl = tl[k]; cd = d; icd = iv[k]; }
        }
        const float lh = __shfl_sync(0xffffffffu, ph, 31);
        const float ll = __shfl_sync(0xffffffffu, pl, 31);
        const int ld = __shfl_sync(0xffffffffu, pd, 31);
        if (df::df_gt(lh, ll, rh, rl)) { rh = lh; rl = ll; rd = ld; }
        base += 32 * kpl;
    }
    *esc_out = __any_sync(0xffffffffu, esc);
    return warp_sum(acc);
}

// Exact measure of POV x of the row, written by lane 0.  count[0] and count[1]
// are the warp's exact and FP64 walks so far.
__device__ __noinline__ void exact_walk(const ExactCtx& c, int x, int lane, unsigned* count)
{
    const int n = min(c.bwd ? x : c.L - 1 - x, c.K);
    int cv;
    if (n < 2) {
        cv = n < 1 ? 0 : 1;
    } else {
        bool esc = c.eta >= 0x1p-42f * df::BEYOND;
        const int s = esc ? 0 : df_walk<XW_KPL>(c, x, 0, 0, 0, n - 1, lane, &esc);
        cv = 1 + (esc ? fp64_walk(c, x, 0, n - 1, lane) : s);
        ++count[0];
        if (esc) ++count[1];
    }
    if (lane == 0 && in_range(x, c.L, 14)) c.cvrow[x] = cv;
}

// Adds to POV x's measure what the targets of block e0 (len steps; FLAG_PREFIX
// and FLAG_WALK: and all after it) add, decided exactly; kind, p0 and plen as in the flag entry.
__device__ __noinline__ void exact_block(const ExactCtx& c, int x, int e0, int len, int p0, int plen, int kind,
                                         int lane, unsigned* count)
{
    const int n = min(c.bwd ? x : c.L - 1 - x, c.K);
    const int last = kind == FLAG_BLOCK ? min(n - 1, e0 + len) : n - 1;
    if (last <= e0) return;
    bool esc = kind == FLAG_WALK;
    const int s = kind == FLAG_WALK ? 0 : kind == FLAG_PREFIX ? df_walk<XW_KPL>(c, x, p0, e0, e0, last, lane, &esc)
                                      : df_walk<4>(c, x, p0, min(p0 + plen, e0), e0, last, lane, &esc);
    const int add = esc ? fp64_walk(c, x, e0, last, lane) : s;
    if (lane == 0 && in_range(x, c.L, 14) && add) atomicAdd(c.cvrow + x, add);
    ++count[0];
    if (esc) ++count[1];
}

// The same for one FLAG_BLOCK entry of at most 16 steps in either block per half-warp (h: the lane's place in its
// half; valid: the half has an entry): one target of the earlier block and one
// of the flagged block per lane.  The maximum of the earlier block is one of
// its near-tied largest slopes, so its error is taken at that block's first
// distance.  Returns whether the half's decisions need the FP64 walk (nothing
// is added then).
__device__ __forceinline__ bool exact_half(const ExactCtx& c, bool valid, int x, int e0, int len, int p0, int plen,
                                           int lane)
{
    const unsigned FULL = 0xffffffffu;
    const float NEG = neg_inf();
    const int h = lane & 15, dir = c.bwd ? -1 : 1;
    int da = 0, db = 0;
    if (valid) {
        const int last = min(min(c.bwd ? x : c.L - 1 - x, c.K) - 1, e0 + len);
        if (p0 + 1 + h <= min(p0 + plen, e0)) da = p0 + 1 + h;
        if (e0 + 1 + h <= last) db = e0 + 1 + h;
    }
    float ah = NEG, al = 0.f, bh = NEG, bl = 0.f, iv = 1.f;
    if (valid) {
        float zh, zl, hh, hl, s, e;
        dem_hl(c, x, zh, zl);
        df::two_sum(zh, c.h0h, s, e);
        e = __fadd_rn(e, __fadd_rn(zl, c.h0l));
        df::two_sum(s, e, hh, hl);
        if (da) {
            dem_hl(c, x + dir * da, zh, zl);
            df::df_slope(zh, zl, hh, hl, da, ah, al);
        }
        if (db) {
            iv = __frcp_rn((float)db);
            dem_hl(c, x + dir * db, zh, zl);
            df::df_slope_iv(zh, zl, hh, hl, db, iv, bh, bl);
        }
    }
    // the maximum before the block, and before each of its targets
    float ph = bh, pl = bl;
#pragma unroll
    for (int o = 1; o < 16; o <<= 1) {
        const float qh = __shfl_xor_sync(FULL, ah, o), ql = __shfl_xor_sync(FULL, al, o);
        if (df::df_gt(qh, ql, ah, al)) { ah = qh; al = ql; }
        const float rh = __shfl_up_sync(FULL, ph, o, 16), rl = __shfl_up_sync(FULL, pl, o, 16);
        if (h >= o && df::df_gt(rh, rl, ph, pl)) { ph = rh; pl = rl; }
    }
    float ch = __shfl_up_sync(FULL, ph, 1, 16), cl = __shfl_up_sync(FULL, pl, 1, 16);
    if (h == 0 || df::df_gt(ah, al, ch, cl)) { ch = ah; cl = al; }
    bool esc = false;
    int add = 0;
    if (db) {
        bool v = true;                       // the first target (no earlier one) is visible
        if (ch > NEG) {
            float s, e;
            df::two_sum(bh, -ch, s, e);
            const float dh = __fadd_rn(s, __fadd_rn(e, __fsub_rn(bl, cl)));
            const float marg = __fmaf_rn(0x1p-40f, fabsf(bh) + fabsf(ch),
                                         4.04f * c.eta * (iv + __frcp_rn((float)(p0 + 1)))) + 0x1p-120f;
            esc = !(fabsf(dh) > marg);
            v = dh > 0.f;
        }
        if (v) add = 2 * db + 1;
    }
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) add += __shfl_xor_sync(FULL, add, o);
    const bool any = (__ballot_sync(FULL, esc) >> (lane & 16) & 0xffffu) != 0u;
    if (valid && !any && h == 0 && add && in_range(x, c.L, 14)) atomicAdd(c.cvrow + x, add);
    return any;
}

// min(a, |b|, |c|).  TVS_CERT_MIN3 selects the three-input minimum of
// sm_100+ (one instruction for two steps of a POV) or two chained minima.
#ifndef TVS_CERT_MIN3
#define TVS_CERT_MIN3 1
#endif
__device__ __forceinline__ float min_abs2(float a, float b, float c)
{
#if TVS_CERT_MIN3
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(fabsf(b)), "f"(fabsf(c)));
    return r;
#else
    return fminf(fminf(a, fabsf(b)), fabsf(c));
#endif
}

// U certified steps of one lane's P POVs (see the derivation above), two
// steps at a time.  y[m] is the window's target x0 + e + m relative to R,
// ng2 the POVs' heights relative to R, negated, in pairs (q, q + 1).  mn[q]
// keeps the smallest |s| of the POV's steps: the block's margin test (mn <
// delta) runs once at its end.  With PACK the differences of a pair of POVs
// go through one packed add wherever their two targets form an aligned pair
// of the window (y[2j], y[2j + 1]: every other step); y - g and y + (-g)
// round alike.
template <int P, int U, bool MASKED, bool FAR, bool PACK, class T>
__device__ __forceinline__ void cert_block(const float* y, const T* __restrict__ tab, int e, const float2* ng2,
                                           float2* M2, float2* acc2, float* mn, int nvalid)
{
    static_assert(U % 2 == 0, "steps go in pairs");
#pragma unroll
    for (int u = 0; u < U; u += 2) {
        float2 sv[2][P / 2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int w = u + k;
            float2 iv, cp;
            dist_pair<FAR>(tab, e, w, iv, cp);
            if (MASKED && w >= nvalid) cp = make_float2(0.f, 0.f);
#pragma unroll
            for (int q = 0; q < P; q += 2) {
                const float2 d = (PACK && (q + w + 1) % 2 == 0)
                                     ? __fadd2_rn(make_float2(y[q + w + 1], y[q + w + 2]), ng2[q / 2])
                                     : make_float2(__fadd_rn(y[q + w + 1], ng2[q / 2].x),
                                                   __fadd_rn(y[q + w + 2], ng2[q / 2].y));
                const float2 x = __fmul2_rn(d, iv);
                const float2 sp = __ffma2_rn(make_float2(-1.f, -1.f), M2[q / 2], x);
                const float2 v = make_float2(sat_pos(sp.x), sat_pos(sp.y));
                acc2[q / 2] = __ffma2_rn(v, cp, acc2[q / 2]);
                M2[q / 2].x = fmaxf(M2[q / 2].x, x.x);
                M2[q / 2].y = fmaxf(M2[q / 2].y, x.y);
                // a masked step's |s| is +inf: it takes no part in the test
                sv[k][q / 2] = (MASKED && w >= nvalid) ? make_float2(pos_inf(), pos_inf()) : sp;
            }
        }
#pragma unroll
        for (int q = 0; q < P; q += 2) {
            mn[q] = min_abs2(mn[q], sv[0][q / 2].x, sv[1][q / 2].x);
            mn[q + 1] = min_abs2(mn[q + 1], sv[0][q / 2].y, sv[1][q / 2].y);
        }
    }
}

// Certified sweep of one staged row (the lane queue of sweep_row).  Every
// target is walked; pruned launches take sweep_rows_skip.
//
// The row is staged in row order for both walk directions.  A group covers
// the samples x0 .. x0 + P - 1 (x0 a multiple of 4, so that every window is
// 16-byte aligned); its POV q is sample x0 + q walking forward, or sample
// x0 + P - 1 - q walking backward, so that in either direction POV q's step
// w meets the window's element q + w + 1: a backward block's window is
// loaded from x0 - e - U and stored reversed.  Backward groups are taken
// from the row's end (the longest walks first).
template <int P, int U, bool LONG, bool RANGED, bool BWD, bool TIERS>
__device__ __forceinline__ void sweep_row_cert(const SweepParams& sp, const CertRow& r,
                                               const float4* __restrict__ tab, int* __restrict__ spill, int lane)
{
    static_assert(P % 4 == 0 && U % 4 == 0, "window loads must stay 16-byte aligned");
    const unsigned FULL = 0xffffffffu;
    const unsigned below = (1u << lane) - 1u;
    const float NEG = neg_inf();
    const float* __restrict__ H = r.H;
    const float* __restrict__ Lo = r.Lo;
    const int L = r.L, K = r.K, tabn = sp.inv_len;
    const int G = (L + P - 1) / P;
    const int klim = K - 1;
    // a backward block's window is stored reversed, so its aligned register
    // pairs hold (y[2j + 1], y[2j]) and only forward walks pack the differences
    constexpr bool PACK = !BWD && TVS_CERT_PACKADD;
    float ia[P];
    float2 ng2[P / 2];               // -g of POV pairs
    float2 M2[P / 2], acc2[P / 2];   // running maxima of POV pairs (packed x - M)
#define CERT_M(q) ((q) % 2 ? M2[(q) / 2].y : M2[(q) / 2].x)
#define CERT_NG(q) ((q) % 2 ? ng2[(q) / 2].y : ng2[(q) / 2].x)
    float Rh = 0.f, c2e = 0.f;
    unsigned lost = 0u, again = 0u;  // as in sweep_rows_skip
    int gi = lane, next = 32;
    int x0 = 0, e = 0, dlim = -1, seg = FLUSH_STEPS;
    bool klimited = false;
    // sample of POV q of the current group, and its walk's target count
    auto pov_x = [&](int q) { return BWD ? x0 + P - 1 - q : x0 + q; };
    auto walk_n = [&](int x) { return min(BWD ? x : L - 1 - x, K); };

    auto start = [&]() {
        x0 = (BWD ? G - 1 - gi : gi) * P;
        // the group's longest walk: its first existing POV in walk order
        const int xl = BWD ? min(x0 + P - 1, L - 1) : x0;
        const int rowlim = BWD ? xl - 1 : L - 2 - xl;
        dlim = min(klim, rowlim);
        klimited = klim < rowlim;
        e = 0;
        seg = FLUSH_STEPS;
        lost = again = 0u;
#pragma unroll
        for (int q = 0; q < P / 2; ++q) acc2[q] = make_float2(0.f, 0.f);
        if (LONG) {
#pragma unroll
            for (int q = 0; q < P; ++q) spill[32 * q] = 0;
        }
        if (dlim < 1) return;                 // no block runs
        // every index the group's blocks use, checked once: the last block
        // starts at elast < dlim
        const int elast = (dlim - 1) / U * U;
        const int wlo = BWD ? x0 - elast - U : x0;           // lowest window start
        const int whi = BWD ? x0 - U : x0 + elast;           // highest window start
        if (!in_range(ROW_PADL + wlo, sp.half, 19) || !in_range(ROW_PADL + whi + P + U - 1, sp.half, 19) ||
            (!(LONG && elast + U > tabn) && !in_range(elast + U - 1, tabn, 11))) {
            dlim = 0;
            lost = (1u << P) - 1u;
            sp.flag_count[2] = 1u;
            return;
        }
        float Rl;
        pov_hl(r, x0, Rh, Rl);
        (void)Rl;
        float gmax = 0.f;
#pragma unroll
        for (int q = 0; q < P; ++q) {
            const int x = pov_x(q);
            float gq = 0.f;
            if (BWD ? (x >= 1 && x <= L - 1) : x <= L - 2) {   // POVs with a target
                float zh, zl;
                pov_hl(r, x, zh, zl);
                gq = __fadd_rn(__fadd_rn(__fsub_rn(zh, Rh), zl), r.h0);
            }
            CERT_NG(q) = -gq;
            gmax = fmaxf(gmax, fabsf(gq));
        }
        c2e = CERT_ABS * __fmaf_rn(5.1f * 0x1p-24f, gmax, r.eg0);
#pragma unroll
        for (int q = 0; q < P; ++q) {
            // target 1 (a sentinel, -inf, when the POV has no target adding
            // area): M starts just below its slope, so that target is visible
            // and outside its margin, and the maximum then is its slope exactly
            const int x = pov_x(q);
            const int t = BWD ? x - 1 : x + 1;
            const float y1 = __fadd_rn(__fsub_rn(H[t], Rh), Lo[t]);
            const float x1 = __fadd_rn(y1, CERT_NG(q));
            const float C = __fmaf_rn(0x1p-6f, fabsf(x1), __fmaf_rn(4.f, c2e, 0x1p-16f));
            // a POV with no target that adds area starts at +inf: nothing is
            // visible to it and no step is inside its margin
            const bool area = BWD ? (x >= 2 && x <= L - 1) : x <= L - 3;
            CERT_M(q) = area ? __fsub_rn(x1, C) : pos_inf();
            ia[q] = 1.f;
        }
    };
    if (gi < G) start();
    for (;;) {
        const bool fin = gi < G && e >= dlim;
        const unsigned need = __ballot_sync(FULL, fin);
        if (need) {
            if (fin) {
                finish_group<P, LONG>(sp, r, lost, pov_x, walk_n,
                                      [&](int q) { return q % 2 ? acc2[q / 2].y : acc2[q / 2].x; }, spill);
                gi = next + __popc(need & below);
                if (gi < G) start(); else gi = G;
            }
            next += __popc(need);
            if (!__any_sync(FULL, gi < G)) break;
            continue;
        }
        if (gi < G) {
            if (LONG && e >= seg) {
                seg += FLUSH_STEPS;
#pragma unroll
                for (int q = 0; q < P; q += 2) {
                    spill[32 * q] += __float2int_rz(acc2[q / 2].x);
                    spill[32 * (q + 1)] += __float2int_rz(acc2[q / 2].y);
                    acc2[q / 2] = make_float2(0.f, 0.f);
                }
            }
            // a margin block of nh window blocks of U steps.  One of several
            // window blocks lies wholly before the group's last needed step (e +
            // nh U <= dlim), so none of them is masked and every window and
            // table entry it reads lies in the ranges start() checked.
            auto blocks_at = [&](int e) {
                return (!TIERS || LONG || e < CERT_NEAR) ? 1
                     : (e >= CERT_FAR && e + 4 * U <= dlim) ? 4
                     : (e + 2 * U <= dlim) ? 2 : 1;
            };
            const int nh = blocks_at(e);
            float2 before[P / 2];    // the measures before the block
#pragma unroll
            for (int q = 0; q < P / 2; ++q) before[q] = acc2[q];
            const float4* __restrict__ tb = tab + e + e / U;
            const float ive = (LONG && e >= tabn) ? __frcp_rn((float)(e + 1)) : tb->x;
            float Ms[P], mn[P];
#pragma unroll
            for (int q = 0; q < P; ++q) {
                Ms[q] = CERT_M(q);
                mn[q] = pos_inf();
            }
#pragma unroll 1
            for (int h = 0; h < nh; ++h) {
                const int eh = e + h * U;                    // this window block's first step
                const int wsh = BWD ? x0 - eh - U : x0 + eh; // its window's first sample
                const bool far = LONG && eh + U > tabn;
                const float4* __restrict__ tbh = tab + eh + eh / U;
                // the window, relative to R (reversed for a backward walk)
                float y[P + U];
                {
                    const float2 nRh = make_float2(-Rh, -Rh);
                    const float* bh = H + wsh;
                    const float* bl = Lo + wsh;
#pragma unroll
                    for (int m = 0; m < P + U; m += 4) {
                        const float4 a = *reinterpret_cast<const float4*>(bh + m);
                        const float4 b = *reinterpret_cast<const float4*>(bl + m);
                        const float2 y0 = __fadd2_rn(__fadd2_rn(make_float2(a.x, a.y), nRh), make_float2(b.x, b.y));
                        const float2 y1 = __fadd2_rn(__fadd2_rn(make_float2(a.z, a.w), nRh), make_float2(b.z, b.w));
                        const float v[4] = {y0.x, y0.y, y1.x, y1.y};
#pragma unroll
                        for (int i = 0; i < 4; ++i) y[BWD ? P + U - 1 - (m + i) : m + i] = v[i];
                    }
                }
                const bool masked = RANGED && klimited && eh + U > dlim;
                if (masked) {
                    if (far) cert_block<P, U, true, true, PACK>(y, tab, eh, ng2, M2, acc2, mn, dlim - eh);
                    else cert_block<P, U, true, false, PACK>(y, tbh, eh, ng2, M2, acc2, mn, dlim - eh);
                } else {
                    if (far) cert_block<P, U, false, true, PACK>(y, tab, eh, ng2, M2, acc2, mn, U);
                    else cert_block<P, U, false, false, PACK>(y, tbh, eh, ng2, M2, acc2, mn, U);
                }
            }
            // the margin test, once the block's last M is known: M only rises
            // within the block, so max(|M| at its start, |M| at its end)
            // bounds |M| at every one of its steps
            const float ce = __fmaf_rn(c2e, ive, CERT_FLOOR);
            unsigned fm = 0u;
#pragma unroll
            for (int q = 0; q < P; ++q) {
                const float dq =
                    __fmaf_rn(CERT_REL, fmaxf(fabsf(Ms[q]), fabsf(CERT_M(q))), __fmaf_rn(c2e, ia[q], ce));
                fm |= mn[q] < dq ? 1u << q : 0u;
            }
            if (fm) {
                // flagged POVs leave the block to the exact pass
                unsigned at = lost ? (unsigned)sp.flag_cap : reserve_flags(sp, __popc(fm));
#pragma unroll
                for (int q = 0; q < P; ++q) {
                    if (!((fm >> q) & 1u)) continue;
                    (q % 2 ? acc2[q / 2].y : acc2[q / 2].x) = q % 2 ? before[q / 2].y : before[q / 2].x;
                    const int x = pov_x(q), p0 = __float2int_rn(__frcp_rn(ia[q])) - 1;
                    const bool rest = (again >> q) & 1u || beside_outlier(c2e, CERT_M(q));
                    if (!flag_block(sp, at++, r.key, r.zmax, r.rev_staged ? L - 1 - x : x, e, nh * U, p0,
                                    blocks_at(p0) * U, rest ? FLAG_PREFIX : FLAG_BLOCK))
                        lost |= 1u << q;
                    if (rest) CERT_M(q) = pos_inf();   // nothing more is visible to it, or flagged
                }
                again |= fm;
            }
#pragma unroll
            for (int q = 0; q < P; ++q)
                if (CERT_M(q) > Ms[q] && !((fm >> q) & 1u)) { ia[q] = ive; again &= ~(1u << q); }
            e += nh * U;
        }
    }
#undef CERT_M
#undef CERT_NG
}

// min(a, b, c), one instruction; a NaN is dropped.
__device__ __forceinline__ float min3(float a, float b, float c)
{
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// Floats that a search may read past the last row's window maxima.
constexpr int WM_SLACK = std::max(SKIP_TESTS, PACK_TESTS) * SKIP_UNROLL / ZS_STRIDE;

// How a pruned walk takes the block that its range limit ends: there is none in
// the launch; in a masked copy of the block's code beside it; or cut short in
// the common code, so that its lanes run with the others (one row per warp,
// 1000^2, 1.5 km: 15.3 ms masked, 14.8 cut; shared rows, 4000^2, 10 km: 205
// masked, 211 cut).
enum class RangeEnd { NONE, MASKED, CUT };

// One round of a searching lane: tests NT blocks from step e on
// against the lines T d + K of its four POVs (see sweep_rows_skip) and returns
// the first step that may hold a visible target (*ready), the walk's end when
// no remaining target can be visible, or the step after the tested blocks.
// x0 and e are multiples of 4.  Blocks past the walk's end are tested against
// what lies up to WM_SLACK entries past the window maxima (or before them,
// walking backward: the end maxima); whatever the outcome, e is then past the
// end and the walk is over.
template <int U, bool BWD, int NT>
__device__ __forceinline__ int skip_blocks(const float2* T2, const float2* K2, bool rising, int x0, int e, int dlim,
                                           const float* __restrict__ WM, const float* __restrict__ ZS,
                                           bool* ready)
{
    const float d = (float)(e + 1);
    const int w0 = (BWD ? x0 - e : x0 + e + U) / ZS_STRIDE;
    float lim[NT], wm[NT];
#pragma unroll
    for (int k = 0; k < NT; ++k) {
        const float dk = d + (float)(k * U);
        const float2 l0 = __ffma2_rn(T2[0], make_float2(dk, dk), K2[0]);
        const float2 l1 = __ffma2_rn(T2[1], make_float2(dk, dk), K2[1]);
        lim[k] = min3(fminf(l0.x, l0.y), l1.x, l1.y);
        wm[k] = WM[BWD ? w0 - k * U / ZS_STRIDE : w0 + k * U / ZS_STRIDE];
    }
    const float end = ZS[(BWD ? x0 - e : x0 + e) / ZS_STRIDE];
    int n = NT;
#pragma unroll
    for (int k = NT - 1; k >= 0; --k)
        if (!(wm[k] <= lim[k])) n = k;
    e = rising && end <= lim[0] ? dlim : e + n * U;
    *ready = n < NT && e < dlim;
    return e;
}

// Pruned certified sweep of a warp's staged rows (2^lgna of them, sp.per_row
// floats apart; `groups` is the most groups of any), or of its share of a row's
// groups (every 2^lgs-th from gsub on): sweep_row_cert's walk, but a lane
// evaluates only the blocks of U steps that can hold a visible target, and
// stops where none is left.  (On fractal terrain 3 to 5 % of the targets of a
// walk are visible; the walks reach their stopping point after about 40 % of
// them, and about 12 % lie in blocks that cannot be skipped.)
//
// The test needs no slope: POV q's exact running maximum theta_a is at least
// thr_q = M_q - 2 delta_q (delta_q bounds |M_q - theta_a| as it does in the
// margin test, taken at the last evaluated block, whose 1 / (e + 1) is
// larger), so a target at distance d that is no higher than the line
//     R + g_q + thr_q d
// is not visible and leaves the maximum as it is.  Over the block's distances
// e + 1 .. e + U the line is lowest at the first when thr_q >= 0, at the last
// otherwise:
//     limit_q = thr_q (e + 1) + k_q,
//     k_q = R + g_q + (U - 1) min(thr_q, 0) - slack,
// and the block is skipped when its window's maximum height (WM) is at most
// min_q limit_q.  The walk is over when every thr_q >= 0 (the lines only
// rise) and the maximum of all remaining targets (ZS: suffix maxima, or
// prefix maxima walking backward) is at most that minimum too.  slack covers
// the rounding of g_q (Eg) and, 2^-20 of |R| and of |g_q|, of the line's start;
// the line's last rounding is relative to its own height, which is that of the
// maximum it is compared with where the two are close: the maxima are raised by
// 2^-20 of themselves, which covers the samples' lo parts too.  The (U - 1) term
// is taken 2^-17 larger.  (A slack of the row's largest |elevation| let one cell
// of -1e9 keep its rows from skipping.)
// A POV with no target that adds area has M = +inf and thr NaN, which the
// minimum drops.
//
// Measured (whole maps, against the walk that only stopped): 2000^2 199 ->
// 85.1 ms, 1000^2 32.7 -> 18.6 ms.  Where every target is visible nothing can be
// skipped and each block pays its tests and lines (level ground from 1.5 m, 8
// directions: 2000^2 16.4 -> 19.6 ms, 4000^2, 2 directions, 47.5 -> 45.0); leaving
// tests out after blocks that were needed gave 18.0 and cost 2000^2 fractal ground
// 85 -> 90.  Bound by the FMA and ALU pipes and by what
// the lanes wait for each other (22 of 32 active, issue slots 67 to 75 %
// used): registers decide how many warps hide the tests' latency, so the
// kernels keep no exact walks of their own (their context cost 200 bytes of
// local memory per lane; 16 warps then lost to 12), form the window as they
// go, and treat the inner groups of a row apart from its ends (92.6 -> 89.1).
//
// END says how the block in which the range limit ends the walks (at the same
// step for every POV) is walked.
//
// Work is done in three warp-wide phases, each with as many lanes as possible:
// finished groups are written and replaced (SKIP_RESTART lanes at a time, or
// when no lane has work); lanes without a block test NT blocks at a
// time until SKIP_READY lanes have one or nobody is searching; the lanes that
// have one evaluate it.  A lane waits while others search or restart, so the
// thresholds trade idle lanes against phases run for a few lanes only.  A
// block is evaluated SKIP_CHUNK steps at a time, with the window formed as it
// goes: the few registers that takes let 20 warps share an SM, and their
// number is what hides the latency of the tests.
template <int P, int U, bool LONG, RangeEnd END, bool BWD, int NT, int CH>
__device__ __forceinline__ void sweep_rows_skip(const SweepParams& sp, const SkipRow* __restrict__ rows,
                                                const float* H0, int lgna, int groups, int lgs, int gsub, int zs_off,
                                                int wm_off,
                                                const float2* __restrict__ tab, int* __restrict__ spill, int lane)
{
    static_assert(P == 4 && U % 8 == 0 && U % CH == 0 && CH % 4 == 0, "groups of four, window loads 16-byte aligned");
    const unsigned FULL = 0xffffffffu;
    const unsigned below = (1u << lane) - 1u;
    const int tabn = sp.inv_len;
    // the group's staged row (the lanes of a warp may be on different ones)
    const SkipRow* r = rows;
    const float* H = H0;             // its hi parts; lo parts, end and window maxima at fixed offsets
    constexpr bool PACK = !BWD && TVS_CERT_PACKADD;
    float2 ia2[P / 2];
    float2 ng2[P / 2];               // -g of POV pairs
    float2 M2[P / 2], acc2[P / 2];   // running maxima and measures of POV pairs
    float2 T2[P / 2], K2[P / 2];     // thr and k of POV pairs
    bool rising = false;             // every thr >= 0
    float Rh = 0.f, c2e = 0.f;
    float level = 0.f;               // R - slack
    unsigned lost = 0u, again = 0u;  // POVs whose walk is taken again; with a flagged block since the last certain rise
    // group (t >> lgna) 2^lgs + gsub of row t & (rows - 1), longest walks first
    const int tasks = (groups - gsub + (1 << lgs) - 1) >> lgs << lgna;
    int next = 32;
    bool has = lane < tasks;
    int x0 = 0, e = 0, dlim = -1, seg = FLUSH_STEPS;
    bool klimited = false, ready = false;
    auto pov_x = [&](int q) { return BWD ? x0 + P - 1 - q : x0 + q; };

    auto start = [&](int task) {
        r = rows + (task & ((1 << lgna) - 1));
        H = H0 + (task & ((1 << lgna) - 1)) * sp.per_row;
        const int L = r->L, gi = ((task >> lgna) << lgs) + gsub, G = (L + P - 1) / P;
        x0 = (BWD ? G - 1 - gi : gi) * P;
        e = 0;
        dlim = -1;
        lost = again = 0u;
        if (gi >= G) { x0 = L; return; }                     // a shorter row of the pack
        const int klim = r->K - 1;
        const int xl = BWD ? min(x0 + P - 1, L - 1) : x0;
        const int rowlim = BWD ? xl - 1 : L - 2 - xl;
        dlim = min(klim, rowlim);
        klimited = klim < rowlim;
        seg = FLUSH_STEPS;
#pragma unroll
        for (int q = 0; q < P / 2; ++q) {
            acc2[q] = make_float2(0.f, 0.f);
            ia2[q] = make_float2(1.f, 1.f);
        }
        if (LONG) {
#pragma unroll
            for (int q = 0; q < P; ++q) spill[32 * q] = 0;
        }
        if (dlim < 1) return;
        ready = true;                                        // the first block is always evaluated
        // the group's samples and its last POV's first target, relative to R
        const float4 a = *reinterpret_cast<const float4*>(H + x0);
        const float4 b = *reinterpret_cast<const float4*>(H + sp.half + x0);
        const float* ht = H + (BWD ? x0 - 1 : x0 + P);
        // all but a row's first and last groups stand on samples staged as
        // they are, and all of their POVs see targets that add area
        const bool inner = x0 > 0 && x0 + P <= L - 2;
        Rh = a.x;
        if (!inner) {                                        // the row's end samples are sentinels when staged
            if (x0 == 0) Rh = r->ends[0];
            else if (x0 == L - 1) Rh = r->ends[2];
        }
        const float2 nRh = make_float2(-Rh, -Rh);
        const float2 y0 = __fadd2_rn(__fadd2_rn(make_float2(a.x, a.y), nRh), make_float2(b.x, b.y));
        const float2 y1 = __fadd2_rn(__fadd2_rn(make_float2(a.z, a.w), nRh), make_float2(b.z, b.w));
        const float yt = __fadd_rn(__fsub_rn(ht[0], Rh), ht[sp.half]);
        const float ys[P + 1] = {BWD ? y1.y : y0.x, BWD ? y1.x : y0.y, BWD ? y0.y : y1.x, BWD ? y0.x : y1.y, yt};
        const float2 rh = *reinterpret_cast<const float2*>(&r->h0);   // h0, eg0
        float gq[P];
        bool area[P];
#pragma unroll
        for (int q = 0; q < P; ++q) {
            gq[q] = __fadd_rn(ys[q], rh.x);
            area[q] = true;
        }
        if (!inner) {
#pragma unroll
            for (int q = 0; q < P; ++q) {
                const int x = pov_x(q);
                if (x == 0) gq[q] = __fadd_rn(__fadd_rn(__fsub_rn(r->ends[0], Rh), r->ends[1]), rh.x);
                if (x == L - 1) gq[q] = __fadd_rn(__fadd_rn(__fsub_rn(r->ends[2], Rh), r->ends[3]), rh.x);
                if (!(BWD ? (x >= 1 && x <= L - 1) : x <= L - 2)) gq[q] = 0.f;   // no target
                area[q] = BWD ? (x >= 2 && x <= L - 1) : x <= L - 3;
            }
        }
        const float gmax = fmaxf(fmaxf(fabsf(gq[0]), fabsf(gq[1])), fmaxf(fabsf(gq[2]), fabsf(gq[3])));
        c2e = CERT_ABS * __fmaf_rn(5.1f * 0x1p-24f, gmax, rh.y);
        level = __fsub_rn(Rh, __fmaf_rn(0x1p-20f, __fmaf_rn(2.f, fabsf(Rh), gmax), __fmul_rn(2.f, c2e)));
        const float c0 = __fmaf_rn(4.f, c2e, 0x1p-16f);
#pragma unroll
        for (int q = 0; q < P; ++q) {
            // as sweep_row_cert: M starts just below the first target's slope
            const float x1 = __fsub_rn(ys[q + 1], gq[q]);
            const float m = area[q] ? __fsub_rn(x1, __fmaf_rn(0x1p-6f, fabsf(x1), c0)) : pos_inf();
            (q % 2 ? ng2[q / 2].y : ng2[q / 2].x) = -gq[q];
            (q % 2 ? M2[q / 2].y : M2[q / 2].x) = m;
        }
    };
    if (tasks <= 0) return;
    if (has) start(lane);
    for (;;) {
        // 1. finished groups: write their measures, hand over their flagged
        // walks, take the next groups
        const bool fin = has && !ready && e >= dlim;
        const unsigned need = __ballot_sync(FULL, fin);
        if (need && (__popc(need) >= SKIP_RESTART || !__any_sync(FULL, has && !fin))) {
            if (fin) {
                const int L = r->L, K = r->K;
                int* cvrow = r->cv;
                const bool rev = r->rev != 0;
                int add[P];                                  // by sample
#pragma unroll
                for (int q = 0; q < P; ++q) {
                    const int i = BWD ? P - 1 - q : q;
                    add[i] = (int)(q % 2 ? acc2[q / 2].y : acc2[q / 2].x) + (LONG ? spill[32 * q] : 0);
                }
                if (dlim >= 1 && x0 > 0 && x0 + P <= L - 2 && !lost) {
                    // every POV has a target
                    int* at = cvrow + (rev ? L - 1 - x0 : x0);
                    const int st = rev ? -1 : 1;
#pragma unroll
                    for (int i = 0; i < P; ++i, at += st) *at = 1 + add[i];
                } else
#pragma unroll
                for (int q = 0; q < P; ++q) {
                    const int x = pov_x(q);
                    if (x >= L) continue;
                    const int n = min(BWD ? x : L - 1 - x, K);
                    const int cv = n >= 1 ? 1 + add[BWD ? P - 1 - q : q] : 0;
                    cvrow[rev ? L - 1 - x : x] = (lost >> q) & 1u ? CV_FLAGGED : cv;
                }
                const int task = next + __popc(need & below);
                has = task < tasks;
                if (has) start(task);
            }
            next += __popc(need);
            if (!__any_sync(FULL, has)) break;
        }
        // 2. lanes without a block look for one
        for (;;) {
            if (has && !ready && e < dlim)
                e = skip_blocks<U, BWD, NT>(T2, K2, rising, x0, e, dlim, H + wm_off, H + zs_off, &ready);
            const unsigned have = __ballot_sync(FULL, ready);
            const unsigned look = __ballot_sync(FULL, has && !ready && e < dlim);
            if (!look || __popc(have) >= SKIP_READY) break;
        }
        // 3. evaluate the blocks found
        if (ready) {
            ready = false;
            if (LONG && e >= seg) {
                // at most FLUSH_STEPS steps of distance between two flushes
                seg = e + FLUSH_STEPS;
#pragma unroll
                for (int q = 0; q < P; q += 2) {
                    spill[32 * q] += __float2int_rz(acc2[q / 2].x);
                    spill[32 * (q + 1)] += __float2int_rz(acc2[q / 2].y);
                    acc2[q / 2] = make_float2(0.f, 0.f);
                }
            }
            const bool far = LONG && e + U > tabn;
            const float2* __restrict__ tb = tab + e + 2 * (e / U);
            const float ive = (LONG && e >= tabn) ? __frcp_rn((float)(e + 1)) : tb->x;
            float mn[P];
            float2 Ms2[P / 2];
            float2 blk2[P / 2];      // the block's share of the measures
#pragma unroll
            for (int q = 0; q < P / 2; ++q) {
                blk2[q] = make_float2(0.f, 0.f);
                Ms2[q] = M2[q];
                mn[2 * q] = mn[2 * q + 1] = pos_inf();
            }
            {
                // the window relative to R, y[m] = sample m of the block's
                // window in walk order, kept P samples back from step to step
                const float2 nRh = make_float2(-Rh, -Rh);
                const float* bh = H + (BWD ? x0 - e : x0 + e);
                const float* bl = bh + sp.half;
                float y[P + CH];
                auto quad = [&](int at, int m) {   // y[m ..] from the four samples at `at`
                    const float4 a = *reinterpret_cast<const float4*>(bh + at);
                    const float4 b = *reinterpret_cast<const float4*>(bl + at);
                    const float2 y0 = __fadd2_rn(__fadd2_rn(make_float2(a.x, a.y), nRh), make_float2(b.x, b.y));
                    const float2 y1 = __fadd2_rn(__fadd2_rn(make_float2(a.z, a.w), nRh), make_float2(b.z, b.w));
                    y[m] = BWD ? y1.y : y0.x;
                    y[m + 1] = BWD ? y1.x : y0.y;
                    y[m + 2] = BWD ? y0.y : y1.x;
                    y[m + 3] = BWD ? y0.x : y1.y;
                };
                quad(0, 0);
                const int steps = min(dlim - e, U);
                // RangeEnd::CUT: POV q's last target is element steps + q.
                // Elements past `steps` are hidden from all POVs and the targets
                // that POVs 1 to 3 still have among them taken one by one.
                const bool cut = END == RangeEnd::CUT && klimited && steps < U;
                if (cut) {
#pragma unroll
                    for (int m = 0; m < P; ++m) y[m] = m > steps ? neg_inf() : y[m];
                }
#pragma unroll 1
                for (int c = 0; c < steps; c += CH) {
#pragma unroll
                    for (int m = P; m < P + CH; m += 4) quad(BWD ? -(c + m) : c + m, m);
                    if (cut) {
#pragma unroll
                        for (int m = P; m < P + CH; ++m) y[m] = c + m > steps ? neg_inf() : y[m];
                    }
                    if (END == RangeEnd::MASKED && klimited && c + CH > steps) {
                        if (far) cert_block<P, CH, true, true, PACK>(y, tab, e + c, ng2, M2, blk2, mn, steps - c);
                        else cert_block<P, CH, true, false, PACK>(y, tb + c, e + c, ng2, M2, blk2, mn, steps - c);
                    } else {
                        if (far) cert_block<P, CH, false, true, PACK>(y, tab, e + c, ng2, M2, blk2, mn, CH);
                        else cert_block<P, CH, false, false, PACK>(y, tb + c, e + c, ng2, M2, blk2, mn, CH);
                    }
#pragma unroll
                    for (int m = 0; m < P; ++m) y[m] = y[m + CH];
                }
                if (cut) {
#pragma unroll
                    for (int q = 1; q < P; ++q) {
                        float2& M = M2[q / 2];
                        float2& A = blk2[q / 2];
#pragma unroll
                        for (int k = 0; k < q; ++k) {
                            const int w = steps - q + k;     // element steps + 1 + k
                            if (w < 0) continue;
                            const int at = BWD ? P - 1 - (steps + 1 + k) : steps + 1 + k;
                            const float yk = __fadd_rn(__fsub_rn(bh[at], Rh), bl[at]);
                            const float iv = far ? __frcp_rn((float)(e + w + 1)) : tb[w].x;
                            const float x = __fmul_rn(__fadd_rn(yk, q % 2 ? ng2[q / 2].y : ng2[q / 2].x), iv);
                            const float sx = __fsub_rn(x, q % 2 ? M.y : M.x);
                            const float add = __fmul_rn(sat_pos(sx), (float)(2 * (e + w) + 3));
                            if (q % 2) { A.y = __fadd_rn(A.y, add); M.y = fmaxf(M.y, x); }
                            else { A.x = __fadd_rn(A.x, add); M.x = fmaxf(M.x, x); }
                            mn[q] = fminf(mn[q], fabsf(sx));
                        }
                    }
                }
            }
            // the margin test of sweep_row_cert, and the lines of the next tests
            const float ce = __fmaf_rn(c2e, ive, CERT_FLOOR);
            float2 dq2[P / 2], ex2[P / 2];               // delta, and mn - delta
#pragma unroll
            for (int q = 0; q < P / 2; ++q) {
                const float2 mb = make_float2(fmaxf(fabsf(Ms2[q].x), fabsf(M2[q].x)),
                                              fmaxf(fabsf(Ms2[q].y), fabsf(M2[q].y)));
                dq2[q] = __ffma2_rn(make_float2(CERT_REL, CERT_REL), mb,
                                    __ffma2_rn(make_float2(c2e, c2e), ia2[q], make_float2(ce, ce)));
                ex2[q] = __ffma2_rn(make_float2(-1.f, -1.f), dq2[q], make_float2(mn[2 * q], mn[2 * q + 1]));
            }
            unsigned fm = 0u;
            if (min3(fminf(ex2[0].x, ex2[0].y), ex2[1].x, ex2[1].y) < 0.f) {
                // flagged POVs leave the block to the exact pass
#pragma unroll
                for (int q = 0; q < P; ++q) fm |= (q % 2 ? ex2[q / 2].y : ex2[q / 2].x) < 0.f ? 1u << q : 0u;
                unsigned at = flag_slots(sp, __popc(fm), full_mark(H + sp.half));
#pragma unroll
                for (int q = 0; q < P; ++q) {
                    if (!((fm >> q) & 1u)) continue;
                    (q % 2 ? blk2[q / 2].y : blk2[q / 2].x) = 0.f;
                    const int p0 = __float2int_rn(__frcp_rn(q % 2 ? ia2[q / 2].y : ia2[q / 2].x)) - 1;
                    const int x = pov_x(q);
                    float& M = q % 2 ? M2[q / 2].y : M2[q / 2].x;
                    const bool rest = (again >> q) & 1u || beside_outlier(c2e, M);
                    if (!flag_block(sp, at++, r->key, r->zmax, r->rev ? r->L - 1 - x : x, e, U, p0, U,
                                    rest ? FLAG_PREFIX : FLAG_BLOCK))
                        lost |= 1u << q;
                    if (rest) M = pos_inf();   // nothing more is visible to it, or flagged
                }
                again |= fm;
            }
#pragma unroll
            for (int q = 0; q < P / 2; ++q) {
                acc2[q] = __fadd2_rn(acc2[q], blk2[q]);
                // (the last rise of a flagged POV stays where it was; a certain
                // rise lies above every earlier target, flagged or not)
                if (M2[q].x > Ms2[q].x && !((fm >> 2 * q) & 1u)) { ia2[q].x = ive; again &= ~(1u << 2 * q); }
                if (M2[q].y > Ms2[q].y && !((fm >> (2 * q + 1)) & 1u)) { ia2[q].y = ive; again &= ~(2u << 2 * q); }
                T2[q] = __ffma2_rn(make_float2(-2.f, -2.f), dq2[q], M2[q]);
                const float2 lv = __ffma2_rn(make_float2(-1.f, -1.f), ng2[q], make_float2(level, level));
                K2[q] = __ffma2_rn(make_float2((float)(U - 1) * 1.00001f, (float)(U - 1) * 1.00001f),
                                   make_float2(fminf(T2[q].x, 0.f), fminf(T2[q].y, 0.f)), lv);
            }
            rising = !(min3(fminf(T2[0].x, T2[0].y), T2[1].x, T2[1].y) < 0.f);
            e += U;
        }
    }
}

// Pruned FP32-decision sweep of one staged row (backward rows staged
// reversed), in the phases of sweep_rows_skip.  A skipped target must be one
// whose single-precision slope fl(fl(z - h) fl(1/d)) is at most M_q, which the
// maximum then keeps: three roundings move a slope by less than 2^-22 of
// itself, so with thr_q = M_q - 2^-21 |M_q| every target no higher than
// h_q + thr_q d qualifies; the line starts 2^-19 of |h_q| lower and the maxima
// are raised for the line's own rounding, as there.
// Every measure is bit for bit the unpruned walk's.  A POV without targets
// has thr = -inf, which keeps its (short) group from skipping.
// 1201 x 777, 180 directions: 19.5 -> 11.5 ms against the walk that only
// stopped (8 POVs and 28 steps per block: larger blocks hold a visible target
// more often, but cost less where all are: level ground, 2000^2, 8 directions 9.8
// ms then, 13.7 so).
template <int P, int U, bool LONG, bool RANGED>
__device__ __forceinline__ void sweep_row_skip32(const SweepParams& sp, const float* __restrict__ F,
                                                 const float* __restrict__ ZS, const float* __restrict__ WM,
                                                 const float2* __restrict__ tab, int* __restrict__ cvrow,
                                                 int* __restrict__ spill, int L, int K, float h0,
                                                 bool rev, int lane)
{
    constexpr int CH = FP32_CHUNK;
    static_assert(P == 4 && U % 8 == 0 && U % CH == 0 && CH % 4 == 0, "groups of four, window loads 16-byte aligned");
    const unsigned FULL = 0xffffffffu;
    const unsigned below = (1u << lane) - 1u;
    const float NEG = neg_inf();
    const int G = (L + P - 1) / P;
    const int klim = K - 1, tabn = sp.inv_len;
    float h[P], M[P];
    float2 acc2[P / 2], T2[P / 2], K2[P / 2];
    bool rising = false, ready = false, klimited = false;
    int gi = lane, next = 32;
    int x0 = 0, e = 0, dlim = -1, seg = FLUSH_STEPS;
    const bool inside = in_range(ROW_PADL + L + P + U, sp.half, 6) && in_range((L - 1) / ZS_STRIDE, sp.zs_len, 7) &&
                        in_range((L + U + 3) / ZS_STRIDE - 1, sp.wm_len, 8) &&
                        (LONG || in_range(min(K, L) + U - 1, tabn, 12));
    if (!inside) return;

    auto start = [&]() {
        x0 = gi * P;
        const int rowlim = L - 2 - x0;
        dlim = min(klim, rowlim);
        klimited = klim < rowlim;
        e = 0;
        seg = FLUSH_STEPS;
        ready = dlim > 0;                                    // the first block is always evaluated
        const float4 a = *reinterpret_cast<const float4*>(F + ROW_PADL + x0);
        h[0] = __fadd_rn(a.x, h0); h[1] = __fadd_rn(a.y, h0);
        h[2] = __fadd_rn(a.z, h0); h[3] = __fadd_rn(a.w, h0);
#pragma unroll
        for (int q = 0; q < P; ++q) {
            M[q] = NEG;
            if (LONG) spill[32 * q] = 0;
        }
#pragma unroll
        for (int q = 0; q < P / 2; ++q) acc2[q] = make_float2(0.f, 0.f);
    };
    if (gi < G) start();
    for (;;) {
        const bool fin = gi < G && !ready && e >= dlim;
        const unsigned need = __ballot_sync(FULL, fin);
        if (need && (__popc(need) >= SKIP_RESTART || !__any_sync(FULL, gi < G && !fin))) {
            if (fin) {
#pragma unroll
                for (int q = 0; q < P; ++q) {
                    const int x = x0 + q;
                    if (x >= L) continue;
                    const float s = q % 2 ? acc2[q / 2].y : acc2[q / 2].x;
                    cvrow[rev ? L - 1 - x : x] =
                        min(L - 1 - x, K) >= 1 ? 1 + (int)s + (LONG ? spill[32 * q] : 0) : 0;
                }
                gi = next + __popc(need & below);
                if (gi < G) start(); else gi = G;
            }
            next += __popc(need);
            if (!__any_sync(FULL, gi < G)) break;
        }
        for (;;) {
            if (gi < G && !ready && e < dlim) e = skip_blocks<U, false, SKIP_TESTS>(T2, K2, rising, x0, e, dlim, WM, ZS, &ready);
            const unsigned have = __ballot_sync(FULL, ready);
            const unsigned look = __ballot_sync(FULL, gi < G && !ready && e < dlim);
            if (!look || __popc(have) >= SKIP_READY) break;
        }
        if (ready) {
            ready = false;
            if (LONG && e >= seg) {
                seg = e + FLUSH_STEPS;
#pragma unroll
                for (int q = 0; q < P; q += 2) {
                    spill[32 * q] += __float2int_rz(acc2[q / 2].x);
                    spill[32 * (q + 1)] += __float2int_rz(acc2[q / 2].y);
                    acc2[q / 2] = make_float2(0.f, 0.f);
                }
            }
            const bool far = LONG && e + U > tabn;
            const float2* __restrict__ tb = tab + e + 2 * (e / U);
            const float* base = F + ROW_PADL + x0 + e;
            float w[P + CH];
            auto quad = [&](int at, int m) {
                const float4 v = *reinterpret_cast<const float4*>(base + at);
                w[m] = v.x; w[m + 1] = v.y; w[m + 2] = v.z; w[m + 3] = v.w;
            };
            quad(0, 0);
            const int steps = min(dlim - e, U);
            // the block that the range limit cuts, as in sweep_rows_skip
            const bool cut = RANGED && klimited && steps < U;
            if (cut) {
#pragma unroll
                for (int m = 0; m < P; ++m) w[m] = m > steps ? NEG : w[m];
            }
#pragma unroll 1
            for (int c = 0; c < steps; c += CH) {
#pragma unroll
                for (int m = P; m < P + CH; m += 4) quad(c + m, m);
                if (cut) {
#pragma unroll
                    for (int m = P; m < P + CH; ++m) w[m] = c + m > steps ? NEG : w[m];
                }
                if (far) sweep_block<P, CH, false, true>(w, tab, e + c, h, M, acc2, CH);
                else sweep_block<P, CH, false, false>(w, tb + c, e + c, h, M, acc2, CH);
#pragma unroll
                for (int m = 0; m < P; ++m) w[m] = w[m + CH];
            }
            if (cut) {
#pragma unroll
                for (int q = 1; q < P; ++q) {
#pragma unroll
                    for (int k = 0; k < q; ++k) {
                        const int u = steps - q + k;
                        if (u < 0) continue;
                        const float iv = far ? __frcp_rn((float)(e + u + 1)) : tb[u].x;
                        const float t = __fmul_rn(__fsub_rn(base[steps + 1 + k], h[q]), iv);
                        const float add = __fmul_rn(fset_gt(t, M[q]), (float)(2 * (e + u) + 3));
                        if (q % 2) acc2[q / 2].y = __fadd_rn(acc2[q / 2].y, add);
                        else acc2[q / 2].x = __fadd_rn(acc2[q / 2].x, add);
                        M[q] = fmaxf(M[q], t);
                    }
                }
            }
            rising = true;
#pragma unroll
            for (int q = 0; q < P; ++q) {
                const float thr = __fmaf_rn(-0x1p-21f, fabsf(M[q]), M[q]);
                const float base0 = __fmaf_rn(-0x1p-19f, fabsf(h[q]), h[q]);
                (q % 2 ? T2[q / 2].y : T2[q / 2].x) = thr;
                (q % 2 ? K2[q / 2].y : K2[q / 2].x) =
                    __fmaf_rn((float)(U - 1) * 1.00001f, fminf(thr, 0.f), base0);
                rising = rising && thr >= 0.f;
            }
            e += U;
        }
    }
}

template <bool LONG>
__device__ __forceinline__ void sweep_item(const ItemRow& it, const float* F, const float4* tab, int tabn, int* cvrow,
                                           int* spill, int lane)
{
    if (it.pov == SMALL_POV)
        sweep_row<SMALL_POV, SMALL_UNROLL, LONG>(F, tab, tabn, cvrow, spill, it.L, it.K, it.h0, it.rev, lane);
    else
        sweep_row<LARGE_POV, LARGE_UNROLL, LONG>(F, tab, tabn, cvrow, spill, it.L, it.K, it.h0, it.rev, lane);
}


// Warps per CTA of the unpruned certified kernels: their
// per-lane state (4 POVs' maxima, heights, margins and last-visible bounds,
// the window relative to the group) takes about 160 registers, which 12 warps
// still leave every thread.  When shared memory holds CERT_WIDE_WARPS warps, a
// second instantiation bounded to 128 registers runs them: the extra warps
// hide more latency than the few spills of its group-restart path cost.
#ifndef TVS_CERT_MAX_WARPS
#define TVS_CERT_MAX_WARPS 12
#endif
constexpr int CERT_MAX_WARPS = TVS_CERT_MAX_WARPS;
#ifndef TVS_CERT_WIDE_WARPS
#define TVS_CERT_WIDE_WARPS 16
#endif
constexpr int CERT_WIDE_WARPS = TVS_CERT_WIDE_WARPS;
// The fewest warps the one-row-per-warp certified kernel runs with; longer
// rows go to warp pairs.
#ifndef TVS_CERT_SINGLE_MIN
#define TVS_CERT_SINGLE_MIN 12
#endif
static_assert(CERT_MAX_WARPS % 2 == 0 && CERT_WIDE_WARPS % 2 == 0, "certified warps come in pairs");

// The FP32-decision sweep.  PRUNE: exact horizon pruning; LONG: the launch
// holds rows with walks of more than LONG_WALK steps (every row then takes
// the flushing walk).  Per warp, shared memory holds the staged row (reversed
// for backward items), its suffix maxima (PRUNE) and the long-walk spill
// (LONG).
template <bool PRUNE, bool LONG, bool RANGED, int WARPS>
__global__ void __launch_bounds__(WARPS * 32, 1) sweep_kernel(SweepParams sp)
{
    extern __shared__ __align__(16) float smem[];
    using Entry = std::conditional_t<PRUNE, float2, float4>;
    Entry* tab = reinterpret_cast<Entry*>(smem);
    int* istart = reinterpret_cast<int*>(smem + sp.tab_floats);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float* Fh = smem + sp.tab_floats + sp.istart_len + warp * sp.per_warp;
    float* ZS = Fh + sp.half;
    float* WM = ZS + sp.zs_len;
    int* spill = reinterpret_cast<int*>(WM + sp.wm_len) + lane;
    // per distance d = m + 1: (1/d, 1/d, 2d + 1, 2d + 1); 1/d correctly rounded
    for (int m = threadIdx.x; m < sp.inv_len; m += blockDim.x) {
        const float r = __frcp_rn((float)(m + 1));
        if constexpr (PRUNE) tab[m + 2 * (m / SKIP_UNROLL)] = make_float2(r, r);
        else tab[m] = make_float4(r, r, (float)(2 * m + 3), (float)(2 * m + 3));
    }
    for (int m = threadIdx.x; m <= sp.ndir; m += blockDim.x) istart[m] = sp.item_start[m];
    __syncthreads();

    int next = 0;
    if (lane == 0) next = (int)atomicAdd(sp.counter, 1u);
    next = __shfl_sync(0xffffffffu, next, 0);
    for (;;) {
        const int item = next;
        if (item >= sp.total_items) break;
        ItemRow it;
        const bool nonempty = decode_item(sp, istart, item, &it);
        if (lane == 0) next = (int)atomicAdd(sp.counter, 1u);
        next = __shfl_sync(0xffffffffu, next, 0);
        if (!nonempty) continue;
        __syncwarp();
        stage_row<false>(sp, it, Fh, nullptr, nullptr, lane);
        __syncwarp();   // the staged row is visible to every lane
        int* cvrow = (it.rev ? sp.cv_bwd : sp.cv_fwd) + it.rowbase;
        if constexpr (PRUNE) {
            end_max<false>(Fh, ZS, it.L, lane);
            window_max<SMALL_POV, SKIP_UNROLL>(Fh, WM, it.L, lane);
            __syncwarp();
            sweep_row_skip32<SMALL_POV, SKIP_UNROLL, LONG, RANGED>(sp, Fh, ZS, WM, tab, cvrow, spill, it.L, it.K, it.h0,
                                                           it.rev, lane);
        } else {
            sweep_item<LONG>(it, Fh, tab, sp.inv_len, cvrow, spill, lane);
        }
    }
}

// The unpruned certified sweep with one row per warp, for launches whose rows leave
// room for at least TVS_CERT_SINGLE_MIN of them (16 warps when they fit, else
// 12): a backward item's row is staged reversed and walked forward, like the
// FP32 sweep's.  Per warp, shared memory holds
// [Fh half][Fl half][ends 4].
template <bool LONG, bool RANGED, int WARPS>
__global__ void __launch_bounds__(WARPS * 32, 1) sweep_cert_kernel(SweepParams sp)
{
    extern __shared__ __align__(16) float smem[];
    float4* tab = reinterpret_cast<float4*>(smem);
    int* istart = reinterpret_cast<int*>(smem + sp.tab_floats);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float* Fh = smem + sp.tab_floats + sp.istart_len + warp * sp.per_warp;
    float* Fl = Fh + sp.half;
    constexpr int U = CERT_UNROLL_SINGLE;
    int* spill = reinterpret_cast<int*>(Fl + sp.half) + lane;
    float* ends = Fh + sp.per_warp - 4;
    for (int m = threadIdx.x; m < sp.inv_len; m += blockDim.x) {
        const float r = __frcp_rn((float)(m + 1));
        tab[m + m / U] = make_float4(r, r, (float)(2 * m + 3), (float)(2 * m + 3));
    }
    for (int m = threadIdx.x; m <= sp.ndir; m += blockDim.x) istart[m] = sp.item_start[m];
    __syncthreads();
    const long long t_start = clock64();

    int next = 0;
    if (lane == 0) next = (int)atomicAdd(sp.counter, 1u);
    next = __shfl_sync(0xffffffffu, next, 0);
    for (;;) {
        const int item = next;
        if (item >= sp.total_items) break;
        ItemRow it;
        const bool nonempty = decode_item(sp, istart, item, &it);
        if (lane == 0) next = (int)atomicAdd(sp.counter, 1u);
        next = __shfl_sync(0xffffffffu, next, 0);
        if (!nonempty) continue;
        __syncwarp();
        const float zmax = stage_row<true>(sp, it, Fh, Fl, ends, lane);
        __syncwarp();   // the staged row is visible to every lane
        if (df::beyond(zmax, it.h0)) {
            hand_over_row(sp, it, it.rev, zmax, it.rev ? sp.cv_bwd : sp.cv_fwd, lane, 32, Fl + ROW_PADL);
            continue;
        }
        const CertRow r = cert_row(sp, it, Fh, Fl, ends, zmax, it.rev ? sp.cv_bwd : sp.cv_fwd, it.rev);
        sweep_row_cert<CERT_POV, U, LONG, RANGED, false, false>(sp, r, tab, spill, lane);
    }
    if (lane == 0) atomicAdd(&g_sweep_stats[3], (unsigned long long)(clock64() - t_start));
}

// The pruned certified sweep of rows that leave room for a warp's own: a warp
// stages 2^lgna walks' rows at a time, walked forward.  With lgna = 0 that is
// one work item (a backward item's row reversed); with more, both walk
// directions of 2^(lgna - 1) consecutive rows, gathered once and stored in
// either order.  The groups of all of them share the lanes' queue: a row of
// 100 samples alone has 25 groups for 32 lanes, and its lanes would wait for
// the longest walk of every row and for its gathers.  60 tiles of 64 to 256
// cells a side: 21.6 -> 14.9 ms, 100 x 100: 309 -> 232 us (packs of one row
// at 20 warps instead of 16: 1000^2 21.9 -> 20.5 ms).  Per warp, shared memory
// holds the rows' SkipRows and per row [Fh half][Fl half][suffix maxima]
// [window maxima].
template <bool RANGED, int WARPS, int NT, int CH>
__global__ void __launch_bounds__(WARPS * 32, 1) sweep_pack_kernel(SweepParams sp)
{
    extern __shared__ __align__(16) float smem[];
    float2* tab = reinterpret_cast<float2*>(smem);
    int* istart = reinterpret_cast<int*>(smem + sp.tab_floats);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int na = 1 << sp.lgna;
    SkipRow* rows = reinterpret_cast<SkipRow*>(smem + sp.tab_floats + sp.istart_len + warp * sp.per_warp);
    float* arrays = reinterpret_cast<float*>(rows + na);
    const int zs_off = 2 * sp.half - ROW_PADL, wm_off = zs_off + sp.zs_len;   // from the hi parts
    constexpr int U = SKIP_UNROLL;
    for (int m = threadIdx.x; m < sp.inv_len; m += blockDim.x) {
        const float r = __frcp_rn((float)(m + 1));
        tab[m + 2 * (m / U)] = make_float2(r, r);
    }
    for (int m = threadIdx.x; m <= sp.ndir; m += blockDim.x) istart[m] = sp.item_start[m];
    __syncthreads();
    const long long t_start = clock64();

    int next = 0;
    if (lane == 0) next = (int)atomicAdd(sp.counter, (unsigned)na);
    next = __shfl_sync(0xffffffffu, next, 0);
    while (next < sp.total_items) {
        const int base = next;
        if (lane == 0) next = (int)atomicAdd(sp.counter, (unsigned)na);
        next = __shfl_sync(0xffffffffu, next, 0);
        __syncwarp();
        int longest = 0;
        for (int a = 0; a < na; a += 2) {      // items base + a and base + a + 1 are one row, both directions
            ItemRow it;
            SkipRow* r = rows + a;
            if (base + a >= sp.total_items || !decode_item(sp, istart, base + a, &it)) {
                if (lane == 0) {
                    r->L = 0;
                    if (na > 1) r[1].L = 0;
                }
                continue;
            }
            float* Fh = arrays + a * sp.per_row;
            float* Fb = Fh + sp.per_row;
            const bool both = na > 1;
            const float zmax = stage_row<true>(sp, it, Fh, Fh + sp.half, r->ends, lane, 0, 1, true,
                                               both ? Fb : nullptr, Fb + sp.half);
            __syncwarp();   // the staged rows are visible to every lane
            if (df::beyond(zmax, it.h0)) {
                const float* lo = Fh + sp.half + ROW_PADL;
                hand_over_row(sp, it, it.rev, zmax, it.rev ? sp.cv_bwd : sp.cv_fwd, lane, 32, lo);
                if (both) hand_over_row(sp, it, true, zmax, sp.cv_bwd, lane, 32, lo);
                if (lane == 0) {
                    r->L = 0;
                    if (both) r[1].L = 0;
                }
                continue;
            }
            if (lane == 0) {
                const bool ok = skip_row(sp, it, it.rev, zmax, it.rev ? sp.cv_bwd : sp.cv_fwd, it.rev, false, r);
                if (both) {
                    skip_row(sp, it, true, zmax, sp.cv_bwd, true, false, r + 1);
                    r[1].ends[0] = r->ends[2]; r[1].ends[1] = r->ends[3];
                    r[1].ends[2] = r->ends[0]; r[1].ends[3] = r->ends[1];
                }
                if (!ok) {
                    r->L = 0;
                    if (both) r[1].L = 0;
                }
            }
            longest = max(longest, it.L);
            for (int b = 0; b <= (both ? 1 : 0); ++b) {
                const float* F = Fh + b * sp.per_row;
                float* ZS = Fh + b * sp.per_row + 2 * sp.half;
                end_max<false>(F, ZS, it.L, lane);
                window_max<CERT_POV, U>(F, ZS + sp.zs_len, it.L, lane);
            }
        }
        __syncwarp();
        if (longest > 0)
            sweep_rows_skip<CERT_POV, U, false, RANGED ? RangeEnd::CUT : RangeEnd::NONE, false, NT, CH>(sp, rows, arrays + ROW_PADL, sp.lgna,
                                                       (longest + CERT_POV - 1) / CERT_POV, 0, 0, zs_off, wm_off, tab,
                                                       nullptr, lane);
    }
    if (lane == 0) atomicAdd(&g_sweep_stats[3], (unsigned long long)(clock64() - t_start));
}

// Barrier of the 2^lgw warps that share row buffer `row` (named barrier 1 + row).
__device__ __forceinline__ void row_sync(int row, int lgw)
{
    asm volatile("bar.sync %0, %1;" :: "r"(1 + row), "r"(32 << lgw) : "memory");
}

// The certified sweep with one staged row per 2^lgw warps, half of which walk
// it forward (items 2p) and half backward (items 2p + 1), so a row's
// double-float samples and end samples are staged once and held once for all
// of them.  The warps of one walk direction take every 2^(lgw - 1)-th group.
// Two warps per row when that fills the SM (rows of up to about 2600 samples),
// more beyond (pruned): 4000-sample rows leave room for 4, and with two warps
// each for 8 warps in all (4000^2, 90 directions, 10 km: 264 ms with two warps
// per row, 204 with four; 5000^2, 8 directions: 74 and 53).  All of them stage a share of the row; the first
// computes its suffix maxima, the second its prefix maxima (pruning).  Each
// warp runs one direction's code only.  Per row, shared memory holds [Fh
// half][Fl half][suffix maxima][prefix maxima][window maxima][ends 4][item and
// zmax exchange][a SkipRow per walk direction]; per warp the long-walk spill.
constexpr int MAX_LGW = 4;
constexpr int ROW_XCH = 4 + (1 << MAX_LGW);   // floats of the exchange

template <bool PRUNE, bool LONG, bool RANGED, int WARPS>
__global__ void __launch_bounds__(WARPS * 32, 1) sweep_pair_kernel(SweepParams sp)
{
    extern __shared__ __align__(16) float smem[];
    using Entry = std::conditional_t<PRUNE, float2, float4>;
    Entry* tab = reinterpret_cast<Entry*>(smem);
    int* istart = reinterpret_cast<int*>(smem + sp.tab_floats);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int lgw = sp.lgw, nw = 1 << lgw;
    const int pair = warp >> lgw, part = warp & (nw - 1), bwd = part & 1;
    const int npairs = blockDim.x >> (5 + lgw);
    float* base = smem + sp.tab_floats + sp.istart_len;
    float* Fh = base + pair * sp.per_pair;
    float* Fl = Fh + sp.half;
    float* ZS = Fl + sp.half + bwd * sp.zs_len;            // this warp's suffix or prefix maxima
    float* WM = Fl + sp.half + 2 * sp.zs_len;              // window maxima (both warps')
    float* ends = WM + sp.wm_len;                          // 4 floats
    constexpr int U = PRUNE ? SKIP_UNROLL : CERT_UNROLL;
    float* xch = ends + 4;                                   // item number and the halves' zmax
    // the row as either walk direction sees it (pruned)
    SkipRow* row = reinterpret_cast<SkipRow*>(xch + ROW_XCH) + bwd;
    constexpr RangeEnd END = RANGED ? RangeEnd::MASKED : RangeEnd::NONE;
    float* own = base + npairs * sp.per_pair + warp * sp.per_warp;
    int* spill = reinterpret_cast<int*>(own) + lane;
    for (int m = threadIdx.x; m < sp.inv_len; m += blockDim.x) {
        const float r = __frcp_rn((float)(m + 1));
        if constexpr (PRUNE) tab[m + 2 * (m / U)] = make_float2(r, r);
        else tab[m + m / U] = make_float4(r, r, (float)(2 * m + 3), (float)(2 * m + 3));
    }
    for (int m = threadIdx.x; m <= sp.ndir; m += blockDim.x) istart[m] = sp.item_start[m];
    __syncthreads();
    const long long t_start = clock64();

    for (;;) {
        if (part == 0 && lane == 0) reinterpret_cast<int*>(xch)[0] = (int)atomicAdd(sp.counter, 2u);
        row_sync(pair, lgw);
        const int pitem = reinterpret_cast<const int*>(xch)[0];   // items pitem (forward), pitem + 1
        if (pitem >= sp.total_items) break;
        ItemRow it;
        const bool nonempty = decode_item(sp, istart, pitem + bwd, &it);
        float zmax = 0.f;
        int* cv = bwd ? sp.cv_bwd : sp.cv_fwd;
        if (nonempty) {
            const float zpart = stage_row<true>(sp, it, Fh, Fl, ends, lane, part, nw, false);
            if (lane == 0) xch[1 + part] = zpart;
            row_sync(pair, lgw);   // the staged row is complete
            for (int m = 1; m <= nw; ++m) zmax = fmaxf(zmax, xch[m]);
        }
        if (nonempty && df::beyond(zmax, it.h0)) {
            hand_over_row(sp, it, bwd != 0, zmax, cv, (part >> 1) * 32 + lane, 16 << lgw, Fl + ROW_PADL);
        } else if (nonempty) {
            if (PRUNE) {   // suffix and prefix maxima and the rows' records by the first two warps (one of each
                           // walk direction), a share of the window maxima by each
                if (part < 2 && lane == 0) {
#pragma unroll
                    for (int m = 0; m < 4; ++m) row->ends[m] = ends[m];
                    if (!skip_row(sp, it, bwd != 0, zmax, cv, false, LONG, row)) row->L = 0;
                }
                if (part == 1) end_max<true>(Fh, ZS, it.L, lane);
                if (part == 0) end_max<false>(Fh, ZS, it.L, lane);
                window_max<CERT_POV, U>(Fh, WM, it.L, lane, part, nw);
                row_sync(pair, lgw);   // every warp sees them
            }
            if constexpr (PRUNE) {
                const float* H = Fh + ROW_PADL;
                const int groups = (row->L + CERT_POV - 1) / CERT_POV;
                const int zs_off = (int)(ZS - H), wm_off = (int)(WM - H);
                if (bwd)
                    sweep_rows_skip<CERT_POV, U, LONG, END, true, SKIP_TESTS, SKIP_CHUNK>(sp, row, H, 0, groups, lgw - 1, part >> 1, zs_off,
                                                                     wm_off, tab, spill, lane);
                else
                    sweep_rows_skip<CERT_POV, U, LONG, END, false, SKIP_TESTS, SKIP_CHUNK>(sp, row, H, 0, groups, lgw - 1, part >> 1, zs_off,
                                                                     wm_off, tab, spill, lane);
            } else {
                const CertRow r = cert_row(sp, it, Fh, Fl, ends, zmax, cv, false);
                if (bwd) sweep_row_cert<CERT_POV, U, LONG, RANGED, true, true>(sp, r, tab, spill, lane);
                else sweep_row_cert<CERT_POV, U, LONG, RANGED, false, true>(sp, r, tab, spill, lane);
            }
        }
        row_sync(pair, lgw);   // both walks are done with the row (and with the exchange slot)
    }
    if (lane == 0) atomicAdd(&g_sweep_stats[3], (unsigned long long)(clock64() - t_start));
}

// The exact pass of a certified launch: every block the sweep flagged
// (a row key, the sample and its entry's kind, the row's |elevation| bound and
// the blocks) is decided again exactly, double-float or FP64 past its margin,
// on samples blended from the DEM as the staging does (the DEM is L2-resident
// while the sweep runs).  Bound by the latency of those gathers.  A warp takes
// two entries at a time: two FLAG_BLOCK entries of 16 steps in one go, a
// half-warp each, what else there is (longer blocks, the rest of walks flagged
// twice since their last rise, whole walks, FP64) with all 32 lanes.  An entry names its row directly (no search of the item
// table) and the counters stay in registers: 12 mixed tiles (7.3 million
// blocks) 214 -> 204 ms, 2000^2 (1.26 million) 95.5 -> 92.6 ms.
// flag_count[0] is the buffer's fill.
constexpr int EXACT_WARPS = 16;

__global__ void __launch_bounds__(EXACT_WARPS * 32, 2) exact_kernel(SweepParams sp)
{
    const int lane = threadIdx.x & 31;
    const unsigned n = min(sp.flag_count[0], (unsigned)sp.flag_cap);
    const long long t_start = clock64();
    unsigned count[2] = {0u, 0u};
    for (unsigned i = 2 * (blockIdx.x * EXACT_WARPS + (threadIdx.x >> 5)); i < n; i += 2 * gridDim.x * EXACT_WARPS) {
        const unsigned at = i + (lane >> 4);
        int4 en = make_int4(0, 0, 0, 0);
        ItemRow it;
        bool ok = at < n;
        if (ok) {
            en = sp.flag_buf[at];
            ok = in_range(en.x >> 16, sp.ndir, 22) && in_range(en.x >> 1 & 0x7fff, sp.dirs[en.x >> 16].R, 24) &&
                 decode_row(sp, en.x >> 16, en.x >> 1 & 0x7fff, (en.x & 1) != 0, &it) &&
                 in_range(en.y & 0xffff, it.L, 23);
        }
        ExactCtx c{};
        if (ok) c = exact_ctx(sp, it, __int_as_float(en.z));
        const int x = en.y & 0xffff, kind = en.y >> 16 & 3, e0 = en.w & 0x3fff, p0 = en.w >> 14;
        const bool half = ok && kind == FLAG_BLOCK && (en.y >> 18 & 15) <= 2 && (en.y >> 22) <= 2;
        bool left = ok;                       // the half's entry is still to do
        if (__any_sync(0xffffffffu, half)) {
            const bool esc = exact_half(c, half, x, e0, (en.y >> 18 & 15) * 8, p0, (en.y >> 22) * 8, lane);
            if (half && !esc) left = false;
            count[0] += __popc(__ballot_sync(0xffffffffu, half && !esc) & 0x00010001u);
        }
        const unsigned todo = __ballot_sync(0xffffffffu, left) & 0x00010001u;
        for (unsigned m = todo; m; m &= m - 1) {
            const int src = __ffs(m) - 1;
            const int key = __shfl_sync(0xffffffffu, en.x, src), y = __shfl_sync(0xffffffffu, en.y, src);
            const int z = __shfl_sync(0xffffffffu, en.z, src), w = __shfl_sync(0xffffffffu, en.w, src);
            decode_row(sp, key >> 16, key >> 1 & 0x7fff, (key & 1) != 0, &it);
            const ExactCtx cc = exact_ctx(sp, it, __int_as_float(z));
            exact_block(cc, y & 0xffff, w & 0x3fff, (y >> 18 & 15) * 8, w >> 14, (y >> 22) * 8, y >> 16 & 3, lane,
                        count);
        }
    }
    if (lane == 0) {
        if (count[0]) atomicAdd(&g_sweep_stats[0], (unsigned long long)count[0]);
        if (count[1]) atomicAdd(&g_sweep_stats[1], (unsigned long long)count[1]);
        atomicAdd(&g_sweep_stats[2], (unsigned long long)(clock64() - t_start));
    }
}

// The walks that found the flag buffer full: their measures are negative.
// Does nothing unless the sweep saw a full buffer; otherwise the measures of
// the whole launch are searched, 32 samples of an item at a time (a few long
// rows would leave most warps without one), evenly spaced, as marked samples
// stand together (a corner of equal no-data cells), and the marked walks walked
// exactly (100 x 100, 60 directions, a third of each side at -9999 seen from its
// own height: 5.0 -> 1.2 ms, with walks as fp64_walk now takes them).
__global__ void __launch_bounds__(EXACT_WARPS * 32, 2) exact_scan_kernel(SweepParams sp)
{
    if (sp.flag_count[2] == 0u) return;
    const int lane = threadIdx.x & 31;
    unsigned count[2] = {0u, 0u};
    const long long units = (long long)sp.total_items * sp.scan_blocks, step = (long long)gridDim.x * EXACT_WARPS;
    for (long long u = (long long)blockIdx.x * EXACT_WARPS + (threadIdx.x >> 5); u < units; u += step) {
        const int item = (int)(u / sp.scan_blocks), x0 = (int)(u % sp.scan_blocks), sx = sp.scan_blocks;
        ItemRow it;
        if (!decode_item(sp, sp.item_start, item, &it) || x0 >= it.L) continue;
        const int* cv = (it.rev ? sp.cv_bwd : sp.cv_fwd) + it.rowbase;
        const int xl = x0 + lane * sx;
        unsigned marked = __ballot_sync(0xffffffffu, xl < it.L && cv[xl] < 0);
        if (!marked) continue;
        ExactCtx c = exact_ctx(sp, it, 0.f);
        float zmax = 0.f;
        for (int x = lane; x < it.L; x += 32) {
            float va, vb;
            unsigned fr;
            dem_pair(c, x, va, vb, fr);
            zmax = fmaxf(zmax, fmaxf(fabsf(va), fabsf(vb)));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) zmax = fmaxf(zmax, __shfl_xor_sync(0xffffffffu, zmax, o));
        c = exact_ctx(sp, it, zmax);
        for (; marked; marked &= marked - 1) exact_walk(c, x0 + (__ffs(marked) - 1) * sx, lane, count);
    }
    if (lane == 0) {
        if (count[0]) atomicAdd(&g_sweep_stats[0], (unsigned long long)count[0]);
        if (count[1]) atomicAdd(&g_sweep_stats[1], (unsigned long long)count[1]);
    }
}

}  // namespace

// A long-walk launch keeps at least this many warps per CTA, shrinking the
// distance table (to no fewer than MIN_TABLE entries) when both do not fit.
constexpr int LONG_MIN_WARPS = 2;
constexpr int MIN_TABLE = 1024;

// Shared-memory sizes of a launch (floats), for rows of up to wmax samples and
// walks of up to dmax steps in a launch of ndir directions.
struct SweepSizes {
    int inv_len, tab, istart;   // distance table (entries, floats) and item table
    int padr, half, zs, wm;     // right pad, one staged array, end maxima, window maxima
    int row;                    // a packed row's arrays
    size_t room;                // what the tables leave (0 if they do not fit)
};

static SweepSizes sweep_sizes(int wmax, int dmax, bool prune, bool cert, int ndir, int smem_optin)
{
    SweepSizes z;
    // the distance table is read up to d = dmax + U (a walk of at most
    // min(K, W) - 1 steps, rounded up to U); dmax <= wmax
    z.inv_len = (std::min(dmax, wmax) + 2 * LARGE_UNROLL + 8 + 1) & ~1;
    z.tab = tab_floats_for(z.inv_len, prune, cert);
    z.istart = (ndir + 1 + 3) & ~3;
    z.padr = prune ? SKIP_PADR : ROW_PADR;
    z.half = (ROW_PADL + 4 + wmax + z.padr + 3) & ~3;
    z.zs = prune ? ((wmax + ZS_STRIDE - 1) / ZS_STRIDE + 4) & ~3 : 0;
    z.wm = prune ? ((wmax + SKIP_UNROLL + 3) / ZS_STRIDE + 4) & ~3 : 0;
    z.row = 2 * z.half + z.zs + z.wm;
    const size_t total = (size_t)smem_optin / 4, fixed = (size_t)z.tab + z.istart + (prune ? WM_SLACK : 0);
    z.room = fixed >= total ? 0 : total - fixed;
    return z;
}

// Certified warps that hold a row of their own in shared memory (launch_sweep
// gives them one when there are at least TVS_CERT_SINGLE_MIN, else rows go to
// pairs of warps).
static size_t cert_single_fit(const SweepSizes& z, bool prune)
{
    return z.room / (size_t)(prune ? SKIP_ROW_FLOATS + z.row : 2 * z.half + 4);
}

// log2 of the rows that PACK_WARPS warps of a packed launch can each stage.
static int pack_fit(const SweepSizes& z)
{
    int lg = 0;
    while (lg < PACK_MAX_LG && (size_t)PACK_WARPS * (size_t)(SKIP_ROW_FLOATS + z.row) * (2u << lg) <= z.room) ++lg;
    return lg;
}

int cert_sweep_class(int wmax, int dmax, int prune, int ndir, int smem_optin)
{
    if (wmax - 2 > LONG_WALK && dmax - 1 > LONG_WALK) return 0;
    const SweepSizes z = sweep_sizes(wmax, dmax, prune != 0, true, ndir, smem_optin);
    const size_t fit = cert_single_fit(z, prune != 0);
    if (fit < (size_t)TVS_CERT_SINGLE_MIN) return 0;
    if (fit < (size_t)CERT_WIDE_WARPS) return CERT_MAX_WARPS;
    return CERT_WIDE_WARPS << (prune ? pack_fit(z) : 0);
}

// Layout of a launch's CTAs in shared memory.
struct SweepLayout {
    bool single, pairs, longw;   // certified: rows of a warp's own, or shared ones; walks of more than LONG_WALK steps
    size_t single_fit;           // certified warps that could hold a row of their own
    size_t fit;                  // units that fit: warps, or the groups of warps that share a row
    int most;                    // most warps of its kernel
    int units, warps;            // units and warps of a CTA
    size_t smem;                 // its bytes
};

// Fills the sizes of sp (ndir and total_items are set) and the layout of a
// launch with rows of up to wmax samples and walks of up to dmax steps; false
// when they do not fit.
static bool sweep_layout(SweepParams& sp, int wmax, int dmax, bool prune, bool cert, int num_sms, int smem_optin,
                         int max_warps, SweepLayout* lay)
{
    const int ndir = sp.ndir, total_items = sp.total_items;
    const SweepSizes z = sweep_sizes(wmax, dmax, prune, cert, ndir, smem_optin);
    sp.inv_len = z.inv_len;
    sp.tab_floats = z.tab;
    sp.istart_len = z.istart;
    sp.padr = z.padr;
    sp.half = z.half;
    sp.zs_len = z.zs;
    sp.wm_len = z.wm;
    sp.per_row = z.row;
    sp.lgna = 0;
    const bool longw = wmax - 2 > LONG_WALK && dmax - 1 > LONG_WALK;
    const int lspill = longw ? 32 * (cert || prune ? CERT_POV : LARGE_POV) : 0;
    // FP32 decisions: one row per warp.  Certified: rows of a warp's own (one,
    // reversed for backward walks, or when pruned up to 2^PACK_MAX_LG) when
    // TVS_CERT_SINGLE_MIN such warps fit, else one row per pair of warps (both
    // staged arrays, the maxima, the end samples, an exchange slot and pruned
    // each warp's SkipRow), and per warp its spill: a row's samples are then
    // held once for both walk directions.
    lay->single_fit = cert ? cert_single_fit(z, prune) : 0;
    const int single_min = TVS_CERT_SINGLE_MIN;
    lay->longw = longw;
    lay->single = cert && !longw && (max_warps == 0 || max_warps >= single_min) &&
                  lay->single_fit >= (size_t)single_min;
    lay->pairs = cert && !lay->single;
    const bool single = lay->single, pairs = lay->pairs;
    if (single && prune) {
        // as many rows as fit, while every warp still finds several packs to
        // claim: the last packs of a launch run alone (100 x 100, 180
        // directions: 232 us with at least 3 packs per warp, 255 with 1)
        const int cap = max_warps == 0 || max_warps >= PACK_WARPS ? pack_fit(z) : 0;
        while (sp.lgna < cap && (long long)total_items >> (sp.lgna + 1) >=
                                    (long long)PACK_MIN_CLAIMS * num_sms * PACK_WARPS)
            ++sp.lgna;
    }
    sp.per_pair = pairs ? 2 * sp.half + 2 * sp.zs_len + sp.wm_len + 4 + ROW_XCH + (prune ? 2 * SKIP_ROW_FLOATS : 0) : 0;
    sp.per_warp = single ? (prune ? (SKIP_ROW_FLOATS + z.row) << sp.lgna : 2 * sp.half + 4)
                : pairs ? lspill
                        : sp.half + sp.zs_len + sp.wm_len + lspill;
    // warps per shared row: more than two where that raises the warps of an SM
    // by a fifth
    sp.lgw = 1;
    if (pairs && prune) {
        const int most = max_warps > 0 ? std::max(std::min(max_warps, SKIP_WARPS), 2) : SKIP_WARPS;
        auto warps_of = [&](int lgw) {
            const size_t unit = (size_t)sp.per_pair + ((size_t)sp.per_warp << lgw);
            return (int)std::min<size_t>(std::max<size_t>(z.room / unit, longw ? 1 : 0), (size_t)(most >> lgw)) << lgw;
        };
        for (int lgw = 2; lgw <= MAX_LGW; ++lgw)
            if (warps_of(lgw) > 0 && 5 * warps_of(lgw) >= 6 * warps_of(sp.lgw)) sp.lgw = lgw;
    }
    // shared memory of one unit: the warps that share a row, or one warp
    const int uw = pairs ? 1 << sp.lgw : 1;
    const size_t unit = (size_t)(sp.per_pair + uw * sp.per_warp) * 4;
    const size_t slack = prune ? WM_SLACK * 4 : 0;   // past the last warp's window maxima
    size_t fixed = (size_t)(sp.tab_floats + sp.istart_len) * 4 + slack;
    if (longw && fixed + (size_t)std::max(1, LONG_MIN_WARPS / uw) * unit > (size_t)smem_optin) {
        // Rows of more than about 10^4 samples: the whole table and several
        // staged rows do not fit together.  Keep LONG_MIN_WARPS warps (or as
        // many as fit) and a table of what is left (at least MIN_TABLE
        // entries); the long-walk sweep computes the entries past its end.
        const size_t base = (size_t)sp.istart_len * 4 + slack;
        int w = std::max(1, LONG_MIN_WARPS / uw);
        const size_t min_tab = (size_t)tab_floats_for(MIN_TABLE, prune, cert) * 4;
        while (w > 1 && base + min_tab + (size_t)w * unit > (size_t)smem_optin) --w;
        if (base + 16 * 4 + (size_t)w * unit >= (size_t)smem_optin) return false;
        // floats that fit, and the most entries whose slots do
        const size_t room = ((size_t)smem_optin - base - (size_t)w * unit) / 16 * 4;
        sp.inv_len = (int)std::min<size_t>((size_t)sp.inv_len, tab_entries_fit(room, prune, cert)) & ~1;
        sp.tab_floats = tab_floats_for(sp.inv_len, prune, cert);
        fixed = (size_t)(sp.tab_floats + sp.istart_len) * 4 + slack;
    }
    if (fixed + unit > (size_t)smem_optin) return false;
    // As many resident units as shared memory and registers allow, in one CTA
    // per SM (the 1/d table is shared by the CTA).
    lay->fit = (smem_optin - fixed) / unit;
    // (unpruned certified launches take 16 warps, of 128 registers, where that many
    // fit, else 12)
    const bool wide = max_warps == 0 || max_warps >= CERT_WIDE_WARPS;
    if (single)
        lay->most = prune ? (sp.lgna > 0 ? PACK_WARPS : SINGLE_WARPS)
                    : wide && lay->single_fit >= (size_t)CERT_WIDE_WARPS ? CERT_WIDE_WARPS : CERT_MAX_WARPS;
    else if (pairs)
        lay->most = prune ? SKIP_WARPS
                    : wide && !longw && lay->fit * 2 >= (size_t)CERT_WIDE_WARPS ? CERT_WIDE_WARPS : CERT_MAX_WARPS;
    else
        lay->most = prune ? FP32_WARPS : SWEEP_MAX_WARPS;
    const int cap = max_warps > 0 ? std::max(std::min(max_warps, lay->most), uw) : lay->most;
    lay->units = (int)std::min<size_t>(lay->fit, (size_t)(cap / uw));
    lay->warps = lay->units * uw;
    lay->smem = fixed + (size_t)lay->units * unit;
    return true;
}

cudaError_t launch_sweep(const DirDev* d_dirs, const JobDev* d_jobs, const int* d_item_start, int ndir,
                         int total_items, const int* rowlo, const int* rowhi, int* cv_fwd, int* cv_bwd, int wmax,
                         int dmax, bool ranged, int prune, int cert, unsigned* counter, int4* flag_buf, unsigned* flag_count,
                         int flag_cap, int num_sms, int smem_optin, int max_warps, cudaStream_t stream)
{
    if (ndir <= 0 || total_items <= 0) return cudaSuccess;
    SweepParams sp;
    sp.dirs = d_dirs; sp.jobs = d_jobs; sp.item_start = d_item_start; sp.rowlo = rowlo;
    sp.rowhi = rowhi; sp.cv_fwd = cv_fwd; sp.cv_bwd = cv_bwd; sp.counter = counter; sp.ndir = ndir;
    sp.total_items = total_items;
    sp.scan_blocks = (wmax + 31) / 32;
    if (cert && !flag_count) return cudaErrorInvalidValue;
    sp.flag_buf = flag_buf;
    sp.flag_count = flag_count;
    sp.flag_cap = flag_buf ? flag_cap : 0;
    SweepLayout lay;
    if (!sweep_layout(sp, wmax, dmax, prune != 0, cert != 0, num_sms, smem_optin, max_warps, &lay))
        return cudaErrorInvalidConfiguration;
    constexpr int CW = CERT_MAX_WARPS, WW = CERT_WIDE_WARPS, FW = SWEEP_MAX_WARPS;
    const bool wide = lay.most == WW, longw = lay.longw;
    void (*kern)(SweepParams);
    if (lay.single) {
        if (!prune) kern = ranged ? (wide ? sweep_cert_kernel<false, true, WW> : sweep_cert_kernel<false, true, CW>)
                                  : (wide ? sweep_cert_kernel<false, false, WW> : sweep_cert_kernel<false, false, CW>);
        else if (sp.lgna > 0) kern = ranged ? sweep_pack_kernel<true, PACK_WARPS, PACK_TESTS, PACK_CHUNK>
                                            : sweep_pack_kernel<false, PACK_WARPS, PACK_TESTS, PACK_CHUNK>;
        else kern = ranged ? sweep_pack_kernel<true, SINGLE_WARPS, SKIP_TESTS, SINGLE_CHUNK>
                           : sweep_pack_kernel<false, SINGLE_WARPS, SKIP_TESTS, SINGLE_CHUNK>;
    } else if (lay.pairs) {
        if (prune && longw) kern = sweep_pair_kernel<true, true, true, SKIP_WARPS>;
        else if (prune) kern = ranged ? sweep_pair_kernel<true, false, true, SKIP_WARPS>
                                      : sweep_pair_kernel<true, false, false, SKIP_WARPS>;
        else if (wide) kern = ranged ? sweep_pair_kernel<false, false, true, WW> : sweep_pair_kernel<false, false, false, WW>;
        else kern = longw ? sweep_pair_kernel<false, true, true, CW> : sweep_pair_kernel<false, false, true, CW>;
    } else {
        if (!prune) kern = longw ? sweep_kernel<false, true, true, FW> : sweep_kernel<false, false, true, FW>;
        else if (longw) kern = sweep_kernel<true, true, true, FP32_WARPS>;
        else kern = ranged ? sweep_kernel<true, false, true, FP32_WARPS> : sweep_kernel<true, false, false, FP32_WARPS>;
    }
    cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)lay.smem);
    if (err != cudaSuccess) return err;
    int per_sm = 0;
    err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, lay.warps * 32, lay.smem);
    if (err != cudaSuccess) return err;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    kern<<<per_sm * num_sms, lay.warps * 32, lay.smem, stream>>>(sp);
    err = cudaGetLastError();
    if (err != cudaSuccess || !cert) return err;
    // the exact pass: no shared memory, as many warps as registers allow
    int xper = 0;
    err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&xper, exact_kernel, EXACT_WARPS * 32, 0);
    if (err != cudaSuccess) return err;
    if (xper < 1) return cudaErrorInvalidConfiguration;
    exact_kernel<<<xper * num_sms, EXACT_WARPS * 32, 0, stream>>>(sp);
    err = cudaGetLastError();
    if (err != cudaSuccess) return err;
    exact_scan_kernel<<<2 * num_sms, EXACT_WARPS * 32, 0, stream>>>(sp);   // two resident CTAs per SM
    return cudaGetLastError();
}

}  // namespace tvs

extern "C" int tvs_debug_sweep_layout(int wmax, int dmax, int ndir, int items, int prune, int fp32_decisions,
                                      int max_warps, int num_sms, int smem_optin, int32_t* out)
{
    if (!out || wmax < 2 || dmax < 1 || ndir < 1 || items < 1 || max_warps < 0 || num_sms < 1) return TVS_ERR_ARG;
    tvs::SweepParams sp{};
    sp.ndir = ndir;
    sp.total_items = items;
    tvs::SweepLayout lay;
    if (!tvs::sweep_layout(sp, wmax, dmax, prune != 0, !fp32_decisions, num_sms, smem_optin, max_warps, &lay))
        return TVS_ERR_OOM;
    out[0] = lay.warps;
    out[1] = lay.pairs ? 1 << sp.lgw : 1;
    out[2] = 1 << sp.lgna;
    return TVS_OK;
}

extern "C" int tvs_debug_sweep_stats(uint64_t* out, int clear)
{
    if (!out) return TVS_ERR_ARG;
    cudaError_t e = cudaDeviceSynchronize();
    if (e == cudaSuccess) e = cudaMemcpyFromSymbol(out, tvs::g_sweep_stats, sizeof(unsigned long long) * 4);
    if (e == cudaSuccess && clear) {
        const unsigned long long zero[4] = {0, 0, 0, 0};
        e = cudaMemcpyToSymbol(tvs::g_sweep_stats, zero, sizeof(zero));
    }
    return e == cudaSuccess ? TVS_OK : TVS_ERR_CUDA;
}

extern "C" int tvs_debug_sweep_check(int32_t* out, int clear)
{
    if (!out) return TVS_ERR_ARG;
    cudaError_t e = cudaDeviceSynchronize();
    if (e == cudaSuccess) e = cudaMemcpyFromSymbol(out, tvs::g_sweep_check, sizeof(int) * 4);
    if (e == cudaSuccess && clear) {
        const int zero[4] = {0, 0, 0, 0};
        e = cudaMemcpyToSymbol(tvs::g_sweep_check, zero, sizeof(zero));
    }
    return e == cudaSuccess ? TVS_OK : TVS_ERR_CUDA;
}

// cf_pair.cuh -- the persistent pair kernel (template; instantiated per kind in cf_pair_*.cu).
//
// Sec. 4.3-4.7 on a GPU.  Every warp repeatedly takes one work item -- an i tile of one cell
// (<= 128 points) against a j range (<= 512 points) of a neighbour cell -- from a global atomic
// cursor, and works through the tile in groups of 32 points: lane l holds one i point in registers,
// translated by the cell-pair shift (Sec. 4.4, Code corrfunc_pbc: the shift is added once per i, not
// per pair).
//
// Gathering: the warp reads the j range 32 points at a time, one per lane, tests each against the
// bounding box of the group's 32 i points (the late entry / early exit of Sec. 4.5, point by point)
// and gathers the points within reach in shared memory as float arrays.  The smallest separation the
// box allows is formed with operations that round monotonically, and the limit lies above the largest
// edge by the FP32 error of that form (CfDevPlan::reach_r), so no pair that counts is dropped.
// Counting: whenever 32 points are gathered (and at the end of the range) every lane forms its pairs
// with them, four at a time: packed FP32x2 separations on cell-relative coordinates -- with the
// shift's low part and the TwoSum residual of the i translation when ravg needs relative accuracy --
// binned through a table over the separation (one byte a cell; outside every bin is a class of it), the
// equally wide pi bins by one multiplication.  A table cell that holds an edge, or a value near a pi
// edge, resolves through the full tables on the squared separation's bits (Sec. 4.7); a value within
// the proven FP32 error band of an edge is not binned: the pair goes to a global queue and is
// re-evaluated in FP64 by the recheck kernel, so counts equal the FP64 result.
//
// What bounds it: instruction issue for the counts (rp-pi 86 to 88 % of the slots, wp 85 %, theta 83 % beside 81 % of the
// shared-memory wavefronts, mocks 78 %), for the sums the shared-memory wavefronts (73 % for r, 88 % for 2M points of
// rp-pi: a 16-byte Kahan update per pair and lane, five atomics per pair of rp-pi) at the 16 warps per SM that their
// histograms leave.  Counting costs 17 (DD(theta), counts only) to 30 (weights and ravg) instructions per gathered
// point and warp, gathering about 70 per 32 j points, so the layout aims at few gathered points per pair in
// range: counted in the kernel, clustered catalogues form 1.34 (1M points, separations to 40) to 1.84 (angles) pairs per
// pair in range, mocks 2.40 (their reach is a sphere, a counted pair lies in a cylinder), where whole cell pairs form 4
// to 8.  Gathering also fills the blocks: a cell's ragged end costs at most three points of a
// range's last block, and a tile's last group shares the warp (below).
// Measured against whole cell pairs with a branch per pair in range (pair kernel, one GB300): DD(r) of
// 1M clustered points with weights and ravg 1.546 -> 0.981 ms, counts to twice the separation
// 5.25 -> 2.06 ms, DD(rp, pi) of 2M points 1.505 -> 0.879 ms, its DR against 4M randoms 5.17 -> 2.70 ms,
// DD(theta) of 1M points 1.176 -> 0.623 ms, DR of the survey cone 5.48 -> 1.81 ms.
//
// Histograms live in shared memory per warp (Sec. 4.8: private histograms, merged once): for
// r / theta / wp one private copy per lane (no bank conflicts, no contention; weighted sums
// Kahan-compensated in FP32), for rp-pi one copy per warp updated by shared atomics (weight and
// ravg sums in fixed point where the host found scales for the terms' range, else FP64).  They are
// merged into the global histogram when a warp moves to another job, after every 2^28 evaluated
// pairs (2^18 with fixed-point sums), and at exit.
//
// The fixed-point sums use 32-bit shared atomics only (64-bit shared atomics are several times
// slower): a term t adds m = round(t * S) (S a power of two the host chose so that every term of
// the sum lies in [2^21, 2^26) units, so that rounding moves a term by at most 2^-22 of itself) to
// two 32-bit words of its slot, m modulo 2^32 and m >> 12.  A warp flushes before its slots can
// hold 2^18 terms: the second word then stays below 2^32 and places the true sum within 2^30 below
// its value times 2^12, and the first word gives the sum exactly (fx_sum).
#pragma once
#include <math_constants.h>

#include "cf_build.h"
#include "cf_device.cuh"

namespace cfpair {

constexpr int KIND_R = 0, KIND_RPPI = 1, KIND_WP = 2, KIND_THETA = 3, KIND_MOCKS = 4;

// rp-pi kinds keep one histogram per warp updated by shared atomics (nb * npi slots)
__host__ __device__ constexpr bool warp_hist(int kind) { return kind == KIND_RPPI || kind == KIND_MOCKS; }

__host__ __device__ __forceinline__ uint32_t align16(uint32_t x) { return (x + 15u) & ~15u; }

// per-warp shared memory: (counts only) two work items, the current and the next | gathered j points |
// histogram
//   gathered points: a ring of GBUF points as 3-7 float arrays (x, y, z[, w][, lo parts of x, y, z])
//   and the points' places in the j range (u16)
// a warp flushes its histograms once it has evaluated more than this many pairs of one job;
// with the item in hand that keeps every flushed batch at <= 2^28 pairs (an item: <= 2^16)
constexpr uint32_t CF_FLUSH_PAIRS = (1u << 28) - (1u << 16);
// with fixed-point sums: fewer than 2^18 terms per slot between flushes
constexpr uint32_t FX_FLUSH_PAIRS = (1u << 18) - (1u << 16);
constexpr uint32_t FX_HI_SHIFT = 12;

// True sum of the fixed-point terms of a slot from its two words: lo = the sum modulo 2^32, hi = the
// sum of (m >> 12).  For fewer than 2^18 terms below 2^26, hi * 2^12 lies in (T - 2^30, T].
__device__ __forceinline__ unsigned long long fx_sum(uint32_t lo, uint32_t hi)
{
    const unsigned long long c = (unsigned long long)hi << FX_HI_SHIFT;
    return c + (uint32_t)(lo - (uint32_t)c);
}
// that sum divided by its scale 2^s: below 2^52 it is the mantissa of 2^52 + T, with any exponent (one FP64
// operation; a conversion and a division take a dozen: 700k points over (rp, pi) with both sums 827 -> 790 us)
__device__ __forceinline__ double fx_value(unsigned long long T, float scale)
{
    const unsigned long long e = (unsigned long long)(1075 + 127 - (__float_as_uint(scale) >> 23)) << 52;
    return __longlong_as_double((long long)(e | T)) - __longlong_as_double((long long)e);
}
constexpr uint32_t GBUF = 64;
// widening of a group's half width on an axis of explicit minimum image, over the side: 64 roundings
constexpr float WRAP_MARGIN = 1.0f / 262144.0f;
// bits of 2^23: a value below 2^22 added to it has its integer part in the low bits of the sum
constexpr uint32_t MAGIC_BITS = 0x4B000000u;
// Counts-only instances run 32 warps per SM on 64 registers: they keep the work item and the next one in
// shared memory (24 registers otherwise).  The others have the registers and need the shared memory.
__host__ __device__ constexpr bool smem_items(bool W, bool R) { return !W && !R; }
__host__ __device__ constexpr uint32_t item_bytes(bool W, bool R) { return smem_items(W, R) ? 2u * sizeof(CfItem) : 0u; }
static_assert(sizeof(CfItem) % 16 == 0, "items are copied 16 bytes at a time");
// Histogram rows past the bins: a separation outside every bin reads class nb, one that the full tables
// must decide class nb + 1.  Counts-only kinds add there as well instead of testing (lane-private rows; one
// word per lane past a per-warp histogram), and nothing reads those rows.
constexpr uint32_t SPARE = 2;
__host__ __device__ __forceinline__ uint32_t warp_hist_bytes(int kind, bool W, bool R, int nslot)
{
    if (warp_hist(kind)) {
        uint32_t b = (((uint32_t)nslot + (W || R ? 0u : 32u)) * 4u + 7u) & ~7u;
        if (W) b += nslot * 8u;
        if (R) b += nslot * 8u;
        return align16(b);
    }
    uint32_t b = (nslot + (W || R ? 0u : SPARE)) * 32u * 4u;
    if (W) b += nslot * 32u * 8u;
    if (R) b += nslot * 32u * 8u;
    return b;
}
__host__ __device__ constexpr bool has_z(int kind) { return kind == KIND_RPPI || kind == KIND_WP; }
// kinds that bin a second value (|dz|; for mocks pi^2)
__host__ __device__ constexpr bool has_pi(int kind) { return has_z(kind) || kind == KIND_MOCKS; }
__host__ __device__ constexpr uint32_t stage_arrays(bool W, bool LO) { return LO ? 7u : (W ? 4u : 3u); }
__host__ __device__ constexpr uint32_t warp_jbuf_bytes(bool W, bool R, bool LO)
{
    return item_bytes(W, R) + stage_arrays(W, LO) * GBUF * 4u + GBUF * 2u + (!W && !R ? 32u : 0u);     // 32: the box
}
__host__ __device__ __forceinline__ uint32_t warp_bytes(int kind, bool W, bool R, bool LO, int nslot)
{
    return warp_jbuf_bytes(W, R, LO) + warp_hist_bytes(kind, W, R, nslot);
}

// per-CTA shared memory past the separation table: the ravg scales per rp bin (rp-pi, mocks), or the
// spare row of the sums of the other kinds (a count, and two Kahan pairs at most, per lane)
__host__ __device__ __forceinline__ uint32_t cta_extra_bytes(int kind, bool W, bool R, int nb)
{
    if (warp_hist(kind)) return align16(4u * (uint32_t)nb);
    return W || R ? 32u * 20u : 0u;
}

// Kahan-compensated FP32 sum: s holds the sum, c the negated lost low part
__device__ __forceinline__ void kahan_step(float &s, float &c, float v)
{
    const float y = v - c;
    const float t = s + y;
    c = (t - s) - y;
    s = t;
}
__device__ __forceinline__ void kahan_add(float2 *p, float v)
{
    float2 sc = *p;
    kahan_step(sc.x, sc.y, v);
    *p = sc;
}

// class of a non-negative value's bit pattern from the full (16-bit) table in global memory
__device__ __forceinline__ uint32_t lut_class(const uint16_t *__restrict__ words, const CfFine *__restrict__ fine,
                                              const CfLut &L, uint32_t vb)
{
    const uint32_t idx = min((max(vb, L.base) - L.base) >> L.shift, L.last);
    uint32_t c = words[L.coff + idx];
    if (c >= CFI_FINE_FLAG) {
        const CfFine f = fine[c - CFI_FINE_FLAG];
        uint32_t seg = (vb >= f.t1 ? 1u : 0u) + (vb >= f.t2 ? 1u : 0u);
        c = (f.code >> (8u * seg)) & 0xFFu;
    }
    return c;
}

__device__ __forceinline__ float f_rcp_approx(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
// denormals as 0 (one instruction): the table sends separations that small to the full tables
__device__ __forceinline__ float f_sqrt_ftz(float x)
{
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ uint32_t lds_u8(uint32_t addr)
{
    uint32_t r;
    asm("ld.shared.u8 %0, [%1];" : "=r"(r) : "r"(addr));
    return r;
}
__device__ __forceinline__ float pick4(const float (&v)[4], int h)
{
    const float a = h & 1 ? v[1] : v[0], b = h & 1 ? v[3] : v[2];
    return h & 2 ? b : a;
}

__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e)
{
    s = a + b;
    float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

__device__ __forceinline__ float wrap1(float d, float L, float invL) { return fmaf(-L, rintf(d * invL), d); }

__device__ __forceinline__ u64 wrap2(u64 d, float L, float invL)
{
    return f2_pack(wrap1(f2_lo(d), L, invL), wrap1(f2_hi(d), L, invL));
}

// queue one pair for the FP64 recheck (rare: kept out of line so the pair loops stay small)
static __device__ __noinline__ void push_recheck(const CfPairArgs &a, uint32_t ip, uint32_t jp, uint32_t job)
{
    const unsigned long long k = atomicAdd(a.qcount, 1ull);
    if (k < a.qcap) a.queue[k] = make_uint4(cf_orig(a.orig, a.pt, ip), cf_orig(a.orig, a.pt, jp), job, 0u);
}

// rp of a counted pair of the mocks kind, for ravg (Appendix A.2.1).  rp^2 = |s x l|^2 / |l|^2,
// and s x l = s x v_i because l = v_i - s / 2: the cancellation that makes s.s - pi^2 inaccurate
// for rp << pi moves into one cross product of exactly known numbers (s as a hi + lo pair from
// the cell-relative coordinates, v_i as float32 plus its lo part), taken by Kahan's difference of
// products (error <= 2u of each component).  ip: the i point; bj: the gathered j point; sh / sl: the
// item's shift, hi and lo.  Rare (counted pairs with ravg
// only), so kept out of line.
template <bool LO>
static __device__ __noinline__ float mocks_rp(const CfPairArgs &a, uint32_t ip, const float *bj,
                                              float shx, float shy, float shz, float slx, float sly, float slz)
{
    const float4 P = a.pt[ip], A = a.pabs[ip];
    const float X[3] = {-P.x, -P.y, -P.z}, Ah[3] = {A.x, A.y, A.z};
    const float ish[3] = {shx, shy, shz}, isl[3] = {slx, sly, slz};
    float XL[3] = {0.f, 0.f, 0.f}, AL[3] = {0.f, 0.f, 0.f}, XJL[3] = {0.f, 0.f, 0.f};
    if (LO) {
        const float4 C = a.plo[ip], D = a.pabslo[ip];
        XL[0] = -C.x; XL[1] = -C.y; XL[2] = -C.z;
        AL[0] = D.x; AL[1] = D.y; AL[2] = D.z;
        XJL[0] = bj[4 * GBUF]; XJL[1] = bj[5 * GBUF]; XJL[2] = bj[6 * GBUF];
    }
    const float XJ[3] = {bj[0], bj[GBUF], bj[2 * GBUF]};   // -X_j
    float sh[3], sl[3], l[3];
#pragma unroll
    for (int d = 0; d < 3; d++) {
        float h, e, h2, e2;
        two_sum(X[d], ish[d], h, e);          // X_i + shift hi, exactly h + e
        two_sum(h, XJ[d], h2, e2);            // - X_j, exactly h2 + e2
        sh[d] = h2;
        sl[d] = ((e + e2) + isl[d]) + (XL[d] + XJL[d]);
        l[d] = fmaf(-0.5f, sh[d], Ah[d]) + (AL[d] - 0.5f * sl[d]);
    }
    float c2 = 0.f;
#pragma unroll
    for (int d = 0; d < 3; d++) {
        const int p = (d + 1) % 3, q = (d + 2) % 3;
        // component d of s x A: s_p A_q - s_q A_p
        const float w = sh[q] * Ah[p];
        const float err = fmaf(sh[q], Ah[p], -w);
        const float f = fmaf(sh[p], Ah[q], -w);
        const float corr = (sh[p] * AL[q] - sh[q] * AL[p]) + (sl[p] * Ah[q] - sl[q] * Ah[p]);
        const float c = (f - err) + corr;
        c2 = fmaf(c, c, c2);
    }
    const float ll = fmaf(l[2], l[2], fmaf(l[1], l[1], l[0] * l[0]));
    return sqrtf(__fdiv_rn(c2, ll));
}

// GH (rp-pi and mocks only): no per-warp histogram; every pair adds straight into the job's global
// histogram (CfPairArgs::ghist).  FX (rp-pi and mocks, per-warp histogram): the weight and ravg sums
// are fixed point (two 32-bit words per slot) at the scales CfPairArgs::fxw / fxr_bin, else FP64.
template <int KIND, bool W, bool R, bool WRAP, bool LO, bool GH, bool FX>
struct Warp {
    const CfPairArgs &a;
    uint32_t lut;           // separation table in shared memory: its address, less MAGIC_BITS
    uint32_t *h_cnt;        // lane-private [nslot][32] (this and the sums: at the lane's column) or
                            // per-warp [nslot]
    float2 *h_w;            // lane-private Kahan pairs of the sum kept (interleaved when both are)
    uint32_t *d_cnt;        // the CTA's spare row: count and sums nobody reads (all of its warps write there without
                            // atomics: what they lose of one another does not matter)
    float2 *d_w;
    double *h_wd, *h_rd;    // per-warp sums (rp-pi, mocks): FP64, or with FX two 32-bit words per slot
                            // (nslot low words, then nslot high words)
    const float *fxr_bin;   // with FX and ravg: the scale of each rp bin's ravg terms (shared memory)
    float *jst;             // gathered j points
    uint16_t *gj;           // their places in the j range
    int lane;
    float Lx, Ly, Lz, iLx, iLy, iLz;

    __device__ Warp(const CfPairArgs &args) : a(args) {}

    // index of a gathered point among the sorted points
    __device__ __forceinline__ uint32_t gidx(const CfItem &it, const float *bs, uint32_t k) const
    {
        return it.jbeg + gj[(bs - jst) + k];
    }
    static __device__ __forceinline__ uint32_t job(const CfItem &it) { return it.meta & CFI_ITEM_JOBMASK; }

    // Table classes of two separations (bin; nb: outside every bin; nb + 1: for the full tables to decide).
    // The cell is the separation times lut_scale, rounded to an integer by adding 2^23; values past the
    // table and NaN clamp to its last cell.
    __device__ __forceinline__ void lut2(float r0, float r1, uint32_t &c0, uint32_t &c1) const
    {
        const u64 n = f2_fma(f2_pack(r0, r1), a.lut_scale2, f2_pack(8388608.0f, 8388608.0f));
        c0 = lds_u8(lut + min(f2_lo_bits(n), a.lut_top));
        c1 = lds_u8(lut + min(f2_hi_bits(n), a.lut_top));
    }

    __device__ __forceinline__ void push(const CfItem &it, uint32_t ip, uint32_t jp) { push_recheck(a, ip, jp, job(it)); }

    // Add to a lane's histogram of r, theta or wp, in bin c where `in` holds and in the CTA's spare row
    // otherwise (no branch: the four pairs' chains overlap)
    __device__ __forceinline__ void add_lane(bool in, uint32_t c, float r, float wp)
    {
        const uint32_t idx = c * 32u;       // the histogram pointers carry the lane
        atomicAdd(in ? h_cnt + idx : d_cnt, 1u);
        if (R && KIND == KIND_THETA) r = 2.0f * asinf(0.5f * r) * 57.29577951308232f;
        if (W && R) {
            // both sums of a lane's bin sit in one 16-byte word (sums, then their compensations): one load,
            // one packed compensated step, one store
            ulonglong2 *p = reinterpret_cast<ulonglong2 *>(in ? h_w + 2u * idx : d_w);
            ulonglong2 v = *p;
            const u64 y = f2_sub(f2_pack(wp, __fmul_rn(wp, r)), v.y);
            const u64 t = f2_add(v.x, y);
            v.y = f2_sub(f2_sub(t, v.x), y);
            v.x = t;
            *p = v;
        } else if (W || R) {
            kahan_add(in ? h_w + idx : d_w, W ? wp : r);
        }
    }

    __device__ __forceinline__ void acc_sh(const CfItem &it, uint32_t slot, uint32_t rbin, float r, float wp)
    {
        if (GH) {
            // no per-warp histogram: straight into the job's global one
            const size_t g = (size_t)job(it) * (uint32_t)a.nslot + slot;
            atomicAdd(a.hcnt + g, 1ull);
            if (W) atomicAdd(a.hw + g, (double)wp);
            if (R) atomicAdd(a.hr + g, (double)(W ? wp * r : r));
            return;
        }
        atomicAdd(h_cnt + slot, 1u);
        if (W) add_sum(h_wd, slot, wp, a.fxw);
        if (R) add_sum(h_rd, slot, W ? wp * r : r, FX ? fxr_bin[rbin] : 0.f);
    }

    // One term of a per-warp sum: with FX m = round(t * scale) into the slot's two 32-bit words (m
    // and m >> 12; the scale is a power of two, so t * scale is exact), else an FP64 add.
    __device__ __forceinline__ void add_sum(double *h, uint32_t slot, float t, float scale) const
    {
        if (FX) {
            uint32_t *w = reinterpret_cast<uint32_t *>(h);
            const uint32_t m = __float2uint_rn(t * scale);
            atomicAdd(w + slot, m);
            atomicAdd(w + a.nslot + slot, m >> FX_HI_SHIFT);
        } else {
            atomicAdd(h + slot, (double)t);
        }
    }

    // The i point of a lane, translated by the item's shift.  A lane past the tile holds NaN: every
    // separation it forms is NaN, which the table puts outside every bin.
    struct IPoint {
        u64 s[3], e[3];         // x_i + shift, and with ravg its low part (in both halves)
        u64 a[3];               // mocks: the absolute position
        float w;
        uint32_t p;             // its index among the sorted points
    };

    __device__ __forceinline__ void load_i(const CfItem &it, uint32_t ip, bool live, IPoint &I) const
    {
        I.p = ip;
        I.w = 0.f;
#pragma unroll
        for (int d = 0; d < 3; d++) {
            I.s[d] = f2_pack(CUDART_NAN_F, CUDART_NAN_F);
            I.e[d] = I.a[d] = 0ull;
        }
        if (!live) return;
        const float4 P = a.pt[ip];
        const float X[3] = {-P.x, -P.y, -P.z};
        float XL[3] = {0.f, 0.f, 0.f};
        if (LO) {
            const float4 l = a.plo[ip];
            XL[0] = -l.x;
            XL[1] = -l.y;
            XL[2] = -l.z;
        }
        if (KIND == KIND_MOCKS) {
            const float4 q = a.pabs[ip];
            I.a[0] = f2_pack(q.x, q.x);
            I.a[1] = f2_pack(q.y, q.y);
            I.a[2] = f2_pack(q.z, q.z);
        }
#pragma unroll
        for (int d = 0; d < 3; d++) {
            if (R) {
                float s, e;
                two_sum(X[d], it.s[d], s, e);
                I.s[d] = f2_pack(s, s);
                const float l = (e + it.slo[d]) + XL[d];
                I.e[d] = f2_pack(l, l);
            } else {
                const float s = X[d] + it.s[d];
                I.s[d] = f2_pack(s, s);
            }
        }
        I.w = P.w;
    }

    // Add the pair with the gathered point bj (weight wj) to the histogram: rp (or r) bin cr, pi bin cz,
    // FP32 separation r
    __device__ __forceinline__ void add_pair(const CfItem &it, const IPoint &I, uint32_t cr, uint32_t cz, float r,
                                             float wj, const float *bj)
    {
        const float wp = W ? __fmul_rn(I.w, wj) : 0.f;
        if (KIND == KIND_MOCKS) {
            if (R) r = mocks_rp<LO>(a, I.p, bj, it.s[0], it.s[1], it.s[2], it.slo[0], it.slo[1],
                                     it.slo[2]);
            acc_sh(it, cr * (uint32_t)a.npi + cz, cr, r, wp);
        } else if (KIND == KIND_RPPI) {
            acc_sh(it, cr * (uint32_t)a.npi + cz, cr, r, wp);
        } else {
            add_lane(true, cr, r, wp);
        }
    }

    // Bin the pairs of this lane's i point with the gathered j points j4 .. j4 + 3 (of the block at bs).
    // All four are formed and classified at once (independent chains, packed arithmetic); there is no
    // test for "in range" before the table: a value past the last edge reads the class outside every
    // bin.  dg: a cell paired with itself; gathered points before position skip do not count for this
    // lane.
    __device__ __forceinline__ void bin4(const CfItem &it, const IPoint &I, const float *bs, uint32_t j4, bool dg,
                                         uint32_t skip)
    {
        const float *b = bs + j4;
        const ulonglong2 xj = *reinterpret_cast<const ulonglong2 *>(b);
        const ulonglong2 yj = *reinterpret_cast<const ulonglong2 *>(b + GBUF);
        const ulonglong2 zj = *reinterpret_cast<const ulonglong2 *>(b + 2 * GBUF);
        u64 q[2], z[2] = {0ull, 0ull};
#pragma unroll
        for (int h = 0; h < 2; h++) {
            u64 dx = f2_add(I.s[0], h ? xj.y : xj.x), dy = f2_add(I.s[1], h ? yj.y : yj.x),
                dz = f2_add(I.s[2], h ? zj.y : zj.x);
            if (R) {
                u64 ex = I.e[0], ey = I.e[1], ez = I.e[2];
                if (LO) {
                    ex = f2_add(ex, *reinterpret_cast<const u64 *>(b + 4 * GBUF + 2 * h));
                    ey = f2_add(ey, *reinterpret_cast<const u64 *>(b + 5 * GBUF + 2 * h));
                    ez = f2_add(ez, *reinterpret_cast<const u64 *>(b + 6 * GBUF + 2 * h));
                }
                dx = f2_add(dx, ex);
                dy = f2_add(dy, ey);
                dz = f2_add(dz, ez);
            }
            if (WRAP) {
                if (Lx > 0.f) dx = wrap2(dx, Lx, iLx);
                if (Ly > 0.f) dy = wrap2(dy, Ly, iLy);
                if (Lz > 0.f) dz = wrap2(dz, Lz, iLz);
            }
            if (KIND == KIND_MOCKS) {
                // DD(rp, pi) of observed positions (Appendix A.2.1): pi^2 = (s.l)^2 / l.l and rp^2 =
                // |s x A_i|^2 / l.l (s x A_i = s x l, because l = A_i - s / 2), whose error scales with
                // rp where s.s - pi^2 would lose everything below the rounding of s.s when rp << pi
                const u64 ax = I.a[0], ay = I.a[1], az = I.a[2];
                const u64 NH = f2_pack(-0.5f, -0.5f);
                const u64 lx = f2_fma(dx, NH, ax), ly = f2_fma(dy, NH, ay), lz = f2_fma(dz, NH, az);
                const u64 sl = f2_fma(dz, lz, f2_fma(dy, ly, f2_mul(dx, lx)));
                const u64 ll = f2_fma(lz, lz, f2_fma(ly, ly, f2_mul(lx, lx)));
                const u64 cx = f2_sub(f2_mul(dy, az), f2_mul(dz, ay));
                const u64 cy = f2_sub(f2_mul(dz, ax), f2_mul(dx, az));
                const u64 cz = f2_sub(f2_mul(dx, ay), f2_mul(dy, ax));
                const u64 c2 = f2_fma(cz, cz, f2_fma(cy, cy, f2_mul(cx, cx)));
                const u64 r = f2_pack(f_rcp_approx(f2_lo(ll)), f_rcp_approx(f2_hi(ll)));
                q[h] = f2_mul(c2, r);
                z[h] = f2_mul(f2_mul(sl, sl), r);
                if (a.near2 > 0.f) {
                    // a midpoint near the observer, where the error bounds do not hold: FP64 when its
                    // s.s may count
                    const u64 ss = f2_fma(dz, dz, f2_fma(dy, dy, f2_mul(dx, dx)));
                    const bool n0 = f2_lo(ll) < a.near2, n1 = f2_hi(ll) < a.near2;
                    if (n0 && f2_lo(ss) < a.near_ss && (!dg || j4 + 2 * h >= skip)) push(it, I.p, gidx(it, bs, j4 + 2 * h));
                    if (n1 && f2_hi(ss) < a.near_ss && (!dg || j4 + 2 * h + 1 >= skip)) push(it, I.p, gidx(it, bs, j4 + 2 * h + 1));
                    const float nan = CUDART_NAN_F;
                    q[h] = f2_pack(n0 ? nan : f2_lo(q[h]), n1 ? nan : f2_hi(q[h]));
                }
            } else {
                q[h] = f2_fma(dy, dy, f2_mul(dx, dx));
                if (!has_pi(KIND)) q[h] = f2_fma(dz, dz, q[h]);
                else z[h] = dz & 0x7FFFFFFF7FFFFFFFull;
            }
        }
        float v2[4] = {f2_lo(q[0]), f2_hi(q[0]), f2_lo(q[1]), f2_hi(q[1])};
        if (dg) {
#pragma unroll
            for (int h = 0; h < 4; h++) v2[h] = j4 + h < skip ? CUDART_NAN_F : v2[h];
        }
        uint32_t c[4], cz[4] = {0u, 0u, 0u, 0u};
        float r4[4];
#pragma unroll
        for (int h = 0; h < 4; h++) r4[h] = f_sqrt_ftz(v2[h]);
        lut2(r4[0], r4[1], c[0], c[1]);
        lut2(r4[2], r4[3], c[2], c[3]);
        float F[4] = {0.f, 0.f, 0.f, 0.f};
        if (has_pi(KIND)) {
            // the pi bins are equally wide: with t = pi / width, t + 2^23 rounded down holds the bin in its
            // low bits, and the fraction's distance from 1/2 says whether a pi edge is near
            const u64 MAGIC = f2_pack(8388608.0f, 8388608.0f), HALF = f2_pack(-0.5f, -0.5f);
#pragma unroll
            for (int h = 0; h < 2; h++) {
                u64 p = z[h];
                if (KIND == KIND_MOCKS) p = f2_pack(f_sqrt_ftz(f2_lo(p)), f_sqrt_ftz(f2_hi(p)));
                const u64 t = f2_mul(p, a.pi_inv2);
                const u64 n = f2_add_rm(t, MAGIC);
                const u64 f = f2_add(f2_sub(t, f2_sub(n, MAGIC)), HALF);
                F[2 * h] = f2_lo(f);
                F[2 * h + 1] = f2_hi(f);
                cz[2 * h] = f2_lo_bits(n);
                cz[2 * h + 1] = f2_hi_bits(n);
            }
        }
        bool odd = max(max(c[0], c[1]), max(c[2], c[3])) > (uint32_t)a.nb;
        if (has_pi(KIND)) odd = odd || fmaxf(fmaxf(fabsf(F[0]), fabsf(F[1])), fmaxf(fabsf(F[2]), fabsf(F[3]))) > a.pi_half;
        if (odd) {
            // a table cell with an edge in it or a value near a pi edge (one pair in a thousand): the full
            // tables decide, and what they call ambiguous goes to the FP64 recheck
            uint32_t todo = 0;
#pragma unroll
            for (int h = 0; h < 4; h++) {
                const bool d = c[h] > (uint32_t)a.nb || (has_pi(KIND) && c[h] < (uint32_t)a.nb && fabsf(F[h]) > a.pi_half);
                todo |= (d ? 1u : 0u) << h;
                c[h] = d ? (uint32_t)a.nb : c[h];
            }
            const float z4[4] = {f2_lo(z[0]), f2_hi(z[0]), f2_lo(z[1]), f2_hi(z[1])};
            for (; todo; todo &= todo - 1u) {
                const int h = __ffs(todo) - 1;
                const uint32_t kr = lut_class(a.lut, a.fine, a.lr, __float_as_uint(pick4(v2, h)));
                const uint32_t kz = has_pi(KIND) ? lut_class(a.lut, a.fine, a.lp, __float_as_uint(pick4(z4, h))) : 0u;
                if (kr == CFI_CLS_OUT || kz == CFI_CLS_OUT) continue;
                if (max(kr, kz) == CFI_CLS_AMB) push(it, I.p, gidx(it, bs, j4 + h));
                else add_pair(it, I, kr, kz, R ? f_sqrt_approx(pick4(v2, h)) : 0.f, W ? b[3 * GBUF + h] : 0.f, b + h);
            }
        }
        float wj[4] = {0.f, 0.f, 0.f, 0.f};
        if (W) {
            const float4 t = *reinterpret_cast<const float4 *>(b + 3 * GBUF);
            wj[0] = t.x; wj[1] = t.y; wj[2] = t.z; wj[3] = t.w;
        }
#pragma unroll
        for (int h = 0; h < 4; h++) {
            bool in = c[h] < (uint32_t)a.nb;
            if (has_pi(KIND)) in = in && cz[h] < a.pi_top;
            const uint32_t kz = cz[h] - MAGIC_BITS;
            if ((W || R) && !warp_hist(KIND)) {
                add_lane(in, c[h], r4[h], W ? __fmul_rn(I.w, wj[h]) : 0.f);
            } else if (W || R || GH) {
                if (in) add_pair(it, I, c[h], kz, r4[h], wj[h], b + h);
            } else if (KIND == KIND_RPPI || KIND == KIND_MOCKS) {
                atomicAdd(h_cnt + (in ? c[h] * (uint32_t)a.npi + kz : (uint32_t)(a.nslot + lane)), 1u);
            } else if (KIND == KIND_WP) {
                atomicAdd(h_cnt + (in ? c[h] : (uint32_t)a.nb) * 32u, 1u);
            } else {
                atomicAdd(h_cnt + c[h] * 32u, 1u);
            }
        }
    }

    // The least separation on one axis between the box (lo, hi) of the group and a point, whose negated coordinate is
    // nx.  With an explicit minimum image (L > 0) the box comes as its centre and half width, the latter
    // widened by L * WRAP_MARGIN: the centre, the wrapped difference and the half width are each off by a few
    // 2^-24 L (|centre - x| stays below 2 L), and so is the kernel's own minimum image of a pair.  Gathering
    // every point there instead formed all pairs of neighbouring cells (pair kernel, without / with this test): DD(r) of
    // 100k points to 0.4 of the side 5.10 / 2.98 ms, with both sums 9.98 / 5.64; DD(rp, pi) of 1M with the line of sight
    // explicit 56.1 / 29.9, with both sums 174 / 108; wp 47.7 / 24.0.
    __device__ __forceinline__ static float gap(float lo, float hi, float nx, float L, float invL)
    {
        if (WRAP && L > 0.f) return fabsf(wrap1(lo + nx, L, invL)) - hi;
        return fmaxf(lo + nx, -hi - nx);
    }

    // Whether a separation of at least (gx, gy, gz) per axis (negative: 0) may count.  Every operation from
    // the boxes on rounds monotonically, so what fails here holds no pair below the limit.
    __device__ __forceinline__ bool within(float gx, float gy, float gz) const
    {
        gx = fmaxf(gx, 0.f);
        gy = fmaxf(gy, 0.f);
        gz = fmaxf(gz, 0.f);
        float t = fmaf(gy, gy, fmaf(gx, gx, -a.reach_r));
        if (has_z(KIND)) return t < 0.f && fmaf(gz, gz, -a.reach_p) < 0.f;
        t = fmaf(gz, gz, t);
        return t < 0.f;
    }

    // One work item: its i tile in groups of 32 points; for each the j points within reach of the
    // group's bounding box are gathered in shared memory and counted 32 at a time.
    __device__ __forceinline__ void run(const CfItem &it)
    {
        const uint32_t icnt = it.cnt & 0xFFFFu, jcnt = it.cnt >> 16, jbeg = it.jbeg;
        const bool diag = (it.meta & CFI_ITEM_DIAG) != 0;
        // Counts over (rp, pi) keep the group's box in shared memory: two loads per 32 points tested take
        // less than the spills that six more registers cost (64 B of spills without, 20 B with).
        constexpr bool BOXS = !W && !R && has_pi(KIND);
        // Groups of few points share the warp (below).  Counts by separation or angle alone do not: the
        // bookkeeping costs their shorter loop 2 to 6 %, more than it saves.
        constexpr bool SPLIT = W || R || has_pi(KIND);
        const uint32_t box = (uint32_t)__cvta_generic_to_shared(gj + GBUF);
        const uint32_t upto = 0xFFFFFFFFu >> (31 - lane);       // the lanes up to this one
#pragma unroll 1
        for (uint32_t i0 = 0; i0 < icnt; i0 += 32u) {
            // a cell paired with itself: only j > i counts, so the points from this group on
            uint32_t j0 = diag ? i0 : 0u;
            const float4 *pj = a.pt + (jbeg + j0 + lane), *lj = LO ? a.plo + (jbeg + j0 + lane) : nullptr;
            float4 P = make_float4(0.f, 0.f, 0.f, 0.f), Q = P;
            if (j0 + lane < jcnt) {
                P = *pj;
                if (LO) Q = *lj;
            }
            IPoint I;
            // A group of at most 16, 8 or 4 points has 2, 4 or 8 lanes per point: lane l has point l % 2^sh and
            // counts every 2^(5 - sh)-th four of the gathered points.  Of a cell's points (50 on average in a
            // sparse catalogue) the last group leaves half of the lanes idle otherwise.  Measured with this and
            // the box above: (rp, pi) counts, 2M points 928 -> 883 us, 2M x 4M 2892 -> 2706 us; mocks 200k x 2M
            // 2287 -> 2140 us; 1M points with separations and weights 1024 -> 985 us.
            const uint32_t left = icnt - i0;
            uint32_t sh = 5u, li = lane, off = 0u, step = 4u;
            if (SPLIT) {
                // (by a vote, so that the compiler sees a value that is the same in all lanes)
                const uint32_t m = __ballot_sync(CF_FULL, lane < left);
                sh = m >> 16 ? 5u : (m >> 8 ? 4u : (m >> 4 ? 3u : 2u));
                li = lane & ((1u << sh) - 1u);
                off = (uint32_t)lane >> sh << 2;
                step = 128u >> sh;
            }
            load_i(it, it.ibeg + i0 + li, li < left, I);
            float lo[3], hi[3];     // the group's box; the NaN of an empty lane drops out
#pragma unroll
            for (int d = 0; d < 3; d++) {
                lo[d] = cf_redux_min(f2_lo(I.s[d]));
                hi[d] = cf_redux_max(f2_lo(I.s[d]));
            }
            if (WRAP) {
                // on an axis of explicit minimum image the box is kept as centre and half width
#pragma unroll
                for (int d = 0; d < 3; d++) {
                    const float L = d == 0 ? Lx : (d == 1 ? Ly : Lz);
                    const float c = 0.5f * lo[d] + 0.5f * hi[d], h = 0.5f * hi[d] - 0.5f * lo[d];
                    lo[d] = L > 0.f ? c : lo[d];
                    hi[d] = L > 0.f ? fmaf(L, WRAP_MARGIN, h) : hi[d];
                }
            }
            if (BOXS && lane == 0) {
                asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(box), "f"(lo[0]), "f"(lo[1]), "f"(lo[2]),
                             "f"(hi[0]) : "memory");
                asm volatile("st.shared.v2.f32 [%0 + 16], {%1, %2};" ::"r"(box), "f"(hi[1]), "f"(hi[2]) : "memory");
            }
            if (BOXS) __syncwarp();
            // head: where the block to count next starts in the ring (0 or 32); fill: points gathered there
            uint32_t head = 0, fill = 0, skip = 0;
            bool dg = diag;
            for (;;) {
#pragma unroll 1
                while (fill < 32u && j0 < jcnt) {
                    const float4 C = P, E = Q;
                    const uint32_t j = j0 + lane;
                    j0 += 32u;
                    pj += 32;
                    if (LO) lj += 32;
                    if (j0 + lane < jcnt) {
                        P = *pj;
                        if (LO) Q = *lj;
                    }
                    bool keep = j < jcnt;
                    {
                        float l0 = lo[0], l1 = lo[1], l2 = lo[2], h0 = hi[0], h1 = hi[1], h2 = hi[2];
                        if (BOXS) {
                            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                                         : "=f"(l0), "=f"(l1), "=f"(l2), "=f"(h0) : "r"(box));
                            asm volatile("ld.shared.v2.f32 {%0, %1}, [%2 + 16];" : "=f"(h1), "=f"(h2) : "r"(box));
                        }
                        keep = keep && within(gap(l0, h0, C.x, Lx, iLx), gap(l1, h1, C.y, Ly, iLy), gap(l2, h2, C.z, Lz, iLz));
                    }
                    const uint32_t m = __ballot_sync(CF_FULL, keep);
                    uint32_t le = upto;
                    if (BOXS) asm volatile("mov.u32 %0, %%lanemask_le;" : "=r"(le));
                    const uint32_t rank = __popc(m & le);
                    if (keep) {
                        const uint32_t k = (head + fill + rank - 1u) & (GBUF - 1u);
                        float *q = jst + k;
                        q[0] = C.x;
                        q[GBUF] = C.y;
                        q[2 * GBUF] = C.z;
                        if (W) q[3 * GBUF] = C.w;
                        if (LO) {
                            q[4 * GBUF] = E.x;
                            q[5 * GBUF] = E.y;
                            q[6 * GBUF] = E.z;
                        }
                        gj[k] = (uint16_t)j;
                    }
                    // in a cell paired with itself the group's own points come first: those up to lane i
                    // (i itself among them) do not count for it
                    if (dg && fill == 0u) skip = SPLIT ? __shfl_sync(CF_FULL, rank, li) : rank;
                    fill += __popc(m);
                }
                if (fill == 0u) break;
                // up to a multiple of step
                if (fill < 32u && lane < (int)step - 1) jst[(head + fill + lane) & (GBUF - 1u)] = CUDART_NAN_F;
                __syncwarp();
                const float *bs = jst + head + off;
                const uint32_t n = min(fill, 32u);
#pragma unroll 1
                for (uint32_t j4 = 0; j4 < n; j4 += step)
                    bin4(it, I, bs, j4, dg, SPLIT ? max(skip, off) - off : skip);
                __syncwarp();       // the block's place is filled again
                head ^= 32u;
                fill -= n;
                dg = false;
            }
        }
    }

    // one lane's sum s - c into a pair of words, or where those could overflow into d
    static __device__ __forceinline__ void add_words(float s, float c, float &h, float &l, double &d)
    {
        if (!(fabsf(s) < 1e36f)) {
            d += (double)s - (double)c;
            return;
        }
        float t, e;
        two_sum(h, s, t, e);
        h = t;
        l += e - c;
    }

    __device__ void flush(uint32_t jb)
    {
        if (GH) return;         // nothing held per warp
        __syncwarp();
        const size_t g0 = (size_t)jb * a.nslot;
        for (int sl = lane; sl < a.nslot; sl += 32) {
            unsigned long long c = 0;
            double ws = 0.0, rs = 0.0;
            if (warp_hist(KIND)) {
                c = h_cnt[sl];
                h_cnt[sl] = 0;
                if (W) {
                    if (FX) {
                        uint32_t *w = reinterpret_cast<uint32_t *>(h_wd);
                        ws = fx_value(fx_sum(w[sl], w[a.nslot + sl]), a.fxw);
                        w[sl] = w[a.nslot + sl] = 0u;
                    } else {
                        ws = h_wd[sl];
                        h_wd[sl] = 0.0;
                    }
                }
                if (R) {
                    if (FX) {
                        uint32_t *w = reinterpret_cast<uint32_t *>(h_rd);
                        rs = fx_value(fx_sum(w[sl], w[a.nslot + sl]), fxr_bin[sl / a.npi]);
                        w[sl] = w[a.nslot + sl] = 0u;
                    } else {
                        rs = h_rd[sl];
                        h_rd[sl] = 0.0;
                    }
                }
            } else {
                // the lanes' sums are added in pairs of float32 words (error-free sums of the high words, the low
                // words with the errors): 32 x 8 FP64 operations per bin would hold each SM's FP64 pipe, 1/64 as
                // fast, at the end of the call (200k points with both sums 330 -> 322 us)
                float wh = 0.f, wl = 0.f, rh = 0.f, rl = 0.f;
                for (int l = 0; l < 32; l++) {
                    const int idx = sl * 32 + ((l + lane) & 31) - lane;
                    c += h_cnt[idx];
                    h_cnt[idx] = 0;
                    if (W && R) {
                        float4 *q = reinterpret_cast<float4 *>(h_w) + idx;
                        const float4 v = *q;
                        add_words(v.x, v.z, wh, wl, ws);
                        add_words(v.y, v.w, rh, rl, rs);
                        *q = make_float4(0.f, 0.f, 0.f, 0.f);
                    } else if (W || R) {
                        float2 *q = h_w + idx;
                        const float2 v = *q;
                        add_words(v.x, v.y, wh, wl, W ? ws : rs);
                        *q = make_float2(0.f, 0.f);
                    }
                }
                if (W || R) (W ? ws : rs) += (double)wh + (double)wl;
                if (W && R) rs += (double)rh + (double)rl;
            }
            if (c) atomicAdd(a.hcnt + g0 + sl, c);
            if (W && ws != 0.0) atomicAdd(a.hw + g0 + sl, ws);
            if (R && rs != 0.0) atomicAdd(a.hr + g0 + sl, rs);
        }
        __syncwarp();
    }
};

// CTA shape the register budget is sized for.  With weights or ravg the lane-private histograms
// (about 13 KB per warp for 20 bins) hold an SM to one CTA, so it may take up to 16 warps (the
// launcher takes as many as fit); count-only CTAs are small, and a budget for 4 of 256 threads per
// SM (64 registers, no spills in the rp-pi instances) keeps more of them resident than one for 3.
__host__ __device__ constexpr int pair_max_threads(bool W, bool R) { return (W || R) ? 512 : 256; }
__host__ __device__ constexpr int pair_min_blocks(bool W, bool R) { return (!W && !R) ? 4 : 1; }

template <int KIND, bool W, bool R, bool WRAP, bool LO, bool GH, bool FX, bool FIRST>
__global__ void __launch_bounds__(pair_max_threads(W, R), pair_min_blocks(W, R))
    pair_kernel(const CfPairArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const CfDevPlan *__restrict__ P = a.plan;
    const uint32_t nl4 = align16(a.nlut8) / 4u;
    // rp-pi / mocks: per rp bin scale of the ravg terms; else with sums the spare row
    float *s_fxr = (float *)(smem + 4u * nl4);
    unsigned char *wbase = (unsigned char *)s_fxr + cta_extra_bytes(KIND, W, R, a.nb);
    for (uint32_t i = threadIdx.x; i < nl4; i += blockDim.x) ((uint32_t *)smem)[i] = ((const uint32_t *)a.lut8)[i];
    if (FX && R)
        for (int i = threadIdx.x; i < a.nb; i += blockDim.x) s_fxr[i] = a.fxr_bin[i];
    const int hslots = GH ? 0 : a.nslot;        // slots of the per-warp histogram
    const uint32_t wb = warp_bytes(KIND, W, R, LO, hslots);
    const uint32_t hoff = warp_jbuf_bytes(W, R, LO);
    unsigned char *my = wbase + (size_t)(threadIdx.x >> 5) * wb;
    {
        // zero this warp's histogram (the buffers need no initial value)
        uint32_t *h = (uint32_t *)(my + hoff);
        const uint32_t words = warp_hist_bytes(KIND, W, R, hslots) / 4u;
        for (uint32_t i = threadIdx.x & 31; i < words; i += 32) h[i] = 0u;
    }
    __syncthreads();

    Warp<KIND, W, R, WRAP, LO, GH, FX> w(a);
    w.lane = threadIdx.x & 31;
    w.fxr_bin = s_fxr;
    w.lut = (uint32_t)__cvta_generic_to_shared(smem) - MAGIC_BITS;
    w.Lx = a.L[0]; w.Ly = a.L[1]; w.Lz = a.L[2];
    w.iLx = a.L[0] > 0.f ? 1.0f / a.L[0] : 0.f;
    w.iLy = a.L[1] > 0.f ? 1.0f / a.L[1] : 0.f;
    w.iLz = a.L[2] > 0.f ? 1.0f / a.L[2] : 0.f;
    w.jst = (float *)(my + item_bytes(W, R));
    w.gj = (uint16_t *)(my + item_bytes(W, R) + stage_arrays(W, LO) * GBUF * 4u);
    w.h_cnt = (uint32_t *)(my + hoff);
    if (warp_hist(KIND)) {
        uint32_t o = (((uint32_t)hslots + (W || R ? 0u : 32u)) * 4u + 7u) & ~7u;
        w.h_wd = (double *)(my + hoff + o);
        w.h_rd = (double *)(my + hoff + o + (W ? hslots * 8u : 0u));
        w.h_w = nullptr;
    } else {
        uint32_t o = a.nslot * 32u * 4u;
        // with both sums they interleave (float4 per lane and bin: w, r, their compensations)
        w.h_w = (float2 *)(my + hoff + o) + (W && R ? 2 : 1) * w.lane;
        // (counts only: there is neither a sum nor a spare row)
        w.d_cnt = W || R ? (uint32_t *)s_fxr + w.lane : nullptr;
        w.d_w = W || R ? (float2 *)(s_fxr + 32) + (W && R ? 2 : 1) * w.lane : nullptr;
        w.h_cnt += w.lane;
        w.h_wd = w.h_rd = nullptr;
    }

    // a list that was cut off is made again: nothing to count then
    const uint32_t nitems = *a.nitems_dev <= a.items_cap ? *a.nitems_dev : 0u;
    int cur = -1;
    // pairs evaluated since the last flush: a warp flushes at the latest every 2^28 (an item holds
    // at most 128 x 512 = 2^16), so no 32-bit count and no fixed-point sum it holds can overflow
    uint32_t pend = 0;
    // the next item is fetched while the current one is processed
    uint32_t t = 0, at = 0;
    // FIRST: a warp's first item is its own number and the cursor hands out those after, so that the warps do
    // not all wait for one word at the start
    if (w.lane == 0) t = FIRST ? blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5) : atomicAdd(a.cursor, 1u);
    t = __shfl_sync(CF_FULL, t, 0);
    CfItem *ring = (CfItem *)my;
    CfItem nx;
    auto fetch = [&](uint32_t k) {
        if (smem_items(W, R)) {
            if (k < nitems && w.lane < (int)(sizeof(CfItem) / 16))
                cp_async16((uint4 *)(ring + at) + w.lane, (const uint4 *)(a.items + k) + w.lane);
            cp_async_commit();
        } else if (k < nitems) {
            nx = a.items[k];
        }
    };
    fetch(t);
    while (t < nitems) {
        uint32_t tn = 0;
        if (w.lane == 0) tn = atomicAdd(a.cursor, 1u) + (FIRST ? a.nwarps : 0u);
        tn = __shfl_sync(CF_FULL, tn, 0);
        auto count = [&](const CfItem &it) {
            const int job = (int)w.job(it);
            if (job != cur || pend > (FX ? FX_FLUSH_PAIRS : CF_FLUSH_PAIRS)) {
                if (cur >= 0) w.flush((uint32_t)cur);
                cur = job;
                pend = 0;
            }
            pend += (it.cnt & 0xFFFFu) * (it.cnt >> 16);
            w.run(it);
        };
        if (smem_items(W, R)) {
            cp_async_wait_all();
            __syncwarp();           // the current item is there, and nobody reads the other place any more
            const CfItem *it = ring + at;
            at ^= 1u;
            fetch(tn);
            count(*it);
        } else {
            const CfItem it = nx;
            fetch(tn);
            count(it);
        }
        t = tn;
    }
    if (smem_items(W, R)) cp_async_wait_all();
    if (cur >= 0) w.flush((uint32_t)cur);
}

template <int KIND, bool W, bool R, bool WRAP, bool LO, bool GH = false, bool FX = false,
          bool FIRST = (W || R || has_pi(KIND))>
cudaError_t launch_variant(const CfPairCfg &c, const CfPairArgs &a, int num_sms, cudaStream_t st, int *grid_out,
                           int *warps_out)
{
    auto k = pair_kernel<KIND, W, R, WRAP, LO, GH, FX, FIRST>;
    int dev;
    cudaGetDevice(&dev);
    int maxsm = 0;
    cudaDeviceGetAttribute(&maxsm, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    const int maxw = pair_max_threads(W, R) / 32;
    int warps = c.warps > 0 ? (c.warps > maxw ? maxw : c.warps) : maxw;
    size_t smem = 0;
    for (; warps >= 1; warps--) {
        smem = cfp_pair_smem(c, warps);
        if (smem <= (size_t)maxsm) break;
    }
    if (warps < 1) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int per_sm = c.ctas_per_sm;
    if (per_sm <= 0) {
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, warps * 32, smem);
        if (e != cudaSuccess) return e;
        if (per_sm < 1) per_sm = 1;
    }
    int grid = per_sm * num_sms;
    CfPairArgs b = a;
    b.nwarps = (uint32_t)(grid * warps);
    k<<<grid, warps * 32, smem, st>>>(b);
    if (grid_out) *grid_out = grid;
    if (warps_out) *warps_out = warps;
    return cudaGetLastError();
}

constexpr uint32_t SHORT_LIST = 40000;       // work items

// global histograms (rp-pi and mocks tables too large for shared memory), fixed-point per-warp sums, or
// the plain form
template <int KIND, bool W, bool R, bool WRAP, bool LO>
cudaError_t launch_one(const CfPairCfg &c, const CfPairArgs &a, int num_sms, cudaStream_t st, int *grid_out,
                       int *warps_out)
{
    if constexpr (warp_hist(KIND))
        if (c.ghist) return launch_variant<KIND, W, R, WRAP, LO, true>(c, a, num_sms, st, grid_out, warps_out);
    if constexpr (warp_hist(KIND) && (W || R))
        if (a.fxw != 0.f || a.fxr != 0.f)
            return launch_variant<KIND, W, R, WRAP, LO, false, true>(c, a, num_sms, st, grid_out, warps_out);
    // Counts by separation or angle: the registers of FIRST slow their loop down by 4.5 % (1M points to a separation
    // of 40: 2347 -> 2452 us), which short lists do not notice (20k points 27 -> 23 us, 6,800 cells by angle
    // 31 -> 29 us, equal at 30,000 items).  The other kinds' loops do not change.
    if constexpr (!W && !R && !has_pi(KIND))
        if (a.items_cap <= SHORT_LIST)
            return launch_variant<KIND, W, R, WRAP, LO, false, false, true>(c, a, num_sms, st, grid_out, warps_out);
    return launch_variant<KIND, W, R, WRAP, LO>(c, a, num_sms, st, grid_out, warps_out);
}

}  // namespace cfpair

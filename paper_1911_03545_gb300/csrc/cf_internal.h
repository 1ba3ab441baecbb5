// cf_internal.h -- descriptors shared by the host planner and the CUDA kernels.
//
// Data layout in device memory (one call = a set of point sets and a set of jobs):
//   point set s (a catalogue, or one side of a cross count) is scattered into cell order by a
//   counting sort (Sec. 4.3: particles of a cell are stored contiguously).  For every point p
//   (global index over all sets) we keep
//     pt[p] = float4(-X, -Y, -Z, w)
//   where X = x - o(cell) is the cell-relative coordinate (Sec. 4.4's shift trick applied per
//   cell), stored negated so that an addition forms a separation; for mocks also
//     pabs[p] = float4(x, y, z, 0), the absolute position rounded to float32
//   and for float64 inputs with ravg the low parts: x - o = X + Xlo, x = float(x) + xlo
//     plo[p] = float4(-Xlo, -Ylo, -Zlo, 0), pabslo[p] = float4(xlo, ylo, zlo, 0) (mocks)
//     orig[p] = index of the point in its input arrays (without weights kept in pt[p].w)
//   cell_start[set cell offset + c] .. [c+1] delimit a cell's points.
//   A work item is one (i tile, j range, shift) triple of a cell pair (Sec. 4.3).
#pragma once
#include <math.h>
#include <stdint.h>

#include "cf.h"

#define CFI_MAX_SETS 4096
#define CFI_MAX_STENCIL 4096
#define CFI_LUT_MAX 8192          // coarse LUT cells (2 B each)
#define CFI_LUT_TARGET 4096       // preferred coarse cells per table
#define CFI_LUT8_CELLS 16384      // cells of the pair kernel's separation table below the last edge
#define CFI_LUT8_CELLS_SUMS 8192  // the same with weights or ravg, whose histograms fill shared memory
#define CFI_FINE_MAX 1024         // fine LUT entries (16 B each)
#define CFI_CLS_OUT 0xFEu         // class: outside every bin
#define CFI_CLS_AMB 0xFFu         // class: within the FP32 error band of an edge
#define CFI_FINE_FLAG 0x100u      // coarse entry >= this: index of a fine entry + flag
#define CFI_MIN_FILL 40.0         // points per cell and set below which the cells are widened (widen_cells)
#define CFI_BIG_FILL 2.0          // times that: points per cell of the typical point's own set that stop the widening
#define CFI_WIDEN_MIN 32768       // points of a call below which they are not
#define CFI_DENSE 800.0           // points per cell of a pair's larger set from which cells are halved (dense_cells)
#define CFI_DENSE_MOCKS 500.0     // the same for mocks,
#define CFI_DENSE_FEW 500.0       // and for r where that set has at most
#define CFI_DENSE_FEW_N (1 << 17) // so many points
#define CFI_DENSE_I_CYL 90.0      // points per cell of the smaller set below which they are not: rp-pi and wp,
#define CFI_DENSE_I_MOCKS 16.0    // mocks (r: those of the larger set)
#define CFI_DENSE_MAX (1 << 24)   // points of a set above which they are not
#define CFI_JMAX 512              // longest j range of a work item

// Pair-kernel item (48 bytes, three 16-byte loads)
struct CfItem {
    uint32_t ibeg;     // first i point (global sorted index)
    uint32_t jbeg;     // first j point
    uint32_t cnt;      // icnt (low 16) | jcnt (high 16)
    uint32_t meta;     // job (low 20 bits) | diag (bit 30)
    float s[3];        // shift hi:  x_i - x_j = (X_i + s + slo) - X_j
    float pad0;
    float slo[3];      // shift lo
    float pad1;
};
#define CFI_ITEM_DIAG (1u << 30)
#define CFI_ITEM_JOBMASK 0xFFFFFu
// most work items and recheck-queue entries of one call: both are indexed in 32 bits, and the
// grid-stride loops and the work cursor run a few thousand past the end
#define CFI_MAX_ENTRIES 0xFFF00000ull   // 2^32 - 2^20

#ifdef __CUDACC__
#define CFI_HD __host__ __device__ __forceinline__
#else
#define CFI_HD inline
#endif

// Work items of a cell pair: every tile of the i cell with every range of the j cell, or of a cell with itself the
// tile pairs a <= b.  64 bits: a cell of 4.2 million points has 65,625 tiles of 64, whose square does not fit 32.
CFI_HD uint64_t cfi_item_count(uint32_t nti, uint32_t ntj, bool diag)
{
    return diag ? (uint64_t)nti * (nti + 1ull) / 2u : (uint64_t)nti * ntj;
}
// below this many tiles and ranges a count stays below CFI_MANY_ITEMS, and 32 of those fit 32 bits
#define CFI_FEW_TILES 8192u
#define CFI_MANY_ITEMS (1u << 26)

// q (q + 1) / 2 without a product larger than it
CFI_HD uint32_t cfi_triangle(uint32_t q) { return ((q + 1u) >> 1) * (q | 1u); }

// The k-th tile pair of a cell with itself, row by row (a = 0: b = 0, 1, ..; then a = 1: b = 1, ..).  Counted from
// the end the rows are a triangle.  k < cfi_item_count(nti, nti, true), which must fit 32 bits.
CFI_HD void cfi_tile_pair(uint32_t nti, uint32_t k, uint32_t &a, uint32_t &b)
{
    const uint32_t t = cfi_triangle(nti) - 1u - k;
    uint32_t q = (uint32_t)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
    while (cfi_triangle(q) > t) q--;
    while (cfi_triangle(q + 1u) <= t) q++;
    a = nti - 1u - q;
    b = nti - 1u - (t - cfi_triangle(q));
}

// A point set (input view + where its sorted points and cells live)
struct CfSetDesc {
    const void *x, *y, *z, *w;   // device pointers of the input arrays
    int64_t n;
    int dtype;                   // 0 f32, 1 f64
    int pad;
    int64_t pbeg;                // first sorted point of this set
    int64_t cbeg;                // first cell of this set in cell_start
};

// A job: count set a (i side) against set b (j side) into histogram slot block `job`
struct CfJobDesc {
    int a, b;
    int autoc;
    int pad;
};

// Coarse/fine bin lookup on the bit pattern of a non-negative float (Sec. 4.7: bins are found
// on squared separations; the bit pattern of a positive float is monotone in its value).
struct CfLut {
    uint32_t base;     // bits of the start of coarse cell 0
    uint32_t shift;    // log2 of a coarse cell width in bit space
    uint32_t last;     // index of the last coarse cell (values above clamp here)
    uint32_t coff;     // offset of the coarse entries in the shared LUT array (in words)
    uint32_t foff;     // offset of the fine entries (in 16-byte units from the fine base)
    uint32_t tail;     // bits from which every value is outside all bins
    uint32_t pad[2];
};

struct CfFine {        // class of v: byte seg of `code`, seg = (v >= t1) + (v >= t2)
    uint32_t t1, t2, code, pad;
};

// Grid parameters (Sec. 4.1 Eq. 3 cell index; Sec. 4.2 refinement)
struct CfGrid {
    int n[3];
    int ncell;
    double lo[3];
    double width[3];
    double inv[3];         // n / extent
    double L[3];           // periodic side (0 when not periodic)
    int periodic;
    int wrap[3];           // explicit minimum image on this axis
    int k[3];
    int nstencil;
};

struct CfStencil {         // neighbour offset per axis; wrap axes enumerate targets (i+d) mod n
    int d[3];
    int pad;
};

#define CFI_MAX_ANG_K 4           // refinement of the angular grid (bands searched: 2k + 1)

// One DEC band of the angular grid (DD(theta) alternative cell list): DEC in [dlo, dhi),
// nra RA cells of width w (radians) over [0, 2 pi), cells base .. base + nra - 1.  da[d] is the RA
// half-width to search in band b + d - k: 2 asin(sin(t / 2) / cos dm) with dm the largest |DEC| of
// both bands (haversine bound), or -1 when every RA cell is searched
struct CfBand {
    double dlo, dhi, w;
    double inv_w;                      // 1 / w
    double da[2 * CFI_MAX_ANG_K + 1];  // RA half-width searched in band b + d - k (negative: every cell)
    int nra, base;
};

// Everything the kernels need for one call
struct CfDevPlan {
    CfGrid g;
    int kind;              // 0 r, 1 rppi, 2 wp, 3 theta, 4 mocks (rp-pi of observed positions)
    int nb;                // r / rp / theta bins
    int npi;               // pi bins (1 for r, theta, wp)
    int nslot;             // nb * npi for rppi and mocks, nb otherwise
    int weighted, ravg, f64lo;
    int nsets, njobs;
    int tile;              // max i tile (64 or 128)
    int jchunk;            // max j range per item
    CfLut lr, lp;          // r/rp/chord LUT, and pi LUT (rppi/wp)
    int nlut8;             // cells of the pair kernel's separation table (one byte each)
    float lut8_scale;      // its cells per unit of separation
    int nlut_words;        // coarse words (both LUTs)
    int nfine;             // fine entries (both LUTs)
    double pimax;
    const double *origin;  // device table of cell origins: axis a, index i at origin[ooff[a] + i]
                           // (angular grid: cell c at origin[3 c + a])
    int ooff[3];
    int ang;               // 1: angular grid (theta): DEC bands x RA cells instead of the 3-D grid
    int nband;
    const CfBand *band;    // device table of the bands
    double adlo, ah;       // lowest band edge and band height (radians)
    double tsearch;        // neighbour-search angle (radians): the largest edge, widened
    float reach_r;         // gathering limit of the pair kernel on the squared separation (mocks: s.s;
                           // rp-pi / wp: rp^2) formed without the shift's low part: above the largest
                           // one that may count by that form's FP32 error
    float reach_p;         // the same on dz^2 (rp-pi / wp)
    int pi_n;              // rp-pi / wp / mocks: pi bins, all of one width (wp: one bin)
    float pi_inv;          // 1 / that width: bin floor(pi * pi_inv)
    float pi_tol;          // a pi * pi_inv within this of an integer may lie in the FP32 band of a pi edge
    float near2;           // mocks: a candidate whose FP32 l.l is below this goes to the FP64
                           // recheck when its s.s is below near_ss (0: no candidate can be)
    float near_ss;
    double smax2;          // mocks: largest |s|^2 of a counted pair (rmax^2 + pimax^2, widened)
    // float32 helpers of the cell build (the FP64 pipe runs at a small fraction of the FP32 rate):
    const float *origin32; // float32 copies of `origin` (exact: origins are multiples of the float32
                           // spacing at their cell's magnitude)
    float inv32[3], lo32[3];   // n / extent and the lower corner per axis, float32
    float cguard[3];       // a float32 cell coordinate within cguard of an integer is recomputed in FP64
    float pmargin[3];      // cell-pair pruning in float32: each gap is shrunk by this (its rounding)
    float e2max32, zmax32; // the largest squared separation / |dz| of a counted pair, rounded up
    double e2[CF_MAX_BINS + 1];     // squared edges (FP64, host-computed)
    double pe[CF_MAX_PIBINS + 1];   // pi edges (mocks: squared pi edges)
};

// cf_build.h -- launchers of the cell-build, work-list and pair-count kernels.
#pragma once
#include <cuda_runtime.h>

#include "cf_internal.h"

// per point set: 3 min keys, 3 max keys, bad, norm deviation, min |v|^2, smallest nonzero |w|,
// largest |w|, negative weights
#define CFB_BBOX_WORDS 12
cudaError_t cfb_bbox(const CfSetDesc *sets, int nsets, int64_t nmax, unsigned long long *out, cudaStream_t st);
// fills out[nsets * CFB_BBOX_WORDS] with the starting values cfb_bbox reduces into
cudaError_t cfb_bbox_init(unsigned long long *out, int nsets, cudaStream_t st);
// key = cell * sub^3 + place of the sub-cell (sub = 1, 2, 4): the counting-sort key of every point
cudaError_t cfb_assign(const CfDevPlan *plan, const CfSetDesc *sets, int nsets, int64_t nmax, int sub,
                       uint32_t *count, uint32_t *key, uint32_t *slot, cudaStream_t st);
// origins of the angular grid's cells (3 per cell) from their (RA, DEC) boxes
cudaError_t cfb_ang_origins(const CfDevPlan *plan, int ncell, double *origin, float *origin32, cudaStream_t st);
int64_t cfb_scan_tmp_words(int64_t n);
// exclusive scan of n counts into out[0..n) and the total into out[n] (and *total_copy if given);
// tmp holds cfb_scan_tmp_words(n) words, *done must be 0 (a ticket counter).  every, if given,
// receives every[i >> every_shift] = out[i] for the multiples i of 2^every_shift up to n (the cell
// starts among the sub-cell starts: cell_start[c] = fstart[c * sub^3]).
cudaError_t cfb_scan(const uint32_t *in, uint32_t *out, int64_t n, uint32_t *tmp, uint32_t *done, cudaStream_t st,
                     uint32_t *total_copy = nullptr, uint32_t *every = nullptr, int every_shift = 0);
cudaError_t cfb_scatter(const CfDevPlan *plan, const CfSetDesc *sets, int nsets, int64_t nmax, int sub,
                        const uint32_t *fstart, const uint32_t *key, const uint32_t *slot, float4 *pt,
                        float4 *pabs, float4 *plo, float4 *pabslo, uint32_t *orig, cudaStream_t st);
// tight point bounding box per cell (6 floats: lo xyz, hi xyz, cell-relative), for cell-pair pruning;
// with gbox (6 floats per point) also the box of every 32-point group of a cell at its first point
cudaError_t cfb_cellbox(const uint32_t *cell_start, int64_t ncell_all, const float4 *pt, float *box, float *gbox,
                        cudaStream_t st);
// the units (job, i cell) whose i cell holds points, appended to live[] (nunits entries) at the
// zeroed counter *nlive
cudaError_t cfb_live_units(const CfDevPlan *plan, const CfSetDesc *sets, const CfJobDesc *jobs,
                           const uint32_t *cell_start, int64_t nunits, uint32_t *live, uint32_t *nlive,
                           cudaStream_t st);
// cbox: the boxes above, or nullptr to visit every stencil neighbour; gbox: the group boxes, or
// nullptr for j ranges over whole cells; live / nlive: the units to visit (cfb_live_units), or
// nullptr for all of them; nunits: units visited at most, for the size of the grid (with a list, mode 0 writes the counts of the listed units only: the
// caller zeroes the rest).  mode 0: per-unit item counts
// into counts[], their number in 64 bits added to *evaluated; mode 1: items at offsets[]; mode 2:
// count and emit in one pass, items reserved on the counter counts[0] (zeroed by the caller), their
// number added to *total64.  Modes 1 and 2 add the pairs the stored items hold to *evaluated.
cudaError_t cfb_items(const CfDevPlan *plan, const CfSetDesc *sets, const CfJobDesc *jobs, const CfStencil *stencil,
                      const uint32_t *cell_start, const float *cbox, const float *gbox, const uint32_t *live,
                      const uint32_t *nlive, int64_t nunits, int mode, uint32_t *counts, const uint32_t *offsets,
                      CfItem *items, uint32_t items_cap, unsigned long long *evaluated, unsigned long long *total64,
                      cudaStream_t st);
// The whole build, from zeroing the call's counters to the work list, in one cooperative launch of one block
// per SM: see cf_one_build_kernel.  3-D grids without group pruning only.
#define CFB_ITEM_BLOCKS 8192    // of the work-list kernel, at most; 8 units at a time each
#define CFB_ITEM_STAGE 256      // work items a block collects in shared memory (stencils of more than 32 entries)
#define CFB_ONE_THREADS 1024
#define CFB_POLLS (1u << 22)       // of a block at a barrier: two to three seconds
#define CFB_ONE_KEYS 49152         // sort keys at most (192 KB of shared memory, beside the 12 KB item stage)
struct CfOneBuild {
    const CfDevPlan *plan;
    const CfSetDesc *sets;
    const CfJobDesc *jobs;
    const CfStencil *stencil;
    int nsets, sub;
    uint32_t npts, nfine;
    uint32_t *zero;              // counters and histograms of the call
    uint32_t zero_words;
    uint32_t *bar;               // the grid barrier's words: arrivals, barriers, given up, poll limit
    uint32_t *count;             // nfine key counts (a multiple of four of them is read): 0 before the launch, and after it
    uint32_t *key, *slot, *cell_start, *orig;
    float4 *pt, *pabs, *plo, *pabslo;
    float *cbox;                 // NULL: no boxes, every stencil neighbour is visited
    CfItem *items;
    uint32_t items_cap;
    uint32_t *nitems;
    unsigned long long *evaluated, *total64;
};
// once per context, on its device: blocks of the launch (0: the device does not take it)
int cfb_one_init(int num_sms);
cudaError_t cfb_one_build(const CfOneBuild &A, int blocks, cudaStream_t st);
cudaError_t cfb_wsq(const CfSetDesc *sets, int nsets, int64_t nmax, double *out, cudaStream_t st);

// ---- pair counting ----
struct CfPairArgs {
    const CfDevPlan *plan;
    const uint8_t *lut8;         // separation table (staged into shared memory)
    const uint16_t *lut;         // coarse entries of the full tables
    const CfFine *fine;          // fine LUT entries
    const CfItem *items;
    const uint32_t *nitems_dev;  // item count written by the work-list scan
    uint32_t items_cap;          // items beyond this were not stored
    uint32_t qcap;
    uint32_t *cursor;
    const float4 *pt;            // (-X, -Y, -Z, w)
    const float4 *pabs;          // mocks: absolute positions
    const float4 *plo, *pabslo;  // low parts (float64 inputs with ravg)
    const uint32_t *orig;        // NULL without weights: the index is in pt's fourth word
    unsigned long long *hcnt;    // [njobs][nslot]
    double *hw;                  // [njobs][nslot]
    double *hr;                  // [njobs][nslot]
    uint4 *queue;                // (orig i, orig j, job, 0)
    unsigned long long *qcount;  // queued pairs, 64-bit so that it cannot wrap (entries >= qcap are dropped)
    float L[3];                  // periodic sides (wrap axes)
    int nb, npi, nslot;
    // the plan's constants (CfDevPlan) as kernel parameters: constant operands instead of registers
    uint64_t lut_scale2;         // lut8_scale, pi_inv in both halves of a packed pair
    uint64_t pi_inv2;
    uint32_t nlut8, lut_top;     // cells of lut8, and the bits of 2^23 + the last one's index
    float reach_r, reach_p, near2, near_ss;
    float pi_half;               // 1/2 - pi_tol: a fraction of pi / width farther from 1/2 may lie near a pi edge
    uint32_t pi_top;             // bits of 2^23 + the number of pi bins
    CfLut lr, lp;
    int ghist;                   // 1: rp-pi / mocks add straight into hcnt/hw/hr (global atomics):
                                 // their per-warp histogram does not fit in shared memory
    float fxw;                   // rp-pi / mocks per-warp weight sums in fixed point (two 32-bit words
                                 // per slot, see cf_pair.cuh) at this power-of-two scale (0: FP64)
    float fxr;                   // nonzero: the ravg sums too, those of rp bin k at scale fxr_bin[k]
    float fxr_bin[CF_MAX_BINS];
    uint32_t nwarps;             // warps of the launch (set by the launcher)
};

// Static configuration of a pair-kernel launch (selects the template instance and the shared
// memory layout).
struct CfPairCfg {
    int kind;          // 0 r, 1 rppi, 2 wp, 3 theta, 4 mocks
    int weighted, ravg, wrap, lo;
    int ghist;         // see CfPairArgs::ghist (no per-warp histogram in shared memory)
    int nlut;          // cells of the squared-separation table in shared memory
    int nslot;
    int nb;            // r / rp / theta bins
    int warps;         // warps per CTA (0: automatic)
    int ctas_per_sm;   // 0: occupancy-derived
};

// Shared-memory bytes of one CTA with `warps` warps.
size_t cfp_pair_smem(const CfPairCfg &c, int warps);

// Launch the persistent pair kernel.  Returns cudaErrorInvalidValue when no CTA shape fits in
// shared memory.  *grid_out receives the number of CTAs launched.
cudaError_t cfp_launch_pair(const CfPairCfg &c, const CfPairArgs &a, int num_sms, cudaStream_t st,
                            int *grid_out, int *warps_out);
// CF_OPT_AUDIT: queue every pair of every work item for the FP64 recheck (launched instead of the
// pair kernel).
cudaError_t cfp_launch_audit(const CfItem *items, const uint32_t *nitems_dev, uint32_t items_cap,
                             const uint32_t *orig, const float4 *pt, uint4 *queue, unsigned long long *qcount,
                             uint32_t qcap, int num_sms, cudaStream_t st);
cudaError_t cfp_launch_recheck(const CfDevPlan *plan, const CfSetDesc *sets, const CfJobDesc *jobs,
                               const uint4 *queue, const unsigned long long *qcount, uint32_t qcap,
                               unsigned long long *hcnt, double *hw, double *hr, size_t hsz, const uint32_t *late,
                               uint32_t *flag, int num_sms, cudaStream_t st);

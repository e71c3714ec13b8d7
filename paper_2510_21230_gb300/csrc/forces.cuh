// forces.cuh -- host side of one LJ + ATM force evaluation on built cells,
// and the replica descriptors; shared by the context API and the
// allocation-free entry point.
#pragma once
#include "atm3.h"
#include "atm3_internal.cuh"
#include "md_kernels.cuh"

namespace atm3 {

constexpr int ATM_MCAP_LIMIT = 2047;  // staged molecules per unit (queue entries pack 11-bit indices)

// Fill a replica descriptor from the public parameters: linked-cell grid
// (n_d = largest k with L_d / k >= r_c, at least 3), cutoffs in FP64 and
// FP32, LJ constants, FP32 prefilter bands of the FP64 decisions (derivation
// in atm_common.cuh).  Returns ATM_OK, ATM_E_INVALID or ATM_E_BOX_TOO_SMALL.
atm_status make_rep(const atm_params& p, long long n, long long mol0, long long cell0, Rep& r);

struct ForceJob {
    Batch b;                 // device replica table
    const Rep* rep_host;     // [R] host copy (plan sizing)
    const double* xl;        // sorted cell-local coordinates FP64, SoA [3n]
    const float* xl32;       // the same in FP32
    const int* start;        // cell_start [ncell + 1]
    const int* cell_sorted;  // [n]
    double* f_lj;            // [3n] sorted order, fully written
    double* f_atm;           // [3n] sorted order
    double* mol_ew;          // [2n]
    unsigned* mol_cnt;       // [2n]
    double* unit_ew;         // [2 ncell]
    unsigned long long* unit_cnt;
    int* status;
    int* work;               // unit counter of the persistent launch
    int trav, trunc, prec;
    int mcap;                // largest unit of the traversal (staged molecules)
    int optin;               // opt-in shared memory per block of the device
    int sms;                 // SMs of the device
    int persistent;          // 1: persistent grid over a unit counter
    int nwarps;              // 0: the plan's default, else 4 or 8
    cudaStream_t st;
    // 3c08 / corner-anchored 3c08 / 3c18, pair rule: LJ evaluated inside the
    // ATM units (f_atm receives LJ + ATM, f_lj is zeroed; E2, W2 and the pair
    // counts go to unit_ew2 / unit_cnt2 instead of mol_ew / mol_cnt)
    int lj = 0;
    double* unit_ew2 = nullptr;
    unsigned long long* unit_cnt2 = nullptr;
    // block traversals: unit size classes (ncls 2 or 3; 1 = none).  Units of
    // at most cuts[0] (then cuts[1]) staged molecules run in launches sized for
    // that bound (2 warps when it is at most 64), the rest in one sized for
    // mcap; ulist [ncls * ncell], ucount [ncls] and work [ncls] are scratch
    int ncls = 1;
    int cuts[2] = {0, 0};
    int* ulist = nullptr;
    int* ucount = nullptr;
    // with a side stream the first class runs on it, forked from st after the
    // class kernel and joined back before the evaluation ends
    cudaStream_t side_st = nullptr;
    cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
    // deterministic mode: fixed work order; the block traversals sum their
    // terms in 64-bit fixed point and f_atm is converted back after them
    int det = 0;
    // FP32 pair rule of the block traversals: [PM_WORDS n] words for the pair
    // bitmaps, computed by one kernel ahead of the units, which assemble
    // their adjacency from them (nullptr: the units decide their own pairs).
    // The caller passes it only when every cell holds at most PM_CELL_MAX
    // molecules (a fuller cell found on the device sets ST_CAPACITY)
    unsigned* pmask = nullptr;
    // pair rule of the block traversals: edge-table capacity in 1/16 edges per
    // staged molecule (256: 16), and where the units record their need
    // (nullptr: not recorded)
    int gpm16 = 256;
    int* emax = nullptr;
    // FP32C pair rule from forward lists (atm_fwd.cuh): largest 18-cell unit
    // (0: not known, the list path is not taken); the unit arrays hold
    // fwd_unit_slots(ncell) entries; whole: every layer owned; lj_apart: the
    // caller wants the LJ force on its own and may get it from the units
    // (unit_ew2 / unit_cnt2 then hold its sums)
    int mcap_fwd = 0;
    bool whole = false;
    bool lj_apart = false;
    // FP64 pair rule from forward lists (atm_list64.cu): the buffers and inputs
    // of List64Args (list nullptr: not taken), cells within PM_CELL_MAX
    const List64Args* l64 = nullptr;
    // wrapped positions, original order, and the sorted -> original index (FP64
    // product rule)
    const double* x = nullptr;
    const int* perm = nullptr;
    const int* runs = nullptr;  // FwdArgs.runs and nruns of FWD_RUN cells (device)
    long long nruns = 0;
    int rc_exp = 0;             // largest rc_exponent of the replicas
};

// distance of r_c from 1 in powers of two
int rc_exponent(const Rep& r);

// how an evaluation from forward lists is launched
struct FwdLaunch {
    bool use = false;  // the job takes the list path
    int lj = 0;        // 0 no LJ, 1 inside fs, 2 apart
    int nwarps = FWD_MAXW, run = FWD_RUN, split = 1;
};
FwdLaunch atm_fwd_plan(const ForceJob& j);
// the same for the FP64 lists (lj 1 or 2)
FwdLaunch atm_list64_plan(const ForceJob& j);
// The FP64 lists' buffers: a row of list64_stride(mcap) entries of 16 bytes for each
// of n molecules, any list of an 18-cell unit of mcap molecules with an eighth for
// units to grow (a liquid at density 0.8: 310 entries, 5 KB a molecule), up to 16 GiB.
constexpr unsigned long long LIST64_MAX_BYTES = 16ull << 30;
inline long long list64_stride(int mcap) { return ((long long)mcap + mcap / 8 + 15) / 8 * 8; }
// the entries a row to allocate now for units of mcap molecules; 0: rows of `have`
// hold them, or they are beyond the limit, or rows of `refused` or fewer entries
// could not be had before (neither is tried again at every evaluation, and rows
// that are there stay)
inline long long list64_rows_wanted(long long n, long long have, long long refused, int mcap)
{
    if (have >= mcap) return 0;
    const long long s = list64_stride(mcap);
    if ((unsigned long long)n * (unsigned long long)s * 16 > LIST64_MAX_BYTES) return 0;
    return refused > 0 && s >= refused ? 0 : s;
}
// the product-rule kernel's warps per CTA (0: the job does not take it) and bytes
// of shared memory
struct ProdLaunch {
    int warps = 0, smem = 0;
};
ProdLaunch atm_prod_plan(const ForceJob& j);
// either
inline bool atm_uses_lists(const ForceJob& j)
{
    return atm_fwd_plan(j).use || atm_list64_plan(j).use;
}
// runs of FWD_RUN cells of one replica's grid
inline long long fwd_runs_of(const Grid& g)
{
    return (long long)((g.nc[0] + FWD_RUN - 1) / FWD_RUN) * g.nc[1] * g.nc[2];
}

cudaError_t enqueue_lj(const ForceJob& j);
// *capacity is set when no kernel configuration fits the unit size
cudaError_t enqueue_atm(const ForceJob& j, size_t* smem_set, bool* capacity);
// the job runs its units in size classes (one more kernel, ncls ATM launches)
bool atm_split_active(const ForceJob& j);
// the job's units take their pairs from bitmaps (one more kernel ahead of them)
bool atm_uses_pair_masks(const ForceJob& j);

}  // namespace atm3

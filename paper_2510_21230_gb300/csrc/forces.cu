// forces.cu -- replica descriptors, argument set-up and launch of the LJ and
// ATM force kernels, shared by the context API (capi.cu) and the
// allocation-free entry point (noalloc.cu).
#include <algorithm>
#include <cmath>
#include <cstdlib>

#include "forces.cuh"

namespace atm3 {

atm_status make_rep(const atm_params& p, long long n, long long mol0, long long cell0, Rep& r)
{
    r = Rep{};
    long long ncell = 1;
    for (int d = 0; d < 3; d++) {
        double L = p.box[d], rc = p.rc;
        if (!(L > 0.0) || !(rc > 0.0) || !std::isfinite(L) || !std::isfinite(rc)) return ATM_E_INVALID;
        double k = std::floor(L / rc);
        if (k < 1.0) k = 1.0;
        while (L / (k + 1.0) >= rc) k += 1.0;
        while (k > 0.0 && L / k < rc) k -= 1.0;
        if (k < 3.0) return ATM_E_BOX_TOO_SMALL;
        if (k > 1.0e6) return ATM_E_INVALID;
        r.g.nc[d] = (int)k;
        r.g.L[d] = L;
        r.g.w[d] = L / k;
        r.g.iw[d] = 1.0 / r.g.w[d];
        r.wf[d] = (float)r.g.w[d];
        ncell *= (long long)k;
    }
    if (ncell > (1ll << 30)) return ATM_E_INVALID;
    if (!std::isfinite(p.nu) || !std::isfinite(p.lj_eps) || !(p.lj_sigma > 0.0) ||
        !std::isfinite(p.dt))
        return ATM_E_INVALID;
    r.g.ncell = ncell;
    r.mol0 = mol0;
    r.n = n;
    r.cell0 = cell0;
    const double rc = p.rc;
    r.rc = rc;
    r.rc2 = rc * rc;
    r.rc6 = r.rc2 * r.rc2 * r.rc2;
    r.nu = p.nu;
    r.dt = p.dt;
    const float rcf = (float)rc;
    r.rcf = rcf;
    r.rc2f = rcf * rcf;
    r.rc6f = r.rc2f * r.rc2f * r.rc2f;
    r.nuf = (float)p.nu;
    const double sig2 = p.lj_sigma * p.lj_sigma;
    const double sc = sig2 / (rc * rc), sc3 = sc * sc * sc;
    r.sig2 = sig2;
    r.eps4 = 4.0 * p.lj_eps;
    r.eps24 = 24.0 * p.lj_eps;
    r.eps48 = 48.0 * p.lj_eps;
    r.ushift = p.lj_shift ? 4.0 * p.lj_eps * (sc3 * sc3 - sc3) : 0.0;
    r.sig2f = (float)r.sig2;
    r.eps4f = (float)r.eps4;
    r.eps24f = (float)r.eps24;
    r.eps48f = (float)r.eps48;
    r.ushiftf = (float)r.ushift;
    const double wmax = std::max(r.g.w[0], std::max(r.g.w[1], r.g.w[2]));
    r.p_lo = (float)(r.rc2 * (1.0 - 1.0 / 4096.0));
    r.p_hi = (float)(r.rc2 * (1.0 + 1.0 / 4096.0));
    r.q_lo = (float)(r.rc6 * (1.0 - 1.0 / 1024.0));
    r.q_hi = (float)(r.rc6 * (1.0 + 1.0 / 1024.0));
    r.dmin = (float)((0.02 * wmax) * (0.02 * wmax));
    const double wmin = std::min(r.g.w[0], std::min(r.g.w[1], r.g.w[2]));
    r.rw2 = (2.0 * wmin) * (2.0 * wmin);
    r.rw2f = (float)r.rw2;
    r.own_z0 = 0;
    r.own_z1 = r.g.nc[2];
    return ATM_OK;
}

int rc_exponent(const Rep& r) { return std::abs(std::ilogb(r.rc)); }

cudaError_t enqueue_lj(const ForceJob& j)
{
    LjArgs<double> l64{};
    LjArgs<float> l32{};
    if (j.prec == 0) {
        l64.b = j.b; l64.n = j.b.ntot; l64.xl = j.xl; l64.xl32 = j.xl32; l64.cell_start = j.start;
        l64.fs = j.f_lj; l64.mol_ew = j.mol_ew;
        l64.mol_cnt = j.mol_cnt;
    } else {
        l32.b = j.b; l32.n = j.b.ntot; l32.xl = j.xl32; l32.xl32 = j.xl32; l32.cell_start = j.start;
        l32.fs = j.f_lj; l32.mol_ew = j.mol_ew;
        l32.mol_cnt = j.mol_cnt;
    }
    return launch_lj(j.prec, l64, l32, j.st);
}

// one ATM launch over all units, or over the listed units (ulist, ucount)
static cudaError_t launch_atm_one(const ForceJob& j, size_t* smem_set, bool* capacity,
                                  const int* ulist, const int* ucount, int* work)
{
    AtmPlan P;
    // the block kernel packs staged indices in 11 bits, the owner kernels in 16
    const int limit = (j.trav == 0 || j.trav == 3) ? 65535 : ATM_MCAP_LIMIT;
    if (j.mcap > limit || !atm_choose_plan(j.trav, j.trunc, j.prec, j.mcap, j.optin, P, j.det, j.gpm16)) {
        *capacity = true;
        return cudaErrorInvalidValue;
    }
    if ((j.nwarps == 2 || j.nwarps == 4 || j.nwarps == 8) && j.trav != 0 && j.trav != 3) {
        AtmPlan Q;
        if (atm_choose_plan_nw(j.trav, j.trunc, j.prec, j.mcap, j.optin, j.nwarps, Q, j.det, j.gpm16)) P = Q;
    }
    cudaError_t e;
    // the deterministic instantiations are other kernels: their attribute is
    // set on its own (smem_set tracks the floating-point ones)
    if (j.det || !smem_set || P.smem > *smem_set) {
        e = j.prec == 0 ? atm_attr_fp64(j.trav, j.trunc, P.smem, j.det)
                        : atm_attr_fp32(j.trav, j.trunc, P.smem, j.det);
        if (e != cudaSuccess) return e;
        if (smem_set && !j.det) *smem_set = P.smem;
    }
    const int lj = j.lj && (j.trav == 1 || j.trav == 2 || j.trav == 4) && j.trunc == 0;
    int ctas = 0;
    if (j.persistent && work) {
        int per_sm = j.prec == 0 ? atm_occupancy_fp64(j.trav, j.trunc, P.nwarps, P.smem, j.det)
                                 : atm_occupancy_fp32(j.trav, j.trunc, P.nwarps, P.smem, j.det);
        ctas = std::max(1, per_sm) * std::max(1, j.sms);
        e = cudaMemsetAsync(work, 0, sizeof(int), j.st);
        if (e != cudaSuccess) return e;
    }
    if (j.prec == 0) {
        AtmArgs<double> a{};
        a.b = j.b; a.n = j.b.ntot; a.xl = j.xl; a.xl32 = j.xl32; a.cell_start = j.start;
        a.fs = j.f_atm; a.unit_ew = j.unit_ew; a.unit_cnt = j.unit_cnt; a.status = j.status;
        a.work = ctas > 0 ? work : nullptr;
        a.mcap = j.mcap;
        a.gcap = P.gcap;
        a.use_d = P.use_d;
        a.acc_mode = P.acc_mode;
        a.pcap = P.pcap;
        a.lj = lj;
        a.unit_ew2 = j.unit_ew2;
        a.unit_cnt2 = j.unit_cnt2;
        a.ulist = ulist;
        a.ucount = ucount;
        a.det = j.det;
        a.emax = j.emax;
        return launch_atm_fp64(j.trav, j.trunc, a, P.nwarps, P.smem, ctas, j.st);
    }
    AtmArgs<float> a{};
    a.b = j.b; a.n = j.b.ntot; a.xl = j.xl32; a.xl32 = j.xl32; a.cell_start = j.start;
    a.fs = j.f_atm; a.unit_ew = j.unit_ew; a.unit_cnt = j.unit_cnt; a.status = j.status;
    a.work = ctas > 0 ? work : nullptr;
    a.mcap = j.mcap;
    a.gcap = P.gcap;
    a.use_d = P.use_d;
    a.acc_mode = P.acc_mode;
    a.pcap = P.pcap;
    a.lj = lj;
    a.unit_ew2 = j.unit_ew2;
    a.unit_cnt2 = j.unit_cnt2;
    a.ulist = ulist;
    a.ucount = ucount;
    a.det = j.det;
    a.pmask = atm_uses_pair_masks(j) ? j.pmask : nullptr;
    a.emax = j.emax;
    return launch_atm_fp32(j.trav, j.trunc, a, P.nwarps, P.smem, ctas, j.st);
}

// The FP32C pair rule of 3c01, 3c18 and 3c08 takes the forward lists (liquid of
// 256,000 molecules at rho* 0.8: five steps 3.57 against 8.42 ms of the pair bitmaps
// and the block kernel; 5,003 molecules 0.14 against 0.28 ms a call).  Left to the
// owner kernel: 3c01 in parts of a domain (owner computes: only owned molecules get a
// force) and in the deterministic mode (its sums need no fixed point, so no term can
// leave the fixed-point range); to the block kernel: the corner-anchored 3c08 (not
// every triangle).  Units that do not fit shared memory are refused before by the
// block kernel's plan: 18 cells lie in four blocks of eight or two units of fourteen,
// and its adjacency holds 900 molecules a unit, the lists 6,500.
FwdLaunch atm_fwd_plan(const ForceJob& j)
{
    FwdLaunch f;
    if (j.prec != 1 || j.trunc != 0 || (j.trav != 0 && j.trav != 1 && j.trav != 2) || j.mcap_fwd <= 0 ||
        (j.trav == 0 && (!j.whole || j.det)))
        return f;
    // LJ apart only for whole systems (in a domain the LJ kernel gives owned
    // molecules their complete force) and in floating point
    f.lj = j.lj && j.trav != 0 ? 1 : (j.lj_apart && j.whole && !j.det ? 2 : 0);
    if (j.trav == 0 && f.lj != 2) return FwdLaunch();  // (no kernel of this form)
    // eight warps and a run of four cells per CTA; one cell, and several CTAs per
    // cell, while the grid would leave SMs without enough warps
    const long long sms = j.sms > 0 ? j.sms : 148, occ = (j.b.ntot + j.b.ncell - 1) / j.b.ncell;
    const long long want = sms * 24;  // warps
    if (j.nruns <= 0 || j.nruns * FWD_MAXW < 2 * want) {
        f.run = 1;
        if (occ <= 4) f.nwarps = 4;
        const long long most = std::min<long long>({FWD_SPLIT, (occ + FWD_MAXW - 1) / FWD_MAXW,
                                                    fwd_unit_slots(j.b.ncell) / j.b.ncell});
        while (f.split < most && j.b.ncell * f.nwarps * f.split < want) f.split++;
    }
    const size_t lim = j.optin > 4096 ? (size_t)j.optin - 4096 : 0;
    auto fits = [&]() {
        return fwd_stage(j.mcap_fwd, f.run) <= 65535 &&
               fwd_smem_plan(j.mcap_fwd, f.run, f.nwarps).total <= lim;
    };
    if (!fits() && f.run > 1) {
        f.run = 1;
        f.split = 1;
    }
    while (f.nwarps > 1 && !fits()) f.nwarps /= 2;
    f.use = fits();
    return f.use ? f : FwdLaunch();  // (no LJ from lists that are not taken)
}

// The FP64 pair rule of 3c01, 3c18 and 3c08 on whole systems, outside the
// deterministic mode and with every cell within the bitmaps' 32 molecules:
// forces and LJ of 32,000 molecules 0.68 ms against 1.67 ms of the block kernel
// and 0.62 ms of the LJ kernel, of 1,000 molecules 0.06 ms against 0.87 ms of the
// owner and LJ kernels.  (Their first test is of FP32 squares, which hold r_c^2 to
// full precision for r_c within 2^+-40.)
FwdLaunch atm_list64_plan(const ForceJob& j)
{
    FwdLaunch f;
    if (j.prec != 0 || j.trunc != 0 || (j.trav != 0 && j.trav != 1 && j.trav != 2) || !j.l64 ||
        !j.l64->list || j.det || !j.whole || j.rc_exp > LIST64_RC_EXP || j.mcap_fwd <= 0 || j.mcap_fwd > j.l64->stride ||
        j.mcap_fwd > 65535)
        return f;
    f.lj = j.lj && j.trav != 0 ? 1 : (j.lj_apart ? 2 : 0);
    if (!f.lj) return f;
    if (j.nruns <= 0 || j.nruns * 2 < j.sms * 8) f.run = 1;  // fewer cells than fill the SMs in runs
    const long long occ = (j.b.ntot + j.b.ncell - 1) / j.b.ncell;
    if (f.run == 1 && j.b.ncell < 4ll * j.sms && occ > FWD_MAXW) f.split = 2;
    if (list64_smem(j.mcap_fwd, f.run) > LIST64_SMEM) f.run = 1;
    f.use = list64_smem(j.mcap_fwd, f.run) <= LIST64_SMEM;
    return f.use ? f : FwdLaunch();
}

// The product rule of 3c01, 3c18, 3c08 and 3c08a outside the deterministic mode (its
// sums are fixed-point, in the block kernel, or in a fixed order, in the owner
// kernel), while two warps' tables fit beside the largest unit (FP64 3c08 with a table of
// 220 molecules' pairs 1.7 ms against 3.2 of the block kernel, one warp beside 230: 5.4
// against 3.6).  32,000 molecules, 3c18 FP32 3.93 -> 1.01 ms a call; 15,001, 3c08 FP64
// 3.74 -> 2.09; 7,811, 3c01 FP64 12.2 -> 3.9; vapours (8,000 molecules, densities 0.001
// to 0.1) 0.2 to 0.9 of the others' times, but for 3c01 in FP64 with units of 14 to 32
// molecules (1.03 to 1.25; of 61 0.84).
// FP64: for r_c within 2^+-16, where the scan's FP32 products of six lengths are far
// from the ends of their range (an r_c of 1e-9, in metres, would find no triplet); the
// other kernels decide in FP64 what FP32 cannot.
ProdLaunch atm_prod_plan(const ForceJob& j)
{
    ProdLaunch l;
    if (j.trunc != 1 || j.trav < 0 || j.trav > 4 || j.trav == 3 || j.det || j.mcap < 1 || j.mcap > 65535 ||
        (j.trav != 0 && j.mcap > ATM_MCAP_LIMIT) || (j.prec == 0 && (!j.x || j.rc_exp > PROD64_RC_EXP)) ||
        (j.trav == 0 && j.prec == 0 && j.mcap < PROD64_OWNER_MIN))
        return l;
    const bool f64 = j.prec == 0;
    const long long fixed = f64 ? prod_smem<double>(j.trav, j.mcap).total : prod_smem<float>(j.trav, j.mcap).total;
    const long long warp = f64 ? prod_warp_smem<double>(j.trav, j.mcap).total
                               : prod_warp_smem<float>(j.trav, j.mcap).total;
    const long long lim = j.optin > 4096 ? (long long)j.optin - 4096 : 0;
    // an SM holds 20 (FP64) or 32 (FP32) warps of these kernels; four, three or two
    // CTAs to it while four warps' tables fit the largest unit and there are units
    // for them; of units of up to 64 molecules, CTAs of four warps
    for (int c = j.mcap <= 64 ? (f64 ? 5 : 8) : (f64 ? 2 : 4); c >= 1; c--) {
        const long long room = std::min<long long>(lim, 233472 / c - 2560);
        if (c > 1 && ((long long)j.b.ncell < (long long)c * j.sms || fixed + 4 * warp > room)) continue;
        if (fixed + 2 * warp > room) return l;
        l.warps = std::min<int>(PROD_MAXW, (f64 ? 20 : 32) / c);
        l.smem = (int)std::min<long long>(room, fixed + l.warps * warp);
        return l;
    }
    return l;
}

template <typename R>
static cudaError_t launch_prod(const ForceJob& j, const R* xl, const ProdLaunch& l)
{
    AtmArgs<R> a{};
    a.b = j.b; a.n = j.b.ntot; a.xl = xl; a.xl32 = j.xl32; a.cell_start = j.start;
    a.fs = j.f_atm; a.unit_ew = j.unit_ew; a.unit_cnt = j.unit_cnt; a.status = j.status;
    a.mcap = j.mcap;
    a.gcap = l.smem;
    a.x = j.x;
    a.perm = j.perm;
    return launch_atm_prod<R>(j.trav, a, l.warps, j.st);
}

static cudaError_t launch_l64(const ForceJob& j, const FwdLaunch& f)
{
    List64Args a = *j.l64;
    a.b = j.b;
    a.n = j.b.ntot;
    a.xl = j.xl;
    a.xl32 = j.xl32;
    a.cell_start = j.start;
    a.cell_sorted = j.cell_sorted;
    a.mol_ew = j.mol_ew;
    a.mol_cnt = j.mol_cnt;
    a.fs = j.f_atm;
    a.fs_lj = j.f_lj;
    a.status = j.status;
    a.mcap = j.mcap_fwd;
    a.run = f.run;
    a.runs = j.runs;
    a.nruns = j.nruns;
    a.split = f.split;
    a.lj = f.lj;
    return launch_list64(a, j.st);
}

static cudaError_t launch_fwd(const ForceJob& j, const FwdLaunch& f)
{
    FwdArgs a{};
    a.b = j.b;
    a.n = j.b.ntot;
    a.xl = j.xl32;
    a.cell_start = j.start;
    a.fs = j.f_atm;
    a.fs_lj = j.f_lj;
    a.unit_ew = j.unit_ew;
    a.unit_cnt = j.unit_cnt;
    a.unit_ew2 = j.unit_ew2;
    a.unit_cnt2 = j.unit_cnt2;
    a.status = j.status;
    a.mcap = j.mcap_fwd;
    a.run = f.run;
    a.runs = j.runs;
    a.nruns = j.nruns;
    a.split = f.split;
    a.lj = f.lj;
    a.trav = j.trav;
    return launch_atm_fwd(a, j.det, f.nwarps, j.st);
}

bool atm_uses_pair_masks(const ForceJob& j)
{
    return j.pmask && j.prec == 1 && j.trunc == 0 && j.trav == 4 && j.b.ntot > 0;
}

bool atm_split_active(const ForceJob& j)
{
    return !atm_uses_lists(j) && !atm_prod_plan(j).warps && j.ncls > 1 && (j.trav == 1 || j.trav == 2 || j.trav == 4) && j.ulist && j.ucount &&
           j.b.ncell > 0;
}

static cudaError_t enqueue_atm_launches(const ForceJob& j, size_t* smem_set, bool* capacity);

cudaError_t enqueue_atm(const ForceJob& j, size_t* smem_set, bool* capacity)
{
    cudaError_t e = enqueue_atm_launches(j, smem_set, capacity);
    // deterministic block traversals left 64-bit fixed-point sums in f_atm
    if (e == cudaSuccess && j.det && (j.trav == 1 || j.trav == 2 || j.trav == 4) && j.b.ntot > 0)
        e = launch_fix_to_double(j.f_atm, 3 * j.b.ntot, j.prec == 0 ? FixBits<double>::B
                                                                   : FixBits<float>::B, j.st);
    return e;
}

// f_atm, and f_lj too, to zero (one operation where f_atm follows f_lj)
static cudaError_t zero_forces(const ForceJob& j, bool lj)
{
    const size_t m = 3 * (size_t)j.b.ntot;
    if (lj && j.f_atm == j.f_lj + m) return cudaMemsetAsync(j.f_lj, 0, 2 * m * sizeof(double), j.st);
    const cudaError_t e = cudaMemsetAsync(j.f_atm, 0, m * sizeof(double), j.st);
    return e == cudaSuccess && lj ? cudaMemsetAsync(j.f_lj, 0, m * sizeof(double), j.st) : e;
}

static cudaError_t enqueue_atm_launches(const ForceJob& j, size_t* smem_set, bool* capacity)
{
    *capacity = false;
    {
        // every launch's plan must fit before anything is enqueued
        AtmPlan P;
        const int limit = (j.trav == 0 || j.trav == 3) ? 65535 : ATM_MCAP_LIMIT;
        if (j.mcap > limit || !atm_choose_plan(j.trav, j.trunc, j.prec, j.mcap, j.optin, P, j.det, j.gpm16)) {
            *capacity = true;
            return cudaErrorInvalidValue;
        }
    }
    cudaError_t e;
    const FwdLaunch f = atm_fwd_plan(j), f64 = atm_list64_plan(j);
    if (f64.use && j.b.ntot > 0) {
        e = zero_forces(j, true);
        return e == cudaSuccess ? launch_l64(j, f64) : e;
    }
    if (f.use) {
        if (j.b.ntot <= 0) return launch_fwd(j, f);
        e = zero_forces(j, f.lj != 0);
        return e == cudaSuccess ? launch_fwd(j, f) : e;
    }
    if (const ProdLaunch l = atm_prod_plan(j); l.warps) {
        if (j.b.ntot > 0) {
            e = cudaMemsetAsync(j.f_atm, 0, 3 * (size_t)j.b.ntot * sizeof(double), j.st);
            if (e != cudaSuccess) return e;
        }
        return j.prec == 0 ? launch_prod<double>(j, j.xl, l) : launch_prod<float>(j, j.xl32, l);
    }
    if (j.trav != 0 && j.trav != 3 && j.b.ntot > 0) {  // owner traversals write every F_i
        e = cudaMemsetAsync(j.f_atm, 0, 3 * (size_t)j.b.ntot * sizeof(double), j.st);
        if (e != cudaSuccess) return e;
    }
    const int lj = j.lj && (j.trav == 1 || j.trav == 2 || j.trav == 4) && j.trunc == 0;
    if (lj && j.b.ntot > 0) {  // the units write LJ + ATM into f_atm
        e = cudaMemsetAsync(j.f_lj, 0, 3 * (size_t)j.b.ntot * sizeof(double), j.st);
        if (e != cudaSuccess) return e;
    }
    if (atm_uses_pair_masks(j)) {
        e = launch_pair_masks(j.b, j.start, j.xl32, j.cell_sorted, j.pmask, j.status, j.st);
        if (e != cudaSuccess) return e;
    }
    if (!atm_split_active(j)) return launch_atm_one(j, smem_set, capacity, nullptr, nullptr, j.work);
    e = launch_unit_classes(j.b, j.start, j.trav, j.ncls, j.cuts[0], j.cuts[1], j.ulist, j.ucount,
                            j.st);
    if (e != cudaSuccess) return e;
    // the small-unit class on the side stream, beside the others: its CTAs
    // fill the SMs the larger units' launch leaves idle in its tail
    const bool side = j.side_st && j.ev_fork && j.ev_join;
    if (side) {
        e = cudaEventRecord(j.ev_fork, j.st);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(j.side_st, j.ev_fork, 0);
        if (e != cudaSuccess) return e;
    }
    for (int k = 0; k < j.ncls && e == cudaSuccess; k++) {
        ForceJob jk = j;
        if (side && k == 0) jk.st = j.side_st;
        if (k < j.ncls - 1) {
            jk.mcap = std::min(j.cuts[k], j.mcap);
            // small units: short phases between the CTA's barriers, so few
            // warps (64-molecule bound: 2 warps measured best on a batch of
            // 64 uneven replicas, against 1 and 4)
            if (j.cuts[k] <= 64) jk.nwarps = 2;
        }
        if (jk.mcap < 1) jk.mcap = 1;
        e = launch_atm_one(jk, smem_set, capacity, j.ulist + (size_t)k * j.b.ncell, j.ucount + k,
                           j.work ? j.work + k : nullptr);
    }
    if (side) {
        // once forked, the side stream is always joined back (a capture
        // must not end with it unjoined, and later work on st must follow
        // what was queued there); the first error is the one returned
        cudaError_t ej = cudaEventRecord(j.ev_join, j.side_st);
        if (ej == cudaSuccess) ej = cudaStreamWaitEvent(j.st, j.ev_join, 0);
        if (e == cudaSuccess) e = ej;
    }
    return e;
}

}  // namespace atm3

// md_kernels.cu -- linked-cell build, LJ pair forces, velocity-Verlet update,
// density profile and the per-replica reductions (in a fixed order).
// Every kernel works on a batch of replicas (a single system is a batch of
// one): per-molecule threads look their replica up in rep_of_mol, per-cell
// threads in rep_of_cell.
#include "md_kernels.cuh"

namespace atm3 {

// ---------------------------------------------------------------- linked cells

// periodic wrap into [0, L): t = x - floor(x/L) L, folded once more if the
// rounding lands outside [0, L).  A value already in [0, L) comes back
// unchanged from those steps (x/L rounds to below 1, or to 1 and then
// x - L and (x - L) + L are exact), so it skips the division.
__device__ __forceinline__ double wrap1(double x, double L)
{
    if (x >= 0.0 && x < L) return x;
    double t = __dsub_rn(x, __dmul_rn(floor(__ddiv_rn(x, L)), L));
    if (t < 0.0) t = __dadd_rn(t, L);
    if (t >= L) t = 0.0;
    return t;
}

// cell coordinate floor(t / w) (correctly rounded quotient) and clamped
// cell-local coordinate in [0, w].  q = t * (1/w) is within 3 units of 2^-53
// |t/w| of the rounded quotient, so when no integer lies within 5 units of q
// both have the same floor and the division is skipped.
__device__ __forceinline__ int bin1(double t, double w, double iw, int n, double& loc)
{
    const double q = __dmul_rn(t, iw);
    const double fq = floor(q);
    const double tol = __dmul_rn(fabs(q), 5.551115123125783e-16);  // 5 * 2^-53
    int c;
    if (__dsub_rn(q, fq) > tol && __dsub_rn(__dadd_rn(fq, 1.0), q) > tol)
        c = (int)fq;
    else
        c = (int)floor(__ddiv_rn(t, w));
    c = c > n - 1 ? n - 1 : (c < 0 ? 0 : c);
    double l = __dsub_rn(t, __dmul_rn((double)c, w));
    l = l < 0.0 ? 0.0 : (l > w ? w : l);
    loc = l;
    return c;
}

// a non-negative finite double to FP32, the mantissa cut off (integer work: a
// conversion takes the FP64 pipe); below 2^-126 zero, from 2^128 infinity
__device__ __forceinline__ float cut32(double t)
{
    const int hi = __double2hiint(t);  // (-0: zero too)
    if (hi >= 0x47f00000) return __int_as_float(0x7f800000);
    return hi < 0x38100000 ? 0.0f
                           : __uint_as_float(((unsigned)(hi - 0x38000000) << 3) | ((unsigned)__double2loint(t) >> 29));
}

// a non-negative double to FP32, rounded to nearest even (integer work again,
// where the result is a normal number below 2^127)
__device__ __forceinline__ float round32(double t)
{
    const unsigned long long u = (unsigned long long)__double_as_longlong(t);
    if (u - 0x3810000000000000ull >= 0x0fd0000000000000ull) return (float)t;
    return __uint_as_float((unsigned)((u + 0x0fffffffull + ((u >> 29) & 1ull)) >> 29) - (896u << 23));
}

// K1: wrap positions in place, global cell id per molecule, cell histogram
// with the arrival rank of each molecule.  A coordinate in [0, L) (one integer
// compare: the bits of non-negative doubles order as they do) stays as it is, and
// its cell comes from an FP32 quotient wherever that lies farther from an integer
// than its error; the FP64 pipe, which takes 16 cycles a warp instruction, is left to
// the others.  256,000 molecules: 22 -> 8.3 us.
__global__ void k_wrap_bin(Batch B, double* __restrict__ x, int* __restrict__ cell_of,
                           int* __restrict__ rank, int* __restrict__ count, int* __restrict__ maxocc,
                           int* __restrict__ status)
{
    after_previous();
    const long long n = B.ntot;
    long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i < 1 + ATM_NUNIT) maxocc[i] = 0;  // (k_unit_max raises them)
    if (i >= n) return;
    const Rep& rp = B.rep[B.rep_of_mol[i]];
    double xv[3];
    for (int d = 0; d < 3; d++) xv[d] = x[d * n + i];
    int cc[3];
    for (int d = 0; d < 3; d++) {
        double t = xv[d];
        if ((unsigned long long)__double_as_longlong(t) >= (unsigned long long)__double_as_longlong(rp.g.L[d])) {
            if (!isfinite(t)) {
                atomicOr(status, ST_NONFINITE);
                t = 0.0;
            }
            t = wrap1(t, rp.g.L[d]);
            x[d * n + i] = t;
        }
        // both factors cut to 2^-23, the product rounded to 2^-24: within 2^-21.6
        const float q = cut32(t) * cut32(rp.g.iw[d]), fq = floorf(q), tol = q * 0x1p-21f;
        const int nc = rp.g.nc[d];
        if (q - fq > tol && (fq + 1.0f) - q > tol) {
            cc[d] = min((int)fq, nc - 1);
        } else {
            double loc;
            cc[d] = bin1(t, rp.g.w[d], rp.g.iw[d], nc, loc);
        }
    }
    int id = (int)rp.cell0 + (cc[2] * rp.g.nc[1] + cc[1]) * rp.g.nc[0] + cc[0];
    cell_of[i] = id;
    rank[i] = atomicAdd(count + id, 1);
}

// K2: exclusive scan of the cell counts (one CTA of 1024 threads, each warp
// owns a contiguous segment); the counts are left at zero
__global__ void __launch_bounds__(1024) k_scan(long long ncell, int* __restrict__ count,
                                               int* __restrict__ start)
{
    after_previous();
    // warp w owns the contiguous segment [w seg, (w + 1) seg) of the cells and
    // reads it 256 consecutive counts at a time (coalesced, eight loads in flight:
    // 19,683 cells 10 -> 8.4 us): its total first, then, after a scan of the 32
    // totals, the exclusive prefix of every cell with a shuffle scan per 32 and
    // a running carry
    constexpr int U = 8;
    __shared__ int s_tot[32];
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long seg = ((ncell + 31) / 32 + 31) / 32 * 32;
    const long long lo = warp * seg, hi = lo + seg < ncell ? lo + seg : ncell;
    int tot = 0;
    for (long long c0 = lo; c0 < hi; c0 += 32 * U) {
        int v[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            const long long c = c0 + 32 * u + lane;
            v[u] = c < hi ? count[c] : 0;
        }
#pragma unroll
        for (int u = 0; u < U; u++) tot += v[u];
    }
    tot = __reduce_add_sync(FULL, tot);
    if (lane == 0) s_tot[warp] = tot;
    __syncthreads();
    if (warp == 0) {
        const int t = s_tot[lane];
        int incl = t;
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(FULL, incl, o);
            if (lane >= o) incl += u;
        }
        s_tot[lane] = incl - t;  // exclusive: the cells before warp lane's segment
        if (lane == 31) start[ncell] = incl;
    }
    __syncthreads();
    int carry = s_tot[warp];
    for (long long c0 = lo; c0 < hi; c0 += 32 * U) {
        int v[U], incl[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            const long long c = c0 + 32 * u + lane;
            incl[u] = v[u] = c < hi ? count[c] : 0;
        }
        for (int o = 1; o < 32; o <<= 1) {
#pragma unroll
            for (int u = 0; u < U; u++) {
                const int t = __shfl_up_sync(FULL, incl[u], o);
                if (lane >= o) incl[u] += t;
            }
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
            const long long c = c0 + 32 * u + lane;
            if (c < hi) {
                start[c] = carry + incl[u] - v[u];
                count[c] = 0;  // for the next build
            }
            carry += __shfl_sync(FULL, incl[u], 31);
        }
    }
}

// out[0] the largest cell, out + 1 the largest staged-molecule count of a
// traversal unit, per traversal: 3c01 (27 cells), 3c18 (base + 13 forward), 3c08
// (2x2x2 block), [ATM_FWD_UNIT] the forward lists' 18 cells (the base cell's layer
// and the next).  From the counts alone (27 independent loads a cell), so it comes
// before the scan and the host can read it while the molecules are sorted.
__global__ void k_unit_max(Batch B, const int* __restrict__ count, int wide, int* __restrict__ out)
{
    after_previous();
    long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    int m01 = 0, m18 = 0, m08 = 0, mw = 0, mf = 0, own = 0;
    if (c < B.ncell) {
        const Rep& rp = B.rep[B.rep_of_cell[c]];
        const int* ct = count + rp.cell0;
        int cx, cy, cz;
        cell_coords(rp.g, c - rp.cell0, cx, cy, cz);
        const int nx = rp.g.nc[0], ny = rp.g.nc[1], nz = rp.g.nc[2];
        const int xs[3] = {cx > 0 ? cx - 1 : nx - 1, cx, cx + 1 < nx ? cx + 1 : 0};
        const int ys[3] = {nx * (cy > 0 ? cy - 1 : ny - 1), nx * cy, nx * (cy + 1 < ny ? cy + 1 : 0)};
        const int zs[3] = {nx * ny * (cz > 0 ? cz - 1 : nz - 1), nx * ny * cz, nx * ny * (cz + 1 < nz ? cz + 1 : 0)};
        int k[27];
#pragma unroll
        for (int t = 0; t < 27; t++) k[t] = ct[zs[t / 9] + ys[(t / 3) % 3] + xs[t % 3]];
#pragma unroll
        for (int t = 0; t < 27; t++) {
            m01 += k[t];
            if (t >= 13) m18 += k[t];
            if (t >= 9) mf += k[t];
            if (t % 3 >= 1 && (t / 3) % 3 >= 1 && t / 9 >= 1) m08 += k[t];
        }
        own = k[13];
        // the wide traversal's 5^3 neighbourhood (only when that traversal is in use)
        for (int t = 0; t < (wide ? 125 : 0); t++)
            mw += ct[cell_at(rp.g, cx, cy, cz, t % 5 - 2, (t / 5) % 5 - 2, t / 25 - 2)];
    }
    // block maximum first: one global atomic per value and block
    __shared__ int s_m[6][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int m[6] = {own, m01, m18, m08, mw, mf};
#pragma unroll
    for (int q = 0; q < 6; q++) {
        const int v = __reduce_max_sync(0xffffffffu, m[q]);
        if (lane == 0) s_m[q][warp] = v;
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        const int q = threadIdx.x;
        int v = 0;
        for (int w = 0; w < nw; w++) v = max(v, s_m[q][w]);
        atomicMax(out + (q == 5 ? 1 + ATM_FWD_UNIT : q), v);
        // the corner-anchored 3c08 stages the same blocks as 3c08
        if (q == 3) atomicMax(out + 5, v);
    }
}

// Unit size classes of the block traversals: unit u (its base cell) holds
// the molecules of its 8 cells (3c08, corner-anchored 3c08) or 14 cells
// (3c18); it goes to the first class whose bound holds them (cut0, then cut1
// when there are three classes; the last class takes the rest).  Class k is
// listed in ulist[k * ncell ..] and counted in counts[k] (zero at launch).
__global__ void k_unit_classes(Batch B, const int* __restrict__ start, int trav, int ncls,
                               int cut0, int cut1, int* __restrict__ ulist,
                               int* __restrict__ counts)
{
    const long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    int cls = -1;
    if (c < B.ncell) {
        const Rep& rp = B.rep[B.rep_of_cell[c]];
        const int* st = start + rp.cell0;
        int cx, cy, cz;
        cell_coords(rp.g, c - rp.cell0, cx, cy, cz);
        int m = 0;
        for (int t = 0; t < 27; t++) {
            int dx, dy, dz;
            offset27(t, dx, dy, dz);
            if (trav == 1 ? t >= 13 : (dx >= 0 && dy >= 0 && dz >= 0)) {
                const long long nc = cell_at(rp.g, cx, cy, cz, dx, dy, dz);
                m += st[nc + 1] - st[nc];
            }
        }
        cls = m <= cut0 ? 0 : ((ncls > 2 && m <= cut1) ? 1 : ncls - 1);
    }
    // one append per class and warp
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    for (int k = 0; k < ncls; k++) {
        const unsigned mk = __ballot_sync(FULL, cls == k);
        if (mk == 0u) continue;
        const int lead = __ffs(mk) - 1;
        int base = 0;
        if (lane == lead) base = atomicAdd(counts + k, __popc(mk));
        base = __shfl_sync(FULL, base, lead);
        if (cls == k) ulist[k * B.ncell + base + __popc(mk & ((1u << lane) - 1u))] = (int)c;
    }
}

// K3a: scatter by arrival rank
__global__ void k_scatter(long long n, const int* __restrict__ cell_of, const int* __restrict__ rank,
                          const int* __restrict__ start, int* __restrict__ list)
{
    after_previous();
    long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= n) return;
    list[start[cell_of[i]] + rank[i]] = (int)i;
}

// K3b+c: a thread per entry of the unsorted lists restores the original index
// order inside its cell (its place is the number of the cell's entries below it)
// and writes, for its sorted slot, the FP64 and FP32 cell-local coordinates (t - c
// w clamped to [0, w], the cell's own c: the binning's arithmetic without its
// division) and the global cell.  Full warps of entries, not a warp per cell, and
// integer compares and conversions: 9 FP64 instructions a warp (256,000 molecules
// in cells of 13: 26 -> 12 us).
__global__ void __launch_bounds__(128) k_cell_order(Batch B, const double* __restrict__ x,
                                                    const int* __restrict__ cell_of,
                                                    const int* __restrict__ start,
                                                    const int* __restrict__ list,
                                                    int* __restrict__ perm, double* __restrict__ xl,
                                                    float* __restrict__ xl32,
                                                    int* __restrict__ cell_sorted)
{
    after_previous();
    const long long n = B.ntot;
    const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (e >= n) return;
    const int i = list[e];
    const int c = cell_of[i];
    double t[3];
    for (int d = 0; d < 3; d++) t[d] = x[d * n + i];
    const int lo = start[c], hi = start[c + 1];
    int s = lo;
    for (int k = lo; k < hi; k++) s += list[k] < i ? 1 : 0;
    const Rep& rp = B.rep[B.rep_of_cell[c]];
    int cc[3];
    cell_coords(rp.g, c - rp.cell0, cc[0], cc[1], cc[2]);
    perm[s] = i;
    cell_sorted[s] = c;
    for (int d = 0; d < 3; d++) {
        const double w = rp.g.w[d];
        // (double)cc, exactly
        const double cd = __dsub_rn(__hiloint2double(0x43300000, cc[d]), 0x1p52);
        double l = __dsub_rn(t[d], __dmul_rn(cd, w));
        // l < 0 ? 0 : (l > w ? w : l)
        const long long b = __double_as_longlong(l), bw = __double_as_longlong(w);
        l = __longlong_as_double(b < 0 ? 0 : (b > bw ? bw : b));
        xl[d * n + s] = l;
        xl32[d * n + s] = round32(l);
    }
}

// ---------------------------------------------------------------- LJ pairs

template <typename R>
struct LjArith;
template <>
struct LjArith<double> {
    static __device__ __forceinline__ double add(double a, double b) { return __dadd_rn(a, b); }
    static __device__ __forceinline__ double sub(double a, double b) { return __dsub_rn(a, b); }
    static __device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
    static __device__ __forceinline__ double rcp(double a) { return __drcp_rn(a); }
};
template <>
struct LjArith<float> {
    static __device__ __forceinline__ float add(float a, float b) { return __fadd_rn(a, b); }
    static __device__ __forceinline__ float sub(float a, float b) { return __fsub_rn(a, b); }
    static __device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
    static __device__ __forceinline__ float rcp(float a) { return __frcp_rn(a); }
};

// LJ (section 5) with owner-computes over the 27-cell neighbourhood: every
// molecule sums its own pair forces (no atomics, deterministic); each pair is
// seen from both ends, so the energy and virial take half per visit.  The
// candidate and interacting counts are those of the half-shell traversal:
// later molecules of the own cell plus the 13 forward cells (what is staged
// after the molecule), so every pair is counted once, by one of its molecules
// (also when the two belong to different domains).
//
// A CTA per base cell stages the 27 cells, a tile at a time.  Eight lanes share a
// molecule: they take its candidates in turn (a broadcast row of 128 bytes for the
// four molecules of a warp), test them in FP32 on unit-frame positions (9
// instructions, within 2^-16 r_c^2 of the canonical square) into a bit each, then
// every lane evaluates its own hits, a sixth of them, with the canonical
// displacement and decision.  With a thread a molecule straight from global memory
// nearly every candidate was a hit of some lane, and the chain of loads bound it:
// FP32, 100,003 molecules 103 -> 67 us, 32,000 molecules 83 -> 34; FP64, 15,001
// molecules 327 -> 142, bound by the FP64 pipe.
constexpr int LJ_PARTS = 8, LJ_TILE = 512;
template <typename R>
__device__ __forceinline__ void lj_cell(const LjArgs<R>& A, const long long u)
{
    typedef LjArith<R> Q;
    constexpr bool f64 = sizeof(R) == 8;
    constexpr unsigned FULL = 0xffffffffu;
    __shared__ float4 S4[LJ_TILE];  // unit-frame position, offset27
    __shared__ int s_g[LJ_TILE];    // sorted index
    __shared__ int s_beg[28], s_g0[27];
    __shared__ float4 s_off[27];
    const int tid = threadIdx.x, lane = tid & 31;
    const long long n = A.n;
    if (A.cell_start[u] == A.cell_start[u + 1]) return;
    const Rep& rp = A.b.rep[A.b.rep_of_cell[u]];
    const int* st = A.cell_start + rp.cell0;
    int cx, cy, cz;
    cell_coords(rp.g, u - rp.cell0, cx, cy, cz);
    if (cz < rp.own_z0 || cz >= rp.own_z1) {
        // another domain's molecules: no pair terms here
        for (int s = A.cell_start[u] + tid; s < A.cell_start[u + 1]; s += blockDim.x) {
            A.fs[s] = A.fs[n + s] = A.fs[2 * n + s] = 0.0;
            A.mol_ew[2 * s] = A.mol_ew[2 * s + 1] = 0.0;
            A.mol_cnt[2 * s] = A.mol_cnt[2 * s + 1] = 0u;
        }
        return;
    }
    if (tid < 32) {
        int cnt = 0;
        if (lane < 27) {
            int dx, dy, dz;
            offset27(lane, dx, dy, dz);
            const long long c = cell_at(rp.g, cx, cy, cz, dx, dy, dz);
            s_g0[lane] = st[c];
            cnt = st[c + 1] - st[c];
            s_off[lane] = make_float4((float)dx, (float)dy, (float)dz, 0.0f);
        }
        int incl = cnt;
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(FULL, incl, o);
            if (lane >= o) incl += v;
        }
        if (lane < 27) s_beg[lane + 1] = incl;
        if (lane == 0) s_beg[0] = 0;
    }
    __syncthreads();
    const int M = s_beg[27], b0 = s_beg[13], M0 = s_beg[14] - b0;  // staged, and the base cell's
    if (M0 == 0) return;
    const float wf0 = rp.wf[0], wf1 = rp.wf[1], wf2 = rp.wf[2];
    const R w0 = f64 ? (R)rp.g.w[0] : (R)wf0, w1 = f64 ? (R)rp.g.w[1] : (R)wf1, w2 = f64 ? (R)rp.g.w[2] : (R)wf2;
    const R rc2 = f64 ? (R)rp.rc2 : (R)rp.rc2f;
    const R sig2 = f64 ? (R)rp.sig2 : (R)rp.sig2f;
    const R eps4 = f64 ? (R)rp.eps4 : (R)rp.eps4f;
    const R eps24 = f64 ? (R)rp.eps24 : (R)rp.eps24f;
    const R eps48 = f64 ? (R)rp.eps48 : (R)rp.eps48f;
    const R ushift = f64 ? (R)rp.ushift : (R)rp.ushiftf;
    // (FP64: the band of its prefilter; a comparison that zeros, infinities and NaN of
    // FP32 pass, so that units far from 1 are decided in FP64)
    const float c_hi = f64 ? rp.p_hi : rp.rc2f * (1.0f + 0x1p-16f);
    const int part = tid % LJ_PARTS;
    auto stage = [&](int base) {
        for (int k = tid; k < LJ_TILE && base + k < M; k += LJ_BLOCK) {
            const int t = base + k;
            int s = 0;  // the last slot that begins at or before t (an empty one has no t)
            for (int h = 16; h > 0; h >>= 1)
                if (s + h < 27 && s_beg[s + h] <= t) s += h;
            const int g = s_g0[s] + t - s_beg[s];
            const float4 o = s_off[s];
            S4[k] = make_float4(A.xl32[g] + o.x * wf0, A.xl32[n + g] + o.y * wf1, A.xl32[2 * n + g] + o.z * wf2,
                                __int_as_float(s));
            s_g[k] = g;
        }
    };
    // molecules of the base cell, 16 at a time
    for (int k0 = 0; k0 < M0; k0 += LJ_BLOCK / LJ_PARTS) {
        const bool valid = k0 + tid / LJ_PARTS < M0;  // (the shuffles want whole warps)
        const int k = min(k0 + tid / LJ_PARTS, M0 - 1), i = b0 + k;
        const long long s = s_g0[13] + k;
        const float fx0 = A.xl32[s], fy0 = A.xl32[n + s], fz0 = A.xl32[2 * n + s];
        R xs = fx0, ys = fy0, zs = fz0;
        if constexpr (f64) {
            xs = A.xl[s];
            ys = A.xl[n + s];
            zs = A.xl[2 * n + s];
        }
        R fx = 0, fy = 0, fz = 0, esum = 0, wsum = 0;
        unsigned pairs = 0;
        for (int base = 0; base < M; base += LJ_TILE) {
            if (k0 == 0 || M > LJ_TILE) {
                __syncthreads();
                stage(base);
                __syncthreads();
            }
            const int e = valid ? min(LJ_TILE, M - base) : 0;
            // 32 of the lane's candidates: c0 + part, c0 + part + 8, ..
            for (int c0 = 0; c0 < e; c0 += 32 * LJ_PARTS) {
                unsigned hit = 0;
                const int m = min(32, (e - c0 - part + LJ_PARTS - 1) / LJ_PARTS);
#pragma unroll 4
                for (int b = 0; b < m; b++) {
                    const float4 p = S4[c0 + part + b * LJ_PARTS];
                    const float dx = p.x - fx0, dy = p.y - fy0, dz = p.z - fz0;
                    const float c = dx * dx + dy * dy + dz * dz;
                    if (f64 ? !(c > c_hi) : c < c_hi) hit |= 1u << b;
                }
                while (hit) {
                    const int q = c0 + part + (__ffs(hit) - 1) * LJ_PARTS, t = base + q;
                    hit &= hit - 1;
                    if (t == i) continue;
                    const long long g = s_g[q];
                    const float4 o = s_off[__float_as_int(S4[q].w)];
                    const R* xl = A.xl;  // (FP32: xl32)
                    const R ddx = Q::add(Q::sub(xl[g], xs), Q::mul((R)o.x, w0));
                    const R ddy = Q::add(Q::sub(xl[n + g], ys), Q::mul((R)o.y, w1));
                    const R ddz = Q::add(Q::sub(xl[2 * n + g], zs), Q::mul((R)o.z, w2));
                    const R a = Q::add(Q::add(Q::mul(ddx, ddx), Q::mul(ddy, ddy)), Q::mul(ddz, ddz));
                    if (!(a < rc2)) continue;
                    if (t > i) pairs++;
                    const R ia = Q::rcp(a);  // correctly rounded: the same value as 1 / a
                    const R s2 = sig2 * ia;
                    const R s3 = s2 * s2 * s2;
                    const R s6 = s3 * s3;
                    const R fw = (eps48 * s6 - eps24 * s3) * ia;  // F_s = -fw d
                    fx -= fw * ddx;
                    fy -= fw * ddy;
                    fz -= fw * ddz;
                    esum += eps4 * (s6 - s3) - ushift;
                    wsum += fw * a;
                }
            }
        }
        for (int o = 1; o < LJ_PARTS; o <<= 1) {
            fx += __shfl_xor_sync(FULL, fx, o);
            fy += __shfl_xor_sync(FULL, fy, o);
            fz += __shfl_xor_sync(FULL, fz, o);
            esum += __shfl_xor_sync(FULL, esum, o);
            wsum += __shfl_xor_sync(FULL, wsum, o);
            pairs += __shfl_xor_sync(FULL, pairs, o);
        }
        if (valid && part == 0) {
            A.fs[s] = (double)fx;
            A.fs[n + s] = (double)fy;
            A.fs[2 * n + s] = (double)fz;
            A.mol_ew[2 * s] = 0.5 * (double)esum;
            A.mol_ew[2 * s + 1] = 0.5 * (double)wsum;
            A.mol_cnt[2 * s] = (unsigned)(M - 1 - i);
            A.mol_cnt[2 * s + 1] = pairs;
        }
    }
}

// One cell per CTA, or (MANY, in vapours) A.per of them, the empty ones passed over
// together (20 molecules in a million cells: 870 us with a CTA each)
template <typename R, bool MANY>
__global__ void __launch_bounds__(LJ_BLOCK) k_lj_owner(const LjArgs<R> A)
{
    after_previous();
    if constexpr (!MANY) {
        lj_cell<R>(A, blockIdx.x);
        return;
    }
    __shared__ unsigned s_full[LJ_BLOCK / 32];
    const long long u0 = (long long)blockIdx.x * A.per, u = u0 + threadIdx.x;
    const unsigned m = __ballot_sync(0xffffffffu, threadIdx.x < A.per && u < A.b.ncell &&
                                                      A.cell_start[u] != A.cell_start[u + 1]);
    if ((threadIdx.x & 31) == 0) s_full[threadIdx.x >> 5] = m;
    __syncthreads();
    for (int w = 0; w < LJ_BLOCK / 32; w++)
        for (unsigned b = s_full[w]; b != 0u; b &= b - 1u) {
            lj_cell<R>(A, u0 + 32 * w + __ffs(b) - 1);
            __syncthreads();  // the tables are free
        }
}

// ---------------------------------------------------------------- integrator

// v += (dt/2) F for every molecule (F = LJ + ATM in sorted order), then, if
// drift, x += dt v; kinetic energy per molecule (after the kick)
__global__ void __launch_bounds__(256) k_kick(Batch B, const int* __restrict__ perm,
                                              const double* __restrict__ f_lj,
                                              const double* __restrict__ f_atm,
                                              double* __restrict__ x, double* __restrict__ v,
                                              int drift, double* __restrict__ ke)
{
    after_previous();
    const long long n = B.ntot;
    long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (s >= n) return;
    int i = perm[s];
    const Rep& rp = B.rep[B.rep_of_mol[i]];
    const double dt = rp.dt, half_dt = 0.5 * rp.dt;
    double k = 0.0;
    for (int d = 0; d < 3; d++) {
        double f = __dadd_rn(f_lj[d * n + s], f_atm[d * n + s]);
        double vv = __dadd_rn(v[d * n + i], __dmul_rn(half_dt, f));
        v[d * n + i] = vv;
        if (drift) x[d * n + i] = __dadd_rn(x[d * n + i], __dmul_rn(dt, vv));
        if (!drift) k += 0.5 * vv * vv;
    }
    if (!drift) ke[i] = k;  // (the second half kick of the step gives the kinetic energy)
}

// the first half kick and the drift from a total force given in the
// original molecule order (a state restored with its forces)
__global__ void __launch_bounds__(256) k_kick_orig(Batch B, const double* __restrict__ f,
                                                   double* __restrict__ x, double* __restrict__ v,
                                                   double* __restrict__ ke)
{
    const long long n = B.ntot;
    long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const Rep& rp = B.rep[B.rep_of_mol[i]];
    const double dt = rp.dt, half_dt = 0.5 * rp.dt;
    double k = 0.0;
    for (int d = 0; d < 3; d++) {
        double vv = __dadd_rn(v[d * n + i], __dmul_rn(half_dt, f[d * n + i]));
        v[d * n + i] = vv;
        x[d * n + i] = __dadd_rn(x[d * n + i], __dmul_rn(dt, vv));
        k += 0.5 * vv * vv;
    }
    ke[i] = k;
}

// kinetic energy per molecule only (no update)
__global__ void __launch_bounds__(256) k_kinetic(long long n, const double* __restrict__ v,
                                                 double* __restrict__ ke)
{
    after_previous();
    long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= n) return;
    double k = 0.0;
    for (int d = 0; d < 3; d++) k += 0.5 * v[d * n + i] * v[d * n + i];
    ke[i] = k;
}

// velocity rescaling thermostat: every velocity of replica r times
// lambda_r = sqrt(T_r (3 N_r - 3) / (2 K_r)) (K_r from the last reduction;
// unchanged when K_r = 0 or N_r < 2), kinetic energies times lambda_r^2
__global__ void __launch_bounds__(256) k_rescale(Batch B, double* __restrict__ v,
                                                 double* __restrict__ ke,
                                                 const ResultDev* __restrict__ res,
                                                 const double* __restrict__ t_target)
{
    const long long n = B.ntot;
    long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int r = B.rep_of_mol[i];
    const double k = res[r].ekin, dof = 3.0 * (double)B.rep[r].n - 3.0;
    if (!(k > 0.0) || !(dof > 0.0)) return;
    const double l2 = t_target[r] * dof / (2.0 * k), l = sqrt(l2);
    for (int d = 0; d < 3; d++) v[d * n + i] *= l;
    ke[i] *= l2;
}

// finiteness check of a state copied from device memory
__global__ void k_check_finite(long long m, const double* __restrict__ a, int* __restrict__ status)
{
    after_previous();
    long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i < m && !isfinite(a[i])) atomicOr(status, ST_NONFINITE);
}

// density profile: histogram of one coordinate of the wrapped positions
__global__ void k_density(Batch B, const double* __restrict__ x, int axis, int nbins,
                          unsigned long long* __restrict__ counts)
{
    const long long n = B.ntot;
    long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int r = B.rep_of_mol[i];
    const double h = B.rep[r].g.L[axis] / (double)nbins;
    int b = (int)floor(x[axis * n + i] / h);
    b = b < 0 ? 0 : (b >= nbins ? nbins - 1 : b);
    atomicAdd(counts + (long long)r * nbins + b, 1ull);
}

// radial distribution: every pair once (forward half shell of the 27 cells,
// later molecules of the own cell) with r < r_max, binned by floor(r / dr) in
// FP64 on the canonical displacement; per-CTA shared histogram of the CTA's
// first replica (molecules of a second replica go straight to global memory).
//
// A warp per molecule, candidates across its lanes: an FP32 square leaves out
// those surely beyond r_max, and the others are queued and take the FP64 pipe 32 at
// a time (displacement, root and quotient, some 35 instructions).  With a thread per
// molecule every candidate of a warp took it, and 2,866 molecules filled 23 CTAs:
// 234 -> 25 us.
constexpr int RDF_WARPS = 16;
__global__ void __launch_bounds__(32 * RDF_WARPS) k_rdf(Batch B, const double* __restrict__ xl,
                                                        const float* __restrict__ xl32,
                                                        const int* __restrict__ start,
                                                        const int* __restrict__ cell_sorted, double rmax,
                                                        int nbins, long long per,
                                                        unsigned long long* __restrict__ counts)
{
    extern __shared__ unsigned hist[];
    __shared__ uint2 s_queue[RDF_WARPS][64];  // molecule (from s0) and slot << 27, partner
    typedef LjArith<double> Q;
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int k = threadIdx.x; k < nbins; k += blockDim.x) hist[k] = 0u;
    __syncthreads();
    const long long n = B.ntot;
    const long long s0 = blockIdx.x * per, s1 = s0 + per < n ? s0 + per : n;
    const int r0 = B.rep_of_cell[cell_sorted[s0]];
    const double dr = rmax / (double)nbins, rmax2 = rmax * rmax;
    uint2* queue = s_queue[warp];
    int qn = 0;
    auto evaluate = [&](uint2 e) {
        const long long s = s0 + (e.x & 0x7ffffffu), q = e.y;
        const int cg = cell_sorted[s], rep = B.rep_of_cell[cg];
        const Rep& rp = B.rep[rep];
        int dx, dy, dz;
        offset27(13 + (int)(e.x >> 27), dx, dy, dz);
        const double sx = Q::mul((double)dx, rp.g.w[0]), sy = Q::mul((double)dy, rp.g.w[1]),
                     sz = Q::mul((double)dz, rp.g.w[2]);
        const double ex = Q::add(Q::sub(xl[q], xl[s]), sx);
        const double ey = Q::add(Q::sub(xl[n + q], xl[n + s]), sy);
        const double ez = Q::add(Q::sub(xl[2 * n + q], xl[2 * n + s]), sz);
        const double r2 = Q::add(Q::add(Q::mul(ex, ex), Q::mul(ey, ey)), Q::mul(ez, ez));
        if (!(r2 < rmax2)) return;
        int b = (int)(sqrt(r2) / dr);
        b = b >= nbins ? nbins - 1 : b;
        if (rep == r0) atomicAdd(hist + b, 1u);
        else atomicAdd(counts + (long long)rep * nbins + b, 1ull);
    };
    for (long long s = s0 + warp; s < s1; s += RDF_WARPS) {
        const int cg = cell_sorted[s];
        const Rep& rp = B.rep[B.rep_of_cell[cg]];
        const int* st = start + rp.cell0;
        int cx, cy, cz;
        cell_coords(rp.g, cg - rp.cell0, cx, cy, cz);
        const float wx = rp.wf[0], wy = rp.wf[1], wz = rp.wf[2];
        // squares up to 12 w^2 from rounded coordinates: within 2^-18 of that (or of the
        // least FP32 numbers; zeros, infinities and NaN pass the test below)
        const float c_hi = (float)rmax2 * (1.0f + 0x1p-20f) + 0x1p-14f * (wx * wx + wy * wy + wz * wz) + 0x1p-144f;
        const float xs = xl32[s], ys = xl32[n + s], zs = xl32[2 * n + s];
        int dx = 0, dy = 0, dz = 0, q0 = 0, q1 = 0;
        if (lane < 14) {
            offset27(13 + lane, dx, dy, dz);
            const long long c = cell_at(rp.g, cx, cy, cz, dx, dy, dz);
            q0 = lane == 0 ? (int)s + 1 : st[c];
            q1 = st[c + 1];
        }
        for (int t = 0; t < 14; t++) {
            const int b = __shfl_sync(FULL, q0, t), e = __shfl_sync(FULL, q1, t);
            if (b >= e) continue;
            const float ox = (float)__shfl_sync(FULL, dx, t) * wx, oy = (float)__shfl_sync(FULL, dy, t) * wy,
                        oz = (float)__shfl_sync(FULL, dz, t) * wz;
            for (int k = b; k < e; k += 32) {
                const int q = k + lane;
                bool keep = false;
                if (q < e) {
                    const float ex = (xl32[q] - xs) + ox, ey = (xl32[n + q] - ys) + oy, ez = (xl32[2 * n + q] - zs) + oz;
                    keep = !(ex * ex + ey * ey + ez * ez > c_hi);
                }
                const unsigned m = __ballot_sync(FULL, keep);
                if (m == 0) continue;
                if (keep) queue[qn + __popc(m & ((1u << lane) - 1u))] = make_uint2((unsigned)(s - s0) | ((unsigned)t << 27), (unsigned)q);
                qn += __popc(m);
                __syncwarp();
                if (qn >= 32) {
                    evaluate(queue[lane]);
                    __syncwarp();
                    if (lane < qn - 32) queue[lane] = queue[32 + lane];
                    qn -= 32;
                    __syncwarp();
                }
            }
        }
    }
    if (lane < qn) evaluate(queue[lane]);
    __syncthreads();
    for (int k = threadIdx.x; k < nbins; k += blockDim.x)
        if (hist[k]) atomicAdd(counts + (long long)r0 * nbins + k, (unsigned long long)hist[k]);
}

// ---------------------------------------------------------------- reductions

// candidate triplets of the cell tasks of unit u (index inside its replica)
// and its half-shell candidate pairs
__device__ void cell_candidates(const Grid& g, const int* st, int trav, long long u,
                                unsigned long long& c3, unsigned long long& c2)
{
    int cx, cy, cz;
    cell_coords(g, u, cx, cy, cz);
    auto C2 = [](unsigned long long m) { return m < 2 ? 0ull : m * (m - 1) / 2; };
    auto C3 = [](unsigned long long m) { return m < 3 ? 0ull : m * (m - 1) * (m - 2) / 6; };
    unsigned long long N[8];           // 3c08's block, by slot
    unsigned long long before = 0, pairs = 0, one = 0, all = 0;  // 3c18: the forward cells so far
    const unsigned long long N0 = (unsigned long long)(st[u + 1] - st[u]);
#pragma unroll
    for (int t = 0; t < 27; t++) {
        const int dx = t % 3 - 1, dy = (t / 3) % 3 - 1, dz = t / 9 - 1;
        if (t < 13 && trav != 0) continue;
        const long long c = cell_at(g, cx, cy, cz, dx, dy, dz);
        const unsigned long long k = (unsigned long long)(st[c + 1] - st[c]);
        all += k;
        if (t > 13) {
            pairs += k * before;
            one += k * C2(N0) + N0 * C2(k);
            before += k;
        }
        if (dx >= 0 && dy >= 0 && dz >= 0) N[dx + 2 * dy + 4 * dz] = k;
    }
    c2 += C2(N0) + N0 * before;
    if (trav == 0) {
        c3 += all > 0 ? N0 * C2(all - 1) : 0ull;
    } else if (trav == 1) {
        c3 += C3(N0) + one + N0 * pairs;
    } else {
        c3 += C3(N0);
#pragma unroll
        for (int s = 0; s < 8; s++)
#pragma unroll
            for (int t = s + 1; t < 8; t++) {
                if ((s & t) == 0) c3 += N[t] * C2(N[s]) + N[s] * C2(N[t]);
#pragma unroll
                for (int v = t + 1; v < 8; v++)
                    if ((s & t & v) == 0) c3 += N[s] * N[t] * N[v];
            }
    }
}

// Two-level reduction in a fixed order (the same sums for the same partials).  Level 1: CTA
// (r, k) sums the k-th of REDUCE_PARTS equal slices of replica r's units and
// molecules (thread-strided, then a fixed tree).  Level 2: one warp per
// replica adds the REDUCE_PARTS partial sums in a fixed tree.  CAND: with the
// candidates of the cells (apart, for their registers).  With many replicas the FP64 pipe
// bounds it, 16 cycles a warp instruction: 240 replicas of 480 molecules 53 us (249 with
// a division in every thread and whole trees for slices of a few), 90 to 100 with CAND.
template <bool CAND>
__global__ void __launch_bounds__(256, CAND ? 4 : 5) k_partial_reduce(ReduceArgs R)
{
    after_previous();
    __shared__ double sd[5][256];
    __shared__ unsigned long long su[4][256];
    const int tid = threadIdx.x;
    const int r = blockIdx.x / REDUCE_PARTS, k = blockIdx.x % REDUCE_PARTS;
    const Rep& rp = R.b.rep[r];
    const long long nu = rp.g.ncell * R.split, uf = rp.cell0 * R.split;
    const long long cu = (nu + REDUCE_PARTS - 1) / REDUCE_PARTS;
    const long long cm = (rp.n + REDUCE_PARTS - 1) / REDUCE_PARTS;
    const long long u0 = uf + k * cu, u1 = min(uf + nu, u0 + cu);
    const long long m0 = rp.mol0 + k * cm, m1 = min(rp.mol0 + rp.n, m0 + cm);
    double e3 = 0, w3 = 0, e2 = 0, w2 = 0, ke = 0;
    unsigned long long c3 = 0, i3 = 0, c2 = 0, v2 = 0;
    for (long long q = u0 + tid; q < u1 && !R.mol_w3; q += 256) {
        e3 += R.unit_ew[2 * q];
        w3 += R.unit_ew[2 * q + 1];
        c3 += R.unit_cnt[2 * q];
        i3 += R.unit_cnt[2 * q + 1];
        if (R.unit_ew2) {
            e2 += R.unit_ew2[2 * q];
            w2 += R.unit_ew2[2 * q + 1];
            c2 += R.unit_cnt2[2 * q];
            v2 += R.unit_cnt2[2 * q + 1];
        }
    }
    if constexpr (CAND) {
        const long long cc = (rp.g.ncell + REDUCE_PARTS - 1) / REDUCE_PARTS;
        const long long l1 = min(rp.g.ncell, (k + 1) * cc);
        for (long long q = k * cc + tid; q < l1; q += 256)
            if (unit_owned(rp, q))
                cell_candidates(rp.g, R.cell_start + rp.cell0, R.cand_trav, q, c3, c2);
        if (!R.unit_ew2 && !R.mol_w3) c2 = 0;  // (counted with the molecules below)
    }
    for (long long q = m0 + tid; q < m1; q += 256) {
        if (!R.unit_ew2) {
            e2 += R.mol_ew[2 * q];
            w2 += R.mol_ew[2 * q + 1];
            c2 += R.mol_cnt[2 * q];
            v2 += R.mol_cnt[2 * q + 1];
        }
        if (R.mol_w3) {
            w3 += R.mol_w3[q];
            i3 += (unsigned long long)R.visits * R.mol_n3[q];
        }
        ke += R.ke[q];
    }
    sd[0][tid] = e2; sd[1][tid] = e3; sd[2][tid] = w2; sd[3][tid] = w3; sd[4][tid] = ke;
    su[0][tid] = c3; su[1][tid] = i3; su[2][tid] = c2; su[3][tid] = v2;
    __syncthreads();
    // a warp to a quantity: the tree over halves, quarters, .. of the 256 (in that
    // order; of slices of up to 32 the other threads have zeros)
    const bool few = max(cu, cm) <= 32;  // (and the cells: no more than units)
    const int lane = tid & 31;
    double* out = reinterpret_cast<double*>(R.part + blockIdx.x);  // e2, e3, w2, w3, ekin; the counts
    auto tree = [&](auto* v) {
        auto half = [&](int t) { return v[t] + v[t + 128]; };
        auto x = few ? v[lane] : (half(lane) + half(lane + 64)) + (half(lane + 32) + half(lane + 96));
        for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
        return x;
    };
    for (int q = tid >> 5; q < 9; q += 8) {
        if (q < 5) {
            const double x = tree(sd[q]);
            if (lane == 0) out[q] = x;
        } else {
            const unsigned long long x = tree(su[q - 5]);
            if (lane == 0) reinterpret_cast<unsigned long long*>(out)[q] = x;
        }
    }
}
static_assert(sizeof(ResultDev) == 72, "nine quantities in their order");

// one warp per replica: lane k holds partials k and k + 32 (added in that
// order), then a fixed shuffle tree; the order is the same for every launch
__global__ void __launch_bounds__(128) k_final_reduce(ReduceArgs R)
{
    after_previous();
    static_assert(REDUCE_PARTS == 64, "two partials per lane");
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int r = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (r >= R.b.R) return;  // whole warps leave together
    const ResultDev& a = R.part[r * REDUCE_PARTS + lane];
    const ResultDev& b = R.part[r * REDUCE_PARTS + 32 + lane];
    double e2 = a.e2 + b.e2, e3 = a.e3 + b.e3, w2 = a.w2 + b.w2, w3 = a.w3 + b.w3;
    double ek = a.ekin + b.ekin;
    unsigned long long c3 = a.n_cand3 + b.n_cand3, i3 = a.n_int3 + b.n_int3;
    unsigned long long c2 = a.n_cand2 + b.n_cand2, i2 = a.n_int2 + b.n_int2;
    for (int o = 16; o > 0; o >>= 1) {
        e2 += __shfl_down_sync(FULL, e2, o);
        e3 += __shfl_down_sync(FULL, e3, o);
        w2 += __shfl_down_sync(FULL, w2, o);
        w3 += __shfl_down_sync(FULL, w3, o);
        ek += __shfl_down_sync(FULL, ek, o);
        c3 += __shfl_down_sync(FULL, c3, o);
        i3 += __shfl_down_sync(FULL, i3, o);
        c2 += __shfl_down_sync(FULL, c2, o);
        i2 += __shfl_down_sync(FULL, i2, o);
    }
    if (lane == 0) {
        ResultDev t;
        t.e2 = e2;
        // u is homogeneous of degree -9 in the distances (divided here, once a replica:
        // beside the partial sums it took 1 us of an SM's FP64 pipe a CTA)
        t.e3 = R.mol_w3 ? w3 / 9.0 : e3;
        t.w2 = w2;
        t.w3 = w3;
        t.ekin = ek;
        t.n_cand3 = c3;
        t.n_int3 = i3;
        t.n_cand2 = c2;
        t.n_int2 = i2;
        R.out[r] = t;
    }
}

// gather sorted-order forces to the original order: which 0 total, 1 LJ, 2 ATM
__global__ void k_gather_forces(long long n, const int* __restrict__ perm,
                                const double* __restrict__ f_lj, const double* __restrict__ f_atm,
                                int which, double* __restrict__ out)
{
    after_previous();
    long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (s >= n) return;
    int i = perm[s];
    for (int d = 0; d < 3; d++) {
        double a = which == 2 ? 0.0 : f_lj[d * n + s];
        double b = which == 1 ? 0.0 : f_atm[d * n + s];
        out[d * n + i] = which == 0 ? __dadd_rn(a, b) : (which == 1 ? a : b);
    }
}

// the deterministic mode's force sums: 64-bit integers in units of 2^-bits,
// read and rewritten in place as doubles (the value is rounded once)
__global__ void k_fix_to_double(double* __restrict__ f, long long m, double scale)
{
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= m) return;
    const long long v = reinterpret_cast<const long long*>(f)[i];
    f[i] = (double)v * scale;
}

// ---------------------------------------------------------------- launchers

static inline unsigned nblk(long long m, int b) { return (unsigned)((m + b - 1) / b); }

cudaError_t launch_cell_counts(const Batch& b, double* x, int* cell_of, int* rank, int* count,
                               int* maxocc, int* status, bool wide, cudaStream_t st)
{
    const long long n = b.ntot;
    if (n > 0) {
        // (at least a thread for every maximum)
        launch_after(k_wrap_bin, nblk(n, MD_BLOCK), MD_BLOCK, 0, st, b, x, cell_of, rank, count, maxocc, status);
    } else {
        const cudaError_t e = cudaMemsetAsync(maxocc, 0, (1 + ATM_NUNIT) * sizeof(int), st);
        if (e != cudaSuccess) return e;
    }
    launch_after(k_unit_max, nblk(b.ncell, MD_BLOCK), MD_BLOCK, 0, st, b, count, wide ? 1 : 0, maxocc);
    return cudaGetLastError();
}

cudaError_t launch_cell_sort(const Batch& b, const double* x, const int* cell_of, const int* rank,
                             int* count, int* start, int* list, int* perm, double* xl, float* xl32,
                             int* cell_sorted, cudaStream_t st)
{
    const long long n = b.ntot;
    launch_after(k_scan, 1, 1024, 0, st, b.ncell, count, start);
    if (n > 0) {
        launch_after(k_scatter, nblk(n, MD_BLOCK), MD_BLOCK, 0, st, n, cell_of, rank, start, list);
        launch_after(k_cell_order, nblk(n, 128), 128, 0, st, b, x, cell_of, start, list, perm, xl, xl32, cell_sorted);
    }
    return cudaGetLastError();
}

cudaError_t launch_unit_classes(const Batch& b, const int* start, int trav, int ncls, int cut0,
                                int cut1, int* ulist, int* counts, cudaStream_t st)
{
    cudaError_t e = cudaMemsetAsync(counts, 0, ncls * sizeof(int), st);
    if (e != cudaSuccess || b.ncell <= 0) return e;
    k_unit_classes<<<nblk(b.ncell, MD_BLOCK), MD_BLOCK, 0, st>>>(b, start, trav, ncls, cut0, cut1,
                                                                  ulist, counts);
    return cudaGetLastError();
}

cudaError_t launch_lj(int prec, const LjArgs<double>& a64, const LjArgs<float>& a32,
                      cudaStream_t st)
{
    long long n = prec == 0 ? a64.n : a32.n;
    if (n <= 0) return cudaSuccess;
    const long long ncell = prec == 0 ? a64.b.ncell : a32.b.ncell;
    LjArgs<double> l64 = a64;
    LjArgs<float> l32 = a32;
    l64.per = l32.per = (int)std::max(1ll, std::min<long long>(LJ_BLOCK, ncell / n));
    const bool many = l64.per > 1;
    if (prec == 0)
        launch_after(many ? k_lj_owner<double, true> : k_lj_owner<double, false>, nblk(ncell, l64.per), LJ_BLOCK, 0,
                     st, l64);
    else
        launch_after(many ? k_lj_owner<float, true> : k_lj_owner<float, false>, nblk(ncell, l32.per), LJ_BLOCK, 0, st,
                     l32);
    return cudaGetLastError();
}

cudaError_t launch_kick(const Batch& b, const int* perm, const double* f_lj, const double* f_atm,
                        double* x, double* v, int drift, double* ke, cudaStream_t st)
{
    if (b.ntot <= 0) return cudaSuccess;
    launch_after(k_kick, nblk(b.ntot, MD_BLOCK), MD_BLOCK, 0, st, b, perm, f_lj, f_atm, x, v, drift, ke);
    return cudaGetLastError();
}

cudaError_t launch_kick_orig(const Batch& b, const double* f, double* x, double* v, double* ke,
                             cudaStream_t st)
{
    if (b.ntot <= 0) return cudaSuccess;
    k_kick_orig<<<nblk(b.ntot, MD_BLOCK), MD_BLOCK, 0, st>>>(b, f, x, v, ke);
    return cudaGetLastError();
}

cudaError_t launch_rescale(const Batch& b, double* v, double* ke, const ResultDev* res,
                           const double* t_target, cudaStream_t st)
{
    if (b.ntot <= 0) return cudaSuccess;
    k_rescale<<<nblk(b.ntot, MD_BLOCK), MD_BLOCK, 0, st>>>(b, v, ke, res, t_target);
    return cudaGetLastError();
}

cudaError_t launch_kinetic(long long n, const double* v, double* ke, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    launch_after(k_kinetic, nblk(n, MD_BLOCK), MD_BLOCK, 0, st, n, v, ke);
    return cudaGetLastError();
}

cudaError_t launch_check_finite(long long m, const double* a, int* status, cudaStream_t st)
{
    if (m <= 0) return cudaSuccess;
    launch_after(k_check_finite, nblk(m, MD_BLOCK), MD_BLOCK, 0, st, m, a, status);
    return cudaGetLastError();
}

cudaError_t launch_final_reduce(const ReduceArgs& r, cudaStream_t st)
{
    launch_after(r.cand_trav >= 0 ? k_partial_reduce<true> : k_partial_reduce<false>, (unsigned)(r.b.R * REDUCE_PARTS),
                 256, 0, st, r);
    launch_after(k_final_reduce, (unsigned)((r.b.R + 3) / 4), 128, 0, st, r);
    return cudaGetLastError();
}

cudaError_t launch_gather_forces(long long n, const int* perm, const double* f_lj,
                                 const double* f_atm, int which, double* out, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    launch_after(k_gather_forces, nblk(n, MD_BLOCK), MD_BLOCK, 0, st, n, perm, f_lj, f_atm, which, out);
    return cudaGetLastError();
}

cudaError_t launch_rdf(const Batch& b, const double* xl, const float* xl32, const int* start,
                       const int* cell_sorted, double rmax, int nbins, unsigned long long* counts, cudaStream_t st)
{
    if (b.ntot <= 0) return cudaSuccess;
    // a molecule a warp, more in CTAs beyond 4,096 (a histogram each)
    const long long per = std::max<long long>(RDF_WARPS, (b.ntot + 4095) / 4096);
    k_rdf<<<nblk(b.ntot, (int)per), 32 * RDF_WARPS, (size_t)nbins * sizeof(unsigned), st>>>(
        b, xl, xl32, start, cell_sorted, rmax, nbins, per, counts);
    return cudaGetLastError();
}

cudaError_t launch_density(const Batch& b, const double* x, int axis, int nbins,
                           unsigned long long* counts, cudaStream_t st)
{
    if (b.ntot <= 0) return cudaSuccess;
    k_density<<<nblk(b.ntot, MD_BLOCK), MD_BLOCK, 0, st>>>(b, x, axis, nbins, counts);
    return cudaGetLastError();
}

cudaError_t launch_fix_to_double(double* f, long long m, int bits, cudaStream_t st)
{
    if (m <= 0) return cudaSuccess;
    k_fix_to_double<<<nblk(m, MD_BLOCK), MD_BLOCK, 0, st>>>(f, m, 1.0 / (double)(1ull << bits));
    return cudaGetLastError();
}

}  // namespace atm3

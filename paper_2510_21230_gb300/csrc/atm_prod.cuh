// atm_prod.cuh -- the product rule of 3c01, 3c18, 3c08 and the corner-anchored 3c08
// in floating point (the deterministic mode and units that do not fit shared
// memory take the owner and block kernels).
//
// Units, staging order and triplets are those kernels' (atm_block.cuh p < q < r;
// 3c01: p a molecule of the base cell, q and r any two others).  Under the
// product rule a side may exceed r_c, so nearly every candidate has to be
// tested; 6 % of them interact in a liquid.
//
// A warp takes a molecule p.  Its rows are the molecules that may form triplets
// with it, positions relative to p: with d the least distance in the unit, two
// molecules at distances D >= D' from p have a third side of at least
// max(d, D - D'), so a product below r_c^3 needs D D' max(d, D - D') < r_c^3,
// hence D d max(d, D - d) < r_c^3.  The rows are sorted by distance (32 bins of
// its square).  Lane j holds a row r and the warp runs through the rows q before
// it, nearer to p, eight at a time and skipping eights whose distances leave no
// hit, two at a time in packed FP32: c = a + b - 2 q.r, a product and a compare, 6
// instructions a round; the results are a bit each in the lane's words.  (Lanes
// that hold the farther row have hits alike: the longest list of 32 lanes is 1.5
// to 1.8 of their mean; with rows in staging order, or lanes that hold the
// nearer row, it is 3 to 5.)  In a liquid 3c18 tests 24 % of its candidates.
//   FP32  3c01 and 3c18 evaluate the canonical displacements of the rows, as the owner
//         kernel does (unit-frame positions, rounded at 2 w, gave 3c01 up to 9 % more
//         rms force error and 3c18 up to 4 than the kernels before; 3c08 and 3c08a
//         are below those with them, and 7 % faster than with canonical rows).  A
//         lane evaluates its own hits, one a turn; nothing is
//         queued, r's force stays in registers and p's too (3c01: compensated),
//         q's goes to shared memory by three reductions.  A lane begins at its own
//         bit of a word, and eight copies of the forces take the lanes in turn,
//         for the far rows of a p share their few near ones (32,000 molecules,
//         3c18: 1.72 ms with one, 0.88 with four, 0.86 with eight).
//   FP64  an instruction takes the FP64 pipe as long for one lane as for 32, so
//         hits are queued, one a lane and turn, and evaluated 32 at a time; lanes
//         hold the nearer row there (hits of one batch meet fewer equal rows).
//         The pair scalars of 3c08 and 3c08a go to a dense table of the unit, and
//         one thread per molecule gathers F_m = sum_y G d(m -> y) at the end;
//         3c18, whose table would not fit, adds forces, and 3c01 keeps p's force
//         in registers.
// The warps' tables are sized by the unit's most rows, not by the largest unit's
// molecules: more warps fit.
//
// 32,000 molecules at density 0.8, 3c18, FP32: 0.86 ms (the block kernel: 3.69), issue
// 55 % and the shared-memory reductions 50 % busy; with rows in staging order and hits
// queued it took 2.1.  15,001 at 0.7, 3c08, FP64: 1.86 ms (3.36), bound by the FP64
// pipe, 69 instructions a triplet of which 43 are its arithmetic.  7,811, 3c01, FP64:
// 3.8 ms a call (12.2).  Units of up to 64 molecules run in CTAs of four warps (see
// atm_prod_plan).
//
// Decisions.  Squares from unit-frame positions are within 2.4e-4 (relative) of
// the canonical FP32 and FP64 ones for sides above 0.02 w, and c = a + b - 2 q.r
// adds 2^-21 (a + b): the scan keeps what is below r_c^6 (1 + 2^-10 + 2 D^6 2^-20
// / r_c^6), D the largest row.  (With a side below 0.02 w the product is below
// 0.06 w^6 <= 0.33 r_c^6: interacting either way.)  The evaluation has the
// product from the differences themselves: in FP32 one above r_c^6 (1 - 2^-10),
// in FP64 one within 2^-30 of r_c^6, is decided by the canonical sorted product.
//
// FP64: positions relative to the unit's frame come from the wrapped positions
// (x - x_0) -+ L, x_0 the base cell's corner: one rounding of values up to 2 w,
// three in the cell-local coordinates.  Bound by the FP64 pipe there, by
// instruction issue in FP32.
#pragma once
#include <type_traits>

#include "atm_block.cuh"

namespace atm3 {

// energy and the three pair scalars g_e = 2 du/d(r_e^2), over 3 nu, of a triplet
// with squared sides a, b and dot product m of the vectors of length a^(1/2),
// b^(1/2): x = a - m, y = b - m, c = x + y (see atm_fwd.cuh)
template <typename R>
__device__ __forceinline__ void prod_terms(R a, R b, R c, R x, R y, R m, R& u, R& ga, R& gb, R& gc)
{
    const R bc = b * c, ac = a * c, ab = a * b;
    R q;
    if constexpr (sizeof(R) == 8) q = ::rsqrt(a * bc);
    else q = rsqrtf(a * bc);
    const R q2 = q * q;
    const R xm = x * m, ym = y * m, xy = x * y;
    const R p = (xy * m) * q2;
    const R z = fma(R(5), p, R(1));
    const R q3 = q * q2, q5 = q3 * q2;
    u = q3 * fma(R(3), p, R(1));
    ga = q5 * fma(-z, bc, fma(a, y, -xm));
    gb = q5 * fma(-z, ac, fma(b, x, -ym));
    gc = q5 * fma(-z, ab, fma(c, m, -xy));
}

// packed pairs of FP32 numbers
__device__ __forceinline__ unsigned long long pk2(float lo, float hi)
{
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void upk2(unsigned long long v, float& lo, float& hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c)
{
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b)
{
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b)
{
    unsigned long long r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

template <int TRAV, typename R>
__device__ __forceinline__ void atm_prod_unit(const AtmArgs<R>& A, const long long u)
{
    constexpr int S = Trav<TRAV>::S;
    constexpr bool F64 = sizeof(R) == 8, OWNER = TRAV == 0;
    constexpr bool CANON = !F64 && (TRAV == 0 || TRAV == 1);  // evaluates canonical displacements
    constexpr bool TABLE = F64 && (TRAV == 2 || TRAV == 4);  // dense pair scalars
    constexpr unsigned FULL = 0xffffffffu;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_beg[S + 1];
    __shared__ int s_cell0[S];
    __shared__ signed char s_off[S][3];
    __shared__ float4 s_offf[CANON ? S : 1];
    __shared__ int s_next, s_dmin, s_rows, s_none;
    __shared__ double s_red[2][PROD_MAXW];
    __shared__ unsigned long long s_redn[PROD_MAXW];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
    const unsigned below = (1u << lane) - 1u;
    const int mcap = A.mcap;
    const Rep& rp = A.b.rep[A.b.rep_of_cell[u]];
    const long long lu = u - rp.cell0, n = A.n;
    auto store_zero = [&]() {
        if (tid == 0) {
            A.unit_ew[2 * u] = A.unit_ew[2 * u + 1] = 0.0;
            A.unit_cnt[2 * u] = A.unit_cnt[2 * u + 1] = 0ull;
        }
    };
    if (!unit_owned(rp, lu)) {
        store_zero();
        return;
    }
    if (warp == 0) unit_slots<TRAV, S>(rp.g, A.cell_start + rp.cell0, lu, s_beg, s_cell0, s_off);
    if (warp == 0) {
        __syncwarp();
        if (lane == 0) {
            s_next = 0;
            s_dmin = 0x7f000000;
            s_rows = 0;
            s_none = s_beg[S] < 3;
        }
    }
    __syncthreads();
    const int M = s_beg[S];
    const int Mp = TRAV == 2 ? M : s_beg[1];  // first molecules p of triplets
    if (M > mcap) {
        if (tid == 0) atomicOr(A.status, ST_CAPACITY);
        store_zero();
        return;
    }
    // no triplet, and no candidate (all of them hold a p); 3c08 is told by shared memory (the
    // test on M itself costs its FP32 kernel registers and 4 % of its time, and saves 3c18 2 %)
    if (TRAV == 2 ? s_none : M < 3 || Mp == 0) {
        store_zero();
        return;
    }
    const ProdSmem plan = prod_smem<R>(TRAV, M);
    float4* S4 = reinterpret_cast<float4*>(smem + plan.off_frame);  // unit-frame position, slot
    double* X = reinterpret_cast<double*>(smem + plan.off_x);       // FP64: unit-frame positions, SoA
    int* sidx = reinterpret_cast<int*>(smem + plan.off_idx);
    R* G = reinterpret_cast<R*>(smem + plan.off_acc);  // TABLE: pair scalars
    R* F = reinterpret_cast<R*>(smem + plan.off_acc);  // else: forces [(3 t + c) PROD_COPIES + copy]
    constexpr int NF = F64 ? 1 : PROD_COPIES;
    int cx, cy, cz;
    cell_coords(rp.g, lu, cx, cy, cz);
    const double r0 = (double)cx * rp.g.w[0], r1 = (double)cy * rp.g.w[1], r2 = (double)cz * rp.g.w[2];
    for (int s = warp; s < S; s += nwarps) {
        const int b = s_beg[s], e = s_beg[s + 1], g0 = s_cell0[s] - b;
        const int ox = s_off[s][0], oy = s_off[s][1], oz = s_off[s][2];
        if (CANON && lane == 0) s_offf[s] = make_float4((float)ox, (float)oy, (float)oz, 0.0f);
        // images of the cells beyond the box edges
        const double sx = cx + ox < 0 ? -rp.g.L[0] : (cx + ox >= rp.g.nc[0] ? rp.g.L[0] : 0.0);
        const double sy = cy + oy < 0 ? -rp.g.L[1] : (cy + oy >= rp.g.nc[1] ? rp.g.L[1] : 0.0);
        const double sz = cz + oz < 0 ? -rp.g.L[2] : (cz + oz >= rp.g.nc[2] ? rp.g.L[2] : 0.0);
        for (int t = b + lane; t < e; t += 32) {
            const int g = g0 + t;
            S4[t] = make_float4(A.xl32[g] + (float)ox * rp.wf[0], A.xl32[n + g] + (float)oy * rp.wf[1],
                                A.xl32[2 * n + g] + (float)oz * rp.wf[2], __int_as_float(s));
            sidx[t] = g;
            if constexpr (F64) {
                const long long o = A.perm[g];
                X[t] = (A.x[o] - r0) + sx;
                X[M + t] = (A.x[n + o] - r1) + sy;
                X[2 * M + t] = (A.x[2 * n + o] - r2) + sz;
            }
        }
    }
    if constexpr (!OWNER) {
        const int na = TABLE ? M * (M - 1) / 2 : 3 * NF * M;
        for (int t = tid; t < na; t += blockDim.x) G[t] = R(0);
    }
    __syncthreads();

    // ---- the least distance in the unit, and the farthest row it leaves
    {
        float d2 = 1e30f;
        for (int c0 = 0; c0 < M; c0 += 32) {
            const int q = min(c0 + lane, M - 1);
            const float4 Q = S4[q];
            for (int r = c0 + 1 + warp; r < M; r += nwarps) {
                const float4 V = S4[r];
                const float ex = V.x - Q.x, ey = V.y - Q.y, ez = V.z - Q.z;
                const float c = ex * ex + ey * ey + ez * ez;
                d2 = fminf(d2, r > q ? c : 1e30f);
            }
        }
        const int b = __reduce_min_sync(FULL, __float_as_int(d2));
        if (lane == 0) atomicMin(&s_dmin, b);
    }
    __syncthreads();
    const float rc6 = F64 ? (float)rp.rc6 : rp.rc6f;
    const float rc3 = sqrtf(rc6) * (1.0f + 0x1p-8f);
    float dmin = 0.0f;  // a lower bound of the distances of the unit
    float d_hi = 4.1f * (rp.wf[0] * rp.wf[0] + rp.wf[1] * rp.wf[1] + rp.wf[2] * rp.wf[2]);
    {
        // below by 2^-10 and the rounding of the positions, the product above by 2^-8
        const float d = sqrtf(__int_as_float(s_dmin)) * (1.0f - 0x1p-10f) - 0x1p-17f * (rp.wf[0] + rp.wf[1] + rp.wf[2]);
        if (d > 0.0f) {
            dmin = d;
            const float D = 0.5f * (d + sqrtf(d * d + 4.0f * rc3 / d));
            d_hi = fminf(d_hi, fmaxf(D * D, 4.0f * d * d) * (1.0f + 0x1p-10f));
        }
    }
    const float binf = 32.0f / d_hi, edge2 = d_hi * (1.0f / 32.0f);  // bins of squared distances
    const float t_hi = rc6 * (1.0f + 0x1p-10f) + 2.0f * d_hi * d_hi * d_hi * 0x1p-20f;
    // ---- the most rows of a p: the warps' tables, and how many warps have one
    // (p outermost: one ballot counts 32 rows)
    auto row_of = [&](const float4& P, int p, int t, float4& V, float& b) -> bool {
        V = S4[min(t, M - 1)];
        V.x = __fsub_rn(V.x, P.x);
        V.y = __fsub_rn(V.y, P.y);
        V.z = __fsub_rn(V.z, P.z);
        b = __fmaf_rn(V.z, V.z, __fmaf_rn(V.y, V.y, __fmul_rn(V.x, V.x)));
        return t < M && b < d_hi && (!OWNER || t != p);
    };
    {
        int most = 0;
        for (int p = warp; p < Mp; p += nwarps) {
            const float4 P = S4[p];
            int np = 0;
            for (int t0 = OWNER ? 0 : p + 1; t0 < M; t0 += 32) {
                float4 V;
                float b;
                np += __popc(__ballot_sync(FULL, row_of(P, p, t0 + lane, V, b)));
            }
            most = max(most, np);
        }
        if (lane == 0) atomicMax(&s_rows, most);
    }
    __syncthreads();
    const ProdWarpSmem wp = prod_warp_smem<R>(TRAV, s_rows);
    // (the launch has room for the tables of one warp with M rows, so >= 1)
    const int active = min(nwarps, (int)((A.gcap - plan.total) / wp.total));
    // the warp's rows: pairs (x0 x1 y0 y1) (z0 z1 b0 b1); again as (x y z, staged index),
    // FP32, or (x y z b), FP64; the eights' bounds; 3c08: the rows that complete an
    // anchored set with slots v, a word per 32 rows and v; the bins
    unsigned char* wb = smem + plan.total + (size_t)min(warp, active - 1) * wp.total;
    float* rows = reinterpret_cast<float*>(wb);
    float4* rows4 = reinterpret_cast<float4*>(wb + wp.rows);
    double2* rows64 = reinterpret_cast<double2*>(wb + wp.rows);
    float2* eights = reinterpret_cast<float2*>(wb + wp.eights);
    unsigned* anch = reinterpret_cast<unsigned*>(wb + wp.anch);
    unsigned* queue = reinterpret_cast<unsigned*>(wb + wp.queue);
    int* bins = reinterpret_cast<int*>(wb + wp.bins);
    unsigned short* rid = reinterpret_cast<unsigned short*>(wb + wp.rid);
    // the canonical decision of a triplet of staged molecules
    auto canonical = [&](int p, int q, int r) -> bool {
        const int sp = __float_as_int(S4[p].w), sq = __float_as_int(S4[q].w), sr = __float_as_int(S4[r].w);
        const long long gp = sidx[p], gq = sidx[q], gr = sidx[r];
        auto square = [&](long long g1, int s1, long long g2, int s2) -> R {
            R dx, dy, dz;
            const R w0 = F64 ? (R)rp.g.w[0] : (R)rp.wf[0], w1 = F64 ? (R)rp.g.w[1] : (R)rp.wf[1],
                    w2 = F64 ? (R)rp.g.w[2] : (R)rp.wf[2];
            return canon_disp<R>(A.xl[g1], A.xl[n + g1], A.xl[2 * n + g1], A.xl[g2], A.xl[n + g2],
                                 A.xl[2 * n + g2], s_off[s2][0] - s_off[s1][0], s_off[s2][1] - s_off[s1][1],
                                 s_off[s2][2] - s_off[s1][2], w0, w1, w2, dx, dy, dz);
        };
        const R rc6r = F64 ? (R)rp.rc6 : (R)rp.rc6f;
        return sorted_product<R>(square(gp, sp, gq, sq), square(gp, sp, gr, sr), square(gq, sq, gr, sr)) < rc6r;
    };

    const R nu3 = R(3) * (F64 ? (R)rp.nu : (R)rp.nuf);
    Sum<R> esum;
    unsigned nint = 0;
    R fpx, fpy, fpz;  // force on p: the lane's share
    Sum<float> fox, foy, foz;  // the same of 3c01 in FP32, compensated
    int qn = 0;
    R* Fl = F + (lane & (NF - 1));  // the lane's copy of the forces
    // FP64: one queued hit, two rows of p, per lane
    auto evaluate64 = [&](int p, unsigned e) {
        if constexpr (F64) {
            const int j = (int)(e & 0xffffu), k = (int)(e >> 16), q = rid[j], r = rid[k];
            const double2 Q0 = rows64[2 * j], Q1 = rows64[2 * j + 1], V0 = rows64[2 * k], V1 = rows64[2 * k + 1];
            const double qx = Q0.x, qy = Q0.y, qz = Q1.x, a = Q1.y;
            const double rx = V0.x, ry = V0.y, rz = V1.x, b = V1.y;
            // (the third side from the difference of the rows: a + b - 2 q.r would lose the
            // digits of a side short against the others, of which this rule has many)
            const double ex = rx - qx, ey = ry - qy, ez = rz - qz, c = ex * ex + ey * ey + ez * ez;
            const double x = -(qx * ex + qy * ey + qz * ez), y = c - x, m = a - x;
            const double abc = a * (b * c);
            if (abc > rp.rc6 * (1.0 - 0x1p-30)) {
                if (abc > rp.rc6 * (1.0 + 0x1p-30)) return;
                if (!canonical(p, min(q, r), max(q, r))) return;
            }
            nint++;
            double uu, ga, gb, gc;
            prod_terms<double>(a, b, c, x, y, m, uu, ga, gb, gc);
            esum.add(uu);
            if constexpr (TABLE) {
                atomicAdd(G + tri_index(p, q), ga);
                atomicAdd(G + tri_index(p, r), gb);
                atomicAdd(G + (q < r ? tri_index(q, r) : tri_index(r, q)), gc);
            } else {
                fpx = fma(ga, qx, fma(gb, rx, fpx));
                fpy = fma(ga, qy, fma(gb, ry, fpy));
                fpz = fma(ga, qz, fma(gb, rz, fpz));
                if constexpr (!OWNER) {
                    const double gx = gc * ex, gy = gc * ey, gz = gc * ez;
                    atomicAdd(F + 3 * q, fma(-ga, qx, gx));
                    atomicAdd(F + 3 * q + 1, fma(-ga, qy, gy));
                    atomicAdd(F + 3 * q + 2, fma(-ga, qz, gz));
                    atomicAdd(F + 3 * r, -fma(gb, rx, gx));
                    atomicAdd(F + 3 * r + 1, -fma(gb, ry, gy));
                    atomicAdd(F + 3 * r + 2, -fma(gb, rz, gz));
                }
            }
        }
    };

    while (warp < active) {
        int p = 0;
        if (lane == 0) p = atomicAdd(&s_next, 1);
        p = __shfl_sync(FULL, p, 0);
        if (p >= Mp) break;
        const float4 P = S4[p];
        if (TRAV == 2 && __float_as_int(P.w) == 7) break;  // no later slot completes an anchored set
        // ---- the rows of p: their number in each bin, then their places (the
        // arithmetic of the two passes is spelt out: they must agree)
        R px = R(0), py = R(0), pz = R(0);
        if constexpr (F64) {
            px = X[p];
            py = X[M + p];
            pz = X[2 * M + p];
        }
        float lx = 0.0f, ly = 0.0f, lz = 0.0f;  // CANON: p lies in the base cell
        if constexpr (CANON) {
            const float* xp = A.xl + sidx[p];
            lx = xp[0];
            ly = xp[n];
            lz = xp[2 * n];
        }
        const int first = OWNER ? 0 : p + 1;
        bins[lane] = 0;
        __syncwarp();
        for (int t0 = first; t0 < M; t0 += 32) {
            float4 V;
            float b;
            if (row_of(P, p, t0 + lane, V, b)) atomicAdd(bins + min((int)(b * binf), 31), 1);
        }
        __syncwarp();
        int np = bins[lane];
        const int mine = np;
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(FULL, np, o);
            if (lane >= o) np += v;
        }
        bins[lane] = np - mine;
        np = __shfl_sync(FULL, np, 31);
        __syncwarp();
        for (int t0 = first; t0 < M; t0 += 32) {
            const int t = t0 + lane;
            float4 V;
            float b;
            if (row_of(P, p, t, V, b)) {
                const int k = atomicAdd(bins + min((int)(b * binf), 31), 1);
                float* to = rows + 8 * (k >> 1) + (k & 1);
                to[0] = V.x;
                to[2] = V.y;
                to[4] = V.z;
                to[6] = b;
                if constexpr (CANON) {
                    const float* xg = A.xl + sidx[t];
                    const float4 o = s_offf[__float_as_int(V.w)];
                    rows4[k] = make_float4(__fadd_rn(__fsub_rn(xg[0], lx), __fmul_rn(o.x, rp.wf[0])),
                                           __fadd_rn(__fsub_rn(xg[n], ly), __fmul_rn(o.y, rp.wf[1])),
                                           __fadd_rn(__fsub_rn(xg[2 * n], lz), __fmul_rn(o.z, rp.wf[2])),
                                           __int_as_float(t));
                } else if constexpr (!F64) {
                    rows4[k] = make_float4(V.x, V.y, V.z, __int_as_float(t));
                } else {
                    rid[k] = (unsigned short)t;
                }
                if constexpr (F64) {
                    const double dx = X[t] - px, dy = X[M + t] - py, dz = X[2 * M + t] - pz;
                    rows64[2 * k] = make_double2(dx, dy);
                    rows64[2 * k + 1] = make_double2(dz, dx * dx + dy * dy + dz * dz);
                }
            }
        }
        __syncwarp();
        // the edges of the bins of an eight's first and last row
        for (int g = lane; 8 * g < np; g += 32) {
            const int k1 = min(8 * g + 7, np - 1);
            const float b0 = rows[32 * g + 6], b1 = rows[8 * (k1 >> 1) + (k1 & 1) + 6];
            eights[g] = make_float2(fmaxf(dmin, sqrtf((float)min((int)(b0 * binf), 31) * edge2) * (1.0f - 0x1p-16f)),
                                    sqrtf((float)(min((int)(b1 * binf), 31) + 1) * edge2) * (1.0f + 0x1p-16f));
        }
        auto staged = [&](int k) -> int { return F64 ? (int)rid[k] : __float_as_int(rows4[k].w); };
        if constexpr (TRAV == 2) {
            for (int k0 = 0; k0 < np; k0 += 32) {
                const int s = k0 + lane < np ? __float_as_int(S4[staged(k0 + lane)].w) : 8;
                unsigned all = 0;
#pragma unroll
                for (int v = 0; v < 8; v++) {
                    const unsigned m = __ballot_sync(FULL, s < 8 && (s & v) == 0);
                    if (lane == v) all = m;
                }
                if (lane < 8) anch[(k0 >> 2) + lane] = all;
            }
        }
        __syncwarp();
        fpx = fpy = fpz = R(0);
        fox = foy = foz = Sum<float>();
        // ---- 32 rows, a row per lane: FP32 with the rows before, FP64 with those after
        for (int r0 = 0; r0 < np; r0 += 32) {
            const int r = r0 + lane;
            const bool own = r < np;
            float Vx = 0.0f, Vy = 0.0f, Vz = 0.0f, b = 0.0f;
            int ri = p, v = 0;
            if (own) {
                if constexpr (!CANON) {
                    const float* vr = rows + 8 * (r >> 1) + (r & 1);
                    Vx = vr[0];
                    Vy = vr[2];
                    Vz = vr[4];
                    b = vr[6];
                } else {
                    const float4 V = rows4[r];
                    Vx = V.x;
                    Vy = V.y;
                    Vz = V.z;
                    b = Vx * Vx + Vy * Vy + Vz * Vz;
                }
                ri = staged(r);
            }
            if constexpr (TRAV == 2) v = __float_as_int(P.w) & __float_as_int(S4[ri].w);
            const unsigned long long vx2 = pk2(-2.0f * Vx, -2.0f * Vx), vy2 = pk2(-2.0f * Vy, -2.0f * Vy),
                                     vz2 = pk2(-2.0f * Vz, -2.0f * Vz), b2 = pk2(b, b);
            const float rl = eights[r0 >> 3].x, rh = eights[min(r0 + 31, np - 1) >> 3].y, lim = rc3 / rl;
            // the lane's hits among rows q0 .. q0 + 31, rotated to the lane's own bit
            auto scan = [&](int q0) -> unsigned {
                unsigned hit = 0;
                const ulonglong2* qq = reinterpret_cast<const ulonglong2*>(rows + 4 * q0);
#pragma unroll
                for (int h = 0; h < 4; h++) {
                    if (q0 + 8 * h >= np) break;
                    const float2 g = eights[(q0 >> 3) + h];
                    if (g.x * fmaxf(dmin, F64 ? g.x - rh : rl - g.y) >= lim) continue;
#pragma unroll
                    for (int i = 4 * h; i < 4 * h + 4; i++) {
                        const ulonglong2 xy = qq[2 * i], zb = qq[2 * i + 1];
                        unsigned long long c = add2(zb.y, b2);
                        c = fma2(zb.x, vz2, c);
                        c = fma2(xy.y, vy2, c);
                        c = fma2(xy.x, vx2, c);
                        float lo, hi;
                        upk2(mul2(mul2(zb.y, b2), c), lo, hi);
                        if (lo < t_hi) hit |= 1u << (2 * i);
                        if (hi < t_hi) hit |= 2u << (2 * i);
                    }
                }
                if (q0 == r0) hit &= F64 ? ~(below << 1 | 1u) : below;
                if (F64 && np - q0 < 32) hit &= (1u << (np - q0)) - 1u;
                if (!own) hit = 0;
                if constexpr (TRAV == 2) hit &= anch[(q0 >> 2) + v];
                return __funnelshift_r(hit, hit, lane);
            };
            if constexpr (F64) {
                for (int q0 = r0; q0 < np; q0 += 32) {
                    unsigned hit = scan(q0);
                    for (;;) {
                        const unsigned m = __ballot_sync(FULL, hit != 0);
                        if (m == 0) break;
                        if (hit) {
                            const unsigned q = (unsigned)(q0 + ((__ffs(hit) - 1 + lane) & 31));
                            queue[qn + __popc(m & below)] = (unsigned)r | (q << 16);
                            hit &= hit - 1;
                        }
                        qn += __popc(m);
                        __syncwarp();
                        if (qn >= 32) {
                            evaluate64(p, queue[lane]);
                            __syncwarp();
                            if (lane < qn - 32) queue[lane] = queue[32 + lane];
                            qn -= 32;
                            __syncwarp();
                        }
                    }
                }
            } else {
                float gr = 0.0f, frx = 0.0f, fry = 0.0f, frz = 0.0f;
                for (int qb = 0; qb <= r0; qb += 128) {
                    unsigned h0 = 0, h1 = 0, h2 = 0, h3 = 0;
                    for (int k = 3; k >= 0; k--) {
                        h3 = h2;
                        h2 = h1;
                        h1 = h0;
                        h0 = qb + 32 * k <= r0 ? scan(qb + 32 * k) : 0u;
                    }
                    int base = qb;
                    // (one hit a lane and turn, the warp together)
                    while (__any_sync(FULL, (h0 | h1 | h2 | h3) != 0)) {
                        if (h0 == 0) {
                            h0 = h1;
                            h1 = h2;
                            h2 = h3;
                            h3 = 0;
                            base += 32;
                        }
                        bool act = h0 != 0;
                        const int q = act ? base + ((__ffs(h0) - 1 + lane) & 31) : 0;
                        h0 &= h0 - 1;
                        const float4 Q = rows4[q];
                        const int qi = __float_as_int(Q.w);
                        const float a = Q.x * Q.x + Q.y * Q.y + Q.z * Q.z;
                        const float ex = Vx - Q.x, ey = Vy - Q.y, ez = Vz - Q.z;
                        const float c = ex * ex + ey * ey + ez * ez;
                        const float t = fmaf(0.5f, b, 0.5f * a), w = fmaf(0.5f, b, -0.5f * a);
                        if (act && a * (b * c) >= rc6 * (1.0f - 0x1p-10f)) act = canonical(p, min(qi, ri), max(qi, ri));
                        __syncwarp();
                        if (act) {
                            nint++;
                            float uu, ga, gb, gc;
                            prod_terms<float>(a, b, c, fmaf(0.5f, c, -w), fmaf(0.5f, c, w), fmaf(-0.5f, c, t), uu, ga,
                                              gb, gc);
                            esum.add(uu);
                            if constexpr (OWNER) {
                                fox.add(fmaf(ga, Q.x, gb * Vx));
                                foy.add(fmaf(ga, Q.y, gb * Vy));
                                foz.add(fmaf(ga, Q.z, gb * Vz));
                            } else {
                                gr += gb;
                                fpx = fmaf(ga, Q.x, fpx);
                                fpy = fmaf(ga, Q.y, fpy);
                                fpz = fmaf(ga, Q.z, fpz);
                                const float gx = gc * ex, gy = gc * ey, gz = gc * ez;
                                frx += gx;
                                fry += gy;
                                frz += gz;
                                atomicAdd(Fl + 3 * NF * qi, fmaf(-ga, Q.x, gx));
                                atomicAdd(Fl + 3 * NF * qi + NF, fmaf(-ga, Q.y, gy));
                                atomicAdd(Fl + 3 * NF * qi + 2 * NF, fmaf(-ga, Q.z, gz));
                            }
                        }
                        __syncwarp();
                    }
                }
                if (own && !OWNER) {
                    fpx = fmaf(gr, Vx, fpx);
                    fpy = fmaf(gr, Vy, fpy);
                    fpz = fmaf(gr, Vz, fpz);
                    atomicAdd(Fl + 3 * NF * ri, -fmaf(gr, Vx, frx));
                    atomicAdd(Fl + 3 * NF * ri + NF, -fmaf(gr, Vy, fry));
                    atomicAdd(Fl + 3 * NF * ri + 2 * NF, -fmaf(gr, Vz, frz));
                }
            }
        }
        if constexpr (F64) {
            if (lane < qn) evaluate64(p, queue[lane]);
            qn = 0;
        }
        if constexpr (!TABLE) {
            using W = std::conditional_t<OWNER, double, R>;
            W f0 = fpx, f1 = fpy, f2 = fpz;
            if constexpr (OWNER && !F64) {
                f0 = fox.get();
                f1 = foy.get();
                f2 = foz.get();
            }
            for (int o = 16; o > 0; o >>= 1) {
                f0 += __shfl_down_sync(FULL, f0, o);
                f1 += __shfl_down_sync(FULL, f1, o);
                f2 += __shfl_down_sync(FULL, f2, o);
            }
            if (lane == 0) {
                if constexpr (OWNER) {
                    double* to = A.fs + sidx[p];
                    to[0] = (double)nu3 * f0;
                    to[n] = (double)nu3 * f1;
                    to[2 * n] = (double)nu3 * f2;
                } else {
                    atomicAdd(F + 3 * NF * p, f0);
                    atomicAdd(F + 3 * NF * p + NF, f1);
                    atomicAdd(F + 3 * NF * p + 2 * NF, f2);
                }
            }
        }
        __syncwarp();  // the rows and the queue are free
    }
    __syncthreads();

    if constexpr (!OWNER) {
        for (int m = tid; m < M; m += blockDim.x) {
            R fx = R(0), fy = R(0), fz = R(0);
            if constexpr (TABLE) {
                // F_m = 3 nu sum over the other molecules y of G d(m -> y)
                const R px = X[m], py = X[M + m], pz = X[2 * M + m];
                const int low = m * (m - 1) / 2;
                for (int y = 0; y < M; y++) {
                    const R g = G[y < m ? low + y : (y > m ? tri_index(m, y) : 0)];
                    if (g == R(0) || y == m) continue;
                    fx = fma(g, X[y] - px, fx);
                    fy = fma(g, X[M + y] - py, fy);
                    fz = fma(g, X[2 * M + y] - pz, fz);
                }
            } else {
                for (int c = 0; c < NF; c++) {
                    fx += F[3 * NF * m + c];
                    fy += F[3 * NF * m + NF + c];
                    fz += F[3 * NF * m + 2 * NF + c];
                }
            }
            double* to = A.fs + sidx[m];
            if (fx != R(0)) atomicAdd(to, (double)(nu3 * fx));
            if (fy != R(0)) atomicAdd(to + n, (double)(nu3 * fy));
            if (fz != R(0)) atomicAdd(to + 2 * n, (double)(nu3 * fz));
        }
    }
    const double nu = F64 ? rp.nu : (double)rp.nuf;
    const double e3 = nu * esum.get();
    unsigned long long cand = 0;
    if constexpr (OWNER) cand = unit_candidates<TRAV, S>(s_beg);
    else if (warp == 0) cand = unit_candidates_warp<TRAV, S>(s_beg);
    // 3c01 finds a triangle from each owner that sees it
    unit_reduce_store<PROD_MAXW>(e3, 9.0 * e3, (unsigned long long)nint, OWNER ? 1.0 / 3.0 : 1.0, cand, A.unit_ew,
                                 A.unit_cnt, u, s_red, s_redn);
}

template <int TRAV, typename R>
__global__ void __launch_bounds__(32 * PROD_MAXW) __maxnreg__(sizeof(R) == 8 ? 96 : 64)
    k_atm_prod(const AtmArgs<R> A)
{
    after_previous();
    atm_prod_unit<TRAV, R>(A, blockIdx.x);
}

}  // namespace atm3

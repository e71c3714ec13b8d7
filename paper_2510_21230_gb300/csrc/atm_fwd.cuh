// atm_fwd.cuh -- the FP32C pair rule from forward lists.
//
// Under the pair rule every traversal over adjacent cells (3c01, 3c18, 3c08)
// finds the same triangles, all sides below r_c, so they are enumerated once,
// at their lowest molecule: within a cell layer molecules are ordered by
// (z, sorted index) and a layer lies below the next one, so the other two
// molecules of a triangle are in the forward list of its lowest one, i -- the
// partners within r_c that lie above it, in i's cell layer or the next (18
// cells).  (No triangle can wind around three layers: its sides would add up
// to less than 3 r_c <= L_z.)  Lists cut by height instead of by half-shell
// cells have nearly one length, 26 +- 3 in a rho* = 0.8 liquid against 26 +- 9,
// and the triangle work goes with its square: 12.7 rounds per molecule
// against 17.5.
//
// One warp takes one molecule i.
//  1. The staged molecules are tested in 32s on unit-frame positions xl + o w,
//     the indices of those within r_c and above i compacted, and the list's
//     rows (canonical displacement d, |d|^2) formed from them.  A square from
//     unit-frame positions is within 1.6e-6 r_c^2 of the canonical one; in a
//     band of 2^-16 around r_c^2, and for equal heights, the canonical form
//     decides, as in the block kernels.
//  2. Lane j keeps row j; in round s = 1 .. n/2 it takes the pair
//     (j, j + s mod n), so every pair of the list is met once with the lanes
//     evenly loaded, and no queue, search or atomic stands between the test
//     and the evaluation: with 61 % of the pairs interacting, evaluating the
//     masked rest costs less than compacting them (the edge-centric block
//     kernel spends 37 % of its time on expanding edges into triangles and
//     4 % on its atomics).  Row k's share of a pair goes to lane k by two shuffles:
//     with g_e = 2 du/d(r_e^2) the force on j is
//         V_j - G_ij d_j,   V_j = sum_k g_jk (d_k - d_j),
//     and that on i is sum_j G_ij d_j; all of it stays in registers.  (V_j as
//     sum_k g_jk d_k - d_j sum_k g_jk is an operation less a pair, but cancels
//     where j and k are close: rms force error of the arithmetic 2.9e-7 against 2.7e-7.)
//     3c01 compensates these sums, as the owner kernel does (2.6e-7): 32,000
//     molecules 111 -> 126 us, 438 in the owner kernel.
//     The third side comes from the rows, |d_k - d_j|^2: within 2.2e-6
//     (relative to r_c^2) of the canonical square (five FP32 roundings of
//     values up to 4/3 r_c per component, in both), so outside a band of
//     2^-16 around r_c^2 it decides as the canonical form does; in the band
//     the canonical form decides.  (The rows are stored twice over, so row
//     j + s needs no wrapped index.)
//  3. A few rows beyond 32 are each met with all lanes' rows, their sums
//     reduced over the warp; longer lists are cut into equal chunks: each chunk
//     with itself as above and with every later one by rotation.
// A CTA takes a run of base cells along x and stages the columns around it
// (three cells of the layer and three of the next per column), so the 18
// cells of every base cell are one contiguous range and staging, latency and
// the unit's sums are paid once for up to four cells.
// The LJ term of the pair (i, j) is evaluated on the list row (the canonical
// displacement), so every pair of the system is met once here too.
// A row's force goes to the FP64 array (fixed point in the deterministic mode)
// by one reduction per component when its list is done: 21 M of them for
// 256,000 molecules, which the L2 takes at over 400 G/s beside the arithmetic.
// Each triangle's energy is added with compensation (a plain sum of a list: steps of
// 256,000 molecules 3 % faster); the virial is 9 times the energy (u is homogeneous of
// degree -9 in the distances).
//
// Bound by instruction issue (72 % of the issue slots on 32,000 molecules, LJ apart:
// 70 M warp instructions, 2.0 MB from DRAM, 0.090 ms; the block kernel 140 M).  256,000
// molecules, rho* = 0.8, in a step (LJ inside): 0.47 ms against 1.16 ms of bitmaps and
// block kernel; by leaving phases out, rounds are six tenths of it, lists 0.07 ms, the
// rows' shares and LJ 0.10, staging and sums of the unit 0.04 (0.10 with one base cell
// per CTA; lists of 33 in two chunks instead of 32 and 1: + 0.07).
#pragma once
#include <type_traits>

#include "atm_common.cuh"

namespace atm3 {

// 1 / sqrt(s) to 2 ulp (s of a triangle: normal range wherever the force is finite)
__device__ __forceinline__ float fwd_rsq(float s)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(s));
    return y;
}

// v in FP64 by integer operations (the conversion instruction runs at the FP64
// pipe's rate, 1/64 of theirs)
__device__ __forceinline__ double fwd_widen(float v)
{
    const unsigned u = __float_as_uint(v), e = u & 0x7f800000u;
    const unsigned bias = e == 0x7f800000u ? 0x70000000u : 0x38000000u;  // not finite: stays so
    const unsigned hi = (u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + bias);
    return e == 0u ? 0.0 : __hiloint2double((int)hi, (int)(u << 29));  // (below 1e-38: zero)
}

// the sum of two float pairs (value s + r, |r| a few ulp of s): error-free
// addition of the values, the rests added
__device__ __forceinline__ void fwd_add_pair(float& s, float& r, float s2, float r2)
{
    const float t = __fadd_rn(s, s2), b = __fsub_rn(t, s);
    const float e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(s2, b));
    r = __fadd_rn(__fadd_rn(r, r2), e);
    s = t;
}

// x, y, z and w summed over the warp: lane 8 d of the result holds component d
__device__ __forceinline__ float fwd_sum4(float x, float y, float z, float w, int lane)
{
    const unsigned FULL = 0xffffffffu;
    const bool b4 = lane & 16, b3 = lane & 8;
    float k0 = b4 ? z : x, k1 = b4 ? w : y;
    k0 += __shfl_xor_sync(FULL, b4 ? x : z, 16);
    k1 += __shfl_xor_sync(FULL, b4 ? y : w, 16);
    float k = b3 ? k1 : k0;
    k += __shfl_xor_sync(FULL, b3 ? k0 : k1, 8);
    for (int o = 4; o > 0; o >>= 1) k += __shfl_xor_sync(FULL, k, o);
    return k;
}

// the same in float pairs
__device__ __forceinline__ float fwd_sum4_pair(float x, float y, float z, float w, int lane)
{
    const unsigned FULL = 0xffffffffu;
    const bool b4 = lane & 16, b3 = lane & 8;
    float k0 = b4 ? z : x, k1 = b4 ? w : y, r0 = 0.0f, r1 = 0.0f;
    fwd_add_pair(k0, r0, __shfl_xor_sync(FULL, b4 ? x : z, 16), 0.0f);
    fwd_add_pair(k1, r1, __shfl_xor_sync(FULL, b4 ? y : w, 16), 0.0f);
    float k = b3 ? k1 : k0, r = b3 ? r1 : r0;
    const float s2 = __shfl_xor_sync(FULL, b3 ? k0 : k1, 8), t2 = __shfl_xor_sync(FULL, b3 ? r0 : r1, 8);
    fwd_add_pair(k, r, s2, t2);
    for (int o = 4; o > 0; o >>= 1) {
        const float s = __shfl_xor_sync(FULL, k, o), t = __shfl_xor_sync(FULL, r, o);
        fwd_add_pair(k, r, s, t);
    }
    return k + r;
}

// sums of a list row: plain FP32, or (COMP) compensated
template <bool COMP>
struct FwdSum {
    float s = 0.f;
    __device__ __forceinline__ void fma(float a, float b) { s = fmaf(a, b, s); }
    __device__ __forceinline__ void add(float v) { s += v; }
    __device__ __forceinline__ float get() const { return s; }
};
template <>
struct FwdSum<true> {
    Sum<float> k;
    __device__ __forceinline__ void fma(float a, float b) { k.add(__fmul_rn(a, b)); }
    __device__ __forceinline__ void add(float v) { k.add(v); }
    __device__ __forceinline__ float get() const { return __fsub_rn(k.s, k.c); }
};

template <int LJ, bool DET, bool COMP>
__device__ __forceinline__ void atm_fwd_unit(const FwdArgs& A, const int u, const int part)
{
    constexpr unsigned FULL = 0xffffffffu;
    typedef Ar<float> Q;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_beg[FWD_CELLS + 1];
    __shared__ int s_cell0[FWD_CELLS];
    __shared__ float4 s_off[FWD_CELLS];   // cell offset from the run's first base cell
    __shared__ int s_base[FWD_RUN + 1];   // molecules of the run's base cells before each
    __shared__ int s_next, s_over;
    __shared__ unsigned long long s_cnt[2][FWD_MAXW];

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nwarps = blockDim.x >> 5;
    const int stage = fwd_stage(A.mcap, A.run);
    const FwdSmem plan = fwd_smem_plan(A.mcap, A.run, nwarps);
    const Rep& rp = A.b.rep[A.b.rep_of_cell[u]];
    const int lu = u - (int)rp.cell0;
    const long long n = A.n;
    float4* P4 = reinterpret_cast<float4*>(smem + plan.off_pos);    // xl, staged cell
    float4* S4 = reinterpret_cast<float4*>(smem + plan.off_frame);  // xl + o w, sorted index
    float4* list = reinterpret_cast<float4*>(smem + plan.off_list) + warp * FWD_ROWS;
    unsigned short* lidx =
        reinterpret_cast<unsigned short*>(smem + plan.off_lidx) + (size_t)warp * plan.icap;

    const int nx = rp.g.nc[0], ny = rp.g.nc[1], nz = rp.g.nc[2];
    const int cx = lu % nx, cy = (lu / nx) % ny, cz = lu / (nx * ny);
    const int len = min(A.run, nx - cx), ncell = 6 * (len + 2);  // base cells, staged cells
    // the partial sums of this CTA, at the run's first cell; none at the others
    const long long slot_out = (long long)u * A.split + part;
    auto store_zero = [&](int from) {
        for (int r = from + tid; r < len; r += blockDim.x) {
            const long long o = 2 * (slot_out + r);
            A.unit_ew[o] = A.unit_ew[o + 1] = 0.0;
            A.unit_cnt[o] = A.unit_cnt[o + 1] = 0ull;
            if (LJ) {
                A.unit_ew2[o] = A.unit_ew2[o + 1] = 0.0;
                A.unit_cnt2[o] = A.unit_cnt2[o + 1] = 0ull;
            }
        }
    };
    if (cz < rp.own_z0 || cz >= rp.own_z1) {  // another domain's units
        store_zero(0);
        return;
    }
    const float wf0 = rp.wf[0], wf1 = rp.wf[1], wf2 = rp.wf[2];
    if (warp == 0) {
        int run = 0;
        for (int s0 = 0; s0 < ncell; s0 += 32) {
            const int s = s0 + lane;
            int cnt = 0;
            if (s < ncell) {
                // column s / 6 (x = cx - 1 ..), then the three cells of this layer and
                // the three of the next
                const int col = s / 6, q = s - 6 * col;
                const int dx = col - 1, dy = (q < 3 ? q : q - 3) - 1, dz = q < 3 ? 0 : 1;
                int x = cx + dx, y = cy + dy, z = cz + dz;
                x = x < 0 ? x + nx : (x >= nx ? x - nx : x);
                y = y < 0 ? y + ny : (y >= ny ? y - ny : y);
                z = z >= nz ? z - nz : z;
                const int c = (int)rp.cell0 + (z * ny + y) * nx + x;
                const int c0 = A.cell_start[c];
                cnt = A.cell_start[c + 1] - c0;
                s_cell0[s] = c0;
                s_off[s] = make_float4((float)dx, (float)dy, (float)dz, 0.f);
            }
            int incl = cnt;
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(FULL, incl, o);
                if (lane >= o) incl += v;
            }
            if (s < ncell) s_beg[s + 1] = run + incl;
            run += __shfl_sync(FULL, incl, 31);
        }
        if (lane == 0) s_beg[0] = 0;
        __syncwarp();
        if (lane == 0) {
            bool over = run > stage;
            int b = 0;
            for (int r = 0; r < len; r++) {
                s_base[r] = b;
                b += s_beg[6 * r + 8] - s_beg[6 * r + 7];
                over = over || s_beg[6 * r + 18] - s_beg[6 * r] > A.mcap;
            }
            s_base[len] = b;
            s_next = part;
            s_over = over;
        }
    }
    __syncthreads();
    if (s_over) {
        if (tid == 0) atomicOr(A.status, ST_CAPACITY);
        store_zero(0);
        return;
    }
    for (int s = warp; s < ncell; s += nwarps) {
        const int b = s_beg[s], e = s_beg[s + 1], g0 = s_cell0[s] - b;
        const float4 o = s_off[s];
        for (int t = b + lane; t < e; t += 32) {
            const int g = g0 + t;
            const float x = A.xl[g], y = A.xl[n + g], z = A.xl[2 * n + g];
            P4[t] = make_float4(x, y, z, __int_as_float(s));
            S4[t] = make_float4(x + o.x * wf0, y + o.y * wf1, z + o.z * wf2, __int_as_float(g));
        }
    }
    __syncthreads();

    const float rc2 = rp.rc2f;
    const float c_lo = rc2 * (1.0f - 0x1p-16f), c_hi = rc2 * (1.0f + 0x1p-16f);
    // v to component d of molecule g's force
    auto add = [&](int d, int g, float v) {
        if constexpr (DET)
            atomicAdd(reinterpret_cast<unsigned long long*>(A.fs) + d * n + g, to_fix_w<float>(v, A.status));
        else
            atomicAdd(A.fs + d * n + g, fwd_widen(v));
    };
    // canonical displacement of two staged molecules and its square
    auto canon = [&](const float4& a, const float4& b) -> float4 {
        const float4 oa = s_off[__float_as_int(a.w)], ob = s_off[__float_as_int(b.w)];
        float4 d;
        d.x = Q::add(Q::sub(b.x, a.x), Q::mul(ob.x - oa.x, wf0));
        d.y = Q::add(Q::sub(b.y, a.y), Q::mul(ob.y - oa.y, wf1));
        d.z = Q::add(Q::sub(b.z, a.z), Q::mul(ob.z - oa.z, wf2));
        d.w = Q::add(Q::add(Q::mul(d.x, d.x), Q::mul(d.y, d.y)), Q::mul(d.z, d.z));
        return d;
    };

    // (the owner kernel that 3c01 had combined its lanes' shares in FP64)
    auto sum4 = [&](float x, float y, float z, float w) -> float {
        return COMP ? fwd_sum4_pair(x, y, z, w, lane) : fwd_sum4(x, y, z, w, lane);
    };
    Sum<float> esum, e2sum, w2sum;
    unsigned nint = 0, n2 = 0;
    const int M0 = s_base[len];

    for (int it = 0;; it++) {
        // molecules part, part + split, .. of the base cells; in the deterministic
        // mode warp w takes a fixed share of them
        int k0 = part + (it * nwarps + warp) * A.split;
        if (!DET) {
            if (lane == 0) k0 = atomicAdd(&s_next, A.split);
            k0 = __shfl_sync(FULL, k0, 0);
        }
        if (k0 >= M0) break;
        int r = 0;
        while (k0 >= s_base[r + 1]) r++;
        const int i = s_beg[6 * r + 7] + k0 - s_base[r];         // staged index
        const int t0 = s_beg[6 * r], t1 = s_beg[6 * r + 18];     // its 18 cells

        // ---- 1. forward list of i
        const float4 si = S4[i];
        int np = 0;
        bool rare = false;  // a square in the band, or another molecule at i's height
#pragma unroll 2
        for (int t = t0 + lane; t < t1 + lane; t += 32) {
            const float4 p = S4[t];
            const float dx = p.x - si.x, dy = p.y - si.y, dz = p.z - si.z;
            const float c = dx * dx + dy * dy + dz * dz;
            // above i: higher in its layer, or the next layer (whose unit-frame
            // height is at least w)
            const bool in = t < t1;
            const bool keep = in && c < c_lo && dz > 0.0f;
            rare = rare || (in && c < c_hi && (c >= c_lo || (dz == 0.0f && t != i)));
            const unsigned m = __ballot_sync(FULL, keep);
            if (keep) lidx[np + __popc(m & ((1u << lane) - 1u))] = (unsigned short)t;
            np += __popc(m);
        }
        const float4 pi = P4[i];
        if (__any_sync(FULL, rare)) {
            // again, with the canonical decision (of equal heights in a layer the
            // later in sorted order is above)
            np = 0;
#pragma unroll 1
            for (int t = t0 + lane; t < t1 + lane; t += 32) {
                bool keep = false;
                if (t < t1 && t != i) {
                    const float4 q = P4[t];
                    const float rz = q.z - pi.z;
                    keep = canon(pi, q).w < rc2 &&
                           (s_off[__float_as_int(q.w)].z > 0.0f || rz > 0.0f ||
                            (rz == 0.0f && __float_as_int(S4[t].w) > __float_as_int(si.w)));
                }
                const unsigned m = __ballot_sync(FULL, keep);
                if (keep) lidx[np + __popc(m & ((1u << lane) - 1u))] = (unsigned short)t;
                np += __popc(m);
            }
        }
        __syncwarp();
        if (np == 0) continue;
        // a row that fills the last chunk: too far from every partner to interact with it
        const float4 far = make_float4(0.f, 0.f, 64.0f * rp.rcf, 4096.0f * rc2);

        float fix = 0.f, fiy = 0.f, fiz = 0.f;  // force on i, this lane's share
        float fjx = 0.f, fjy = 0.f, fjz = 0.f;  // (LJ apart) its LJ part
        // sums of the lane's row j: V = sum g_jk (d_k - d_j), G = g_ij, over 3 nu
        struct RowSum {
            FwdSum<COMP> Vx, Vy, Vz, G;
            __device__ __forceinline__ void add(float gi, float gjk, float ex, float ey, float ez)
            {
                G.add(gi);
                Vx.fma(gjk, ex);
                Vy.fma(gjk, ey);
                Vz.fma(gjk, ez);
            }
        };
        Sum<float> es;  // energies of the list's triangles, over nu
        // The triangle of rows Dj (lane) and Dk: with the squared sides a, b, c
        // and x = (a + c - b) / 2, y = (b + c - a) / 2, m = (a + b - c) / 2,
        //     2 du/da = 3 nu q^5 (a y - x m - b c (1 + 5 x y m q^2)), cyclic,
        //     u = nu q^3 (1 + 3 x y m q^2), q = (a b c)^(-1/2).
        // decide(c): the third side's decision; e = d_k - d_j
        auto triangle = [&](const float4& Dj, const float4& Dk, auto decide, float& ga, float& gb,
                            float& gc, float& ex, float& ey, float& ez) {
            const float a = Dj.w, b = Dk.w;
            ex = Dk.x - Dj.x, ey = Dk.y - Dj.y, ez = Dk.z - Dj.z;
            const float c = ex * ex + ey * ey + ez * ez;
            const bool keep = decide(c);
            nint += keep ? 1u : 0u;
            const float t = fmaf(0.5f, b, 0.5f * a), w = fmaf(0.5f, b, -0.5f * a);
            const float x = fmaf(0.5f, c, -w), y = fmaf(0.5f, c, w), m = fmaf(-0.5f, c, t);
            const float bc = b * c, ac = a * c, ab = a * b;
            const float q = keep ? fwd_rsq(a * bc) : 0.0f;
            const float q2 = q * q;
            const float xm = x * m, ym = y * m, xy = x * y;
            const float p = (x * ym) * q2;
            const float z = fmaf(5.0f, p, 1.0f);
            const float q3 = q * q2, q5 = q3 * q2;
            es.add(q3 * fmaf(3.0f, p, 1.0f));
            ga = q5 * fmaf(-z, bc, fmaf(a, y, -xm));
            gb = q5 * fmaf(-z, ac, fmaf(b, x, -ym));
            gc = q5 * fmaf(-z, ab, fmaf(c, m, -xy));
        };
        // a row's share when its sums are complete; first: with its LJ term
        const float nu3 = 3.0f * rp.nuf;
        auto finish = [&](const float4& D, int t, const RowSum& R, bool first) {
            const int g = __float_as_int(S4[t].w);
            float G = nu3 * R.G.get();
            if (LJ && first) {
                // LJ pair scalar of (i, j): F_i = g d(i -> j); the LJ kernel's
                // expressions on the same displacement
                const float a = D.w;
                const float ia = __frcp_rn(a);
                const float s2 = rp.sig2f * ia;
                const float s3 = s2 * s2 * s2;
                const float s6 = s3 * s3;
                const float fw = (rp.eps48f * s6 - rp.eps24f * s3) * ia;
                e2sum.add(rp.eps4f * (s6 - s3) - rp.ushiftf);
                w2sum.add(fw * a);
                n2++;
                if (LJ == 2) {
                    const float gx = fw * D.x, gy = fw * D.y, gz = fw * D.z;
                    double* to = A.fs_lj + g;
                    atomicAdd(to, fwd_widen(gx));
                    atomicAdd(to + n, fwd_widen(gy));
                    atomicAdd(to + 2 * n, fwd_widen(gz));
                    fjx -= gx;
                    fjy -= gy;
                    fjz -= gz;
                } else {
                    G -= fw;
                }
            }
            add(0, g, fmaf(-G, D.x, nu3 * R.Vx.get()));
            add(1, g, fmaf(-G, D.y, nu3 * R.Vy.get()));
            add(2, g, fmaf(-G, D.z, nu3 * R.Vz.get()));
            fix = fmaf(G, D.x, fix);
            fiy = fmaf(G, D.y, fiy);
            fiz = fmaf(G, D.z, fiz);
        };

        bool whole = np > 32 + FWD_EXTRA;  // a longer list, or a third side in the band
        if (!whole) {
            // h rows one to a lane, and the few beyond 32 (each met with all the
            // others).  The rows that lanes beyond the list read may be stale.
            const int h = min(np, 32), nextra = np - h;
            const bool own = lane < h, extra = lane < nextra;
            const int tj = own ? lidx[lane] : i, te = extra ? lidx[32 + lane] : i;
            const float4 Dj = own ? canon(pi, P4[tj]) : far;
            float4 De = far;
            if (nextra) {
                if (extra) {
                    De = canon(pi, P4[te]);
                    list[64 + lane] = De;
                }
            }
            if (own) {
                list[lane] = Dj;
                list[lane + h] = Dj;
            }
            __syncwarp();
            const unsigned n_before = nint;
            float dev = c_hi;  // least distance of a third side's square from r_c^2
            RowSum R, RE;
            const float4* up = list + lane;        // row lane + s (mod h)
            const float4* down = list + lane + h;  // row lane - s
            auto near = [&](float c, bool ok) {
                const float x = c - rc2;
                dev = fminf(dev, fabsf(x));
                return ok && x < 0.0f;
            };
            auto shift = [&](int s, bool ok) {
                const float4 Dk = up[s], Ds = down[-s];
                float ga, gb, gc, ex, ey, ez;
                triangle(Dj, Dk, [&](float c) { return near(c, ok); }, ga, gb, gc, ex, ey, ez);
                R.add(ga, gc, ex, ey, ez);
                // (unsigned: a negative lane - s is the larger)
                const unsigned src = min((unsigned)(lane - s), (unsigned)(lane - s + h));
                gb = __shfl_sync(FULL, gb, (int)src);
                gc = __shfl_sync(FULL, gc, (int)src);
                R.add(gb, gc, Ds.x - Dj.x, Ds.y - Dj.y, Ds.z - Dj.z);
            };
            const int odd = (h - 1) >> 1;
#pragma unroll 2
            for (int s = 1; s <= odd; s++) shift(s, own);
            // the pairs (j, j + h / 2), once
            if ((h & 1) == 0) shift(h >> 1, lane < (h >> 1));
            if (nextra) {
#pragma unroll 1
                for (int e = 0; e < nextra; e++) {
                    // row 32 + e with the 32 rows, then with the extra ones before it
                    FwdSum<COMP> sx, sy, sz, sg;
                    const float4 Dk = list[64 + e];
#pragma unroll 1
                    for (int pass = 0; pass < 2; pass++) {
                        const float4 D = pass ? De : Dj;
                        float ga, gb, gc, ex, ey, ez;
                        triangle(D, Dk, [&](float c) { return near(c, pass ? lane < e : true); }, ga, gb, gc, ex, ey,
                                 ez);
                        if (pass) RE.add(ga, gc, ex, ey, ez);
                        else R.add(ga, gc, ex, ey, ez);
                        sg.add(gb);
                        sx.fma(gc, ex);
                        sy.fma(gc, ey);
                        sz.fma(gc, ez);
                        if (e == 0) break;
                    }
                    const float v = sum4(sx.get(), sy.get(), sz.get(), sg.get());
                    const float vx = __shfl_sync(FULL, v, 0), vy = __shfl_sync(FULL, v, 8),
                                vz = __shfl_sync(FULL, v, 16), vg = __shfl_sync(FULL, v, 24);
                    if (lane == e) {
                        RE.Vx.add(-vx);
                        RE.Vy.add(-vy);
                        RE.Vz.add(-vz);
                        RE.G.add(vg);
                    }
                }
            }
            // (a lane without a row has a far one, whose sides are in no band)
            whole = __any_sync(FULL, dev < c_hi - rc2);
            if (!whole) {
                if (own) {
                    finish(Dj, tj, R, true);
                    esum.add(es.s);
                    esum.add(-es.c);
                }
                if (nextra && extra) finish(De, te, RE, true);
            } else {
                nint = n_before;
                es = Sum<float>();
            }
        }
        if (whole) {
            // equal chunks of h rows; rows beyond the warp's table are formed again
            // each time
            const int nch = (np + 31) >> 5, h = (np + nch - 1) / nch;
            const bool table = nch * h <= FWD_ROWS;
            __syncwarp();
            if (table)
                for (int k = lane; k < nch * h; k += 32) list[k] = k < np ? canon(pi, P4[lidx[k]]) : far;
            __syncwarp();
            auto row = [&](int k) -> float4 {
                if (table) return list[k];
                return k < np ? canon(pi, P4[lidx[k]]) : far;
            };
            const int l0 = lane < h ? lane : 0;
#pragma unroll 1
            for (int J = 0; J < np; J += h) {
                const bool own = lane < h && J + lane < np;
                const float4 Dj = row(J + l0);
                const int tj = own ? lidx[J + lane] : i;
                RowSum R;
                // the chunk with itself (K = J: shifts 1 .. h / 2), then with the later
                // ones (all h shifts)
#pragma unroll 1
                for (int K = J; K < np; K += h) {
                    RowSum RK;
                    const float4 Dl = row(K + l0);
                    int k = l0, src = l0;
#pragma unroll 1
                    for (int s = 0; s < (K == J ? (h >> 1) + 1 : h); s++) {
                        if (K > J || s > 0) {
                            const float4 Dk = row(K + k), Ds = row(J + src);
                            const bool ok = own && K + k < np && !(K == J && 2 * s == h && lane >= s);
                            float ga, gb, gc, ex, ey, ez;
                            triangle(Dj, Dk, [&](float c) {
                                if (!ok || c >= c_hi) return false;
                                return c < c_lo || canon(P4[tj], P4[lidx[K + k]]).w < rc2;
                            }, ga, gb, gc, ex, ey, ez);
                            R.add(ga, gc, ex, ey, ez);
                            gb = __shfl_sync(FULL, gb, src);
                            gc = __shfl_sync(FULL, gc, src);
                            RK.add(gb, gc, Ds.x - Dl.x, Ds.y - Dl.y, Ds.z - Dl.z);
                        }
                        k = k + 1 == h ? 0 : k + 1;
                        src = src == 0 ? h - 1 : src - 1;
                    }
                    if (lane < h && K + lane < np) finish(Dl, lidx[K + lane], RK, false);
                }
                if (own) {
                    finish(Dj, tj, R, true);
                    esum.add(es.s);
                    esum.add(-es.c);
                }
                es = Sum<float>();
            }
        }
        const int d = lane >> 3;
        const bool mine = lane < 24 && (lane & 7) == 0;
        const float fi = sum4(fix, fiy, fiz, 0.0f);
        if (mine) add(d, __float_as_int(si.w), fi);
        if (LJ == 2) {
            const float fj = fwd_sum4(fjx, fjy, fjz, 0.0f, lane);
            if (mine) atomicAdd(A.fs_lj + d * n + __float_as_int(si.w), fwd_widen(fj));
        }
        __syncwarp();  // the list is read to the end before the next one is written
    }
    // every lane's E3, E2, W2 (value, rest) over the warp's list rows
    float2* sums = reinterpret_cast<float2*>(list);
    sums[lane] = make_float2(esum.s, -esum.c);
    if (LJ) {
        sums[32 + lane] = make_float2(e2sum.s, -e2sum.c);
        sums[64 + lane] = make_float2(w2sum.s, -w2sum.c);
    }
    {
        // counts in halves of 16 bits, so that a warp's sums fit 32
        const unsigned lo = __reduce_add_sync(FULL, nint & 0xffffu), hi = __reduce_add_sync(FULL, nint >> 16);
        const unsigned l2 = __reduce_add_sync(FULL, n2 & 0xffffu), h2 = __reduce_add_sync(FULL, n2 >> 16);
        if (lane == 0) {
            s_cnt[0][warp] = ((unsigned long long)hi << 16) + lo;
            s_cnt[1][warp] = ((unsigned long long)h2 << 16) + l2;
        }
    }
    store_zero(1);
    __syncthreads();

    // ---- sums of the unit: quantity w of E3, E2, W2 by warp w (mod the warps),
    // in pairs of floats
    for (int w = warp; w < (LJ ? 3 : 1); w += nwarps) {
        float v = 0.f, r = 0.f;
        for (int q = 0; q < nwarps; q++) {
            const float2 p = reinterpret_cast<const float2*>(smem + plan.off_list)[q * (2 * FWD_ROWS) + 32 * w + lane];
            fwd_add_pair(v, r, p.x, p.y);
        }
        for (int o = 16; o > 0; o >>= 1) {
            const float v2 = __shfl_down_sync(FULL, v, o), r2 = __shfl_down_sync(FULL, r, o);
            fwd_add_pair(v, r, v2, r2);
        }
        if (lane == 0) {
            const double x = (double)v + (double)r;
            unsigned long long cnt = 0;
            if (w < 2)
                for (int q = 0; q < nwarps; q++) cnt += s_cnt[w][q];
            if (w == 0) {
                const double e = (double)rp.nuf * x;
                A.unit_ew[2 * slot_out] = e;
                A.unit_ew[2 * slot_out + 1] = 9.0 * e;
                A.unit_cnt[2 * slot_out] = 0ull;  // candidates: counted by the reduction
                A.unit_cnt[2 * slot_out + 1] = A.trav == 0 ? 3 * cnt : cnt;  // 3c01 counts owner visits
            } else if (w == 1) {
                A.unit_ew2[2 * slot_out] = x;
                A.unit_cnt2[2 * slot_out] = 0ull;
                A.unit_cnt2[2 * slot_out + 1] = cnt;
            } else {
                A.unit_ew2[2 * slot_out + 1] = x;
            }
        }
    }
}

// One CTA per run of base cells along x (one cell per run, and split > 1 CTAs
// dealt its molecules, for systems of too few cells to fill the GPU).
// LJ: 0 none, 1 into fs, 2 apart.  COMP (3c01): compensated sums, at three CTAs
// to an SM for their registers
template <int LJ, bool DET, bool COMP>
__global__ void __launch_bounds__(32 * FWD_MAXW, COMP ? 3 : 4) k_atm_fwd(const FwdArgs A)
{
    after_previous();
    const int b = (int)(A.split > 1 ? blockIdx.x / A.split : blockIdx.x);
    int u = b;
    if (A.run > 1) {
        if (A.runs) {
            u = A.runs[b];
        } else {  // one replica
            const int nx = A.b.rep[0].g.nc[0], nseg = (nx + A.run - 1) / A.run;
            u = b / nseg * nx + b % nseg * A.run;
        }
    }
    atm_fwd_unit<LJ, DET, COMP>(A, u, A.split > 1 ? (int)(blockIdx.x % A.split) : 0);
}

}  // namespace atm3

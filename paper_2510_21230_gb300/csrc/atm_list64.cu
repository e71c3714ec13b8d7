// atm_list64.cu -- the FP64 pair rule of 3c01, 3c18 and 3c08 from forward lists
// in global memory.
//
// The FP64 pipe does two lanes per clock and SM, 1/64 of the FP32 rate, and a
// warp instruction takes its 16 cycles whatever lanes are active (measured:
// the same time for 1, 8, 16 and 32 lanes).  So everything but the triangle
// terms themselves is taken off it: decisions go through FP32 (only squares in a
// band of 2^-16 around r_c^2 are decided in FP64), interacting pairs are
// compacted so that every lane of an evaluation is a triangle, and the sums of
// the pair scalars G_e are reductions that the L2 performs.  Three kernels:
//
//  1. k_list64: the forward lists of atm_fwd.cuh (a molecule's partners within
//     r_c above it, 18 cells), written to global memory with a bitmap of the
//     partners per cell, from which the place of a partner in a list is found;
//     the pair scalars of the list's edges start at zero.
//  2. k_tri64: a warp per molecule i.  Every pair of its list is tested in FP32
//     (rotation), the hits queued and 32 triangles evaluated at a time.  With
//     the rows d_j, d_k and m = d_j . d_k, x = a - m, y = b - m, c = x + y,
//         g_a = 2 du/da = 3 nu q^5 (a y - x m - b c (1 + 5 x y m q^2)), cyclic,
//     34 FP64 instructions a triangle with the reciprocal square root (87 in
//     the block kernel).  g of the two edges at i is added to i's list, that of
//     (j, k) to the list of the lower of the two.
//  3. k_edge64: a warp per molecule sums F = sum_e G_e d and the virial
//     W3 = -sum_e G_e d^2 over its edges (E3 = W3 / 9: u is homogeneous of
//     degree -9), and evaluates LJ on the same displacements.
//
// Displacements come from the wrapped positions and the box, (x_j - x_i) -+ L,
// one rounding where the cell-local coordinates of the block kernels take
// three; decisions stay the canonical ones on cell-local coordinates.
//
// Kernel 2 is bound by the FP64 pipe: 32,000 molecules 0.51 ms (block kernel
// 1.67 ms), where 6.65 M triplets at 34 instructions of 16 cycles take 0.36 ms.
// Kernel 3 0.13 ms with LJ apart (LJ kernel 0.62 ms), kernel 1 0.04 ms.
#include "atm_common.cuh"

namespace atm3 {

namespace {

constexpr int L64_ROWS = 64;  // rows a warp of k_tri64 keeps (longer lists: formed again)

// 18-cell slot: column (x offset + 1) * 6, then the three cells of the layer
// (y offset + 1) and the three of the next
__device__ __forceinline__ void slot18(int s, int& dx, int& dy, int& dz)
{
    const int col = s / 6, q = s - 6 * col;
    dx = col - 1;
    dy = (q < 3 ? q : q - 3) - 1;
    dz = q < 3 ? 0 : 1;
}

// d(i -> j) from wrapped positions: i in cell (cx, cy, cz), j in the cell at
// offset (dx, dy, dz)
struct Frame64 {
    const double* x;
    const int* perm;
    long long n;
    int cx, cy, cz, nx, ny, nz;
    double L0, L1, L2, xi, yi, zi;
    __device__ __forceinline__ void set(const List64Args& A, const Rep& rp, long long gi)
    {
        x = A.x;
        perm = A.perm;
        n = A.n;
        nx = rp.g.nc[0];
        ny = rp.g.nc[1];
        nz = rp.g.nc[2];
        L0 = rp.g.L[0];
        L1 = rp.g.L[1];
        L2 = rp.g.L[2];
        const int lu = A.cell_sorted[gi] - (int)rp.cell0;
        cx = lu % nx;
        cy = lu / nx % ny;
        cz = lu / (nx * ny);
        const long long o = perm[gi];
        xi = x[o];
        yi = x[n + o];
        zi = x[2 * n + o];
    }
    __device__ __forceinline__ void disp(int g, int slot, double& dx, double& dy, double& dz) const
    {
        int ox, oy, oz;
        slot18(slot, ox, oy, oz);
        const long long o = perm[g];
        const double sx = cx + ox < 0 ? -L0 : (cx + ox >= nx ? L0 : 0.0);
        const double sy = cy + oy < 0 ? -L1 : (cy + oy >= ny ? L1 : 0.0);
        const double sz = cz + oz >= nz ? L2 : 0.0;
        dx = (x[o] - xi) + sx;
        dy = (x[n + o] - yi) + sy;
        dz = (x[2 * n + o] - zi) + sz;
    }
    // d(g -> h) of two partners in 18-cell slots s and t: exact for a close pair
    __device__ __forceinline__ void between(int g, int s, int h, int t, double& dx, double& dy, double& dz) const
    {
        int ox, oy, oz, px, py, pz;
        slot18(s, ox, oy, oz);
        slot18(t, px, py, pz);
        const long long o = perm[g], p = perm[h];
        auto image = [](int c, int m) { return c < 0 ? -1 : (c >= m ? 1 : 0); };
        dx = (x[p] - x[o]) + (double)(image(cx + px, nx) - image(cx + ox, nx)) * L0;
        dy = (x[n + p] - x[n + o]) + (double)(image(cy + py, ny) - image(cy + oy, ny)) * L1;
        dz = (x[2 * n + p] - x[2 * n + o]) + (double)(image(cz + pz, nz) - image(cz + oz, nz)) * L2;
    }
};

// c is below an eighth of the larger of a and b (by the bits of their high words: no
// FP64 instruction; a negative c is)
__device__ __forceinline__ bool small_side(double a, double b, double c)
{
    return __double2hiint(c) + (3 << 20) < max(__double2hiint(a), __double2hiint(b));
}

// v (one per lane and component) summed over the warp: lane 8 d holds component d
__device__ __forceinline__ double sum3_64(double x, double y, double z, int lane)
{
    const unsigned FULL = 0xffffffffu;
    const bool b4 = lane & 16, b3 = lane & 8;
    double k0 = b4 ? z : x, k1 = b4 ? 0.0 : y;
    const double s0 = __shfl_xor_sync(FULL, b4 ? x : z, 16);
    const double s1 = __shfl_xor_sync(FULL, b4 ? y : 0.0, 16);
    k0 += s0;
    k1 += s1;
    double k = (b3 ? k1 : k0) + __shfl_xor_sync(FULL, b3 ? k0 : k1, 8);
    for (int o = 4; o > 0; o >>= 1) k += __shfl_xor_sync(FULL, k, o);
    return k;
}

}  // namespace

// One CTA per run of base cells along x (as k_atm_fwd)
__global__ void __launch_bounds__(32 * FWD_MAXW) k_list64(const List64Args A)
{
    after_previous();
    constexpr unsigned FULL = 0xffffffffu;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_beg[FWD_CELLS + 1];
    __shared__ int s_cell0[FWD_CELLS];
    __shared__ int s_base[FWD_RUN + 1];
    __shared__ int s_over;
    __shared__ unsigned s_word[FWD_MAXW][18];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
    int u = (int)(blockIdx.x / A.split);
    const int part = (int)(blockIdx.x % A.split);
    if (A.run > 1) {
        if (A.runs) {
            u = A.runs[u];
        } else {  // one replica
            const int nx = A.b.rep[0].g.nc[0], nseg = (nx + A.run - 1) / A.run;
            u = u / nseg * nx + u % nseg * A.run;
        }
    }
    const Rep& rp = A.b.rep[A.b.rep_of_cell[u]];
    const int lu = u - (int)rp.cell0;
    const long long n = A.n;
    const int stage = fwd_stage(A.mcap, A.run);
    float4* S4 = reinterpret_cast<float4*>(smem);  // unit-frame position, sorted index
    unsigned char* sslot = smem + 16 * (size_t)(stage + 32);
    const int nx = rp.g.nc[0], ny = rp.g.nc[1], nz = rp.g.nc[2];
    const int cx = lu % nx, cy = (lu / nx) % ny, cz = lu / (nx * ny);
    const int len = min(A.run, nx - cx), ncell = 6 * (len + 2);
    if (warp == 0) {
        int run = 0;
        for (int s0 = 0; s0 < ncell; s0 += 32) {
            const int s = s0 + lane;
            int cnt = 0;
            if (s < ncell) {
                int dx, dy, dz;
                slot18(s, dx, dy, dz);
                int x = cx + dx, y = cy + dy, z = cz + dz;
                x = x < 0 ? x + nx : (x >= nx ? x - nx : x);
                y = y < 0 ? y + ny : (y >= ny ? y - ny : y);
                z = z >= nz ? z - nz : z;
                const int c = (int)rp.cell0 + (z * ny + y) * nx + x;
                const int c0 = A.cell_start[c];
                cnt = A.cell_start[c + 1] - c0;
                s_cell0[s] = c0;
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
            for (int s = 0; s < ncell; s++) over = over || s_beg[s + 1] - s_beg[s] > PM_CELL_MAX;
            s_base[len] = b;
            s_over = over;
        }
    }
    __syncthreads();
    const bool over = s_over;
    const int M0 = s_base[len];
    if (over) {
        // a unit beyond the capacity (flagged): its molecules keep empty lists
        if (tid == 0) atomicOr(A.status, ST_CAPACITY);
        for (int k = tid; k < M0; k += blockDim.x) {
            int r = 0;
            while (k >= s_base[r + 1]) r++;
            const long long g = s_cell0[6 * r + 7] + k - s_base[r];
            A.count[g] = 0;
            for (int q = 0; q < 18; q++) A.place[g * 18 + q] = make_uint2(0u, 0u);  // (others look here)
        }
        return;
    }
    const float wf0 = rp.wf[0], wf1 = rp.wf[1], wf2 = rp.wf[2];
    for (int s = warp; s < ncell; s += nwarps) {
        const int b = s_beg[s], e = s_beg[s + 1], g0 = s_cell0[s] - b;
        int dx, dy, dz;
        slot18(s, dx, dy, dz);
        for (int t = b + lane; t < e; t += 32) {
            const int g = g0 + t;
            S4[t] = make_float4(A.xl32[g] + (float)dx * wf0, A.xl32[n + g] + (float)dy * wf1,
                                A.xl32[2 * n + g] + (float)dz * wf2, __int_as_float(g));
            sslot[t] = (unsigned char)s;
        }
    }
    __syncthreads();
    // FP32 squares of unit-frame differences are within 6.5e-6 r_c^2 of the FP64
    // ones (rounded coordinates up to 5 w, w <= 4/3 r_c, and the rounded w)
    const float rc2f = (float)rp.rc2;
    const float c_lo = rc2f * (1.0f - 0x1p-16f), c_hi = rc2f * (1.0f + 0x1p-16f);
    for (int k0 = part + warp * A.split; k0 < M0; k0 += nwarps * A.split) {
        int r = 0;
        while (k0 >= s_base[r + 1]) r++;
        const int i = s_beg[6 * r + 7] + k0 - s_base[r];
        const int t0 = s_beg[6 * r], t1 = s_beg[6 * r + 18];
        const float4 si = S4[i];
        const int gi = __float_as_int(si.w);
        uint2* list = A.list + (long long)gi * A.stride;
        double* G = A.G + (long long)gi * A.stride;
        if (lane < 18) s_word[warp][lane] = 0u;
        __syncwarp();
        int np = 0;
        for (int t = t0 + lane; t < t1 + lane; t += 32) {
            const float4 p = S4[t];
            const float dx = p.x - si.x, dy = p.y - si.y, dz = p.z - si.z;
            const float c = dx * dx + dy * dy + dz * dz;
            const bool in = t < t1;
            bool keep = in && c < c_lo && dz > 0.0f;
            if (in && c < c_hi && t != i && (c >= c_lo || dz == 0.0f)) {
                // in the band, or at i's height: the canonical FP64 decision (of
                // equal heights in a layer the later in sorted order is above)
                int ox, oy, oz;
                slot18(sslot[t], ox, oy, oz);
                const long long g = __float_as_int(p.w);
                double ex, ey, ez;
                const double d2 = canon_disp<double>(
                    A.xl[gi], A.xl[n + gi], A.xl[2 * n + gi], A.xl[g], A.xl[n + g], A.xl[2 * n + g],
                    ox - r, oy, oz, rp.g.w[0], rp.g.w[1], rp.g.w[2], ex, ey, ez);
                keep = d2 < rp.rc2 &&
                       (oz > 0 || dz > 0.0f || (dz == 0.0f && __float_as_int(p.w) > gi));
            }
            const unsigned m = __ballot_sync(FULL, keep);
            if (keep) {
                const int pos = np + __popc(m & ((1u << lane) - 1u));
                const int s = sslot[t], b = t - s_beg[s];
                list[pos] = make_uint2((unsigned)__float_as_int(p.w), (unsigned)(s - 6 * r) | ((unsigned)b << 8));
                G[pos] = 0.0;
                atomicOr(&s_word[warp][s - 6 * r], 1u << b);
            }
            np += __popc(m);
        }
        __syncwarp();
        // the bitmap and the place of its first partner in the list, per cell
        const unsigned w = lane < 18 ? s_word[warp][lane] : 0u;
        int incl = __popc(w);
        const int own = incl;
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(FULL, incl, o);
            if (lane >= o) incl += v;
        }
        if (lane < 18) A.place[(long long)gi * 18 + lane] = make_uint2(w, (unsigned)(incl - own));
        if (lane == 0) A.count[gi] = np;
        __syncwarp();
    }
}

// One warp per molecule
__global__ void __launch_bounds__(128) k_tri64(const List64Args A)
{
    constexpr unsigned FULL = 0xffffffffu;
    __shared__ double s_row[4][L64_ROWS][4];   // d(i -> j), |d|^2
    __shared__ float4 s_f[4][L64_ROWS];        // d in FP32, the molecule's own height
    __shared__ uint2 s_meta[4][L64_ROWS];      // sorted index, slot | place in its cell << 8
    __shared__ unsigned s_queue[4][64];        // j | k << 16
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long i = blockIdx.x * 4ll + warp;
    if (i >= A.n) return;  // whole warps leave together
    const int np = A.count[i];
    if (np < 2) {
        if (lane == 0) A.mol_n3[i] = 0u;
        return;
    }
    const long long n = A.n;
    const Rep& rp = A.b.rep[A.b.rep_of_mol[i]];
    Frame64 F;
    F.set(A, rp, i);
    const uint2* list = A.list + i * A.stride;
    double* G = A.G + i * A.stride;
    const bool table = np <= L64_ROWS;
    auto form = [&](uint2 e, double& dx, double& dy, double& dz, float4& f) {
        F.disp((int)e.x, (int)(e.y & 0xffu), dx, dy, dz);
        f = make_float4((float)dx, (float)dy, (float)dz, A.xl32[2 * n + e.x]);
    };
    if (table)
        for (int k = lane; k < np; k += 32) {
            const uint2 e = list[k];
            double dx, dy, dz;
            float4 f;
            form(e, dx, dy, dz, f);
            s_row[warp][k][0] = dx;
            s_row[warp][k][1] = dy;
            s_row[warp][k][2] = dz;
            s_row[warp][k][3] = dx * dx + dy * dy + dz * dz;
            s_f[warp][k] = f;
            s_meta[warp][k] = e;
        }
    __syncwarp();
    auto meta = [&](int k) -> uint2 { return table ? s_meta[warp][k] : list[k]; };
    auto row32 = [&](int k) -> float4 {
        if (table) return s_f[warp][k];
        double dx, dy, dz;
        float4 f;
        form(list[k], dx, dy, dz, f);
        return f;
    };
    auto row64 = [&](int k, double& dx, double& dy, double& dz, double& a) {
        if (table) {
            dx = s_row[warp][k][0];
            dy = s_row[warp][k][1];
            dz = s_row[warp][k][2];
            a = s_row[warp][k][3];
        } else {
            float4 f;
            form(list[k], dx, dy, dz, f);
            a = dx * dx + dy * dy + dz * dz;
        }
    };
    const double nu3 = 3.0 * rp.nu;
    // triangle (i, j, k) of list rows j and k
    auto evaluate = [&](unsigned e) {
        const int j = (int)(e & 0xffffu), k = (int)(e >> 16);
        double xj, yj, zj, a, xk, yk, zk, b;
        row64(j, xj, yj, zj, a);
        row64(k, xk, yk, zk, b);
        double m = xj * xk + yj * yk + zj * zk;
        double x = a - m, y = b - m, c = x + y;
        // c by cancellation keeps fewer digits than the rows have where it is below
        // a + b by more than 16 (measured against extended precision on triangles of a
        // liquid's sides: rms force error 4.1e-15 above that line, where displacements
        // of three roundings each and their differences give 4.8e-15; 1.4e-13 at 1/256);
        // there it comes from the two positions (1.6e-15).  A liquid has next to none.
        if (small_side(a, b, c)) {
            const uint2 ej = meta(j), ek = meta(k);
            double ex, ey, ez;
            F.between((int)ej.x, (int)(ej.y & 0xffu), (int)ek.x, (int)(ek.y & 0xffu), ex, ey, ez);
            c = ex * ex + ey * ey + ez * ez;
            x = -(xj * ex + yj * ey + zj * ez);
            y = c - x;
            m = a - x;
        }
        const double bc = b * c, ac = a * c, ab = a * b;
        const double q = rsqrt(a * bc);
        const double q2 = q * q;
        const double xm = x * m, ym = y * m, xy = x * y;
        const double z = fma(5.0 * q2, xy * m, 1.0);
        const double q5 = (nu3 * q) * (q2 * q2);
        const double ga = q5 * fma(-z, bc, fma(a, y, -xm));
        const double gb = q5 * fma(-z, ac, fma(b, x, -ym));
        const double gc = q5 * fma(-z, ab, fma(c, m, -xy));
        atomicAdd(G + j, ga);
        atomicAdd(G + k, gb);
        // the edge (j, k) is in the list of the lower of the two
        const uint2 ej = meta(j), ek = meta(k);
        int jx, jy, jz, kx, ky, kz;
        slot18((int)(ej.y & 0xffu), jx, jy, jz);
        slot18((int)(ek.y & 0xffu), kx, ky, kz);
        const float hj = table ? s_f[warp][j].w : A.xl32[2 * n + ej.x];
        const float hk = table ? s_f[warp][k].w : A.xl32[2 * n + ek.x];
        const bool up = kz != jz ? kz > jz : (hk != hj ? hk > hj : ek.x > ej.x);  // k above j
        const int sg = up ? 1 : -1;
        const int s = ((kx - jx) * sg + 1) * 6 + (kz != jz ? 3 : 0) + (ky - jy) * sg + 1;
        const long long low = up ? ej.x : ek.x;
        const unsigned bit = (up ? ek.y : ej.y) >> 8;
        const uint2 pl = A.place[low * 18 + s];
        const unsigned pos = pl.y + __popc(pl.x & ((1u << bit) - 1u));
        atomicAdd(A.G + low * A.stride + pos, gc);
    };
    // every pair of the list once, 32 rows at a time: rows j and j + s (mod np),
    // s = 1 .. np / 2 (the last shift of an even list meets its pairs twice)
    const float rc2f = (float)rp.rc2;
    const float c_lo = rc2f * (1.0f - 0x1p-16f), c_hi = rc2f * (1.0f + 0x1p-16f);
    int qn = 0;
    unsigned nint = 0;
    for (int j0 = 0; j0 < np; j0 += 32) {
        const int j = j0 + lane;
        const float4 fj = row32(j < np ? j : 0);
        int k = j;
        for (int s = 1; s <= np >> 1; s++) {
            k = k + 1 == np ? 0 : k + 1;
            const bool ok = j < np && !(2 * s == np && j >= s);
            bool keep = false;
            if (ok) {
                const float4 fk = row32(k);
                const float ex = fk.x - fj.x, ey = fk.y - fj.y, ez = fk.z - fj.z;
                const float c = ex * ex + ey * ey + ez * ez;
                keep = c < c_lo;
                if (!keep && c < c_hi) {
                    const uint2 ej = meta(j), ek = meta(k);
                    int jx, jy, jz, kx, ky, kz;
                    slot18((int)(ej.y & 0xffu), jx, jy, jz);
                    slot18((int)(ek.y & 0xffu), kx, ky, kz);
                    double dx, dy, dz;
                    keep = canon_disp<double>(A.xl[ej.x], A.xl[n + ej.x], A.xl[2 * n + ej.x], A.xl[ek.x],
                                              A.xl[n + ek.x], A.xl[2 * n + ek.x], kx - jx, ky - jy, kz - jz,
                                              rp.g.w[0], rp.g.w[1], rp.g.w[2], dx, dy, dz) < rp.rc2;
                }
            }
            const unsigned m = __ballot_sync(FULL, keep);
            if (keep) s_queue[warp][qn + __popc(m & ((1u << lane) - 1u))] = (unsigned)j | ((unsigned)k << 16);
            qn += __popc(m);
            nint += __popc(m);
            __syncwarp();
            if (qn >= 32) {
                evaluate(s_queue[warp][lane]);
                __syncwarp();
                if (lane < qn - 32) s_queue[warp][lane] = s_queue[warp][32 + lane];
                qn -= 32;
                __syncwarp();
            }
        }
    }
    if (lane < qn) evaluate(s_queue[warp][lane]);
    if (lane == 0) A.mol_n3[i] = nint;
}

// One warp per molecule.  LJ: 1 into fs, 2 apart
template <int LJ>
__global__ void __launch_bounds__(128) k_edge64(const List64Args A)
{
    const int lane = threadIdx.x & 31;
    const long long n = A.n, i = blockIdx.x * 4ll + (threadIdx.x >> 5);
    if (i >= n) return;  // whole warps leave together
    const int np = A.count[i];
    const Rep& rp = A.b.rep[A.b.rep_of_mol[i]];
    double fx = 0.0, fy = 0.0, fz = 0.0, lx = 0.0, ly = 0.0, lz = 0.0, e2 = 0.0, w2 = 0.0, w3 = 0.0;
    if (np > 0) {
        Frame64 F;
        F.set(A, rp, i);
        for (int k = lane; k < np; k += 32) {
            const uint2 e = A.list[i * A.stride + k];
            double dx, dy, dz;
            F.disp((int)e.x, (int)(e.y & 0xffu), dx, dy, dz);
            const double a = dx * dx + dy * dy + dz * dz;
            double g = A.G[i * A.stride + k];
            w3 = fma(-g, a, w3);
            const double ia = __drcp_rn(a);
            const double s2 = rp.sig2 * ia;
            const double s3 = s2 * s2 * s2;
            const double fw = (rp.eps48 * s3 - rp.eps24) * (s3 * ia);
            e2 += rp.eps4 * (s3 * s3 - s3) - rp.ushift;
            w2 = fma(fw, a, w2);
            double* to = A.fs + e.x;
            if (LJ == 1) {
                g -= fw;
            } else {
                const double px = fw * dx, py = fw * dy, pz = fw * dz;
                double* tl = A.fs_lj + e.x;
                atomicAdd(tl, px);
                atomicAdd(tl + n, py);
                atomicAdd(tl + 2 * n, pz);
                lx -= px;
                ly -= py;
                lz -= pz;
            }
            const double px = g * dx, py = g * dy, pz = g * dz;
            if (g != 0.0) {
                atomicAdd(to, -px);
                atomicAdd(to + n, -py);
                atomicAdd(to + 2 * n, -pz);
            }
            fx += px;
            fy += py;
            fz += pz;
        }
        const bool mine = lane < 24 && (lane & 7) == 0;
        const double f = sum3_64(fx, fy, fz, lane);
        if (mine) atomicAdd(A.fs + (lane >> 3) * n + i, f);
        if (LJ == 2) {
            const double l = sum3_64(lx, ly, lz, lane);
            if (mine) atomicAdd(A.fs_lj + (lane >> 3) * n + i, l);
        }
        const double s = sum3_64(e2, w2, w3, lane);
        if (lane == 0) A.mol_ew[2 * i] = s;
        if (lane == 8) A.mol_ew[2 * i + 1] = s;
        if (lane == 16) A.mol_w3[i] = s;
    } else {
        if (lane < 2) A.mol_ew[2 * i + lane] = 0.0;
        if (lane == 2) A.mol_w3[i] = 0.0;
    }
    if (lane == 0) {
        A.mol_cnt[2 * i] = 0u;  // candidates: counted by the reduction
        A.mol_cnt[2 * i + 1] = (unsigned)np;
    }
}

size_t list64_smem(int mcap, int run) { return 17 * (size_t)(fwd_stage(mcap, run) + 32); }

cudaError_t launch_list64(const List64Args& a, cudaStream_t s)
{
    if (a.n <= 0 || a.b.ncell <= 0) return cudaSuccess;
    const size_t smem = list64_smem(a.mcap, a.run);
    cudaError_t e = cudaFuncSetAttribute(k_list64, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)LIST64_SMEM);
    if (e != cudaSuccess) return e;
    const long long units = a.run > 1 ? a.nruns : a.b.ncell;
    launch_after(k_list64, (unsigned)(units * a.split), 32 * FWD_MAXW, smem, s, a);
    const unsigned grid = (unsigned)((a.n + 3) / 4);
    // (not launch_after: CTAs that come while others still run pile up on the SMs that
    // are free first, and the FP64 pipe of each SM is the bound: ten steps of the two
    // replay systems 1,736 us so, 1,448 thus)
    k_tri64<<<grid, 128, 0, s>>>(a);
    if (a.lj == 1) k_edge64<1><<<grid, 128, 0, s>>>(a);
    else k_edge64<2><<<grid, 128, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace atm3

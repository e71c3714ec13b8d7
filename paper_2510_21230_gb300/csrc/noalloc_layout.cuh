// noalloc_layout.cuh -- the scratch array of the allocation-free entry point
// (noalloc.cu): where its arrays lie, in bytes from its beginning.
#pragma once
#include "atm3.h"
#include "atm3_internal.cuh"
#include "md_kernels.cuh"

namespace atm3 {

constexpr size_t NA_ALIGN = 256;
constexpr size_t na_al(size_t v) { return (v + NA_ALIGN - 1) & ~(NA_ALIGN - 1); }

constexpr long long NA_N = ATM_NOALLOC_MAX_N;
constexpr long long NA_C = ATM_NOALLOC_MAX_CELLS;

// What a call must find at zero, back to back for its n molecules and ncell cells
// so that one operation clears it: the status word (behind the results), the
// occupancy maxima, the cell counts, the replica of every cell and molecule, the
// kinetic energies.  (The cell build leaves its counts at zero, but a call that
// overlaps another or ends early does not, and counts too high would send the next
// call's molecules beyond their arrays.)
struct NaZero {
    size_t status, maxocc, count, rep_of_cell, rep_of_mol, ke, end;
};

constexpr NaZero na_zero_at(size_t o, long long n, long long ncell)
{
    NaZero Z{};
    Z.status = o;      o = na_al(o + sizeof(int));
    Z.maxocc = o;      o = na_al(o + (1 + ATM_NUNIT) * sizeof(int));
    Z.count = o;       o = na_al(o + (size_t)ncell * sizeof(int));
    Z.rep_of_cell = o; o = na_al(o + (size_t)ncell * sizeof(int));
    Z.rep_of_mol = o;  o = na_al(o + (size_t)n * sizeof(int));
    Z.ke = o;          o = na_al(o + (size_t)n * sizeof(double));
    Z.end = o;
    return Z;
}

struct NaLayout {
    size_t rep, x, cell_of, rank, start, perm, cell_sorted, xl, xl32, f_lj, unit_ew, unit_cnt, unit_ew2,
        unit_cnt2, mol_ew, mol_cnt, res, zero, total;
};

constexpr NaLayout na_layout()
{
    NaLayout L{};
    size_t o = 0;
    L.rep = o;         o = na_al(o + sizeof(Rep));
    L.x = o;           o = na_al(o + 3 * NA_N * sizeof(double));
    L.cell_of = o;     o = na_al(o + NA_N * sizeof(int));
    L.rank = o;        o = na_al(o + NA_N * sizeof(int));
    L.start = o;       o = na_al(o + (NA_C + 1) * sizeof(int));
    L.perm = o;        o = na_al(o + NA_N * sizeof(int));
    L.cell_sorted = o; o = na_al(o + NA_N * sizeof(int));
    L.xl = o;          o = na_al(o + 3 * NA_N * sizeof(double));
    L.xl32 = o;        o = na_al(o + 3 * NA_N * sizeof(float));
    L.f_lj = o;        o = na_al(o + 6 * NA_N * sizeof(double));  // f_atm behind it
    L.unit_ew = o;     o = na_al(o + 2 * NA_C * sizeof(double));
    L.unit_cnt = o;    o = na_al(o + 2 * NA_C * sizeof(unsigned long long));
    L.unit_ew2 = o;    o = na_al(o + 2 * NA_C * sizeof(double));
    L.unit_cnt2 = o;   o = na_al(o + 2 * NA_C * sizeof(unsigned long long));
    L.mol_ew = o;      o = na_al(o + 2 * NA_N * sizeof(double));
    L.mol_cnt = o;     o = na_al(o + 2 * NA_N * sizeof(unsigned));
    L.res = o;         o = na_al(o + (1 + REDUCE_PARTS) * sizeof(ResultDev));
    L.zero = o;        o = na_zero_at(o, NA_N, NA_C).end;
    L.total = o;
    return L;
}
constexpr NaLayout NA = na_layout();

constexpr NaZero na_zero(long long n, long long ncell) { return na_zero_at(NA.zero, n, ncell); }

}  // namespace atm3

// internal.h -- data layouts shared by the host planner (topology.cpp) and the
// CUDA kernels (solve.cu).  Not part of the public ABI.
//
// Every molecule is described by a "program": a compact, 16-byte aligned blob of
// 16-bit indices that a team of threads (one warp, or one CTA for large molecules)
// copies next to its numerical state and then interprets once per Newton iteration.
//
// Constraint numbering inside a molecule is the ELIMINATION POSITION p (0..nc-1):
// pivots are sorted by level, so the pivots of one level are contiguous.
//
// LU form: A = L U with L unit lower triangular and U upper triangular (diagonal
// d_j).  L is stored unscaled, Lt[q,j] = L[q,j] d_j, together with inv_j = 1 / d_j,
// so that every entry is computed by the same division-free expression:
//   DIAG j        d_j     = a_jj - sum_m Lt[j,m] inv_m U[m,j];   inv_j = 1 / d_j
//                 y_j     = sigma_j - sum_m Lt[j,m] inv_m y_m     (forward solve, fused)
//   U (j,q)       U[j,q]  = a_jq - sum_m Lt[j,m] inv_m U[m,q]    for q in N+(j)
//   L (q,j)       Lt[q,j] = a_qj - sum_m Lt[q,m] inv_m U[m,j]    for q in N+(j)
// where N+(j) are the later neighbours of j in the filled graph and m runs over
// earlier pivots adjacent to both row and column.  Task t writes value slot t.
// Within a level the DIAG tasks come first, then for each pivot its U row and its
// L column.  The backward solve is delta_j = inv_j (y_j - sum_{q in N+(j)} U[j,q] delta_q).
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define ILVES_HD __host__ __device__ __forceinline__
#else
#define ILVES_HD inline
#endif

namespace ilves {

constexpr uint32_t kNoAtom32 = 0xFFFFFFFFu;

// Program words of large molecules (32-bit, run by a whole CTA or several); the batched
// kernel's molecules have a program of their own (BatchLayout).
//   Task (large molecules): row, col of the target entry; atomsign = (shared atom << 1) |
//         (sign product < 0), the dummy atom for fill entries, unused for DIAG tasks;
//         tstart = first term.  Task t's terms are [tstart_t, tstart_{t+1}); a sentinel
//         task ends the list.
//   TermWide: l = slot of Lt[row, m], u = slot of U[m, col], m = the earlier pivot.
//   Piv:  diag = first slot of the pivot's U row (its L column follows), nup = |N+(pivot)|.
//   ConA: local atom ids (i, j) of the constraint at position p.
// inc[e] = p << 1 | (atom is the second atom of constraint p)
struct Task { uint32_t row, col, atomsign, tstart; };
struct ConA { uint32_t i, j; };
struct Piv { uint32_t diag, nup; };
struct TermWide { uint32_t l, u, m, pad; };

// Words of a batched molecule's program.  Its values are two to a slot: off-diagonal pair k of the
// factor (U[j,q], L[q,j]), then pivot p at batch_pivot_base + p, then a zero.
// PairWord: row j (8) | column q (8) << 8 | shared atom (9) << 16 | negative sign product (1) << 25.
struct PairWord {
    static constexpr uint32_t kMaxAtom = 511;
    static ILVES_HD uint32_t row(uint32_t w) { return w & 0xFFu; }
    static ILVES_HD uint32_t col(uint32_t w) { return (w >> 8) & 0xFFu; }
    static ILVES_HD uint32_t atom(uint32_t w) { return (w >> 16) & 0x1FFu; }
    static ILVES_HD uint32_t neg(uint32_t w) { return (w >> 25) & 1u; }
    static ILVES_HD uint32_t make(uint32_t row, uint32_t col, uint32_t atomsign) {
        return row | (col << 8) | ((atomsign >> 1) << 16) | ((atomsign & 1u) << 25);
    }
};
// HeadWord of an item that has terms: slot (12) | pivot (1) << 12 | pairs of terms past the first
// (5) << 13 | its first pair of terms (14) << 18.  16384 pairs are 128 KB of terms; stars of
// up to 57 bonds, whose factor is full, stay below (176 KB with their float64 values).
struct HeadWord {
    static constexpr uint32_t kMaxTerms = 63, kMaxPairs = 16384;
    static ILVES_HD uint32_t slot(uint32_t h) { return h & 0xFFFu; }
    static ILVES_HD bool diag(uint32_t h) { return ((h >> 12) & 1u) != 0u; }
    static ILVES_HD uint32_t more(uint32_t h) { return (h >> 13) & 31u; }
    static ILVES_HD uint32_t first(uint32_t h) { return h >> 18; }
    static ILVES_HD uint32_t make(uint32_t slot, bool diag, uint32_t pairs, uint32_t first) {
        return slot | (diag ? 1u << 12 : 0u) | ((pairs - 1u) << 13) | (first << 18);
    }
};
// TermWord of item (j, q) and earlier pivot m: slots of the pairs (m, j) (12) and (m, q) (12) << 12
// (a pivot's term: the same slot twice) | m (8) << 24.
struct TermWord {
    static ILVES_HD uint32_t a(uint32_t t) { return t & 0xFFFu; }
    static ILVES_HD uint32_t b(uint32_t t) { return (t >> 12) & 0xFFFu; }
    static ILVES_HD uint32_t m(uint32_t t) { return t >> 24; }
    static ILVES_HD uint32_t make(uint32_t a, uint32_t b, uint32_t m) { return a | (b << 12) | (m << 24); }
};
// Substitution record of a batched molecule's pivot, two words: first pair of its row (12) |
// entries of the row (8) << 12 | column of the first (8) << 20, columns of the next three (8 each).
#ifdef __CUDACC__
struct BackWord {
    static ILVES_HD uint32_t slot(uint2 w) { return w.x & 0xFFFu; }
    static ILVES_HD uint32_t n(uint2 w) { return (w.x >> 12) & 0xFFu; }
    static ILVES_HD uint32_t q(uint2 w, int k) { return k == 0 ? w.x >> 20 : (w.y >> (8 * (k - 1))) & 0xFFu; }
};
#endif
constexpr uint32_t kNoInc = 0x8000u;  // an absent incidence of a batched molecule's atom

constexpr uint32_t kCompactMaxConstraints = 256, kCompactMaxSlots = 4096;
// Threads of the team that solves one molecule of the batched kernel (whole warps; three
// warps cut the passes of wide levels at no cost in residency, which shared memory
// limits to about eight molecules per SM), the batched kernel's CTA size bound and its
// molecule slots per CTA.  Measured on the 4096-tree batch (mixed, kernel only, an early version
// with one task per factor entry): 32 threads 224 us, 64 195 us, 96 185 us, 128 206 us.
#ifndef ILVES_SLOT_THREADS
#define ILVES_SLOT_THREADS 96
#endif
constexpr int kSlotThreads = ILVES_SLOT_THREADS;
constexpr int kSlotCtaThreads = 768;
constexpr int kMaxSlotsPerCta = kSlotCtaThreads / kSlotThreads;
// Narrow class: molecules of at most narrow_atoms atoms get one-warp teams, up to
// kNarrowSlotsPerCta per CTA beside its 96-thread teams.  Their slices are small, so an SM's
// shared memory holds about three times as many of them: a batch of 4096 trees of 50-100 atoms
// (mixed) takes 87 us against 108 on 96-thread teams, 8192 of 20-50 atoms 95 against 141.  On
// batches of mixed sizes (20-200 atoms, mixed / float64 / float-float) they gain 3 % at best and
// lose in the other precisions (up to 60 atoms: 124 / 344 / 143 us against 127 / 327 / 131), so
// the automatic choice keeps those on 96 threads and leaves the threshold to the autotuner.
constexpr int kNarrowThreads = 32;
constexpr int kNarrowSlotsPerCta = kSlotCtaThreads / kNarrowThreads;
constexpr int kDefaultNarrowAtoms = 100;

ILVES_HD uint32_t align16(uint32_t b) { return (b + 15u) & ~15u; }

// Program of a batched molecule (16-byte aligned sections).  `staged` = bytes a team copies
// into shared memory (everything but con_gid, which is read from the global copy of the
// blob); `bytes` = the whole blob.
//   head      BatchHead
//   con       uint32 x nc            local atoms i | j << 16 of each position
//   back      uint32 x 2 nc          substitution records (BackWord)
//   lvl_piv   uint16 x (nlevel + 1)  positions of each level
//   lvl_hdr   uint16 x (nlevel + 1)  headers of each level (level 0 has none)
//   inc4      uint16 x 4 na          first four incidences of each atom in ascending position,
//                                    p << 1 | (atom is the second atom of p), else kNoInc
//   over_ptr  uint16 x (nover + 1)   incidences past the fourth of atoms [0, nover) (local atoms
//   over      uint16 x nover_inc     are ordered by decreasing degree)
//   aslot     uint16 x na            local atom of each atom slot (ascending global order)
//   pairs     uint32 x npair         PairWord of every off-diagonal pair of A and its fill, pivot
//                                    by pivot
//   hdr       uint32 x nhdr          HeadWord of the items that have terms, level by level (in a
//                                    level by decreasing number of terms)
//   terms     uint32 x nterm         TermWords, each item's completed to an even number by a term
//                                    of the zero slot
struct BatchSizes { int32_t na, nc, npair, nlevel, nhdr, nterm, nover, nover_inc; };
// wide32, wide16: the first level from which on no level has more than 32, 16 items with terms;
// wide_piv: the first level from which on no level has more than 32 pivots.
struct BatchHead { uint16_t wide32, wide16, wide_piv, pad[5]; };
struct BatchLayout {
    uint32_t con, back, lvl_piv, lvl_hdr, inc4, over_ptr, over, aslot, pairs, hdr, terms, staged, con_gid, bytes;
};
ILVES_HD BatchLayout batch_layout(const BatchSizes& z) {
    BatchLayout L;
    uint32_t o = (uint32_t)sizeof(BatchHead);
    L.con = o;       o = align16(o + 4u * z.nc);
    L.back = o;      o = align16(o + 8u * z.nc);
    L.lvl_piv = o;   o = align16(o + 2u * (z.nlevel + 1));
    L.lvl_hdr = o;   o = align16(o + 2u * (z.nlevel + 1));
    L.inc4 = o;      o = align16(o + 8u * z.na);
    L.over_ptr = o;  o = align16(o + (z.nover > 0 ? 2u * (z.nover + 1) : 0u));
    L.over = o;      o = align16(o + 2u * z.nover_inc);
    L.aslot = o;     o = align16(o + 2u * z.na);
    L.pairs = o;     o = align16(o + 4u * z.npair);
    L.hdr = o;       o = align16(o + 4u * z.nhdr);
    L.terms = o;     o = align16(o + 4u * z.nterm);
    L.staged = o;
    L.con_gid = o;   o = align16(o + 4u * z.nc);
    L.bytes = o;
    return L;
}
// Slot of pivot 0 among the values of a batched molecule.  Not before 3 na - 2 nc, so that the
// set-up's staging of x_old (24 na bytes from rf on) ends before the pivots' values, whose
// second component holds the starting multipliers by then.
ILVES_HD int32_t batch_pivot_base(int32_t na, int32_t nc, int32_t npair) {
    const int32_t st = 3 * na - 2 * nc;
    return npair > st ? npair : st;
}
// State of a batched molecule, after its program.  Float64-class values (float64, or
// float-float pairs of the same size) take 8 bytes; lp_bytes is the factor element size.  Atom
// arrays x (SoA), w (2 w; the float-float mode: w), wl (4 w; one more atom, of zero weight, for
// the fill); per constraint rho (SoA; with `disp`, the float-float mode, only its low float
// parts), s (`disp`: x_unc,i - x_unc,j), d2, lam, the rows rhof (.w = 4 (w_i + w_j)) and rf; c the
// factor, two values to a slot: pairs, pivots (1 / pivot, solve vector), the zero, and three
// slots that substitution may read past a row's end.
struct BatchState { uint32_t x, w, wl, rho, s, d2, lam, rhof, rf, c, bytes; };
ILVES_HD BatchState batch_state(uint32_t na, uint32_t nc, uint32_t npair, uint32_t lp_bytes, bool disp) {
    BatchState S;
    uint32_t o = 0;
    S.x = o;    o = align16(o + 24u * na);
    S.w = o;    o = align16(o + 8u * (na + 1));
    S.wl = o;   o = align16(o + lp_bytes * (na + 1));
    S.rho = o;  o = align16(o + (disp ? 12u : 24u) * nc);
    S.s = o;    o = align16(o + (disp ? 24u * nc : 0u));
    S.d2 = o;   o = align16(o + 8u * nc);
    S.lam = o;  o = align16(o + 8u * nc);
    S.rhof = o; o = align16(o + 4u * lp_bytes * nc);
    S.rf = o;   o = align16(o + 4u * lp_bytes * nc);
    S.c = o;
    o = align16(o + 2u * lp_bytes * ((uint32_t)batch_pivot_base((int32_t)na, (int32_t)nc, (int32_t)npair) + nc + 4u));
    S.bytes = o;
    return S;
}

// Program of a large molecule, in global memory.  Partitioned molecules add the Schur-contribution tables (see SepInfo, Contrib).
struct ProgLayout {
    uint32_t seg, con_atoms, piv, lvl_task, lvl_piv, inc_ptr, inc, tasks, terms, sep_info, cptr, cent, pprog_off,
        pprog, con_gid, bytes;
};

// Partitioned molecules: the separator block's entries receive the terms of interior
// pivots (the Schur complement contributions) from the parts that own those pivots.
// Part q computes, for each Contrib entry of its list, the partial sums over terms
// [e0, e1) of task `task` (all with the earlier pivot m inside part q):
//   sum L[row,m] inv_m U[m,col]   and, for a DIAG task, sum L[row,m] inv_m y_m
// into slot `slot` (0 or 1) of that task.  The separator phase then subtracts the
// `ngroups` slots and the remaining terms [b_start, end) itself.
struct SepInfo { uint32_t b_start, ngroups; };
struct Contrib { uint32_t task, slot, e0, e1; };

// Part programs (partitioned molecules): each part's factorisation and back substitution
// again, in 16-bit part-local indices, small enough to stage in the shared memory of the
// part's CTA.  Positions, task slots and atoms count from the part's first; a row or
// column that is a separator is coded 0x8000 | k, k indexing the part's separator table
// (global positions); a fill entry's atom is 0xFFFF.  Terms are stored thread by thread
// for a team of kPartThreads, like the warp programs.  Layout (16-byte aligned sections):
//   header    PartProgHeader
//   lvl_piv   uint16 x (nlev + 1)       local positions of each level
//   lvl_task  uint16 x (nlev + 1)       local task slots of each level
//   septab    int32  x nsep             global positions of the separators referenced
//   lane_term uint32 x kPartThreads     first term of each team thread
//   piv       uint32 x np               U-row slot | (number of U-row entries << 16)
//   aorder    uint16 x na               the part's atoms in update order (decreasing degree)
//   tasks     uint2  x nt               (row | col << 16, atom | neg << 16 | nterm << 24)
//   terms     uint2  x nterm            (l | u << 16, m)
//   contribs  uint2  x ncontrib         the part's Schur contributions (see Contrib):
//                                       (CT slot | DIAG << 31, first cterm | count << 16)
//   cterms    uint2  x ncterm           their terms, (l | u << 16, m)
// followed, in shared memory only, by a scratch section (not in the blob) that holds the
// separators' current and reference rows and solution values during a phase.
constexpr int kPartThreads = 256;
constexpr uint32_t kPartSep = 0x8000u, kPartNoAtom = 0xFFFFu;
struct PartProgHeader { uint32_t np, nt, na, nlev, nsep, nterm, ncontrib, ncterm; };
struct PartProgLayout {
    uint32_t lvl_piv, lvl_task, septab, lane_term, piv, aorder, tasks, terms, contribs, cterms, scratch, bytes;
};
constexpr uint32_t kPartSepScratch = 2u * 32u + 8u;  // per separator: two rows and a value (float64)
ILVES_HD PartProgLayout part_prog_layout(uint32_t np, uint32_t nt, uint32_t na, uint32_t nlev, uint32_t nsep,
                                         uint32_t nterm, uint32_t ncontrib, uint32_t ncterm) {
    PartProgLayout L;
    uint32_t o = (uint32_t)sizeof(PartProgHeader);
    L.lvl_piv = o;   o = align16(o + 2u * (nlev + 1));
    L.lvl_task = o;  o = align16(o + 2u * (nlev + 1));
    L.septab = o;    o = align16(o + 4u * nsep);
    L.lane_term = o; o = align16(o + 4u * (uint32_t)kPartThreads);
    L.piv = o;       o = align16(o + 4u * np);
    L.aorder = o;    o = align16(o + 2u * na);
    L.tasks = o;     o = align16(o + 8u * nt);
    L.terms = o;     o = align16(o + 8u * nterm);
    L.contribs = o;  o = align16(o + 8u * ncontrib);
    L.cterms = o;    o = align16(o + 8u * ncterm);
    L.scratch = o;   o = align16(o + kPartSepScratch * nsep);
    L.bytes = o;
    return L;
}

// Separator program (partitioned molecules): the separator block's factorisation in
// indices local to the block (positions from the first separator, task slots from the
// first separator task), staged in the shared memory of the CTA that solves the block.
// A term whose eliminated pivot is a separator is (l | u << 16, m); one whose pivot is an
// interior pivot (beyond the parts' contribution slots) is (0xFFFFFFFF, global term index).
//   header    SepProgHeader
//   lvl_piv   uint16 x (nlev + 1)
//   lvl_task  uint16 x (nlev + 1)
//   piv       uint32 x nsep             U-row slot | (number of U-row entries << 16)
//   tasks     uint2  x (nt + 1)         (row | col << 16, first term | ngroups << 30), sentinel
//   terms     uint2  x nterm
struct SepProgHeader { uint32_t nsep, nt, nlev, nterm; };
struct SepProgLayout { uint32_t lvl_piv, lvl_task, piv, tasks, terms, bytes; };
constexpr uint32_t kSepInterior = 0xFFFFFFFFu;
ILVES_HD SepProgLayout sep_prog_layout(uint32_t nsep, uint32_t nt, uint32_t nlev, uint32_t nterm) {
    SepProgLayout L;
    uint32_t o = (uint32_t)sizeof(SepProgHeader);
    L.lvl_piv = o;   o = align16(o + 2u * (nlev + 1));
    L.lvl_task = o;  o = align16(o + 2u * (nlev + 1));
    L.piv = o;       o = align16(o + 4u * nsep);
    L.tasks = o;     o = align16(o + 8u * (nt + 1));
    L.terms = o;     o = align16(o + 8u * nterm);
    L.bytes = o;
    return L;
}

// Overlapping domains (OPM, supplement Sec. 3): one connected system solved as a
// quasi-Newton iteration over domains.  Atoms are cut into contiguous parts; part d owns
// the constraints whose smaller atom it holds, and its domain adds the atoms within
// `overlap` edges of its atoms; the domain's system is A restricted to the constraints
// between domain atoms, factorised and solved by one CTA in shared memory, and only the
// owned constraints' corrections are kept.  Blob of an OPM molecule:
//   OpmBlobHeader, dom_off uint32 x (n_dom + 1) (byte offsets of the domain programs from
//   the blob start), con_gid int32 x nc (global id of each molecule-local constraint), then
//   the domain programs.  Domain program (indices local to the domain, 16-byte aligned
//   sections):
//   header    DomProgHeader
//   lvl_piv   uint16 x (nlev + 1)       positions of each level
//   lvl_task  uint16 x (nlev + 1)       task slots of each level
//   lane_term uint32 x kPartThreads     first term of each team thread
//   piv       uint32 x nc               U-row slot | (number of U-row entries << 16)
//   con       uint32 x nc               local atoms i | j << 16 of position p
//   con_ml    uint32 x nc               molecule-local constraint | (owned << 31)
//   atom_ml   int32  x na               molecule-local atom of each domain atom (owned atoms
//                                       first, in order, then the halo)
//   inc_ptr   uint16 x (na_own + 1)     incidence of the owned atoms
//   inc       uint16 x n_inc            position p << 1 | (atom is the second atom of p)
//   aorder    uint16 x na_own           owned atoms in update order (decreasing degree)
//   tasks     uint2  x nt               (row | col << 16, atom | neg << 16 | nterm << 24)
//   terms     uint32 x nterm            l | u << 11 | m << 22 (DomTerm), thread by thread
// so a domain has fewer than 2048 task slots and 1024 constraints.
struct DomTerm {
    static constexpr uint32_t kMaxSlots = 2048, kMaxCons = 1024;
    static ILVES_HD uint32_t l(uint32_t t) { return t & 0x7FFu; }
    static ILVES_HD uint32_t u(uint32_t t) { return (t >> 11) & 0x7FFu; }
    static ILVES_HD uint32_t m(uint32_t t) { return t >> 22; }
    static ILVES_HD uint32_t make(uint32_t l, uint32_t u, uint32_t m) { return l | (u << 11) | (m << 22); }
};
struct OpmBlobHeader { uint32_t n_dom, overlap, pad0, pad1; };
struct DomProgHeader { uint32_t na, na_own, nc, nt, nterm, nlev, n_inc, pad; };
struct DomProgLayout {
    uint32_t lvl_piv, lvl_task, lane_term, piv, con, con_ml, atom_ml, inc_ptr, inc, aorder, tasks, terms, bytes;
};
ILVES_HD DomProgLayout dom_prog_layout(uint32_t na, uint32_t na_own, uint32_t nc, uint32_t nt, uint32_t nterm,
                                       uint32_t nlev, uint32_t n_inc) {
    DomProgLayout L;
    uint32_t o = (uint32_t)sizeof(DomProgHeader);
    L.lvl_piv = o;   o = align16(o + 2u * (nlev + 1));
    L.lvl_task = o;  o = align16(o + 2u * (nlev + 1));
    L.lane_term = o; o = align16(o + 4u * (uint32_t)kPartThreads);
    L.piv = o;       o = align16(o + 4u * nc);
    L.con = o;       o = align16(o + 4u * nc);
    L.con_ml = o;    o = align16(o + 4u * nc);
    L.atom_ml = o;   o = align16(o + 4u * na);
    L.inc_ptr = o;   o = align16(o + 2u * (na_own + 1));
    L.inc = o;       o = align16(o + 2u * n_inc);
    L.aorder = o;    o = align16(o + 2u * na_own);
    L.tasks = o;     o = align16(o + 8u * nt);
    L.terms = o;     o = align16(o + 4u * nterm);
    L.bytes = o;
    return L;
}
// Shared-memory state of a domain behind its program (Mode sizes: hp = 8 bytes of the
// float64 class, lp = factor element size): X (SoA, 3 na float64), WL (na + 1, lp; the
// extra atom has zero weight), W (na_own float64), RHO (SoA, 3 nc float64), RHOF and RF
// (nc x 4 lp; .w = w_i + w_j and 1 / pivot), D2 (nc float64), Y (nc lp), V (nt lp).  With
// `disp` (float-float mode) X holds displacements x - x_unc, RHO only the low float parts
// of rho (the high parts are RHOF.xyz) and SK the differences x_unc,i - x_unc,j (SoA, 3 nc
// float-float pairs); the float64-class values are float-float pairs in the same 8 bytes.
struct DomStateLayout { uint32_t x, wl, w, rho, sk, rhof, rf, d2, y, v, bytes; };
ILVES_HD DomStateLayout dom_state_layout(uint32_t na, uint32_t na_own, uint32_t nc, uint32_t nt, uint32_t lp,
                                         bool disp = false) {
    DomStateLayout S;
    uint32_t o = 0;
    S.x = o;    o = align16(o + 24u * na);
    S.wl = o;   o = align16(o + lp * (na + 1));
    S.w = o;    o = align16(o + 8u * na_own);
    S.rho = o;  o = align16(o + (disp ? 12u : 24u) * nc);
    S.sk = o;   o = align16(o + (disp ? 24u * nc : 0u));
    S.rhof = o; o = align16(o + 4u * lp * nc);
    S.rf = o;   o = align16(o + 4u * lp * nc);
    S.d2 = o;   o = align16(o + 8u * nc);
    S.y = o;    o = align16(o + lp * nc);
    S.v = o;    o = align16(o + lp * nt);
    S.bytes = o;
    return S;
}

// Segment table (n_seg + 1 rows of {first position, first level-table entry, first atom}):
// one segment for an ordinary molecule; for a partitioned molecule one per part, then the
// separators (constraints between parts), whose atom range is empty.
struct SegRow { int32_t piv, lvl, atom; };

ILVES_HD ProgLayout prog_layout(uint32_t na, uint32_t nc, uint32_t ntask, uint32_t nterm,
                                uint32_t nlevel, uint32_t n_seg = 1, uint32_t n_sept = 0, uint32_t n_cent = 0,
                                uint32_t pprog_bytes = 0) {
    ProgLayout L;
    uint32_t o = 0;
    L.seg = o;       o = align16(o + 12u * (n_seg + 1));
    L.con_atoms = o; o = align16(o + (uint32_t)sizeof(ConA) * nc);
    L.piv = o;       o = align16(o + (uint32_t)sizeof(Piv) * nc);
    L.lvl_task = o;  o = align16(o + 4u * (nlevel + 1));
    L.lvl_piv = o;   o = align16(o + 4u * (nlevel + 1));
    L.inc_ptr = o;   o = align16(o + 4u * (na + 1));
    L.inc = o;       o = align16(o + 8u * nc);
    L.tasks = o;     o = align16(o + (uint32_t)sizeof(Task) * (ntask + 1));
    L.terms = o;     o = align16(o + (uint32_t)sizeof(TermWide) * nterm);
    const bool parted = n_seg > 1;
    L.sep_info = o;  o = align16(o + (parted ? 8u * n_sept : 0u));
    L.cptr = o;      o = align16(o + (parted ? 4u * n_seg : 0u));  // n_parts + 1 = n_seg entries
    L.cent = o;      o = align16(o + (parted ? 16u * n_cent : 0u));
    L.pprog_off = o; o = align16(o + (pprog_bytes ? 4u * (n_seg + 1) : 0u));  // parts, separators, end
    L.pprog = o;     o = align16(o + pprog_bytes);
    L.con_gid = o;   o = align16(o + 4u * nc);
    L.bytes = o;
    return L;
}

// Numerical state of a large molecule, in the workspace.  Float64-class values (float64,
// or float-float pairs of the same size) take 8 bytes; lp_bytes is the factor element
// size (4 for float32, 8 for float64); 3-vectors of the factor precision take 4
// elements and use the fourth: rhof[p].w holds w_i + w_j (the weight of a DIAG entry),
// rf[p].w holds 1 / pivot p of the current factor.  Atom arrays have na + 1 entries:
// the extra atom has zero weight and is what fill entries of the pattern point at.
// With `disp` (float-float mode) the state keeps displacements x - x_unc and the
// per-constraint differences s_k = x_unc,i - x_unc,j, and rho keeps only the low
// float parts of rho (the high parts are rhof.xyz).
struct StateLayout {
    uint32_t x, w, wl, rho, s, d2, lam, rhof, y, rf, vals, bytes;
};

ILVES_HD StateLayout state_layout(uint32_t na, uint32_t nc, uint32_t ntask, uint32_t lp_bytes, bool disp) {
    StateLayout S;
    const uint32_t vp = 4u * lp_bytes;
    uint32_t o = 0;
    S.x = o;      o = align16(o + 24u * na);             // SoA: x[0..na), y[..], z[..]
    S.w = o;      o = align16(o + 8u * (na + 1));
    S.wl = o;     o = align16(o + lp_bytes * (na + 1));
    S.rho = o;    o = align16(o + (disp ? 12u : 24u) * nc);  // SoA
    S.s = o;      o = align16(o + (disp ? 24u * nc : 0u));
    S.d2 = o;     o = align16(o + 8u * nc);
    S.lam = o;    o = align16(o + 8u * nc);
    S.rhof = o;   o = align16(o + vp * nc);
    S.y = o;      o = align16(o + (lp_bytes > 4u ? lp_bytes : 4u) * nc);
    S.rf = o;     o = align16(o + vp * nc);
    S.vals = o;   o = align16(o + lp_bytes * ntask);
    S.bytes = o;
    return S;
}

constexpr size_t kStaticScratchBytes = size_t(16) << 20;  // see ilves_solve_static_scratch

// One molecule as the kernels see it.
struct MolDesc {
    int64_t blob_off;    // byte offset of the program blob in the blob buffer (16-B aligned)
    int64_t work_off;    // large path: byte offset of the numerical state in the workspace
    int32_t atom_base;   // first global atom if the molecule's atoms are contiguous, else -1
    int32_t gid_off;     // offset of this molecule's global atom ids in atom_gid[]
    int32_t mol_id;      // output index (molecules ordered by smallest atom)
    int32_t nterm;
    int32_t ntask;
    int32_t na, nc;
    int32_t nlevel;  // level-table entries - 1 (for one segment: its number of levels)
    int32_t n_seg;   // 1, or parts + 1 for a partitioned molecule
    int32_t n_sept;  // partitioned: tasks of the separator segment (they are the last ones)
    int32_t n_cent;  // partitioned: Schur contribution entries over all parts
    int32_t pprog_bytes;  // partitioned: bytes of the segment programs (parts, then separators)
    int32_t opm;          // overlapping domains: overlap depth (0 = not solved by domains)
    int32_t n_hdr, n_over, n_over_inc, n_pair;  // batched: see BatchSizes (nterm: the completed terms)
};
ILVES_HD BatchSizes batch_sizes(const MolDesc& D) {
    return BatchSizes{D.na, D.nc, D.n_pair, D.nlevel, D.n_hdr, D.nterm, D.n_over, D.n_over_inc};
}

}  // namespace ilves

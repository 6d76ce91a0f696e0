// batched.cuh -- one molecule of the batched kernel, solved by the team of a slot with its
// program (BatchLayout) and state in shared memory.  Included by solve.cu.
//
// What bounds it.  A molecule's solve is a chain of dependent passes (per Newton step: the
// violations, the assembly, about eight elimination levels, as many substitution levels, the
// position update) on a team that shares its SM with seven others.  A warp issues an
// instruction of such a chain every five cycles or so, so a pass costs what its busiest warp
// has to issue; and a float64 instruction holds its scheduler's pipe for 66 cycles whatever
// the number of active lanes.  Hence:
//  - A's pattern is symmetric, so the entries U[j,q] and L[q,j] are one item of two values: they
//    share the pivots of their terms, their term words, and two 2-value loads serve both.
//    A pivot and its right-hand side are another such item (its second sum is the forward
//    solve), so every lane of a level runs the same instructions;
//  - in float64, where the two sums would be two float64 instructions, the two lanes of a pair
//    take one each;
//  - the whole matrix is assembled in one pass, so a level has one round of independent loads
//    in front of its sums, and a lane reads the program words of its next item while it holds
//    the current one;
//  - levels of at most 32 items or pivots, the last ones, belong to the team's first warp
//    alone, which orders them with warp barriers while the others wait;
//  - terms come in pairs (the odd one is completed by a zero), incidences four to a word pair;
//  - no pass is unrolled.  Eight teams are in different passes at any time, and both classes of
//    teams and both kinds of solve have code of their own, so the passes' code has to stay in the
//    instruction caches: unrolled four times by the compiler, 1.5 (float-float) and 0.6 (mixed)
//    of a warp's stall cycles an issue were waits for instructions, 1.7 and 0.9 with one-warp teams
//    beside the others; now 0.7 and 0.3 (135 -> 127 us mixed, 151 -> 129 us float-float).  The copies
//    of inputs and outputs are left to the compiler: rolled, every store of a multiplier waits for
//    its index, which costs a batch on page-locked host buffers 5 % (4096 trees: 288 against 268 us).
// Measured (4096 trees of 20-200 atoms, 96-thread teams; one task per entry and one atom per lane
// before): mixed 162.0 -> 132.4 us, float64 541 -> 417 us; 8192 trees of 20-50 atoms on one-warp
// teams 121.7 -> 95.4 us.  The mixed batch issues on every other cycle (its teams wait on one
// another and on shared memory); the float64 batch fills three quarters of the float64 pipe.
#pragma once

namespace ilves {

template <class Mode>
struct BatchMol {
    using LP = typename Mode::LP;
    using V4 = typename Mode::V4;
    struct alignas(2 * sizeof(LP)) V2 { LP x, y; };
    static constexpr bool DF = Mode::df;
    static constexpr bool kF32 = sizeof(LP) == 4;
    int na, nc, npair, nlevel, nover, zero;
    const BatchHead* head;
    const uint32_t* con;  // local atoms i | j << 16 of each position
    const uint2* back;    // substitution record of each pivot (BackWord)
    const uint16_t *lvl_piv, *lvl_hdr;
    const uint2* inc4;    // first four incidences of each atom
    const uint16_t *over_ptr, *over, *aslot;
    const uint32_t* pairs;  // PairWord of every off-diagonal pair
    const uint32_t* hdr;    // HeadWord of the items that have terms
    const uint2* terms;     // two TermWords
    const int32_t* con_gid;  // global memory
    double *X, *W, *RHO, *SK, *D2, *LAM;
    float* RHOL;
    LP* WL;
    V4 *RHOF, *RF;  // RHOF[p].w = 4 (w_i + w_j)
    V2* C;          // pair k: (U[j,q], L[q,j]); then, at PV, pivot p: (1 / pivot, solve vector);
    V2* PV;         // then the zero
    double* STG;    // x_old gathered AoS (set-up only; aliases RF and the pairs)
    const MolDesc& D;
    const SolveArgs& A;
    float tolf;

    __device__ __forceinline__ BatchMol(const MolDesc& d, const BatchLayout& L, uint8_t* slice, const SolveArgs& a,
                                        const uint8_t* gprog)
        : D(d), A(a) {
        na = d.na;
        nc = d.nc;
        npair = d.n_pair;
        nlevel = d.nlevel;
        nover = d.n_over;
        tolf = (float)a.tol;
        const int pbase = batch_pivot_base(na, nc, npair);
        zero = pbase + nc;
        head = reinterpret_cast<const BatchHead*>(slice);
        con = reinterpret_cast<const uint32_t*>(slice + L.con);
        back = reinterpret_cast<const uint2*>(slice + L.back);
        lvl_piv = reinterpret_cast<const uint16_t*>(slice + L.lvl_piv);
        lvl_hdr = reinterpret_cast<const uint16_t*>(slice + L.lvl_hdr);
        inc4 = reinterpret_cast<const uint2*>(slice + L.inc4);
        over_ptr = reinterpret_cast<const uint16_t*>(slice + L.over_ptr);
        over = reinterpret_cast<const uint16_t*>(slice + L.over);
        aslot = reinterpret_cast<const uint16_t*>(slice + L.aslot);
        pairs = reinterpret_cast<const uint32_t*>(slice + L.pairs);
        hdr = reinterpret_cast<const uint32_t*>(slice + L.hdr);
        terms = reinterpret_cast<const uint2*>(slice + L.terms);
        con_gid = reinterpret_cast<const int32_t*>(gprog + L.con_gid);
        uint8_t* st = slice + L.staged;
        const BatchState S = batch_state(na, nc, npair, sizeof(LP), DF);
        X = reinterpret_cast<double*>(st + S.x);
        W = reinterpret_cast<double*>(st + S.w);
        WL = reinterpret_cast<LP*>(st + S.wl);
        RHO = reinterpret_cast<double*>(st + S.rho);
        RHOL = reinterpret_cast<float*>(st + S.rho);
        SK = reinterpret_cast<double*>(st + S.s);
        D2 = reinterpret_cast<double*>(st + S.d2);
        LAM = reinterpret_cast<double*>(st + S.lam);
        RHOF = reinterpret_cast<V4*>(st + S.rhof);
        RF = reinterpret_cast<V4*>(st + S.rf);
        C = reinterpret_cast<V2*>(st + S.c);
        PV = C + pbase;
        STG = reinterpret_cast<double*>(st + S.rf);
    }
    // global atom of atom slot o (the molecule's atoms in ascending global order); local atom a
    // sits in the slot whose entry of aslot is a (local atoms are ordered by degree)
    __device__ __forceinline__ int64_t slot_gid(int o) const {
        return D.atom_base >= 0 ? (int64_t)D.atom_base + o : (int64_t)A.atom_gid[D.gid_off + o];
    }
    __device__ __forceinline__ int32_t gid_of_con(int p) const { return __ldg(con_gid + p); }

    // ---- S1: one batch of asynchronous gathers, then local passes.  x_old -> STG (AoS); x_unc
    //      -> X (SoA; AoS in the float-float mode, where X is free until the displacements
    //      start); inv_mass -> W, d -> D2, lambda0 -> LAM as raw values.  The reads run over atom
    //      slots, so consecutive lanes read consecutive addresses.
    __device__ __forceinline__ void s1_gather(int r0, int ts) {
        for (int p = r0; p < nc; p += ts) {
            const int32_t g = gid_of_con(p);
            cp_async8(D2 + p, A.d + g);
            if (A.lambda0 && !A.start_diag) cp_async4(LAM + p, A.lambda0 + g);
        }
        for (int e = r0; e < 3 * na; e += ts) {
            const int o = e / 3, c = e - 3 * o, a = (int)aslot[o];
            const int64_t g = 3 * slot_gid(o) + c;
            cp_async8(STG + 3 * a + c, A.x_old + g);
            cp_async8(DF ? X + 3 * a + c : X + c * na + a, A.x_unc + g);
        }
        for (int o = r0; o < na; o += ts) cp_async8(W + aslot[o], A.inv_mass + slot_gid(o));
        cp_async_wait_all();
    }
    // The weights are kept scaled by exact powers of two, WL = 4 w (the factor of every entry
    // of A) and, in the float64 modes, W = 2 w (that of every position update), which takes a
    // product out of each entry and an addition out of each update term without changing a bit.
    __device__ __forceinline__ void s1_atom(int a) {
        const double w = W[a];
        W[a] = DF ? as_bits(df_split(w)) : w + w;
        WL[a] = LP(4) * to_lp<LP>(w);
    }
    __device__ __forceinline__ void s1_dummy() {
        W[na] = 0.0;
        WL[na] = LP(0);
    }
    __device__ __forceinline__ void s1_constraint(int p) {
        const int i = (int)(con[p] & 0xFFFFu), j = (int)(con[p] >> 16);
        const double rx = STG[3 * i] - STG[3 * j];
        const double ry = STG[3 * i + 1] - STG[3 * j + 1];
        const double rz = STG[3 * i + 2] - STG[3 * j + 2];
        V4 v;
        v.x = to_lp<LP>(rx);
        v.y = to_lp<LP>(ry);
        v.z = to_lp<LP>(rz);
        v.w = WL[i] + WL[j];
        RHOF[p] = v;
        const double dd = D2[p];
        if constexpr (DF) {
            RHOL[p] = df_split(rx).lo;
            RHOL[nc + p] = df_split(ry).lo;
            RHOL[2 * nc + p] = df_split(rz).lo;
            D2[p] = as_bits(df_split(dd * dd));
            SK[p] = as_bits(df_split(X[3 * i] - X[3 * j]));
            SK[nc + p] = as_bits(df_split(X[3 * i + 1] - X[3 * j + 1]));
            SK[2 * nc + p] = as_bits(df_split(X[3 * i + 2] - X[3 * j + 2]));
        } else {
            RHO[p] = rx;
            RHO[nc + p] = ry;
            RHO[2 * nc + p] = rz;
            D2[p] = dd * dd;
        }
        float l0 = A.lambda0 ? *reinterpret_cast<const float*>(LAM + p) : 0.0f;
        if (A.start_diag) {  // x_unc is in X (AoS in the float-float mode, else SoA)
            float u[3];
            for (int c = 0; c < 3; ++c)
                u[c] = DF ? narrow(X[3 * i + c]) - narrow(X[3 * j + c]) : narrow(X[c * na + i]) - narrow(X[c * na + j]);
            l0 = diag_start(u[0], u[1], u[2], narrow(STG[3 * i]) - narrow(STG[3 * j]),
                            narrow(STG[3 * i + 1]) - narrow(STG[3 * j + 1]),
                            narrow(STG[3 * i + 2]) - narrow(STG[3 * j + 2]), narrow(dd),
                            0.25f * (f32_of(WL[i]) + f32_of(WL[j])));
        }
        LAM[p] = DF ? as_bits(dfloat{l0, 0.0f}) : widen(l0);
        PV[p].y = (LP)l0;
    }

    // ---- S2: violation of constraint p (float64 class), Jacobian row, right-hand side (rows =
    //      false: ILVES-F, which assembles A(x_old, x_old) from the reference rows alone)
    __device__ __forceinline__ void violation(int p, uint32_t ij, bool& conv, bool& bad, bool rows) {
        const int i = (int)(ij & 0xFFFFu), j = (int)(ij >> 16);
        V4 v;
        LP y;
        bool cv, bd;
        if constexpr (DF) {
            const dfloat rx = df_add(as_df(SK[p]), df_sub(as_df(X[i]), as_df(X[j])));
            const dfloat ry = df_add(as_df(SK[nc + p]), df_sub(as_df(X[na + i]), as_df(X[na + j])));
            const dfloat rz = df_add(as_df(SK[2 * nc + p]), df_sub(as_df(X[2 * na + i]), as_df(X[2 * na + j])));
            const dfloat d2 = as_df(D2[p]);
            // |r|^2 - d^2: exact products of the high words, two-sums of the big terms, every
            // rounding error collected in a small tail
            const float px = __fmul_rn(rx.hi, rx.hi), ex = __fmaf_rn(rx.hi, rx.hi, -px);
            const float py = __fmul_rn(ry.hi, ry.hi), ey = __fmaf_rn(ry.hi, ry.hi, -py);
            const float pz = __fmul_rn(rz.hi, rz.hi), ez = __fmaf_rn(rz.hi, rz.hi, -pz);
            float s1, e1, s2, e2, s3, e3;
            two_sum(px, py, s1, e1);
            two_sum(s1, pz, s2, e2);
            two_sum(s2, -d2.hi, s3, e3);
            float cross = __fmul_rn(rx.hi, rx.lo);
            cross = __fmaf_rn(ry.hi, ry.lo, cross);
            cross = __fmaf_rn(rz.hi, rz.lo, cross);
            const float tail = ((ex + ey) + (ez + e1)) + ((e2 + e3) - d2.lo) + (cross + cross);
            const float sg = s3 + tail;
            cv = fabsf(sg) <= tolf * d2.hi;
            bd = nonfinite(sg);
            v.x = rx.hi;
            v.y = ry.hi;
            v.z = rz.hi;
            y = sg;
        } else {
            const double d2 = D2[p];
            const double rx = X[i] - X[j], ry = X[na + i] - X[na + j], rz = X[2 * na + i] - X[2 * na + j];
            const double sg = fma(rx, rx, fma(ry, ry, fma(rz, rz, -d2)));
            cv = within(sg, A.tol, d2);
            bd = nonfinite(sg);
            v.x = to_lp<LP>(rx);
            v.y = to_lp<LP>(ry);
            v.z = to_lp<LP>(rz);
            y = to_lp<LP>(sg);
        }
        v.w = LP(0);
        conv = conv && cv;
        bad = bad || bd;
        PV[p].y = y;
        if (rows) RF[p] = v;
    }

    // ---- S3: every entry a = 4 s s' w_atom r_row . rho_col of A: the pivots (w = w_i + w_j),
    //      those of level 0 already inverted, then the pairs.  R: the Jacobian rows, or the
    //      reference rows (ILVES-F).
    __device__ __forceinline__ static LP dot(const V4& r, const V4& p) { return r.x * p.x + r.y * p.y + r.z * p.z; }
    __device__ __forceinline__ void assemble(const V4* R, int r0, int ts, bool& singular) {
        if (r0 == 0) C[zero] = V2{LP(0), LP(0)};
        const int n0 = lvl_piv[1];
#pragma unroll 1
        for (int p = r0; p < nc; p += ts) {
            const V4 rr = R[p], pp = RHOF[p];
            LP a = pp.w * dot(rr, pp);
            if (p < n0) {
                singular = singular | pivot_vanished<Mode>(a, a);
                a = lp_rcp(a);
            }
            PV[p].x = a;
        }
#pragma unroll 1
        for (int k = r0; k < npair; k += ts) {
            const uint32_t w = pairs[k];
            const int j = (int)PairWord::row(w), q = (int)PairWord::col(w);
            const V4 rj = R[j], pq = RHOF[q], rq = R[q], pj = RHOF[j];
            const LP wa = WL[PairWord::atom(w)], c = PairWord::neg(w) ? -wa : wa;
            C[k] = V2{c * dot(rj, pq), c * dot(rq, pj)};
        }
    }

    // ---- S4 + forward S5, levels [l0, l1) (entered after a barrier; one after every level).
    //      Item k: its two values minus its terms',
    //        U[j,q] -= (L[j,m] inv_m) U[m,q],   L[q,j] -= (L[q,m] inv_m) U[m,j],
    //      with a = (U, L)[m,j], b = (U, L)[m,q]; pivot j (a = b) instead
    //        d_j -= (L[j,m] inv_m) U[m,j],      -(L[j,m] inv_m) y_m, added to y_j,
    //      and d_j is inverted.  kW lanes take part; in float64 the two lanes of a pair share an
    //      item and take one sum each, and every level begins by scaling the previous level's
    //      L[.,m] with inv_m, once instead of in every term: half the float64 instructions of
    //      the terms for one more barrier a level (the products and their order are the same).
    //      kForward (ILVES-F with its stored factor): y alone.
    //      kOne: no level has more items than kW lanes hold.
    template <int kW, bool kForward, bool kOne, class Sync>
    __device__ __forceinline__ void eliminate(int l0, int l1, int r, bool& singular, Sync sync) {
        constexpr int kI = kF32 ? kW : kW / 2;
        const int g = kF32 ? r : r >> 1;
        const bool second = !kF32 && (r & 1);
        int hb = lvl_hdr[l0], he = lvl_hdr[l0 + 1], hn = lvl_hdr[min(l0 + 2, l1)];
        uint32_t h = 0u;
        uint2 x = make_uint2(0u, 0u);
        if (hb + g < he) {
            h = hdr[hb + g];
            x = terms[HeadWord::first(h)];
        }
        for (int l = l0; l < l1; ++l) {
            const int hq = lvl_hdr[min(l + 3, l1)];  // levels: this [hb, he), then [he, hn), [hn, hq)
            if constexpr (!kF32 && !kForward) {
                const int s1 = (int)BackWord::slot(back[lvl_piv[l]]);
#pragma unroll 1
                for (int k = (int)BackWord::slot(back[lvl_piv[l - 1]]) + r; k < s1; k += kW)
                    C[k].y *= PV[PairWord::row(pairs[k])].x;
                sync();
            }
            int k = hb + g;
            bool mine = k < he;
            if (!mine && he + g < hn) {
                h = hdr[he + g];
                x = terms[HeadWord::first(h)];
            }
            while (mine) {
                const bool diag = HeadWord::diag(h);
                const int s = (int)HeadWord::slot(h), nm = (int)HeadWord::more(h);
                const uint2* tq = terms + HeadWord::first(h) + 1;  // the item's further term pairs
                const V2 v = C[s];
                LP e1, e2;  // float64: e1 alone, the sum of this lane
                if constexpr (kF32) {
                    e1 = v.x;
                    e2 = diag ? LP(0) : v.y;
                } else {
                    e1 = second ? (diag ? LP(0) : v.y) : v.x;
                    e2 = LP(0);
                }
                auto term = [&](uint32_t w) {
                    if constexpr (kF32) {
                        const V2 pm = PV[TermWord::m(w)];
                        const V2 a = C[TermWord::a(w)], b = C[TermWord::b(w)];
                        const LP ua = diag ? pm.y : a.x;
                        if constexpr (!kForward) e1 -= (a.y * pm.x) * b.x;
                        e2 -= (b.y * pm.x) * ua;
                    } else {
                        const LP lv = C[second ? TermWord::b(w) : TermWord::a(w)].y;
                        LP uv = C[second ? TermWord::a(w) : TermWord::b(w)].x;
                        if (diag && second) uv = PV[TermWord::m(w)].y;
                        e1 -= lv * uv;
                    }
                };
                const uint2 xc = x;
                k += kI;
                mine = !kOne && k < he;
                const int kn = mine ? k : he + g;
                const bool more = kn < (mine ? he : hn);
                uint32_t h2 = h;
                if (more) h2 = hdr[kn];
                x = *tq;  // (unused past the item's last pair; stays in the slice)
                if (!kForward || diag) {
                    term(xc.x);
                    term(xc.y);
#pragma unroll 1
                    for (int q = 0; q < nm; ++q) {
                        const uint2 xn = x;
                        x = *++tq;
                        term(xn.x);
                        term(xn.y);
                    }
                }
                h = h2;
                if (more) x = terms[HeadWord::first(h)];
                if constexpr (kF32) {
                    if (diag) {
                        V2 o = v;
                        if constexpr (!kForward) {
                            singular = singular | pivot_vanished<Mode>(e1, v.x);
                            o.x = lp_rcp(e1);
                        }
                        o.y = v.y + e2;
                        C[s] = o;
                    } else if constexpr (!kForward) {
                        C[s] = V2{e1, e2};
                    }
                } else if (second) {
                    if (diag) C[s].y = v.y + e1;
                    else if constexpr (!kForward) C[s].y = e1;
                } else if constexpr (!kForward) {
                    if (diag) {
                        singular = singular | pivot_vanished<Mode>(e1, v.x);
                        e1 = lp_rcp(e1);
                    }
                    C[s].x = e1;
                }
            }
            sync();
            hb = he;
            he = hn;
            hn = hq;
        }
    }

    // ---- backward S5, delta_p = inv_p (y_p - sum_q U[p,q] delta_q), levels l1 - 1 down to l0
    //      (entered after a barrier; one after every level but level 0).  A lane reads its next
    //      pivot's record, right-hand side and row of U, all final, ahead of the barrier that
    //      ends the level, so only the other pivots' values are read after it.
    struct Ahead {
        uint2 rec;
        V2 v;
        LP u[4];
    };
    __device__ __forceinline__ void fetch_values(Ahead& o, int p) const {
        const V2* row = C + BackWord::slot(o.rec);
        o.v = PV[p];
#pragma unroll
        for (int k = 0; k < 4; ++k) o.u[k] = row[k].x;  // past the row's end: unused
    }
    __device__ __forceinline__ void finish_pivot(const Ahead& o, int p) {
        const int nu = (int)BackWord::n(o.rec);
        LP z[4], d = o.v.y;
#pragma unroll
        for (int k = 0; k < 4; ++k) z[k] = PV[BackWord::q(o.rec, k)].y;
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (k < nu) d -= o.u[k] * z[k];
        if (nu > 4) {
            const int us = (int)BackWord::slot(o.rec);
#pragma unroll 1
            for (int k = 4; k < nu; ++k) d -= C[us + k].x * PV[PairWord::col(pairs[us + k])].y;
        }
        PV[p].y = d * o.v.x;
    }
    template <int kW, class Sync>
    __device__ __forceinline__ void substitute(int l0, int l1, int r, Sync sync) {
        int pb = lvl_piv[l1 - 1], pe = lvl_piv[l1], pn = lvl_piv[max(l1 - 2, l0)];
        Ahead cur{};
        if (pb + r < pe) {
            cur.rec = back[pb + r];
            fetch_values(cur, pb + r);
        }
        for (int l = l1 - 1; l >= l0; --l) {
            const int pq = lvl_piv[max(l - 2, l0)];  // levels: this [pb, pe), then [pn, pb), [pq, pn)
            Ahead nxt = cur;
            const bool next = pn + r < pb;
            if (next) nxt.rec = back[pn + r];
            if (pb + r < pe) finish_pivot(cur, pb + r);
            if (next) fetch_values(nxt, pn + r);
#pragma unroll 1
            for (int p = pb + r + kW; p < pe; p += kW) {
                Ahead o;
                o.rec = back[p];
                fetch_values(o, p);
                finish_pivot(o, p);
            }
            if (l > 0) sync();
            cur = nxt;
            pe = pb;
            pb = pn;
            pn = pq;
        }
    }

    // the linear solve: levels below head->wide are the team's, the others the first warp's
    // (entered after a barrier; ends without one)
    template <class Team, bool kForward>
    __device__ __forceinline__ void solve_linear(const Team& tm, bool& singular) {
        const int r = tm.rank(), nl = nlevel;
        const auto warp_sync = [] { __syncwarp(); };
        if constexpr (Team::kWarp) {
            if (nl > 1) eliminate<32, kForward, false>(1, nl, r, singular, warp_sync);
            substitute<32>(0, nl, r, warp_sync);
        } else {
            const auto team_sync = [&] { tm.sync(); };
            const int le = kF32 ? head->wide32 : head->wide16, lb = head->wide_piv;
            if (le > 1) eliminate<Team::kSize, kForward, false>(1, le, r, singular, team_sync);
            if (r < 32) {
                if (nl > le) eliminate<32, kForward, true>(le, nl, r, singular, warp_sync);
                if (nl > lb) substitute<32>(lb, nl, r, warp_sync);
            }
            if (lb > 0) {
                tm.sync();
                substitute<Team::kSize>(0, lb, r, team_sync);
            }
        }
    }

    // ---- S6: x_a -= w_a sum_k s_k(a) 2 delta_k rho_k   (PV.y holds delta, or lambda0), one
    //      coordinate of one atom per lane: 3 na items over the lanes, atoms by decreasing
    //      degree, leave the busiest warp of a tree of 110 atoms 12 float64 instructions (one
    //      atom per lane: 21).  A predicated float64 instruction takes its slot with no lane on,
    //      so the second to fourth incidences are behind warp votes (145.6 -> 141.2 us mixed).
    //      The sum runs over the incidences in ascending position.
    //      In the mixed mode the corrections are widened to float64 once, not in every
    //      coordinate's lane: dlt is LAM for the starting multipliers, then the rows' space RF
    //      (free until the next violations), which lambda_acc fills.
    __device__ __forceinline__ static double signed64(double v, unsigned inc) {
        return __hiloint2double(__double2hiint(v) ^ (int)(inc << 31), __double2loint(v));
    }
    // The float-float mode takes a whole atom per lane: its terms are float32 instructions, of which
    // no warp has too few lanes on, and three lanes to an atom would repeat the incidence, the
    // correction and the loop (4096 / 1001 trees, diagonal start: 150.8 / 52.3 us by coordinates,
    // 148.8 / 50.1 by atoms).
    struct Sum3 { dfloat x, y, z; };
    __device__ __forceinline__ void term_df(unsigned v, Sum3& s) const {
        const int p = (int)((v >> 1) & 0xFFu);
        const float dl = (float)PV[p].y, k = (v & 1u) ? -(dl + dl) : (dl + dl);
        const V4 hi = RHOF[p];
        s.x = df_add(s.x, df_mul_f(dfloat{(float)hi.x, RHOL[p]}, k));
        s.y = df_add(s.y, df_mul_f(dfloat{(float)hi.y, RHOL[nc + p]}, k));
        s.z = df_add(s.z, df_mul_f(dfloat{(float)hi.z, RHOL[2 * nc + p]}, k));
    }
    __device__ __forceinline__ void update_df(int r0, int ts) {
#pragma unroll 1
        for (int a = r0; a < na; a += ts) {
            const uint2 v = inc4[a];
            const unsigned v1 = v.x >> 16, v2 = v.y & 0xFFFFu, v3 = v.y >> 16;
            Sum3 s{{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
            term_df(v.x, s);
            if (!(v1 & kNoInc)) term_df(v1, s);
            if (!(v2 & kNoInc)) term_df(v2, s);
            if (!(v3 & kNoInc)) term_df(v3, s);
            if (a < nover)
#pragma unroll 1
                for (int e = over_ptr[a]; e < over_ptr[a + 1]; ++e) term_df(over[e], s);
            const dfloat w = as_df(W[a]);
            X[a] = as_bits(df_sub(as_df(X[a]), df_mul(w, s.x)));
            X[na + a] = as_bits(df_sub(as_df(X[na + a]), df_mul(w, s.y)));
            X[2 * na + a] = as_bits(df_sub(as_df(X[2 * na + a]), df_mul(w, s.z)));
        }
    }
    template <int kStride>
    __device__ __forceinline__ void update(const double* dlt, int r0, int ts) {
        const int n = 3 * na;
        uint2 rec = make_uint2(0u, 0u);
        if (r0 < n) rec = inc4[r0 / 3];
#pragma unroll 1
        for (int q = r0; q < n; q += ts) {
            const int a = q / 3, c = q - 3 * a;
            const uint2 v = rec;
            if (q + ts < n) rec = inc4[(q + ts) / 3];
            double* xp = X + c * na + a;
            const unsigned v1 = v.x >> 16, v2 = v.y & 0xFFFFu, v3 = v.y >> 16;
            // the four products' operands first, then the float64 chain
            const int p0 = (int)((v.x >> 1) & 0xFFu), p1 = (int)((v1 >> 1) & 0xFFu);
            const int p2 = (int)((v2 >> 1) & 0xFFu), p3 = (int)((v3 >> 1) & 0xFFu);
            const double* rho = RHO + c * nc;
            const double d0 = dlt[kStride * p0], d1 = dlt[kStride * p1], d2 = dlt[kStride * p2],
                         d3 = dlt[kStride * p3];
            const double h0 = rho[p0], h1 = rho[p1], h2 = rho[p2], h3 = rho[p3];
            const double w = W[a], x = *xp;
            double s = fma(signed64(d0, v.x), h0, 0.0);
            const unsigned act = __activemask();
            if (__any_sync(act, !(v1 & kNoInc))) {
                if (!(v1 & kNoInc)) s = fma(signed64(d1, v1), h1, s);
                if (__any_sync(act, !(v2 & kNoInc))) {
                    if (!(v2 & kNoInc)) s = fma(signed64(d2, v2), h2, s);
                    if (__any_sync(act, !(v3 & kNoInc))) {
                        if (!(v3 & kNoInc)) s = fma(signed64(d3, v3), h3, s);
                    }
                }
            }
            if (a < nover)
#pragma unroll 1
                for (int e = over_ptr[a]; e < over_ptr[a + 1]; ++e) {
                    const unsigned o = over[e];
                    const int p = (int)((o >> 1) & 0xFFu);
                    s = fma(signed64(dlt[kStride * p], o), rho[p], s);
                }
            *xp = fma(-w, s, x);
        }
    }
    __device__ __forceinline__ void lambda_acc(int p) {
        if constexpr (DF) {
            LAM[p] = as_bits(df_add_f(as_df(LAM[p]), (float)PV[p].y));
        } else {
            const double dl = to_hp(PV[p].y);
            LAM[p] = LAM[p] + dl;
            if constexpr (kF32) reinterpret_cast<double*>(RF)[2 * p] = dl;
        }
    }
    __device__ __forceinline__ const double* corrections() const {
        return reinterpret_cast<const double*>(kF32 ? (const void*)RF : (const void*)&PV[0].y);
    }

    // ---- S7: the positions, one coordinate per lane in global order; the multipliers.  The
    //      float-float mode adds x_unc, which it reads again: first, all of a lane's coordinates at
    //      once (into the rows' space, free by now), since a read behind each write is a
    //      round trip each, over the host link a long one (x_out may be x_unc): 2500 trees on
    //      page-locked buffers 238 -> 210 us.
    __device__ __forceinline__ void out_atoms(int r0, int ts) {
        if constexpr (DF) {
            for (int e = r0; e < 3 * na; e += ts) cp_async8(STG + e, A.x_unc + 3 * slot_gid(e / 3) + e % 3);
            cp_async_wait_all();
        }
        for (int e = r0; e < 3 * na; e += ts) {
            const int o = e / 3, c = e - 3 * o, a = (int)aslot[o];
            const int64_t g = 3 * slot_gid(o) + c;
            if constexpr (DF) A.x_out[g] = STG[e] + df_join(as_df(X[c * na + a]));
            else A.x_out[g] = X[c * na + a];
        }
    }
    __device__ __forceinline__ void out_lambda(int p) {
        const double l = LAM[p];
        A.lambda_out[gid_of_con(p)] = DF ? df_join(as_df(l)) : l;
    }
};

template <class Mode, class Team>
__device__ void solve_batched(const Team& tm, const MolDesc& D, const BatchLayout& L, uint8_t* slice,
                              const SolveArgs& A, const uint8_t* gprog) {
    BatchMol<Mode> M(D, L, slice, A, gprog);
    const int na = M.na, nc = M.nc, r0 = tm.rank(), ts = Team::kSize;
    // ---- S1
    M.s1_gather(r0, ts);
    tm.sync();
#pragma unroll 1
    for (int a = r0; a < na; a += ts) M.s1_atom(a);
    if (r0 == 0) M.s1_dummy();
    tm.sync();
#pragma unroll 1
    for (int p = r0; p < nc; p += ts) M.s1_constraint(p);
    tm.sync();
    if constexpr (Mode::df) {  // displacements start at zero
#pragma unroll 1
        for (int q = r0; q < 3 * na; q += ts) M.X[q] = 0.0;
        tm.sync();
    }
    if (A.has_start()) {  // x = x_unc - M^-1 G(x_old)^T lambda0
        if constexpr (Mode::df) M.update_df(r0, ts);
        else if constexpr (sizeof(typename Mode::LP) == 8) M.template update<2>(M.corrections(), r0, ts);
        else M.template update<1>(M.LAM, r0, ts);
        tm.sync();
    }
    int status = ILVES_MOL_MAX_ITER, iters = A.max_iter;
    for (int it = 0;; ++it) {
        bool conv = true, bad = false;
#pragma unroll 1
        for (int p = r0; p < nc; p += ts) M.violation(p, M.con[p], conv, bad, !A.chord);
        if (tm.all(conv && !bad)) {
            status = ILVES_MOL_CONVERGED;
            iters = it;
            break;
        }
        // a non-finite violation ends the solve in this iteration, before anything moves; it is
        // voted on together with the pivots
        if (it >= A.max_iter) {
            if (tm.any(bad)) status = ILVES_MOL_NONFINITE;
            break;
        }
        if constexpr (Team::kWarp) tm.sync();  // a warp's vote does not order memory
        bool singular = false;
        if (!A.chord || it == 0) {
            M.assemble(A.chord ? M.RHOF : M.RF, r0, ts, singular);  // ILVES-F: A(x_old, x_old), once
            tm.sync();
            M.template solve_linear<Team, false>(tm, singular);
        } else {
            M.template solve_linear<Team, true>(tm, singular);
        }
        if (tm.any(singular || bad)) {  // also the barrier after the last level
            status = tm.any(bad) ? ILVES_MOL_NONFINITE : ILVES_MOL_SINGULAR_PIVOT;
            iters = it;
            break;
        }
        if constexpr (Team::kWarp) tm.sync();
#pragma unroll 1
        for (int p = r0; p < nc; p += ts) M.lambda_acc(p);
        if constexpr (!Mode::df && sizeof(typename Mode::LP) == 4) tm.sync();
        if constexpr (Mode::df) M.update_df(r0, ts);
        else M.template update<2>(M.corrections(), r0, ts);
        tm.sync();
    }
    M.out_atoms(r0, ts);
    if (A.lambda_out)
        for (int p = r0; p < nc; p += ts) M.out_lambda(p);
    if (r0 == 0) {
        if (A.iterations_out) A.iterations_out[D.mol_id] = iters;
        if (A.status_out) A.status_out[D.mol_id] = status;
    }
}

}  // namespace ilves

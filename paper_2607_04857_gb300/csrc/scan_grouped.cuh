// The grouped step form of the dense scans (included by scan_impl.cuh, which has its helpers).
//
// The min over a step's columns is half of a state's work and only finds the rare states at or
// below the threshold.  The walk runs in groups of 16 Gray steps.  Steps 1..15 of a group flip the
// register rows 0-3, in the same pattern in every group but for the sign of row 3, which alternates:
// the group's 16 states of a column are its value with rows 0-3 clear plus every subset of the four
// rows, so its minimum over the group is its value at the first state plus an offset, the sum of the
// rows' negative parts, less M_3 when row 3 is set there.  At a group's first state each thread takes
// the exact minimum m of its columns; with D the smallest offset of its columns (two values per thread
// and unit, one per sign of row 3), no column falls below m + D in the group.  With min E_L over the
// group's states from the tables, m + D > u - min E_L in every lane proves that the group holds no
// candidate, and it runs its 15 column updates alone.  Every state gets its column update either way.
//
// A group the first test cannot clear takes a second one, each column with its own offset (kept in
// shared memory): the exact minimum over the group, with no slack but E_L's.  Groups that fail it
// (n=36: 0.002% of them, n=48 Max-Cut 0.004%) are walked state by state.
//
// What bounds it (GB300, cycles per 16-column step per scheduler): eight f32x2 adds 17.4 (both halves
// of the FMA pipe); sixteen int32 adds as long when half of them issue to the FMA pipe's heavy half and
// half to the ALU pipe (group_updates).
#pragma once

namespace qubo {

// Integer columns: half of a group's updates are multiply-adds.  Register rows 0-3 of the columns
// updated so are held divided by an odd constant c (modulo 2^32, where c has an inverse), and
// x +- c (M / c) is one instruction with two register operands that issues to the FMA pipe's heavy
// half.  c is no short sum of powers of two, which would become shifts and adds on the ALU pipe, and
// its inverse comes as an argument: with both known the compiler cancels them.
template <class TC>
__host__ __device__ constexpr bool mad_slot(int row, int q)  // row 0 flips at odd steps, rows 1-3 at even ones
{
    return std::is_integral_v<TC> && row < 4 && (row == 0 ? q % 2 == 1 : q % 2 == 0);
}
template <class TC>
__host__ __device__ constexpr TC mad_factor(int row, int q) { return mad_slot<TC>(row, q) ? (TC)kMad : (TC)1; }
template <bool NEG, class TC>
__device__ __forceinline__ void mad_row(TC &x, TC part)
{
    if constexpr (NEG)
        asm("mad.lo.s32 %0, %1, %2, %0;" : "+r"(x) : "r"(part), "n"((int32_t)(0u - kMad)));
    else
        asm("mad.lo.s32 %0, %1, %2, %0;" : "+r"(x) : "r"(part), "n"((int32_t)kMad));
}
// Register row values as the walk keeps them (kept) from plain ones, once per unit.
template <class TC, int S, int NR>
__device__ __forceinline__ void keep_mad_rows(TC (&Mr)[NR][S], uint32_t inverse)
{
    static_for<NR>([&](auto rc) {
        static_for<S>([&](auto qc) {
            constexpr int r = decltype(rc)::value, q = decltype(qc)::value;
            if constexpr (mad_slot<TC>(r, q))
                Mr[r][q] = (TC)((uint32_t)Mr[r][q] * inverse);
        });
    });
}

// x += a (NEG: x -= a) as the minimum of the sum and a cap that no column value reaches (an
// operand in the instruction): an add that issues to the ALU pipe.  int32 columns stay below 2^30 in
// magnitude; packed words stay below 2^32 - 1 (the host admits plans whose columns stay below 32767).
template <bool NEG>
__device__ __forceinline__ void capped_add(int32_t &x, int32_t a)
{
    x = __viaddmin_s32(x, NEG ? -a : a, 1 << 30);
}
template <bool NEG>
__device__ __forceinline__ void capped_add(uint32_t &x, uint32_t a)
{
    x = __viaddmin_u32(x, NEG ? 0u - a : a, 0xfffffffeu);
}

// The column updates of a skipped group.  FP32 adds are not reassociated.  Integer adds are: the
// compiler would fold a run of them into one (or, as opaque instructions, in pairs into 3-input
// adds), and the energies between would never be formed.  So a column's capped adds alternate with
// multiply-adds by kMad, which no add next to them can be merged with, in a checkerboard over steps
// and columns, so that every step feeds both integer pipes.  All 240 updates of a group are issued
// (instruction count).  A whole n=38 scan takes 21.2 cycles per 16-column step, tests and set-up
// included; of the other forms measured, a skipped group alone took 23.4 with every second step's
// adds predicated, 26.2 with every add predicated and 31.6 for plain adds with the min over the columns.
template <class TC, int S, int ADDM, int PAR, int NR>
__device__ __forceinline__ void group_updates(TC (&E)[S], const TC (&Mr)[NR][S])
{
    static_for<15>([&](auto tc) {
        constexpr int t = decltype(tc)::value + 1, kk = ctzc(t);
        constexpr bool neg = kk == 3 ? PAR != 0 : ((t >> (kk + 1)) & 1) != 0;
        if constexpr (std::is_integral_v<TC>) {
            static_for<S>([&](auto qc) {
                constexpr int q = decltype(qc)::value;
                if constexpr (mad_slot<TC>(kk, q))
                    mad_row<neg>(E[q], Mr[kk][q]);
                else
                    capped_add<neg>(E[q], Mr[kk][q]);
            });
        } else {
            add_row<TC, S, ADDM, neg>(E, Mr[kk]);
        }
    });
}

// Sums that round down (FP32) or are exact.
__device__ __forceinline__ float add_down(float a, float b) { return __fadd_rd(a, b); }
__device__ __forceinline__ int32_t add_down(int32_t a, int32_t b) { return a + b; }
__device__ __forceinline__ int64_t add_down(int64_t a, int64_t b) { return a + b; }

// One work unit of the grouped form: all 2^(B+L) states with fixed bits x_f = unit, L >= 5.
// FP32 columns that hold integers: m + D is summed rounding down and u - min E_L is exact (both
// stay below 2^24).  FP32 columns of float Q take 16 ulp of beta (geps) off m + D, more than the
// rounding of the group's 15 adds and of the E_L add, and round u - min E_L up, so a group is
// skipped only when the step-by-step path records nothing in it.  int32: summed in int64.
//
// NG groups are unrolled per body: 4 (a body flips rows 0-4 with compile-time signs and row RC = 5
// between its halves) for long launches, 1 for short ones, where the first pass through the code
// waits on instruction fetch (about 0.2 us per 128 bytes) longer than the scan takes.
template <class T, int S, int RC, int NG, bool K1, int ADDM>
__device__ __forceinline__ void scan_unit_grouped(const ScanArgs &a, const Inst &d, int inst, uint64_t unit,
                                                  typename Tr<T>::TP &Treg, int lane, typename Tr<T>::TC *stage,
                                                  typename Tr<T>::TP *wsm, typename Tr<T>::TC *anc,
                                                  typename Tr<T>::TC *neg)
{
    using F = typename Tr<T>::FU;
    using TC = typename Tr<T>::TC;
    using TP = typename Tr<T>::TP;
    constexpr bool kFp = std::is_same_v<TC, float>;
    constexpr int V = VecOf<TC>::V;
    constexpr int G = S / V;
    constexpr int LOGV = ilog2c(V), LOGG = ilog2c(G);
    constexpr int B = LOGV + 5 + LOGG, NB = 1 << B;
    static_assert((RC == 4 && NG == 1) || (RC == 5 && NG == 4), "a body's flips below row RC are register rows");
    constexpr int NR = 4 + ilog2c(NG);  // rows a body flips
    const int n = d.n, L = d.L, k = d.k, BL = B + L;
    InstState *st = a.state + inst;

    // fields of the set fixed bits and c(x_f), as in scan_unit
    F f0, cx;
    if constexpr (std::is_same_v<F, float>) {
        double f0d, cxd;
        unit_fields<T, double>(d.W64, n, k, BL, unit, lane, f0d, cxd);
        f0 = (float)f0d;
        cx = (float)cxd;
    } else {
        unit_fields<T, F>(unit_matrix<T>(d), n, k, BL, unit, lane, f0, cx);
    }
    __syncwarp();
    if (lane >= B && lane < BL)
        wsm[lane - B] = (TP)f0;
    __syncwarp();
    F lin_t, lin_e[V], lin_g[G];
    column_fields<F, V, G>(f0, lane, lin_t, lin_e, lin_g);

    // initial columns (walked bits all zero) and register rows M_r + w_r
    const TC *Es = (const TC *)d.Es;
    const TC *Mt = (const TC *)d.M;
    TC E[S];
#pragma unroll
    for (int g = 0; g < G; ++g) {
        TC ev[V];
        vload<TC>(Es + (g * 32 + lane) * V, ev);
#pragma unroll
        for (int e = 0; e < V; ++e)
            E[g * V + e] = (TC)((F)ev[e] + (lin_e[e] + lin_t + lin_g[g]));
    }
    if constexpr (Tr<T>::kFloat) {
#pragma unroll
        for (int g = 0; g < G; ++g)
            *(typename VecOf<TC>::type *)(anc + (g * 32 + lane) * V) = vjoin(E + g * V);
    }
    TC Mr[RC][S];
#pragma unroll
    for (int r = 0; r < RC; ++r) {
        const F wr = __shfl_sync(kFull, f0, B + r);
#pragma unroll
        for (int g = 0; g < G; ++g) {
            TC mv[V];
            vload<TC>(Mt + (size_t)r * NB + (g * 32 + lane) * V, mv);
#pragma unroll
            for (int e = 0; e < V; ++e)
                Mr[r][g * V + e] = (TC)((F)mv[e] + wr);
        }
    }

    // the offsets (rows 0-3 clear at the first state) and D, summed rounding down
    using DB = std::conditional_t<kFp, float, int64_t>;  // the bound as the test takes it
    DB Dgrp[2];
    {
        TC d0{}, d1{};
#pragma unroll
        for (int g = 0; g < G; ++g) {
            TC nv[V];
#pragma unroll
            for (int e = 0; e < V; ++e) {
                const int q = g * V + e;
                nv[e] = emin(Mr[0][q], (TC)0);
#pragma unroll
                for (int r = 1; r < 4; ++r)
                    nv[e] = add_down(nv[e], emin(Mr[r][q], (TC)0));
                const TC odd = add_down(nv[e], -Mr[3][q]);
                d0 = q ? emin(d0, nv[e]) : nv[e];
                d1 = q ? emin(d1, odd) : odd;
            }
            *(typename VecOf<TC>::type *)(neg + (g * 32 + lane) * V) = vjoin(nv);
        }
        Dgrp[0] = (DB)d0;
        Dgrp[1] = (DB)d1;
    }
    keep_mad_rows(Mr, a.mad_inverse);

    {
        const TP tg = Tr<T>::thr_load(st);
        Treg = K1 ? min(Treg, tg) : tg;
    }
    const TP mu = (TP)a.margin;
    const int32_t clampC = d.clampC;
    TP P = (TP)cx;  // c(x_f) + coupling of the walked rows >= RC that are set
    TP u = Treg + mu - P;
    TC uc = to_col<T>(u, clampC);

    // flip of a walked row kk >= RC (row from memory, run-time sign)
    auto high_flip = [&](int kk, int sgn) {
        if (!QUBO_DCHECK(kk >= RC && kk < L, st, 1))
            kk = RC;
        const TC *row = Mt + (size_t)kk * NB;
        const TC sg = (TC)sgn;
#pragma unroll
        for (int g = 0; g < G; ++g) {
            TC mv[V];
            vload<TC>(row + (g * 32 + lane) * V, mv);
#pragma unroll
            for (int e = 0; e < V; e += 2) {
                if constexpr (kFp) {
                    fma_f32x2(E[g * V + e], E[g * V + e + 1], mv[e], mv[e + 1], sg);
                } else {
                    E[g * V + e] += sg * mv[e];
                    E[g * V + e + 1] += sg * mv[e + 1];
                }
            }
        }
        P = P + (TP)sgn * wsm[kk];
        u = Treg + mu - P;
        uc = to_col<T>(u, clampC);
    };

    // float scans: rebuild the columns and P from the base columns and the rows of the set walked
    // bits at walk step i (a multiple of 2^(RC+1), so the register rows are clear); the largest
    // difference to the incremental values is the drift (see scan_unit)
    TC dl = 0;
    auto reanchor = [&](int i) {
        const int gi = i ^ (i >> 1);
        TP Pf = (TP)cx;
        TC fr[S];
#pragma unroll
        for (int g = 0; g < G; ++g) {
            TC bv[V];
            vsplit(*(const typename VecOf<TC>::type *)(anc + (g * 32 + lane) * V), bv);
#pragma unroll
            for (int e = 0; e < V; ++e)
                fr[g * V + e] = bv[e];
        }
        for (unsigned bits = (unsigned)gi >> RC; bits; bits &= bits - 1) {
            int r = RC + __ffs(bits) - 1;
            if (!QUBO_DCHECK(r < L, st, 2))
                r = RC;
            Pf = Pf + wsm[r];
            const TC *row = Mt + (size_t)r * NB;
#pragma unroll
            for (int g = 0; g < G; ++g) {
                TC mv[V];
                vload<TC>(row + (g * 32 + lane) * V, mv);
#pragma unroll
                for (int e = 0; e < V; ++e)
                    fr[g * V + e] = fr[g * V + e] + mv[e];
            }
        }
#pragma unroll
        for (int q = 0; q < S; ++q) {
            const TC dd = E[q] - fr[q];  // exact for close values
            const TC ad = dd < 0 ? -dd : dd;
            dl = dl > ad ? dl : ad;
            E[q] = fr[q];
        }
        const TC dp = (TC)(P < Pf ? Pf - P : P - Pf);
        dl = dl > dp ? dl : dp;
        P = Pf;
        u = Treg + mu - P;
        uc = to_col<T>(u, clampC);
    };
    // anchor period in bodies minus one; -1 (never) without mid-walk anchors
    constexpr int LOGBODY = 4 + ilog2c(NG), BODY = 1 << LOGBODY;
    const int amask = (Tr<T>::kFloat && d.anchor > RC && d.anchor < L) ? (1 << (d.anchor - LOGBODY)) - 1 : -1;

    const TC *ELp = (const TC *)d.EL;
    const TC *ELg = ELp + (1 << L);  // min E_L over each group
    const uint64_t cbase = unit << BL;

    // The group of 16 states whose first is in E: the tests, then the column updates; true (for
    // the warp) when a column may be at or below the threshold in one of its states.  PAR: sign of row
    // 3 (2: par, at run time).
    auto run_group = [&](auto parc, int par, TC elg) -> bool {
        constexpr int PAR = decltype(parc)::value;
        const bool odd = PAR == 2 ? par != 0 : PAR == 1;
        const TC m0 = tree_min<TC, 3, S>(E);
        const DB D = odd ? Dgrp[1] : Dgrp[0];
        auto above = [&](DB low) {  // no state of the group is at or below the threshold
            if constexpr (Tr<T>::kFloat)
                return __fadd_rd(low, -d.geps) > __fsub_ru(uc, elg);
            else if constexpr (kFp)
                return low > uc - elg;
            else
                return low > (int64_t)uc - elg;
        };
        auto updates = [&] {
            if constexpr (PAR == 2) {
                if (odd)
                    group_updates<TC, S, ADDM, 1>(E, Mr);
                else
                    group_updates<TC, S, ADDM, 0>(E, Mr);
            } else {
                group_updates<TC, S, ADDM, PAR>(E, Mr);
            }
        };
        // the exact minimum over the group of each column (with row 3 set, less M_3)
        auto refined = [&] {
            TC low[S];
#pragma unroll
            for (int g = 0; g < G; ++g) {
                TC nv[V];
                vsplit(*(const typename VecOf<TC>::type *)(neg + (g * 32 + lane) * V), nv);
#pragma unroll
                for (int e = 0; e < V; ++e) {
                    const int q = g * V + e;
                    low[q] = add_down(odd ? add_kept_row(E[q], (TC)-1, mad_factor<TC>(3, q), Mr[3][q]) : E[q], nv[e]);
                }
            }
            return (DB)tree_min<TC, 3, S>(low);
        };
        const bool clear = __all_sync(kFull, above(add_down((DB)m0, D)));
        if constexpr (kFp && NG > 1) {
            // a copy of the updates for the rare side: the common one stays straight-line code (0.8%)
            if (__builtin_expect(clear, 1)) {
                updates();
                return false;
            }
            const bool hit = !__all_sync(kFull, above(refined()));
            updates();
            return hit;
        } else {
            bool hit = false;
            if (!clear)
                hit = !__all_sync(kFull, above(refined()));
            updates();
            return hit;
        }
    };

    // Rare: offer the staged columns in mask of walk step i (P = Pp, E_L = elp).
    auto record_staged = [&](int i, TP Pp, TC elp, unsigned mask) {
        const uint64_t cb = cbase | ((uint64_t)(i ^ (i >> 1)) << B);
        const TP Ep = Pp + (TP)elp;
        const TP least = record_warp<T>(
            a, inst, mask, lane, [&](int q) { return (TP)stage[q * 32 + lane] + Ep; },
            [&](int q) { return cb | (uint32_t)(((q / V) * 32 + lane) * V + (q % V)); });
        if (K1 && least < Treg) {
            Treg = least;
            if (lane == 0)
                Tr<T>::thr_min(st, least);
        }
    };
    // Columns of walk step i of the body from those of step j: the register rows, and with NG > 1 row
    // RC, whose Gray bits differ.
    const TC *rowRC = Mt + (size_t)RC * NB;
    [[maybe_unused]] auto move = [&](TC (&x)[S], int i, int j) {
        const int gi = i ^ (i >> 1), gj = j ^ (j >> 1);
        TC sr[NR];
#pragma unroll
        for (int r = 0; r < NR; ++r)
            sr[r] = (TC)(((gi >> r) & 1) - ((gj >> r) & 1));
        static_for<G>([&](auto gc) {
            constexpr int g = decltype(gc)::value;
            TC mv[V];
            if constexpr (NG > 1)
                vload<TC>(rowRC + (g * 32 + lane) * V, mv);
            static_for<V>([&](auto ec) {
                constexpr int e = decltype(ec)::value, q = g * V + e;
                static_for<(NR < RC ? NR : RC)>([&](auto rc) {
                    constexpr int r = decltype(rc)::value;
                    x[q] = add_kept_row(x[q], sr[r], mad_factor<TC>(r, q), Mr[r][q]);
                });
                if constexpr (NG > 1)
                    x[q] = x[q] + sr[RC] * mv[e];
            });
        });
    };
    // The states of the body's groups in hits (the same for the warp), E being the body's last one.  Integer columns (exact)
    // are moved to each group's first state, walked through it and moved back; FP32 columns are
    // left alone and every state is rebuilt from the last one.  Pmid: P before the flip of row RC.
    auto record_hits = [&](int i0, unsigned hits, TP Pmid) {
        const int iend = i0 + BODY - 1;
        auto prefix = [&](int i) {
            return NG == 1 || (((i ^ (i >> 1)) ^ (iend ^ (iend >> 1))) >> RC & 1) == 0 ? P : Pmid;
        };
        if constexpr (Tr<T>::kFloat) {
            const int gend = iend ^ (iend >> 1);
#pragma unroll 1
            for (int p = 0; p < BODY; ++p) {
                if (!((hits >> (p >> 4)) & 1u))
                    continue;
                if (__any_sync(kFull, gave_up(a)))
                    break;
                const int i = i0 + p, gp = i ^ (i >> 1);
                TC sr[NR];
#pragma unroll
                for (int r = 0; r < NR; ++r)
                    sr[r] = (TC)(((gp >> r) & 1) - ((gend >> r) & 1));
                const TP Pp = prefix(i);
                const TC elp = ELp[i], tp = to_col<T>(Treg + mu - Pp, clampC) - elp;
                unsigned mask = 0;
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    TC mv[V];
                    if constexpr (NG > 1)
                        vload<TC>(rowRC + (g * 32 + lane) * V, mv);
#pragma unroll
                    for (int e = 0; e < V; ++e) {
                        const int q = g * V + e;
                        TC x = E[q];
#pragma unroll
                        for (int r = 0; r < NR && r < RC; ++r)
                            x = x + sr[r] * Mr[r][q];
                        if constexpr (NG > 1)
                            x = x + sr[RC] * mv[e];
                        stage[q * 32 + lane] = x;
                        mask |= x <= tp ? 1u << q : 0u;
                    }
                }
                if (__any_sync(kFull, mask != 0))
                    record_staged(i, Pp, elp, mask);
            }
        } else {
            int at = iend;
#pragma unroll 1
            for (int p = 0; p < BODY; ++p) {
                if (!((hits >> (p >> 4)) & 1u))
                    continue;
                if (p % 16 == 0) {
                    move(E, i0 + p, at);
                } else {
                    const int row = __ffs(p) - 1;
                    const TC sg = ((p + i0) >> (row + 1)) & 1 ? (TC)-1 : (TC)1;
                    static_for<4>([&](auto rc) {
                        constexpr int r = decltype(rc)::value;
                        if (row == r)
                            static_for<S>([&](auto qc) {
                                constexpr int q = decltype(qc)::value;
                                E[q] = add_kept_row(E[q], sg, mad_factor<TC>(r, q), Mr[r][q]);
                            });
                    });
                }
                at = i0 + p;
                const TP Pp = prefix(at);
                const TC elp = ELp[at], tp = to_col<T>(Treg + mu - Pp, clampC) - elp;
                if (!__any_sync(kFull, tree_min<TC, 3, S>(E) <= tp))
                    continue;
                unsigned mask = 0;
#pragma unroll
                for (int q = 0; q < S; ++q) {
                    stage[q * 32 + lane] = E[q];
                    mask |= E[q] <= tp ? 1u << q : 0u;
                }
                record_staged(at, Pp, elp, mask);
            }
            move(E, iend, at);
        }
        u = Treg + mu - P;
        uc = to_col<T>(u, clampC);
    };

    const int nblk = 1 << (L - LOGBODY);
    if (!QUBO_DCHECK(L >= RC + 1 && L <= kMaxWalkBits && nblk * BODY == (1 << L), st, 3))
        return;
#pragma unroll 1
    for (int blk = 0; blk < nblk; ++blk) {
        const int i0 = blk * BODY;
        TC elg[NG];
        if constexpr (NG == VecOf<TC>::V)
            vload<TC>(ELg + blk * NG, elg);
        else
            elg[0] = __ldg(ELg + blk);
        if (blk) {  // the step into the body
            const int kk = __ffs(i0) - 1;
            high_flip(kk, ((i0 >> (kk + 1)) & 1) ? -1 : 1);
            if constexpr (Tr<T>::kFloat) {
                if ((blk & amask) == 0)
                    reanchor(i0);
            }
        }
        TP Pmid = P;
        unsigned hits = 0;
        if constexpr (NG == 1) {
            hits = run_group(std::integral_constant<int, 2>{}, blk & 1, elg[0]);
        } else {
            static_for<NG>([&](auto gc) {
                constexpr int g = decltype(gc)::value, p0 = 16 * g, kk = g > 0 ? ctzc(p0) : 0;
                if constexpr (g > 0 && kk < RC) {
                    add_row<TC, S, ADDM, ((p0 >> (kk + 1)) & 1) != 0>(E, Mr[kk]);
                } else if constexpr (g > 0) {
                    Pmid = P;
                    high_flip(RC, (blk & 1) ? -1 : 1);
                }
                if (run_group(std::integral_constant<int, g & 1>{}, 0, elg[g]))
                    hits |= 1u << g;
            });
        }
        if (hits)
            record_hits(i0, hits, Pmid);
    }

    if constexpr (Tr<T>::kFloat) {
        // the walk ends at step 2^L - 1 (g = 2^(L-1)): the last segment's drift
        reanchor((1 << L) - 1);
        double dmax = (double)dl;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            dmax = fmax(dmax, __shfl_xor_sync(kFull, dmax, o));
        if (lane == 0)
            atomicMax(&st->drift, (unsigned long long)__double_as_longlong(dmax));
    }
}

// One work unit of the grouped form in packed 16-bit columns (see scan_unit_packed for the lanes).
// E_L is stored minus the lane bias, so lane + stored E_L is the column's energy without P.  D takes
// the offsets of both lanes; the host admits only plans whose rows 0-3 move a column by at most 32767.
template <int S, int RC, int NG, bool K1>
__device__ __forceinline__ void scan_unit_packed_grouped(const ScanArgs &a, const Inst &d, int inst, uint64_t unit,
                                                         int32_t &Treg, int lane, uint32_t *stage, int32_t *wsm,
                                                         uint32_t *neg)
{
    using T = i16p;
    using F = int32_t;
    constexpr int V = 4, G = S / V;
    constexpr int LOGV = ilog2c(V), LOGG = ilog2c(G);
    constexpr int B = LOGV + 5 + LOGG + 1;
    constexpr int NW = 1 << (B - 1);  // words per table row
    static_assert((RC == 4 && NG == 1) || (RC == 5 && NG == 4), "a body's flips below row RC are register rows");
    constexpr int NR = 4 + ilog2c(NG);
    const int n = d.n, L = d.L, k = d.k, BL = B + L;
    InstState *st = a.state + inst;

    F f0, cx;
    unit_fields<T>(unit_matrix<T>(d), n, k, BL, unit, lane, f0, cx);
    __syncwarp();
    if (lane >= B && lane < BL)
        wsm[lane - B] = f0;
    __syncwarp();
    F lin_t, lin_e[V], lin_g[G];
    column_fields<F, V, G>(f0, lane, lin_t, lin_e, lin_g);
    const F vtop = __shfl_sync(kFull, f0, B - 1);

    const int32_t *Es = (const int32_t *)d.Es;
    const uint32_t *Mt = (const uint32_t *)d.M;
    uint32_t E[S];
#pragma unroll
    for (int g = 0; g < G; ++g) {
        int32_t lo[V], hi[V];
        vload<int32_t>(Es + (g * 32 + lane) * V, lo);
        vload<int32_t>(Es + NW + (g * 32 + lane) * V, hi);
#pragma unroll
        for (int e = 0; e < V; ++e) {
            const F lin = lin_e[e] + lin_t + lin_g[g];
            E[g * V + e] = (uint32_t)(lo[e] + lin + kLaneBias) + ((uint32_t)(hi[e] + lin + vtop + kLaneBias) << 16);
        }
    }
    uint32_t Mr[RC][S];
#pragma unroll
    for (int r = 0; r < RC; ++r) {
        const uint32_t wr2 = (uint32_t)__shfl_sync(kFull, f0, B + r) * 65537u;
#pragma unroll
        for (int g = 0; g < G; ++g) {
            uint32_t mv[V];
            vload<uint32_t>(Mt + (size_t)r * NW + (g * 32 + lane) * V, mv);
#pragma unroll
            for (int e = 0; e < V; ++e)
                Mr[r][g * V + e] = mv[e] + wr2;
        }
    }
    // the offsets per lane and D over both lanes; a row's word is x + 65536 y with both moves in
    // [-32768, 32767]
    int32_t Dgrp[2] = {0x7fffffff, 0x7fffffff};
#pragma unroll
    for (int g = 0; g < G; ++g) {
        uint32_t nv[V];
#pragma unroll
        for (int e = 0; e < V; ++e) {
            int32_t nx = 0, ny = 0, x = 0, y = 0;
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const uint32_t w = Mr[r][g * V + e];
                x = (int32_t)(int16_t)(w & 0xffffu);
                y = (int32_t)(w - (uint32_t)x) >> 16;
                nx += min(x, 0);
                ny += min(y, 0);
            }
            nv[e] = (uint32_t)nx + ((uint32_t)ny << 16);
            Dgrp[0] = __vimin3_s32(Dgrp[0], nx, ny);
            Dgrp[1] = __vimin3_s32(Dgrp[1], nx - x, ny - y);
        }
        *(uint4 *)(neg + (g * 32 + lane) * V) = vjoin(nv);
    }
    keep_mad_rows(Mr, a.mad_inverse);

    {
        const int32_t tg = Tr<T>::thr_load(st);
        Treg = K1 ? min(Treg, tg) : tg;
    }
    const int32_t mu = (int32_t)a.margin;
    int32_t P = cx;
    int32_t u = Treg + mu - P;
    auto high_flip = [&](int kk, int sgn) {
        if (!QUBO_DCHECK(kk >= RC && kk < L, st, 4))
            kk = RC;
        const uint32_t *row = Mt + (size_t)kk * NW;
        const uint32_t sg = (uint32_t)sgn;
#pragma unroll
        for (int g = 0; g < G; ++g) {
            uint32_t mv[V];
            vload<uint32_t>(row + (g * 32 + lane) * V, mv);
#pragma unroll
            for (int e = 0; e < V; ++e)
                E[g * V + e] += sg * mv[e];
        }
        P = P + sgn * wsm[kk];
        u = Treg + mu - P;
    };

    const int32_t *ELp = (const int32_t *)d.EL;
    const int32_t *ELg = ELp + (1 << L);
    const uint64_t cbase = unit << BL;
    auto lane_min = [](uint32_t w) { return min((int32_t)(w & 0xffffu), (int32_t)(w >> 16)); };

    // as in scan_unit_grouped, in lane units
    auto run_group = [&](auto parc, int par, int32_t elg) -> bool {
        constexpr int PAR = decltype(parc)::value;
        const bool odd = PAR == 2 ? par != 0 : PAR == 1;
        const int32_t m0 = lane_min(tree_min<uint32_t, 3, S>(E));
        bool hit = false;
        if (__builtin_expect(!__all_sync(kFull, m0 + (odd ? Dgrp[1] : Dgrp[0]) > u - elg), 0)) {
            uint32_t low[S];  // each lane a column value of the group, so no carry leaves it
#pragma unroll
            for (int g = 0; g < G; ++g) {
                uint32_t nv[V];
                vsplit(*(const uint4 *)(neg + (g * 32 + lane) * V), nv);
#pragma unroll
                for (int e = 0; e < V; ++e) {
                    const int q = g * V + e;
                    low[q] = (odd ? E[q] - mad_factor<uint32_t>(3, q) * Mr[3][q] : E[q]) + nv[e];
                }
            }
            hit = !__all_sync(kFull, lane_min(tree_min<uint32_t, 3, S>(low)) > u - elg);
        }
        if constexpr (PAR == 2) {
            if (odd)
                group_updates<uint32_t, S, 0, 1>(E, Mr);
            else
                group_updates<uint32_t, S, 0, 0>(E, Mr);
        } else {
            group_updates<uint32_t, S, 0, PAR>(E, Mr);
        }
        return hit;
    };

    constexpr int LOGBODY = 4 + ilog2c(NG), BODY = 1 << LOGBODY;
    auto record_state = [&](int i, int32_t Pp) {
        const int32_t els = ELp[i], tp = Treg + mu - Pp - els;
        if (!__any_sync(kFull, lane_min(tree_min<uint32_t, 3, S>(E)) <= tp))
            return;
        unsigned mask = 0;  // bit 2 q + h: half h of word q
#pragma unroll
        for (int q = 0; q < S; ++q) {
            stage[q * 32 + lane] = E[q];
            mask |= (int32_t)(E[q] & 0xffffu) <= tp ? 1u << (2 * q) : 0u;
            mask |= (int32_t)(E[q] >> 16) <= tp ? 2u << (2 * q) : 0u;
        }
        const uint64_t cb = cbase | ((uint64_t)(i ^ (i >> 1)) << B);
        const int32_t least = record_warp<T>(
            a, inst, mask, lane,
            [&](int q) {
                const uint32_t word = stage[(q >> 1) * 32 + lane];
                return (int32_t)((q & 1) ? (word >> 16) : (word & 0xffffu)) + els + Pp;
            },
            [&](int q) {
                const int w = q >> 1;
                return cb | (uint32_t)(((w / V) * 32 + lane) * V + (w % V) + ((q & 1) ? NW : 0));
            });
        if (K1 && least < Treg) {
            Treg = least;
            if (lane == 0)
                Tr<T>::thr_min(st, least);
        }
    };
    const uint32_t *rowRC = Mt + (size_t)RC * NW;
    auto move = [&](int i, int j) {
        const int gi = i ^ (i >> 1), gj = j ^ (j >> 1);
        uint32_t sr[NR];
#pragma unroll
        for (int r = 0; r < NR; ++r)
            sr[r] = (uint32_t)(((gi >> r) & 1) - ((gj >> r) & 1));
        static_for<G>([&](auto gc) {
            constexpr int g = decltype(gc)::value;
            uint32_t mv[V];
            if constexpr (NG > 1)
                vload<uint32_t>(rowRC + (g * 32 + lane) * V, mv);
            static_for<V>([&](auto ec) {
                constexpr int e = decltype(ec)::value, q = g * V + e;
                static_for<(NR < RC ? NR : RC)>([&](auto rc) {
                    constexpr int r = decltype(rc)::value;
                    E[q] += sr[r] * mad_factor<uint32_t>(r, q) * Mr[r][q];
                });
                if constexpr (NG > 1)
                    E[q] += sr[RC] * mv[e];
            });
        });
    };
    auto record_hits = [&](int i0, unsigned hits, int32_t Pmid) {
        const int iend = i0 + BODY - 1;
        int at = iend;
#pragma unroll 1
        for (int p = 0; p < BODY; ++p) {
            if (!((hits >> (p >> 4)) & 1u))
                continue;
            if (p % 16 == 0) {
                move(i0 + p, at);
            } else {
                const int row = __ffs(p) - 1;
                const uint32_t sg = ((p + i0) >> (row + 1)) & 1 ? ~0u : 1u;
                static_for<4>([&](auto rc) {
                    constexpr int r = decltype(rc)::value;
                    if (row == r)
                        static_for<S>([&](auto qc) {
                            constexpr int q = decltype(qc)::value;
                            E[q] += sg * mad_factor<uint32_t>(r, q) * Mr[r][q];
                        });
                });
            }
            at = i0 + p;
            const int ga = at ^ (at >> 1), ge = iend ^ (iend >> 1);
            record_state(at, NG == 1 || ((ga ^ ge) >> RC & 1) == 0 ? P : Pmid);
        }
        move(iend, at);
        u = Treg + mu - P;
    };

    const int nblk = 1 << (L - LOGBODY);
    if (!QUBO_DCHECK(L >= RC + 1 && L <= kMaxWalkBits && nblk * BODY == (1 << L), st, 5))
        return;
#pragma unroll 1
    for (int blk = 0; blk < nblk; ++blk) {
        const int i0 = blk * BODY;
        int32_t elg[NG];
        if constexpr (NG == 4)
            vload<int32_t>(ELg + blk * NG, elg);
        else
            elg[0] = __ldg(ELg + blk);
        if (blk) {
            const int kk = __ffs(i0) - 1;
            high_flip(kk, ((i0 >> (kk + 1)) & 1) ? -1 : 1);
        }
        int32_t Pmid = P;
        unsigned hits = 0;
        if constexpr (NG == 1) {
            hits = run_group(std::integral_constant<int, 2>{}, blk & 1, elg[0]);
        } else {
            static_for<NG>([&](auto gc) {
                constexpr int g = decltype(gc)::value, p0 = 16 * g, kk = g > 0 ? ctzc(p0) : 0;
                if constexpr (g > 0 && kk < RC) {
                    add_row<uint32_t, S, 0, ((p0 >> (kk + 1)) & 1) != 0>(E, Mr[kk]);
                } else if constexpr (g > 0) {
                    Pmid = P;
                    high_flip(RC, (blk & 1) ? -1 : 1);
                }
                if (run_group(std::integral_constant<int, g & 1>{}, 0, elg[g]))
                    hits |= 1u << g;
            });
        }
        if (hits)
            record_hits(i0, hits, Pmid);
    }
}

}  // namespace qubo

// Scan and table-build kernels instantiated for the int64_t accumulator: the plain kernel (variant 0)
// and the grouped one on two 32-bit limbs (variant 1).
#include "scan_impl.cuh"

namespace qubo {

namespace {
// ---- grouped scan of int64 energies on two limbs -------------------------------------------------
// A column's energy is held as hi * 2^s + lo, two int32 values that are updated separately: a table
// row is split once into hi and lo (|lo| <= 2^(s-1)), and the walk adds the halves without carrying
// from one to the other.  The lo of a column is then the sum of the lo of its base and of at most
// kLimbMaxWalkBits = 14 set rows, |lo| <= 15 * 2^(s-1) < 8 * 2^s, and with s = max(1, ceil(log2 beta) - 29)
// <= 26 both limbs stay below 2^30 (beta < 2^55).  A state costs two int32 updates, no 64-bit minimum: the group
// test of scan_grouped.cuh runs on the hi limbs alone, E > u - min E_L being certain when
// hi > ((u - min E_L) >> s) + 8 (at 16 set rows a group that holds the minimum can pass it).  Groups it cannot clear are walked state by state in int64.
// What bounds it: the two integer pipes, 32 updates per 16-column step (two limbs).  n=34, entries up to
// 2^30: the plain kernel (64-bit adds and minima, 217 cycles per step) takes 5.8 ms, this one 1.35 ms (51).
constexpr int kLimbCols = 16, kLimbRows = 4;
constexpr int kLimbSlack = 8;  // of a hi limb against the energy, in units of 2^s
static_assert(kLimbMaxWalkBits + 1 < 2 * kLimbSlack, "the sum of the low limbs");

__device__ __forceinline__ void split_limbs(int64_t v, int s, int32_t &hi, int32_t &lo)
{
    const int64_t l = (int64_t)((uint64_t)v << (64 - s)) >> (64 - s);
    lo = (int32_t)l;
    hi = (int32_t)((v - l) >> s);
}

struct LimbShared {
    int64_t stage[kLimbCols * 32];
    int32_t neg[kLimbCols * 32];  // negative parts of rows 0-3, hi limbs
    int64_t wsm[kMaxWalkBits];
};

template <bool K1>
__device__ __forceinline__ void scan_unit_limbs(const ScanArgs &a, const Inst &d, int inst, uint64_t unit,
                                                int64_t &Treg, int lane, LimbShared &sm)
{
    using T = int64_t;
    constexpr int S = kLimbCols, RC = kLimbRows, V = 4, G = S / V, B = 9, NB = 1 << B;
    const int n = d.n, L = d.L, k = d.k, BL = B + L, s = d.limb;
    InstState *st = a.state + inst;
    int64_t f0, cx;
    unit_fields<T>(unit_matrix<T>(d), n, k, BL, unit, lane, f0, cx);
    __syncwarp();
    if (lane >= B && lane < BL)
        sm.wsm[lane - B] = f0;
    __syncwarp();
    int64_t lin_t, lin_e[V], lin_g[G];
    column_fields<int64_t, V, G>(f0, lane, lin_t, lin_e, lin_g);

    const int64_t *Es = (const int64_t *)d.Es;
    const int32_t *Mt = (const int32_t *)d.M;  // per row: hi limbs, then lo limbs
    int32_t Eh[S], El[S], Mh[RC][S], Ml[RC][S];
#pragma unroll
    for (int g = 0; g < G; ++g) {
        int64_t ev[V];
        const int j = (g * 32 + lane) * V;
        vsplit(__ldg((const longlong2 *)(Es + j)), *(int64_t(*)[2])ev);
        vsplit(__ldg((const longlong2 *)(Es + j + 2)), *(int64_t(*)[2])(ev + 2));
#pragma unroll
        for (int e = 0; e < V; ++e)
            split_limbs(ev[e] + (lin_e[e] + lin_t + lin_g[g]), s, Eh[g * V + e], El[g * V + e]);
    }
#pragma unroll
    for (int r = 0; r < RC; ++r) {
        const int64_t wr = __shfl_sync(kFull, f0, B + r);
#pragma unroll
        for (int g = 0; g < G; ++g) {
            const int j = (g * 32 + lane) * V;
            int32_t h[V], l[V];
            vload<int32_t>(Mt + (size_t)r * 2 * NB + j, h);
            vload<int32_t>(Mt + (size_t)r * 2 * NB + NB + j, l);
#pragma unroll
            for (int e = 0; e < V; ++e)
                split_limbs((int64_t)h[e] * ((int64_t)1 << s) + l[e] + wr, s, Mh[r][g * V + e], Ml[r][g * V + e]);
        }
    }
    int64_t Dgrp[2];
    {
        int32_t d0 = 0x7fffffff, d1 = 0x7fffffff;
#pragma unroll
        for (int g = 0; g < G; ++g) {
            int32_t nv[V];
#pragma unroll
            for (int e = 0; e < V; ++e) {
                const int q = g * V + e;
                nv[e] = min(Mh[0][q], 0) + min(Mh[1][q], 0) + min(Mh[2][q], 0) + min(Mh[3][q], 0);
                d0 = min(d0, nv[e]);
                d1 = min(d1, nv[e] - Mh[3][q]);
            }
            *(int4 *)(sm.neg + (g * 32 + lane) * V) = vjoin(nv);
        }
        Dgrp[0] = d0;
        Dgrp[1] = d1;
    }
    keep_mad_rows(Mh, a.mad_inverse);
    keep_mad_rows(Ml, a.mad_inverse);

    {
        const int64_t tg = Tr<T>::thr_load(st);
        Treg = K1 ? min(Treg, tg) : tg;
    }
    const int64_t mu = (int64_t)a.margin;
    int64_t P = cx, u = Treg + mu - P;
    const int64_t *ELp = (const int64_t *)d.EL;
    const int64_t *ELg = ELp + (1 << L);
    const uint64_t cbase = unit << BL;

    // walk steps 1..15 of a group, every state recorded that reaches the threshold (rare)
    auto checked_updates = [&](bool odd, int i0) {
#pragma unroll 1
        for (int t = 0; t < 16; ++t) {
            if (t) {
                const int row = __ffs(t) - 1;
                const int32_t sg = (row == 3 ? odd : ((t >> (row + 1)) & 1) != 0) ? -1 : 1;
                static_for<RC>([&](auto rc) {
                    constexpr int r = decltype(rc)::value;
                    if (row == r)
                        static_for<S>([&](auto qc) {
                            constexpr int q = decltype(qc)::value;
                            const uint32_t f = (uint32_t)sg * mad_factor<uint32_t>(r, q);
                            Eh[q] = (int32_t)((uint32_t)Eh[q] + f * (uint32_t)Mh[r][q]);
                            El[q] = (int32_t)((uint32_t)El[q] + f * (uint32_t)Ml[r][q]);
                        });
                });
            }
            const int i = i0 + t;
            const int64_t el = ELp[i], tp = u - el;
            if (!__any_sync(kFull, (int64_t)tree_min<int32_t, 3, S>(Eh) <= (tp >> s) + kLimbSlack))
                continue;
            unsigned mask = 0;
#pragma unroll
            for (int q = 0; q < S; ++q) {
                const int64_t x = (int64_t)Eh[q] * ((int64_t)1 << s) + El[q];
                sm.stage[q * 32 + lane] = x;
                mask |= x <= tp ? 1u << q : 0u;
            }
            if (!__any_sync(kFull, mask != 0))
                continue;
            const uint64_t cb = cbase | ((uint64_t)(i ^ (i >> 1)) << B);
            const int64_t least = record_warp<T>(
                a, inst, mask, lane, [&](int q) { return sm.stage[q * 32 + lane] + el + P; },
                [&](int q) { return cb | (uint32_t)(((q / V) * 32 + lane) * V + (q % V)); });
            if (K1 && least < Treg) {
                Treg = least;
                u = Treg + mu - P;
                if (lane == 0)
                    Tr<T>::thr_min(st, least);
            }
        }
    };

    const int ngrp = 1 << (L - 4);
    if (!QUBO_DCHECK(L >= RC + 1 && L <= kLimbMaxWalkBits, st, 9))
        return;
#pragma unroll 1
    for (int g = 0; g < ngrp; ++g) {
        const int64_t elg = __ldg(ELg + g);
        const bool odd = g & 1;
        if (g) {  // row 4 + z into the group's first state
            const int z = __ffs(g) - 1, row = RC + z;
            const int32_t sg = ((g >> (z + 1)) & 1) ? -1 : 1;
            const int32_t *src = Mt + (size_t)row * 2 * NB + lane * V;
#pragma unroll
            for (int c = 0; c < G; ++c) {
                int32_t h[V], l[V];
                vload<int32_t>(src + c * 32 * V, h);
                vload<int32_t>(src + NB + c * 32 * V, l);
#pragma unroll
                for (int e = 0; e < V; ++e) {
                    Eh[c * V + e] += sg * h[e];
                    El[c * V + e] += sg * l[e];
                }
            }
            P += sg * sm.wsm[row];
            u = Treg + mu - P;
        }
        const int64_t limit = ((u - elg) >> s) + kLimbSlack;
        if (!__all_sync(kFull, (int64_t)tree_min<int32_t, 3, S>(Eh) + (odd ? Dgrp[1] : Dgrp[0]) > limit)) {
            int32_t low[S];
            static_for<G>([&](auto cc) {
                constexpr int c = decltype(cc)::value;
                int32_t nv[V];
                vsplit(*(const int4 *)(sm.neg + (c * 32 + lane) * V), nv);
                static_for<V>([&](auto ec) {
                    constexpr int e = decltype(ec)::value, q = c * V + e;
                    const uint32_t m3 = mad_factor<uint32_t>(3, q) * (uint32_t)Mh[3][q];
                    low[q] = (int32_t)((uint32_t)Eh[q] - (odd ? m3 : 0u)) + nv[e];
                });
            });
            if (!__all_sync(kFull, (int64_t)tree_min<int32_t, 3, S>(low) > limit)) {
                checked_updates(odd, 16 * g);
                continue;
            }
        }
        if (odd) {
            group_updates<int32_t, S, 0, 1>(Eh, Mh);
            group_updates<int32_t, S, 0, 1>(El, Ml);
        } else {
            group_updates<int32_t, S, 0, 0>(Eh, Mh);
            group_updates<int32_t, S, 0, 0>(El, Ml);
        }
    }
}

template <bool K1>
__global__ void __launch_bounds__(kScanThreads, 2) scan_limb_kernel(const ScanArgs a)
{
    __shared__ __align__(16) LimbShared sh_all[kScanThreads / 32];
    const int lane = threadIdx.x & 31;
    LimbShared &sm = sh_all[threadIdx.x >> 5];
    int64_t Treg = 0;
    persistent_units<int64_t, 1>(a, lane, Treg, [&](const Inst &d, int inst, uint64_t unit) {
        scan_unit_limbs<K1>(a, d, inst, unit, Treg, lane, sm);
    });
}

template <bool K1>
constexpr auto plain_kernel()
{
    constexpr int kS = cols_per_thread(sizeof(int64_t), 0);
    static_assert(ilog2c(32 * kS) == suffix_bits(sizeof(int64_t), 0), "suffix bits must match the column layout");
    static_assert(kS == kLimbCols, "both kernels take the same suffix split");
    return scan_kernel<int64_t, kS, kVariantRegRows[0], K1, kVariantMinBlocks[0], kVariantAddMode[0],
                       kVariantMinInputs[0]>;
}

template <bool K1>
auto pick(int variant)
{
    return variant == kLimbVariant ? scan_limb_kernel<K1> : plain_kernel<K1>();
}
}  // namespace

template <>
cudaError_t launch_tables_t<int64_t>(const Inst *d_inst, int n_inst, int max_entries, cudaStream_t s)
{
    if (n_inst <= 0)
        return cudaSuccess;
    const int threads = 256;
    int bx = (max_entries + threads - 1) / threads;
    if (bx < 1)
        bx = 1;
    if (bx > 4096)
        bx = 4096;
    tables_kernel<int64_t><<<dim3(bx, n_inst), threads, 0, s>>>(d_inst);
    return cudaGetLastError();
}

template <>
cudaError_t launch_scan_t<int64_t>(const ScanArgs &a, int blocks, int variant, cudaStream_t s)
{
    auto k = a.k1 ? pick<true>(variant) : pick<false>(variant);
    k<<<blocks, kScanThreads, 0, s>>>(a);
    return cudaGetLastError();
}

template <>
int scan_blocks_per_sm_t<int64_t>(bool k1, int variant)
{
    int nb = 0;
    auto k = k1 ? pick<true>(variant) : pick<false>(variant);
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, kScanThreads, 0);
    return e == cudaSuccess ? nb : -1;
}

}  // namespace qubo

// qs_rowquant.cuh -- quantising rows of a state (Sec. 3, "Levels and storage") in the row layout,
// shared by the row-unit write-back and the pack kernel (sm_103a).
//
// Row layout: TPR = dv / 32 lanes per row, each owning 32 consecutive value columns, i.e. a
// word-aligned run of 32 codes (4w bytes); RPB = 32 / TPR rows per warp.  Warps take batches of RPB
// rows in order of output width, so that the code arithmetic of a warp is specialised for one width
// and its rows' searches end at similar candidates.
#pragma once

#include "qs_common.cuh"

namespace qs {

template <int DV>
struct RowQuant {
    static constexpr int TPR = DV / 32;
    static constexpr int RPB = 32 / TPR;
    static constexpr int KPT = kNFit / TPR;   // candidate steps each lane of a row prepares
    // A row's candidate table: kNFit / 2 pairs of 16 bytes.  So that the rows of a warp read one pair
    // from different banks they are permuted by row at dv = 128, where 8 KB for 8 warps is what two
    // CTAs per SM leave, and padded at dv = 64 (an operation less per round: Mamba-2 802 against
    // 812 us).
    static constexpr int kTable = kNFit / 2 + (TPR == 2 ? 1 : 0);
    static constexpr int kSwizzle = TPR == 2 ? 0 : kNFit / 2 - 1;
};

// (n, 1/n, kMagic - n, kMagic + n) of a width, n = 2^(w-1) - 1 (0 below 2 bits).
__device__ __forceinline__ float4 width_consts(int w) {
    const float n = w >= 2 ? static_cast<float>((1 << (w - 1)) - 1) : 0.0f;
    return make_float4(n, w >= 2 ? __frcp_rn(n) : 0.0f, kMagic - n, kMagic + n);
}

// The lane's codes occupy the 4W bytes at byte 4 W q of the row (q = its part), a whole number of
// words: code c of the run sits at bits [c W, c W + W) of those words.

// Packing.  With t_c = fl(x_c / Delta) + kMagic (round to nearest even; its bit pattern is
// kMagicBits + q_c), the stored code u_c = clamp(q_c + n, 0, 2n) is one add-min-relu on the bits;
// codes are shifted into the lane's words (codes that straddle two words add their high bits to
// the next word).
template <int W, int C>
__device__ __forceinline__ void run_put(uint32_t (&wd)[W], uint32_t u) {
    constexpr int bp = C * W, k = bp >> 5, sh = bp & 31;
    wd[k] += u << sh;
    if constexpr (sh + W > 32) wd[k + 1] += u >> (32 - sh);
}

// PAIRS: the product and the rounding add as packed operations, which the compiler may fuse into
// one (a code at x / Delta within an ulp of a half-integer can then fall the other way); otherwise one
// by one, each rounded, with the clamp on the floats (a NaN gets the lowest code).
template <int W, int C, bool PAIRS>
struct RunEncode {
    __device__ __forceinline__ static void go(uint32_t (&wd)[W], const float2 (&xv)[16], float2 i2, int off, int top) {
        if constexpr (!PAIRS) {
            const float n = static_cast<float>(top / 2);
            const float tx = code_magic(xv[C / 2].x, i2.x, kMagic - n, kMagic + n);
            const float ty = code_magic(xv[C / 2].y, i2.y, kMagic - n, kMagic + n);
            run_put<W, C>(wd, static_cast<uint32_t>(__float_as_int(tx) + off));
            run_put<W, C + 1>(wd, static_cast<uint32_t>(__float_as_int(ty) + off));
            RunEncode<W, C + 2, PAIRS>::go(wd, xv, i2, off, top);
            return;
        }
        const float2 t = __fadd2_rn(__fmul2_rn(xv[C / 2], i2), make_float2(kMagic, kMagic));
        run_put<W, C>(wd, static_cast<uint32_t>(__viaddmin_s32_relu(__float_as_int(t.x), off, top)));
        run_put<W, C + 1>(wd, static_cast<uint32_t>(__viaddmin_s32_relu(__float_as_int(t.y), off, top)));
        RunEncode<W, C + 2, PAIRS>::go(wd, xv, i2, off, top);
    }
};
template <int W, bool PAIRS>
struct RunEncode<W, 32, PAIRS> {
    __device__ __forceinline__ static void go(uint32_t (&)[W], const float2 (&)[16], float2, int, int) {}
};

// MAXA: alignment of the row starts (16 bytes for dv = 128, 8 for dv = 64).
template <int NWD, int MAXA>
__device__ __forceinline__ void store_words(uint8_t* dst, const uint32_t (&wd)[NWD]) {
    if constexpr (NWD % 4 == 0 && MAXA >= 16) {
#pragma unroll
        for (int k = 0; k < NWD; k += 4)
            *reinterpret_cast<uint4*>(dst + 4 * k) = make_uint4(wd[k], wd[k + 1], wd[k + 2], wd[k + 3]);
    } else if constexpr (NWD % 2 == 0) {
#pragma unroll
        for (int k = 0; k < NWD; k += 2) *reinterpret_cast<uint2*>(dst + 4 * k) = make_uint2(wd[k], wd[k + 1]);
    } else {
#pragma unroll
        for (int k = 0; k < NWD; ++k) reinterpret_cast<uint32_t*>(dst)[k] = wd[k];
    }
}

// Quantise + pack the lane's 32 values (row of width W) to dst (4W bytes at byte 4 W q of a row
// aligned to MAXA bytes): q = clamp(rint(x / Delta), -n, n), offset binary.
template <int W, int MAXA, bool EXACT>
__device__ __forceinline__ void pack_run(const float2 (&xv)[16], float inv, uint8_t* dst) {
    if constexpr (W == 1) {
        // sign bit, code 1 for x < 0 (negative zero counts as positive)
        uint32_t wd[1] = {0u};
#pragma unroll
        for (int c = 0; c < 16; ++c) {
            wd[0] |= (xv[c].x < 0.0f ? 1u : 0u) << (2 * c);
            wd[0] |= (xv[c].y < 0.0f ? 2u : 0u) << (2 * c);
        }
        store_words<1, MAXA>(dst, wd);
    } else if constexpr (W >= 2) {
        constexpr int n = (1 << (W - 1)) - 1;
        uint32_t wd[W];
#pragma unroll
        for (int k = 0; k < W; ++k) wd[k] = 0u;
        RunEncode<W, 0, !EXACT>::go(wd, xv, make_float2(inv, inv), n - static_cast<int>(kMagicBits), 2 * n);
        store_words<W, MAXA>(dst, wd);
    }
}

template <int MAXA, bool EXACT = false>
__device__ __forceinline__ void pack_row(int w, const float2 (&xv)[16], float inv, uint8_t* dst) {
    switch (w) {
#define QS_W(N) case N: pack_run<N, MAXA, EXACT>(xv, inv, dst); break;
        QS_W(1) QS_W(2) QS_W(3) QS_W(4) QS_W(5) QS_W(6) QS_W(7) QS_W(8)
        QS_W(9) QS_W(10) QS_W(11) QS_W(12) QS_W(13) QS_W(14) QS_W(15) QS_W(16)
#undef QS_W
        default: break;
    }
}

// One warp: the DK rows in order of output width and, within a width, of the factor last fitted
// (a close predictor of the next), any order among equals.  Widths 2..16 come first in ascending
// order (the narrowest rows have the longest range-factor search), then widths 1 and 0; within a
// width the smaller factors first (the search runs from the largest factor down, so they search
// longest).  A counting sort over the 17 x 16 keys: histogram, exclusive scan, ranks from the
// atomics.  hist: 17 * kNFit + 16 ints of shared memory.  key(i): width and factor of row i.
template <int DK, class Key>
__device__ __forceinline__ void order_rows(uint8_t* order, int* hist, int lane, Key key_of) {
    constexpr int PER = DK / 32, NK = 17 * kNFit, KPL = (NK + 31) / 32;
    for (int k = lane; k < NK; k += 32) hist[k] = 0;
    __syncwarp();
    int key[PER], rank[PER];
#pragma unroll
    for (int jj = 0; jj < PER; ++jj) {
        int w, f;
        key_of(lane * PER + jj, w, f);
        key[jj] = ((min(w, 16) + 15) % 17) * kNFit + (f & (kNFit - 1));
        rank[jj] = atomicAdd(&hist[key[jj]], 1);
    }
    __syncwarp();
    int cnt[KPL], sum = 0;
#pragma unroll
    for (int m = 0; m < KPL; ++m) {
        const int k = lane * KPL + m;
        cnt[m] = sum;
        sum += k < NK ? hist[k] : 0;
    }
    int incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int n = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += n;
    }
    __syncwarp();
#pragma unroll
    for (int m = 0; m < KPL; ++m) {
        const int k = lane * KPL + m;
        if (k < NK) hist[k] = incl - sum + cnt[m];
    }
    __syncwarp();
#pragma unroll
    for (int jj = 0; jj < PER; ++jj) order[hist[key[jj]] + rank[jj]] = static_cast<uint8_t>(lane * PER + jj);
}

// The factor search of a warp's batch: av the lane's 32 magnitudes, m4 the maxima of four
// disjoint parts of them, R the row's range (equal over its lanes), w its width with constants wc; table: the row's candidate table, in
// the warp's own shared memory.  Returns the row's best factor index (kNFit - 1 for
// rows below 2 bits and zero rows) and its step in D (untouched below 2 bits).  TIES: also says, in
// `close`, whether another candidate's error lies within a relative 2^-19 (n + 2) of the best: more
// than approximate reciprocals, one rounding instead of two before the rint, and another order
// of the sum can change an error (a position in steps moves by at most n 2^-22, and an error
// by 8 times that, where every element sat on a rounding boundary).
template <int DV, bool TIES = false>
__device__ __forceinline__ int fit_rows(const float2 (&av)[16], const float (&m4)[4], float R, int w, float4 wc, const float* fitf,
                                        float4* table, int lane, float& D, bool* close = nullptr) {
    constexpr int TPR = RowQuant<DV>::TPR, KPT = RowQuant<DV>::KPT;
    const int q = lane % TPR, sw = (lane / TPR) & RowQuant<DV>::kSwizzle;
    __syncwarp();   // the previous batch's rows are done with the candidate table
    // the row's 16 candidate steps, KPT per lane.  The search takes approximate
    // reciprocals; the chosen step's IEEE reciprocal is taken for the codes.
#pragma unroll
    for (int kk = 0; kk < KPT; kk += 2) {
        const int k = q * KPT + kk;   // even
        float2 d, iv;
        cand_pair(__fmul2_rn(*reinterpret_cast<const float2*>(fitf + k), make_float2(R, R)), wc.y, d, iv);
        table[(k / 2) ^ sw] = make_float4(iv.x, -d.x, iv.y, -d.y);
    }
    __syncwarp();
    // squared error of the candidates (levels clamped at n): e = |x| - q Delta,
    // q = min(rint(|x| / Delta), n); the smallest wins, ties to the larger factor.
    // Candidates are taken from the largest factor down, two per round (independent
    // work for the warp).  Every element at or above n Delta_k quantises to n, so the
    // clipping error of some of them is a lower bound on candidate k's error that
    // grows as k falls: once it exceeds the best error found (with a 2^-10 margin for
    // rounding), no smaller factor can win.  The round's second candidate is evaluated
    // even when its bound already rules it out; it then cannot win the comparison.
    const float nf = wc.x, off = level_offset(nf), nulp = nf * kLevelUlp;
    // A candidate's bound.  dv = 128: from 4 maxima of 8 elements per lane, summed over the row's
    // lanes (about half an evaluation per row fewer than from the 4 lane maxima: KDA decode 357
    // against 360 us per token, pack 78 against 80); made one round ahead, beside the evaluations.
    // dv = 64: from the row's 2 lane maxima, without a sum (Mamba-2, whose wider rows stop
    // early: 201 against 206 us).
    float mx[2];
    if constexpr (TPR == 2) {
        const float lmax = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3]));
        mx[0] = lmax;
        mx[1] = __shfl_xor_sync(kFull, lmax, 1);
    }
    auto bound = [&](float d_ulp) {
        float lb = 0.0f;
#pragma unroll
        for (int j = 0; j < (TPR == 2 ? 2 : 4); ++j) {
            const float e = fmaxf(fmaf(nulp, d_ulp, TPR == 2 ? mx[j & 1] : m4[j]), 0.0f);
            lb = fmaf(e, e, lb);
        }
        if constexpr (TPR != 2) {
#pragma unroll
            for (int o = 1; o < TPR; o <<= 1) lb += __shfl_xor_sync(kFull, lb, o);
        }
        return lb;
    };
    const float2 noff = make_float2(-off, -off);
    const bool live = w >= 2 && R > 0.0f;   // a zero row keeps the largest factor
    float bsse = INFINITY, second = INFINITY;
    int bk = kNFit - 1;
    const float near = 1.0f + 0x1p-19f * (nf + 2.0f);
    // the bound's margin: 2^-10, or what `close` has to see
    const float margin = TIES ? fmaxf(1.0f + 0x1p-10f, near * near) : 1.0f + 0x1p-10f;
    // each round's two candidates are loaded one round ahead
    float4 next = table[(kNFit / 2 - 1) ^ sw];
    float lbA = 0.0f;   // the first round always runs
#pragma unroll 1
    for (int k = kNFit - 1; k >= 0; k -= 2) {
        // candidates k and k - 1 in one round
        const float2 cA = make_float2(next.z, next.w), cB = make_float2(next.x, next.y);
        if constexpr (TPR == 2) lbA = bound(cA.y);
        const bool goA = live && lbA <= bsse * margin;
        if constexpr (TPR == 2) {
            if (k >= 3) next = table[(k / 2 - 1) ^ sw];
        }
        if (!__any_sync(kFull, goA)) break;
        if constexpr (TPR != 2) {
            if (k >= 3) next = table[(k / 2 - 1) ^ sw];
            lbA = bound(next.w);
        }
        const float2 dA = make_float2(cA.y, cA.y), dB = make_float2(cB.y, cB.y);
        float2 aA0 = make_float2(0.0f, 0.0f), aA1 = aA0, aB0 = aA0, aB1 = aA0;
#pragma unroll
        for (int c = 0; c < 16; c += 2) {
            const float2 t0 = make_float2(round_level(av[c].x, cA.x, off), round_level(av[c].y, cA.x, off));
            const float2 t1 = make_float2(round_level(av[c + 1].x, cA.x, off), round_level(av[c + 1].y, cA.x, off));
            const float2 u0 = make_float2(round_level(av[c].x, cB.x, off), round_level(av[c].y, cB.x, off));
            const float2 u1 = make_float2(round_level(av[c + 1].x, cB.x, off), round_level(av[c + 1].y, cB.x, off));
            const float2 e0 = __ffma2_rn(__fadd2_rn(t0, noff), dA, av[c]);
            const float2 e1 = __ffma2_rn(__fadd2_rn(t1, noff), dA, av[c + 1]);
            const float2 f0 = __ffma2_rn(__fadd2_rn(u0, noff), dB, av[c]);
            const float2 f1 = __ffma2_rn(__fadd2_rn(u1, noff), dB, av[c + 1]);
            aA0 = __ffma2_rn(e0, e0, aA0);
            aA1 = __ffma2_rn(e1, e1, aA1);
            aB0 = __ffma2_rn(f0, f0, aB0);
            aB1 = __ffma2_rn(f1, f1, aB1);
        }
        float tA = (aA0.x + aA0.y) + (aA1.x + aA1.y);
        float tB = (aB0.x + aB0.y) + (aB1.x + aB1.y);
#pragma unroll
        for (int o = 1; o < TPR; o <<= 1) {
            tA += __shfl_xor_sync(kFull, tA, o);
            tB += __shfl_xor_sync(kFull, tB, o);
        }
        if constexpr (TIES) second = fminf(second, fminf(fmaxf(tA, tB), fmaxf(fminf(tA, tB), bsse)));
        if (goA && tA < bsse) {
            bsse = tA;
            bk = k;
        }
        if (live && tB < bsse) {
            bsse = tB;
            bk = k - 1;
        }
    }
    if (w >= 2) D = -reinterpret_cast<const float2*>(table + ((bk / 2) ^ sw))[bk & 1].y * kLevelUlp;
    if constexpr (TIES) *close = live && !(second > bsse * near);
    return bk;
}

// Sum of a row in a fixed order: C consecutive values added one by one, for each 32nd of the row,
// and those 32 sums by halves (l and l + 16, then l and l + 8, ...).  part: the lane's 32 / C sums.
template <int DV>
struct RowSum {
    static constexpr int C = DV / 32, NP = 32 / C;
    __device__ __forceinline__ static float total(float (&part)[NP]) {
#pragma unroll
        for (int o = RowQuant<DV>::TPR / 2; o > 0; o >>= 1)
#pragma unroll
            for (int j = 0; j < NP; ++j) part[j] += __shfl_xor_sync(kFull, part[j], o);
#pragma unroll
        for (int o = NP / 2; o > 0; o >>= 1)
#pragma unroll
            for (int j = 0; j < o; ++j) part[j] += part[j + o];
        return part[0];
    }
};

__device__ __forceinline__ float lane_value(const float2 (&v)[16], int c) { return c & 1 ? v[c / 2].y : v[c / 2].x; }

// The factor search with IEEE reciprocals, products and sums rounded one by one, and the row's
// errors summed in RowSum's order: what decides between candidates whose errors are close.
template <int DV>
__device__ __noinline__ int fit_rows_exact(const float2 (&av)[16], float R, float4 wc, const float* fitf, float& D) {
    float best = INFINITY;
    int bk = kNFit - 1;
#pragma unroll 1
    for (int k = kNFit - 1; k >= 0; --k) {
        const float Dk = cand_step(fitf[k], R, wc.y), inv = step_rcp(Dk);
        float part[RowSum<DV>::NP];
#pragma unroll
        for (int c = 0; c < 32; ++c) {
            const float a = lane_value(av, c);
            const float t = fminf(__fadd_rn(__fmul_rn(a, inv), kMagic), wc.w);
            const float e = fmaf(-__fsub_rn(t, kMagic), Dk, a);
            float& s = part[c / RowSum<DV>::C];
            s = fmaf(e, e, c % RowSum<DV>::C == 0 ? 0.0f : s);
        }
        const float tot = RowSum<DV>::total(part);
        if (tot < best) {
            best = tot;
            bk = k;
        }
    }
    D = cand_step(fitf[bk], R, wc.y);
    return bk;
}

}  // namespace qs

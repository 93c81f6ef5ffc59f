// qs_pack_row.cuh -- pack and unpack for the row allocation unit (sm_103a): a dense state into the
// packed form (Sec. 3, "Levels and storage") and back.
#pragma once

#include "qs_rowquant.cuh"

namespace qs {

// ---- pack ------------------------------------------------------------------------------------
// One CTA of 4 warps per head.  Two warps make the row offsets (prefix sum of the widths, with
// the layout check) and the order of the rows by width; then every warp claims batches of RPB rows,
// loads each lane's 32 consecutive values of its row straight from the dense state, and quantises
// and stores them without any exchange beyond the row's TPR lanes.  16 warps per SM: the loads of
// some hide behind the searches of the others.
// What bounds it: the search's FP32 work (47 lane-instructions per element in all; issue 59 %, FMA pipe
// 56 % of the time, the loads' latency next), ahead of HBM (64 KB read per head).  64 x 32 heads of 128 x 128, 4 bits: 78 us (151 MB, 1.9 TB/s); 214 us with all
// 16 candidates of every row in scalar arithmetic, a row spread over a warp.  Results are those of that
// arithmetic bit for bit (each product and sum of a code rounded by itself, near ties between factors
// decided by fit_rows_exact); without that it took 80 us when it took 88 with it.
template <int DK, int DV>
struct alignas(16) PackSmem {
    static constexpr int NW = 4;
    float4 cand[NW][RowQuant<DV>::RPB][RowQuant<DV>::kTable];
    float4 wc[17];
    alignas(8) float fitf[kNFit];
    int off[DK];
    int hist[17 * kNFit + 16];
    uint8_t w[DK], order[DK];
    int flag, next;
};

// The dense state's alignment: 4 bytes with BY4, else vec: 16 (else 8).
template <int DK, int DV, bool BY4>
__global__ void __launch_bounds__(128, 4) pack_row_kernel(const __grid_constant__ StepParams p, bool vec) {
    using RQ = RowQuant<DV>;
    constexpr int TPR = RQ::TPR, RPB = RQ::RPB, NB = DK / RPB, NW = PackSmem<DK, DV>::NW;
    __shared__ PackSmem<DK, DV> sm;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = blockIdx.x, b = g / p.H;
    const size_t rb = static_cast<size_t>(g) * DK;
    const long long hoff = p.out_head_off[g];
    constexpr int PER = DK / 32;
    if (warp == 0) {
        int loc[PER], sum = 0;
        bool bad = false;
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            const int w = p.out_widths[rb + lane * PER + j];
            sm.w[lane * PER + j] = static_cast<uint8_t>(w);
            bad |= w > 16;
            loc[j] = sum;
            sum += w * (DV / 8);
        }
        int incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int n = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += n;
        }
#pragma unroll
        for (int j = 0; j < PER; ++j) sm.off[lane * PER + j] = incl - sum + loc[j];
        const int total = __shfl_sync(kFull, incl, 31);
        bad = __any_sync(kFull, bad) || hoff + total > p.region_bytes || hoff % (DV == 128 ? 16 : 8) != 0 ||
              total > p.stage_bytes;
        if (lane == 0) {
            sm.flag = bad ? 1 : 0;
            sm.next = NW;
        }
    } else if (warp == 1) {
        order_rows<DK>(sm.order, sm.hist, lane, [&](int i, int& w, int& f) {
            w = p.out_widths[rb + i];
            f = 0;
        });
    } else if (warp == 2) {
        if (lane < kNFit) sm.fitf[lane] = fit_factor(lane);
    } else if (lane < 17) {
        sm.wc[lane] = width_consts(lane);
    }
    __syncthreads();
    if (sm.flag) {
        if (tid == 0) raise_status(p.status, QS_DEV_LAYOUT);
        return;
    }
    uint8_t* out = p.out_payload + static_cast<size_t>(b) * p.region_bytes + hoff;
    const int q = lane % TPR;
    auto claim = [&]() {
        int n = 0;
        if (lane == 0) n = atomicAdd(&sm.next, 1);
        return __shfl_sync(kFull, n, 0);
    };
    for (int bat = warp; bat < NB; bat = claim()) {
        const int i = sm.order[bat * RPB + lane / TPR];
        const int w = sm.w[i];
        float2 xv[16], av[16];
        if (p.dense_in != nullptr) {
            const float* src = p.dense_in + (rb + i) * DV + 32 * q;
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                if constexpr (BY4) {
                    xv[2 * c] = make_float2(src[4 * c], src[4 * c + 1]);
                    xv[2 * c + 1] = make_float2(src[4 * c + 2], src[4 * c + 3]);
                } else if (vec) {
                    const float4 v = __ldcs(reinterpret_cast<const float4*>(src + 4 * c));
                    xv[2 * c] = make_float2(v.x, v.y);
                    xv[2 * c + 1] = make_float2(v.z, v.w);
                } else {
                    xv[2 * c] = *reinterpret_cast<const float2*>(src + 4 * c);
                    xv[2 * c + 1] = *reinterpret_cast<const float2*>(src + 4 * c + 2);
                }
            }
        } else {
#pragma unroll
            for (int c = 0; c < 16; ++c) xv[c] = make_float2(0.0f, 0.0f);
        }
        float m4[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int c = 0; c < 16; ++c) {
            av[c] = make_float2(fabsf(xv[c].x), fabsf(xv[c].y));
            m4[c & 3] = fmaxf(m4[c & 3], fmaxf(av[c].x, av[c].y));
        }
        const float lmax = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3]));
        float R = lmax;
#pragma unroll
        for (int o = 1; o < TPR; o <<= 1) R = fmaxf(R, __shfl_xor_sync(kFull, R, o));
        float D = 0.0f;
        int fidx = p.in_fidx ? p.in_fidx[rb + i] : kNFit - 1;
        if (__any_sync(kFull, w == 1)) {   // 1-bit rows: mean |x|
            float part[RowSum<DV>::NP];
#pragma unroll
            for (int c = 0; c < 32; ++c) {
                float& s = part[c / RowSum<DV>::C];
                s = (c % RowSum<DV>::C == 0 ? 0.0f : s) + lane_value(av, c);
            }
            const float sum = RowSum<DV>::total(part);
            if (w == 1) D = f16_round(__fdiv_rn(sum, static_cast<float>(DV)));
        }
        bool close = false;
        const int bk = fit_rows<DV, true>(av, m4, R, w, sm.wc[w], sm.fitf, sm.cand[warp][lane / TPR], lane, D, &close);
        if (w >= 2) fidx = bk;
        if (__any_sync(kFull, close)) {
            // near ties (a few rows in a million at 4 bits): decided in a fixed arithmetic, which
            // does not depend on how the search is computed
            float De = 0.0f;
            const int be = fit_rows_exact<DV>(av, R, sm.wc[w], sm.fitf, De);
            if (close) {
                fidx = be;
                D = De;
            }
        }
        if (q == 0) {
            p.out_scales[rb + i] = f16_bits(D);
            p.out_fidx[rb + i] = static_cast<uint8_t>(fidx);
            if (p.range) p.range[rb + i] = R;
        }
        pack_row<DV == 128 ? 16 : 8, true>(w, xv, w >= 2 ? step_rcp(D) : 0.0f, out + sm.off[i] + 4 * w * q);
    }
}

template <int DK, int DV>
cudaError_t launch_pack_row_t(const qstate_cfg& cfg, const StepParams& p, cudaStream_t stream) {
    StepParams q = p;
    q.stage_bytes = DK * DV * cfg.bmax / 8;
    const uintptr_t at = reinterpret_cast<uintptr_t>(p.dense_in);
    auto kern = at % 8 == 0 ? pack_row_kernel<DK, DV, false> : pack_row_kernel<DK, DV, true>;
    kern<<<cfg.B * cfg.H, 128, 0, stream>>>(q, at % 16 == 0);
    return cudaGetLastError();
}

// ---- unpack ----------------------------------------------------------------------------------
// One CTA of 8 warps per head, small enough for 6 CTAs per SM: a head is two dependent loads
// (widths and payload, both issued at once) and 64 KB of stores, and many heads in flight keep the
// stores going.  The payload window is taken from the neighbouring head offsets so that its copy
// does not wait for the sum of the widths; if the widths ask for more, the rest is copied after.
// Lanes decode four consecutive codes and store 16 bytes; at dv = 64 the half-warps take
// alternate rows.  A dense state that is not 16-byte aligned: every 32nd (16th) column to a lane, so that
// its 4-byte stores have no gaps.
// What bounds it: HBM, 64 KB written per head.  64 x 32 heads of 128 x 128, 4 bits: 26.6 us (151 MB,
// 5.7 TB/s); 45 us with two CTAs of 256 threads per SM, whose loads, prefix sum and stores followed one
// another.
template <int DK, int DV>
struct alignas(16) UnpackSmem {
    float4 deq[DK];   // (A, S, B, width): x = (2^23 + u - A) S + B
    int off[DK];
    int total, flag, pad[2];
};

// VEC: the dense state is 16-byte aligned.
template <int DK, int DV, bool VEC>
__global__ void __launch_bounds__(256, 6) unpack_row_kernel(const __grid_constant__ StepParams p) {
    extern __shared__ __align__(16) uint8_t smem_raw[];
    UnpackSmem<DK, DV>& sm = *reinterpret_cast<UnpackSmem<DK, DV>*>(smem_raw);
    uint8_t* pay = smem_raw + sizeof(UnpackSmem<DK, DV>);
    constexpr int kVec = DV == 128 ? 16 : 8;   // alignment of rows
    using Vec = typename std::conditional<DV == 128, uint4, uint2>::type;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = blockIdx.x, b = g / p.H, h = g - b * p.H;
    const size_t rb = static_cast<size_t>(g) * DK;
    const long long hoff = p.in_head_off[g];
    const long long hend = h + 1 < p.H ? static_cast<long long>(p.in_head_off[g + 1]) : p.region_bytes;
    const uint8_t* src = p.in_payload + static_cast<size_t>(b) * p.region_bytes + hoff;
    const bool sane = hoff % kVec == 0 && hoff <= hend && hend <= p.region_bytes;
    const int first = sane ? static_cast<int>(min(hend - hoff, static_cast<long long>(p.stage_bytes))) / kVec * kVec : 0;
    for (int i = tid; i < first / kVec; i += 256) reinterpret_cast<Vec*>(pay)[i] = __ldcs(reinterpret_cast<const Vec*>(src) + i);
    if (warp == 0) {
        constexpr int PER = DK / 32;
        int loc[PER], sum = 0;
        bool bad = false;
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            const int w = p.in_widths[rb + lane * PER + j];
            bad |= w > 16;
            loc[j] = sum;
            sum += w * (DV / 8);
        }
        int incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int n = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += n;
        }
#pragma unroll
        for (int j = 0; j < PER; ++j) sm.off[lane * PER + j] = incl - sum + loc[j];
        const int total = __shfl_sync(kFull, incl, 31);
        bad = __any_sync(kFull, bad) || hoff + total > p.region_bytes || hoff % kVec != 0 || total > p.stage_bytes;
        if (lane == 0) {
            sm.total = total;
            sm.flag = bad ? 1 : 0;
        }
    } else if (tid >= 64 && tid < 64 + DK) {
        // w >= 2: q Delta; w = 1: +-m; w = 0: 0 (float(u) is 2^23 + u built from the code's bits)
        const int i = tid - 64, w = min(static_cast<int>(p.in_widths[rb + i]), 16);
        const float D = f16_value(p.in_scales[rb + i]);
        sm.deq[i] = make_float4(8388608.0f + static_cast<float>(w >= 2 ? (1 << (w - 1)) - 1 : 0),
                                w >= 2 ? D : (w == 1 ? -2.0f * D : 0.0f), w == 1 ? D : 0.0f, __int_as_float(w));
    }
    __syncthreads();
    if (sm.flag) {
        if (tid == 0) raise_status(p.status, QS_DEV_LAYOUT);
        return;
    }
    if (sm.total > first) {   // offsets that are not those of the widths
        for (int i = first / kVec + tid; i < sm.total / kVec; i += 256)
            reinterpret_cast<Vec*>(pay)[i] = reinterpret_cast<const Vec*>(src)[i];
        __syncthreads();
    }
    constexpr int RS = 128 / DV;   // rows that a warp decodes at once
    const int half = lane / (32 / RS), cl = lane % (32 / RS);
    if constexpr (!VEC) {
#pragma unroll 2
        for (int r = warp * RS + half; r < DK; r += 8 * RS) {
            const float4 dq = sm.deq[r];
            const int w = __float_as_int(dq.w);
            const uint32_t* words = reinterpret_cast<const uint32_t*>(pay + sm.off[r]);
            float* o = p.dense_out + (rb + r) * DV;
#pragma unroll
            for (int col = cl; col < DV; col += 32 / RS) {
                const int P = col * w, idx = P >> 5;
                const uint32_t u = __funnelshift_r(words[idx], words[idx + 1], P & 31) & ((1u << w) - 1u);
                o[col] = fmaf(__fsub_rn(__uint_as_float(kTwo23Bits | u), dq.x), dq.y, dq.z);
            }
        }
        return;
    }
    float* dst = p.dense_out + rb * DV + cl * 4;
#pragma unroll 4
    for (int r = warp * RS + half; r < DK; r += 8 * RS) {
        const float4 dq = sm.deq[r];
        const int w = __float_as_int(dq.w);
        const uint32_t* words = reinterpret_cast<const uint32_t*>(pay + sm.off[r]);
        const int P = cl * 4 * w, idx = P >> 5, sh = P & 31;
        const uint32_t mask = (1u << w) - 1u;
        const uint32_t lo = __funnelshift_r(words[idx], words[idx + 1], sh);
        const uint32_t hi = __funnelshift_r(words[idx + 1], words[idx + 2], sh);
        const uint64_t chunk = (static_cast<uint64_t>(hi) << 32) | lo;
        float x[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const uint32_t u = static_cast<uint32_t>(chunk >> (c * w)) & mask;
            x[c] = fmaf(__fsub_rn(__uint_as_float(kTwo23Bits | u), dq.x), dq.y, dq.z);
        }
        __stcs(reinterpret_cast<float4*>(dst + r * DV), make_float4(x[0], x[1], x[2], x[3]));
    }
}

template <int DK, int DV>
cudaError_t launch_unpack_row_t(const qstate_cfg& cfg, const StepParams& p, cudaStream_t stream) {
    StepParams q = p;
    q.stage_bytes = DK * DV * cfg.bmax / 8;
    const int smem = static_cast<int>(sizeof(UnpackSmem<DK, DV>)) + q.stage_bytes + 16;   // 12 readable bytes
    const bool vec = (reinterpret_cast<uintptr_t>(p.dense_out) & 15) == 0;
    auto kern = vec ? unpack_row_kernel<DK, DV, true> : unpack_row_kernel<DK, DV, false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    kern<<<cfg.B * cfg.H, 256, smem, stream>>>(q);
    return cudaGetLastError();
}

}  // namespace qs

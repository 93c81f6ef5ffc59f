// qs_fp32.cu -- Eq. (1) on an unquantised FP32 state (qstate_scan_fp32).
//
// An FP32 state does not change on its way through memory, so a call's tokens run in one launch
// with the state in registers: it is read once and written once, whatever the write-back period.
//
// The value columns of a head are independent (p_j, u_j, o_j and column j of the state need only
// column j and the token's row vectors), so a CTA of 4 warps takes 64 columns of a head and a warp
// 16 of them over all key rows, with no exchange between warps.  Lane (rg, cg) = (lane / 2,
// lane % 2) owns RL = dk / 16 rows x 8 columns (two runs of 4, so that a lane pair's 16-byte accesses
// fill 32-byte sectors).  Per token it reads its rows' d, k and q from
// shared memory (24 bytes per row for 8 columns x 4 multiply-adds: with 4 columns per lane the
// shared-memory path would be as busy as the FMA pipe), decays, and forms p = a^T S' and r = q^T S'
// over its rows with row pairs as packed operands (d, k and q come from memory as pairs); 15
// shuffles of recursive halving leave each lane one of the warp's 32 sums; u goes round through
// shared memory.  The inputs of 8 tokens are copied ahead with cp.async while the 8 before them
// run; the rates become decays in place.  Two CTA barriers per 8 tokens.
//
// What bounds it: 4 FMA-pipe operations per element and token (the pipe is 54 % busy) and, between
// them, the chain of each token's sums, which the 16 warps per SM do not quite hide.  16 x 32 heads
// of 128 x 128, 32 tokens: 74 us; 463 us with a launch per token, each reading and writing the
// state (67 MB).
// Calls of one or two tokens, which are little but the state's way through memory, have a kernel of their
// own (below).
#include "qs_common.cuh"

namespace qs {

namespace {

constexpr int kTB = 8;       // tokens per staged block
constexpr int kCols = 64;    // value columns per CTA
constexpr int kFpThreads = 128;

enum : int { kEraseNone = 0, kEraseDelta = 1, kEraseGeneral = 2 };

// One block's inputs: k, q and the decays of the rows, v of the CTA's columns, beta; a and w under
// general erasure.
template <int DK, int ERASE>
struct alignas(16) FpStage {
    float k[kTB][DK], q[kTB][DK], d[kTB][DK];
    float v[kTB][kCols];
    float a[ERASE == kEraseGeneral ? kTB : 1][DK], w[ERASE == kEraseGeneral ? kTB : 1][kCols];
    float beta[kTB];
    float pad[4];
};

template <int DK, int ERASE>
struct alignas(16) FpSmem {
    FpStage<DK, ERASE> st[2];
    float u[kFpThreads / 32][16];   // per warp
};

__device__ __forceinline__ void fp_cp16(float* smem, const float* gmem) {
    const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(smem));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void fp_cp4(float* smem, const float* gmem) {
    const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(smem));
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(s), "l"(gmem) : "memory");
}

// Halve the values a lane holds: lanes with bit `off` keep the upper N / 2 sums, the others the
// lower ones.
template <int N>
__device__ __forceinline__ void halve(float (&v)[16], int lane, int off) {
    const bool upper = (lane & off) != 0;
#pragma unroll
    for (int i = 0; i < N / 2; ++i) {
        const float send = upper ? v[i] : v[i + N / 2];
        const float keep = upper ? v[i + N / 2] : v[i];
        v[i] = keep + __shfl_xor_sync(kFull, send, off);
    }
}

// vec: bit 0 token inputs, bit 1 the state are 16-byte aligned.
template <int DK, int ERASE>
__global__ void __launch_bounds__(kFpThreads, 4) scan_fp32_kernel(const __grid_constant__ StepParams p, int dv, int vec) {
    constexpr int RL = DK / 16;   // rows per lane
    using Sm = FpSmem<DK, ERASE>;
    using St = FpStage<DK, ERASE>;
    extern __shared__ __align__(16) uint8_t smem_raw[];
    Sm& sm = *reinterpret_cast<Sm*>(smem_raw);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int parts = dv / kCols;
    const int bh = blockIdx.x / parts, c0 = (blockIdx.x - bh * parts) * kCols;
    const int b = bh / p.H, h = bh - b * p.H;
    // the lane's rows: four from 4 rg on, of every 64 (so that the lanes of a warp read a vector's
    // 64 values without gaps, on all banks)
    const int i0 = (lane >> 1) * 4;
    auto row = [](int r) { return (r / 4) * 64 + r % 4; };   // + i0
    // and columns: 4 from j0 on and 4 from j0 + 8 on, so that a lane pair's 16-byte accesses fill sectors
    const int j0 = c0 + 16 * warp + 4 * (lane & 1);

    auto issue = [&](St& S, int t0) {
        const int nt = min(kTB, p.t_end - t0);
        const size_t tok = (static_cast<size_t>(b) * p.T + t0) * p.H + h;   // + t H
        auto rows = [&](float (*dst)[DK], const float* src) {
            if (vec & 1) {
                for (int c = tid; c < nt * (DK / 4); c += kFpThreads) {
                    const int t = c / (DK / 4), i = c % (DK / 4) * 4;
                    fp_cp16(&dst[t][i], src + (tok + static_cast<size_t>(t) * p.H) * DK + i);
                }
            } else {
                for (int c = tid; c < nt * DK; c += kFpThreads) {
                    const int t = c / DK, i = c % DK;
                    fp_cp4(&dst[t][i], src + (tok + static_cast<size_t>(t) * p.H) * DK + i);
                }
            }
        };
        auto cols = [&](float (*dst)[kCols], const float* src) {
            if (vec & 1) {
                for (int c = tid; c < nt * (kCols / 4); c += kFpThreads) {
                    const int t = c / (kCols / 4), j = c % (kCols / 4) * 4;
                    fp_cp16(&dst[t][j], src + (tok + static_cast<size_t>(t) * p.H) * dv + c0 + j);
                }
            } else {
                for (int c = tid; c < nt * kCols; c += kFpThreads) {
                    const int t = c / kCols, j = c % kCols;
                    fp_cp4(&dst[t][j], src + (tok + static_cast<size_t>(t) * p.H) * dv + c0 + j);
                }
            }
        };
        rows(S.k, p.k);
        rows(S.q, p.q);
        if (p.decay_row && !p.s_code) rows(S.d, p.s);
        cols(S.v, p.v);
        if constexpr (ERASE == kEraseGeneral) {
            rows(S.a, p.a_in);
            cols(S.w, p.w_in);
        }
        if (ERASE == kEraseDelta && tid < nt) fp_cp4(&S.beta[tid], p.beta + tok + static_cast<size_t>(tid) * p.H);
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };

    issue(sm.st[0], p.t_begin);
    // the lane's state: rows in pairs, (row 2m, row 2m + 1) of each column
    float2 x[RL / 2][8];
    const float* src = p.dense_in + (static_cast<size_t>(bh) * DK + i0) * dv + j0;
#pragma unroll
    for (int r = 0; r < RL; ++r) {
        float t[8];
        if (vec & 2) {
            const float4 lo = *reinterpret_cast<const float4*>(src + row(r) * dv);
            const float4 hi = *reinterpret_cast<const float4*>(src + row(r) * dv + 8);
            t[0] = lo.x; t[1] = lo.y; t[2] = lo.z; t[3] = lo.w;
            t[4] = hi.x; t[5] = hi.y; t[6] = hi.z; t[7] = hi.w;
        } else {
#pragma unroll
            for (int c = 0; c < 8; ++c) t[c] = src[row(r) * dv + (c & 3) + 2 * (c & 4)];
        }
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            if (r & 1) x[r / 2][c].y = t[c];
            else x[r / 2][c].x = t[c];
        }
    }

    int buf = 0;
    for (int t0 = p.t_begin; t0 < p.t_end; t0 += kTB, buf ^= 1) {
        St& S = sm.st[buf];
        const int nt = min(kTB, p.t_end - t0);
        asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        __syncthreads();   // this block's inputs have landed; every warp is done with the one before
        if (t0 + kTB < p.t_end) issue(sm.st[buf ^ 1], t0 + kTB);
        {
            // rates -> decays; a thread keeps its row
            const int i = tid % DK;
            float rate[kTB * DK / kFpThreads];
            constexpr int step = kFpThreads / DK;
#pragma unroll
            for (int m = 0; m < kTB / step; ++m) {
                const int t = tid / DK + m * step;
                rate[m] = 1.0f;
                if (t >= nt) continue;
                const size_t tok = (static_cast<size_t>(b) * p.T + t0 + t) * p.H + h;
                if (p.s_code) {
                    const size_t ch = p.decay_row ? static_cast<size_t>(h) * DK + i : h;
                    const int code = p.s_code[p.decay_row ? tok * DK + i : tok];
                    rate[m] = __ldg(p.s_lut + ch * p.L + min(code, p.L - 1));
                } else {
                    rate[m] = p.decay_row ? S.d[t][i] : __ldg(p.s + tok);
                }
            }
            bool bad = false;
#pragma unroll
            for (int m = 0; m < kTB / step; ++m) {
                bad |= !(rate[m] > 0.0f) || !(rate[m] < INFINITY);
                S.d[tid / DK + m * step][i] = expf(-rate[m]);
            }
            if (bad) raise_status(p.status, QS_DEV_RATE);
        }
        __syncthreads();
#pragma unroll 1
        for (int t = 0; t < nt; ++t) {
            float2 pp[8], rr[8], kq2 = make_float2(0.0f, 0.0f);
#pragma unroll
            for (int c = 0; c < 8; ++c) pp[c] = rr[c] = make_float2(0.0f, 0.0f);
#pragma unroll
            for (int m = 0; m < RL / 2; m += 2) {
                const float4 d4 = *reinterpret_cast<const float4*>(&S.d[t][i0 + 32 * m]);
                const float4 k4 = *reinterpret_cast<const float4*>(&S.k[t][i0 + 32 * m]);
                const float4 q4 = *reinterpret_cast<const float4*>(&S.q[t][i0 + 32 * m]);
                float4 a4 = k4;   // delta rule: a = beta k, with beta taken out of the sum
                if constexpr (ERASE == kEraseGeneral) a4 = *reinterpret_cast<const float4*>(&S.a[t][i0 + 32 * m]);
                const float2 d2[2] = {make_float2(d4.x, d4.y), make_float2(d4.z, d4.w)};
                const float2 k2[2] = {make_float2(k4.x, k4.y), make_float2(k4.z, k4.w)};
                const float2 q2[2] = {make_float2(q4.x, q4.y), make_float2(q4.z, q4.w)};
                const float2 a2[2] = {make_float2(a4.x, a4.y), make_float2(a4.z, a4.w)};
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    kq2 = __ffma2_rn(k2[e], q2[e], kq2);
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        x[m + e][c] = __fmul2_rn(x[m + e][c], d2[e]);
                        if constexpr (ERASE != kEraseNone) pp[c] = __ffma2_rn(x[m + e][c], a2[e], pp[c]);
                        rr[c] = __ffma2_rn(x[m + e][c], q2[e], rr[c]);
                    }
                }
            }
            // sums over the 16 row groups: lane bits 4..1 end as (r or p, column bits 2, 1, 0);
            // without erasure bit 4 only halves the rows
            float s[16];
            float kq = kq2.x + kq2.y;
#pragma unroll
            for (int o = 2; o < 32; o <<= 1) kq += __shfl_xor_sync(kFull, kq, o);
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                s[c] = pp[c].x + pp[c].y;
                s[8 + c] = rr[c].x + rr[c].y;
            }
            if constexpr (ERASE != kEraseNone) {
                halve<16>(s, lane, 16);
            } else {
#pragma unroll
                for (int c = 0; c < 8; ++c) s[c] = s[8 + c];
            }
            halve<8>(s, lane, 8);
            halve<4>(s, lane, 4);
            halve<2>(s, lane, 2);
            if constexpr (ERASE == kEraseNone) s[0] += __shfl_xor_sync(kFull, s[0], 16);
            const int jl = 4 * (lane & 1) + ((lane & 8) ? 8 : 0) + ((lane & 4) ? 2 : 0) + ((lane & 2) ? 1 : 0);
            const int jc = 16 * warp + jl;   // the lane's column within the CTA's
            const float vj = S.v[t][jc];
            // u = w o v - p (w = beta 1, p = beta k^T S' for the delta rule; a = 0, w = 1 without)
            float u = vj;
            if constexpr (ERASE == kEraseDelta) u = __fmul_rn(S.beta[t], __fsub_rn(vj, s[0]));
            if constexpr (ERASE == kEraseGeneral) u = __fsub_rn(__fmul_rn(S.w[t][jc], vj), s[0]);
            if constexpr (ERASE != kEraseNone) {
                const float other = __shfl_xor_sync(kFull, u, 16);
                u = lane < 16 ? u : other;   // lanes below 16 hold p, the others r
            }
            if (lane < 16) sm.u[warp][jl] = u;
            __syncwarp();
            if (lane >= 16)   // o = S^T q = r + u (k . q)
                p.o[((static_cast<size_t>(b) * p.T + t0 + t) * p.H + h) * dv + c0 + jc] = fmaf(u, kq, s[0]);
            const float4 ua = *reinterpret_cast<const float4*>(&sm.u[warp][4 * (lane & 1)]);
            const float4 ub = *reinterpret_cast<const float4*>(&sm.u[warp][4 * (lane & 1) + 8]);
            const float us[8] = {ua.x, ua.y, ua.z, ua.w, ub.x, ub.y, ub.z, ub.w};
#pragma unroll
            for (int m = 0; m < RL / 2; m += 2) {
                const float4 k4 = *reinterpret_cast<const float4*>(&S.k[t][i0 + 32 * m]);
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    x[m][c] = __ffma2_rn(make_float2(k4.x, k4.y), make_float2(us[c], us[c]), x[m][c]);
                    x[m + 1][c] = __ffma2_rn(make_float2(k4.z, k4.w), make_float2(us[c], us[c]), x[m + 1][c]);
                }
            }
            __syncwarp();   // u is read before the next token's
        }
    }

    float* dst = p.dense_out + (static_cast<size_t>(bh) * DK + i0) * dv + j0;
#pragma unroll
    for (int r = 0; r < RL; ++r) {
        float t[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) t[c] = r & 1 ? x[r / 2][c].y : x[r / 2][c].x;
        if (vec & 2) {
            *reinterpret_cast<float4*>(dst + row(r) * dv) = make_float4(t[0], t[1], t[2], t[3]);
            *reinterpret_cast<float4*>(dst + row(r) * dv + 8) = make_float4(t[4], t[5], t[6], t[7]);
        } else {
#pragma unroll
            for (int c = 0; c < 8; ++c) dst[row(r) * dv + (c & 3) + 2 * (c & 4)] = t[c];
        }
    }
}

// ---- a call of few tokens ----------------------------------------------------------------------
// Such a call is its state's way through memory.  Same CTAs (64 columns of a head, 4 warps), but half a
// warp holds 256 bytes of a row and a warp's rows lie beside each other, so that a 16-byte access of the warp
// takes 4 lines of the L1 (16 in the kernel above); the price is an exchange between the warps
// for each token's sums, three barriers per token.  16 x 32 heads of 128 x 128, one token: 13.6 us from HBM
// (67 MB, 4.9 TB/s) and 9.0 us from L2; the kernel above 16.6 and 14.1, one CTA of 8 warps to a head 16.4 and 11.4.
// Two tokens 15.7 and 11.1 (16.9 and 14.7), three 17.2 and 12.9 (17.5 and 15.6), four 19.0 and 14.8 (18.9 and 17.1);
// 64 x 32 heads, two 53 and 53 (52 and 52), three 58 and 57: hence up to two.  The readouts' error against
// 64 bits is the kernel above's (8.9e-8 and 8.8e-8 for one token, 9.5e-8 both for two).
constexpr int kShortTokens = 2;

template <int DK, int ERASE>
__global__ void __launch_bounds__(kFpThreads, 4) scan_fp32_short_kernel(const __grid_constant__ StepParams p, int dv) {
    constexpr int RT = DK / 8;   // rows per thread: 8 r + rg
    __shared__ float4 dakq[DK];  // decay, a (delta rule: k), k, q of the token's rows
    __shared__ __align__(16) float red[2][4][kCols], us[kCols];
    __shared__ float wsum[DK / 32];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, rg = tid >> 4, cl = (tid & 15) * 4;
    const int parts = dv / kCols;
    const int bh = blockIdx.x / parts, c0 = (blockIdx.x - bh * parts) * kCols;
    const int b = bh / p.H, h = bh - b * p.H;
    const size_t at = (static_cast<size_t>(bh) * DK + rg) * dv + c0 + cl;   // + 8 r dv
    float2 x[RT][2];
#pragma unroll
    for (int r = 0; r < RT; ++r) {
        const float4 v = *reinterpret_cast<const float4*>(p.dense_in + at + static_cast<size_t>(8 * r) * dv);
        x[r][0] = make_float2(v.x, v.y);
        x[r][1] = make_float2(v.z, v.w);
    }
#pragma unroll 1
    for (int t = p.t_begin; t < p.t_end; ++t) {
        const size_t tok = (static_cast<size_t>(b) * p.T + t) * p.H + h;
        if (t > p.t_begin) __syncthreads();   // the token before is done with its rows and u
        float vj = 0.0f, wj = 1.0f;
        if (tid < kCols) {
            vj = p.v[tok * dv + c0 + tid];
            if constexpr (ERASE == kEraseDelta) wj = p.beta[tok];
            if constexpr (ERASE == kEraseGeneral) wj = p.w_in[tok * dv + c0 + tid];
        }
        if (tid < DK) {
            const float k = p.k[tok * DK + tid], q = p.q[tok * DK + tid];
            float a = k, rate;
            if constexpr (ERASE == kEraseGeneral) a = p.a_in[tok * DK + tid];
            if (p.s_code) {
                const size_t ch = p.decay_row ? static_cast<size_t>(h) * DK + tid : h;
                rate = p.s_lut[ch * p.L + min(static_cast<int>(p.s_code[p.decay_row ? tok * DK + tid : tok]), p.L - 1)];
            } else {
                rate = p.s[p.decay_row ? tok * DK + tid : tok];
            }
            if (!(rate > 0.0f) || !(rate < INFINITY)) raise_status(p.status, QS_DEV_RATE);
            dakq[tid] = make_float4(expf(-rate), a, k, q);
            const float kq = warp_sum(k * q);
            if (lane == 0) wsum[warp] = kq;
        }
        __syncthreads();
        // (four runs of RT / 4 rows summed by halves, so that the sums round no worse than the kernel above's)
        float2 pp[2], rr[2];
        auto run = [&](int r0, float2 (&ps)[2], float2 (&rs)[2]) {
#pragma unroll
            for (int i = 0; i < RT / 4; ++i) {
                const int r = r0 + i;
                const float4 f = dakq[8 * r + rg];
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    x[r][c] = __fmul2_rn(x[r][c], make_float2(f.x, f.x));
                    if constexpr (ERASE != kEraseNone)
                        ps[c] = i == 0 ? __fmul2_rn(x[r][c], make_float2(f.y, f.y)) : __ffma2_rn(x[r][c], make_float2(f.y, f.y), ps[c]);
                    rs[c] = i == 0 ? __fmul2_rn(x[r][c], make_float2(f.w, f.w)) : __ffma2_rn(x[r][c], make_float2(f.w, f.w), rs[c]);
                }
            }
        };
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            float2 p0[2], r0[2], p1[2], r1[2];
            run(half * (RT / 2), p0, r0);
            run(half * (RT / 2) + RT / 4, p1, r1);
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                if constexpr (ERASE != kEraseNone) {
                    p0[c] = __fadd2_rn(p0[c], p1[c]);
                    pp[c] = half == 0 ? p0[c] : __fadd2_rn(pp[c], p0[c]);
                }
                r0[c] = __fadd2_rn(r0[c], r1[c]);
                rr[c] = half == 0 ? r0[c] : __fadd2_rn(rr[c], r0[c]);
            }
        }
        // the warp's two halves, then the four warps
        auto both = [&](float2 v) {
            return make_float2(v.x + __shfl_xor_sync(kFull, v.x, 16), v.y + __shfl_xor_sync(kFull, v.y, 16));
        };
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            if constexpr (ERASE != kEraseNone) pp[c] = both(pp[c]);
            rr[c] = both(rr[c]);
        }
        if (lane < 16) {
            if constexpr (ERASE != kEraseNone)
                *reinterpret_cast<float4*>(&red[0][warp][cl]) = make_float4(pp[0].x, pp[0].y, pp[1].x, pp[1].y);
            *reinterpret_cast<float4*>(&red[1][warp][cl]) = make_float4(rr[0].x, rr[0].y, rr[1].x, rr[1].y);
        }
        __syncthreads();
        if (tid < kCols) {
            float P = 0.0f;
            if constexpr (ERASE != kEraseNone) P = (red[0][0][tid] + red[0][1][tid]) + (red[0][2][tid] + red[0][3][tid]);
            const float R = (red[1][0][tid] + red[1][1][tid]) + (red[1][2][tid] + red[1][3][tid]);
            float kq = wsum[0] + wsum[1];
            if constexpr (DK == 128) kq += wsum[2] + wsum[3];
            // as above: u = beta (v - p), w o v - p, or v
            float u = vj;
            if constexpr (ERASE == kEraseDelta) u = __fmul_rn(wj, __fsub_rn(vj, P));
            if constexpr (ERASE == kEraseGeneral) u = __fsub_rn(__fmul_rn(wj, vj), P);
            us[tid] = u;
            p.o[tok * dv + c0 + tid] = fmaf(u, kq, R);
        }
        __syncthreads();
        const float4 u = *reinterpret_cast<const float4*>(&us[cl]);
#pragma unroll
        for (int r = 0; r < RT; ++r) {
            const float k = dakq[8 * r + rg].z;
            x[r][0] = __ffma2_rn(make_float2(k, k), make_float2(u.x, u.y), x[r][0]);
            x[r][1] = __ffma2_rn(make_float2(k, k), make_float2(u.z, u.w), x[r][1]);
        }
    }
#pragma unroll
    for (int r = 0; r < RT; ++r)
        *reinterpret_cast<float4*>(p.dense_out + at + static_cast<size_t>(8 * r) * dv) =
            make_float4(x[r][0].x, x[r][0].y, x[r][1].x, x[r][1].y);
}

template <int DK, int ERASE>
cudaError_t launch_fp32_t(const StepParams& p, int dv, int vec, cudaStream_t stream) {
    if (p.t_end - p.t_begin <= kShortTokens && (vec & 2)) {
        scan_fp32_short_kernel<DK, ERASE><<<p.B * p.H * (dv / kCols), kFpThreads, 0, stream>>>(p, dv);
        return cudaGetLastError();
    }
    const int smem = static_cast<int>(sizeof(FpSmem<DK, ERASE>));
    cudaError_t e = cudaFuncSetAttribute(scan_fp32_kernel<DK, ERASE>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    scan_fp32_kernel<DK, ERASE><<<p.B * p.H * (dv / kCols), kFpThreads, smem, stream>>>(p, dv, vec);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_scan_fp32(int dk, int dv, const StepParams& p, cudaStream_t stream) {
    auto aligned = [](const void* q) { return (reinterpret_cast<uintptr_t>(q) & 15) == 0; };
    const bool inputs = aligned(p.k) && aligned(p.q) && aligned(p.v) && aligned(p.s) && (!p.general || (aligned(p.a_in) && aligned(p.w_in)));
    const int vec = (inputs ? 1 : 0) | (aligned(p.dense_in) ? 2 : 0);
    const int erase = p.general ? kEraseGeneral : p.erase ? kEraseDelta : kEraseNone;
    if (dk == 128)
        return erase == kEraseGeneral ? launch_fp32_t<128, kEraseGeneral>(p, dv, vec, stream)
               : erase == kEraseDelta ? launch_fp32_t<128, kEraseDelta>(p, dv, vec, stream)
                                      : launch_fp32_t<128, kEraseNone>(p, dv, vec, stream);
    return erase == kEraseGeneral ? launch_fp32_t<64, kEraseGeneral>(p, dv, vec, stream)
           : erase == kEraseDelta ? launch_fp32_t<64, kEraseDelta>(p, dv, vec, stream)
                                  : launch_fp32_t<64, kEraseNone>(p, dv, vec, stream);
}

}  // namespace qs

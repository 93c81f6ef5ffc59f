// qs_alloc.cu -- bit allocation (Sec. 3 "State bit allocation": Eq. 3, Eq. 4 and the integer
// rounding to the layer budget), one CTA per batch element.
//
// Weights c_i = Gamma_hat_i Rtilde_i^2 are formed in FP32 with one IEEE rounding per operation
// (Gamma_hat = (1 - m_s) / (expm1(m_r) + m_s), expm1 from its Taylor series), so they are
// reproducible bit for bit.  Rounding Eq. (4) to nearest, clipping and adjusting to the budget
// by the rounding remainders hands out bits in decreasing order of their marginal value
// c_i 4^{-b}: the result is the set of the M = total - N b_min most valuable bits (i, b),
// b in (b_min, b_max].  For FP32 c the order of c 4^{-b} is the order of the integer key
// bits(c) - b 2^24 (a power-of-4 scaling moves only the exponent field), so the kernel finds
// the M-th largest key from integer counts -- no logarithm, no floating-point
// comparison -- and gives bits tied at the threshold to the lowest unit indices.  The M-th
// largest key is found from a histogram of the keys' high parts, a second one of the leading
// 7 of their low 24 bits, and a count of the few keys (about 32 of 4096 units) left in that bin.
//
// What bounds it: one CTA's latency.  The data (13 bytes per unit) is nothing; the launch is a
// chain of short phases between CTA barriers, each instruction of which runs once per launch, so
// that its fetch costs more than its execution.  So a thread keeps its UPT consecutive units in
// registers from the statistics (one 16-byte load per array) to the widths, what few calls need
// stays out of the straight line (other_weight), and each phase is as few instructions as it
// can be.  Per launch, back to back, against the kernel it replaces (1024 threads for any size,
// statistics and keys in shared memory, 16-term series, a radix select of 8-bit digits):
//     units   64 (1 head 64 x 64)        7.1 -> 2.6 us
//     units   16 (16 heads, head unit)   6.3 -> 2.8 us
//     units 2048                         9.7 -> 4.4 us
//     units 4096                        12.4 -> 6.1 us
//     units 8192, groups of 1024        23.4 -> 11.9 us (the row-order sum of a group: 1024
//                                       dependent additions)
//     units 16384                       38.0 -> 19.9 us
#include "qs_common.cuh"

namespace qs {

namespace {

constexpr int kThreads = 1024;               // at most
constexpr int kListMax = 128;                // keys ranked directly, one thread each (= kBins)
constexpr int kGroupPad = 4;                 // floats between two groups' R^2 in shared memory
// Keys: the bits of a weight in [2^-60, 2^60], so E = key >> 24 is in 33..93 and the high parts of
// its keys in 17..92; a null weight's keys lie below all of them; a thread without a unit
// reaches no high part.  128 bins hold them all.
constexpr int kNullKey = 16 << 24;
constexpr int kNoKey = 0;
constexpr int kBins = 128, kBPL = kBins / 32;

// expm1 by its Taylor series (degree 16, Horner), the argument halved while above 1 (an infinite one
// cannot be halved; its series is infinite as it is).
__device__ __noinline__ float expm1_series(float x, const AllocParams& p) {
    if (!(x > 0.0f)) return 0.0f;
    int halvings = 0;
    while (x > 1.0f && x < INFINITY) {
        x = __fmul_rn(x, 0.5f);
        ++halvings;
    }
    float t = p.e1[16];
#pragma unroll 1
    for (int k = 15; k >= 1; --k) t = __fadd_rn(__fmul_rn(t, x), p.e1[k]);
    float y = __fmul_rn(t, x);
    for (int i = 0; i < halvings; ++i) y = __fmul_rn(y, __fadd_rn(y, 2.0f));
    return y;
}

// The same on (0, 2^-3): the terms above x^9 change no bit of the result there (checked for every
// float of that range; each later rounding absorbs them.  From 2^-3 up a few arguments do differ).
// The erasure statistic of a unit key averages about 0.7/dk, so nearly all units come this way.
constexpr float kShortSeries = 0.125f;
__device__ __forceinline__ float expm1_short(float x, const float* e1) {
    float p = e1[9];
#pragma unroll
    for (int k = 8; k >= 1; --k) p = __fadd_rn(__fmul_rn(p, x), e1[k]);
    return __fmul_rn(p, x);
}

}  // namespace

// The part of an allocation weight that does not depend on ranges, one IEEE rounding per
// operation: Gamma_hat of Eq. 3 outside the range of the short series, and the alternatives of
// Table 1.
__device__ __noinline__ float other_weight(int kind, float ms, float mr, const AllocParams& p) {
    if (kind == QSTATE_WEIGHT_PERSIST) return __fdiv_rn(1.0f, ms);
    if (kind == QSTATE_WEIGHT_WBFACTOR) {
        float pw = 1.0f, bb = __fsub_rn(1.0f, ms);   // (1 - m_s)^C, low bit first
#pragma unroll 1
        for (int e = p.C; e > 0; e >>= 1) {
            if (e & 1) pw = __fmul_rn(pw, bb);
            bb = __fmul_rn(bb, bb);
        }
        return __fdiv_rn(1.0f, __fsub_rn(1.0f, pw));
    }
    if (mr < 0.0f) mr = 0.0f;
    return __fdiv_rn(__fsub_rn(1.0f, ms), __fadd_rn(expm1_series(mr, p), ms));
}

// Inclusive prefix sum over the warp.
__device__ __forceinline__ int warp_prefix(int v, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int n = __shfl_up_sync(kFull, v, o);
        if (lane >= o) v += n;
    }
    return v;
}

// One warp: the bin of kBins whose suffix count (bins >= it, highest first) first reaches `rank`
// (1-based), *above the count of the bins above it and *left its own.  c: the counts of bins
// kBins - 1 - kBPL lane, then one lower each.
__device__ __forceinline__ int warp_select(const int (&c)[kBPL], int rank, int lane, int* above, int* left) {
    int run[kBPL], s = 0;
#pragma unroll
    for (int k = 0; k < kBPL; ++k) run[k] = s += c[k];
    const int excl = warp_prefix(s, lane) - s;
    const int want = rank - excl;   // the lane with 0 < want <= s holds the bin
    int k0 = 0, own = c[0], up = 0;
#pragma unroll
    for (int k = 1; k < kBPL; ++k)
        if (run[k - 1] < want) {
            k0 = k;
            own = c[k];
            up = run[k - 1];
        }
    const int src = __ffs(__ballot_sync(kFull, want >= 1 && want <= s)) - 1;
    *above = __shfl_sync(kFull, excl + up, src);
    *left = __shfl_sync(kFull, own, src);
    return kBins - 1 - kBPL * src - __shfl_sync(kFull, k0, src);
}

// Shared memory after the R^2 and the group means:
struct AllocTail {
    int hist[kBins];
    alignas(16) int list[kListMax];       // unused places hold -1
    int hbytes[1024];                     // payload bytes per head
    int hs, rank, low, left, cnt, ties;   // selection (see below)
    int wties[kThreads / 32];             // tied units per warp
    int wsum[kThreads / 32];              // sum of widths, then of payload bytes, per warp
};

// UPT consecutive units per thread.  PLAIN: the weights are Eq. 3's (weight_kind OURS) and, for
// UPT > 1, the arrays aligned for 16-byte loads (p.vec); otherwise any weight and alignment.
template <int UPT, bool PLAIN>
__global__ void __launch_bounds__(kThreads, 1) alloc_kernel(const __grid_constant__ AllocParams p) {
    extern __shared__ __align__(16) uint8_t smem[];
    const int N = p.units, NT = blockDim.x;
    const int gsz = p.group_heads * p.dk;
    const int ngroups = p.ngroups;
    float* R2s = reinterpret_cast<float*>(smem);
    float* gmean = R2s + (p.unit_row ? N + ngroups * kGroupPad : 0);
    AllocTail& sm = *reinterpret_cast<AllocTail*>(gmean + ((ngroups + 3) & ~3));
    const size_t base = static_cast<size_t>(blockIdx.x) * N;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, u0 = tid * UPT;
    const int J = p.bmax - p.bmin, M = p.above_min;
    int w[UPT];
    chain_wait();

    if (p.uniform || M == 0) {
        // equal weights: M / N bits for every unit, and the rest to the lowest indices
        const int each = p.bmin + M / N, extra = M % N;
#pragma unroll
        for (int k = 0; k < UPT; ++k) w[k] = each + (u0 + k < extra ? 1 : 0);
    } else {
        const int kind = PLAIN ? static_cast<int>(QSTATE_WEIGHT_OURS) : p.weight_kind;
        // 1. statistics (from L2: the write-back has just written them); R^2 to shared memory, its
        //    groups kGroupPad words apart so that the lanes that sum different groups in lockstep
        //    hit different banks
        float R[UPT], ms[UPT], mr[UPT];
        const bool some = u0 < N;
        if (UPT > 1 && (PLAIN || (p.vec && kind != QSTATE_WEIGHT_SHUFFLE))) {
            if constexpr (UPT > 1) {
#pragma unroll
                for (int k = 0; k < UPT; k += 4) {
                    float4 t = make_float4(0.0f, 0.0f, 0.0f, 0.0f), a = t, b = t;
                    if (some) {
                        t = *reinterpret_cast<const float4*>(p.range + base + u0 + k);
                        a = *reinterpret_cast<const float4*>(p.ema_s + base + u0 + k);
                        if (PLAIN || kind != QSTATE_WEIGHT_NOERASE)
                            b = *reinterpret_cast<const float4*>(p.ema_r + base + u0 + k);
                    }
                    R[k] = t.x; R[k + 1] = t.y; R[k + 2] = t.z; R[k + 3] = t.w;
                    ms[k] = a.x; ms[k + 1] = a.y; ms[k + 2] = a.z; ms[k + 3] = a.w;
                    mr[k] = b.x; mr[k + 1] = b.y; mr[k + 2] = b.z; mr[k + 3] = b.w;
                }
            }
        } else {
            // SHUFFLE: the statistics of unit pi(u) (below 2^28 + 2^14: 32 bits)
            int pi = !PLAIN && kind == QSTATE_WEIGHT_SHUFFLE ? (p.shuf_a * u0 + p.shuf_b) % N : 0;
#pragma unroll
            for (int k = 0; k < UPT; ++k) {
                const int u = u0 + k;
                R[k] = mr[k] = 0.0f;
                ms[k] = 1.0f;
                if (u < N) {
                    int us = u;
                    if (!PLAIN && kind == QSTATE_WEIGHT_SHUFFLE) {
                        us = pi;
                        pi += p.shuf_a;
                        if (pi >= N) pi -= N;
                    }
                    if (p.unit_row) R[k] = p.range[base + u];
                    ms[k] = p.ema_s[base + us];
                    if (PLAIN || kind != QSTATE_WEIGHT_NOERASE) mr[k] = p.ema_r[base + us];
                }
            }
        }
        for (int k = tid; k < kBins; k += NT) {
            sm.hist[k] = 0;
            sm.list[k] = -1;
        }
        if (tid == 0) sm.cnt = 0;
        int gi = 0;   // the thread's group (UPT divides dk)
        float* r2 = nullptr;
        if (p.unit_row) {
            gi = p.gshift >= 0 ? u0 >> p.gshift : u0 / gsz;
            r2 = R2s + u0 + gi * kGroupPad;
#pragma unroll
            for (int k = 0; k < UPT; ++k) R[k] = __fmul_rn(R[k], R[k]);
            if (some) {
                if constexpr (UPT > 1) {
#pragma unroll
                    for (int k = 0; k < UPT; k += 4)
                        *reinterpret_cast<float4*>(r2 + k) = make_float4(R[k], R[k + 1], R[k + 2], R[k + 3]);
                } else {
                    *r2 = R[0];
                }
            }
            __syncthreads();
            // 2. mean R^2 of each output-normalisation group, summed in row order by one thread: a
            //    chain of gsz dependent additions, its operands loaded ahead 16 bytes at a time
            //    (gsz is a multiple of 64), beside the weights' decay parts in the other warps
            if (tid < ngroups) {
                const float4* rg = reinterpret_cast<const float4*>(R2s + tid * (gsz + kGroupPad));
                float acc = 0.0f;
                auto add4 = [&](const float4& v) {
                    acc = __fadd_rn(acc, v.x);
                    acc = __fadd_rn(acc, v.y);
                    acc = __fadd_rn(acc, v.z);
                    acc = __fadd_rn(acc, v.w);
                };
                float4 a0 = rg[0], a1 = rg[1], a2 = rg[2], a3 = rg[3];
#pragma unroll 1
                for (int r = 0; r < gsz / 4; r += 8) {
                    const float4 b0 = rg[r + 4], b1 = rg[r + 5], b2 = rg[r + 6], b3 = rg[r + 7];
                    add4(a0); add4(a1); add4(a2); add4(a3);
                    const int nr = r + 8 < gsz / 4 ? r + 8 : 0;
                    a0 = rg[nr]; a1 = rg[nr + 1]; a2 = rg[nr + 2]; a3 = rg[nr + 3];
                    add4(b0); add4(b1); add4(b2); add4(b3);
                }
                gmean[tid] = __fdiv_rn(acc, static_cast<float>(gsz));
            }
        }
        float c[UPT];
        // Gamma_hat (Eq. 3), for the weights that have it
        if (PLAIN || kind == QSTATE_WEIGHT_OURS || kind == QSTATE_WEIGHT_GAMMA_RAW || kind == QSTATE_WEIGHT_NOERASE ||
            kind == QSTATE_WEIGHT_SHUFFLE) {
            bool rare = false;
#pragma unroll
            for (int k = 0; k < UPT; ++k) rare |= !(mr[k] < kShortSeries) || mr[k] < 0.0f;
            // (-0 and 0 give expm1 = +-0, which adds nothing to m_s)
#pragma unroll
            for (int k = 0; k < UPT; ++k)
                c[k] = __fdiv_rn(__fsub_rn(1.0f, ms[k]), __fadd_rn(expm1_short(mr[k], p.e1), ms[k]));
            if (rare) {
#pragma unroll
                for (int k = 0; k < UPT; ++k)
                    if (!(mr[k] < kShortSeries) || mr[k] < 0.0f) c[k] = other_weight(kind, ms[k], mr[k], p);
            }
        } else {
            const bool flat = kind == QSTATE_WEIGHT_RANGE || kind == QSTATE_WEIGHT_NRANGE;
#pragma unroll
            for (int k = 0; k < UPT; ++k) c[k] = flat ? 1.0f : other_weight(kind, ms[k], mr[k], p);
        }
        if (p.unit_row) {
            __syncthreads();
            // times R^2 over its group's mean (or R^2, or that factor alone)
            const float m = some ? gmean[gi] : 0.0f;
            const bool raw = !PLAIN && (kind == QSTATE_WEIGHT_RANGE || kind == QSTATE_WEIGHT_GAMMA_RAW);
            const bool alone = !PLAIN && (kind == QSTATE_WEIGHT_RANGE || kind == QSTATE_WEIGHT_NRANGE);
#pragma unroll
            for (int k = 0; k < UPT; ++k) {
                const float f = raw ? R[k] : m > 0.0f ? __fdiv_rn(R[k], m) : 1.0f;
                c[k] = alone ? f : __fmul_rn(c[k], f);
            }
        } else {
            __syncthreads();   // the histogram is zero
        }

        // 3. integer keys; those of unit u's bits b_min + j (j = 1..J) are key_u - j 2^24, i.e.
        //    high part E - j and low part L with E = key_u >> 24, L = key_u & 0xFFFFFF.  Histogram
        //    of E (lanes with equal E add together).  A unit beyond N reaches no bin.
        int key[UPT];
#pragma unroll
        for (int k = 0; k < UPT; ++k) {
            const float cc = c[k] > 0x1p60f ? 0x1p60f : c[k];
            key[k] = cc >= 0x1p-60f ? __float_as_int(cc) : kNullKey;
            if (u0 + k >= N) key[k] = kNoKey;
            const int E = key[k] >> 24;
            const unsigned peers = __match_any_sync(kFull, E);
            if ((peers & ((1u << lane) - 1u)) == 0) atomicAdd(&sm.hist[E], __popc(peers));
        }
        __syncthreads();

        // 4. V = the M-th largest key: its high part.  The keys with high part h number
        //    #{E > h} - #{E > h + J}; with the counts of E by lane in descending order, both
        //    suffix counts come from one prefix sum over the warp, kept in shared memory.
        if (warp == 0) {
            const int top = kBins - 1 - kBPL * lane;
            int c[kBPL], s = 0;
#pragma unroll
            for (int k = 0; k < kBPL; ++k) {
                c[k] = s;   // of the lane's bins above this one
                s += sm.hist[top - k];
            }
            const int excl = warp_prefix(s, lane) - s;
            __syncwarp();
#pragma unroll
            for (int k = 0; k < kBPL; ++k) sm.hist[top - k] = c[k] = excl + c[k];   // #{E > h}
            __syncwarp();
#pragma unroll
            for (int k = 0; k < kBPL; ++k) c[k] -= top - k + J < kBins ? sm.hist[top - k + J] : 0;
            int above, left;
            const int h = warp_select(c, M, lane, &above, &left);
            __syncwarp();
#pragma unroll
            for (int k = 0; k < kBPL; ++k) sm.hist[top - k] = 0;
            if (lane == 0) {
                sm.hs = h;             // high part of V
                sm.rank = M - above;   // rank of V among the keys with that high part
            }
        }
        __syncthreads();
        const int Hs = sm.hs;
        // its low 24 bits, among the units whose keys reach high part Hs: the leading 7 from a
        // histogram, the others by ranking the keys of that bin directly when they are few
        // (else by histograms of the next 7, 7 and 3: many equal weights)
        int pre = 0, ties = 0, need = 0;
#pragma unroll 1
        for (int known = 24, sh = 17;; known = sh, sh = max(sh - 7, 0)) {
#pragma unroll
            for (int k = 0; k < UPT; ++k) {
                const int d = (key[k] >> 24) - Hs, L = key[k] & 0xFFFFFF;
                if (d >= 1 && d <= J && ((L ^ pre) >> known) == 0) atomicAdd(&sm.hist[(L >> sh) & ((1 << (known - sh)) - 1)], 1);
            }
            __syncthreads();
            if (warp == 0) {
                const int top = kBins - 1 - kBPL * lane;
                int c[kBPL], above, left;
#pragma unroll
                for (int k = 0; k < kBPL; ++k) c[k] = sm.hist[top - k];
                const int bin = warp_select(c, sm.rank, lane, &above, &left);
                __syncwarp();
#pragma unroll
                for (int k = 0; k < kBPL; ++k) sm.hist[top - k] = 0;
                if (lane == 0) {
                    sm.rank -= above;
                    sm.low = pre | (bin << sh);
                    sm.left = left;
                }
            }
            __syncthreads();
            pre = sm.low;
            ties = sm.left;
            need = sm.rank;
            if (sh == 0) break;   // `ties` equal keys are left, `need` of which get a bit
            if (ties <= kListMax) {
#pragma unroll
                for (int k = 0; k < UPT; ++k) {
                    const int d = (key[k] >> 24) - Hs, L = key[k] & 0xFFFFFF;
                    if (d >= 1 && d <= J && ((L ^ pre) >> sh) == 0) sm.list[atomicAdd(&sm.cnt, 1)] = L;
                }
                __syncthreads();
#pragma unroll 1
                for (int i = tid; i < ties; i += NT) {
                    const int mine = sm.list[i];
                    int gt = 0, eq = 0;
#pragma unroll 2
                    for (int j = 0; j < ties; j += 4) {
                        const int4 o = *reinterpret_cast<const int4*>(sm.list + j);
                        gt += (o.x > mine ? 1 : 0) + (o.y > mine ? 1 : 0) + (o.z > mine ? 1 : 0) + (o.w > mine ? 1 : 0);
                        eq += (o.x == mine ? 1 : 0) + (o.y == mine ? 1 : 0) + (o.z == mine ? 1 : 0) + (o.w == mine ? 1 : 0);
                    }
                    if (gt < need && need <= gt + eq) {   // equal keys write the same values
                        sm.low = mine;
                        sm.left = need - gt;
                        sm.ties = eq;
                    }
                }
                __syncthreads();
                pre = sm.low;
                need = sm.left;
                ties = sm.ties;
                break;
            }
        }
        if (tid == 0 && (need < 1 || need > ties)) raise_status(p.status, QS_DEV_LAYOUT);

        // 5. widths: bits strictly above V, plus tied bits to the lowest unit indices
        int before = 0;   // tied units below the thread's
        if (need < ties) {
            int mine = 0;
#pragma unroll
            for (int k = 0; k < UPT; ++k) {
                const int d = (key[k] >> 24) - Hs;
                mine += d >= 1 && d <= J && (key[k] & 0xFFFFFF) == pre ? 1 : 0;
            }
            const int incl = warp_prefix(mine, lane);
            if (lane == 31) sm.wties[warp] = incl;
            __syncthreads();
            before = incl - mine;
            for (int i = 0; i < warp; ++i) before += sm.wties[i];
        }
#pragma unroll
        for (int k = 0; k < UPT; ++k) {
            const int d = (key[k] >> 24) - Hs, L = key[k] & 0xFFFFFF;
            w[k] = p.bmin + min(max(d - (L > pre ? 0 : 1), 0), J);
            if (d >= 1 && d <= J && L == pre) {
                w[k] += before < need ? 1 : 0;
                ++before;
            }
        }
    }

    // 6. widths out; head offsets: exclusive prefix sum of the heads' payload bytes (row unit: the
    //    dk / UPT consecutive lanes of a head sum its widths)
    if (UPT > 1 && (PLAIN || p.vec)) {
        if constexpr (UPT > 1) {
            if (u0 < N)
#pragma unroll
                for (int k = 0; k < UPT; k += 4)
                    *reinterpret_cast<uint32_t*>(p.widths + base + u0 + k) =
                        static_cast<uint32_t>(w[k] | (w[k + 1] << 8) | (w[k + 2] << 16) | (w[k + 3] << 24));
        }
    } else {
#pragma unroll
        for (int k = 0; k < UPT; ++k)
            if (u0 + k < N) p.widths[base + u0 + k] = static_cast<uint8_t>(w[k]);
    }
    if (p.unit_row) {
        int sum = 0;
#pragma unroll
        for (int k = 0; k < UPT; ++k) sum += w[k];
        if constexpr (UPT == 1) {   // a head spans dk / 32 warps
            sum = __reduce_add_sync(kFull, sum);
            if (lane == 0) sm.wsum[warp] = sum;
            __syncthreads();
            const int wph = p.dk / 32;
            if (tid < p.H) {
                sum = 0;
                for (int i = 0; i < wph; ++i) sum += sm.wsum[tid * wph + i];
                sm.hbytes[tid] = sum * (p.dv / 8);
            }
        } else {
            const int lanes = p.dk / UPT;   // a power of two, at most 32
            for (int o = lanes >> 1; o > 0; o >>= 1) sum += __shfl_xor_sync(kFull, sum, o);
            if (u0 < N && (tid & (lanes - 1)) == 0) sm.hbytes[u0 >> (p.dk == 128 ? 7 : 6)] = sum * (p.dv / 8);
        }
    } else {
#pragma unroll
        for (int k = 0; k < UPT; ++k)
            if (u0 + k < N) sm.hbytes[u0 + k] = w[k] * p.dk * p.dv / 8;
    }
    __syncthreads();
    // 32 heads at a time by one warp, or, of many, 32 by each warp (1024 heads, head unit: 7.1 us a
    // launch by one warp, 3.6; 256: 3.7 and 2.9; 65: 3.0 and 2.8)
    if (p.H <= 64) {
        if (warp != 0) return;
        int carry = 0;
#pragma unroll 1
        for (int h0 = 0; h0 < p.H; h0 += 32) {
            const int h = h0 + lane;
            const int v = h < p.H ? sm.hbytes[h] : 0;
            const int incl = warp_prefix(v, lane);
            if (h < p.H)
                p.head_off[static_cast<size_t>(blockIdx.x) * p.H + h] = static_cast<uint32_t>(carry + incl - v);
            carry += __shfl_sync(kFull, incl, 31);
        }
    } else {
        const int v = tid < p.H ? sm.hbytes[tid] : 0;
        const int incl = warp_prefix(v, lane);
        if (lane == 31) sm.wsum[warp] = incl;
        __syncthreads();
        const int carry = __reduce_add_sync(kFull, lane < warp ? sm.wsum[lane] : 0);
        if (tid < p.H) p.head_off[static_cast<size_t>(blockIdx.x) * p.H + tid] = static_cast<uint32_t>(carry + incl - v);
    }
}

template <int UPT, bool PLAIN>
static cudaError_t launch_alloc_t(const AllocParams& p, cudaStream_t stream) {
    const size_t smem = static_cast<size_t>(p.unit_row ? p.units + p.ngroups * kGroupPad : 0) * 4 +
                        static_cast<size_t>((p.ngroups + 3) & ~3) * 4 + sizeof(AllocTail);
    const int threads = ((p.units + UPT - 1) / UPT + 31) & ~31;
    cudaError_t e = cudaFuncSetAttribute(alloc_kernel<UPT, PLAIN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(smem));
    if (e != cudaSuccess) return e;
    return launch_chained(alloc_kernel<UPT, PLAIN>, p.B, threads, smem, stream, p.early != 0, p);
}

cudaError_t launch_alloc(const AllocParams& p_in, cudaStream_t stream) {
    AllocParams p = p_in;
    const int gsz = p.group_heads * p.dk;
    p.ngroups = p.unit_row ? p.units / gsz : 0;
    p.gshift = -1;
    if ((gsz & (gsz - 1)) == 0)
        for (p.gshift = 0; (1 << p.gshift) < gsz;) ++p.gshift;
    p.above_min = static_cast<int>(p.total - static_cast<long long>(p.units) * p.bmin);   // <= 16384 * 16
    auto aligned = [](const void* q, uintptr_t n) { return (reinterpret_cast<uintptr_t>(q) & (n - 1)) == 0; };
    const bool ours = p.uniform || p.weight_kind == QSTATE_WEIGHT_OURS;
    // row unit: N is a multiple of 64, so every batch element is aligned as the arrays are
    p.vec = p.unit_row && aligned(p.widths, 4) &&
                    (p.uniform || (aligned(p.ema_s, 16) && aligned(p.ema_r, 16) && aligned(p.range, 16)))
                ? 1 : 0;
    if (p.units <= 1024) return ours ? launch_alloc_t<1, true>(p, stream) : launch_alloc_t<1, false>(p, stream);
    // Other weights and alignments: 8 units per thread up to 8192 units as below.  One batch element, range
    // weights: 8192 units 9.9 us, 16384 19.5 us (38 and 66 us with 16 units per thread at 8192, the
    // decay part evaluated for every weight kind by the full series, and 4-byte loads); shuffled decay weights
    // 13.9 and 34.9 us (38.8 and 70); statistics off 16 bytes 13.9 and 35 us (20.1 and 36).
    if (!ours || !p.vec)
        return p.units <= 4096   ? launch_alloc_t<4, false>(p, stream)
               : p.units <= 8192 ? launch_alloc_t<8, false>(p, stream)
                                 : launch_alloc_t<16, false>(p, stream);
    // Units per thread: as few as 1024 threads allow, for the latency of a launch with few batch
    // elements (4096 units: 6.9 us with 4 per thread, 7.4 us with 8).  Launches of many run beside
    // write-backs, whose CTAs they displace: 512 threads there.  KDA decode in four partitions, per token
    // with 4 and with 8 units per thread: partitions of 2 batch elements of 4096 units 27.4 and 27.5 us, of 8
    // 51.2 and 48.7, of 16 97.0 and 96.1, of 32 183.9 and 178.1, of 64 355.8 and 344.4; of 3072 units 25.4 and
    // 26.2, 40.8 and 39.4, 76.6 and 77.2, 140.0 and 136.7, 273.5 and 262.6.  In one chain, where nothing runs
    // beside them: 16 batch elements 35.4 and 35.7, 32 61.0 and 61.2, 64 100.3 and 100.8.  Hence 8 from the
    // size on at which it gains for both.  At 8192 units the same would be 16 per thread,
    // which cost more than it gave (Mamba-2: 211 against 210 us).
    if (p.units <= 4096) return p.units > 2048 && p.B >= 32 ? launch_alloc_t<8, true>(p, stream) : launch_alloc_t<4, true>(p, stream);
    if (p.units <= 8192) return launch_alloc_t<8, true>(p, stream);
    return launch_alloc_t<16, true>(p, stream);
}

}  // namespace qs

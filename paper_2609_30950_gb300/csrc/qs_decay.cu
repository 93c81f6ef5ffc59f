// qs_decay.cu -- log-uniform decay-gate quantiser (Sec. 3, "Decay-gate quantization").
//
// Three passes over the rates s (count samples x nchan channels, channel fastest):
//   1. per-channel min / max (integer atomics on the bit patterns: rates are positive floats,
//      whose bit patterns order like the values), accumulated into lut[., 0] and lut[., L-1];
//   2. per channel, FP64 levels l_k = exp(lo + k step) and thresholds
//      exp(lo + (k - 1/2) step), lo/hi = log min/max, step = (hi - lo)/(L - 1), rounded to FP32
//      (l_0 = min and l_{L-1} = max exactly);
//   3. codes = number of thresholds <= s, one byte per rate.
// Passes 1 and 3 are bound by HBM (4 bytes read, then 4 read and 1 written per rate).  A lane keeps
// its 4 channels for the whole launch: minima, maxima and thresholds stay in registers, with 4
// 16-byte loads in flight, and the rows of a block meet in shared memory before one atomic per
// channel.  Pass 1 sweeps the rows upwards and pass 3 downwards, so that pass 3 finds the rates
// read last in L2.  16 x 1024 x 4096 rates, 4 levels:
// 103 us (52 + 6 + 43 and the launches; 335 MB of the 603 MB from HBM in pass 3's share, 89 MB less
// than without the turn); 175 us with one rate per load and the thresholds read per rate.  Blocks that
// take 4 KB of a row at once instead of 512 bytes: 110 us.
#include <algorithm>
#include <mutex>

#include "qs_common.cuh"

namespace qs {

namespace {

__global__ void decay_init_kernel(float* lut, int nchan, int L) {
    const int ch = blockIdx.x * blockDim.x + threadIdx.x;
    if (ch < nchan) {
        lut[static_cast<size_t>(ch) * L] = INFINITY;
        lut[static_cast<size_t>(ch) * L + L - 1] = 0.0f;
    }
}

// How a launch walks the rates 16 bytes at a time: LC lanes cover P = 4 LC consecutive values, a
// chunk of one row's channels (P divides nchan) or several whole rows (nchan divides P), so a lane's
// channels are fixed; 256 / LC such strips per block step through the strips of its chunk.  Other
// channel counts (ANY, one chunk) take a number of blocks for which the step is a
// multiple of nchan: a lane's channels are fixed too, but differ between the strips of a block.
struct Walk {
    long long total, pitch;   // values in whole groups of 4; between a chunk's consecutive strips
    long long strips;         // strips per chunk
    int chunks, nchan;
    int tail;                 // values after the whole groups (0 to 3), by the first block's first threads
};
constexpr int kAnyChannels = 1024;   // heads, at most
constexpr int kDecayThreads = 256, kInFlight = 4;
// Blocks per SM, all resident, so that the sweeps keep their order: by the registers that the
// thresholds take.
constexpr int kMinmaxBlocks = 5;
constexpr uint32_t kMaxRate = 0x7f7fffffu;   // the largest finite float
constexpr int codes_blocks(int lm1) { return lm1 <= 3 ? 5 : lm1 <= 7 ? 3 : 2; }

// ANYC: with ANY, the most channels (256 or kAnyChannels: the shared extrema are set and read for each);
// else 0.
template <int LC, int ANYC>
__global__ void __launch_bounds__(kDecayThreads, kMinmaxBlocks) decay_minmax_rows_kernel(const float* __restrict__ s, const Walk wk, int L,
                                                                          float* lut, int* status) {
    constexpr int RS = kDecayThreads / LC;
    __shared__ uint4 smn[RS][LC], smx[RS][LC];
    constexpr bool ANY = ANYC > 0;
    constexpr int NC = ANY ? ANYC : 4 * LC;
    __shared__ uint32_t cmn[NC], cmx[NC];
    const int lane = threadIdx.x % LC, sub = threadIdx.x / LC;
    const int chunk = blockIdx.x % wk.chunks;
    const long long slices = gridDim.x / wk.chunks, step = slices * RS;
    const long long off = static_cast<long long>(chunk) * 4 * LC + lane * 4;
    const long long r0 = static_cast<long long>(blockIdx.x / wk.chunks) * RS + sub;
    const long long d = step * wk.pitch;                    // values from one of the lane's strips to the next
    long long mine = r0 < wk.strips ? (wk.strips - 1 - r0) / step + 1 : 0;
    const uint32_t* at = reinterpret_cast<const uint32_t*>(s) + r0 * wk.pitch + off;
    if (mine > 0 && (r0 + (mine - 1) * step) * wk.pitch + off >= wk.total) --mine;   // last strip of a short walk
    // On the bit patterns, unsigned: a rate is good from 1 to kMaxRate, so the extrema tell at the
    // end whether any was bad (two operations per rate; testing each took the ALU as long as
    // reading it takes)
    uint4 mn = make_uint4(~0u, ~0u, ~0u, ~0u), mx = make_uint4(0u, 0u, 0u, 0u);
    auto take = [&](const uint4& x) {
        mn.x = min(mn.x, x.x); mn.y = min(mn.y, x.y); mn.z = min(mn.z, x.z); mn.w = min(mn.w, x.w);
        mx.x = max(mx.x, x.x); mx.y = max(mx.y, x.y); mx.z = max(mx.z, x.z); mx.w = max(mx.w, x.w);
    };
    long long m = 0;
    for (; m + kInFlight <= mine; m += kInFlight) {
        uint4 x[kInFlight];
#pragma unroll
        for (int k = 0; k < kInFlight; ++k) x[k] = __ldg(reinterpret_cast<const uint4*>(at + (m + k) * d));
#pragma unroll
        for (int k = 0; k < kInFlight; ++k) take(x[k]);
    }
    for (; m < mine; ++m) take(__ldg(reinterpret_cast<const uint4*>(at + m * d)));
    const bool bad = mine > 0 && (min(min(mn.x, mn.y), min(mn.z, mn.w)) < 1u || max(max(mx.x, mx.y), max(mx.z, mx.w)) > kMaxRate);
    auto good = [](uint32_t v, uint32_t& lo, uint32_t& hi) {
        if (v < 1u || v > kMaxRate) return false;
        lo = min(lo, v);
        hi = max(hi, v);
        return true;
    };
    if (bad) {
        // once more, the good rates only
        raise_status(status, QS_DEV_RATE);
        mn = make_uint4(~0u, ~0u, ~0u, ~0u);
        mx = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll 1
        for (m = 0; m < mine; ++m) {
            const uint4 x = __ldg(reinterpret_cast<const uint4*>(at + m * d));
            good(x.x, mn.x, mx.x);
            good(x.y, mn.y, mx.y);
            good(x.z, mn.z, mx.z);
            good(x.w, mn.w, mx.w);
        }
    }
    smn[sub][lane] = mn;
    smx[sub][lane] = mx;
    for (int i = threadIdx.x; i < NC; i += kDecayThreads) {
        cmn[i] = kMaxRate + 1u;   // infinity
        cmx[i] = 0u;
    }
    __syncthreads();
    // the extrema of the block's 1024 values in turn, then of each channel among them
    const uint32_t *vmn = reinterpret_cast<const uint32_t*>(smn), *vmx = reinterpret_cast<const uint32_t*>(smx);
    const int nc = ANY ? wk.nchan : min(wk.nchan, 4 * LC);
    if constexpr (ANY) {
        // the block's values follow one another from a multiple of 1024 on: every nc-th is a channel's
        const long long first = static_cast<long long>(blockIdx.x) * 4 * kDecayThreads;
        if (ANYC <= kDecayThreads || nc <= kDecayThreads) {
            const int per = kDecayThreads / nc * nc, t = threadIdx.x;
            if (t < per) {
                uint32_t lo = ~0u, hi = 0u;
                for (int i = t; i < 4 * kDecayThreads; i += per) {
                    lo = min(lo, vmn[i]);
                    hi = max(hi, vmx[i]);
                }
                const int ch = static_cast<int>((first + t) % nc);
                atomicMin(&cmn[ch], lo);
                atomicMax(&cmx[ch], hi);
            }
        } else {
            for (int i = threadIdx.x; i < 4 * kDecayThreads; i += kDecayThreads) {
                const int ch = static_cast<int>((first + i) % nc);
                atomicMin(&cmn[ch], vmn[i]);
                atomicMax(&cmx[ch], vmx[i]);
            }
        }
    } else {
        for (int i = threadIdx.x; i < 4 * LC; i += kDecayThreads) {
            uint32_t lo = ~0u, hi = 0u;
            for (int k = 0; k < RS; ++k) {
                lo = min(lo, vmn[k * 4 * LC + i]);
                hi = max(hi, vmx[k * 4 * LC + i]);
            }
            atomicMin(&cmn[i % nc], lo);
            atomicMax(&cmx[i % nc], hi);
        }
    }
    if (blockIdx.x == 0 && static_cast<int>(threadIdx.x) < wk.tail) {
        const long long e = wk.total + threadIdx.x;
        uint32_t lo = ~0u, hi = 0u;
        if (!good(__ldg(reinterpret_cast<const uint32_t*>(s) + e), lo, hi)) raise_status(status, QS_DEV_RATE);
        atomicMin(&cmn[e % nc], lo);
        atomicMax(&cmx[e % nc], hi);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nc; i += kDecayThreads) {
        if (ANYC > 256 && cmx[i] == 0u) continue;   // no good rate of this channel here
        float* l = lut + (static_cast<size_t>(chunk) * 4 * LC + i) * L;
        atomicMin(reinterpret_cast<uint32_t*>(l), cmn[i]);
        atomicMax(reinterpret_cast<uint32_t*>(l + L - 1), cmx[i]);
    }
}

// Any channel count and alignment (unaligned rates; more than 256 heads with few samples or no
// multiple of 4): thread e0 visits elements e0, e0 + S, e0 + 2S, ... with S a
// multiple of nchan, so its channel is fixed.
__global__ void decay_minmax_kernel(const float* __restrict__ s, long long total, int nchan,
                                    int L, float* lut, int* status) {
    const long long S = static_cast<long long>(gridDim.x) * blockDim.x;
    const long long e0 = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
    const int ch = static_cast<int>(e0 % nchan);
    float mn = INFINITY, mx = 0.0f;
    bool bad = false;
    for (long long e = e0; e < total; e += S) {
        const float x = __ldg(s + e);
        if (x > 0.0f && x < INFINITY) {
            mn = fminf(mn, x);
            mx = fmaxf(mx, x);
        } else {
            bad = true;
        }
    }
    if (bad) raise_status(status, QS_DEV_RATE);
    if (e0 < total) {
        atomicMin(reinterpret_cast<int*>(lut + static_cast<size_t>(ch) * L), __float_as_int(mn));
        atomicMax(reinterpret_cast<int*>(lut + static_cast<size_t>(ch) * L + L - 1), __float_as_int(mx));
    }
}

// FP64 arithmetic bounds this pass (4096 channels of 4 levels: 8192 logarithms and 20480
// exponentials), so its lanes are kept full: a block takes `per` channels, a thread per logarithm
// and then a thread per exponential.  4096 channels of 4 levels: 6.3 us (a thread per channel,
// one warp to a block: 9.4 us; four warps: 9.2 us).
constexpr int kLevelThreads = 160, kLevelChannels = 32;
__global__ void __launch_bounds__(kLevelThreads) decay_levels_kernel(float* lut, float* thr, int nchan, int L, int per,
                                                                     int* status) {
    __shared__ double lg[kLevelChannels][2];
    const int c0 = blockIdx.x * per, nc = min(per, nchan - c0);
    if (static_cast<int>(threadIdx.x) < 2 * nc) {
        const int c = threadIdx.x >> 1, hi = threadIdx.x & 1;
        const float* l = lut + static_cast<size_t>(c0 + c) * L;
        const float mn = l[0], mx = l[L - 1];
        const bool ok = mn > 0.0f && mx < INFINITY && mn <= mx;
        if (!ok && hi) raise_status(status, QS_DEV_RATE);
        lg[c][hi] = ok ? log(static_cast<double>(hi ? mx : mn)) : NAN;   // NaN: no levels
    }
    __syncthreads();
    // items 0 .. L-2 of a channel: thresholds 1 .. L-1; then levels 1 .. L-2
    const int items = 2 * L - 3;
    for (int i = threadIdx.x; i < nc * items; i += kLevelThreads) {
        const int c = i / items, it = i - c * items;
        const double lo = lg[c][0], hi = lg[c][1];
        if (!(lo <= hi)) continue;
        const double step = __ddiv_rn(__dsub_rn(hi, lo), static_cast<double>(L - 1));
        const bool level = it >= L - 1;
        const int k = level ? it - (L - 2) : it + 1;
        const double at = level ? static_cast<double>(k) : __dsub_rn(static_cast<double>(k), 0.5);
        const float v = static_cast<float>(exp(__dadd_rn(lo, __dmul_rn(at, step))));
        if (level) lut[static_cast<size_t>(c0 + c) * L + k] = v;
        else thr[static_cast<size_t>(c0 + c) * (L - 1) + k - 1] = v;
    }
}

// Codes from the last strip down.  LM1 thresholds for each of the lane's 4 channels in registers.
template <int LC, int LM1, bool ANY>
__global__ void __launch_bounds__(kDecayThreads, codes_blocks(LM1)) decay_codes_rows_kernel(const float* __restrict__ s, const Walk wk,
                                                                         const float* __restrict__ thr,
                                                                         uint8_t* __restrict__ codes) {
    constexpr int RS = kDecayThreads / LC;
    const int lane = threadIdx.x % LC, sub = threadIdx.x / LC;
    const int chunk = blockIdx.x % wk.chunks;
    const long long slices = gridDim.x / wk.chunks, step = slices * RS;
    const long long off = static_cast<long long>(chunk) * 4 * LC + lane * 4;
    const long long r0 = static_cast<long long>(blockIdx.x / wk.chunks) * RS + sub;   // strips from the end
    float th[4][LM1];
    if (blockIdx.x == 0 && static_cast<int>(threadIdx.x) < wk.tail) {
        const long long e = wk.total + threadIdx.x;
        const float x = __ldg(s + e), *t = thr + static_cast<size_t>(e % wk.nchan) * LM1;
        int c = 0;
        for (int k = 0; k < LM1; ++k) c += x >= __ldg(t + k) ? 1 : 0;
        codes[e] = static_cast<uint8_t>(c);
    }
    if (r0 >= wk.strips) return;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const size_t ch = ANY ? static_cast<size_t>(((wk.strips - 1 - r0) * wk.pitch + off + j) % wk.nchan)
                              : static_cast<size_t>(chunk) * 4 * LC + (lane * 4 + j) % min(wk.nchan, 4 * LC);
#pragma unroll
        for (int k = 0; k < LM1; ++k) th[j][k] = __ldg(thr + ch * LM1 + k);
    }
    const long long d = step * wk.pitch;
    long long left = (wk.strips - 1 - r0) / step + 1;
    long long e = (wk.strips - 1 - r0) * wk.pitch + off;
    if (left > 0 && e >= wk.total) {   // last strip of a short walk
        e -= d;
        --left;
    }
    auto code = [&](const float4& x) {
        const float xs[4] = {x.x, x.y, x.z, x.w};
        uint32_t packed = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            uint32_t c = 0;
#pragma unroll
            for (int m = 0; m < LM1; ++m) c += xs[j] >= th[j][m] ? 1u : 0u;
            packed |= c << (8 * j);
        }
        return packed;
    };
    for (; left >= kInFlight; left -= kInFlight, e -= kInFlight * d) {
        float4 x[kInFlight];
#pragma unroll
        for (int k = 0; k < kInFlight; ++k) x[k] = __ldcs(reinterpret_cast<const float4*>(s + e - k * d));
#pragma unroll
        for (int k = 0; k < kInFlight; ++k) __stcs(reinterpret_cast<uint32_t*>(codes + e - k * d), code(x[k]));
    }
    for (; left > 0; --left, e -= d)
        __stcs(reinterpret_cast<uint32_t*>(codes + e), code(__ldcs(reinterpret_cast<const float4*>(s + e))));
}

__global__ void decay_codes_generic_kernel(const float* __restrict__ s, long long total, int nchan,
                                           int LM1, const float* __restrict__ thr,
                                           uint8_t* __restrict__ codes) {
    const long long stride = static_cast<long long>(gridDim.x) * blockDim.x;
    for (long long e = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; e < total; e += stride) {
        const float x = __ldg(s + e);
        const float* t = thr + static_cast<size_t>(e % nchan) * LM1;
        int c = 0;
        for (int k = 0; k < LM1; ++k) c += (x >= __ldg(t + k)) ? 1 : 0;
        codes[e] = static_cast<uint8_t>(c);
    }
}

long long gcd_ll(long long a, long long b) { return b == 0 ? a : gcd_ll(b, a % b); }

}  // namespace

cudaError_t launch_quant_decay(const float* s, long long count, int nchan, int g, uint8_t* codes,
                               float* lut, float* thr, int* status, cudaStream_t stream) {
    const int L = 1 << g;
    const long long total = count * nchan;
    decay_init_kernel<<<(nchan + 255) / 256, 256, 0, stream>>>(lut, nchan, L);
    // The 16-byte walk where a lane's channels can stay fixed: row decay always (channels a multiple
    // of 64), and heads; codes of up to 16 levels, whose thresholds fit in registers.
    // A rate at a time, every thread's extrema went to the few channels by global atomics: call by
    // call from a cold L2, 118 x 256 x 12 rates took 221 us and 256 x 1024 x 1 took 360 us; the walk
    // takes 30 and 28 us (of which 14 us are the call and its four launches).
    // Above 256 heads the walk needs nchan / gcd(nchan, 1024) blocks, all resident (2 per SM at 16 levels):
    // heads in fours, at most 255 blocks.  4 levels, calls replayed in a graph: 65536 samples of 1020 heads
    // 106 us, 264 a rate at a time; 4096 of 260 15 and 32; 1024 of 1000 14.6 and 16.7, of 1020 17.0 and
    // 16.2; 64 of 1000 12.1 and 9.8, hence the line at 1024 samples.
    const bool aligned = (reinterpret_cast<uintptr_t>(s) & 15) == 0 && (reinterpret_cast<uintptr_t>(codes) & 3) == 0;
    const bool fixed = nchan % 128 == 0 || 128 % nchan == 0;
    const bool heads = nchan % 64 != 0 && (nchan <= 256 || (nchan <= kAnyChannels && nchan % 4 == 0 && count >= 1024));
    const int lc = fixed || heads ? 32 : nchan % 64 == 0 ? 16 : 0;
    const bool any = lc == 32 && !fixed;
    const bool walk = aligned && lc > 0;
    Walk wk = {};
    long long turn = 1;   // blocks after which a strip meets the same channels again
    if (walk) {
        const int P = 4 * lc;
        wk.tail = static_cast<int>(total & 3);
        wk.total = total - wk.tail;
        wk.nchan = nchan;
        wk.chunks = any ? 1 : std::max(1, nchan / P);
        wk.pitch = any ? P : std::max(nchan, P);
        wk.strips = (wk.total + wk.pitch - 1) / wk.pitch;
        if (any) turn = nchan / gcd_ll(nchan, 4 * kDecayThreads);
    }
    // resident blocks, a whole number per chunk; fewer when there are not two strips for each lane
    auto blocks_of = [&](int per_sm, long long most = 1LL << 31) {
        const long long rs = kDecayThreads / lc;
        const long long want = std::min(most, std::max(1LL, static_cast<long long>(device_sm_count()) * per_sm / wk.chunks));
        const long long b = std::max(1LL, std::min(want, (wk.strips + rs * 2 - 1) / (rs * 2)));
        return static_cast<unsigned>(wk.chunks * (any ? std::max(turn, b / turn * turn) : b));
    };
    if (walk) {
        // of many heads, each block's extrema are as many atomics: 16 samples to a block at least (4096
        // samples of 1000 heads, 4 levels: 30 us without this)
        const long long most = any && nchan > 256 ? std::max(1LL, count / 16) : 1LL << 31;
#define QS_DM(LC, ANYC) decay_minmax_rows_kernel<LC, ANYC><<<blocks_of(kMinmaxBlocks, most), kDecayThreads, 0, stream>>>(s, wk, L, lut, status)
        if (any && nchan > 256) QS_DM(32, kAnyChannels);
        else if (any) QS_DM(32, 256);
        else if (lc == 32) QS_DM(32, 0);
        else QS_DM(16, 0);
#undef QS_DM
    } else {
        // S = a multiple of lcm(nchan, 256) near (SMs x 8) CTAs of 256 threads
        const long long lcm = static_cast<long long>(nchan) / gcd_ll(nchan, 256) * 256;
        const long long target = static_cast<long long>(device_sm_count()) * 8 * 256;
        long long S = std::max(lcm, (target / lcm) * lcm);
        while (S / 256 > 0x7fffffffLL) S -= lcm;
        decay_minmax_kernel<<<static_cast<unsigned>(S / 256), 256, 0, stream>>>(s, total, nchan, L, lut, status);
    }
    const int per = std::min(kLevelChannels, std::max(1, kLevelThreads / (2 * L - 3)));
    decay_levels_kernel<<<(nchan + per - 1) / per, kLevelThreads, 0, stream>>>(lut, thr, nchan, L, per, status);
    const unsigned blocks = static_cast<unsigned>(device_sm_count()) * 8u;
    if (walk && L <= 16) {
#define QS_DC(LC, LM1, ANY) \
    decay_codes_rows_kernel<LC, LM1, ANY><<<blocks_of(codes_blocks(LM1)), kDecayThreads, 0, stream>>>(s, wk, thr, codes)
#define QS_DL(LC, ANY)                     \
    if (L == 2) QS_DC(LC, 1, ANY);         \
    else if (L == 4) QS_DC(LC, 3, ANY);    \
    else if (L == 8) QS_DC(LC, 7, ANY);    \
    else QS_DC(LC, 15, ANY)
        if (any) {
            QS_DL(32, true);
        } else if (lc == 32) {
            QS_DL(32, false);
        } else {
            QS_DL(16, false);
        }
#undef QS_DL
#undef QS_DC
    } else {
        decay_codes_generic_kernel<<<blocks, 256, 0, stream>>>(s, total, nchan, L - 1, thr, codes);
    }
    return cudaGetLastError();
}

// ---- variant without caller-supplied threshold buffer -------------------------------------------
// The thresholds are an intermediate of the quantiser.  Callers that must not allocate device
// memory of their own keep them here: one file-scope array per device (every GPU that loads
// the library holds it until the process exits), shared by all calls on that device.
constexpr long long kDecayScratchFloats = 65536;   // 256 KiB: channels x (2^g - 1) thresholds
static __device__ __align__(256) float g_decay_thr_scratch[kDecayScratchFloats];

namespace {
constexpr int kMaxDev = 64;
std::mutex g_scratch_mu;
float* g_scratch_addr[kMaxDev] = {};
unsigned long long g_scratch_ctx[kMaxDev] = {};
}  // namespace

long long quant_decay_scratch_capacity() { return kDecayScratchFloats; }

// Device address of the threshold scratch on the current device, looked up on the first call
// made with that device current (a host-side lookup: make it before any stream capture), and
// again whenever the device's context has been created anew since (its module, and with it
// the array, may then sit at another address).
cudaError_t quant_decay_scratch(float** out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDev) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_scratch_mu);
    unsigned long long ctx = 0;
    const bool known = current_context_id(&ctx);
    if (!g_scratch_addr[dev] || !known || ctx != g_scratch_ctx[dev]) {
        void* ptr = nullptr;
        e = cudaGetSymbolAddress(&ptr, g_decay_thr_scratch);
        if (e != cudaSuccess) return e;
        g_scratch_addr[dev] = static_cast<float*>(ptr);
        g_scratch_ctx[dev] = current_context_id(&ctx) ? ctx : 0ull;
    }
    *out = g_scratch_addr[dev];
    return cudaSuccess;
}

}  // namespace qs

// First convolution (one input channel) on the tensor cores.
//
// Per output pixel the layer is a dot product of k*k depth values with each of C1 filters: far too short a
// reduction for the CUDA cores to do cheaply (C1 * k*k multiply-adds per pixel, one instruction each), but
// one tcgen05.mma of K = 16 covers a 3x3 window for 128 pixels and all filters at once.  Four kinds of warps:
//   loader    the frame rows a stage of T x 128 output pixels needs are one contiguous run of memory (also across
//             frames): one untiled bulk copy brings them into shared memory
//   builders  one pixel per thread: the window's rows as aligned pairs of fp16 pixels from that run, put together
//             in registers and written as the 16-byte pieces of the pixel's im2col row, in the unswizzled K-major
//             core-matrix layout (8 rows x 16 bytes per core matrix)
//   MMA       one thread
//   epilogue  ReLU + bf16 conversion in one instruction per pair, the one-bit ReLU gates the backward pass reads, and per
//             warp and 32 pixels x 32 channels one bulk tensor store from a swizzled 2 KB tile
// A window row starts at an even or odd column of the frame, so it is taken as aligned pairs: the K axis is laid out as
// (window row, pair, element of the pair), with one element per row that lies outside the window and meets a zero filter
// entry.  The filters are converted from the bf16 shadow to fp16 once per CTA, so that both operands are fp16 and the
// depth values enter exactly; the bias rides in two spare K slots as a pair of fp16 values (high part, remainder)
// against a constant 1.  fp32 accumulation in tensor memory.
// What bounds it: the output's way to HBM and, on a level with it, the instructions of builders and epilogue (everything
// about a group's shape is a template argument for that reason).  Copying every pair from global memory into its place
// by itself (4 bytes per copy, 15 per pixel of a 5x5 window, each store a four-way bank conflict) was bound by the
// copies.  4096 frames, 4-byte copies per pair -> rows (HBM time): 320x240 5x5 32 filters 2.05 -> 1.06 ms (0.88); 160x120 3x3 32 filters
// 0.41 -> 0.25 (0.22); 160x120 3x3 16 filters normalised 0.51 -> 0.29 (0.22).
// Frames must hold finite values (an Inf or NaN beside a window would meet a zero weight) and have an even
// width.
#include "conv1_window.h"
#include "gemm.cuh"
#include "launch.cuh"
#include "tcgen05.cuh"
#include "tma_host.cuh"

namespace {

using namespace tc;

constexpr int kMaxStages = 4;
constexpr int kRaw = 3;          // runs of frame rows in flight
constexpr int kBuildWarps = 8;   // two groups of 128 threads on alternate tiles
constexpr int kEpiWarps = 16;    // four per TMEM lane quarter, which take the column groups in turn
constexpr int kLoadWarp = kBuildWarps, kMmaWarp = kBuildWarps + 1, kEpiWarp0 = kBuildWarps + 2;
constexpr int kThreads = (kBuildWarps + 2 + kEpiWarps) * 32;
constexpr size_t kSmemMax = 227 * 1024;
constexpr int kStgBytes = 2048;  // an epilogue warp's staging tile; it has two

struct Args {
    CUtensorMap map_out, map_xhat;
    const bf16 *W;      // [C1][k*k] bf16
    const float *bias;  // [C1]
    uint32_t *bits;     // [M][C1 / 32], [M] half words for C1 = 16, or null
    const float *ln_gamma, *ln_beta;  // layer normalisation over the C1 channels of a pixel (null: none; C1 = 16 or 32)
    float *ln_rstd;     // [M]
    long long M;        // output pixels
    long long words;    // 32-bit words of all frames
    int Hi, Wi, Ho, Wo, C1;
    int tiles;   // 128-pixel tiles
    int stages;
    uint32_t raw_bytes;  // room for one run of frame rows
    int32_t *status;
};

struct Pipe {
    uint64_t rfull[kRaw], rempty[kRaw];
    uint64_t full[kMaxStages], empty[kMaxStages];
    uint64_t tfull[4], tempty[4];
    uint32_t tmem_slot;
    int abort_flag;
    long long raw_word[kRaw];  // first word of the run in each buffer
    alignas(16) float gamma[32], beta[32];
};

// Unswizzled K-major operand image: element (row r, column k) of a tile with KP columns lives at
// (r / 8) * (KP / 8) * 128 + (k / 8) * 128 + (r % 8) * 16 + (k % 8) * 2 bytes.
__device__ __forceinline__ uint32_t core_offset(int r, int kchunk, int KP) {
    return (uint32_t)(r >> 3) * (uint32_t)(KP >> 3) * 128u + (uint32_t)kchunk * 128u + (uint32_t)(r & 7) * 16u;
}

__device__ __forceinline__ uint64_t desc_nosw(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}

// kind::f16 with fp16 A and B (format 0), fp32 D, both K-major.
__host__ __device__ constexpr uint32_t idesc_f16(int M, int N) {
    return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// K layout of a window (conv1_window.h): halves 2 KS NP and 2 KS NP + 1 carry the constant 1 for the two bias parts; the rest up to KP are
// zero, as are the filter entries of kernel columns outside 0 .. KS-1.
template <int KS>
struct Win : Window<KS> {
    static constexpr int KP = (2 * Window<KS>::KW + 2 + 15) / 16 * 16;  // halves per im2col row
};

// Output pixel of a walk through the frames, advanced without divisions.
struct PixAt {
    int ow, oh, ib;
    __device__ void init(const Args &a, long long m) {
        ow = (int)(m % a.Wo);
        const long long t = m / a.Wo;
        oh = (int)(t % a.Ho);
        ib = (int)(t / a.Ho);
    }
    __device__ void advance(const Args &a, int d_w, int d_h) {  // by d_h rows and d_w < Wo pixels
        ow += d_w;
        oh += d_h;
        if (ow >= a.Wo) { ow -= a.Wo; ++oh; }
        while (oh >= a.Ho) { oh -= a.Ho; ++ib; }
    }
};

// T: tiles per stage (one barrier round trip and one accumulator hand-over each).
// DIRECT: builders read the frames from global memory themselves; for frames so wide that a run does not fit.
// CW: channels of an epilogue group, 32 or (C1 no multiple of 32) 16.  LN: layer normalisation (C1 == CW).
// (depth is the last argument: a prepared launch is made again with other frames.)
template <int KS, int T, bool DIRECT, int CW, bool LN>
__global__ void __launch_bounds__(kThreads, 1) conv1_tc_kernel(const __grid_constant__ Args a, const __half *depth) {
    using WN = Win<KS>;
    constexpr int K2 = KS * KS, KP = WN::KP, P = WN::P, ODD = WN::ODD, NP = WN::NP, KW = WN::KW;
    constexpr uint32_t kTileBytes = 128u * KP * 2u, kStageBytes = T * kTileBytes;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int N = a.C1, S = a.stages;
    // im2col stages, filters, epilogue staging, frame rows, pipeline state
    uint8_t *bsm = smem + (size_t)S * kStageBytes;                 // filters [N][KP] fp16
    const uint32_t stg_off = (uint32_t)S * kStageBytes + (((uint32_t)(N * KP * 2) + 1023u) & ~1023u);
    const uint32_t raw_off = stg_off + (uint32_t)kEpiWarps * 2u * kStgBytes;
    Pipe *pipe = reinterpret_cast<Pipe *>(smem + raw_off + (size_t)kRaw * a.raw_bytes);
    volatile int *abort_flag = &pipe->abort_flag;
    const int warp = warp_index(), lane = threadIdx.x & 31;
    const uint32_t acc_cols = tmem_cols_for(T * N);                // T accumulators side by side
    const int nacc_log = acc_cols * 4 <= 512 ? 2 : 1, nacc = 1 << nacc_log;
    const uint32_t ncols = acc_cols * nacc;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kRaw; ++s) {
            mbar_init(&pipe->rfull[s], 1);
            mbar_init(&pipe->rempty[s], kBuildWarps * 32);
        }
        for (int s = 0; s < S; ++s) {
            mbar_init(&pipe->full[s], kBuildWarps * 32);
            mbar_init(&pipe->empty[s], 1);
        }
        for (int i = 0; i < nacc; ++i) {
            mbar_init(&pipe->tfull[i], 1);
            mbar_init(&pipe->tempty[i], kEpiWarps * 32);
        }
        pipe->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kMmaWarp) tmem_alloc(&pipe->tmem_slot, ncols);
    grid_wait();
    // filters in the K layout of the window, bias parts in the two slots behind it, zeros elsewhere
    for (int i = threadIdx.x; i < N * KP; i += kThreads) {
        const int n = i / KP, k = i - n * KP;
        float f = 0.f;
        if (k < 2 * KW) {
            const int w = k >> 1, kh = w / NP, kw = 2 * (w - kh * NP) + (k & 1) - ODD;
            if (kw >= 0 && kw < KS) f = bf2f(a.W[n * K2 + kh * KS + kw]);
        } else if (k == 2 * KW) {
            f = __half2float(__float2half_rn(a.bias[n]));
        } else if (k == 2 * KW + 1) {
            f = a.bias[n] - __half2float(__float2half_rn(a.bias[n]));
        }
        *reinterpret_cast<__half *>(bsm + core_offset(n, k >> 3, KP) + (k & 7) * 2) = __float2half_rn(f);
    }
    if (a.ln_gamma && threadIdx.x < 32) {
        pipe->gamma[threadIdx.x] = (int)threadIdx.x < N ? a.ln_gamma[threadIdx.x] : 0.f;
        pipe->beta[threadIdx.x] = (int)threadIdx.x < N ? a.ln_beta[threadIdx.x] : 0.f;
    }
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = pipe->tmem_slot;
    const uint32_t smem_base = smem_u32(smem);

    // contiguous run of stages (T tiles each) for this CTA
    const int nstage_all = (a.tiles + T - 1) / T;
    const int q = nstage_all / (int)gridDim.x, rem = nstage_all - q * (int)gridDim.x, b = (int)blockIdx.x;
    const int s0 = b * q + (b < rem ? b : rem), ns = q + (b < rem ? 1 : 0);
    const int Wh = a.Wi >> 1;  // 32-bit words per frame row

    if (warp == kLoadWarp) {
        // ---------------- loader: one bulk copy per stage.  The few words in front of the first or behind the last
        // 16-byte unit of all frames (where the unit would reach outside them) are copied by hand.
        if (!DIRECT && lane == 0) {
            const uint32_t *frames = reinterpret_cast<const uint32_t *>(depth);
            const uintptr_t lo_all = reinterpret_cast<uintptr_t>(frames), hi_all = lo_all + (uintptr_t)a.words * 4;
            PixAt first, last;
            first.init(a, (long long)s0 * T * 128);
            last.init(a, (long long)s0 * T * 128 + T * 128 - 1);
            const int d_w = (T * 128) % a.Wo, d_h = (T * 128) / a.Wo;
            const int images = (int)(a.M / ((long long)a.Ho * a.Wo));
            bool ok = true;
            int s = 0, li = 0;
            uint32_t ph = 0;
            for (; li < ns; ++li) {
                ok = mbar_wait(&pipe->rempty[s], ph ^ 1u, abort_flag, a.status);
                if (!ok) break;
                int eb = last.ib, eh = last.oh;
                if (eb >= images) { eb = images - 1; eh = a.Ho - 1; }
                const long long r0 = (long long)first.ib * a.Hi + max(0, 2 * first.oh - P);
                const long long r1 = (long long)eb * a.Hi + min(a.Hi, 2 * eh + P + 1);
                const uintptr_t lo = lo_all + (uintptr_t)(r0 * Wh) * 4, hi = lo_all + (uintptr_t)(r1 * Wh) * 4;
                const uintptr_t origin = lo & ~uintptr_t(15);
                uintptr_t c_lo = origin, c_hi = (hi + 15) & ~uintptr_t(15);
                if (c_lo < lo_all) c_lo += 16;
                if (c_hi > hi_all) c_hi -= 16;
                uint8_t *raw = smem + raw_off + (size_t)s * a.raw_bytes;
                for (uintptr_t p = lo; p < c_lo && p < hi; p += 4)
                    *reinterpret_cast<uint32_t *>(raw + (p - origin)) = *reinterpret_cast<const uint32_t *>(p);
                for (uintptr_t p = c_hi > lo ? c_hi : lo; p < hi; p += 4)
                    *reinterpret_cast<uint32_t *>(raw + (p - origin)) = *reinterpret_cast<const uint32_t *>(p);
                pipe->raw_word[s] = (long long)(origin - lo_all) / 4;
                const uint32_t bytes = c_hi > c_lo ? (uint32_t)(c_hi - c_lo) : 0u;
                mbar_arrive_expect_tx(&pipe->rfull[s], bytes);
                if (bytes) bulk_load(smem_u32(raw) + (uint32_t)(c_lo - origin), reinterpret_cast<const void *>(c_lo), bytes, &pipe->rfull[s]);
                first.advance(a, d_w, d_h);
                last.advance(a, d_w, d_h);
                if (++s == kRaw) { s = 0; ph ^= 1u; }
            }
            if (!ok)
                for (int i = max(0, li - kRaw); i < li; ++i) {  // bounded wait for the copies in flight
                    const long long c0 = clock64();
                    while (!mbar_try_wait(&pipe->rfull[i % kRaw], (i / kRaw) & 1))
                        if (clock64() - c0 > kWaitCycles / 4) break;
                }
        }
        __syncwarp();
    } else if (warp < kBuildWarps) {
        // ---------------- builders: thread r of group q fills row r of tiles q, q + 2, .. of every stage
        const int grp = threadIdx.x >> 7, r = threadIdx.x & 127;
        const uint32_t *frames = reinterpret_cast<const uint32_t *>(depth);
        const int d_w = 256 % a.Wo, d_h = 256 / a.Wo;
        long long m = ((long long)s0 * T + grp) * 128 + r;
        PixAt at;
        at.init(a, m);
        const uint32_t row_off = core_offset(r, 0, KP);
        bool ok = true;
        int s = 0, rs = 0;
        uint32_t ph = 0, rph = 0;
        for (int li = 0; li < ns; ++li) {
            long long raw_word = 0;
            if (!DIRECT) {
                ok = mbar_wait(&pipe->rfull[rs], rph, abort_flag, a.status);
                if (!ok) break;
                raw_word = pipe->raw_word[rs];
            }
            ok = mbar_wait(&pipe->empty[s], ph ^ 1u, abort_flag, a.status);
            if (!ok) break;
            const uint32_t raw = smem_base + raw_off + (uint32_t)rs * a.raw_bytes;
#pragma unroll
            for (int g = 0; g < T / 2; ++g) {
                const bool live = m < a.M;
                const int ih0 = 2 * at.oh - P, pw0 = at.ow - (P + ODD) / 2;  // first window row; its first pair, in words
                const long long w0 = ((long long)at.ib * a.Hi + ih0) * Wh + pw0;
                const uint32_t a0 = raw + (uint32_t)(int)(w0 - raw_word) * 4u;
                uint32_t w[KP / 2];
#pragma unroll
                for (int kh = 0; kh < KS; ++kh) {
                    const bool rok = live && (unsigned)(ih0 + kh) < (unsigned)a.Hi;
#pragma unroll
                    for (int qq = 0; qq < NP; ++qq) {
                        const bool pok = rok && (unsigned)(pw0 + qq) < (unsigned)Wh;
                        uint32_t v = 0u;
                        if (DIRECT) {
                            if (pok) v = __ldg(frames + w0 + (long long)kh * Wh + qq);
                        } else if (pok) {
                            asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(a0 + (uint32_t)(kh * Wh + qq) * 4u));
                        }
                        w[kh * NP + qq] = v;
                    }
                }
#pragma unroll
                for (int k = KW; k < KP / 2; ++k) w[k] = k == KW ? 0x3C003C00u : 0u;  // 1.0 against the two bias parts, then zeros
                const uint32_t dst = smem_base + (uint32_t)s * kStageBytes + (uint32_t)(2 * g + grp) * kTileBytes + row_off;
#pragma unroll
                for (int c = 0; c < KP / 8; ++c)
                    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst + (uint32_t)c * 128u), "r"(w[4 * c]), "r"(w[4 * c + 1]),
                                 "r"(w[4 * c + 2]), "r"(w[4 * c + 3])
                                 : "memory");
                m += 256;
                at.advance(a, d_w, d_h);
            }
            fence_async_smem();
            mbar_arrive(&pipe->full[s]);
            if (!DIRECT) mbar_arrive(&pipe->rempty[rs]);
            if (++s == S) { s = 0; ph ^= 1u; }
            if (++rs == kRaw) { rs = 0; rph ^= 1u; }
        }
    } else if (warp == kMmaWarp) {
        // ---------------- MMA issue: T tiles per stage, each into its own columns of the accumulator
        const uint32_t idesc = idesc_f16(128, N);
        const uint32_t sbo = (uint32_t)(KP >> 3) * 128u;
        const uint64_t dB = desc_nosw(smem_u32(bsm), 128u, sbo);
        const uint64_t dA0 = desc_nosw(smem_base, 128u, sbo);
        const uint32_t a_hi = (uint32_t)(dA0 >> 32), b_hi = (uint32_t)(dB >> 32);
        bool ok = true;
        int s = 0;
        uint32_t ph = 0;
        for (int li = 0; li < ns && ok; ++li) {
            const int acc = li & (nacc - 1);
            ok = mbar_wait_warp(&pipe->tempty[acc], ((li >> nacc_log) & 1) ^ 1, abort_flag, a.status);
            if (!ok) break;
            ok = mbar_wait_warp(&pipe->full[s], ph, abort_flag, a.status);
            if (!ok) break;
            tc_fence_after();
            if (elect_one()) {
                uint32_t la = (uint32_t)dA0 + (uint32_t)s * (kStageBytes >> 4);
                uint32_t td = tmem_base + acc * acc_cols;
#pragma unroll
                for (int g = 0; g < T; ++g, la += kTileBytes >> 4, td += N) {
#pragma unroll
                    for (int kk = 0; kk < KP / 16; ++kk)  // 16 columns = two core matrices = 256 bytes
                        umma_bf16_lh(td, la + kk * 16, a_hi, (uint32_t)dB + kk * 16, b_hi, idesc, kk > 0 ? 1u : 0u);
                }
                umma_commit(&pipe->empty[s]);
                umma_commit(&pipe->tfull[acc]);
            }
            __syncwarp();
            if (++s == S) { s = 0; ph ^= 1u; }
        }
    } else {
        // ---------------- epilogue: TMEM lane = pixel of a tile; warp w reads lanes 32 (w % 4) .. +31; the
        // warps of a lane quarter take the groups of 32 accumulator columns in turn (16 when C1 is not a multiple
        // of 32).  A group is 32 pixels x CW channels: one box of the output tensor.
        const int ew = warp - kEpiWarp0, lg = warp & 3, part = ew >> 2;
        constexpr uint32_t rbo = CW * 2u;
        const uint32_t sw = CW == 32 ? (uint32_t)(lane >> 1) & 3u : (uint32_t)(lane >> 2) & 1u;
        const uint32_t stg0 = smem_base + stg_off + (uint32_t)ew * 2u * kStgBytes;
        int buf = 0;
        // writes this lane's CW bf16 values (packed pairs) into the next staging tile and hands it to the copy engine
        auto emit = [&](const CUtensorMap *map, const uint32_t (&pk)[CW / 2], int c0, long long m0) {
            const uint32_t stg = stg0 + (uint32_t)buf * kStgBytes;
            if (lane == 0) bulk_wait_read<1>();  // the store before last has read this tile
            __syncwarp();
#pragma unroll
            for (int j = 0; j < CW / 8; ++j)
                asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(stg + (uint32_t)lane * rbo + (((uint32_t)j ^ sw) << 4)),
                             "r"(pk[4 * j]), "r"(pk[4 * j + 1]), "r"(pk[4 * j + 2]), "r"(pk[4 * j + 3])
                             : "memory");
            fence_async_smem();
            __syncwarp();
            if (lane == 0) {
                if (m0 < a.M) tma_store_2d(map, stg, c0, (int)m0);
                bulk_commit();
            }
            buf ^= 1;
        };
        bool ok = true;
        for (int li = 0; li < ns && ok; ++li) {
            const int acc = li & (nacc - 1);
            ok = mbar_wait(&pipe->tfull[acc], (li >> nacc_log) & 1, abort_flag, a.status);
            if (!ok) break;
            tc_fence_after();
            const uint32_t lane_base = tmem_base + acc * acc_cols + ((uint32_t)(lg * 32) << 16);
            for (int cc = part * CW; cc < T * N; cc += (kEpiWarps / 4) * CW) {   // column of the accumulator: tile g, channel c0
                const int g = cc / N, c0 = cc - g * N;
                const long long m0 = ((long long)(s0 + li) * T + g) * 128 + lg * 32;  // first pixel of this warp
                float v[CW];
                if constexpr (CW == 32) tmem_ld32(lane_base + (uint32_t)cc, v);
                else tmem_ld16(lane_base + (uint32_t)cc, v);
                uint32_t pk[CW / 2];
                uint32_t gate = 0;
                if (LN) {
                    // layer normalisation over the CW = C1 channels this thread holds: two passes in registers
                    float sum = 0.f, sq = 0.f;
#pragma unroll
                    for (int i = 0; i < CW; ++i) sum += v[i];
                    const float mean = sum / (float)CW;
#pragma unroll
                    for (int i = 0; i < CW; ++i) sq += (v[i] - mean) * (v[i] - mean);
                    const float rs = rsqrtf(sq / (float)CW + kLnEps);
#pragma unroll
                    for (int i = 0; i < CW; ++i) v[i] = (v[i] - mean) * rs;
#pragma unroll
                    for (int j = 0; j < CW / 2; ++j) pk[j] = pack_bf16x2(v[2 * j], v[2 * j + 1]);
                    emit(&a.map_xhat, pk, c0, m0);
                    if (m0 + lane < a.M) a.ln_rstd[m0 + lane] = rs;
#pragma unroll
                    for (int i = 0; i < CW; ++i) v[i] = fmaf(pipe->gamma[c0 + i], v[i], pipe->beta[c0 + i]);
                }
#pragma unroll
                for (int j = 0; j < CW / 2; ++j) {
                    pk[j] = relu_pack_bf16x2(v[2 * j], v[2 * j + 1]);
                    gate = gate_bits_add(gate, pk[j], j);
                }
                if (a.bits && m0 + lane < a.M) {
                    if (CW == 32) a.bits[(m0 + lane) * (N >> 5) + (c0 >> 5)] = gate;
                    else reinterpret_cast<uint16_t *>(a.bits)[m0 + lane] = gate_half(gate);
                }
                emit(&a.map_out, pk, c0, m0);
            }
            tc_fence_before();
            mbar_arrive(&pipe->tempty[acc]);
        }
        if (lane == 0) bulk_wait_all();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kMmaWarp) {
        tc_fence_after();
        tmem_dealloc(tmem_base, ncols);
    }
}

template <int KS, int T, bool DIRECT, int CW, bool LN>
int launch_one(const Args &a, const __half *depth, size_t smem, cudaStream_t st) {
    static PerDevice<bool> set;
    const auto fn = conv1_tc_kernel<KS, T, DIRECT, CW, LN>;
    PPO_TRY(ppo_once_per_device(set, [&] { return ppo_allow_smem(fn, kSmemMax); }));
    const int sms = ppo_num_sms(), nstage = (a.tiles + T - 1) / T;
    return ppo_launch(fn, dim3(nstage < sms ? nstage : sms), dim3(kThreads), smem, st, a, depth);
}

template <int KS, int T, int CW>
int launch(Args &a, const __half *depth, cudaStream_t st) {
    constexpr int KP = Win<KS>::KP;
    constexpr size_t stage = (size_t)T * 128 * KP * 2;
    a.stages = (int)(96 * 1024 / stage);
    a.stages = a.stages > kMaxStages ? kMaxStages : (a.stages < 2 ? 2 : a.stages);
    const size_t fixed = (size_t)a.stages * stage + ((size_t)(a.C1 * KP * 2 + 1023) / 1024) * 1024 +
                         (size_t)kEpiWarps * 2 * kStgBytes + sizeof(Pipe) + 1024;
    if (fixed > kSmemMax) return PPO_ERR_UNSUPPORTED;
    // rows of a stage's run: its first and last output rows are at most (T * 128 - 1 + Wo - 1) / Wo apart, two frame rows each
    const long long rows = 2ll * ((T * 128 - 1 + a.Wo - 1) / a.Wo) + 2 * (KS / 2) + 1;
    const long long raw = (rows * a.Wi * 2 + 32 + 15) / 16 * 16;
    const bool direct = fixed + kRaw * (size_t)raw > kSmemMax;
    a.raw_bytes = direct ? 0u : (uint32_t)raw;
    const size_t smem = fixed + kRaw * (size_t)a.raw_bytes;
    if (a.ln_gamma) return direct ? launch_one<KS, T, true, CW, true>(a, depth, smem, st) : launch_one<KS, T, false, CW, true>(a, depth, smem, st);
    return direct ? launch_one<KS, T, true, CW, false>(a, depth, smem, st) : launch_one<KS, T, false, CW, false>(a, depth, smem, st);
}

template <int KS>
int launch_c(Args &a, const __half *depth, cudaStream_t st) {
    if (a.C1 % 32 == 0) return launch<KS, 4, 32>(a, depth, st);
    return a.C1 == 16 ? launch<KS, 8, 16>(a, depth, st) : launch<KS, 4, 16>(a, depth, st);  // 8 tiles: 128 accumulator columns
}

}  // namespace

// out[m][co] = relu(bias[co] + sum_tap depth(m, tap) * W[co][tap]) as bf16; `bits` (optional, C1 % 32 == 0 or C1 = 16) gets the
// ReLU gates.  Returns PPO_ERR_UNSUPPORTED (nothing launched) for shapes it does not cover: C1 must be a multiple
// of 16 up to 64 (not 48 when bits are wanted), k in {3, 5, 7}, the frame width even and the frames 4-byte aligned.
int conv1_tc_fwd(const __half *depth, const bf16 *W, const float *bias, bf16 *out, uint32_t *bits, int rows, int Hi,
                 int Wi, int Ho, int Wo, int C1, int ks, const float *ln_gamma, const float *ln_beta, bf16 *ln_xhat,
                 float *ln_rstd, int32_t *status, cudaStream_t st) {
    if (!status || C1 % 16 != 0 || C1 > 64 || C1 < 16 || (bits && C1 % 32 != 0 && C1 != 16)) return PPO_ERR_UNSUPPORTED;
    if (ln_gamma && ((C1 != 16 && C1 != 32) || !ln_beta || !ln_xhat || !ln_rstd)) return PPO_ERR_UNSUPPORTED;
    if (Wi % 2 != 0 || !ppo_aligned(depth, 4)) return PPO_ERR_UNSUPPORTED;
    Args a = {};
    a.W = W; a.bias = bias; a.bits = bits;
    a.ln_gamma = ln_gamma; a.ln_beta = ln_beta; a.ln_rstd = ln_rstd;
    a.M = (long long)rows * Ho * Wo;
    a.words = (long long)rows * Hi * (Wi / 2);
    a.Hi = Hi; a.Wi = Wi; a.Ho = Ho; a.Wo = Wo; a.C1 = C1;
    const long long tiles = (a.M + 127) / 128;
    if (tiles <= 0) return PPO_OK;
    if (a.M > 0x7fffff00ll) return PPO_ERR_UNSUPPORTED;  // pixels are coordinates of the output map
    a.tiles = (int)tiles;
    a.status = status;
    const int CW = C1 % 32 == 0 ? 32 : 16;
    const long long dims[2] = {C1, a.M}, str[1] = {2ll * C1};
    const int box[2] = {CW, 32};
    PPO_TRY(make_map_strided(&a.map_out, out, 2, dims, str, box));
    if (ln_gamma) PPO_TRY(make_map_strided(&a.map_xhat, ln_xhat, 2, dims, str, box));
    if (ks == 3) return launch_c<3>(a, depth, st);
    if (ks == 5) return launch_c<5>(a, depth, st);
    if (ks == 7) return launch_c<7>(a, depth, st);
    return PPO_ERR_UNSUPPORTED;
}

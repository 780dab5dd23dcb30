// The fully connected layers behind the encoder as one launch per direction (sm_100a).
//
// Layer by layer they are a chain of kernels of 6 to 12 us that each do a microsecond of work: the rest is launching, filling a
// pipeline, fetching weights and draining.  Rows do not depend on one another, so a tile of rows goes through all layers in one
// cluster of 4 or 8 CTAs: a CTA owns a slice of each layer's columns, weights stream into their own ring of stages
// without waiting for anybody, and between two layers the CTAs of the cluster exchange their columns through L2, a release, an
// arrival at each other's barriers and an acquire: some 2500 cycles instead of a kernel boundary.
// Measured (us, separate launches -> here): 16 rows 1024-512-512-256-13 25 -> 16.5; 1024 rows 96-256-13 15 -> 8.7, and back
// 13 -> 8.2; 4096 rows 64-512-512-256-13 37 -> 21 each way.
// Sums run in the order of the separate kernels (gemm_tma.cu): same bits.
//
// Every wait is bounded: on a time-out the kernel records PPO_ERR_TIMEOUT, waits (bounded) for its copies, frees its
// tensor memory and returns.
#include "exchange.h"
#include "gemm.cuh"
#include "launch.cuh"
#include "tcgen05.cuh"
#include "tma_host.cuh"

namespace {

using namespace tc;

constexpr int kEpiWarps = 8;
constexpr int kThreads = (4 + kEpiWarps) * 32;  // warp 0: rows, 1: MMA issue and TMEM owner, 2: weights, 3: maps, 4 ..: epilogue
constexpr int kMaxStages = 16;
constexpr int kMaxSlice = 256;                  // columns of a layer a CTA can own
constexpr size_t kSmemMax = 227 * 1024;
constexpr int kCopy = 16 * 1024;                // bytes of a stage, except for slices of more than 128 columns
constexpr uint32_t kStage = 4096;               // staging of an epilogue warp: 32 rows x 128 bytes

struct Layer {
    CUtensorMap mapA, mapB;
    int chunks, rb;       // of the reduction, and bytes of a row of one
    int g;                // chunks of a stage (a copy brings them): more than one where the reduction is whole chunks
    int N, n;             // columns; of them in a CTA's slice
    int mode, ldo;
    const float *bias;
    bf16 *out;
    float *out_f32;
    const bf16 *mask;
};

struct Args {
    Layer l[kMlpLayers];
    int nl, rows, Mt;          // rows of a tile: 32, 64 or 128
    int sA, sB;                // stages
    uint32_t a_slot, b_slot;   // their bytes
    uint32_t tmem_cols;
    int32_t *status;
};

struct Pipe {
    uint64_t fullA[kMaxStages], emptyA[kMaxStages], fullB[kMaxStages], emptyB[kMaxStages], tfull;
    uint64_t ready[ChainExchange::barriers(kMlpLayers)];  // of the exchange behind each layer
    uint32_t tmem_slot;
    int abort_flag;
    alignas(16) float bias[kMlpLayers * kMaxSlice];
};

// Barrier of the epilogue that also ANDs a condition over it (a bounded wait that ran out in one warp ends all).
__device__ __forceinline__ bool epi_all(bool ok) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.b32 p, %1, 0;\n\t"
        "bar.red.and.pred q, 1, %2, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"(ok ? 1u : 0u), "n"(kEpiWarps * 32)
        : "memory");
    return r != 0;
}

__device__ __forceinline__ void drain(uint64_t *full, int it, int S) {
    for (int i = max(0, it - S); i < it; ++i) {
        const long long t0 = clock64();
        while (!mbar_try_wait(&full[i % S], (i / S) & 1))
            if (clock64() - t0 > kWaitCycles / 4) break;
    }
}

template <int CS>
__device__ __forceinline__ void chain(const Args &a, const MlpEnds &e, uint8_t *raw) {
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(raw) + 1023) & ~uintptr_t(1023));
    const uint32_t base = smem_u32(smem), b_base = base + (uint32_t)a.sA * a.a_slot;  // (an MMA's rows behind the last A stage lie in B's)
    const uint32_t stg_off = (uint32_t)a.sA * a.a_slot + (uint32_t)a.sB * a.b_slot;
    Pipe *pipe = reinterpret_cast<Pipe *>(smem + stg_off + kEpiWarps * kStage);
    volatile int *abort_flag = &pipe->abort_flag;
    const int warp = warp_index(), lane = threadIdx.x & 31;
    const int rank = (int)blockIdx.x % CS, row0 = (int)blockIdx.x / CS * a.Mt;

    if (threadIdx.x == 0) {
        for (int s = 0; s < a.sA; ++s) {
            mbar_init(&pipe->fullA[s], 1);
            mbar_init(&pipe->emptyA[s], 1);
        }
        for (int s = 0; s < a.sB; ++s) {
            mbar_init(&pipe->fullB[s], 1);
            mbar_init(&pipe->emptyB[s], 1);
        }
        mbar_init(&pipe->tfull, 1);
        for (int i = 0; i < ChainExchange::barriers(kMlpLayers); ++i) mbar_init(&pipe->ready[i], CS);
        pipe->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) tmem_alloc(&pipe->tmem_slot, a.tmem_cols);
    if (warp == 3 && lane < 2 * a.nl) {
        const CUtensorMap *m = lane & 1 ? &a.l[lane >> 1].mapB : &a.l[lane >> 1].mapA;
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(m)) : "memory");
    }
    __syncwarp();
    cluster_arrive();  // the barriers exist before anyone arrives at a neighbour's: all threads wait for it once, later
    grid_wait();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = pipe->tmem_slot;

    // (what a layer's loops need is taken out of the parameters before them: indexed by layer and read in the loop, they made a copy
    // cost 430 cycles and a chunk's MMAs 570)
    if (warp == 0) {
        int s = 0, it = 0;
        uint32_t ph = 0;
        bool ok = true;
        for (int l = 0; l < a.nl && ok; ++l) {
            const int chunks = a.l[l].chunks, rb = a.l[l].rb, g = a.l[l].g, N = a.l[l].N, n = a.l[l].n;
            const CUtensorMap *const map = &a.l[l].mapA;
            if (l > 0) {  // what the cluster has left for this layer
                ok = cluster_mbar_wait(&pipe->ready[ChainExchange::barrier(l - 1)], ChainExchange::parity(l - 1), abort_flag, a.status);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                fence_proxy_global();
            }
            if (rank * n >= N) continue;
            if (l == 0 && e.dout) {  // the epilogue fills the first stage
                it = s = 1;
                continue;
            }
            const uint32_t bytes = (uint32_t)(g * a.Mt * rb);
            for (int k = 0; k < chunks; k += g, ++it) {
                ok = mbar_wait_warp(&pipe->emptyA[s], ph ^ 1u, abort_flag, a.status);
                if (!ok) break;
                const int c0 = g > 1 ? 0 : k * (rb >> 1), c2 = g > 1 ? k : 0;
                if (elect_one()) {
                    mbar_arrive_expect_tx(&pipe->fullA[s], bytes);
                    tma_load_4d(base + (uint32_t)s * a.a_slot, map, &pipe->fullA[s], c0, row0, c2, 0);
                }
                __syncwarp();
                if (++s == a.sA) { s = 0; ph ^= 1u; }
            }
        }
        if (!ok && lane == 0) drain(pipe->fullA, it, a.sA);
        __syncwarp();
    } else if (warp == 2) {
        int s = 0, it = 0;
        uint32_t ph = 0;
        bool ok = true;
        for (int l = 0; l < a.nl && ok; ++l) {
            const int chunks = a.l[l].chunks, rb = a.l[l].rb, g = a.l[l].g, n = a.l[l].n, col0 = rank * n;
            const CUtensorMap *const map = &a.l[l].mapB;
            if (col0 >= a.l[l].N) continue;
            const uint32_t bytes = (uint32_t)(g * n * rb);
            for (int k = 0; k < chunks; k += g, ++it) {
                ok = mbar_wait_warp(&pipe->emptyB[s], ph ^ 1u, abort_flag, a.status);
                if (!ok) break;
                const int c0 = g > 1 ? 0 : k * (rb >> 1), c2 = g > 1 ? k : 0;
                if (elect_one()) {
                    mbar_arrive_expect_tx(&pipe->fullB[s], bytes);
                    tma_load_4d(b_base + (uint32_t)s * a.b_slot, map, &pipe->fullB[s], c0, col0, c2, 0);
                }
                __syncwarp();
                if (++s == a.sB) { s = 0; ph ^= 1u; }
            }
        }
        if (!ok && lane == 0) drain(pipe->fullB, it, a.sB);
        __syncwarp();
    } else if (warp == 1) {
        // the accumulator of the layer before has been read: the rows of this one wait for the cluster's arrivals, this CTA's
        // epilogue among them
        const int sA = a.sA, sB = a.sB;
        const uint32_t a_slot16 = a.a_slot >> 4, b_slot16 = a.b_slot >> 4;
        int sa = 0, sb = 0;
        uint32_t pa = 0, pb = 0;
        bool ok = true;
        for (int l = 0; l < a.nl && ok; ++l) {
            const int chunks = a.l[l].chunks, n = a.l[l].n, g = a.l[l].g;
            if (rank * n >= a.l[l].N) continue;
            const uint32_t rb = (uint32_t)a.l[l].rb, idesc = instr_desc(128, n, 0, 0);
            const uint64_t d0 = smem_desc_sw(base, 16, 8u * rb, rb);
            const uint32_t lo = (uint32_t)d0, hi = (uint32_t)(d0 >> 32), b_lo = lo + ((b_base - base) >> 4);
            const uint32_t a16 = (uint32_t)a.Mt * rb >> 4, b16 = (uint32_t)n * rb >> 4;
            const bool wide = rb == 128;
            uint32_t accum = 0;
            for (int k = 0; k < chunks; k += g) {
                ok = mbar_wait_warp(&pipe->fullB[sb], pb, abort_flag, a.status);
                if (!ok) break;
                ok = mbar_wait_warp(&pipe->fullA[sa], pa, abort_flag, a.status);
                if (!ok) break;
                tc_fence_after();
                const int nval = min(g, chunks - k);
                uint32_t la = lo + (uint32_t)sa * a_slot16, lb = b_lo + (uint32_t)sb * b_slot16;
                for (int c = 0; c < nval; ++c, la += a16, lb += b16) {
                    if (elect_one()) {
                        umma_bf16_lh(tmem, la, hi, lb, hi, idesc, accum);
                        if (wide) {
                            umma_bf16_lh(tmem, la + 2, hi, lb + 2, hi, idesc, 1u);
                            umma_bf16_lh(tmem, la + 4, hi, lb + 4, hi, idesc, 1u);
                            umma_bf16_lh(tmem, la + 6, hi, lb + 6, hi, idesc, 1u);
                        }
                    }
                    accum = 1u;
                }
                if (elect_one()) {
                    umma_commit(&pipe->emptyA[sa]);
                    umma_commit(&pipe->emptyB[sb]);
                }
                __syncwarp();
                if (++sa == sA) { sa = 0; pa ^= 1u; }
                if (++sb == sB) { sb = 0; pb ^= 1u; }
            }
            if (ok && elect_one()) umma_commit(&pipe->tfull);
            __syncwarp();
        }
    } else if (warp >= 4) {
        const int lg = warp & 3, half = (warp - 4) >> 2, et = (int)threadIdx.x - 128;
        const int grow = row0 + lg * 32 + lane;  // this thread's row: its tensor-memory lane
        uint4 *const stg = reinterpret_cast<uint4 *>(smem + stg_off + (uint32_t)(warp - 4) * kStage);
        const int rr0 = lane >> 2, piece = lane & 3, sw = (lane >> 1) & 3;
        const bool rows_here = lg * 32 < a.Mt;
        bool joined = false;  // waited for the cluster's start
        // Behind this CTA's stores: one release, an arrival at every CTA's barrier of the exchange behind layer l.
        auto publish = [&](bool ok, int l) -> bool {
            if (!epi_all(ok)) return false;
            if (!joined) cluster_wait();
            joined = true;
            if (warp == 4) {
                if (lane < CS) arrive_in_cta(&pipe->ready[ChainExchange::barrier(l)], (uint32_t)lane);
                __syncwarp();
            }
            return true;
        };
        {   // biases of all layers (a thread has at most one of each); the first use is behind a barrier
            float b[kMlpLayers];
#pragma unroll
            for (int l = 0; l < kMlpLayers; ++l)
                b[l] = l < a.nl && a.l[l].bias && et < a.l[l].n && rank * a.l[l].n + et < a.l[l].N ? __ldg(a.l[l].bias + rank * a.l[l].n + et) : 0.f;
#pragma unroll
            for (int l = 0; l < kMlpLayers; ++l) pipe->bias[l * kMaxSlice + et] = b[l];
            epi_all(true);
        }
        if (e.dout) {
            // The head's gradient as bf16: every CTA makes the tile's rows for itself, straight into the first stage (32-byte rows,
            // their two pieces swapped in every other four), and its share of them for the weight gradient.
            const int per = a.Mt / CS;
            for (int i = et; i < a.Mt * 2; i += kEpiWarps * 32) {
                const int row = i >> 1, p = i & 1, r = row0 + row;
                float v[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const int j = 8 * p + k;
                    v[k] = 0.f;
                    if (r < a.rows && j < e.A) v[k] = __ldg(e.dmean + (size_t)r * e.A + j);
                    else if (r < a.rows && j == e.A) v[k] = __ldg(e.dvalue + r);
                }
                const uint4 o = make_uint4(pack_bf16x2(v[0], v[1]), pack_bf16x2(v[2], v[3]), pack_bf16x2(v[4], v[5]), pack_bf16x2(v[6], v[7]));
                asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(base + (uint32_t)row * 32u + (((uint32_t)p ^ (((uint32_t)row >> 2) & 1u)) << 4)),
                             "r"(o.x), "r"(o.y), "r"(o.z), "r"(o.w)
                             : "memory");
                if (r < a.rows && row / per == rank) *reinterpret_cast<uint4 *>(e.dout + (size_t)r * 16 + 8 * p) = o;
            }
            fence_async_smem();
            epi_all(true);
            if (et == 0 && rank * a.l[0].n < a.l[0].N) mbar_arrive(&pipe->fullA[0]);
        }
        uint32_t tph = 0;
        for (int l = 0; l < a.nl; ++l) {
            const int N = a.l[l].N, n = a.l[l].n, mode = a.l[l].mode, ldo = a.l[l].ldo, col0 = rank * n;
            bf16 *const out = a.l[l].out;
            float *const out_f32 = a.l[l].out_f32;
            const bf16 *const mask = a.l[l].mask;
            bool ok = true;
            if (col0 < N && rows_here) {
                // 16 bytes of the gate for each of this lane's four stores of a group, fetched ahead (see gemm_tma.cu)
                uint4 gate[4];
                auto fetch = [&](int g) {
#pragma unroll
                    for (int ps = 0; ps < 4; ++ps) {
                        const int r = row0 + lg * 32 + ps * 8 + rr0, c = col0 + g + piece * 8;
                        gate[ps] = make_uint4(0, 0, 0, 0);
                        if (g < n && r < a.rows && g + piece * 8 < n && c < N)
                            gate[ps] = __ldg(reinterpret_cast<const uint4 *>(mask + (size_t)r * ldo + c));
                    }
                };
                if (mode == MLP_GATED) fetch(half * 32);
                ok = mbar_wait(&pipe->tfull, tph, abort_flag, a.status);
                ok = __all_sync(0xffffffffu, ok);
                tc_fence_after();
                const uint32_t tm = tmem + ((uint32_t)(lg * 32) << 16);
#pragma unroll 1
                for (int g = half * 32; ok && g < n; g += 64) {
                    float v[32] = {};
                    tmem_ld16(tm + (uint32_t)g, v);
                    if (g + 16 < n) tmem_ld16(tm + (uint32_t)g + 16u, v + 16);  // (else nothing made of those is stored)
                    if (mode == MLP_HEAD) {
                        if (grow < a.rows) {
#pragma unroll
                            for (int i = 0; i < 16; ++i) {
                                const int c = col0 + g + i;
                                v[i] += pipe->bias[l * kMaxSlice + g + i];
                                if (c < e.A) e.mean[(size_t)grow * e.A + c] = v[i];
                                else if (c == e.A) e.value[grow] = v[i];
                            }
                            if (e.eps && col0 + g == 0) {  // (at most 16 columns: they are all here)
                                float lp = 0.f;
#pragma unroll
                                for (int i = 0; i < 15; ++i)
                                    if (i < e.A) e.action[(size_t)grow * e.A + i] = sample_action(v[i], __ldg(e.logsigma + i), __ldg(e.eps + (size_t)grow * e.A + i), lp);
                                e.logp[grow] = lp;
                            }
                        }
                        continue;
                    }
                    if (mode == MLP_F32) {  // 32 rows x 128 bytes, 16-byte pieces swizzled by the row
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            stg[lane * 8 + (j ^ (lane & 7))] = make_uint4(__float_as_uint(v[4 * j]), __float_as_uint(v[4 * j + 1]),
                                                                          __float_as_uint(v[4 * j + 2]), __float_as_uint(v[4 * j + 3]));
                        __syncwarp();
#pragma unroll
                        for (int ps = 0; ps < 8; ++ps) {
                            const int rr = ps * 4 + (lane >> 3), p8 = lane & 7, r = row0 + lg * 32 + rr, c = col0 + g + p8 * 4;
                            if (r < a.rows && g + p8 * 4 < n && c < N)
                                *reinterpret_cast<uint4 *>(out_f32 + (size_t)r * ldo + c) = stg[rr * 8 + (p8 ^ (rr & 7))];
                        }
                        __syncwarp();
                        continue;
                    }
                    uint32_t pk[16];
                    if (mode == MLP_RELU) {
                        const float4 *bp = reinterpret_cast<const float4 *>(pipe->bias + l * kMaxSlice + g);
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            const float4 b = bp[q];
                            pk[2 * q] = relu_pack_bf16x2(v[4 * q] + b.x, v[4 * q + 1] + b.y);
                            pk[2 * q + 1] = relu_pack_bf16x2(v[4 * q + 2] + b.z, v[4 * q + 3] + b.w);
                        }
                    } else {
#pragma unroll
                        for (int j = 0; j < 16; ++j) pk[j] = pack_bf16x2(v[2 * j], v[2 * j + 1]);
                    }
#pragma unroll
                    for (int j = 0; j < 4; ++j) stg[lane * 4 + (j ^ sw)] = make_uint4(pk[4 * j], pk[4 * j + 1], pk[4 * j + 2], pk[4 * j + 3]);
                    __syncwarp();
#pragma unroll
                    for (int ps = 0; ps < 4; ++ps) {
                        const int rr = ps * 8 + rr0, r = row0 + lg * 32 + rr, c = col0 + g + piece * 8;
                        if (r < a.rows && g + piece * 8 < n && c < N) {
                            uint4 o = stg[rr * 4 + (piece ^ ((rr >> 1) & 3))];
                            if (mode == MLP_GATED) {
                                o.x &= gate_open(gate[ps].x); o.y &= gate_open(gate[ps].y);
                                o.z &= gate_open(gate[ps].z); o.w &= gate_open(gate[ps].w);
                            }
                            *reinterpret_cast<uint4 *>(out + (size_t)r * ldo + c) = o;
                        }
                    }
                    if (mode == MLP_GATED) fetch(g + 64);
                    __syncwarp();
                }
                tc_fence_before();
            }
            if (col0 < N) tph ^= 1u;
            if (l + 1 < a.nl && !publish(ok, l)) break;
        }
        __syncwarp();
        if (!joined) cluster_wait();
    }
    if (warp < 4) {
        __syncwarp();
        cluster_wait();
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();  // no CTA leaves while a neighbour may arrive at its barriers
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, a.tmem_cols);
    }
}

__global__ void __cluster_dims__(4, 1, 1) __launch_bounds__(kThreads, 1) mlp_chain4_kernel(const __grid_constant__ Args a, const __grid_constant__ MlpEnds e) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    chain<4>(a, e, smem_raw);
}
__global__ void __cluster_dims__(8, 1, 1) __launch_bounds__(kThreads, 1) mlp_chain8_kernel(const __grid_constant__ Args a, const __grid_constant__ MlpEnds e) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    chain<8>(a, e, smem_raw);
}

// CTAs per cluster and rows per tile, or false.  Clusters of eight cut the columns finer, but cudaOccupancyMaxActiveClusters gives 15
// of them on a B200's 148 SMs (33 of four); a second wave would cost as much as it saves.  Below that the smallest tile that still
// leaves one wave.  The two counts are the part's, not asked for in every call: where fewer fit, clusters run one after another.
bool shape(int rows, int &cs, int &Mt) {
    cs = 8;
    for (Mt = 32; Mt <= 128; Mt *= 2)
        if ((rows + Mt - 1) / Mt <= 15) return true;
    cs = 4;
    Mt = 128;
    return (rows + 127) / 128 <= 33;
}

}  // namespace

bool mlp_covers(const MlpLayer *layers, int nl, int rows) {
    int cs, Mt;
    if (nl < 1 || nl > kMlpLayers || rows < 1 || !shape(rows, cs, Mt)) return false;
    for (int i = 0; i < nl; ++i) {
        const MlpLayer &y = layers[i];
        const bool narrow = y.ldx == 16 && y.K <= 16;
        if (!narrow && (y.K < 64 || y.K % 8 != 0 || y.ldx % 8 != 0)) return false;
        if (y.ldw % 8 != 0 || (y.mode == MLP_HEAD ? y.N > 16 : y.N % 8 != 0)) return false;
        if ((y.N + cs - 1) / cs > kMaxSlice - 15) return false;
    }
    return true;
}

int mlp_chain(const MlpLayer *layers, int nl, int rows, const MlpEnds &ends, int32_t *status, cudaStream_t st) {
    if (!status || !mlp_covers(layers, nl, rows)) return PPO_ERR_UNSUPPORTED;
    Args a = {};
    int cs;
    shape(rows, cs, a.Mt);
    a.nl = nl;
    a.rows = rows;
    a.status = status;
    int n_max = 0;
    for (int i = 0; i < nl; ++i) {
        const MlpLayer &x = layers[i];
        Layer &y = a.l[i];
        const bool narrow = x.ldx == 16 && x.K <= 16;  // the head's gradient, rows padded to 16
        const int CB = narrow ? 16 : 64;
        y.rb = 2 * CB;
        y.chunks = (x.K + CB - 1) / CB;
        y.N = x.N;
        y.n = ((x.N + cs - 1) / cs + 15) / 16 * 16;
        y.mode = x.mode; y.ldo = x.ldo;
        y.bias = x.bias;
        y.out = x.out; y.out_f32 = x.out_f32; y.mask = x.mask;
        // a copy costs its warp some 150 cycles: chunks of a few KB go out several at a time
        const bool whole = x.K % CB == 0;
        y.g = whole ? kCopy / ((a.Mt > y.n ? a.Mt : y.n) * y.rb) : 1;
        y.g = y.g < 1 ? 1 : (y.g < y.chunks ? y.g : y.chunks);
        const long long da[4] = {y.g > 1 ? CB : (narrow ? 16 : x.K), rows, y.g > 1 ? y.chunks : 1, 1};
        const long long db[4] = {y.g > 1 ? CB : x.ldw, x.N, y.g > 1 ? y.chunks : 1, 1};
        const long long sa[3] = {2ll * x.ldx, 2ll * CB, 2ll * x.ldx * rows}, sb[3] = {2ll * x.ldw, 2ll * CB, 2ll * x.ldw * x.N};
        const int ba[4] = {CB, a.Mt, y.g, 1}, bb[4] = {CB, y.n, y.g, 1};
        PPO_TRY(make_map_strided(&y.mapA, x.X, 4, da, sa, ba));
        PPO_TRY(make_map_strided(&y.mapB, x.W, 4, db, sb, bb));
        n_max = y.n > n_max ? y.n : n_max;
    }
    a.tmem_cols = 32;
    while ((int)a.tmem_cols < n_max) a.tmem_cols *= 2;
    a.a_slot = kCopy;  // 128 rows of a chunk at most
    a.b_slot = n_max * 128 > kCopy ? (uint32_t)n_max * 128u : kCopy;
    const size_t room = kSmemMax - sizeof(Pipe) - kEpiWarps * kStage - 1024;
    a.sA = (int)((80 * 1024) / a.a_slot);
    if (a.sA > kMaxStages) a.sA = kMaxStages;
    a.sB = (int)((room - (size_t)a.sA * a.a_slot) / a.b_slot);
    if (a.sB > kMaxStages) a.sB = kMaxStages;
    if (a.sB < 2) return PPO_ERR_UNSUPPORTED;
    const size_t smem = (size_t)a.sA * a.a_slot + (size_t)a.sB * a.b_slot + kEpiWarps * kStage + sizeof(Pipe) + 1024;
    const auto fn = cs == 8 ? mlp_chain8_kernel : mlp_chain4_kernel;
    static PerDevice<bool> set[2];
    PPO_TRY(ppo_once_per_device(set[cs == 8], [&] { return ppo_allow_smem(fn, kSmemMax); }));
    return ppo_launch(fn, dim3((unsigned)((rows + a.Mt - 1) / a.Mt * cs)), dim3(kThreads), smem, st, a, ends);
}

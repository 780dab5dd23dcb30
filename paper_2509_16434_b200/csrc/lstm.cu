// The time loop of a recurrent layer as one persistent kernel per direction (sm_100a).
//
// A step's product with W_h is small (Be x 4H x H) and every step waits for the one before it: launch by launch the loop is
// a chain of 13 us GEMMs and 5 us cell kernels that mostly wait, for W_h from L2, for the pipeline to fill, for the
// launch.  Here a CTA keeps its slice of W_h in shared memory for all steps, the cell runs on the accumulator (forward) or
// between two exchanges (backward) with c and its gradient in registers, and the CTAs of a tile of 32, 64 or 128 envs exchange
// h (or the gate gradients) through global memory once per step, with counters for each group of four of them.  Backward's other
// exchange, the partial products of the four slabs of a reduction, goes by st.async into shared memory of the cluster the four
// form; through global memory only where tiles of 128 envs fit but not as clusters.  What a step costs (cycles of 16000, forward, 256 envs x 1024 units): 7300 for the 256 KB of h (or of one gate's gradients) a CTA
// pulls through L2 and their MMAs (all CTAs together take 11 TB/s), 700 + 2500 for the accumulator's way to the cell and the
// cell, 1250 until the release has seen its stores done, 2000 until the readers have seen it.
// The arithmetic is that of the step-by-step path, sum by sum: same bits.
//
// All CTAs of a launch have to be resident at once (cooperative launch, one CTA per SM); every wait is bounded: on a
// time-out the kernel records PPO_ERR_TIMEOUT, waits (bounded) for its copies and returns, and the last CTA to leave
// clears the counters whatever happened.
#include "gemm.cuh"
#include "launch.cuh"
#include "lstm.cuh"
#include "tcgen05.cuh"
#include "tma_host.cuh"

namespace {

using namespace tc;

constexpr int kCellWarps = 16;
constexpr int kThreads = (2 + kCellWarps) * 32;  // warp 0: TMA producer, warp 1: MMA issue and TMEM owner
constexpr int kMaxStages = 16;
constexpr uint32_t kBBytes = 64 * 128;  // weights of one 64-wide chunk of the reduction: 64 rows

// A tile is 32 U envs, U = 1, 2 or 4: a cell thread works on U units of one env, and 512 of them on 16 units of the tile.  Fewer
// envs per tile means more CTAs, each with less to pull, to compute and to write; the MMA takes 128 rows all the same, those
// behind the tile's read whatever lies there and nobody looks at their results.  The smallest tile whose CTAs all fit is
// taken (us per step, forward / backward; 119 envs x 512 units, tiles of 128 -> 32: 6.2 / 6.4 -> 4.3 / 4.4).
__host__ __device__ constexpr int tile_envs(int U) { return 32 * U; }
__host__ __device__ constexpr uint32_t a_bytes(int U) { return (uint32_t)tile_envs(U) * 128u; }  // envs of one chunk
__host__ __device__ constexpr uint32_t x_bytes(int U) { return (uint32_t)tile_envs(U) * 256u; }  // the accumulator on its way to other threads
constexpr size_t kSmemMax = 227 * 1024;

struct Args {
    CUtensorMap mapA;  // forward: h_prev [T * Be][H]; backward: gate gradients [T * Be][4H]
    CUtensorMap mapB;  // forward: W_h [4H][H], boxes of 16 rows; backward: W_h^T [H][4H], boxes of 64 rows
    int T, Be, H, per_tile, stages;  // per_tile: CTAs of a tile of envs
    const uint8_t *done;
    const float *xg, *bias, *h_init, *c_init;        // forward
    const float *dtop;                               // backward
    float *gates, *c, *cprev;
    bf16 *h, *hprev, *dg;
    float *dhc;
    unsigned int *counters;  // two rows of 32 per tile (see below); the first word behind them counts the CTAs that have left
    int32_t *status;
};

struct Pipe {
    uint64_t full[kMaxStages], empty[kMaxStages], tfull, wfull, parts;  // parts: the cluster's partial products
    uint32_t tmem_slot;
    int abort_flag;
};

__device__ __forceinline__ void cell_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kCellWarps * 32) : "memory"); }
__device__ __forceinline__ bool cell_all(bool ok) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.b32 p, %1, 0;\n\t"
        "bar.red.and.pred q, 1, %2, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"(ok ? 1u : 0u), "n"(kCellWarps * 32)
        : "memory");
    return r != 0;
}
// Counters of a tile of envs, a row of 32 for each exchange.  Word k of the first: CTAs that have published their 16 units of
// chunk k of the reduction (64 units, four CTAs a step); of the second (backward): slabs that have published their partial
// products of units 64 k .. 64 k + 63.  A reader waits for the four writers of what it reads next instead of for all the tile's
// CTAs, whose slowest is some 2000 of a step's 16000 cycles behind (256 envs x 1024 units), and one row is one line to poll.
__device__ __forceinline__ unsigned int *chunk_counters(const Args &a, int mt) { return a.counters + mt * 64; }
__device__ __forceinline__ unsigned int *part_counters(const Args &a, int mt) { return a.counters + mt * 64 + 32; }
// Arrival at a counter, by one thread behind a barrier of the threads whose writes it publishes.
__device__ __forceinline__ void tile_arrive(unsigned int *counter) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(counter) : "memory");
}
__device__ __forceinline__ unsigned int load_acquire(const unsigned int *p) {
    unsigned int v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
// Bounded wait until a counter has reached `target`.
__device__ bool tile_wait(const unsigned int *counter, unsigned int target, volatile int *abort_flag, int32_t *status) {
    const long long t0 = clock64();
    while (load_acquire(counter) < target) {
        if (*abort_flag) return false;
        if (clock64() - t0 > kWaitCycles) {
            *abort_flag = 1;
            ppo_report(status, PPO_ERR_TIMEOUT);
            return false;
        }
    }
    return true;
}

// U consecutive values, aligned to their size.
template <int U>
__device__ __forceinline__ void load_u(const float *p, float *v) {
    if constexpr (U == 4) {
        const float4 t = *reinterpret_cast<const float4 *>(p);
        v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
    } else if constexpr (U == 2) {
        const float2 t = *reinterpret_cast<const float2 *>(p);
        v[0] = t.x; v[1] = t.y;
    } else {
        v[0] = *p;
    }
}
template <int U>
__device__ __forceinline__ void store_u(float *p, const float *v) {
    if constexpr (U == 4) *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
    else if constexpr (U == 2) *reinterpret_cast<float2 *>(p) = make_float2(v[0], v[1]);
    else *p = v[0];
}
// The same as bf16, packed.
template <int U>
struct Packed;
template <>
struct Packed<4> { using T = uint2; };
template <>
struct Packed<2> { using T = uint32_t; };
template <>
struct Packed<1> { using T = uint16_t; };
template <int U>
__device__ __forceinline__ typename Packed<U>::T pack_u(const float *v) {
    if constexpr (U == 4) return make_uint2(pack_bf16x2(v[0], v[1]), pack_bf16x2(v[2], v[3]));
    else if constexpr (U == 2) return pack_bf16x2(v[0], v[1]);
    else return __bfloat16_as_ushort(__float2bfloat16_rn(v[0]));
}
template <int U>
__device__ __forceinline__ void store_bf16_u(bf16 *p, typename Packed<U>::T v) { *reinterpret_cast<typename Packed<U>::T *>(p) = v; }

template <int U>
__device__ __forceinline__ void lds_u(uint32_t addr, float *v) {
    if constexpr (U == 4) asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]) : "r"(addr) : "memory");
    else if constexpr (U == 2) asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v[0]), "=f"(v[1]) : "r"(addr) : "memory");
    else asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v[0]) : "r"(addr) : "memory");
}

// The exchange tile [envs][64 floats], 16 pieces of 16 bytes a row.  Tensor memory hands a thread a row; global memory
// wants neighbouring lanes on one row (a lane per row made every load and store of the cell 32 lines: 9000 cycles of a
// backward step went into the load-store unit, and polls of the counters queued behind them; 256 envs x 1024 units, 16 steps:
// forward 187 -> 154 us, backward 258 -> 184).  Piece p of row r sits at
// p ^ f(r), f running through eight values over eight rows with its high bit first: a row per lane on the way in, four or
// sixteen pieces of a row on neighbouring lanes on the way out, neither meets a bank twice.
__device__ __forceinline__ uint32_t xch_addr(uint32_t base, int row, int piece) {
    return base + (uint32_t)row * 256u + (((uint32_t)piece ^ (((uint32_t)row & 1u) << 2 | (((uint32_t)row >> 1) & 3u))) << 4);
}
// This warp's 16 accumulator columns into the tile.
__device__ __forceinline__ void xch_put(uint32_t base, uint32_t tmem, int lg, int lane, int grp) {
    float v[16];
    tmem_ld16(tmem + ((uint32_t)(lg * 32) << 16) + (uint32_t)(16 * grp), v);
    tc_fence_before();
#pragma unroll
    for (int j = 0; j < 4; ++j)
        asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(xch_addr(base, lg * 32 + lane, 4 * grp + j)), "f"(v[4 * j]),
                     "f"(v[4 * j + 1]), "f"(v[4 * j + 2]), "f"(v[4 * j + 3])
                     : "memory");
}
// Place of 16 bytes (piece 0 .. 3) of row `row` in slab `slab` of the partial products a CTA receives, [4][4 pieces][envs]: a
// warp that sends a piece of 32 rows fills 512 bytes on end, and four pieces of a row on neighbouring lanes do not meet a
// bank twice on the way out.
template <int U>
__device__ __forceinline__ uint32_t part_addr(uint32_t base, int slab, int row, int piece) {
    return base + (uint32_t)(slab * 4 + piece) * (uint32_t)(tile_envs(U) * 16) + (((uint32_t)row ^ ((uint32_t)piece << 1)) << 4);
}
// 16 bytes into another CTA's shared memory; its barrier counts them.
__device__ __forceinline__ void send16(uint32_t dst, uint32_t bar, const float *v) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(dst), "f"(v[0]),
                 "f"(v[1]), "f"(v[2]), "f"(v[3]), "r"(bar)
                 : "memory");
}
// Everything the two kernels share around the cell: barriers, tensor memory, the resident weight slice, the stream of A
// chunks and the MMAs.
struct Frame {
    Pipe *pipe;
    uint32_t smem_base, b_base, x_base, tmem;
    int warp, lane, mt, q, chunks, S;
};

template <int U>
__device__ __forceinline__ Frame frame_begin(const Args &a, uint8_t *raw) {
    Frame f;
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(raw) + 1023) & ~uintptr_t(1023));
    f.chunks = a.H >> 6;
    f.S = a.stages;
    f.smem_base = smem_u32(smem);
    f.b_base = f.smem_base + (uint32_t)f.S * a_bytes(U);  // (an MMA's rows behind the last stage's lie in the weights)
    f.x_base = f.b_base + (uint32_t)f.chunks * kBBytes;
    f.pipe = reinterpret_cast<Pipe *>(smem + (size_t)f.S * a_bytes(U) + (size_t)f.chunks * kBBytes + x_bytes(U));
    f.warp = warp_index();
    f.lane = threadIdx.x & 31;
    f.mt = (int)blockIdx.x / a.per_tile;
    f.q = (int)blockIdx.x - f.mt * a.per_tile;
    if (threadIdx.x == 0) {
        for (int s = 0; s < f.S; ++s) {
            mbar_init(&f.pipe->full[s], 1);
            mbar_init(&f.pipe->empty[s], 1);
        }
        mbar_init(&f.pipe->tfull, 1);
        mbar_init(&f.pipe->wfull, 1);
        mbar_init(&f.pipe->parts, 1);
        f.pipe->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (f.warp == 1) tmem_alloc(&f.pipe->tmem_slot, 64);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    f.tmem = f.pipe->tmem_slot;
    return f;
}

__device__ __forceinline__ void frame_end(const Args &a, const Frame &f) {
    tc_fence_before();
    __syncthreads();
    if (f.warp == 1) {
        tc_fence_after();
        tmem_dealloc(f.tmem, 64);
    }
    // the last CTA to leave clears the counters for the next launch
    const int words = (int)gridDim.x / a.per_tile * 64;
    if (threadIdx.x == 0) {
        __threadfence();
        f.pipe->tmem_slot = atomicAdd(a.counters + words, 1u) == gridDim.x - 1 ? 1u : 0u;
    }
    __syncthreads();
    if (f.pipe->tmem_slot)
        for (int i = threadIdx.x; i <= words; i += kThreads) a.counters[i] = 0u;
}

// Producer warp: the A chunks of one step (columns col0 .. col0 + H of the tile's rows from row0 on), each as soon as its four CTAs
// have published it `target / 4` times.  Lane k watches chunk k; the copies go out in order.
template <int U>
__device__ __forceinline__ bool produce_step(const Args &a, const Frame &f, unsigned int target, int col0, int row0, int &s, uint32_t &ph,
                                             int &it) {
    volatile int *abort_flag = &f.pipe->abort_flag;
    const unsigned int *mine = chunk_counters(a, f.mt) + f.lane;
    bool seen = f.lane >= f.chunks;
    uint32_t ready = 0;
    const long long t0 = clock64();
    for (int k = 0; k < f.chunks; ++k, ++it) {
        while (!((ready >> k) & 1u)) {
            if (!seen) seen = load_acquire(mine) >= target;
            ready = __ballot_sync(0xffffffffu, seen);
            if ((ready >> k) & 1u) {
                __syncwarp();  // a vote orders no memory: what lane k has acquired is passed on to the lane that issues the copy
                fence_proxy_global();
                break;
            }
            bool stop = false;
            if (f.lane == 0) {
                stop = *abort_flag != 0;
                if (!stop && clock64() - t0 > kWaitCycles) {
                    *abort_flag = 1;
                    ppo_report(a.status, PPO_ERR_TIMEOUT);
                    stop = true;
                }
            }
            if (__any_sync(0xffffffffu, stop)) return false;
        }
        if (!mbar_wait_warp(&f.pipe->empty[s], ph ^ 1u, abort_flag, a.status)) return false;
        if (elect_one()) {
            mbar_arrive_expect_tx(&f.pipe->full[s], a_bytes(U));
            tma_load_2d(f.smem_base + (uint32_t)s * a_bytes(U), &a.mapA, &f.pipe->full[s], col0 + k * 64, row0);
        }
        __syncwarp();
        if (++s == f.S) { s = 0; ph ^= 1u; }
    }
    return true;
}
__device__ __forceinline__ void drain(const Frame &f, int it) {
    for (int i = max(0, it - f.S); i < it; ++i) {
        const long long t0 = clock64();
        while (!mbar_try_wait(&f.pipe->full[i % f.S], (i / f.S) & 1))
            if (clock64() - t0 > kWaitCycles / 4) break;
    }
}

// MMAs of one step into the 64 accumulator columns (warp 1).
template <int U>
__device__ __forceinline__ bool mma_step(const Args &a, const Frame &f, int &s, uint32_t &ph) {
    constexpr uint32_t idesc = instr_desc(128, 64, 0, 0);
    const uint64_t d0 = smem_desc_sw(f.smem_base, 16, 1024, 128);
    const uint32_t lo = (uint32_t)d0, hi = (uint32_t)(d0 >> 32), b_lo = lo + ((f.b_base - f.smem_base) >> 4);
    for (int k = 0; k < f.chunks; ++k) {
        if (!mbar_wait_warp(&f.pipe->full[s], ph, &f.pipe->abort_flag, a.status)) return false;
        tc_fence_after();
        if (elect_one()) {
            const uint32_t la = lo + (uint32_t)s * (a_bytes(U) >> 4), lb = b_lo + (uint32_t)k * (kBBytes >> 4);
            umma_bf16_lh(f.tmem, la, hi, lb, hi, idesc, k > 0 ? 1u : 0u);
#pragma unroll
            for (int j = 1; j < 4; ++j) umma_bf16_lh(f.tmem, la + 2 * j, hi, lb + 2 * j, hi, idesc, 1u);
            umma_commit(&f.pipe->empty[s]);
        }
        __syncwarp();
        if (++s == f.S) { s = 0; ph ^= 1u; }
    }
    if (elect_one()) umma_commit(&f.pipe->tfull);
    __syncwarp();
    return true;
}

// Forward over all steps of one layer.  CTA q of a tile owns units 16 q .. 16 q + 15: accumulator column 16 g + j is gate g
// of unit 16 q + j.
template <int U>
__global__ void __launch_bounds__(kThreads, 1) lstm_fwd_kernel(const __grid_constant__ Args a) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const Frame f = frame_begin<U>(a, smem_raw);
    unsigned int *counter = chunk_counters(a, f.mt) + (f.q >> 2);  // of this CTA's units
    const int H = a.H, u0 = f.q * 16, row0 = f.mt * tile_envs(U);
    volatile int *abort_flag = &f.pipe->abort_flag;
    if (f.warp == 0) {
        if (f.lane == 0) {
            mbar_arrive_expect_tx(&f.pipe->wfull, (uint32_t)f.chunks * kBBytes);
            for (int k = 0; k < f.chunks; ++k)
                for (int g = 0; g < 4; ++g)
                    tma_load_2d(f.b_base + (uint32_t)k * kBBytes + (uint32_t)g * 2048u, &a.mapB, &f.pipe->wfull, k * 64, g * H + u0);
        }
        __syncwarp();
        int s = 0, it = 0;
        uint32_t ph = 0;
        bool ok = true;
        for (int t = 0; t < a.T && ok; ++t) ok = produce_step<U>(a, f, 4u * (unsigned)(t + 1), 0, t * a.Be + row0, s, ph, it);
        if (!ok && f.lane == 0) drain(f, it);
        __syncwarp();
    } else if (f.warp == 1) {
        int s = 0;
        uint32_t ph = 0;
        bool ok = mbar_wait_warp(&f.pipe->wfull, 0, abort_flag, a.status);
        for (int t = 0; t < a.T && ok; ++t) ok = mma_step<U>(a, f, s, ph);
    } else {
        // thread of the cell: env `row` of the tile, units j0 .. j0 + U - 1, columns col .. of each gate's 16
        const int lg = f.warp & 3, grp = (f.warp - 2) >> 2, ct = (int)threadIdx.x - 64, row = ct * U >> 4, col = ct * U & 15, e = row0 + row;
        const bool live = e < a.Be, issuer = ct == 0;
        const int j0 = u0 + col;
        float cp[U], bias[4][U];
#pragma unroll
        for (int k = 0; k < U; ++k) cp[k] = 0.f;
#pragma unroll
        for (int g = 0; g < 4; ++g) load_u<U>(a.bias + g * H + j0, bias[g]);
        if (live) {  // the state the first step starts from
            const size_t i = (size_t)e * H + j0;
            float hv[U];
            load_u<U>(a.h_init + i, hv);
            load_u<U>(a.c_init + i, cp);
            store_bf16_u<U>(a.hprev + i, pack_u<U>(hv));
            store_u<U>(a.cprev + i, cp);
        }
        cell_sync();
        if (issuer) tile_arrive(counter);
        for (int t = 0; t < a.T; ++t) {
            const size_t r = (size_t)t * a.Be + e;
            float xg[4][U];
            bool reset = false;
            if (live) {  // ahead of the wait: they do not depend on this step's product
#pragma unroll
                for (int g = 0; g < 4; ++g) load_u<U>(a.xg + r * 4 * H + g * H + j0, xg[g]);
                reset = a.done[r] != 0;
            }
            const bool ok = mbar_wait(&f.pipe->tfull, t & 1, abort_flag, a.status);
            tc_fence_after();
            if (lg * 32 < tile_envs(U) && __all_sync(0xffffffffu, ok)) xch_put(f.x_base, f.tmem, lg, f.lane, grp);  // gate `grp` of the 16 units
            if (!cell_all(ok)) break;
            float gi[U], gf[U], gg[U], go[U], cv[U];
            typename Packed<U>::T hb = {};
            if (live) {
                float hg[4][U], hv[U];
#pragma unroll
                for (int g = 0; g < 4; ++g) lds_u<U>(xch_addr(f.x_base, row, 4 * g + (col >> 2)) + 4u * (col & 3), hg[g]);
#pragma unroll
                for (int k = 0; k < U; ++k) {
                    lstm_cell(xg[0][k] + hg[0][k] + bias[0][k], xg[1][k] + hg[1][k] + bias[1][k], xg[2][k] + hg[2][k] + bias[2][k],
                              xg[3][k] + hg[3][k] + bias[3][k], cp[k], gi[k], gf[k], gg[k], go[k], cv[k], hv[k]);
                }
                hb = pack_u<U>(hv);
                if (t + 1 < a.T) store_bf16_u<U>(a.hprev + (r + a.Be) * H + j0, reset ? typename Packed<U>::T{} : hb);
            }
            if (t + 1 < a.T) {  // what the others wait for goes first, the rest behind it
                cell_sync();
                if (issuer) tile_arrive(counter);
            }
            if (live) {
                store_bf16_u<U>(a.h + r * H + j0, hb);
                float *gp = a.gates + r * 4 * H + j0;
                store_u<U>(gp, gi);
                store_u<U>(gp + H, gf);
                store_u<U>(gp + 2 * H, gg);
                store_u<U>(gp + 3 * H, go);
                store_u<U>(a.c + r * H + j0, cv);
#pragma unroll
                for (int k = 0; k < U; ++k) cp[k] = reset ? 0.f : cv[k];
                if (t + 1 < a.T) store_u<U>(a.cprev + (r + a.Be) * H + j0, cp);
            }
        }
    }
    frame_end(a, f);
}

// Back-propagation through all steps of one layer: gate gradients dg of every step.  The product dg W_h of a step reduces
// over 4 H columns in four slabs (one gate each) whose partial products are added in order: CTA q = (64 units, slab) forms
// one, and as a cell it works on units 16 q .. 16 q + 15, a quarter of the same 64.
// CLUSTER: the four slabs of a slice are a cluster and send one another their partial products from the accumulator
// straight into shared memory, data and signal in one; the way through global memory (store, release, poll, load) takes 9000
// of a step's 20000 cycles, and so does shared memory that the others read behind a release (a release waits for all its
// thread's block has under way).  A place is free again when the next product arrives: that needs gate gradients of all the
// tile's cells, who had read it by then.
template <int U, bool CLUSTER>
__device__ __forceinline__ void bwd_steps(const Args &a, uint8_t *smem_raw) {
    const Frame f = frame_begin<U>(a, smem_raw);
    const int H = a.H, row0 = f.mt * tile_envs(U), slab = f.q & 3, slice = f.q >> 2, n0 = slice * 64;
    unsigned int *const cells = chunk_counters(a, f.mt) + slice;  // of this CTA's units as a cell
    unsigned int *const parts = part_counters(a, f.mt) + slice;
    volatile int *abort_flag = &f.pipe->abort_flag;
    if (f.warp == 0) {
        if (f.lane == 0) {
            mbar_arrive_expect_tx(&f.pipe->wfull, (uint32_t)f.chunks * kBBytes);
            for (int k = 0; k < f.chunks; ++k)
                tma_load_2d(f.b_base + (uint32_t)k * kBBytes, &a.mapB, &f.pipe->wfull, slab * H + k * 64, n0);
        }
        __syncwarp();
        int s = 0, it = 0;
        uint32_t ph = 0;
        bool ok = true;
        for (int t = a.T - 1, i = 0; t > 0 && ok; --t, ++i) ok = produce_step<U>(a, f, 4u * (unsigned)(i + 1), slab * H, t * a.Be + row0, s, ph, it);
        if (!ok && f.lane == 0) drain(f, it);
        __syncwarp();
    } else if (f.warp == 1) {
        int s = 0;
        uint32_t ph = 0;
        bool ok = mbar_wait_warp(&f.pipe->wfull, 0, abort_flag, a.status);
        for (int t = a.T - 1; t > 0 && ok; --t) ok = mma_step<U>(a, f, s, ph);
    } else {
        // as a cell: env `row` of the tile, units j0 .. j0 + U - 1, columns col .. of the CTA's 16
        const int lg = f.warp & 3, grp = (f.warp - 2) >> 2, ct = (int)threadIdx.x - 64, row = ct * U >> 4, col = ct * U & 15, e = row0 + row;
        const bool live = e < a.Be, issuer = ct == 0;
        const int j0 = f.q * 16 + col;
        const size_t step = (size_t)a.Be * H;
        float dcc[U], dtop[U], g4[4][U], cv[U], cp[U];
#pragma unroll
        for (int k = 0; k < U; ++k) dcc[k] = 0.f;
        uint8_t done = 0;
        // What the forward pass left for step t.  It comes from HBM in a burst of 57 KB per CTA (7 MB in all: 3500 cycles), so it is
        // asked for while the step before multiplies.
        auto fetch = [&](int t) {
            if (!live) return;
            const size_t r = (size_t)t * a.Be + e;
            load_u<U>(a.dtop + r * H + j0, dtop);
#pragma unroll
            for (int g = 0; g < 4; ++g) load_u<U>(a.gates + r * 4 * H + g * H + j0, g4[g]);
            load_u<U>(a.c + r * H + j0, cv);
            load_u<U>(a.cprev + r * H + j0, cp);
            done = a.done[r];
        };
        fetch(a.T - 1);
        for (int t = a.T - 1, i = 0; t >= 0; --t, ++i) {
            const size_t r = (size_t)t * a.Be + e;
            const bool last = t == a.T - 1, carry = !last && done == 0;
            if (!last) {  // the partial products of the step after this one (their four writers had seen all cells of that step, so
                          // the places of the step before were free)
                bool ok = true;
                if (CLUSTER) ok = cluster_mbar_wait(&f.pipe->parts, (uint32_t)(i - 1) & 1u, abort_flag, a.status);
                else if (issuer) ok = tile_wait(parts, 4u * (unsigned)i, abort_flag, a.status);
                if (!cell_all(ok)) break;
            }
            if (live) {
                float dhn[U];
#pragma unroll
                for (int k = 0; k < U; ++k) dhn[k] = 0.f;
                if (carry) {
                    float p[4][U];
#pragma unroll
                    for (int s = 0; s < 4; ++s) {
                        if constexpr (CLUSTER) {
                            lds_u<U>(part_addr<U>(f.x_base, s, row, col >> 2) + 4u * (col & 3), p[s]);
                        } else {  // written by other CTAs of this launch
                            const float4 v = __ldcg(reinterpret_cast<const float4 *>(a.dhc + s * step + (size_t)e * H + j0));
                            p[s][0] = v.x; p[s][1] = v.y; p[s][2] = v.z; p[s][3] = v.w;
                        }
                    }
#pragma unroll
                    for (int s = 0; s < 4; ++s)
#pragma unroll
                        for (int k = 0; k < U; ++k) dhn[k] += p[s][k];
                }
                float di[U], df[U], dgg[U], dgo[U];
#pragma unroll
                for (int k = 0; k < U; ++k)
                    lstm_cell_back(dtop[k] + dhn[k], carry ? dcc[k] : 0.f, g4[0][k], g4[1][k], g4[2][k], g4[3][k], cv[k], cp[k], di[k],
                                   df[k], dgg[k], dgo[k], dcc[k]);
                bf16 *o = a.dg + r * 4 * H + j0;
                store_bf16_u<U>(o, pack_u<U>(di));
                store_bf16_u<U>(o + H, pack_u<U>(df));
                store_bf16_u<U>(o + 2 * H, pack_u<U>(dgg));
                store_bf16_u<U>(o + 3 * H, pack_u<U>(dgo));
            }
            if (t == 0) break;
            cell_sync();
            if (issuer) {
                if (CLUSTER) mbar_arrive_expect_tx(&f.pipe->parts, x_bytes(U));  // what the four CTAs will send for this step
                tile_arrive(cells);
            }
            fetch(t - 1);
            // this CTA's partial product, 64 columns a row: columns 16 k .. 16 k + 15 are what cell k of the slice needs
            const bool ok = mbar_wait(&f.pipe->tfull, i & 1, abort_flag, a.status);
            tc_fence_after();
            if constexpr (CLUSTER) {
                if (lg * 32 < tile_envs(U) && __all_sync(0xffffffffu, ok)) {  // (else the abort flag ends all warps at the next wait for the parts)
                    float v[16];
                    tmem_ld16(f.tmem + ((uint32_t)(lg * 32) << 16) + (uint32_t)(16 * grp), v);
                    tc_fence_before();
                    const uint32_t bar = in_cta(smem_u32(&f.pipe->parts), (uint32_t)grp);
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        send16(in_cta(part_addr<U>(f.x_base, slab, lg * 32 + f.lane, k), (uint32_t)grp), bar, v + 4 * k);
                }
                continue;
            }
            static_assert(CLUSTER || U == 4, "the way through global memory is written for tiles of 128 envs");
            if (__all_sync(0xffffffffu, ok)) xch_put(f.x_base, f.tmem, lg, f.lane, grp);
            if (!cell_all(ok)) break;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int rr = k * 32 + (ct >> 4), piece = ct & 15;
                if (row0 + rr >= a.Be) continue;
                float v[4];
                lds_u<4>(xch_addr(f.x_base, rr, piece), v);
                __stcg(reinterpret_cast<float4 *>(a.dhc + slab * step + (size_t)(row0 + rr) * H + n0) + piece, make_float4(v[0], v[1], v[2], v[3]));
            }
            cell_sync();
            if (issuer) tile_arrive(parts);
        }
    }
    if (CLUSTER) {  // no CTA leaves while another may write to its shared memory
        if (*abort_flag) {  // (sends of a step that was given up land meanwhile; a finished step has waited for its own)
            const long long t0 = clock64();
            while (clock64() - t0 < 100000) {
            }
        }
        __syncwarp();
        cluster_sync();
    }
    frame_end(a, f);
}

__global__ void __launch_bounds__(kThreads, 1) lstm_bwd_kernel(const __grid_constant__ Args a) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    bwd_steps<4, false>(a, smem_raw);
}
template <int U>
__global__ void __cluster_dims__(4, 1, 1) __launch_bounds__(kThreads, 1) lstm_bwd_cluster_kernel(const __grid_constant__ Args a) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    bwd_steps<U, true>(a, smem_raw);
}

// ---- one step: acting ----

// A sequence of one step has nothing to keep resident and nobody to exchange with: x W_x^T and h W_h^T of M envs and U units
// (4 U columns, gate g of unit j at g U + j) run through one pipeline into two accumulators, and the cell works on their sum.
// Separate launches for W_x x and the step had each its own pipeline to fill, and 512 envs x 1024 units, too many for the
// time loop, took four of them.  What bounds it: the bytes a CTA pulls through L2 (M + 4 U rows of every chunk).
// Measured (us per layer): 16 envs x 1024 units 16.7 -> 7.7; 512 envs x 1024 units 32 -> 19.
struct StepArgs {
    CUtensorMap mapX, mapH, mapWx, mapWh;
    int Be, H;
    int chunksX, gX, chunksH, gH;  // chunks of the two reductions, and of them in a copy
    int stages;
    const float *bias, *cprev;
    float *gates, *c;
    bf16 *h;
    int32_t *status;
};
constexpr int kStepG = 2;  // chunks of a stage

template <int M, int U>
__global__ void __launch_bounds__(kThreads, 1) lstm_step_kernel(const __grid_constant__ StepArgs a, const __grid_constant__ LstmStepEnds ends) {
    constexpr uint32_t kA = M * 128u, kB = 4u * U * 128u, kStageBytes = kStepG * (kA + kB);
    constexpr int W = M * U >= 2048 ? 4 : (M * U >= 1024 ? 2 : 1);  // units of a thread in a pass over the cells
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int S = a.stages, H = a.H;
    const uint32_t base = smem_u32(smem), x_base = base + (uint32_t)S * kStageBytes;  // (an MMA's rows behind M lie in what follows)
    Pipe *pipe = reinterpret_cast<Pipe *>(smem + (size_t)S * kStageBytes + (size_t)M * U * 16);
    volatile int *abort_flag = &pipe->abort_flag;
    const int warp = warp_index(), lane = threadIdx.x & 31;
    const int slices = H / U, mt = (int)blockIdx.x / slices, u0 = ((int)blockIdx.x - mt * slices) * U, row0 = mt * M;
    constexpr uint32_t ncols = 8 * U < 32 ? 32 : 8 * U;
    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(&pipe->full[s], 1);
            mbar_init(&pipe->empty[s], 1);
        }
        mbar_init(&pipe->tfull, 1);
        pipe->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) tmem_alloc(&pipe->tmem_slot, ncols);
    grid_wait();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = pipe->tmem_slot;

    if (warp == 0) {
        int s = 0, it = 0;
        uint32_t ph = 0;
        bool ok = true;
        for (int part = 0; part < 2 && ok; ++part) {
            const int chunks = part ? a.chunksH : a.chunksX, g = part ? a.gH : a.gX;
            const CUtensorMap *const ma = part ? &a.mapH : &a.mapX, *const mb = part ? &a.mapWh : &a.mapWx;
            for (int k = 0; k < chunks; k += g, ++it) {
                ok = mbar_wait_warp(&pipe->empty[s], ph ^ 1u, abort_flag, a.status);
                if (!ok) break;
                const uint32_t dst = base + (uint32_t)s * kStageBytes;
                const int c0 = g > 1 ? 0 : k * 64, ck = g > 1 ? k : 0;
                if (elect_one()) {
                    mbar_arrive_expect_tx(&pipe->full[s], (uint32_t)g * (kA + kB));
                    tma_load_4d(dst, ma, &pipe->full[s], c0, row0, ck, 0);
                    tma_load_4d(dst + kStepG * kA, mb, &pipe->full[s], c0, u0, 0, ck);
                }
                __syncwarp();
                if (++s == S) { s = 0; ph ^= 1u; }
            }
        }
        if (!ok && lane == 0)
            for (int i = max(0, it - S); i < it; ++i) {
                const long long t0 = clock64();
                while (!mbar_try_wait(&pipe->full[i % S], (i / S) & 1))
                    if (clock64() - t0 > kWaitCycles / 4) break;
            }
        __syncwarp();
    } else if (warp == 1) {
        constexpr uint32_t idesc = instr_desc(128, 4 * U, 0, 0);
        const uint64_t d0 = smem_desc_sw(base, 16, 1024, 128);
        const uint32_t lo = (uint32_t)d0, hi = (uint32_t)(d0 >> 32);
        int s = 0;
        uint32_t ph = 0;
        bool ok = true;
        for (int part = 0; part < 2 && ok; ++part) {
            const int chunks = part ? a.chunksH : a.chunksX, g = part ? a.gH : a.gX;
            const uint32_t td = tmem + (part ? 4u * U : 0u);
            uint32_t accum = 0;
            for (int k = 0; k < chunks; k += g) {
                ok = mbar_wait_warp(&pipe->full[s], ph, abort_flag, a.status);
                if (!ok) break;
                tc_fence_after();
                const int nval = min(g, chunks - k);
                uint32_t la = lo + (uint32_t)s * (kStageBytes >> 4), lb = la + (kStepG * kA >> 4);
                for (int c = 0; c < nval; ++c, la += kA >> 4, lb += kB >> 4) {
                    if (elect_one()) {
                        umma_bf16_lh(td, la, hi, lb, hi, idesc, accum);
                        umma_bf16_lh(td, la + 2, hi, lb + 2, hi, idesc, 1u);
                        umma_bf16_lh(td, la + 4, hi, lb + 4, hi, idesc, 1u);
                        umma_bf16_lh(td, la + 6, hi, lb + 6, hi, idesc, 1u);
                    }
                    accum = 1u;
                }
                if (elect_one()) umma_commit(&pipe->empty[s]);
                __syncwarp();
                if (++s == S) { s = 0; ph ^= 1u; }
            }
        }
        if (ok && elect_one()) umma_commit(&pipe->tfull);
        __syncwarp();
    } else {
        const int lg = warp & 3, grp = (warp - 2) >> 2, ct = (int)threadIdx.x - 64;
        auto place = [&](int row, int col) {  // of a float of the exchange tile [M][4 U] (see xch_addr)
            return x_base + (uint32_t)row * (16u * U) +
                   ((((uint32_t)col >> 2) ^ (((uint32_t)row & 1u) << 2 | (((uint32_t)row >> 1) & 3u))) << 4) + 4u * ((uint32_t)col & 3u);
        };
        const bool ok = mbar_wait(&pipe->tfull, 0, abort_flag, a.status);
        tc_fence_after();
        if (lg * 32 < M && __all_sync(0xffffffffu, ok)) {
            const uint32_t tm = tmem + ((uint32_t)(lg * 32) << 16);
#pragma unroll
            for (int b = grp; b < U / 4; b += 4) {
                float x[16], h[16];
                tmem_ld16(tm + 16u * b, x);
                tmem_ld16(tm + 4u * U + 16u * b, h);
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(place(lg * 32 + lane, 16 * b + 4 * j)), "f"(x[4 * j] + h[4 * j]),
                                 "f"(x[4 * j + 1] + h[4 * j + 1]), "f"(x[4 * j + 2] + h[4 * j + 2]), "f"(x[4 * j + 3] + h[4 * j + 3])
                                 : "memory");
            }
            tc_fence_before();
        }
        if (cell_all(ok)) {
#pragma unroll 1
            for (int i = ct * W; i < M * U; i += kCellWarps * 32 * W) {
                const int row = i / U, col = i - row * U, e = row0 + row, j = u0 + col;
                if (e >= a.Be) break;
                const size_t r = (size_t)e * H + j, r4 = (size_t)e * 4 * H + j;
                float p[4][W], b[4][W], cp[W], gi[W], gf[W], gg[W], go[W], cv[W], hv[W];
                load_u<W>(a.cprev + r, cp);
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    load_u<W>(a.bias + g * H + j, b[g]);
                    lds_u<W>(place(row, g * U + col), p[g]);
                }
#pragma unroll
                for (int k = 0; k < W; ++k)
                    lstm_cell(p[0][k] + b[0][k], p[1][k] + b[1][k], p[2][k] + b[2][k], p[3][k] + b[3][k], cp[k], gi[k], gf[k], gg[k], go[k], cv[k], hv[k]);
                store_u<W>(a.gates + r4, gi);
                store_u<W>(a.gates + r4 + H, gf);
                store_u<W>(a.gates + r4 + 2 * H, gg);
                store_u<W>(a.gates + r4 + 3 * H, go);
                store_u<W>(a.c + r, cv);
                store_bf16_u<W>(a.h + r, pack_u<W>(hv));
                if (ends.h_out) {
                    const bool reset = ends.done[e] != 0;
#pragma unroll
                    for (int k = 0; k < W; ++k) {
                        hv[k] = reset ? 0.f : bf2f(__float2bfloat16_rn(hv[k]));
                        cv[k] = reset ? 0.f : cv[k];
                    }
                    store_u<W>(ends.h_out + r, hv);
                    store_u<W>(ends.c_out + r, cv);
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, ncols);
    }
}

// Shape part for tiles of 32 U envs; false where the layer or the sequence does not fit: a slice of W_h has to leave room for
// the exchange and two chunks of A (four of 128 envs at H = 1024), and all CTAs have to be resident at once.
bool plan(Args &a, int T, int Be, int H, int U, int &ctas, size_t &smem) {
    if (H % 64 != 0 || H > 2048 || T < 1 || Be < 1) return false;
    a.T = T; a.Be = Be; a.H = H;
    a.per_tile = H / 16;
    const long long tiles = (Be + tile_envs(U) - 1) / tile_envs(U), n = tiles * a.per_tile;
    if (n > ppo_num_sms() || 2 * tiles + 1 > kLstmCounters) return false;
    const size_t fixed = (size_t)(H / 64) * kBBytes + x_bytes(U) + sizeof(Pipe) + 1024;
    if (fixed + 2 * a_bytes(U) > kSmemMax) return false;
    a.stages = (int)((kSmemMax - fixed) / a_bytes(U));
    if (a.stages > kMaxStages) a.stages = kMaxStages;
    smem = fixed + (size_t)a.stages * a_bytes(U);
    ctas = (int)n;
    return true;
}

template <int M, int U>
int launch_step(StepArgs &a, int in, const LstmSteps &p, const bf16 *X, const bf16 *Wx, const bf16 *Wh, const LstmStepEnds &ends, cudaStream_t st) {
    const long long H = p.H, Be = p.Be;
    auto maps = [&](CUtensorMap &ma, CUtensorMap &mb, const bf16 *A, const bf16 *B, int K, int &chunks, int &g) -> int {
        chunks = (K + 63) / 64;
        g = K % 64 == 0 && chunks > 1 ? kStepG : 1;
        const bool many = g > 1;
        const long long da[4] = {many ? 64 : K, Be, many ? chunks : 1, 1}, sa[3] = {2ll * K, 128, 2ll * K * Be};
        const long long db[4] = {many ? 64 : K, H, 4, many ? chunks : 1}, sb[3] = {2ll * K, 2ll * K * H, 128};
        const int ba[4] = {64, M, g, 1}, bb[4] = {64, U, 4, g};
        PPO_TRY(make_map_strided(&ma, A, 4, da, sa, ba));
        return make_map_strided(&mb, B, 4, db, sb, bb);
    };
    PPO_TRY(maps(a.mapX, a.mapWx, X, Wx, in, a.chunksX, a.gX));
    PPO_TRY(maps(a.mapH, a.mapWh, p.hprev, Wh, (int)H, a.chunksH, a.gH));
    const size_t stage = (size_t)kStepG * (M + 4 * U) * 128, fixed = (size_t)M * U * 16 + sizeof(Pipe) + 1024;
    a.stages = (int)((kSmemMax - fixed) / stage);
    if (a.stages > kMaxStages) a.stages = kMaxStages;
    static PerDevice<bool> set;
    PPO_TRY(ppo_once_per_device(set, [] { return ppo_allow_smem(lstm_step_kernel<M, U>, kSmemMax); }));
    const unsigned ctas = (unsigned)((Be + M - 1) / M * (H / U));
    return ppo_launch(lstm_step_kernel<M, U>, dim3(ctas), dim3(kThreads), (size_t)a.stages * stage + fixed, st, a, ends);
}

// Whether `ctas` CTAs in clusters of four are resident at once: clusters fit the groups of SMs less tightly than single CTAs (33
// of them on 148 SMs).
template <typename F>
int clusters_fit(F *fn, int ctas, size_t smem, bool &fit) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ctas);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = 4;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    int clusters = 0;
    PPO_CUDA_CHECK(cudaOccupancyMaxActiveClusters(&clusters, fn, &cfg));
    fit = 4ll * clusters >= ctas;
    return PPO_OK;
}

template <int U>
int launch_fwd(Args &a, const LstmSteps &p, int ctas, size_t smem, cudaStream_t st) {
    const long long H = p.H, rows = (long long)p.T * p.Be;
    const long long da[2] = {H, rows}, sa[1] = {2 * H};
    const int ba[2] = {64, tile_envs(U)};
    PPO_TRY(make_map_strided(&a.mapA, p.hprev, 2, da, sa, ba));
    static PerDevice<bool> set;
    PPO_TRY(ppo_once_per_device(set, [] { return ppo_allow_smem(lstm_fwd_kernel<U>, kSmemMax); }));
    return ppo_launch_together(lstm_fwd_kernel<U>, dim3(ctas), dim3(kThreads), smem, st, a);
}

int map_dg(Args &a, const LstmSteps &p, bf16 *dg, int envs) {
    const long long H = p.H, rows = (long long)p.T * p.Be;
    const long long da[2] = {4 * H, rows}, sa[1] = {8 * H};
    const int ba[2] = {64, envs};
    return make_map_strided(&a.mapA, dg, 2, da, sa, ba);
}

// PPO_ERR_UNSUPPORTED where the tiles' clusters do not all fit.
template <int U>
int launch_bwd_clusters(Args &a, const LstmSteps &p, bf16 *dg, cudaStream_t st) {
    int ctas = 0;
    size_t smem = 0;
    if (!plan(a, p.T, p.Be, p.H, U, ctas, smem)) return PPO_ERR_UNSUPPORTED;
    static PerDevice<bool> set;
    PPO_TRY(ppo_once_per_device(set, [] { return ppo_allow_smem(lstm_bwd_cluster_kernel<U>, kSmemMax); }));
    bool fit = false;
    PPO_TRY(clusters_fit(lstm_bwd_cluster_kernel<U>, ctas, smem, fit));
    if (!fit) return PPO_ERR_UNSUPPORTED;
    PPO_TRY(map_dg(a, p, dg, tile_envs(U)));
    return ppo_launch_together(lstm_bwd_cluster_kernel<U>, dim3(ctas), dim3(kThreads), smem, st, a);
}

}  // namespace

int lstm_fwd_steps(const LstmSteps &p, const bf16 *Wh, const float *xg, const float *bias, const float *h_init, const float *c_init,
                   int32_t *status, cudaStream_t st) {
    Args a = {};
    int ctas = 0, U = 1;
    size_t smem = 0;
    while (U <= 4 && !plan(a, p.T, p.Be, p.H, U, ctas, smem)) U *= 2;
    if (!status || U > 4 || !ppo_aligned(h_init, 16) || !ppo_aligned(c_init, 16)) return PPO_ERR_UNSUPPORTED;
    const long long H = p.H;
    const long long db[2] = {H, 4 * H}, sb[1] = {2 * H};
    const int bb[2] = {64, 16};
    PPO_TRY(make_map_strided(&a.mapB, Wh, 2, db, sb, bb));
    a.done = p.done;
    a.xg = xg; a.bias = bias; a.h_init = h_init; a.c_init = c_init;
    a.gates = p.gates; a.c = p.c; a.cprev = p.cprev; a.h = p.h; a.hprev = p.hprev;
    a.counters = p.counters;
    a.status = status;
    if (U == 1) return launch_fwd<1>(a, p, ctas, smem, st);
    return U == 2 ? launch_fwd<2>(a, p, ctas, smem, st) : launch_fwd<4>(a, p, ctas, smem, st);
}

int lstm_bwd_steps(const LstmSteps &p, const bf16 *WhT, const float *dtop, bf16 *dg, float *dhc, int32_t *status, cudaStream_t st) {
    Args a = {};
    int ctas = 0;
    size_t smem = 0;
    if (!status || !plan(a, p.T, p.Be, p.H, 4, ctas, smem)) return PPO_ERR_UNSUPPORTED;
    const long long H = p.H;
    const long long db[2] = {4 * H, H}, sb[1] = {8 * H};
    const int bb[2] = {64, 64};
    PPO_TRY(make_map_strided(&a.mapB, WhT, 2, db, sb, bb));
    a.done = p.done;
    a.dtop = dtop; a.dg = dg; a.dhc = dhc;
    a.gates = p.gates; a.c = p.c; a.cprev = p.cprev;
    a.counters = p.counters;
    a.status = status;
    int s = launch_bwd_clusters<1>(a, p, dg, st);
    if (s == PPO_ERR_UNSUPPORTED) s = launch_bwd_clusters<2>(a, p, dg, st);
    if (s == PPO_ERR_UNSUPPORTED) s = launch_bwd_clusters<4>(a, p, dg, st);
    if (s != PPO_ERR_UNSUPPORTED) return s;
    plan(a, p.T, p.Be, p.H, 4, ctas, smem);
    PPO_TRY(map_dg(a, p, dg, tile_envs(4)));
    static PerDevice<bool> set;
    PPO_TRY(ppo_once_per_device(set, [] { return ppo_allow_smem(lstm_bwd_kernel, kSmemMax); }));
    return ppo_launch_together(lstm_bwd_kernel, dim3(ctas), dim3(kThreads), smem, st, a);
}

int lstm_one_step(const LstmSteps &p, const bf16 *X, int in, const bf16 *Wx, const bf16 *Wh, const float *bias, const LstmStepEnds &ends,
                  int32_t *status, cudaStream_t st) {
    if (!status || p.T != 1 || p.H % 64 != 0 || in < 64 || in % 8 != 0) return PPO_ERR_UNSUPPORTED;
    StepArgs a = {};
    a.Be = p.Be; a.H = p.H;
    a.bias = bias; a.cprev = p.cprev;
    a.gates = p.gates; a.c = p.c; a.h = p.h;
    a.status = status;
    // the shape with the fewest bytes per CTA whose CTAs all run at once; the largest up to two waves
    const long long sms = ppo_num_sms();
    auto ctas = [&](int M, int U) { return (long long)((p.Be + M - 1) / M) * (p.H / U); };
    if (ctas(32, 8) <= sms) return launch_step<32, 8>(a, in, p, X, Wx, Wh, ends, st);
    if (ctas(32, 16) <= sms) return launch_step<32, 16>(a, in, p, X, Wx, Wh, ends, st);
    if (ctas(64, 16) <= sms) return launch_step<64, 16>(a, in, p, X, Wx, Wh, ends, st);
    if (ctas(128, 16) <= sms) return launch_step<128, 16>(a, in, p, X, Wx, Wh, ends, st);
    if (ctas(128, 32) <= 2 * sms) return launch_step<128, 32>(a, in, p, X, Wx, Wh, ends, st);
    return PPO_ERR_UNSUPPORTED;
}

// 3x3 stride-2 convolutions whose weights fit in shared memory: forward and input gradient as one kind of GEMM on
// halo tiles (sm_100a).
//
// The forward pass of a stride-2 convolution reads its input through four planes, the parities of row and column: plane
// (py, px) holds the pixels (2v + py, 2u + px) and is a plain 4-D tensor to the copy engine (base and strides adjusted).
// In its plane every kernel tap is a shift by 0 or -1.  The input gradient reads one plane, dY itself, at shifts 0 or
// +1.  So a tile of Wt x R outputs (of I images) needs, per plane, one box of (Wt + 1) x (R + 1) cells, and the A operand
// of a tap is that box read from another start address: row m of the MMA is cell m + shift.  The swizzle is a function
// of the shared-memory address, so a matrix may start at any row of a swizzled image.  Rows that fall on the halo
// column or row compute values nobody stores.
//
// Against one box per tap (gemm_tma.cu) this brings a third to a half of the bytes into shared memory with one copy per
// plane, and all three serial streams that bounded these layers get shorter: the copy-issuing thread, the MMA-issuing
// thread (unrolled taps; no zero blocks in the input gradient), and the epilogue (outputs leave as one bulk tensor store
// per 64 columns and tile, clipped at the edges by the copy engine, instead of a shuffle, a load and a store per 16 bytes;
// ReLU gates are fetched a tile ahead).  The weights stay in shared memory for the life of the CTA.  Sums run in the same
// order as in gemm_tma.cu: the results are the same bits.
// Measured, 4096 rows alone (tap boxes -> here; in brackets the HBM time of inputs, gates and outputs): 32 -> 64 channels on
// 160 x 120 forward 2.22 -> 1.25 ms (1.17), input gradient 3.25 -> 1.28 (1.2); 64 -> 128 on 80 x 60 forward 1.20 -> 0.98
// (0.58; tap boxes whose tiles go in pairs of CTAs take 0.90, and that forward pass), input gradient 1.58 -> 1.01 to 1.07 (0.6).
#include <cuda.h>

#include "conv1_window.h"
#include "gemm.cuh"
#include "halo_plan.h"
#include "launch.cuh"
#include "tcgen05.cuh"
#include "tma_host.cuh"

namespace {

using namespace tc;
using namespace halo;

// An epilogue group works on a tile, the groups of a CTA on alternate ones.  A group has four warps, one per TMEM lane
// quarter: fewer meet at its barriers, and two tiles are drained at a time.  Where shared memory holds only one CTA per SM
// and two staging buffers, a group has eight warps, two per lane quarter, which share out the columns.

enum { FWD = 0, FWD_LN = 1, DG = 2 };

template <int EPW>
__device__ __forceinline__ void epi_sync(int eg) { asm volatile("bar.sync %0, %1;" ::"r"(1 + eg), "n"(EPW * 32) : "memory"); }

// The sign bits of bytes 1 and 3, each replicated over its half word (prmt.b32 in its sign-replicating form).
__device__ __forceinline__ uint32_t half_signs(uint32_t x) {
    uint32_t r;
    asm("prmt.b32 %0, %1, 0, 0xBB99;" : "=r"(r) : "r"(x));
    return r;
}
// Pair j of the 32-channel gate word (bits j and 16 + j) as a mask over the two halves.
__device__ __forceinline__ uint32_t gate_mask(uint32_t gate, int j) { return half_signs(gate << (15 - j)); }

// Slots in the order they become free: four bits each, the next one lowest.  Producer and MMA warp walk the same
// sequence, so a slot that is read for the last time early in a tile takes the next tile's first load.
struct SlotQueue {
    uint32_t q;
    int n;
    __device__ void init(int slots) {
        q = 0x76543210u;
        n = slots;
    }
    __device__ int pop() {
        const int s = (int)(q & 15u);
        q >>= 4;
        --n;
        return s;
    }
    __device__ void push(int s) {
        q = (q & ~(15u << (4 * n))) | ((uint32_t)s << (4 * n));
        ++n;
    }
};

struct TileAt {
    int n, y, x;  // first image, row and column of the tile
    __device__ void init(const Args &a, int t) {
        const int xs = t % a.xsegs;
        t /= a.xsegs;
        const int ys = t % a.ysegs;
        n = t / a.ysegs * a.I;
        x = xs * a.Wt;
        y = ys * a.R;
    }
    __device__ void next(const Args &a) {
        x += a.Wt;
        if (x >= a.Wr) {
            x = 0;
            y += a.R;
            if (y >= a.Hr) {
                y = 0;
                n += a.I;
            }
        }
    }
};

// Barrier of an epilogue group that also ANDs a condition over them (a bounded wait that ran out in one warp ends all).
template <int EPW>
__device__ __forceinline__ bool epi_all(bool ok, int eg) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.b32 p, %1, 0;\n\t"
        "bar.red.and.pred q, %3, %2, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"(ok ? 1u : 0u), "n"(EPW * 32), "r"(1 + eg)
        : "memory");
    return r != 0;
}

// A kernel parameter in a register: several roles that each read theirs in their loops evict one another's from the constant
// cache, and a reading then takes a few hundred cycles.
__device__ __forceinline__ int held(int v) {
    asm volatile("" : "+r"(v));
    return v;
}

// A walk through the row groups of a CTA: the barriers' index and parity, the group's place in its image, and the ring slot of its first
// pixel (negative while that lies in front of the CTA's run).
struct GroupWalk {
    int groups, ysegs, group_px, last_px, ring_px;
    int i, k, slot;
    uint32_t ph;
    __device__ void init(const Args &a, const First &f, int k0, int slot0) {
        groups = held(f.groups); ysegs = held(a.ysegs); group_px = held(f.group_px); last_px = held(f.last_px); ring_px = held(f.ring_px);
        i = 0; k = k0; slot = slot0; ph = 0;
    }
    __device__ int px() const { return k == ysegs - 1 ? last_px : group_px; }
    __device__ void next() {
        slot += px();
        if (slot >= ring_px) slot -= ring_px;
        if (++i == groups) { i = 0; ph ^= 1u; }
        if (++k == ysegs) k = 0;
    }
};

// Place of the 16-byte piece `piece` of ring pixel `row`, two to a line.  Neighbouring lanes of the epilogue write every second pixel,
// ldmatrix reads eight in a row: both go to eight different 16-byte columns of the 128-byte lines.
__device__ __forceinline__ uint32_t ring_offset(int row, int piece) {
    const int line = row >> 1, q = (row & 1) * 4 + piece;
    return (uint32_t)line * 128u + ((uint32_t)(q ^ (line & 7)) << 4);
}

// Builder warp bw: the window tiles of the pixels p0 .. p1, [32 px][TP] bf16, four trips to a stage; trip bw % 4 of every second
// stage.
// The builders also stand between ring and sums, whose loop is the kernel's longest chain: a stage is handed over when its pixels
// have arrived in the ring, and the first of them gives a row group back when it has seen the stage it ends in summed.
__device__ __forceinline__ void first_windows(const First &f, int H1, int W1, const __half *depth, int p0, int p1, const GroupWalk &at, int bw,
                                              uint8_t *patch, FirstPipe *pipe, int32_t *status) {
    constexpr int TP = Window<kFirstK>::TP;
    const int lane = threadIdx.x & 31, nstages = (p1 - p0 + kStagePx - 1) / kStagePx;
    const uint32_t *const frames = reinterpret_cast<const uint32_t *>(depth);
    const int Hf = held(f.Hf), Wh = held(f.Wh);
    H1 = held(H1);
    W1 = held(W1);
    int m = p0 + (bw >> 2) * kStagePx + (bw & 3) * kTrip + lane;
    WindowWalk<kFirstK> px;
    px.init(m, W1, H1);
    const int d_oh = 2 * kStagePx / W1, d_ow = 2 * kStagePx - d_oh * W1;
    uint32_t raw[Window<kFirstK>::KW];
    bool live = false;
    auto fetch = [&]() {  // a trip's loads, a turn ahead of their use
        live = m < p1;
        px.fetch(frames, Hf, Wh, live, raw);
        m += 2 * kStagePx;
        px.advance(d_ow, d_oh, W1, H1);
    };
    fetch();
    uint8_t *const mine = patch + (size_t)((bw & 3) * kTrip + lane) * (TP * 2);
    GroupWalk seen = at, done = at;
    int avail = at.slot, ended = at.slot + at.px();  // pixels of the run that have arrived; end of group `done`
    for (int s = bw >> 2; s < nstages; s += 2) {
        uint32_t wv[TP / 2];
        window_row<kFirstK>(raw, live, wv);
        fetch();
        const int slot = s & (kWinStages - 1);
        if (!mbar_wait_warp(&pipe->pempty[slot], (uint32_t)(s / kWinStages & 1) ^ 1u, &pipe->abort_flag, status)) return;
        put_row(mine + (size_t)slot * (kStagePx * TP * 2), lane, wv);
        if (ring_gives_back(bw))
            for (; ended <= ring_summed(s); ended += done.px()) {  // (the first stages have nothing before them)
                if (lane == 0) mbar_arrive(&pipe->gempty[done.i]);
                done.next();
            }
        const int end = ring_needs(s, p1 - p0);
        while (avail < end) {
            if (!mbar_wait_warp(&pipe->gfull[seen.i], seen.ph, &pipe->abort_flag, status)) return;
            avail += seen.px();
            seen.next();
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&pipe->pfull[slot]);
    }
}

// dW1[co][tap] = sum over pixels dZ1[px][co] x[px][tap] as mma.sync m16n8k16 with the pixel as K, dZ1 from the ring in which the
// epilogue leaves it and x from the builders' window tiles.  The pixels are summed in the runs, the trips of 32 and the blocks
// of conv1_wgrad_mma_kernel: the same bits.  A run is one chain of dependent products, 25 cycles for 16 pixels, and a fragment load
// takes its warp 16 to 20: a unit of all 16 rows (pair elements of the window) x 16 channels per warp, its fragments two trips ahead.  Finer
// units make shorter chains of more shared-memory reads: 8 channels a unit 490 us, 16 channels 450 to 475.
__device__ __forceinline__ void first_sums(const First &f, int p0, int p1, int block0, int ring_px, int unit, uint32_t ring, uint32_t patch,
                                           FirstPipe *pipe, int32_t *status) {
    using WN = Window<kFirstK>;
    constexpr int TP = WN::TP, KW = WN::KW, NP = WN::NP, ODD = WN::ODD, K1 = kFirstK, K2 = K1 * K1, C1 = kFirstC;
    const int lane = threadIdx.x & 31, mi = lane >> 3, r = lane & 7;
    // held: registers are allotted otherwise without it (a backward pass of two layers, 4096 rows of 160 x 120: 926 us, with it 920)
    const int uj = 2 * held(unit & (kUnits - 1));
    uint32_t a_off[2], b_off[2];
#pragma unroll
    for (int ks = 0; ks < 2; ++ks) {
        const int ar = 16 * ks + r + (mi >= 2 ? 8 : 0), c = (mi & 1) ^ piece_swizzle(ar, TP * 2);
        a_off[ks] = (uint32_t)(ar * (TP * 2) + (c << 4));
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) b_off[j] = ring_offset(lane, uj + j);  // (a trip starts at a multiple of 32 pixels)
    const int total = p1 - p0, nstages = (total + kStagePx - 1) / kStagePx;
    const int run_trips = held(f.px_per_warp / kTrip);
    const uint32_t ring_end = ring + (uint32_t)ring_px * (C1 * 2);  // (whole stages)
    float *out = f.part + (size_t)block0 * (C1 * (K2 + 1));
    float acc[2][4] = {}, sum[2][4] = {};
    int left = run_trips, run = 0;
    // The end of a run: eight of them, in order, make a block.
    auto flush = [&](bool last) {
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                sum[j][q] += acc[j][q];
                acc[j][q] = 0.f;
            }
        left = run_trips;
        if (++run < 8 && !last) return;
        const int g = lane >> 2, c = lane & 3;
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int t = g + (q & 2 ? 8 : 0), co = 8 * (uj + j) + 2 * c + (q & 1);
                const int kh = (t >> 1) / NP, kw = 2 * ((t >> 1) - kh * NP) + (t & 1) - ODD;
                if (t < 2 * KW && kw >= 0 && kw < K1) out[co * K2 + kh * K1 + kw] = sum[j][q];
                else if (t == 2 * KW) out[C1 * K2 + co] = sum[j][q];
                sum[j][q] = 0.f;
            }
        run = 0;
        out += C1 * (K2 + 1);
    };
    constexpr uint32_t kX = kTrip * TP * 2, kZ = kTrip * C1 * 2;  // bytes of a trip
    constexpr int LA = 2;                            // trips that are fetched ahead
    uint32_t af[2 * LA][2][4], bf[2 * LA][2][4];     // fragments
    auto fetch_z = [&](int b, uint32_t zs) {
#pragma unroll
        for (int j = 0; j < 2; ++j) ldmatrix_x4_trans(zs + b_off[j], bf[b][j][0], bf[b][j][1], bf[b][j][2], bf[b][j][3]);
    };
    auto fetch_x = [&](int b, int ks, uint32_t xs) {
        ldmatrix_x4_trans(xs + a_off[ks], af[b][ks][0], af[b][ks][1], af[b][ks][2], af[b][ks][3]);
    };
    auto products = [&](int b, int ks) {
#pragma unroll
        for (int j = 0; j < 2; ++j) mma_bf16_16816(acc[j], af[b][ks], bf[b][j][2 * ks], bf[b][j][2 * ks + 1]);
    };
    uint32_t xs = patch, zs = ring, ph = 0;
    int ps = 0;
    if (!mbar_wait_warp(&pipe->pfull[0], 0, &pipe->abort_flag, status)) return;
    if (nstages > 1) {
#pragma unroll
        for (int t = 0; t < LA; ++t) {
            fetch_z(t, zs + t * kZ);
            fetch_x(t, 0, xs + t * kX);
            fetch_x(t, 1, xs + t * kX);
        }
    }
#pragma unroll 1
    for (int s = 0; s + 1 < nstages; ++s) {
        const int old = ps;
        uint32_t xn = xs, zn = zs;  // of the stage that trip t + LA is in
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const int b = t % (2 * LA), n = (t + LA) % (2 * LA), u = (t + LA) & 3;
            products(b, 0);
            if (t + LA == 4) {
                zn = zs + 4 * kZ;
                if (zn == ring_end) zn = ring;
                xn = xs + 4 * kX;
                if (++ps == kWinStages) {
                    ps = 0;
                    xn = patch;
                    ph ^= 1u;
                }
                if (!mbar_wait_warp(&pipe->pfull[ps], ph, &pipe->abort_flag, status)) return;
            }
            fetch_z(n, zn + u * kZ);
            fetch_x(n, 0, xn + u * kX);
            products(b, 1);
            fetch_x(n, 1, xn + u * kX);
            if (t < 3 && --left == 0) flush(false);
        }
        xs = xn;
        zs = zn;
        __syncwarp();  // (the release covers what all lanes read)
        if (lane == 0) mbar_arrive(&pipe->pempty[old]);
        if (--left == 0) flush(false);
    }
    // the last stage, trip by trip
#pragma unroll 1
    for (int px = (nstages - 1) * kStagePx; px < total; px += kTrip, xs += kX, zs += kZ) {
        fetch_z(0, zs);
        fetch_x(0, 0, xs);
        fetch_x(0, 1, xs);
        const int rest = total - px;
        if (rest < kTrip) {  // behind the last pixel the ring holds something else
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int k = 8 * q + 2 * (lane & 3);
#pragma unroll
                for (int j = 0; j < 2; ++j) bf[0][j][q] &= (k < rest ? 0xFFFFu : 0u) | (k + 1 < rest ? 0xFFFF0000u : 0u);
            }
        }
        products(0, 0);
        products(0, 1);
        if (--left == 0 || rest <= kTrip) flush(rest <= kTrip);
    }
}

// GC: columns of an output group, i.e. of one pixel of one store (16, 32 or 64; its bytes are the swizzled row).
// KS: K = 16 steps per channel chunk (1, 2 or 4: rows of 32, 64 or 128 bytes).
// EPW: warps of an epilogue group, 4 or 8.
// FIRST: the first layer's weight gradient takes the place of the output (input gradient, EPW 4, GC = kFirstC).
template <int MODE, int GC, int KS, int EPW, bool FIRST>
__device__ __forceinline__ void halo_body(const Args &a, const First &f, const __half *depth, uint8_t *smem_raw) {
    constexpr int NH = EPW == 4 ? 2 : 1;  // halves of 64 columns a warp works on
    constexpr uint32_t kPatchBytes = kWinStages * kStagePx * Window<kFirstK>::TP * 2;
    static_assert(!FIRST || (MODE == DG && GC == kFirstC && EPW == 4), "");
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const uint32_t smem_base = smem_u32(smem);
    // A slots, then weights (reads of the last slot's halo rows may run on into them), output staging, pipeline state
    const uint32_t w_base = smem_base + a.slots_bytes;
    const uint32_t w_bytes = (uint32_t)a.nchunks * a.w_chunk;
    const uint32_t stg_off = (a.slots_bytes + w_bytes + 1023u) & ~1023u;
    Pipe *pipe = reinterpret_cast<Pipe *>(smem + stg_off + (FIRST ? (size_t)f.ring_bytes + kPatchBytes : (size_t)(a.nbuf * a.neg) * a.stg_bytes));
    [[maybe_unused]] FirstPipe *const hand = static_cast<FirstPipe *>(pipe);  // (FIRST)
    volatile int *abort_flag = &pipe->abort_flag;
    const int warp = warp_index(), lane = threadIdx.x & 31;
    const int nacc = a.nacc;
    const uint32_t ncols = (uint32_t)(a.acc_cols * nacc);

    if (threadIdx.x == 0) {
        for (int s = 0; s < a.slots; ++s) {
            mbar_init(&pipe->full[s], 1);
            mbar_init(&pipe->empty[s], 1);
        }
        for (int i = 0; i < nacc; ++i) {
            mbar_init(&pipe->tfull[i], 1);
            mbar_init(&pipe->tempty[i], EPW * 32);
        }
        mbar_init(&pipe->wfull, 1);
        if constexpr (FIRST) {
            for (int i = 0; i < f.groups; ++i) {
                mbar_init(&hand->gfull[i], (uint32_t)(a.xsegs * EPW * 32));
                mbar_init(&hand->gempty[i], 1);
            }
            for (int i = 0; i < kWinStages; ++i) {
                mbar_init(&hand->pfull[i], kStagePx / kTrip);
                mbar_init(&hand->pempty[i], kUnits);
            }
        }
        pipe->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) tmem_alloc(&pipe->tmem_slot, ncols);
    grid_wait();
    if (MODE == FWD || MODE == FWD_LN)
        for (int i = threadIdx.x; i < a.N; i += (int)blockDim.x) {
            pipe->bias[i] = a.bias[i];
            if (MODE == FWD_LN) {
                pipe->gamma[i] = a.ln_gamma[i];
                pipe->beta[i] = a.ln_beta[i];
            }
        }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = pipe->tmem_slot;

    // contiguous run of tiles for this CTA
    const int q = a.tiles / (int)gridDim.x, rem = a.tiles - q * (int)gridDim.x, bid = (int)blockIdx.x;
    int t0 = bid * q + (bid < rem ? bid : rem), nt = q + (bid < rem ? 1 : 0);
    // with the first layer's sums: the tiles of the row groups that hold the pixels of its blocks
    int p0 = 0, p1 = 0, block0 = 0;
    GroupWalk first_group;
    if constexpr (FIRST) {
        const int bq = f.blocks / (int)gridDim.x, br = f.blocks - bq * (int)gridDim.x, nb = bq + (bid < br ? 1 : 0);
        block0 = bid * bq + (bid < br ? bid : br);
        p0 = block0 * 8 * f.px_per_warp;
        p1 = (int)min((long long)f.M, (long long)(block0 + nb) * 8 * f.px_per_warp);
        auto group_of = [&](int px, int &k, int &start) -> int {  // its number over all images, and where it starts
            const int img = px / (a.Hi * a.Wi), in = px - img * a.Hi * a.Wi;
            k = in / f.group_px;
            start = img * a.Hi * a.Wi + k * f.group_px;
            return img * a.ysegs + k;
        };
        int k, start, k1, start1;
        const int g0 = group_of(p0, k, start), g1 = group_of(p1 - 1, k1, start1);
        first_group.init(a, f, k, start - p0);
        t0 = g0 * a.xsegs;
        nt = (g1 - g0 + 1) * a.xsegs;
    }

    if (warp == 0) {
        {
            if (elect_one()) mbar_arrive_expect_tx(&pipe->wfull, w_bytes);
            for (int c = 0; c < a.nchunks; ++c)
                for (int i = 0; i < a.nwl; ++i)
                    if (elect_one()) tma_load_2d(w_base + (uint32_t)c * a.w_chunk + a.wl[i].off, &a.mapW, &pipe->wfull, a.wl[i].k0 + c * a.CB, 0);
            TileAt t;
            t.init(a, t0);
            SlotQueue sq;
            sq.init(a.slots);
            uint32_t phase = 0, armed = 0;  // per slot: parity of its next use; whether it was ever filled
            bool ok = true;
            for (int li = 0; li < nt && ok; ++li, t.next(a)) {
                uint32_t used = 0;  // the tile's slots in the order of its loads
                for (int i = 0; i < a.nloads; ++i) {  // forward: the planes in the order of their first tap; else the chunks
                    const int p = a.nplanes == 4 ? 3 - i : 0, s = sq.pop();
                    const Plane &pl = a.planes[p];
                    used |= (uint32_t)s << (4 * i);
                    ok = mbar_wait_warp(&pipe->empty[s], (~phase >> s) & 1u, abort_flag, a.status);
                    if (!ok) break;
                    phase ^= 1u << s;
                    armed |= 1u << s;
                    if (elect_one()) {
                        mbar_arrive_expect_tx(&pipe->full[s], pl.bytes);
                        tma_load_4d(smem_base + (uint32_t)s * a.slot_bytes, &a.mapA[p], &pipe->full[s], a.nplanes == 4 ? 0 : i * a.CB,
                                    t.x + pl.ox, t.y + pl.oy, t.n);
                    }
                    __syncwarp();
                }
                if (a.nplanes == 4) used = (used >> 8) | (used << 8 & 0xFF00u);  // planes 01 and 00 are done first
                for (int i = 0; i < a.nloads; ++i) sq.push((int)(used >> (4 * i)) & 15);
            }
            if (!ok) {  // bounded wait for the copies in flight
                for (int s = 0; s < a.slots; ++s) {
                    if (!((armed >> s) & 1u)) continue;
                    const long long c0 = clock64();
                    while (!mbar_try_wait(&pipe->full[s], (~phase >> s) & 1u))
                        if (clock64() - c0 > kWaitCycles / 4) break;
                }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // One thread feeds the tensor core and its instruction stream is what bounds the narrow layers, so the taps of a
        // plane are unrolled: everything but the slot's address is a constant of the launch.
        // The sums run in the order tap, channel (and shift, channel), whatever the order of the loads.
        constexpr bool kFwd = MODE == FWD || MODE == FWD_LN;
        constexpr uint32_t rb = KS * 32u, sbo = 8u * rb;
        const uint64_t d0 = smem_desc_sw(smem_base, 16, sbo, rb);
        const uint32_t a_lo0 = (uint32_t)d0, d_hi = (uint32_t)(d0 >> 32);
        const uint32_t w_lo0 = a_lo0 + ((w_base - smem_base) >> 4);
        const uint32_t slot16 = a.slot_bytes >> 4, wchunk16 = a.w_chunk >> 4;
        SlotQueue sq;
        sq.init(a.slots);
        int acc = 0;
        uint32_t phase = 0, aph = 1u;  // parities of the slots; parity that says the accumulator has been drained
        bool ok = mbar_wait_warp(&pipe->wfull, 0, abort_flag, a.status);
        auto taps = [&](int o, uint32_t la0, uint32_t lb0, uint32_t tmem_d, uint32_t accum) {
            const Op &op = a.ops[o];
            const uint32_t la = la0 + op.a16, lb = lb0 + op.b16, td = tmem_d + op.dcol, id = op.idesc;
            umma_bf16_lh(td, la, d_hi, lb, d_hi, id, accum);
#pragma unroll
            for (int k = 1; k < KS; ++k) umma_bf16_lh(td, la + 2 * k, d_hi, lb + 2 * k, d_hi, id, 1u);
        };
        for (int li = 0; li < nt && ok; ++li) {
            ok = mbar_wait_warp(&pipe->tempty[acc], aph, abort_flag, a.status);
            if (!ok) break;
            tc_fence_after();
            const uint32_t tmem_d = tmem_base + (uint32_t)(acc * a.acc_cols);
            if (kFwd) {
                // planes 11, 10, 01, 00 sit in four consecutive slots; taps in raster order need them in that order
                int sl[4];
                uint32_t la[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    sl[i] = sq.pop();
                    la[i] = a_lo0 + (uint32_t)sl[i] * slot16;
                }
#pragma unroll
                for (int t = 0; t < 9; ++t) {
                    constexpr int kLoad[9] = {0, 1, 0, 2, 3, 2, 0, 1, 0};  // load that brings the tap's plane
                    const int i = kLoad[t];
                    if (t < 2 || t == 3 || t == 4) {
                        ok = mbar_wait_warp(&pipe->full[sl[i]], (phase >> sl[i]) & 1u, abort_flag, a.status);
                        if (!ok) break;
                        tc_fence_after();
                    }
                    if (elect_one()) {
                        taps(t, la[i], w_lo0, tmem_d, t > 0 ? 1u : 0u);
                        if (t == 5) {
                            umma_commit(&pipe->empty[sl[2]]);
                            umma_commit(&pipe->empty[sl[3]]);
                        }
                    }
                    __syncwarp();
                }
                if (!ok) break;
                if (elect_one()) {
                    umma_commit(&pipe->empty[sl[0]]);
                    umma_commit(&pipe->empty[sl[1]]);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    phase ^= 1u << sl[i];
                    sq.push(sl[i ^ 2]);
                }
            } else {
                uint32_t used = 0;
                for (int c = 0; c < a.nchunks; ++c) {
                    const int s = sq.pop();
                    used |= (uint32_t)s << (4 * c);
                    ok = mbar_wait_warp(&pipe->full[s], (phase >> s) & 1u, abort_flag, a.status);
                    if (!ok) break;
                    phase ^= 1u << s;
                }
                if (!ok) break;
                tc_fence_after();
                if (elect_one()) {
#pragma unroll
                    for (int o = 0; o < 4; ++o) {
                        uint32_t lb = w_lo0;
                        for (int c = 0; c < a.nchunks; ++c, lb += wchunk16) {
                            const int s = (int)(used >> (4 * c)) & 15;
                            taps(o, a_lo0 + (uint32_t)s * slot16, lb, tmem_d, o > 0 || c > 0 ? 1u : 0u);
                            if (o == 3) umma_commit(&pipe->empty[s]);
                        }
                    }
                }
                for (int c = 0; c < a.nchunks; ++c) sq.push((int)(used >> (4 * c)) & 15);
            }
            if (elect_one()) umma_commit(&pipe->tfull[acc]);
            __syncwarp();
            if (++acc == nacc) { acc = 0; aph ^= 1u; }
        }
    } else if (FIRST && warp >= 10) {
        if constexpr (FIRST) {
            const uint32_t patch_off = stg_off + f.ring_bytes;
            if (warp < 10 + kBuildWarps) first_windows(f, a.Hi, a.Wi, depth, p0, p1, first_group, warp - 10, smem + patch_off, hand, a.status);
            else first_sums(f, p0, p1, block0, first_group.ring_px, warp - 10 - kBuildWarps, smem_base + stg_off, smem_base + patch_off, hand, a.status);
        }
    } else {
        // ---------------- epilogue: warp reads TMEM lanes 32 (warp % 4) .. +31 and, of every 64 columns, half `h`
        const int lg = warp & 3, eg = (warp - 2) / EPW, h = EPW == 4 ? 0 : ((warp - 2) >> 2) & 1;
        const int m = lg * 32 + lane;
        const int ci = m / (a.Rp * a.Wp), mr = m - ci * a.Rp * a.Wp, cr = mr / a.Wp, cx = mr - cr * a.Wp;
        const bool cell = ci < a.I && cr < a.R && cx < a.Wt;  // an output of the tile, not a halo cell
        const int srow = (ci * a.R + cr) * a.Wt + cx;         // its row in the dense staging tile
        const bool issuer = threadIdx.x == 64 + eg * EPW * 32;
        constexpr uint32_t RBO = GC * 2;                      // bytes of a staged row
        const uint32_t sx = GC == 64 ? (uint32_t)(srow & 7) : (GC == 32 ? (uint32_t)(srow >> 1) & 3u : (uint32_t)(srow >> 2) & 1u);
        const uint32_t grp_bytes = a.stg_bytes / (uint32_t)a.stg_row * RBO;    // of an output group's part of a staging buffer
        const int nsteps = (a.N + 63) >> 6;
        int acc = eg, buf = 0;  // nacc is even where there are two groups
        uint32_t aph = 0;
        TileAt t;
        t.init(a, t0 + (eg < nt ? eg : 0));
        // columns col .. col + 7 (of the step's 64) of this thread's row
        auto put = [&](uint32_t stg, int col, uint4 v) {
            const uint32_t grp = (uint32_t)col / GC, piece = ((uint32_t)col % GC) >> 3;
            const uint32_t addr = stg + grp * grp_bytes + (uint32_t)srow * RBO + ((piece ^ sx) << 4);
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
        };
        auto stage_free = [&]() {  // the store that last read this buffer is done (asked by the thread that issued it)
            if (issuer) {
                if (a.nbuf == 2) bulk_wait_read<1>();
                else bulk_wait_read<0>();
            }
        };
        auto store_step = [&](uint32_t stg, int s, const CUtensorMap *maps) {
            fence_async_smem();
            epi_sync<EPW>(eg);
            if (issuer) {
#pragma unroll
                for (int g = 0; g < 64 / GC; ++g) {
                    const int col = s * 64 + g * GC, grp = col / GC;
                    if (col >= a.N) break;
                    if (MODE == FWD || MODE == FWD_LN) {
                        tma_store_4d(maps, stg + (uint32_t)g * grp_bytes, col, t.x, t.y, t.n);
                    } else {  // parity classes in the order 00, 01, 11, 10
                        const int ph = grp >> 1, pw = (grp == 1 || grp == 2) ? 1 : 0;
                        if (2 * t.y + ph < a.Hi && 2 * t.x + pw < a.Wi)
                            tma_store_4d(maps + grp, stg + (uint32_t)g * grp_bytes, 0, t.x, t.y, t.n);
                    }
                }
                bulk_commit();
            }
            if (++buf == a.nbuf) buf = 0;
        };
        const uint32_t stg0 = smem_base + stg_off + (uint32_t)(eg * a.nbuf) * a.stg_bytes;
        // ReLU gates of the pixels this thread's columns belong to.  They are fetched a tile ahead: this warp is what the
        // tile waits for, so a load on its own tile's path would cost its whole latency.
        uint32_t gate[4], gate_n[4];
        auto fetch_gates = [&](const TileAt &at) {
            const int n = at.n + ci, y = at.y + cr, x = at.x + cx;
            const bool live = cell && n < a.B && y < a.Hr && x < a.Wr;
            if (MODE == DG) {
                auto word = [&](int col) -> uint32_t {  // gates of the class that owns column col (a half word for 16 channels)
                    const int grp = col / GC, iy = 2 * y + (grp >> 1), ix = 2 * x + ((grp == 1 || grp == 2) ? 1 : 0);
                    if (col >= a.N || !live || iy >= a.Hi || ix >= a.Wi) return 0u;
                    const long long px = ((long long)n * a.Hi + iy) * a.Wi + ix;
                    if (GC == 16) return __ldg(reinterpret_cast<const uint16_t *>(a.mask_bits) + px);
                    return __ldg(a.mask_bits + px * (GC / 32 > 0 ? GC / 32 : 1) + (GC == 64 ? (col >> 5) & 1 : 0));
                };
#pragma unroll
                for (int k = 0; k < 4; ++k) {  // step k / NH, half k % NH (EPW == 4: at most 128 columns)
                    const int col = (k / NH) * 64 + (EPW == 4 ? k % NH : h) * 32;
                    if (GC == 16) gate_n[k] = k < NH ? gate_of_halves(word(col), word(col + 16)) : 0u;  // 64 columns: one step
                    else gate_n[k] = word(col);
                }
            }
        };
        TileAt t_next = t;
        if (eg < nt) fetch_gates(t);
        if constexpr (FIRST) {
            // The input gradient of the first layer's output goes into the ring its weight gradient is summed from, pixel by pixel.
            GroupWalk grp = first_group;
            const int xsegs = held(a.xsegs), Hi = held(a.Hi), Wi = held(a.Wi), B = held(a.B), Hr = held(a.Hr), Wr = held(a.Wr);
            int xs = 0;  // of the tile in its row group
            auto next_tile = [&]() {
                if (++xs == xsegs) {
                    xs = 0;
                    grp.next();
                }
            };
            for (int k = 0; k < eg; ++k) next_tile();
            const uint32_t ring = smem_base + stg_off;
            for (int li = eg; li < nt; li += a.neg, t = t_next) {
                const int n = t.n + ci, y = t.y + cr, x = t.x + cx;
                const bool live = cell && n < B && y < Hr && x < Wr;
#pragma unroll
                for (int k = 0; k < 4; ++k) gate[k] = gate_n[k];
                for (int k = 0; k < a.neg; ++k) t_next.next(a);
                if (li + a.neg < nt) fetch_gates(t_next);
                const int gi = grp.i, slot = grp.slot;
                const uint32_t gph = grp.ph;
                for (int k = 0; k < a.neg; ++k) next_tile();
                if (!mbar_wait_warp(&hand->gempty[gi], gph ^ 1u, abort_flag, a.status)) break;
                if (!mbar_wait_warp(&pipe->tfull[acc], aph, abort_flag, a.status)) break;
                tc_fence_after();
                const uint32_t lane_base = tmem_base + (uint32_t)(acc * a.acc_cols) + ((uint32_t)(lg * 32) << 16);
#pragma unroll 1
                for (int q = 0; q < 4; ++q) {  // classes (rolled: the roles' loops share the instruction cache)
                    float v[32];
                    tmem_ld32(lane_base + (uint32_t)(32 * q), v);
                    if (q == 3) {
                        tc_fence_before();
                        mbar_arrive(&pipe->tempty[acc]);
                    }
                    const uint32_t gw = q == 0 ? gate[0] : (q == 1 ? gate[1] : (q == 2 ? gate[2] : gate[3]));
                    const int ph = q >> 1, pw = (q ^ ph) & 1;
                    int row = slot + (2 * cr + ph) * Wi + 2 * x + pw;
                    const bool put_it = live && row >= 0 && 2 * y + ph < Hi && 2 * x + pw < Wi;
                    if (row >= grp.ring_px) row -= grp.ring_px;
                    uint32_t pk[16];
#pragma unroll
                    for (int j = 0; j < 16; ++j) pk[j] = pack_bf16x2(v[2 * j], v[2 * j + 1]) & gate_mask(gw, j);
                    if (put_it) {
#pragma unroll
                        for (int c = 0; c < 4; ++c)
                            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(ring + ring_offset(row, c)), "r"(pk[4 * c]),
                                         "r"(pk[4 * c + 1]), "r"(pk[4 * c + 2]), "r"(pk[4 * c + 3])
                                         : "memory");
                    }
                }
                mbar_arrive(&hand->gfull[gi]);
                acc += a.neg;
                if (acc >= nacc) { acc = eg; aph ^= 1u; }
            }
        } else
        for (int li = eg; li < nt; li += a.neg, t = t_next) {
            const int n = t.n + ci, y = t.y + cr, x = t.x + cx;
            const bool live = cell && n < a.B && y < a.Hr && x < a.Wr;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (MODE == DG) gate[k] = gate_n[k];
            }
            for (int k = 0; k < a.neg; ++k) t_next.next(a);
            if (li + a.neg < nt) fetch_gates(t_next);
            stage_free();
            const bool ok = epi_all<EPW>(mbar_wait(&pipe->tfull[acc], aph, abort_flag, a.status), eg);
            if (!ok) break;
            tc_fence_after();
            const uint32_t lane_base = tmem_base + (uint32_t)(acc * a.acc_cols) + ((uint32_t)(lg * 32) << 16);
            if (MODE == FWD_LN) {
                // Layer normalisation over the N channels of this thread's row.  32 channels stay in registers; more are
                // walked three times in tensor memory (mean, variance about it, result).  Normalised values and outputs of 32
                // channels leave with one hand-over.
                const long long px = ((long long)n * a.Hr + y) * a.Wr + x;
                const bool one = a.N == 32;
                float v[32];
                float sum = 0.f, sq = 0.f;
                auto load = [&](int c0) {
                    tmem_ld32(lane_base + (uint32_t)c0, v);
#pragma unroll
                    for (int i = 0; i < 32; ++i) v[i] += pipe->bias[c0 + i];
                };
                for (int c0 = 0; c0 < a.N; c0 += 32) {
                    load(c0);
#pragma unroll
                    for (int i = 0; i < 32; ++i) sum += v[i];
                }
                const float mean = sum / (float)a.N;
                for (int c0 = 0; c0 < a.N; c0 += 32) {
                    if (!one) load(c0);
#pragma unroll
                    for (int i = 0; i < 32; ++i) {
                        v[i] -= mean;
                        sq += v[i] * v[i];
                    }
                }
                const float rs = rsqrtf(sq / (float)a.N + kLnEps);
                if (live) a.ln_rstd[px] = rs;
#pragma unroll 1
                for (int c0 = 0; c0 < a.N; c0 += 32) {
                    if (!one) {
                        load(c0);
#pragma unroll
                        for (int i = 0; i < 32; ++i) v[i] -= mean;
                    }
                    if (c0 + 32 == a.N) {
                        tc_fence_before();
                        mbar_arrive(&pipe->tempty[acc]);
                    }
                    if (c0 > 0) {
                        stage_free();
                        epi_sync<EPW>(eg);
                    }
                    const uint32_t stg = stg0 + (uint32_t)buf * a.stg_bytes;
                    uint32_t w = 0;
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        uint32_t xh[4], rl[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const int c = 8 * k + 2 * i;
                            const float x0 = v[c] * rs, x1 = v[c + 1] * rs;
                            xh[i] = pack_bf16x2(x0, x1);
                            rl[i] = relu_pack_bf16x2(fmaf(pipe->gamma[c0 + c], x0, pipe->beta[c0 + c]),
                                                     fmaf(pipe->gamma[c0 + c + 1], x1, pipe->beta[c0 + c + 1]));
                            w = gate_bits_add(w, rl[i], 4 * k + i);
                        }
                        if (cell) {
                            put(stg, 8 * k, make_uint4(xh[0], xh[1], xh[2], xh[3]));
                            put(stg, 32 + 8 * k, make_uint4(rl[0], rl[1], rl[2], rl[3]));
                        }
                    }
                    if (a.out_bits && live) a.out_bits[px * (a.N >> 5) + (c0 >> 5)] = w;
                    fence_async_smem();
                    epi_sync<EPW>(eg);
                    if (issuer) {
                        tma_store_4d(&a.mapX, stg, c0, t.x, t.y, t.n);
                        tma_store_4d(&a.mapO[0], stg + grp_bytes, c0, t.x, t.y, t.n);
                        bulk_commit();
                    }
                    if (++buf == a.nbuf) buf = 0;
                }
                acc += a.neg;
                if (acc >= nacc) { acc = eg; aph ^= 1u; }
                continue;
            }
#pragma unroll 1
            for (int s = 0; s < nsteps; ++s) {
                if (s > 0) {
                    stage_free();
                    epi_sync<EPW>(eg);
                }
                const uint32_t stg = stg0 + (uint32_t)buf * a.stg_bytes;
#pragma unroll
                for (int q = 0; q < NH; ++q) {
                    const int hh = EPW == 4 ? q : h, c0 = s * 64 + hh * 32;
                    const bool mine = c0 < a.N;  // uniform in a warp
                    float v[32];
                    if (mine) tmem_ld32(lane_base + (uint32_t)c0, v);
                    if (s == nsteps - 1 && q == NH - 1) {  // the accumulator has been read by this warp
                        tc_fence_before();
                        mbar_arrive(&pipe->tempty[acc]);
                    }
                    if (!mine) continue;
                    if (MODE == FWD) {
                        const float4 *bp = reinterpret_cast<const float4 *>(pipe->bias + c0);
#pragma unroll
                        for (int k = 0; k < 8; ++k) {
                            const float4 b4 = bp[k];
                            v[4 * k] += b4.x; v[4 * k + 1] += b4.y; v[4 * k + 2] += b4.z; v[4 * k + 3] += b4.w;
                        }
                        uint32_t pk[16], w = 0;
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            pk[j] = a.relu ? relu_pack_bf16x2(v[2 * j], v[2 * j + 1]) : pack_bf16x2(v[2 * j], v[2 * j + 1]);
                            w = gate_bits_add(w, pk[j], j);
                        }
                        if (cell) {
#pragma unroll
                            for (int k = 0; k < 4; ++k) put(stg, hh * 32 + 8 * k, make_uint4(pk[4 * k], pk[4 * k + 1], pk[4 * k + 2], pk[4 * k + 3]));
                        }
                        if (a.out_bits && live) a.out_bits[(((long long)n * a.Hr + y) * a.Wr + x) * (a.N >> 5) + (c0 >> 5)] = w;
                    } else if (cell) {
                        const int gk = s * NH + q;
                        const uint32_t gw = gk == 0 ? gate[0] : (gk == 1 ? gate[1] : (gk == 2 ? gate[2] : gate[3]));
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            uint32_t pk[4];
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                pk[j] = pack_bf16x2(v[8 * k + 2 * j], v[8 * k + 2 * j + 1]) & gate_mask(gw, 4 * k + j);
                            }
                            put(stg, hh * 32 + 8 * k, make_uint4(pk[0], pk[1], pk[2], pk[3]));
                        }
                    }
                }
                store_step(stg, s, a.mapO);
            }
            acc += a.neg;
            if (acc >= nacc) { acc = eg; aph ^= 1u; }
        }
        if (issuer) bulk_wait_all();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, ncols);
    }
}

template <int MODE, int GC, int KS, int EPW>
__global__ void __maxnreg__(96) conv_halo_kernel(const __grid_constant__ Args a) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    halo_body<MODE, GC, KS, EPW, false>(a, First{}, nullptr, smem_raw);
}

// The input gradient of the second convolution and from it, on chip, the weight gradient of the first one, which is all it is for: the
// gradient of the first layer's output, the largest of all, does not go through HBM (2.5 GB of writes and reads at 4096 rows of
// 160 x 120 and 32 channels).  Its tiles' rows go into a ring of pixels in the order of the image, builder warps make the windows
// of the frames, and two warps sum runs of pixels (mma.sync, as conv1_wgrad_mma_kernel: same bits).  What bounds it: the epilogue,
// whose two groups need 720 of the 800 cycles that 128 pixels take; the chain of a run needs 500, the tensor core 215.  Nothing is near
// a limit of the chip (counters at 1024 rows: 2.0 instructions per cycle, shared memory's pipe 30 %, tensor pipe 25 %, DRAM 21 %).
// Measured at that size: 330 + 290 us -> 460, a minibatch 3.22 -> 3.12 ms.
// (depth is the last argument: a prepared launch is made again with other frames.)
constexpr int kFirstThreads = (10 + kBuildWarps + kUnits) * 32;
template <int KS>
__global__ void __launch_bounds__(kFirstThreads, 1) conv_halo_first_kernel(const __grid_constant__ Args a, const __grid_constant__ First f, const __half *depth) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    halo_body<DG, kFirstC, KS, 4, true>(a, f, depth, smem_raw);
}

// --------------------------------------------------------------------- host ----

template <int MODE, int GC, int KS, int EPW>
int launch_one(const Args &a, cudaStream_t st) {
    static PerDevice<bool> set;
    const auto fn = conv_halo_kernel<MODE, GC, KS, EPW>;
    PPO_TRY(ppo_once_per_device(set, [&] { return ppo_allow_smem(fn, kSmemMax); }));
    const int ctas = ppo_num_sms() * a.per_sm;
    return ppo_launch(fn, dim3((unsigned)(a.tiles < ctas ? a.tiles : ctas)), dim3((2 + a.neg * EPW) * 32), a.smem, st, a);
}

template <int MODE, int GC, int EPW>
int launch_ks(const Args &a, cudaStream_t st) {
    const int ks = a.CB >> 4;
    if (ks == 4) return launch_one<MODE, GC, 4, EPW>(a, st);
    return ks == 2 ? launch_one<MODE, GC, 2, EPW>(a, st) : launch_one<MODE, GC, 1, EPW>(a, st);
}

template <int MODE, int GC>
int launch_epw(const Args &a, cudaStream_t st) {
    return a.epw == 4 ? launch_ks<MODE, GC, 4>(a, st) : launch_ks<MODE, GC, 8>(a, st);
}

int launch(const Args &a, int mode, int GC, cudaStream_t st) {
    if (mode == FWD) return GC == 64 ? launch_epw<FWD, 64>(a, st) : (GC == 32 ? launch_epw<FWD, 32>(a, st) : launch_epw<FWD, 16>(a, st));
    if (mode == FWD_LN) return launch_ks<FWD_LN, 32, 4>(a, st);
    return GC == 64 ? launch_epw<DG, 64>(a, st) : (GC == 32 ? launch_epw<DG, 32>(a, st) : launch_epw<DG, 16>(a, st));
}

// Channels per chunk of a C-channel source, or 0.
int chunk_of(int C) { return C % 64 == 0 ? 64 : (C % 32 == 0 ? 32 : (C % 16 == 0 ? 16 : 0)); }

}  // namespace

int halo_conv_fwd(const ConvGeom &g, const bf16 *X, const bf16 *W, const FwdEpilogue &e, int32_t *status, cudaStream_t st) {
    if (!status || g.k != 3 || g.pad != 1 || g.Hi < 2 || g.Wi < 2) return PPO_ERR_UNSUPPORTED;
    if (!e.out || (e.ldo && e.ldo != g.Co) || g.Co % 16 != 0 || g.Co > 256) return PPO_ERR_UNSUPPORTED;
    // Outputs that are no multiple of 32 leave in groups of 16 columns; gate bits and layer normalisation work on 32.  (32 -> 48
    // channels, 1024 rows of 31 x 38: tap boxes 37 us, here 25; 16 -> 48, 384 rows of 96 x 117: 92 and 53.)
    if (g.Co % 32 != 0 && (e.out_bits || e.ln_gamma)) return PPO_ERR_UNSUPPORTED;
    const int CB = chunk_of(g.Ci);
    if (CB == 0 || CB != g.Ci || (size_t)9 * g.Ci * g.Co * 2 > 160 * 1024) return PPO_ERR_UNSUPPORTED;
    // 128 outputs of 64 channels: the weights leave no room for the next tile's planes, and tap boxes whose tiles go in pairs are shorter
    // (4096 rows of 15 x 20 outputs 253 us here, 221 there; of 30 x 40 1043 and 900).  With layer normalisation it is the other way
    // round (512 rows of 8 x 10 outputs 22 and 28 us: their epilogue walks each row three times and is the longer side there).
    if (CB == 64 && g.Co >= 128 && !e.ln_gamma && tma_fwd_in_pairs(g)) return PPO_ERR_UNSUPPORTED;
    Args a = {};
    a.CB = CB;
    a.rb = CB * 2;
    a.nchunks = 1;
    a.N = g.Co;
    a.nplanes = a.nloads = 4;
    a.nwl = 9;
    a.w_box = (uint32_t)(g.Co * a.rb);
    a.w_chunk = 9u * a.w_box;
    a.ln_gamma = e.ln_gamma;
    if (!plan(a, g.Wo, g.Ho, g.B)) return PPO_ERR_UNSUPPORTED;
    for (int p = 0; p < 4; ++p) {
        const int py = p >> 1, px = p & 1;
        Plane &pl = a.planes[p];
        for (int ky = 0; ky < 3; ++ky)
            for (int kx = 0; kx < 3; ++kx) {
                if ((ky == 1 ? 0 : 1) != py || (kx == 1 ? 0 : 1) != px) continue;
                const int t = ky * 3 + kx;
                a.ops[t] = {(uint32_t)(((ky == 2 ? 1 : 0) * a.Wp + (kx == 2 ? 1 : 0)) * a.rb) >> 4, (uint32_t)t * a.w_box >> 4, 0u,
                            instr_desc(128, a.N, 0, 0)};
                a.wl[t] = {t * g.Ci, (uint32_t)t * a.w_box};
            }
        pl.ox = -px;
        pl.oy = -py;
        const int rows = a.I > 1 ? a.R + 1 : a.R + py;
        pl.bytes = (uint32_t)(a.I * rows * a.Wp * a.rb);
        const long long dims[4] = {g.Ci, (g.Wi - px + 1) / 2, (g.Hi - py + 1) / 2, g.B};
        const long long str[3] = {4ll * g.Ci, 4ll * g.Wi * g.Ci, 2ll * g.Hi * g.Wi * g.Ci};
        const int box[4] = {CB, a.Wp, rows, a.I};
        const int s = make_map_strided(&a.mapA[p], X + ((size_t)py * g.Wi + px) * g.Ci, 4, dims, str, box);
        if (s != PPO_OK) return s;
    }
    {
        const long long dims[2] = {g.K(), g.Co}, str[1] = {2ll * g.K()};
        const int box[2] = {CB, a.N};
        const int s = make_map_strided(&a.mapW, W, 2, dims, str, box);
        if (s != PPO_OK) return s;
    }
    const int GC = g.Co % 64 == 0 && !e.ln_gamma ? 64 : (g.Co % 32 == 0 ? 32 : 16);
    const long long dims[4] = {g.Co, g.Wo, g.Ho, g.B};
    const long long str[3] = {2ll * g.Co, 2ll * g.Wo * g.Co, 2ll * g.Ho * g.Wo * g.Co};
    const int box[4] = {GC, a.Wt, a.R, a.I};
    int s = make_map_strided(&a.mapO[0], e.out, 4, dims, str, box);
    if (s != PPO_OK) return s;
    a.bias = e.bias;
    a.relu = e.relu;
    a.out_bits = e.out_bits;
    if (e.out_bits && !e.relu) return PPO_ERR_UNSUPPORTED;
    if (e.ln_gamma) {
        if (!e.ln_beta || !e.ln_xhat || !e.ln_rstd || !e.relu) return PPO_ERR_UNSUPPORTED;
        s = make_map_strided(&a.mapX, e.ln_xhat, 4, dims, str, box);
        if (s != PPO_OK) return s;
        a.ln_beta = e.ln_beta;
        a.ln_rstd = e.ln_rstd;
    }
    a.status = status;
    return launch(a, e.ln_gamma ? FWD_LN : FWD, GC, st);
}

// Shape part of the input gradient's arguments; false where the layer is not covered.
static bool dgrad_shape(Args &a, const ConvGeom &g, int ldy, int wt_ld) {
    if (g.k != 3 || g.pad != 1 || g.Hi < 2 || g.Wi < 2 || ldy != g.Co) return false;
    if (g.Ci != 16 && g.Ci != 32 && g.Ci != 64) return false;
    const int CB = chunk_of(g.Co);
    if (CB == 0 || wt_ld < g.Co || wt_ld % 8 != 0 || (size_t)9 * g.Ci * g.Co * 2 > 160 * 1024) return false;
    a.CB = CB;
    a.rb = CB * 2;
    a.nchunks = g.Co / CB;
    a.N = 4 * g.Ci;
    a.nplanes = 1;
    a.nloads = a.nchunks;
    a.w_box = (uint32_t)(g.Ci * a.rb);
    a.w_chunk = 9u * a.w_box;
    return a.nchunks <= kMaxSlots;
}
static bool plan_dgrad(Args &a, const ConvGeom &g, int ldy, int wt_ld, const DgradEpilogue &e) {
    if (!e.out || e.out_f32 || e.ksplit > 1 || !e.mask_bits) return false;
    return dgrad_shape(a, g, ldy, wt_ld) && plan(a, (g.Wi + 1) / 2, (g.Hi + 1) / 2, g.B);
}

bool halo_dgrad_covers(const ConvGeom &g, int ldy, int wt_ld, const DgradEpilogue &e) {
    if (g.k != 3) return false;
    Args a = {};
    return plan_dgrad(a, g, ldy, wt_ld, e);
}

// The four parity classes (ph, pw) of input pixels (2y + ph, 2x + pw) side by side in the order 00, 01, 11, 10: the
// classes that have a tap at a given shift of dY are then neighbours (all four at (0, 0), 01 | 11 at (0, 1), 11 | 10 at
// (1, 0), 11 at (1, 1)), so every shift is one MMA of just those columns and no product with a zero weight is formed.
static constexpr int cls_ph[4] = {0, 0, 1, 1}, cls_pw[4] = {0, 1, 1, 0};

// What the planned tiles read.
static int dgrad_operands(Args &a, const ConvGeom &g, const bf16 *dY, const bf16 *Wt, int wt_ld) {
    const int CB = a.CB;
    int nb = 0, no = 0;
    for (int dy = 0; dy < 2; ++dy)
        for (int dx = 0; dx < 2; ++dx) {
            const int first = nb;
            int c0 = -1;
            for (int c = 0; c < 4; ++c) {
                if (cls_ph[c] < dy || cls_pw[c] < dx) continue;
                if (c0 < 0) c0 = c;
                const int tap = (cls_ph[c] + 1 - 2 * dy) * 3 + cls_pw[c] + 1 - 2 * dx;
                a.wl[nb] = {tap * wt_ld, (uint32_t)nb * a.w_box};
                ++nb;
            }
            a.ops[no++] = {(uint32_t)((dy * a.Wp + dx) * a.rb) >> 4, (uint32_t)first * a.w_box >> 4, (uint32_t)(c0 * g.Ci),
                           instr_desc(128, (nb - first) * g.Ci, 0, 0)};
        }
    a.nwl = nb;
    a.planes[0] = {0, 0, (uint32_t)(a.I * a.Rp * a.Wp * a.rb)};
    {
        const long long dims[4] = {g.Co, g.Wo, g.Ho, g.B};
        const long long str[3] = {2ll * g.Co, 2ll * g.Wo * g.Co, 2ll * g.Ho * g.Wo * g.Co};
        const int box[4] = {CB, a.Wp, a.Rp, a.I};
        int s = make_map_strided(&a.mapA[0], dY, 4, dims, str, box);
        if (s != PPO_OK) return s;
        const long long wd[2] = {9ll * wt_ld, g.Ci}, ws[1] = {18ll * wt_ld};
        const int wb[2] = {CB, g.Ci};
        s = make_map_strided(&a.mapW, Wt, 2, wd, ws, wb);
        if (s != PPO_OK) return s;
    }
    a.Hi = g.Hi;
    a.Wi = g.Wi;
    return PPO_OK;
}

int halo_conv_dgrad(const ConvGeom &g, const bf16 *dY, int ldy, const bf16 *Wt, int wt_ld, const DgradEpilogue &e,
                    int32_t *status, cudaStream_t st) {
    Args a = {};
    if (!status || !plan_dgrad(a, g, ldy, wt_ld, e)) return PPO_ERR_UNSUPPORTED;
    PPO_TRY(dgrad_operands(a, g, dY, Wt, wt_ld));
    for (int c = 0; c < 4; ++c) {
        const int ph = cls_ph[c], pw = cls_pw[c];
        const long long dims[4] = {g.Ci, (g.Wi - pw + 1) / 2, (g.Hi - ph + 1) / 2, g.B};
        const long long str[3] = {4ll * g.Ci, 4ll * g.Wi * g.Ci, 2ll * g.Hi * g.Wi * g.Ci};
        const int box[4] = {g.Ci, a.Wt, a.R, a.I};
        const int s = make_map_strided(&a.mapO[c], e.out + ((size_t)ph * g.Wi + pw) * g.Ci, 4, dims, str, box);
        if (s != PPO_OK) return s;
    }
    a.mask_bits = e.mask_bits;
    a.status = status;
    return launch(a, DG, g.Ci, st);
}

// Where it pays: first layers of 3x3 and 32 channels, second ones of 64 or 32 (one chunk), from 4 M pixels of the first layer, in tiles of
// that many of them on average.  Backward passes of three layers, us, the two kernels -> this one, by output channels of the second:
//   channels, 4 M pixels of 160 x 120 and of 320 x 240 frames   64: 350 -> 321, 356 -> 326; 32: 258 -> 245, 256 -> 242; 16: 404 -> 414,
//            408 -> 412; 48 (three chunks): 555 -> 565, 597 -> 598; 128 (two, in smaller tiles): 485 -> 500, 495 -> 626
//   tiles, 4 M pixels   64: 255 to 262 pixels (258 x 182, 262 x 196) 361 -> 367, 367 -> 369; 336 and 344 (84 x 64, 86 x 63) 367 -> 373, 367
//            -> 369; from 350 on 3 to 14 % less (30 sizes of frames; one alike).  32: 286 to 345 (52 x 44, 60 x 45, 310 x 230) 307 -> 315,
//            287 -> 305, 260 -> 270; 353 to 360 (530 x 31, 92 x 61, 60 x 48) 270 -> 287, 273 -> 283, 285 -> 293; 380 and 385 (100 x 75,
//            88 x 70) 281 -> 281, 275 -> 277; from 390 on 0 to 8 % less.  An epilogue group takes its time per tile, the two kernels
//            theirs per pixel.
//   pixels, 64   19.7 M (160 x 120) 1460 -> 1330, 6.7 M (130 x 100) 10 less of a minibatch of 870, 1.4 M (84 x 64) 6 more of 280
// 5x5 windows (twice the fragments, 2.5 times the loads of a builder) take longer than the two kernels at all sizes, and so do 16 channels
// of the first layer: half as much dX to keep out of HBM for the same chain.
static bool first_shape(Args &a, First &f, const ConvGeom &g, int ldy, int wt_ld, const uint32_t *mask_bits, const FirstGrad &q) {
    if (q.k != kFirstK || g.Ci != kFirstC || (g.Co != 32 && g.Co != 64) || !mask_bits || q.Wf % 2 != 0) return false;
    const long long M = (long long)g.B * g.Hi * g.Wi;
    if (M < 4000000 || M > 0x7fff0000ll) return false;  // (pixels are 32-bit numbers here)
    return dgrad_shape(a, g, ldy, wt_ld) && plan_first(a, f, g.Hi, g.Wi, g.B) && M >= (g.Co == 64 ? 350ll : 390ll) * a.tiles;
}

template <int KS>
static int launch_first(const Args &a, const First &f, const __half *depth, cudaStream_t st) {
    const int sms = ppo_num_sms();
    static PerDevice<bool> set;
    const auto fn = conv_halo_first_kernel<KS>;
    PPO_TRY(ppo_once_per_device(set, [&] { return ppo_allow_smem(fn, kSmemMax); }));
    return ppo_launch(fn, dim3((unsigned)(f.blocks < sms ? f.blocks : sms)), dim3(kFirstThreads), a.smem, st, a, f, depth);
}

int halo_dgrad_first(const ConvGeom &g, const bf16 *dY, int ldy, const bf16 *Wt, int wt_ld, const uint32_t *mask_bits, const FirstGrad &q,
                     const __half *depth, int32_t *status, cudaStream_t st) {
    Args a = {};
    First f = {};
    if (!status || !ppo_aligned(depth, 4) || !first_shape(a, f, g, ldy, wt_ld, mask_bits, q)) return PPO_ERR_UNSUPPORTED;
    PPO_TRY(dgrad_operands(a, g, dY, Wt, wt_ld));
    a.mask_bits = mask_bits;
    a.status = status;
    f.Hf = q.Hf;
    f.Wh = q.Wf / 2;
    f.M = g.B * g.Hi * g.Wi;
    f.px_per_warp = q.px_per_warp;
    f.blocks = q.blocks;
    f.part = q.part;
    return a.CB == 64 ? launch_first<4>(a, f, depth, st) : launch_first<2>(a, f, depth, st);
}

// Tiles of the halo kernels (conv_halo.cu) and the division of an SM's memory that goes with them.  Plain C++.
#pragma once
#include <cuda.h>
#include <stddef.h>
#include <stdint.h>

#include "conv1_window.h"

#ifdef __CUDACC__
#define PPO_HALO_FN __host__ __device__ constexpr
#else
#define PPO_HALO_FN constexpr
#endif

namespace halo {

constexpr int kMaxSlots = 8;
constexpr int kMaxGroups = 8;   // row groups of the ring between the input gradient and the first layer's weight gradient
constexpr int kWinStages = 4;   // stages of window tiles, of four trips of 32 pixels each
constexpr int kTrip = 32, kStagePx = 4 * kTrip;
constexpr int kBuildWarps = 8;  // in two sets of four
constexpr int kFirstK = 3, kFirstC = 32;  // of the first layer: 3x3, 32 channels
static_assert(Window<kFirstK>::TP == 16, "one row of fragments");
constexpr int kUnits = kFirstC / 16;  // warps that sum
constexpr int kMaxOps = 9;
constexpr size_t kSmemMax = 227 * 1024;

// One tap of a plane: CB / 16 MMAs over the channels of a chunk.
struct Op {
    uint32_t a16;    // start of the A rows inside the plane's box, in 16-byte units
    uint32_t b16;    // start of the weights of chunk 0, in 16-byte units
    uint32_t dcol;   // first accumulator column
    uint32_t idesc;  // instruction descriptor (column count)
};

struct Plane {
    int ox, oy;      // box origin relative to the tile's first output cell
    uint32_t bytes;  // of its box
};

struct WLoad {       // one box of weights: rows of one tap (all chunks loaded one after the other)
    int k0;          // column of the weight matrix, without the chunk
    uint32_t off;    // destination of chunk 0
};

struct Args {
    CUtensorMap mapA[4];    // planes
    CUtensorMap mapW;
    CUtensorMap mapO[4];    // output groups (forward: one map, the group is the first coordinate)
    CUtensorMap mapX;       // normalised values
    Op ops[kMaxOps];
    Plane planes[4];
    WLoad wl[kMaxOps];
    int nplanes, nwl, nchunks, nloads, CB, rb;
    uint32_t w_chunk;       // bytes of the weights of one chunk
    uint32_t w_box;         // bytes of one box of weights
    uint32_t slot_bytes, slots_bytes;  // of one slot; of all of them, rounded up
    uint32_t stg_bytes;     // of a staging buffer
    int stg_row;            // of a row of it, over all its output groups
    int epw;                // warps of an epilogue group
    int slots, nbuf, neg;   // slots, staging buffers per epilogue group, epilogue groups
    int Wt, R, I, Wp, Rp;   // tile: Wt x R outputs of I images; cells per box row and box rows per image
    int xsegs, ysegs, tiles;
    int Hr, Wr, B;          // grid of outputs (forward) or of 2x2 input blocks (input gradient)
    int N;                  // accumulator columns
    int acc_cols, nacc;
    int Hi, Wi;             // input gradient: the image that is written
    const float *bias;
    int relu;
    uint32_t *out_bits;
    const uint32_t *mask_bits;
    const float *ln_gamma, *ln_beta;
    float *ln_rstd;
    int per_sm;             // CTAs an SM holds
    size_t smem;
    int32_t *status;
};

// The first layer's weight gradient behind the input gradient of the second (see first_sums).
struct First {
    int Hf, Wh;             // frame rows, and 32-bit words of one
    int M, px_per_warp;     // pixels of the first layer's output; of one of the eight runs that make a block of partial sums
    int blocks;             // blocks of partial sums, dealt out over the CTAs
    int groups, ring_px;    // row groups in flight, pixels of the ring
    int group_px, last_px;  // pixels of a group of 2 R rows, and of the last one of an image
    uint32_t ring_bytes;
    float *part;            // [block][C1 k k (dW order) | C1 (db)]
};

struct Pipe {
    uint64_t full[kMaxSlots], empty[kMaxSlots], tfull[4], tempty[4], wfull;
    uint32_t tmem_slot;
    int abort_flag;
    alignas(16) float bias[256], gamma[256], beta[256];
};
// With the ring's barriers, which take no room in the kernels without one: 192 bytes more cost one in ten plain forward grids of 32 -> 48
// channels a slot.
struct FirstPipe : Pipe {
    uint64_t gfull[kMaxGroups], gempty[kMaxGroups], pfull[kWinStages], pempty[kWinStages];
};


inline uint32_t stage_rows_bytes(int rows, int row_bytes) { return ((uint32_t)(rows * row_bytes) + 1023u) & ~1023u; }

// Tile rectangle whose loads (`loads` slots) and staging buffers (`bufs`) fit into `room` bytes: fewest tiles over the
// whole grid, then fewest loaded cells.  The M rows of a tile (halo cells included, except behind its last row) have to
// fit into the 128 rows of an MMA.
inline bool choose_tile(Args &a, int Wr, int Hr, int B, size_t room, int loads, int bufs) {
    long long best_t = -1, best_c = 0;
    for (int xs = 1; xs <= Wr && xs <= 64; ++xs) {
        const int Wt = (Wr + xs - 1) / xs, Wp = Wt + 1;
        if (Wt > 128) continue;
        int top = (128 - Wt) / Wp + 1;
        if (top > Hr) top = Hr;
        for (int R = top; R >= 1; --R) {
            const int ysegs = (Hr + R - 1) / R;
            if (R < top && (Hr + R) / (R + 1) == ysegs) continue;  // a taller tile makes as few segments
            const int Re = (Hr + ysegs - 1) / ysegs;
            int I = 1;
            if (ysegs == 1 && xs == 1) {
                const int per = (Re + 1) * Wp, last = (Re - 1) * Wp + Wt;
                I = 1 + (128 - last) / per;
                if (I > B) I = B;
            }
            auto fits = [&](int img) {
                const size_t slot = ((size_t)img * (Re + 1) * Wp * a.rb + 127) & ~size_t(127);
                return (size_t)loads * slot + (size_t)bufs * stage_rows_bytes(img * Re * Wt, a.stg_row) <= room;
            };
            while (I > 1 && !fits(I)) --I;
            if (!fits(I)) continue;
            const long long tiles = (long long)((B + I - 1) / I) * ysegs * ((Wr + Wt - 1) / Wt);
            const long long cells = tiles * I * (Re + 1) * Wp;
            if (best_t < 0 || tiles < best_t || (tiles == best_t && cells < best_c)) {
                best_t = tiles; best_c = cells;
                a.Wt = Wt; a.R = Re; a.I = I;
            }
        }
    }
    if (best_t < 0 || best_t > 0x3fffffff) return false;
    a.Wp = a.Wt + 1;
    a.Rp = a.R + 1;
    a.xsegs = (Wr + a.Wt - 1) / a.Wt;
    a.ysegs = (Hr + a.R - 1) / a.R;
    a.tiles = (int)best_t;
    a.Hr = Hr; a.Wr = Wr; a.B = B;
    return true;
}

// Division of shared and tensor memory, and the tile that goes with it.  A tile's loads (four planes, or one box per chunk)
// are all held at once.  Two CTAs per SM, one epilogue group each, where the weights and a full-sized tile's loads and
// staging fit into half of it; else one CTA with two epilogue groups, if need be with a smaller tile.  The epilogue is
// the longest chain of a tile (read the accumulator, convert, stage, hand over, wait until the copy engine has read the
// buffer), so it is what the second CTA or group is for; a CTA's only group stages into two buffers if they fit.  What
// room is left goes to more slots, for the next tile's loads.
inline bool plan(Args &a, int Wr, int Hr, int B) {
    const size_t w = ((size_t)a.nchunks * a.w_chunk + 1023) & ~size_t(1023);
    const size_t fixed = w + sizeof(Pipe) + 1024 + 1024;  // alignment of the base and behind the slots
    a.stg_row = a.N == 32 && !a.ln_gamma ? 64 : 128;  // 64 columns, or 32 and the normalised values beside the outputs
    a.acc_cols = 32;
    while (a.acc_cols < a.N) a.acc_cols *= 2;
    const size_t half = kSmemMax / 2 - 512;
    Args best = a;
    if (!choose_tile(best, Wr, Hr, B, size_t(1) << 30, a.nloads, 1)) return false;
    for (int two = a.N <= 128 ? 1 : 0; two >= 0; --two) {
        const size_t room = two ? half : kSmemMax;
        if (fixed >= room) continue;
        // Four-warp groups (see the top of the file) cost a second staging buffer: worth it for the input gradient (32
        // channels: 1.49 -> 1.29 ms), a single step of 32 columns and normalised rows; a plain forward tile of 64 columns and
        // more wants the room for its next two planes (1.30 against 1.48 ms).
        a.epw = a.ln_gamma || (two && (a.nloads != 4 || a.N == 32)) ? 4 : 8;
        a.nacc = (two ? 256 : 512) / a.acc_cols;
        if (a.nacc > 4) a.nacc = 4;
        if (a.nacc < 2) continue;
        a.neg = two ? 8 / a.epw : 2;
        if (a.neg > a.nacc) a.neg = a.nacc;  // a group has accumulators of its own
        const int least = a.nloads == 4 || two ? a.nloads : a.nloads + 1;
        if (!choose_tile(a, Wr, Hr, B, room - fixed, least, a.neg)) continue;
        if (two && a.tiles > best.tiles) continue;  // no smaller tile for the sake of a second CTA
        a.slot_bytes = (uint32_t)(a.I * a.Rp * a.Wp * a.rb + 127) & ~127u;
        a.stg_bytes = stage_rows_bytes(a.I * a.R * a.Wt, a.stg_row);
        // a second staging buffer comes before more slots where a step stages twice (normalised values, then outputs) or a
        // tile is one load; a plain forward tile wants its next two planes first (32 -> 64 channels: 1.45 -> 1.29 ms)
        const int before = a.nloads == 4 && !a.ln_gamma ? a.nloads + 2 : least;
        a.nbuf = two && (size_t)before * a.slot_bytes + 2 * (size_t)(a.neg * a.stg_bytes) <= room - fixed ? 2 : 1;
        a.slots = (int)((room - fixed - (size_t)(a.nbuf * a.neg) * a.stg_bytes) / a.slot_bytes);
        if (a.slots > kMaxSlots) a.slots = kMaxSlots;
        a.slots_bytes = ((uint32_t)a.slots * a.slot_bytes + 1023u) & ~1023u;
        a.smem = a.slots_bytes + w + (size_t)(a.nbuf * a.neg) * a.stg_bytes + sizeof(Pipe) + 1024;
        a.per_sm = two ? 2 : 1;
        return true;
    }
    return false;
}

// Hand-overs of the ring.  A wait by parity sees a phase only until the next one of the same barrier is complete, and takes the phase
// before the last for it: a waiter may be neither two phases behind nor two ahead.
//
// Row groups are given back by one builder, in order.  An epilogue group that has tiles in every second row group only (one tile each)
// looks at a barrier at every second use where the number of row groups in flight is odd, and leans on this: what it saw given back
// for its last tile came behind all that was given back before.
PPO_HALO_FN bool ring_gives_back(int builder) { return builder == 0; }
// End of what has been summed, in pixels of the run, when a builder is let into stage s.
PPO_HALO_FN int ring_summed(int s) { return (s - kWinStages + 1) * kStagePx; }
// Pixels of the run that a builder waits for before it hands its trip of stage s over: those of the whole stage, which is handed over with
// the last of its four trips anyway.  With its own trip's alone a row group behind them that ends in the same stage could be summed,
// given back and filled again before this builder, by then stages behind, looked at it for the first time.
PPO_HALO_FN int ring_needs(int s, int total) {
    const int end = (s + 1) * kStagePx;
    return end < total ? end : total;
}

// Division of shared memory and the tile for the input gradient whose output stays on chip: room for the loads of a tile and one more,
// and a ring of at least two row groups; fewest tiles, then the lowest groups.
inline bool plan_first(Args &a, First &f, int Hi, int Wi, int B) {
    const int Wr = (Wi + 1) / 2, Hr = (Hi + 1) / 2, C1 = kFirstC;
    const size_t w = ((size_t)a.nchunks * a.w_chunk + 1023) & ~size_t(1023);
    const size_t patch = (size_t)kWinStages * kStagePx * Window<kFirstK>::TP * 2;
    const size_t fixed = w + patch + sizeof(FirstPipe) + 2048;
    if (fixed >= kSmemMax) return false;
    const size_t room = kSmemMax - fixed;
    auto ring_of = [&](int groups, int R) -> size_t {  // whole stages
        return (size_t)((groups * 2 * R * Wi + kStagePx - 1) / kStagePx * kStagePx) * C1 * 2;
    };
    auto slot_of = [&](int R, int Wp) -> size_t { return ((size_t)(R + 1) * Wp * a.rb + 127) & ~size_t(127); };
    long long best_t = -1;
    int least = 0;
    for (int xs = 1; xs <= Wr && xs <= 64; ++xs) {
        const int Wt = (Wr + xs - 1) / xs, Wp = Wt + 1;
        if (Wt > 128) continue;
        int top = (128 - Wt) / Wp + 1;
        if (top > Hr) top = Hr;
        for (int R = top; R >= 1; --R) {
            const int ysegs = (Hr + R - 1) / R, Re = (Hr + ysegs - 1) / ysegs;
            if ((Hr + Re - 1) / Re != ysegs) continue;
            // Groups in flight.  A builder that waits in stage s stands behind a stage (s or, of the other set, s - 1) in which all was
            // given back that ended kWinStages stages before that: at most this many stages' pixels, of whole groups, are not.
            const int ahead = kWinStages + 1;
            int touch = 2;
            for (int i = 0; i < ysegs; ++i) {
                int sum = 0, n = 2;
                for (int k = i;; k = k + 1 == ysegs ? 0 : k + 1, ++n) {
                    sum += (k == ysegs - 1 ? Hi - 2 * Re * (ysegs - 1) : 2 * Re) * Wi;
                    if (sum > ahead * kStagePx) break;
                }
                touch = n > touch ? n : touch;
            }
            if (touch > kMaxGroups) continue;
            if ((size_t)(a.nloads + 1) * slot_of(Re, Wp) + 1024 + ring_of(touch, Re) > room) continue;
            const long long tiles = (long long)B * ysegs * ((Wr + Wt - 1) / Wt);
            if (best_t < 0 || tiles < best_t || (tiles == best_t && Re < a.R)) {
                best_t = tiles;
                a.Wt = Wt; a.R = Re;
                least = touch;
            }
        }
    }
    if (best_t < 0 || best_t > 0x3fffffff) return false;
    a.I = 1;
    a.Wp = a.Wt + 1;
    a.Rp = a.R + 1;
    a.xsegs = (Wr + a.Wt - 1) / a.Wt;
    a.ysegs = (Hr + a.R - 1) / a.R;
    a.tiles = (int)best_t;
    a.Hr = Hr; a.Wr = Wr; a.B = B;
    a.epw = 4;
    a.neg = 2;
    a.acc_cols = a.N;
    a.nacc = 4;
    a.slot_bytes = (uint32_t)slot_of(a.R, a.Wp);
    f.groups = least;
    while (f.groups < 3 && (size_t)(a.nloads + 1) * a.slot_bytes + 1024 + ring_of(f.groups + 1, a.R) <= room) ++f.groups;
    f.group_px = 2 * a.R * Wi;
    f.last_px = (Hi - 2 * a.R * (a.ysegs - 1)) * Wi;
    f.ring_bytes = (uint32_t)ring_of(f.groups, a.R);
    f.ring_px = (int)(f.ring_bytes / (C1 * 2));
    a.slots = (int)((room - 1024 - f.ring_bytes) / a.slot_bytes);
    if (a.slots > kMaxSlots) a.slots = kMaxSlots;
    a.slots_bytes = ((uint32_t)a.slots * a.slot_bytes + 1023u) & ~1023u;
    a.smem = a.slots_bytes + w + f.ring_bytes + patch + sizeof(FirstPipe) + 1024;
    return true;
}

}  // namespace halo

// Windows of the first layer (stride 2, one channel) as aligned pairs of fp16 frame pixels, for the kernels that form its output
// (conv1_tc.cu) and its weight gradient (encoder.cu and, behind the second layer's input gradient, conv_halo.cu: the same sums bit for bit).
#pragma once
#include <stdint.h>

// Pair q of window row kh covers frame columns 2 ow - P - ODD + 2 q (+1); element e of it is kernel column 2 q + e - ODD, which for one
// element per row lies outside 0 .. KS-1.
template <int KS>
struct Window {
    static constexpr int P = KS / 2, ODD = P & 1, NP = (KS + ODD + 1) / 2, KW = KS * NP;  // pairs of a row, of the window
    // rows of the weight gradient: one per pair element and one for the bias
    static constexpr int TP = (2 * KW + 1 + 15) / 16 * 16;
};

#ifdef __CUDACC__
#include "common.cuh"

// A lane's walk through the pixels of the first layer's output, without divisions behind the first.
template <int KS>
struct WindowWalk {
    using WN = Window<KS>;
    int ow, oh;
    long long b;
    __device__ __forceinline__ void init(long long m, int Wo, int Ho) {
        ow = (int)(m % Wo);
        const long long t = m / Wo;
        oh = (int)(t % Ho);
        b = t / Ho;
    }
    __device__ __forceinline__ void advance(int d_ow, int d_oh, int Wo, int Ho) {  // by d_oh rows and d_ow < Wo pixels
        ow += d_ow;
        if (ow >= Wo) { ow -= Wo; ++oh; }
        oh += d_oh;
        while (oh >= Ho) { oh -= Ho; ++b; }
    }
    // The window's pairs, zero outside the frame (Hi rows of Wh pairs); all zero if not live.  A pair outside is a predicated load that leaves
    // its zero.
    __device__ __forceinline__ void fetch(const uint32_t *frames, int Hi, int Wh, bool live, uint32_t (&raw)[WN::KW]) const {
        const int pw0 = ow - (WN::P + WN::ODD) / 2, ih0 = 2 * oh - WN::P;
        const uint32_t *row = frames + ((b * Hi + ih0) * Wh + pw0);
        bool cok[WN::NP];
#pragma unroll
        for (int q = 0; q < WN::NP; ++q) cok[q] = live && (unsigned)(pw0 + q) < (unsigned)Wh;
#pragma unroll
        for (int kh = 0; kh < KS; ++kh) {
            const bool rok = (unsigned)(ih0 + kh) < (unsigned)Hi;
#pragma unroll
            for (int q = 0; q < WN::NP; ++q) {
                raw[kh * WN::NP + q] = 0u;
                if (rok && cok[q]) raw[kh * WN::NP + q] = __ldg(row + q);
            }
            row += Wh;
        }
    }
};

// 16-byte piece c of row r of a tile sits at piece c ^ f(r): rows of 32, 64 or 128 bytes would otherwise put the same piece of several
// rows into the same banks, on the way in as on the way out (ldmatrix reads a column of pieces).
__device__ __forceinline__ int piece_swizzle(int r, int row_bytes) {
    return row_bytes == 128 ? r & 7 : (row_bytes == 64 ? (r >> 1) & 3 : (row_bytes == 32 ? (r >> 2) & 1 : 0));
}

// The window as a row of a tile of [TP] bf16, with a column of ones (the bias gradient) behind it where live; and its way into row r.
template <int KS>
__device__ __forceinline__ void window_row(const uint32_t (&raw)[Window<KS>::KW], bool live, uint32_t (&wv)[Window<KS>::TP / 2]) {
    constexpr int TP = Window<KS>::TP, KW = Window<KS>::KW;
#pragma unroll
    for (int k = 0; k < TP / 2; ++k) wv[k] = 0u;
#pragma unroll
    for (int k = 0; k < KW; ++k) {
        const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&raw[k]));
        wv[k] = pack_bf16x2(f.x, f.y);
    }
    if (live) wv[KW] = 0x00003F80u;  // (1.0, 0) as bf16
}
template <int N>
__device__ __forceinline__ void put_row(uint8_t *row, int r, const uint32_t (&wv)[N]) {
#pragma unroll
    for (int c = 0; c < N / 4; ++c)
        *reinterpret_cast<uint4 *>(row + ((c ^ piece_swizzle(r, N * 4)) * 16)) = make_uint4(wv[4 * c], wv[4 * c + 1], wv[4 * c + 2], wv[4 * c + 3]);
}

__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t addr, uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(addr));
}
__device__ __forceinline__ void mma_bf16_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
#endif

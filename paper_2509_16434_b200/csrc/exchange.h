// Barriers of the exchanges between the layers of a chain (mlp.cu).  Plain C++.
//
// Behind layer l every CTA of a cluster arrives once at barrier `barrier(l)` of every CTA, and whoever reads layer l's columns
// waits there for the phase of parity `parity(l)`.  A wait by parity sees a phase only until the next one of the same barrier is
// complete, and a CTA that owns no columns of a layer arrives for it without its reader having looked at the layer before.  So
// every exchange has a barrier of its own, whose only phase stays complete.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define PPO_EXCHANGE_FN __host__ __device__ constexpr
#else
#define PPO_EXCHANGE_FN constexpr
#endif

struct ChainExchange {
    PPO_EXCHANGE_FN static int barriers(int layers) { return layers - 1; }
    PPO_EXCHANGE_FN static int barrier(int l) { return l; }
    PPO_EXCHANGE_FN static uint32_t parity(int) { return 0u; }
};

// Kernel launches that can be recorded and replayed.
//
// Preparing a launch of the GEMM kernels (tile shapes, up to 64 tensor maps, a few KB of arguments) costs the host several
// microseconds, and a learner makes the same launches with the same arguments over and over.  So the operations of a
// model remember the launches they made under a key of everything the preparation read (shapes and pointers); the next
// call with the same key only enqueues them.
//
// Every kernel launched by ppo_launch starts with grid_wait(): the launch carries the programmatic-serialization attribute, so
// the next kernel of the stream may be set up while the one before it drains, and reads or writes memory only after that
// wait.  (Letting it start earlier still, as soon as every block of the one before it runs, costs 1 to 5 %: the waiting
// blocks take room from the second stream's kernels.)
// Measured: host time of a forward pass of the recurrent policy 140 -> 53 us; TrainPPO of 4 x 1024 rows of 64 x 64, where
// launches and gaps count, 1258 -> 944 us together with the launches that were merged.
#pragma once
#include <tuple>
#include <vector>

#include "common.cuh"
#include "plan_store.h"

// Everything the kernels in front of this one in the stream wrote is visible behind this.
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

struct LaunchRecord {
    const void *fn;
    dim3 grid, block;
    size_t smem;
    bool together;                 // all blocks resident at once (cooperative launch)
    std::vector<char> bytes;       // argument values one after the other
    std::vector<uint32_t> offset;  // where each starts
};

struct PlanKey {
    int op, unused;
    ConvGeom g;
    const void *p[12];
    long long v[6];
};

using Launches = std::vector<LaunchRecord>;

struct ppo_plans : PlanStore<PlanKey, Launches> {
    ppo_plans() : PlanStore(1024) {}  // operations of one model; a few MB of host memory
};

// The record of the operation being prepared on this thread (null: none).
extern thread_local Launches *ppo_recording;

int ppo_enqueue(const void *fn, dim3 grid, dim3 block, size_t smem, bool together, cudaStream_t st, void **argv);

template <typename... P, typename... A>
int ppo_launch_as(bool together, void (*fn)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A... args) {
    static_assert(sizeof...(P) == sizeof...(A), "argument count");
    void *argv[sizeof...(A)];
    int n = 0;
    // converted to the parameter types before their addresses are taken
    std::tuple<std::remove_const_t<P>...> vals(static_cast<std::remove_const_t<P>>(args)...);
    std::apply([&](auto &...v) { ((argv[n++] = (void *)&v), ...); }, vals);
    if (ppo_recording) {
        LaunchRecord r;
        r.fn = reinterpret_cast<const void *>(fn);
        r.grid = grid;
        r.block = block;
        r.smem = smem;
        r.together = together;
        n = 0;
        const size_t sizes[] = {sizeof(P)...};
        for (size_t i = 0; i < sizeof...(P); ++i) {
            r.offset.push_back((uint32_t)r.bytes.size());
            const char *src = static_cast<const char *>(argv[i]);
            r.bytes.insert(r.bytes.end(), src, src + sizes[i]);
        }
        ppo_recording->push_back(std::move(r));
    }
    return ppo_enqueue(reinterpret_cast<const void *>(fn), grid, block, smem, together, st, argv);
}
template <typename... P, typename... A>
int ppo_launch(void (*fn)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A... args) {
    return ppo_launch_as(false, fn, grid, block, smem, st, args...);
}
// For kernels whose blocks wait for one another: the launch fails unless they can all be resident at once.
template <typename... P, typename... A>
int ppo_launch_together(void (*fn)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A... args) {
    return ppo_launch_as(true, fn, grid, block, smem, st, args...);
}

// Enqueues a recorded operation.
int ppo_replay(const Launches &launches, cudaStream_t st);

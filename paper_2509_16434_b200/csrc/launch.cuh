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

// The operation being prepared on this thread.
struct Recording {
    Launches launches;
    bool complete = true;  // false: memory ran out on the way; the launches were made all the same
};
extern thread_local Recording *ppo_recording;  // null: none
void ppo_record(const void *fn, dim3 grid, dim3 block, size_t smem, bool together, void *const *argv, const size_t *sizes, size_t n) noexcept;

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
        const size_t sizes[] = {sizeof(P)...};
        ppo_record(reinterpret_cast<const void *>(fn), grid, block, smem, together, argv, sizes, sizeof...(P));
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

// Enqueues a recorded operation.  last (null: none): what takes the place of the last argument of every launch, last_bytes long; for
// arguments that are no part of the preparation, such as the addresses of results, and of the key neither.
int ppo_replay(const Launches &launches, cudaStream_t st, const void *last = nullptr, size_t last_bytes = 0);

// Recorded launches (see launch.cuh).
#include <tuple>

#include "launch.cuh"

thread_local std::vector<LaunchRecord> *ppo_recording = nullptr;

static const size_t kMaxPlans = 1024;  // of one model; a few MB of host memory

static uint64_t hash_key(const PlanKey &k) {
    uint64_t h = 1469598103934665603ull;
    const char *c = reinterpret_cast<const char *>(&k);
    for (size_t i = 0; i + 8 <= sizeof(k); i += 8) {
        uint64_t w;
        memcpy(&w, c + i, 8);
        h = (h ^ w) * 1099511628211ull;
        h ^= h >> 29;
    }
    return h;
}

int ppo_enqueue(const void *fn, dim3 grid, dim3 block, size_t smem, bool together, cudaStream_t st, void **argv) {
    cudaLaunchConfig_t c = {};
    c.gridDim = grid;
    c.blockDim = block;
    c.dynamicSmemBytes = smem;
    c.stream = st;
    cudaLaunchAttribute at[1];
    if (together) {
        at[0].id = cudaLaunchAttributeCooperative;
        at[0].val.cooperative = 1;
    } else {
        at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[0].val.programmaticStreamSerializationAllowed = 1;
    }
    c.attrs = at;
    c.numAttrs = 1;
    ppo_count_launches(1);
    PPO_CUDA_CHECK(cudaLaunchKernelExC(&c, fn, argv));
    return PPO_OK;
}

PlanEntry *ppo_find_plan(ppo_plans *plans, const PlanKey &key) {
    auto range = plans->map.equal_range(hash_key(key));
    for (auto it = range.first; it != range.second; ++it)
        if (memcmp(&it->second.key, &key, sizeof(key)) == 0) return &it->second;
    return nullptr;
}

int ppo_replay(const PlanEntry &e, cudaStream_t st) {
    for (const LaunchRecord &r : e.launches) {
        void *argv[32];
        const size_t n = r.offset.size();
        if (n > 32) return PPO_ERR_CUDA;
        for (size_t i = 0; i < n; ++i) argv[i] = const_cast<char *>(r.bytes.data()) + r.offset[i];
        const int s = ppo_enqueue(r.fn, r.grid, r.block, r.smem, r.together, st, argv);
        if (s != PPO_OK) return s;
    }
    return PPO_OK;
}

void ppo_store_plan(ppo_plans *plans, const PlanKey &key, std::vector<LaunchRecord> &&launches) {
    if (plans->map.size() >= kMaxPlans) plans->map.clear();
    PlanEntry e;
    e.key = key;
    e.launches = std::move(launches);
    plans->map.emplace(hash_key(key), std::move(e));
}

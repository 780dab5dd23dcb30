// Recorded launches (see launch.cuh).
#include "launch.cuh"

thread_local Recording *ppo_recording = nullptr;

void ppo_record(const void *fn, dim3 grid, dim3 block, size_t smem, bool together, void *const *argv, const size_t *sizes, size_t n) noexcept {
    try {
        LaunchRecord r;
        r.fn = fn;
        r.grid = grid;
        r.block = block;
        r.smem = smem;
        r.together = together;
        for (size_t i = 0; i < n; ++i) {
            r.offset.push_back((uint32_t)r.bytes.size());
            const char *src = static_cast<const char *>(argv[i]);
            r.bytes.insert(r.bytes.end(), src, src + sizes[i]);
        }
        ppo_recording->launches.push_back(std::move(r));
    } catch (...) {
        ppo_recording->complete = false;
    }
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

int ppo_replay(const Launches &launches, cudaStream_t st, const void *last, size_t last_bytes) {
    for (const LaunchRecord &r : launches) {
        void *argv[32];
        const size_t n = r.offset.size();
        if (n > 32) return PPO_ERR_CUDA;
        for (size_t i = 0; i < n; ++i) argv[i] = const_cast<char *>(r.bytes.data()) + r.offset[i];
        if (last) {
            if (n == 0 || r.bytes.size() - r.offset[n - 1] != last_bytes) return PPO_ERR_CUDA;
            argv[n - 1] = const_cast<void *>(last);
        }
        const int s = ppo_enqueue(r.fn, r.grid, r.block, r.smem, r.together, st, argv);
        if (s != PPO_OK) return s;
    }
    return PPO_OK;
}

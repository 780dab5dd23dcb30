// Rollout buffer D on the learner GPU (Algorithm 2): slab carving, write_step, GAE with
// advantage normalisation, and the seeded permutation gather.
#include <atomic>
#include <new>

#include "common.cuh"
#include "launch.cuh"

// ------------------------------------------------------------------ status ----

static __device__ int32_t g_ppo_status;

int32_t *ppo_device_status_ptr() {
    static PerDevice<int32_t *> ptrs;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return nullptr;
    return ptrs.get(dev, []() -> int32_t * {
        void *p = nullptr;
        return cudaGetSymbolAddress(&p, g_ppo_status) == cudaSuccess ? static_cast<int32_t *>(p) : nullptr;
    });
}

static std::atomic<unsigned long long> g_launches{0};

void ppo_count_launches(int n) { g_launches.fetch_add((unsigned long long)n, std::memory_order_relaxed); }

extern "C" uint64_t ppo_launch_count(void) { return g_launches.load(std::memory_order_relaxed); }

int ppo_num_sms() {
    static PerDevice<int> sms;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 148;
    return sms.get(dev, [dev] {
        int n = 0;
        return cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && n > 0 ? n : 148;
    });
}

int ppo_work_sequence(cudaStream_t st, uint64_t *seq) {
    cudaStreamCaptureStatus status;
    unsigned long long id = 0;
    PPO_CUDA_CHECK(cudaStreamGetCaptureInfo(st, &status, &id));
    *seq = status == cudaStreamCaptureStatusNone ? kEagerWork : kEagerWork + 1 + id;  // ids are never given out twice
    return PPO_OK;
}

int ppo_clear_once(uint64_t *made, void *p, size_t bytes, cudaStream_t st) {
    uint64_t seq;
    PPO_TRY(ppo_work_sequence(st, &seq));
    if (*made == seq) return PPO_OK;
    PPO_CUDA_CHECK(cudaMemsetAsync(p, 0, bytes, st));
    ppo_count_launches(1);
    *made = seq;
    return PPO_OK;
}

extern "C" const char *ppo_status_string(int s) {
    switch (s) {
        case PPO_OK: return "ok";
        case PPO_ERR_INVALID_ARG: return "invalid argument";
        case PPO_ERR_SHAPE: return "shape mismatch";
        case PPO_ERR_ALIGN: return "misaligned pointer";
        case PPO_ERR_STATE: return "call out of order";
        case PPO_ERR_CUDA: return "CUDA error";
        case PPO_ERR_TIMEOUT: return "device-side wait timed out";
        case PPO_ERR_UNSUPPORTED: return "unsupported shape";
        default: return "unknown status";
    }
}

extern "C" int ppo_poll_status(void *stream) {
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int32_t *p = ppo_device_status_ptr();
    if (!p) return PPO_ERR_CUDA;
    int32_t host = 0;
    if (cudaMemcpyAsync(&host, p, sizeof(host), cudaMemcpyDeviceToHost, st) != cudaSuccess) return PPO_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return PPO_ERR_CUDA;
    if (host != 0) {
        if (cudaMemsetAsync(p, 0, sizeof(host), st) != cudaSuccess) return PPO_ERR_CUDA;
        if (cudaStreamSynchronize(st) != cudaSuccess) return PPO_ERR_CUDA;
    }
    return host;
}

// ------------------------------------------------------------------ layout ----

static const int kMaxGaeBlocks = 4096;

static bool desc_ok(const ppo_buffer_desc *d) {
    return d && d->N > 0 && d->T > 0 && d->H > 0 && d->W > 0 && d->P > 0 && d->A > 0 &&
           (long long)d->N * d->T < (1ll << 31);
}

static size_t field_bytes(const ppo_buffer_desc *d, int field, int depth_elem) {
    size_t M = (size_t)d->N * d->T;
    switch (field) {
        case PPO_FIELD_DEPTH: return M * d->H * d->W * (size_t)depth_elem;
        case PPO_FIELD_PROPRIO: return M * d->P * 4;
        case PPO_FIELD_ACTION: return M * d->A * 4;
        case PPO_FIELD_LOGP:
        case PPO_FIELD_VALUE:
        case PPO_FIELD_REWARD:
        case PPO_FIELD_ADV:
        case PPO_FIELD_RET: return M * 4;
        case PPO_FIELD_DONE: return M;
        case PPO_FIELD_SCRATCH: return (size_t)kMaxGaeBlocks * 2 * sizeof(double);
        default: return 0;
    }
}

extern "C" size_t ppo_buffer_field_bytes(const ppo_buffer_desc *d, int field, int depth_elem_bytes) {
    if (!desc_ok(d) || field < 0 || field >= PPO_NUM_FIELDS) return 0;
    if (depth_elem_bytes != 2 && depth_elem_bytes != 4) return 0;
    return field_bytes(d, field, depth_elem_bytes);
}

extern "C" size_t ppo_buffer_bytes(const ppo_buffer_desc *d) {
    if (!desc_ok(d)) return 0;
    size_t total = 0;
    for (int f = 0; f < PPO_NUM_FIELDS; ++f) total += ppo_align_up(field_bytes(d, f, 2), 256);
    return total;
}

extern "C" int ppo_buffer_alloc(const ppo_buffer_desc *d, void *dev_storage, size_t bytes, ppo_buffer **out) {
    if (!out) return PPO_ERR_INVALID_ARG;
    *out = nullptr;
    if (!desc_ok(d) || !dev_storage) return PPO_ERR_INVALID_ARG;
    if (!ppo_aligned(dev_storage, 256)) return PPO_ERR_ALIGN;
    if (bytes < ppo_buffer_bytes(d)) return PPO_ERR_SHAPE;
    ppo_buffer *b = new (std::nothrow) ppo_buffer();
    if (!b) return PPO_ERR_INVALID_ARG;
    b->d = *d;
    b->base = static_cast<char *>(dev_storage);
    b->bytes = bytes;
    size_t off = 0;
    for (int f = 0; f < PPO_NUM_FIELDS; ++f) {
        b->field_off[f] = off;
        off += ppo_align_up(field_bytes(d, f, 2), 256);
    }
    b->gae_valid = false;
    b->gae_blocks = 0;
    b->barrier_made = kNotMade;
    *out = b;
    return PPO_OK;
}

extern "C" int ppo_buffer_free(ppo_buffer *b) {
    if (!b) return PPO_ERR_INVALID_ARG;
    delete b;
    return PPO_OK;
}

extern "C" void *ppo_buffer_field_ptr(const ppo_buffer *b, int field) {
    if (!b || field < 0 || field >= PPO_NUM_FIELDS) return nullptr;
    return b->base + b->field_off[field];
}

template <typename T>
static T *slab(const ppo_buffer *b, int field) {
    return reinterpret_cast<T *>(b->base + b->field_off[field]);
}

// -------------------------------------------------------------- write_step ----

struct CopySeg {
    const char *src;
    char *dst;
    unsigned long long bytes;
    uint32_t block_end;  // blocks of the segments up to and including this one
    uint32_t vec;        // 16 or 4 when both ends and the size allow such accesses, else 1
};
struct CopySegs {
    CopySeg s[7];
};

constexpr uint32_t kCopyBlockBytes = 16384;  // per block: four 128-bit accesses in flight per thread

template <typename V>
__device__ __forceinline__ void copy_strided(const char *src, char *dst, uint32_t bytes) {
    const V *s = reinterpret_cast<const V *>(src);
    V *d = reinterpret_cast<V *>(dst);
    const uint32_t n = bytes / sizeof(V);
    uint32_t i = threadIdx.x;
    for (; i + 3 * 256 < n; i += 4 * 256) {
        const V a = __ldcs(s + i), b = __ldcs(s + i + 256), c = __ldcs(s + i + 512), e = __ldcs(s + i + 768);
        __stcs(d + i, a);
        __stcs(d + i + 256, b);
        __stcs(d + i + 512, c);
        __stcs(d + i + 768, e);
    }
    for (; i < n; i += 256) __stcs(d + i, __ldcs(s + i));
}

// A pure copy, bound by HBM.  Every block moves one 16 KB piece of one segment: the blocks are dealt out in proportion
// to the segments' sizes (a grid with one row of blocks per segment spends most of its time starting the empty blocks
// of the six small ones: 36 us instead of 14 us for the 39 MB of a 1024-env step of 160 x 120 frames).
__global__ void __launch_bounds__(256) write_step_kernel(const __grid_constant__ CopySegs segs) {
    grid_wait();
    uint32_t k = 0, first = 0;
    while (blockIdx.x >= segs.s[k].block_end) first = segs.s[k++].block_end;
    const CopySeg &sg = segs.s[k];
    const unsigned long long off = (unsigned long long)(blockIdx.x - first) * kCopyBlockBytes;
    const unsigned long long left = sg.bytes - off;
    const uint32_t bytes = left < kCopyBlockBytes ? (uint32_t)left : kCopyBlockBytes;
    if (sg.vec == 16) copy_strided<uint4>(sg.src + off, sg.dst + off, bytes);
    else if (sg.vec == 4) copy_strided<uint32_t>(sg.src + off, sg.dst + off, bytes);
    else copy_strided<uint8_t>(sg.src + off, sg.dst + off, bytes);
}

// Copies up to 7 per-env arrays of one step into slab row t (null sources are skipped).
static int write_fields(ppo_buffer *b, int t, const void *const srcs[7], void *stream) {
    const ppo_buffer_desc &d = b->d;
    const size_t N = d.N;
    const int fields[7] = {PPO_FIELD_DEPTH, PPO_FIELD_PROPRIO, PPO_FIELD_ACTION, PPO_FIELD_LOGP,
                           PPO_FIELD_VALUE, PPO_FIELD_REWARD, PPO_FIELD_DONE};
    const size_t per_env[7] = {(size_t)d.H * d.W * 2, (size_t)d.P * 4, (size_t)d.A * 4, 4, 4, 4, 1};
    CopySegs segs;
    int n = 0;
    unsigned long long blocks = 0;
    for (int i = 0; i < 7; ++i) {
        if (!srcs[i]) continue;
        size_t bytes = N * per_env[i];
        char *dst = b->base + b->field_off[fields[i]] + (size_t)t * bytes;
        const uintptr_t bits = reinterpret_cast<uintptr_t>(srcs[i]) | reinterpret_cast<uintptr_t>(dst) | bytes;
        blocks += (bytes + kCopyBlockBytes - 1) / kCopyBlockBytes;
        if (blocks > 0x7fffffffull) return PPO_ERR_UNSUPPORTED;
        segs.s[n].src = static_cast<const char *>(srcs[i]);
        segs.s[n].dst = dst;
        segs.s[n].bytes = bytes;
        segs.s[n].block_end = (uint32_t)blocks;
        segs.s[n].vec = bits % 16 == 0 ? 16u : (bits % 4 == 0 ? 4u : 1u);
        ++n;
    }
    b->gae_valid = false;
    if (n == 0) return PPO_OK;
    PPO_TRY(ppo_launch(write_step_kernel, dim3((unsigned)blocks), dim3(256), 0, static_cast<cudaStream_t>(stream), segs));
    return PPO_OK;
}

extern "C" int ppo_buffer_write_step(ppo_buffer *b, int t, const void *depth, const float *proprio,
                                     const float *action, const float *logp, const float *value, const float *reward,
                                     const uint8_t *done, void *stream) {
    if (!b || !depth || !proprio || !action || !logp || !value || !reward || !done) return PPO_ERR_INVALID_ARG;
    if (t < 0 || t >= b->d.T) return PPO_ERR_INVALID_ARG;
    const void *srcs[7] = {depth, proprio, action, logp, value, reward, done};
    return write_fields(b, t, srcs, stream);
}

extern "C" int ppo_buffer_write_obs(ppo_buffer *b, int t, const void *depth, const float *proprio, void *stream) {
    if (!b || !depth || !proprio) return PPO_ERR_INVALID_ARG;
    if (t < 0 || t >= b->d.T) return PPO_ERR_INVALID_ARG;
    const void *srcs[7] = {depth, proprio, nullptr, nullptr, nullptr, nullptr, nullptr};
    return write_fields(b, t, srcs, stream);
}

extern "C" int ppo_buffer_write_outcome(ppo_buffer *b, int t, const float *reward, const uint8_t *done, void *stream) {
    if (!b || !reward || !done) return PPO_ERR_INVALID_ARG;
    if (t < 0 || t >= b->d.T) return PPO_ERR_INVALID_ARG;
    const void *srcs[7] = {nullptr, nullptr, nullptr, nullptr, nullptr, reward, done};
    return write_fields(b, t, srcs, stream);
}

// --------------------------------------------------------------------- GAE ----

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// Sum over the block; the result is valid in thread 0.  Fixed reduction order.
__device__ __forceinline__ double block_sum(double v, double *sh /*[32]*/) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    v = warp_sum(v);
    __syncthreads();
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    if (wid == 0) {
        v = (lane < (int)((blockDim.x + 31) >> 5)) ? sh[lane] : 0.0;
        v = warp_sum(v);
    }
    return v;
}

// One thread per env: reverse scan over t with the loads of UNR steps issued together.
// Reads r, V (fp32) and d (u8), writes A and R: 17 B per env-step.  Each block leaves the
// fp64 sums of A and A^2 of its envs in partials[2*blockIdx.x .. +1].
template <int UNR>
__global__ void __launch_bounds__(128) gae_scan_kernel(const float *__restrict__ reward,
                                                       const float *__restrict__ value,
                                                       const uint8_t *__restrict__ done,
                                                       const float *__restrict__ last_value, float gamma,
                                                       float gamma_lambda, float *__restrict__ adv,
                                                       float *__restrict__ ret, int T, int N,
                                                       double *__restrict__ partials) {
    grid_wait();
    __shared__ double sh[32];
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    double s1 = 0.0, s2 = 0.0;
    if (n < N) {
        float v_next = last_value[n];
        float a_next = 0.f;
        int t = T - 1;
        for (; t >= UNR - 1; t -= UNR) {
            float r[UNR], v[UNR];
            uint8_t d[UNR];
#pragma unroll
            for (int u = 0; u < UNR; ++u) {
                size_t i = (size_t)(t - u) * N + n;
                r[u] = __ldcs(reward + i);
                v[u] = __ldcs(value + i);
                d[u] = __ldcs(done + i);
            }
#pragma unroll
            for (int u = 0; u < UNR; ++u) {
                size_t i = (size_t)(t - u) * N + n;
                float nd = d[u] ? 0.f : 1.f;
                float delta = r[u] + gamma * v_next * nd - v[u];
                float a = delta + gamma_lambda * nd * a_next;
                __stcs(adv + i, a);
                __stcs(ret + i, a + v[u]);
                s1 += (double)a;
                s2 += (double)a * (double)a;
                v_next = v[u];
                a_next = a;
            }
        }
        for (; t >= 0; --t) {
            size_t i = (size_t)t * N + n;
            float r = reward[i], v = value[i];
            float nd = done[i] ? 0.f : 1.f;
            float delta = r + gamma * v_next * nd - v;
            float a = delta + gamma_lambda * nd * a_next;
            adv[i] = a;
            ret[i] = a + v;
            s1 += (double)a;
            s2 += (double)a * (double)a;
            v_next = v;
            a_next = a;
        }
    }
    s1 = block_sum(s1, sh);
    s2 = block_sum(s2, sh);
    if (threadIdx.x == 0) {
        partials[2 * blockIdx.x] = s1;
        partials[2 * blockIdx.x + 1] = s2;
    }
}

// Every block reduces the per-block partial sums in the same fixed order (deterministic),
// then normalises its share of the advantages in place with 128-bit accesses.
__global__ void __launch_bounds__(256) adv_normalize_kernel(float *__restrict__ adv, long long M,
                                                            const double *__restrict__ partials, int nparts,
                                                            float *__restrict__ stats_out) {
    grid_wait();
    __shared__ double sh[32];
    __shared__ float s_mean, s_inv;
    double s1 = 0.0, s2 = 0.0;
    for (int i = threadIdx.x; i < nparts; i += blockDim.x) {
        s1 += partials[2 * i];
        s2 += partials[2 * i + 1];
    }
    s1 = block_sum(s1, sh);
    s2 = block_sum(s2, sh);
    if (threadIdx.x == 0) {
        double mean = s1 / (double)M;
        double var = (M > 1) ? (s2 - s1 * mean) / (double)(M - 1) : 0.0;
        double sd = sqrt(var > 0.0 ? var : 0.0);
        s_mean = (float)mean;
        s_inv = (float)(1.0 / (sd + 1e-8));
        if (blockIdx.x == 0 && stats_out) {
            stats_out[0] = (float)mean;
            stats_out[1] = (float)sd;
        }
    }
    __syncthreads();
    const float mean = s_mean, inv = s_inv;
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long nth = (long long)gridDim.x * blockDim.x;
    const long long n4 = M >> 2;
    float4 *a4 = reinterpret_cast<float4 *>(adv);
    for (long long i = tid; i < n4; i += nth) {
        float4 x = a4[i];
        x.x = (x.x - mean) * inv;
        x.y = (x.y - mean) * inv;
        x.z = (x.z - mean) * inv;
        x.w = (x.w - mean) * inv;
        a4[i] = x;
    }
    for (long long i = (n4 << 2) + tid; i < M; i += nth) adv[i] = (adv[i] - mean) * inv;
}

// GAE, the moments of the advantages and their normalisation in ONE launch, for buffers whose scan blocks are all
// resident at once (cooperative launch): scan as gae_scan_kernel does, a grid barrier, then every block reduces the
// per-block partial sums in the same fixed order and normalises the advantages of its own envs (which it wrote
// itself).  The barrier is a counter that wraps to zero on the last arrival (so it needs no reset) and a generation
// word the last arriver bumps; its wait is bounded: on a time-out the block records PPO_ERR_TIMEOUT and returns
// without normalising.
__global__ void __launch_bounds__(128) gae_fused_kernel(const float *__restrict__ reward, const float *__restrict__ value,
                                                        const uint8_t *__restrict__ done,
                                                        const float *__restrict__ last_value, float gamma,
                                                        float gamma_lambda, float *__restrict__ adv,
                                                        float *__restrict__ ret, int T, int N, double *partials,
                                                        unsigned int *barrier /*[2]: counter, generation*/,
                                                        float *__restrict__ stats_out, int32_t *status) {
    grid_wait();
    __shared__ double sh[32];
    __shared__ float s_mean, s_inv;
    __shared__ int s_ok;
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    double s1 = 0.0, s2 = 0.0;
    if (n < N) {
        float v_next = last_value[n], a_next = 0.f;
        for (int t = T - 1; t >= 0; --t) {
            const size_t i = (size_t)t * N + n;
            const float r = __ldcs(reward + i), v = __ldcs(value + i);
            const float nd = __ldcs(done + i) ? 0.f : 1.f;
            const float delta = r + gamma * v_next * nd - v;
            const float a = delta + gamma_lambda * nd * a_next;
            adv[i] = a;
            ret[i] = a + v;
            s1 += (double)a;
            s2 += (double)a * (double)a;
            v_next = v;
            a_next = a;
        }
    }
    s1 = block_sum(s1, sh);
    s2 = block_sum(s2, sh);
    if (threadIdx.x == 0) {
        partials[2 * blockIdx.x] = s1;
        partials[2 * blockIdx.x + 1] = s2;
        __threadfence();
        volatile unsigned int *gen = barrier + 1;
        const unsigned int my_gen = *gen;
        int ok = 1;
        if (atomicInc(barrier, gridDim.x - 1) == gridDim.x - 1) {
            __threadfence();
            atomicAdd(barrier + 1, 1u);
        } else {
            const long long t0 = clock64();
            while (*gen == my_gen) {
                if (clock64() - t0 > 2000000000ll) {  // ~1 s
                    ppo_report(status, PPO_ERR_TIMEOUT);
                    ok = 0;
                    break;
                }
            }
        }
        __threadfence();
        s_ok = ok;
    }
    __syncthreads();
    if (!s_ok) return;
    const long long M = (long long)N * T;
    double t1 = 0.0, t2 = 0.0;
    for (int i = threadIdx.x; i < (int)gridDim.x; i += blockDim.x) {
        t1 += __ldcg(partials + 2 * i);
        t2 += __ldcg(partials + 2 * i + 1);
    }
    t1 = block_sum(t1, sh);
    t2 = block_sum(t2, sh);
    if (threadIdx.x == 0) {
        const double mean = t1 / (double)M;
        const double var = (M > 1) ? (t2 - t1 * mean) / (double)(M - 1) : 0.0;
        const double sd = sqrt(var > 0.0 ? var : 0.0);
        s_mean = (float)mean;
        s_inv = (float)(1.0 / (sd + 1e-8));
        if (blockIdx.x == 0 && stats_out) {
            stats_out[0] = (float)mean;
            stats_out[1] = (float)sd;
        }
    }
    __syncthreads();
    if (n < N) {
        const float mean = s_mean, inv = s_inv;
        for (int t = 0; t < T; ++t) {
            const size_t i = (size_t)t * N + n;
            adv[i] = (adv[i] - mean) * inv;
        }
    }
}

// Blocks of gae_fused_kernel that can be resident at once on the current device (0: cooperative launch unavailable).
static int gae_fused_capacity() {
    static PerDevice<int> cap;  // + 1
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    return cap.get(dev, [dev] {
        int coop = 0, per_sm = 0;
        if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) == cudaSuccess && coop &&
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, gae_fused_kernel, 128, 0) == cudaSuccess)
            return per_sm * ppo_num_sms() + 1;
        return 1;
    }) - 1;
}

extern "C" int ppo_compute_gae(ppo_buffer *b, const float *last_value, float gamma, float lambda, int normalize,
                               float *stats_out, void *stream) {
    if (!b || !last_value) return PPO_ERR_INVALID_ARG;
    if (!(gamma >= 0.f && gamma <= 1.f) || !(lambda >= 0.f && lambda <= 1.f)) return PPO_ERR_INVALID_ARG;
    const int N = b->d.N, T = b->d.T;
    const int threads = 128;
    const int blocks = ppo_cdiv(N, threads);
    if (blocks > kMaxGaeBlocks) return PPO_ERR_UNSUPPORTED;  // N <= 524288 envs
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    double *partials = slab<double>(b, PPO_FIELD_SCRATCH);
    // normalize == 2: one cooperative launch, possible when the whole scan is resident at once (every configuration
    // of the workloads).  Measured, it is no faster than the two plain launches (24 against 18 microseconds at 1024
    // envs x 16 steps: a cooperative launch and its grid barrier cost more than the second launch they save), so it
    // is an option, not the default.  The last 8 bytes of the scratch slab hold the grid barrier; they are free
    // while blocks < kMaxGaeBlocks.
    if (normalize == 2 && (blocks >= kMaxGaeBlocks || blocks > gae_fused_capacity())) return PPO_ERR_UNSUPPORTED;
    if (normalize == 2) {
        unsigned int *barrier = reinterpret_cast<unsigned int *>(partials + 2 * kMaxGaeBlocks) - 2;
        PPO_TRY(ppo_clear_once(&b->barrier_made, barrier, 8, st));
        const float *reward = slab<float>(b, PPO_FIELD_REWARD), *value = slab<float>(b, PPO_FIELD_VALUE);
        const uint8_t *done = slab<uint8_t>(b, PPO_FIELD_DONE);
        float *adv = slab<float>(b, PPO_FIELD_ADV), *ret = slab<float>(b, PPO_FIELD_RET);
        float gl = gamma * lambda;
        int32_t *status = ppo_device_status_ptr();
        int Ti = T, Ni = N;
        void *args[] = {&reward, &value, &done, &last_value, &gamma, &gl, &adv, &ret, &Ti, &Ni, &partials, &barrier,
                        &stats_out, &status};
        PPO_CUDA_CHECK(cudaLaunchCooperativeKernel((const void *)gae_fused_kernel, dim3(blocks), dim3(threads), args, 0, st));
        PPO_LAUNCH_CHECK();
        b->gae_valid = true;
        b->gae_blocks = blocks;
        return PPO_OK;
    }
    PPO_TRY(ppo_launch(gae_scan_kernel<8>, dim3(blocks), dim3(threads), 0, st, slab<float>(b, PPO_FIELD_REWARD), slab<float>(b, PPO_FIELD_VALUE),
                                                   slab<uint8_t>(b, PPO_FIELD_DONE), last_value, gamma,
                                                   gamma * lambda, slab<float>(b, PPO_FIELD_ADV),
                                                   slab<float>(b, PPO_FIELD_RET), T, N, partials));
    if (normalize) {
        const long long M = (long long)N * T;
        int nb = ppo_cdiv(M, 256 * 4 * 4);
        int cap = ppo_num_sms() * 8;
        if (nb > cap) nb = cap;
        if (nb < 1) nb = 1;
        PPO_TRY(ppo_launch(adv_normalize_kernel, dim3(nb), dim3(256), 0, st, slab<float>(b, PPO_FIELD_ADV), M, partials, blocks, stats_out));
    }
    b->gae_valid = true;
    b->gae_blocks = blocks;
    return PPO_OK;
}

// ------------------------------------------------------------ GAE, no allocation ----

// Scratch of ppo_gae_static: the per-block partial sums the scan leaves for the normalisation pass.
// Lives in the library image, so every device that loads the library holds these 64 KB until exit.
static __device__ __align__(256) double g_gae_static_scratch[2 * kMaxGaeBlocks];

// Device address of the scratch array on the current device (nullptr on error).  The array's name is
// only a host-side handle; kernels must be given the address cudaGetSymbolAddress returns.
static double *gae_static_scratch_ptr() {
    static PerDevice<double *> ptrs;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return nullptr;
    return ptrs.get(dev, []() -> double * {
        void *p = nullptr;
        return cudaGetSymbolAddress(&p, g_gae_static_scratch) == cudaSuccess ? static_cast<double *>(p) : nullptr;
    });
}

extern "C" int ppo_gae_static(const float *reward, const float *value, const uint8_t *done, const float *last_value,
                              int T, int N, float gamma, float lambda, int normalize, float *adv, float *ret,
                              float *stats_out, void *stream) {
    if (!reward || !value || !done || !last_value || !adv || !ret) return PPO_ERR_INVALID_ARG;
    if (T <= 0 || N <= 0 || (long long)T * N >= (1ll << 31)) return PPO_ERR_INVALID_ARG;
    if (!(gamma >= 0.f && gamma <= 1.f) || !(lambda >= 0.f && lambda <= 1.f)) return PPO_ERR_INVALID_ARG;
    if (N > PPO_GAE_STATIC_MAX_ENVS) return PPO_ERR_UNSUPPORTED;  // more envs than the fixed scratch covers
    if (!ppo_aligned(adv, 16)) return PPO_ERR_ALIGN;
    const int threads = 128;
    const int blocks = ppo_cdiv(N, threads);
    double *partials = gae_static_scratch_ptr();
    if (!partials) return PPO_ERR_CUDA;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // every partial a later pass reads is written by this launch first: nothing has to start at zero
    PPO_TRY(ppo_launch(gae_scan_kernel<8>, dim3(blocks), dim3(threads), 0, st, reward, value, done, last_value, gamma, gamma * lambda, adv, ret, T, N,
                                                   partials));
    if (normalize) {
        const long long M = (long long)N * T;
        int nb = ppo_cdiv(M, 256 * 4 * 4);
        const int cap = ppo_num_sms() * 8;
        nb = nb > cap ? cap : (nb < 1 ? 1 : nb);
        PPO_TRY(ppo_launch(adv_normalize_kernel, dim3(nb), dim3(256), 0, st, adv, M, partials, blocks, stats_out));
    }
    return PPO_OK;
}

// ------------------------------------------------------------------ gather ----

struct PermParams {
    uint32_t key[6];
    uint32_t M;
    int h;
    uint32_t mask;
};

__host__ __device__ __forceinline__ uint32_t perm_mix(uint32_t x) {
    x ^= x >> 16;
    x *= 0x9E3779B9u;
    x ^= x >> 15;
    x *= 0x6A09E667u;
    x ^= x >> 16;
    return x;
}

static PermParams make_perm(uint64_t seed, uint32_t epoch, uint32_t M) {
    PermParams p;
    const uint32_t lo = (uint32_t)seed, hi = (uint32_t)(seed >> 32);
    for (uint32_t j = 0; j < 6; ++j)
        p.key[j] = perm_mix(lo ^ perm_mix(hi + 0x9E3779B9u * (j + 1)) ^ perm_mix(epoch + 0xBB67AE85u * (j + 1)));
    int bits = 0;
    while ((1ull << bits) < (unsigned long long)M) ++bits;
    p.h = (bits + 1) / 2 < 1 ? 1 : (bits + 1) / 2;
    p.mask = (1u << p.h) - 1u;
    p.M = M;
    return p;
}

__device__ __forceinline__ uint32_t perm_apply(const PermParams &p, uint32_t i) {
    uint32_t x = i;
    do {
        uint32_t L = x >> p.h, R = x & p.mask;
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            uint32_t nr = L ^ (perm_mix(R ^ p.key[j]) & p.mask);
            L = R;
            R = nr;
        }
        x = (L << p.h) | R;
    } while (x >= p.M);
    return x;
}

struct GatherArgs {
    const char *depth;
    const float *proprio, *action, *logp, *value, *adv, *ret;
    char *o_depth;
    float *o_proprio, *o_action, *o_logp, *o_value, *o_adv, *o_ret;
    uint32_t *o_index;
    uint32_t start;      // first position of this minibatch in the permuted order
    uint32_t rows;       // B
    uint32_t frame;      // bytes of a frame
    uint32_t chunks;     // CTAs per row
    int P, A;
    // sequence minibatches: envs are permuted, not samples; row = t * seq_Be + e holds sample t * N + pi(start + e)
    uint32_t seq_Be;     // 0: flat minibatch
    uint32_t N;
    const uint8_t *done;
    uint8_t *o_done;
};

// Sample that row `row` of the minibatch holds.
__device__ __forceinline__ uint32_t gather_sample(const GatherArgs &g, const PermParams &p, uint32_t row) {
    if (!g.seq_Be) return perm_apply(p, g.start + row);
    const uint32_t t = row / g.seq_Be, e = row - t * g.seq_Be;
    return t * g.N + perm_apply(p, g.start + e);
}

// The row's small fields, by one CTA of the row: a thread's value of sample s, and its place in row `row`.
__device__ __forceinline__ float small_load(const GatherArgs &g, uint32_t s) {
    const int t = threadIdx.x;
    if (t < g.P) return g.proprio[(size_t)s * g.P + t];
    if (t >= 64 && t < 64 + g.A) return g.action[(size_t)s * g.A + (t - 64)];
    if (t == 128) return g.logp[s];
    if (t == 129) return g.value[s];
    if (t == 130) return g.adv[s];
    if (t == 131) return g.ret[s];
    if (t == 133 && g.o_done) return __uint_as_float(g.done[s]);
    return 0.f;
}
__device__ __forceinline__ void small_store(const GatherArgs &g, uint32_t row, uint32_t s, float v) {
    const int t = threadIdx.x;
    if (t < g.P) g.o_proprio[(size_t)row * g.P + t] = v;
    if (t >= 64 && t < 64 + g.A) g.o_action[(size_t)row * g.A + (t - 64)] = v;
    if (t == 128) g.o_logp[row] = v;
    if (t == 129) g.o_value[row] = v;
    if (t == 130) g.o_adv[row] = v;
    if (t == 131) g.o_ret[row] = v;
    if (t == 132 && g.o_index) g.o_index[row] = s;
    if (t == 133 && g.o_done) g.o_done[row] = (uint8_t)__float_as_uint(v);
}

// Bytes Q * 4 + h / 8 .. + 16 of the 32 bytes a | b (h = 0 or 16 bits).
template <int Q>
__device__ __forceinline__ uint4 window16(const uint4 &a, const uint4 &b, uint32_t h) {
    const uint32_t w[9] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, 0u};
    return make_uint4(__funnelshift_r(w[Q], w[Q + 1], h), __funnelshift_r(w[Q + 1], w[Q + 2], h),
                      __funnelshift_r(w[Q + 2], w[Q + 3], h), __funnelshift_r(w[Q + 3], w[Q + 4], h));
}
__device__ __forceinline__ uint4 window16(const uint4 &a, const uint4 &b, uint32_t q, uint32_t h) {
    return q == 0 ? window16<0>(a, b, h) : (q == 1 ? window16<1>(a, b, h) : (q == 2 ? window16<2>(a, b, h) : window16<3>(a, b, h)));
}

constexpr uint32_t kGatherUnits = 1024;  // 16-byte units a CTA moves: four per thread

// One CTA copies one chunk (at most 16 KB) of one row's depth frame, 128-bit accesses, all four loads of a thread in
// flight at once; chunk 0 also copies the row's small fields.  Bound by HBM, as long as the permutation stays out of the
// way: its six rounds, repeated while the walk leaves [0, M), are up to a thousand instructions, and when every warp of
// a CTA works them out for itself they fill the issue slots (math-pipe stalls at 25 % DRAM).  So one warp does it for
// the CTA.  Measured: 5.9 -> 6.4 TB/s at 32768 rows of 160 x 120; persistent CTAs that work out the next sample between
// loads and stores, or several chunks per CTA, are slower.
// RAGGED: frames whose byte count is no multiple of 16.  Source and destination of a row are then misaligned against
// each other by some even number of bytes: every aligned unit of the destination is assembled from two aligned units of
// the source (the second one is the neighbouring lane's, for the last lane a load that hits L1), counted from a 128-byte line so
// that a warp stores whole lines; the few bytes in front of the first and behind the last whole unit go as single pixels.  The loads stay inside
// the depth slab, which is padded to 256 bytes and followed by others.  Measured: 82 -> 61 us for 6700 rows of 90 x 122
// against a pixel per access, 50 with eight blocks per SM (the second unit in registers of its own made it five).
template <bool RAGGED>
__global__ void __launch_bounds__(256, 8) gather_kernel(const __grid_constant__ GatherArgs g, const __grid_constant__ PermParams p) {
    grid_wait();
    const uint32_t row = blockIdx.x / g.chunks, chunk = blockIdx.x - row * g.chunks;
    __shared__ uint32_t s_sample;
    if (threadIdx.x < 32) {
        const uint32_t v = gather_sample(g, p, row);
        if (threadIdx.x == 0) s_sample = v;
    }
    __syncthreads();
    const uint32_t s = s_sample;
    const char *src = g.depth + (size_t)s * g.frame;
    char *dst = g.o_depth + (size_t)row * g.frame;
    int lead = 0, tail = 0, skew = 0;
    uint32_t shift = 0;
    if (RAGGED) {
        const int head = (int)((16u - (uint32_t)(reinterpret_cast<uintptr_t>(dst) & 15u)) & 15u);
        lead = (uint32_t)head < g.frame ? head : (int)g.frame;  // bytes before the first whole unit
        tail = (int)((g.frame - lead) & 15u);
        skew = (int)((reinterpret_cast<uintptr_t>(dst + lead) >> 4) & 7u);  // unit -skew starts a line
        shift = (uint32_t)(reinterpret_cast<uintptr_t>(src + lead) & 15u);
    }
    const int units = (int)((g.frame - lead) >> 4);
    const int per = RAGGED ? ((units + skew + (int)g.chunks - 1) / (int)g.chunks + 7) & ~7 : (units + (int)g.chunks - 1) / (int)g.chunks;
    const int u0 = (int)chunk * per - skew, lo = max(u0, 0), hi = min(u0 + per, units);
    const uint4 *src16 = reinterpret_cast<const uint4 *>(src + lead - shift);
    uint4 *dst16 = reinterpret_cast<uint4 *>(dst + lead);
    const int t0 = u0 + (int)threadIdx.x;
    uint4 a[4];
    const int last = RAGGED && shift ? hi : hi - 1;  // the unit behind the last one supplies its rest
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int u = t0 + 256 * k;
        if (u >= lo && u <= last) a[k] = RAGGED ? __ldg(src16 + u) : __ldcs(src16 + u);
    }
    // Ragged frames are small ones as well: the small fields and the ends of the frame are under way with the rest, behind it they
    // would be another trip to memory (4.35 -> 4.57 TB/s for 49 x 66).  Whole ones are bound by HBM and lose 1 %.
    const int t = threadIdx.x;
    const size_t done = (size_t)lead + (size_t)units * 16;
    float small = 0.f;
    uint32_t ends = 0;  // a pixel of the head and one of the tail
    if (RAGGED && chunk == 0) {
        small = small_load(g, s);
        if (2 * t < lead) ends = reinterpret_cast<const uint16_t *>(src)[t];
        if (2 * t < tail) ends |= (uint32_t)reinterpret_cast<const uint16_t *>(src + done)[t] << 16;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int u = t0 + 256 * k;
        if (RAGGED && shift) {
            uint4 b = make_uint4(__shfl_down_sync(0xffffffffu, a[k].x, 1), __shfl_down_sync(0xffffffffu, a[k].y, 1),
                                 __shfl_down_sync(0xffffffffu, a[k].z, 1), __shfl_down_sync(0xffffffffu, a[k].w, 1));
            if (u >= lo && u < hi) {
                if ((threadIdx.x & 31) == 31) b = __ldg(src16 + u + 1);
                __stcs(dst16 + u, window16(a[k], b, shift >> 2, (shift & 2u) * 8u));
            }
        } else if (u >= lo && u < hi) {
            __stcs(dst16 + u, a[k]);
        }
    }
    if (chunk == 0) {
        if (RAGGED) {
            if (2 * t < lead) reinterpret_cast<uint16_t *>(dst)[t] = (uint16_t)ends;
            if (2 * t < tail) reinterpret_cast<uint16_t *>(dst + done)[t] = (uint16_t)(ends >> 16);
        }
        small_store(g, row, s, RAGGED ? small : small_load(g, s));
    }
}

static int gather_impl(const ppo_buffer *b, uint64_t seed, uint32_t epoch, int mb_index, int num_minibatches,
                       const ppo_minibatch *out, uint8_t *done_out, bool sequences, void *stream);

extern "C" int ppo_shuffle_gather_minibatch(const ppo_buffer *b, uint64_t seed, uint32_t epoch, int mb_index,
                                            int num_minibatches, const ppo_minibatch *out, void *stream) {
    return gather_impl(b, seed, epoch, mb_index, num_minibatches, out, nullptr, false, stream);
}

extern "C" int ppo_shuffle_gather_sequences(const ppo_buffer *b, uint64_t seed, uint32_t epoch, int mb_index,
                                            int num_minibatches, const ppo_minibatch *out, uint8_t *done_out, void *stream) {
    if (!done_out) return PPO_ERR_INVALID_ARG;
    return gather_impl(b, seed, epoch, mb_index, num_minibatches, out, done_out, true, stream);
}

static int gather_impl(const ppo_buffer *b, uint64_t seed, uint32_t epoch, int mb_index, int num_minibatches,
                       const ppo_minibatch *out, uint8_t *done_out, bool sequences, void *stream) {
    if (!b || !out) return PPO_ERR_INVALID_ARG;
    if (num_minibatches <= 0 || mb_index < 0 || mb_index >= num_minibatches) return PPO_ERR_INVALID_ARG;
    // what is permuted and cut into minibatches: the samples, or the envs (each with all its T steps)
    const long long M = sequences ? (long long)b->d.N : (long long)b->d.N * b->d.T;
    if (M % num_minibatches != 0) return PPO_ERR_SHAPE;
    const long long per = M / num_minibatches;
    const long long B = sequences ? per * b->d.T : per;
    if (out->B != B) return PPO_ERR_SHAPE;
    if (!out->depth_f16 || !out->proprio || !out->action || !out->logp_old || !out->value_old || !out->adv ||
        !out->ret)
        return PPO_ERR_INVALID_ARG;
    if (!ppo_aligned(out->depth_f16, 16)) return PPO_ERR_ALIGN;
    if (!b->gae_valid) return PPO_ERR_STATE;
    const size_t frame = (size_t)b->d.H * b->d.W * 2;
    const bool vec16 = frame % 16 == 0;
    if (b->d.P > 64 || b->d.A > 64) return PPO_ERR_UNSUPPORTED;
    GatherArgs g;
    g.depth = b->base + b->field_off[PPO_FIELD_DEPTH];
    g.proprio = slab<float>(b, PPO_FIELD_PROPRIO);
    g.action = slab<float>(b, PPO_FIELD_ACTION);
    g.logp = slab<float>(b, PPO_FIELD_LOGP);
    g.value = slab<float>(b, PPO_FIELD_VALUE);
    g.adv = slab<float>(b, PPO_FIELD_ADV);
    g.ret = slab<float>(b, PPO_FIELD_RET);
    g.o_depth = static_cast<char *>(out->depth_f16);
    g.o_proprio = out->proprio;
    g.o_action = out->action;
    g.o_logp = out->logp_old;
    g.o_value = out->value_old;
    g.o_adv = out->adv;
    g.o_ret = out->ret;
    g.o_index = out->index;
    g.start = (uint32_t)(mb_index * per);
    g.rows = (uint32_t)B;
    g.seq_Be = sequences ? (uint32_t)per : 0u;
    g.N = (uint32_t)b->d.N;
    g.done = slab<uint8_t>(b, PPO_FIELD_DONE);
    g.o_done = done_out;
    g.frame = (uint32_t)frame;
    // at most kGatherUnits units per CTA, so a frame of 38 400 B becomes 3 chunks; a ragged frame's chunks count
    // from the line its first unit lies in and are rounded up to whole lines
    g.chunks = (uint32_t)(vec16 ? (frame / 16 + kGatherUnits - 1) / kGatherUnits : (frame / 16 + 7) / (kGatherUnits - 8) + 1);
    g.P = b->d.P;
    g.A = b->d.A;
    const long long ctas = B * g.chunks;
    if (ctas > 0x7fffffffll || frame > 0x7fffffffull) return PPO_ERR_UNSUPPORTED;
    PermParams p = make_perm(seed, epoch, (uint32_t)M);
    if (vec16) PPO_TRY(ppo_launch(gather_kernel<false>, dim3((unsigned)ctas), dim3(256), 0, static_cast<cudaStream_t>(stream), g, p));
    else PPO_TRY(ppo_launch(gather_kernel<true>, dim3((unsigned)ctas), dim3(256), 0, static_cast<cudaStream_t>(stream), g, p));
    return PPO_OK;
}

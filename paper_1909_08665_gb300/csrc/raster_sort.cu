// raster_sort.cu -- the recorded spikes in (instance, step, id) order, sorted on
// the device before they are copied to the host (Sec. 3.1.2: output spike
// times of all neurons are recorded).
//
// The step kernels append spikes as they come: by partition or by warp, in no
// order within a step.  A reader wants them by step and neuron, and sorting
// 470,000 spikes (one second of the full network) on the host took 37 ms
// beside 26 ms of simulation.  Here the steps are the buckets of a counting
// sort: a histogram over (instance, step), its exclusive scan, a scatter of
// the spikes' keys, and each bucket's few dozen keys ranked against each other.
// A bucket is a warp's work up to kWarpGroup keys; larger ones (the initial
// volley of an unrelaxed network) are split once more, into kBins by the top
// bits of their keys, by a CTA.  Very long spans put 2^k steps into a bucket,
// so that the histogram stays at kMaxGroups words per instance at most.  Up to
// kSmall spikes, the reads of a closed loop, take one launch that counts,
// sorts, clears the lists and writes into mapped host memory, and one wait:
// the spikes of ten steps of the 10 % network in 22 us, 51 with copies of the
// counts and of each array.
// Measured: reading one second of the full network (470,000 spikes) 0.30 ms,
// 0.15 of it for the copies; the 64 instances' 370,000 spikes of 100 ms 2.0 ms
// in 64 reads, 30.5 with the buckets and the sorts on the host.  Bound by the
// seven launches and the one-CTA scan, not by the 4 MB it moves.
#include <algorithm>
#include <cstring>
#include <vector>

#include "snn_internal.cuh"

namespace snn {
namespace {

constexpr int kThreads = 256;
constexpr uint32_t kSmall = 1024;              // spikes sorted by one CTA in one launch
constexpr uint32_t kWarpGroup = 512;           // largest bucket a warp ranks
constexpr int kBigThreads = 512;
constexpr int kBinBits = 10, kBins = 1 << kBinBits;
constexpr long long kMaxGroups = 1ll << 20;    // buckets in all, beyond one per instance

struct SortParams {
    const uint32_t* counts;          // [n_part] recorded spikes (may exceed cap_part)
    const uint32_t* step_in;         // [n_part][cap_part]
    const uint32_t* id_in;
    uint32_t cap_part;
    int32_t n_part, n_inst;
    const int32_t* goff;             // [n_inst + 1] first id of each instance; unused for one
    uint32_t t_lo;                   // first step that may occur
    uint32_t per_inst;               // buckets of one instance
    uint32_t n_groups;
    uint32_t n;                      // spikes the arrays below hold
    int32_t id_bits, shift;          // 2^shift steps share a bucket
    uint32_t* group;                 // [n_groups] counts, then ends of the buckets
    unsigned long long* key;         // [n] keys, bucket by bucket
    unsigned long long* key2;        // [n] the same, large buckets binned
    uint32_t* step_out;
    uint32_t* id_out;
};

__device__ __forceinline__ uint32_t instance_of(const SortParams& p, uint32_t id) {
    int a = 0, b = p.n_inst;         // goff[a] <= id < goff[b]
    while (b - a > 1) {
        const int m = (a + b) >> 1;
        if ((uint32_t)__ldg(&p.goff[m]) <= id) a = m;
        else b = m;
    }
    return (uint32_t)a;
}

__device__ __forceinline__ uint32_t group_of(const SortParams& p, uint32_t step, uint32_t id) {
    return instance_of(p, id) * p.per_inst + min((step - p.t_lo) >> p.shift, p.per_inst - 1u);
}

// f(step, id) for every recorded spike of partition blockIdx.x
template <typename F>
__device__ __forceinline__ void for_each_spike(const SortParams& p, F f) {
    const uint32_t m = min(__ldg(&p.counts[blockIdx.x]), p.cap_part);
    const size_t base = (size_t)blockIdx.x * p.cap_part;
    for (uint32_t i = blockIdx.y * kThreads + threadIdx.x; i < m; i += gridDim.y * kThreads)
        f(__ldg(&p.step_in[base + i]), __ldg(&p.id_in[base + i]));
}

__global__ void __launch_bounds__(kThreads) k_sort_count(const __grid_constant__ SortParams p) {
    for_each_spike(p, [&](uint32_t s, uint32_t id) { atomicAdd(&p.group[group_of(p, s, id)], 1u); });
}

// exclusive scan of the bucket counts, in place (one CTA, 8 buckets a thread)
__global__ void __launch_bounds__(1024) k_sort_scan(const __grid_constant__ SortParams p) {
    __shared__ uint32_t s_w[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t carry = 0;
    for (uint32_t base = 0; base < p.n_groups; base += 8u * 1024u) {
        uint32_t v[8], sum = 0;
        const uint32_t i0 = base + threadIdx.x * 8u;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            v[k] = i0 + k < p.n_groups ? p.group[i0 + k] : 0u;
            sum += v[k];
        }
        uint32_t x = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) s_w[warp] = x;
        __syncthreads();
        uint32_t w = s_w[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        const uint32_t before = warp ? __shfl_sync(0xffffffffu, w, warp - 1) : 0u;
        uint32_t at = carry + before + x - sum;
        carry += __shfl_sync(0xffffffffu, w, 31);
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            if (i0 + k < p.n_groups) p.group[i0 + k] = at;
            at += v[k];
        }
    }
}

// keys into their buckets; group[] ends up as the buckets' ends
__global__ void __launch_bounds__(kThreads) k_sort_scatter(const __grid_constant__ SortParams p) {
    for_each_spike(p, [&](uint32_t s, uint32_t id) {
        const uint32_t at = atomicAdd(&p.group[group_of(p, s, id)], 1u);
        const uint32_t low = (s - p.t_lo) & ((1u << p.shift) - 1u);
        if (at < p.n) p.key[at] = ((unsigned long long)low << p.id_bits) | id;
    });
}

// one warp ranks `n` keys at key[b..) (equal keys keep their order) and writes
// their steps and ids
__device__ __forceinline__ void rank_keys(const SortParams& p, const unsigned long long* key, uint32_t b,
                                          uint32_t n, uint32_t step0) {
    const uint32_t lane = threadIdx.x & 31u;
    for (uint32_t i0 = 0; i0 < n; i0 += 32u) {
        const uint32_t i = i0 + lane;
        const unsigned long long mine = i < n ? key[b + i] : 0ull;
        uint32_t rank = 0;
#pragma unroll 4
        for (uint32_t j = 0; j < n; ++j) {
            const unsigned long long k = key[b + j];
            rank += k < mine || (k == mine && j < i) ? 1u : 0u;
        }
        if (i < n) {
            p.step_out[b + rank] = step0 + (uint32_t)(mine >> p.id_bits);
            p.id_out[b + rank] = (uint32_t)mine & ((1u << p.id_bits) - 1u);
        }
    }
}

// bucket g's keys are [b, b + n): within the arrays even if the lists were changed
// since their spikes were counted
__device__ __forceinline__ void bucket(const SortParams& p, uint32_t g, uint32_t& b, uint32_t& n) {
    b = g ? min(p.group[g - 1], p.n) : 0u;
    n = min(p.group[g], p.n) - b;
}

__device__ __forceinline__ uint32_t first_step(const SortParams& p, uint32_t g) {
    return p.t_lo + ((g % p.per_inst) << p.shift);
}

__global__ void __launch_bounds__(kThreads) k_sort_groups(const __grid_constant__ SortParams p) {
    const uint32_t warps = gridDim.x * (kThreads / 32);
    for (uint32_t g = (blockIdx.x * kThreads + threadIdx.x) >> 5; g < p.n_groups; g += warps) {
        uint32_t b, n;
        bucket(p, g, b, n);
        if (n <= kWarpGroup) rank_keys(p, p.key, b, n, first_step(p, g));
    }
}

// buckets above kWarpGroup: binned by the top kBinBits of their keys, each bin
// ranked by a warp
__global__ void __launch_bounds__(kBigThreads) k_sort_large(const __grid_constant__ SortParams p) {
    __shared__ uint32_t s_bin[kBins + 1], s_at[kBins], s_w[kBigThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int bin_shift = max(0, p.id_bits + p.shift - kBinBits);
    auto bin_of = [&](unsigned long long k) { return (uint32_t)min(k >> bin_shift, (unsigned long long)(kBins - 1)); };
    for (uint32_t g = blockIdx.x; g < p.n_groups; g += gridDim.x) {
        uint32_t b, n;
        bucket(p, g, b, n);
        if (n <= kWarpGroup) continue;
        for (int k = tid; k < kBins; k += kBigThreads) s_bin[k] = 0u;
        __syncthreads();
        for (uint32_t i = tid; i < n; i += kBigThreads) atomicAdd(&s_bin[bin_of(p.key[b + i])], 1u);
        __syncthreads();
        // exclusive scan, two bins a thread
        const uint32_t v0 = s_bin[2 * tid], v1 = s_bin[2 * tid + 1];
        uint32_t x = v0 + v1;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) s_w[warp] = x;
        __syncthreads();
        uint32_t at = x - v0 - v1;
        for (int w = 0; w < warp; ++w) at += s_w[w];
        s_bin[2 * tid] = s_at[2 * tid] = at;
        s_bin[2 * tid + 1] = s_at[2 * tid + 1] = at + v0;
        if (tid == 0) s_bin[kBins] = n;
        __syncthreads();
        for (uint32_t i = tid; i < n; i += kBigThreads) {
            const unsigned long long k = p.key[b + i];
            p.key2[b + atomicAdd(&s_at[bin_of(k)], 1u)] = k;
        }
        __syncthreads();
        for (int k = warp; k < kBins; k += kBigThreads / 32) {
            const uint32_t lo = s_bin[k], hi = s_bin[k + 1];
            if (hi > lo) rank_keys(p, p.key2, b + lo, hi - lo, first_step(p, g));
        }
        __syncthreads();
    }
}
static_assert(kBins == 2 * kBigThreads, "two bins a thread in the scan");

// At most kSmall spikes: one CTA, one launch, all keys in shared memory.  It
// also counts: head[0], head[1] are the halves of the number of spikes (clamped
// counts), head[2] is 1 if a list ran out of capacity.  Up to kSmall spikes are
// sorted out, and the lists are cleared; of more nothing else happens.
__global__ void __launch_bounds__(kSmall) k_sort_small(const __grid_constant__ SortParams p, uint32_t* counts,
                                                       uint32_t* head) {
    __shared__ unsigned long long s_key[kSmall];
    __shared__ uint32_t s_off[kStepThreads + 1], s_w[32];
    __shared__ unsigned long long s_sum[32];
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    const uint32_t raw = tid < (uint32_t)p.n_part ? counts[tid] : 0u;
    const uint32_t m = min(raw, p.cap_part);
    const bool lost = __syncthreads_or(raw > p.cap_part) != 0;
    // the lists' places, exact as far as they are used: a list counts as kSmall
    // + 1 spikes at most, so the sum tells whether there are more than kSmall
    const uint32_t few = min(m, kSmall + 1u);
    uint32_t x = few;
    unsigned long long sum = m;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= (uint32_t)o) x += y;
        sum += __shfl_xor_sync(0xffffffffu, sum, o);
    }
    if (lane == 31u) {
        s_w[warp] = x;
        s_sum[warp] = sum;
    }
    __syncthreads();
    uint32_t off = x - few;
    for (uint32_t w = 0; w < warp; ++w) off += s_w[w];
    if (tid <= (uint32_t)p.n_part) s_off[tid] = off;
    __syncthreads();
    const uint32_t n = s_off[p.n_part];
    if (tid == 0) {
        sum = 0ull;
        for (uint32_t w = 0; w * 32u < (uint32_t)p.n_part; ++w) sum += s_sum[w];
        head[0] = (uint32_t)sum;
        head[1] = (uint32_t)(sum >> 32);
        head[2] = lost ? 1u : 0u;
    }
    if (n > kSmall) return;
    if (tid < (uint32_t)p.n_part) counts[tid] = 0u;
    unsigned long long mine = ~0ull;
    uint32_t step = 0, id = 0;
    if (tid < n) {
        int a = 0, b = p.n_part;     // s_off[a] <= tid < s_off[b]
        while (b - a > 1) {
            const int k = (a + b) >> 1;
            if (s_off[k] <= tid) a = k;
            else b = k;
        }
        const size_t at = (size_t)a * p.cap_part + (tid - s_off[a]);
        step = __ldg(&p.step_in[at]);
        id = __ldg(&p.id_in[at]);
        mine = ((((unsigned long long)instance_of(p, id) << 32) | (step - p.t_lo)) << p.id_bits) | id;
    }
    s_key[tid] = mine;
    __syncthreads();
    if (tid < n) {
        uint32_t rank = 0;
#pragma unroll 4
        for (uint32_t j = 0; j < n; ++j) {
            const unsigned long long k = s_key[j];
            rank += k < mine || (k == mine && j < tid) ? 1u : 0u;
        }
        p.step_out[rank] = step;
        p.id_out[rank] = id;
    }
}

// arrays of n words side by side into (mapped host) memory
__global__ void __launch_bounds__(kThreads) k_read_arrays(const uint32_t* a, const uint32_t* b, const uint32_t* c,
                                                          int n, int total, uint32_t* out) {
    const int i = blockIdx.x * kThreads + threadIdx.x;
    if (i < total) out[i] = i < n ? a[i] : i < 2 * n ? b[i - n] : c[i - 2 * n];
}

template <typename T>
cudaError_t grow(T** p, size_t* cap, size_t need) {
    if (*cap >= need) return cudaSuccess;
    cudaFree(*p);
    *p = nullptr;
    *cap = 0;
    const cudaError_t e = cudaMalloc(reinterpret_cast<void**>(p), sizeof(T) * need);
    if (e == cudaSuccess) *cap = need;
    return e;
}

SortParams common_params(const RasterList& in) {
    SortParams p = {};
    p.counts = in.counts;
    p.step_in = in.step;
    p.id_in = in.id;
    p.cap_part = in.cap_part;
    p.n_part = in.n_part;
    p.n_inst = in.n_inst;
    p.goff = in.goff;
    p.t_lo = in.t_lo;
    p.id_bits = 1;
    while (p.id_bits < 31 && (in.n_ids >> p.id_bits) != 0) ++p.id_bits;
    return p;
}

}  // namespace

cudaError_t host_stage(HostStage* st, size_t bytes, uint32_t** host, uint32_t** dev) {
    if (st->bytes < bytes) {
        host_stage_free(st);
        cudaError_t e = cudaHostAlloc(&st->host, bytes, cudaHostAllocMapped);
        if (e == cudaSuccess) e = cudaHostGetDevicePointer(&st->dev, st->host, 0);
        if (e != cudaSuccess) {
            host_stage_free(st);
            return e;
        }
        st->bytes = bytes;
    }
    *host = static_cast<uint32_t*>(st->host);
    *dev = static_cast<uint32_t*>(st->dev);
    return cudaSuccess;
}

void host_stage_free(HostStage* st) {
    if (st->host) cudaFreeHost(st->host);
    st->host = st->dev = nullptr;
    st->bytes = 0;
}

cudaError_t read_arrays(int count, const uint32_t* const* dev_src, uint32_t* const* host_dst, int n,
                        HostStage* stage, cudaStream_t s) {
    std::lock_guard<std::mutex> hold(stage->mu);
    uint32_t *host = nullptr, *dev = nullptr;
    const int total = count * n;
    cudaError_t e = host_stage(stage, sizeof(uint32_t) * (size_t)total, &host, &dev);
    if (e != cudaSuccess) return e;
    k_read_arrays<<<(total + kThreads - 1) / kThreads, kThreads, 0, s>>>(
        dev_src[0], count > 1 ? dev_src[1] : nullptr, count > 2 ? dev_src[2] : nullptr, n, total, dev);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    for (int k = 0; k < count && e == cudaSuccess; ++k)
        if (host_dst[k]) std::memcpy(host_dst[k], host + (size_t)k * n, sizeof(uint32_t) * (size_t)n);
    return e;
}

void raster_sort_free(RasterSort* w) {
    void* ptrs[] = {w->group, w->key, w->step, w->id};
    for (void* p : ptrs) cudaFree(p);
    *w = RasterSort();
}

void raster_sort_done(RasterSort* w) {
    if (w->step_cap > kSortKeep) raster_sort_free(w);
}

cudaError_t raster_read_small(const RasterList& in, uint32_t* counts, HostStage* stage, cudaStream_t s,
                              RasterSmall* out) {
    constexpr size_t kHead = 4;
    uint32_t *host = nullptr, *dev = nullptr;
    cudaError_t e = host_stage(stage, (kHead + 2 * (size_t)kSmall) * sizeof(uint32_t), &host, &dev);
    if (e != cudaSuccess) return e;
    SortParams p = common_params(in);
    p.step_out = dev + kHead;
    p.id_out = dev + kHead + kSmall;
    k_sort_small<<<1, kSmall, 0, s>>>(p, counts, dev);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return e;
    out->n = (uint64_t)host[1] << 32 | host[0];
    out->lost = host[2] != 0u;
    out->done = out->n <= kSmall;
    out->step = host + kHead;
    out->id = host + kHead + kSmall;
    return cudaSuccess;
}

cudaError_t raster_sort_host(const RasterList& in, uint64_t n, uint64_t limit, const int32_t* goff,
                             uint32_t* steps, uint32_t* ids, cudaStream_t s) {
    constexpr size_t kPiece = 1u << 20;
    std::vector<uint32_t> cnt(in.n_part), st(kPiece), id(kPiece);
    std::vector<uint64_t> key;                   // step since t_lo, id
    key.reserve(n);
    cudaError_t e = cudaMemcpyAsync(cnt.data(), in.counts, sizeof(uint32_t) * in.n_part, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    for (int c = 0; c < in.n_part && e == cudaSuccess; ++c) {
        const size_t m = std::min(cnt[c], in.cap_part), base = (size_t)c * in.cap_part;
        for (size_t at = 0; at < m && e == cudaSuccess; at += kPiece) {
            const size_t k = std::min(kPiece, m - at);
            e = cudaMemcpyAsync(st.data(), in.step + base + at, sizeof(uint32_t) * k, cudaMemcpyDeviceToHost, s);
            if (e == cudaSuccess)
                e = cudaMemcpyAsync(id.data(), in.id + base + at, sizeof(uint32_t) * k, cudaMemcpyDeviceToHost, s);
            if (e == cudaSuccess) e = cudaStreamSynchronize(s);
            for (size_t i = 0; i < k; ++i) key.push_back((uint64_t)(st[i] - in.t_lo) << 32 | id[i]);
        }
    }
    if (e != cudaSuccess) return e;
    std::sort(key.begin(), key.end());
    if (in.n_inst > 1) {
        auto inst = [&](uint64_t x) { return std::upper_bound(goff, goff + in.n_inst + 1, (int32_t)(uint32_t)x) - goff; };
        std::stable_sort(key.begin(), key.end(), [&](uint64_t a, uint64_t b) { return inst(a) < inst(b); });
    }
    limit = std::min<uint64_t>(limit, key.size());
    for (uint64_t i = 0; i < limit; ++i) {
        if (steps) steps[i] = in.t_lo + (uint32_t)(key[i] >> 32);
        if (ids) ids[i] = (uint32_t)key[i];
    }
    return cudaSuccess;
}

cudaError_t raster_sort(RasterSort* w, const RasterList& in, size_t n, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    if (n > 0xffffffffull) return cudaErrorMemoryAllocation;     // 32-bit places
    SortParams p = common_params(in);
    const long long span = std::max<long long>(1, in.t_span);
    const long long most = std::max<long long>(1, kMaxGroups / in.n_inst);
    while ((((span - 1) >> p.shift) + 1) > most) ++p.shift;
    p.per_inst = (uint32_t)(((span - 1) >> p.shift) + 1);
    p.n_groups = p.per_inst * (uint32_t)in.n_inst;
    p.n = (uint32_t)n;
    cudaError_t e = grow(&w->step, &w->step_cap, n);
    if (e == cudaSuccess) e = grow(&w->id, &w->id_cap, n);
    if (e == cudaSuccess) e = grow(&w->group, &w->group_cap, p.n_groups);
    if (e == cudaSuccess) e = grow(&w->key, &w->key_cap, 2 * n);
    if (e != cudaSuccess) {
        raster_sort_free(w);
        if (e == cudaErrorMemoryAllocation) cudaGetLastError();      // not sticky: the caller sorts on the host
        return e;
    }
    p.step_out = w->step;
    p.id_out = w->id;
    p.group = w->group;
    p.key = w->key;
    p.key2 = w->key + n;
    e = cudaMemsetAsync(p.group, 0, sizeof(uint32_t) * p.n_groups, s);
    if (e != cudaSuccess) return e;
    // about 4 spikes a thread, at most 8 CTAs per SM in all
    const size_t per_part = n / (size_t)in.n_part + 1;
    const unsigned y = (unsigned)std::min<size_t>(std::max<size_t>(1216 / in.n_part, 1), (per_part + 1023) / 1024);
    k_sort_count<<<dim3(in.n_part, y), kThreads, 0, s>>>(p);
    k_sort_scan<<<1, 1024, 0, s>>>(p);
    k_sort_scatter<<<dim3(in.n_part, y), kThreads, 0, s>>>(p);
    const unsigned warps = (p.n_groups + kThreads / 32 - 1) / (kThreads / 32);
    k_sort_groups<<<std::min(warps, 2432u), kThreads, 0, s>>>(p);
    k_sort_large<<<std::min(p.n_groups, 304u), kBigThreads, 0, s>>>(p);
    return cudaGetLastError();
}

}  // namespace snn

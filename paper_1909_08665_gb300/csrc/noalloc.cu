// noalloc.cu -- snn_step_noalloc: the time-step kernel on caller-owned device
// memory, for callers that must not allocate device memory at run time.
//
// A closed-loop application that steps the network every 0.1 ms (a robot
// controller, an experiment rig driven in real time) typically reserves all
// of its device memory once, from its own pool, and may not call cudaMalloc
// or cudaFree while it runs: those calls can synchronise the whole device
// and take an unbounded time.  This entry point therefore allocates nothing.
// The caller passes the network, the state and the output buffers as device
// pointers; the kernel's scratch (spike messages and status words) lives in
// the file-scope array g_noalloc_scratch below, which every GPU that loads
// this library holds (about 4.3 MiB) until the process exits.
//
// The kernel has the step kernel's structure (step_kernel.cuh): CTA c owns the
// neurons [c n / P, (c + 1) n / P), state in registers, ring slice in shared
// memory for the launch, spikes exchanged as tagged messages, the spikes of
// step t - 1 delivered after the membrane update of step t.  What it cannot
// have is the step kernel's per-network store (pre-decoded rows, run bounds):
// it reads the caller's packed rows.  Rows ascend by target, so a partition's
// run of a row is contiguous, and where it lies follows from the connection
// probabilities: about len f words into the row, f the expected share of its
// words below the partition, give or take sqrt(len f (1 - f)).  A warp spreads
// 32 probes over the words within kNaSigmas of that, then loads the words
// between the two probes that enclose the run and tests each word's target;
// the probes touched most of those sectors already.  It walks on in either
// direction where the outermost probe does not prove the run complete, so any
// rows of ascending targets give the right result, and rows like the network's
// own cost one L2 round trip.  What bounds a step is that trip, the message's and the run's,
// and in large networks the SM's own intake: a probe costs a 32-byte sector,
// 1 KB per (spike, partition).  Measured, us per step at full size, in the
// versions in which each was decided: 64 probes over the whole row 6.07 and
// every word of the window loaded and tested 6.34, against 5.15 with 32 probes
// of the window; four rows per warp at once 5.15, one 4.48; 16 or 8 probes 4.80
// and 4.90, 32 4.48; 512 threads 4.48, 1024 4.13; the count at the CTA barrier
// 4.13, published by the last warp on a barrier of its own 3.91 (now 3.87).
//
// What it replaced, one warp walking each spike's whole row with an L2 atomic
// per word between two grid barriers, was bound by the chain of a row's
// dependent loads: 130 us per step at full size, 48 us at the 10 % scale; now
// 3.87 and 1.69.
//
// The paper has no counterpart of this entry point.
#include <algorithm>
#include <cstring>
#include <mutex>

#include "../../include/snn.h"
#include "step_kernel.cuh"

namespace snn {

int host_step_constants(const snn_config* cfg, float prop[4], float cdc[kMaxPop],
                        uint64_t pois[kMaxPop][kPoisTable], int32_t* wext_q, int32_t* n_ref);
int set_error(int code, const char* msg);
int set_cuda_error(cudaError_t e, const char* what);

namespace {

// Threads per CTA: a step of a small network waits on L2 round trips and
// barriers, which cost less with 16 warps; in larger ones every warp has
// spikes to deliver and 32 hide more of their loads.  us per step with 512 /
// 1024 threads: scale 0.1 1.81 / 2.05, 0.5
// 2.81 / 2.85, 0.7 3.53 / 3.40, 1.0 4.59 / 4.13
constexpr int kNaFewThreads = 512, kNaManyThreads = 1024;
constexpr int kNaWide = 42000;          // neurons from which on 1024 threads are taken
constexpr int kNaPart = 512;            // most partitions, and the neurons of one where SMs allow
constexpr int kNaMaxDevices = 64;
constexpr int kNaChunk = 384;           // spikes listed at once
constexpr int kNaInline = 3;            // spikes read together with a message header (64 B)
constexpr int kNaWave = 2;              // words of a row per lane before the first add
constexpr uint32_t kNaProbes = 32;      // probes of a window, one per lane
// half width of the window over the expected run, in standard deviations: one
// (spike, partition) pair in 4e4 has to walk on, about one step in 6 at full
// size (46 spikes x 151 partitions)
constexpr float kNaSigmas = 4.2f;
// scratch: [8] status, [9] abort, from kNaHeader on the spike messages
// [4][n_part][stride] of 64-bit words.  Every word carries its own tag in its
// top bits (the launch step / 4 + 1: four messages rotate), so a matching tag
// is the wait and the data at once.  Word 0 is the count; words 2 + 2 i and
// 3 + 2 i, i < kNaInline, are a spike's id and row length (kNaLong: look it up
// in row_ptr) and its row's start, so that the usual few spikes of a partition
// need no row_ptr lookup on the consumer's side; words 8 + i - kNaInline are
// the ids of the others.
constexpr int kNaTagShift = 41;         // 23-bit tags: n_steps <= 2^24
constexpr unsigned long long kNaValMask = (1ull << kNaTagShift) - 1ull;
constexpr int kNaLenBits = 22;          // id (19 bits) << 22 | row length
constexpr uint32_t kNaLong = (1u << kNaLenBits) - 1u;
constexpr size_t kNaHeader = 64;
constexpr size_t kNaMsgWords = 4 * ((size_t)SNN_NOALLOC_MAX_NEURONS + 16 * (size_t)kNaPart);
constexpr size_t kNaScratchWords = kNaHeader + 2 * kNaMsgWords;

static __device__ __align__(256) uint32_t g_noalloc_scratch[kNaScratchWords];

struct NaParams {
    int32_t n, n_pop, n_part, ncmax, w_span, msg_stride;
    int32_t pop_start[kMaxPop + 1];
    float P22, P21, P11, theta;
    float cdc[kMaxPop];
    float prob[kMaxPop][kMaxPop];       // relative connection probabilities [target][source]
    int32_t n_ref, wext_q, mode;
    uint32_t key0, key1;
    int64_t t0;
    int32_t n_steps;
    uint64_t timeout_ns;
    uint32_t pois_m1[kMaxPop][kPoisTable];  // Poisson thresholds minus 1
    const unsigned long long* row_ptr;
    const uint32_t* words;
    const int32_t* wtab;
    float* u;
    float* i_syn;
    int32_t* refr;
    int32_t* ring;                      // [64][n]
    uint32_t* ras_step;
    uint32_t* ras_id;
    uint32_t* ras_n;
    uint32_t ras_cap;
    unsigned long long* counters;
    uint32_t* status;                   // caller's word: | 1 on a timed-out wait
    uint32_t* scratch;                  // device address of g_noalloc_scratch
    unsigned long long* msg;            // its message words
};

// shared memory (bytes): thresholds, scan partials, flags, the expected window
// of each source population's rows, the list of rows to deliver (the first
// word of the window, its place in the row, the window's length, the row's
// length, the source population), the weight-table rows of the
// partition's target populations, each local neuron's offset into them, then
// the ring slice [64][ncmax] where it fits
struct NaSmem {
    uint32_t pois, warp, misc, rs, win, la, lw, rl, rq, w, popo, ring, total;
};

__host__ __device__ inline NaSmem na_smem(int ncmax, int w_span, bool smem_ring) {
    NaSmem L;
    uint32_t o = 0;
    L.rs = o;     o += kNaChunk * 8;
    L.pois = o;   o += kMaxPop * kPoisTable * 4;
    L.warp = o;   o += 32 * 4;
    L.misc = o;   o += 32 * 4;
    L.win = o;    o += kMaxPop * 16;
    L.la = o;     o += kNaChunk * 4;
    L.lw = o;     o += kNaChunk * 4;
    L.rl = o;     o += kNaChunk * 4;
    L.w = o;      o += (uint32_t)w_span * kPopWords * 4;
    L.rq = o;     o += kNaChunk;
    L.popo = o;   o += align_up((uint32_t)ncmax * 2, 4);
    L.ring = o;
    if (smem_ring) o += (uint32_t)kRing * (uint32_t)ncmax * 4;
    L.total = o;
    return L;
}

// poll one message word until it carries `tag`; false once a wait gave up
__device__ inline bool na_poll(const NaParams& p, const unsigned long long* at, uint32_t tag,
                               unsigned long long& w) {
    uint64_t t_start = 0;
    uint32_t iter = 0;
    while ((uint32_t)(w >> kNaTagShift) != tag) {
        if (iter == 0) t_start = globaltimer_ns();
        if ((++iter & 31u) == 0u) {
            if (ld_relaxed_gpu(p.scratch + 9) != 0u) return false;
            if (globaltimer_ns() - t_start > p.timeout_ns || iter > 0x7fffffffu) {
                atomicOr(p.scratch + 8, kStatusTimeout);
                atomicOr(p.status, kStatusTimeout);
                atomicExch(p.scratch + 9, 1u);
                return false;
            }
        }
        w = __ldcg(at);
    }
    return true;
}

// the expected position of partition [lo, hi) in a row of source population q,
// as shares of the row's length, and the window's half width per sqrt(length)
__device__ float4 na_window(const NaParams& p, int q, int32_t lo, int32_t hi) {
    float below = 0.f, upto = 0.f, total = 0.f;
    for (int k = 0; k < p.n_pop; ++k) {
        const int32_t a = p.pop_start[k], b = p.pop_start[k + 1];
        const float w = p.prob[k][q];
        total += w * (float)(b - a);
        below += w * (float)(min(max(lo, a), b) - a);
        upto += w * (float)(min(max(hi, a), b) - a);
    }
    const bool some = total > 0.f;
    const float f0 = some ? below / total : (float)lo / (float)p.n;
    const float f1 = some ? upto / total : (float)hi / (float)p.n;
    const float var = fmaxf(f0 * (1.f - f0), f1 * (1.f - f1));
    return make_float4(f0, f1, kNaSigmas * sqrtf(fmaxf(var, 0.f)), 0.f);
}

// ring[i] += w where ok (a predicated reduction, no branch)
template <bool SMEM_RING>
__device__ __forceinline__ void na_add(int32_t* ring, uint32_t ring_s, size_t i, int32_t w, bool ok) {
    if (SMEM_RING)
        asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t@q red.shared.add.s32 [%0], %1;\n\t}"
                     ::"r"(ring_s + 4u * (uint32_t)i), "r"(w), "r"((uint32_t)ok) : "memory");
    else
        asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t@q red.global.add.s32 [%0], %1;\n\t}"
                     ::"l"(ring + i), "r"(w), "r"((uint32_t)ok) : "memory");
}

// distance of the probes of a window of n words
__device__ __forceinline__ uint32_t na_gap(uint32_t n) { return (n + kNaProbes - 1u) / kNaProbes; }

struct NaList {
    unsigned long long* rs;             // words + rs: the window's first word
    uint32_t* a;                        // its place in the row
    uint32_t* w;                        // words of the window
    uint32_t* len;                      // words of the row
    uint8_t* q;                         // source population
};

// the listed rows' words that target neurons [lo, hi), added into ring slots
// tb + delay: cell(slot, local) = ring[slot * stride + local]
template <int THREADS, bool SMEM_RING>
__device__ __forceinline__ void na_deliver(const NaParams& p, const NaList& list, const int32_t* s_w,
                                           const uint16_t* s_popo, uint32_t m, uint32_t tb,
                                           uint32_t lo, uint32_t hi, int32_t* ring, size_t stride) {
    constexpr uint32_t kNaWarps = THREADS / 32;
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const uint32_t nc = hi - lo;
    const uint32_t ring_s = SMEM_RING ? (uint32_t)__cvta_generic_to_shared(ring) : 0u;
    // branch-free, so that the lookups of a batch's words overlap
    auto add = [&](uint32_t word, const int32_t* wq) {
        const uint32_t local = (word & kTgtMask) - lo;
        const bool ok = local < nc;
        const uint32_t l = ok ? local : 0u;
        const uint32_t slot = (tb + ((word >> kTgtBits) & 63u)) & (kRing - 1);
        na_add<SMEM_RING>(ring, ring_s, slot * stride + l, wq[s_popo[l] + (word >> 25)], ok);
    };
    constexpr uint32_t kOut = kTgtMask;              // no neuron has this index
    static_assert(kNaProbes == 32u, "one probe per lane");
    for (uint32_t i = warp; i < m; i += kNaWarps) {
        // (the branches on the list and on lengths are the same for all lanes)
        const uint32_t n = list.w[i], gap = na_gap(n);
        const uint32_t* row = p.words + list.rs[i];  // the window's first word
        uint32_t probe = kOut;
        if (lane * gap < n) probe = __ldg(row + lane * gap) & kTgtMask;
        const uint32_t nl = __popc(__ballot_sync(0xffffffffu, probe < lo));
        const uint32_t nh = __popc(__ballot_sync(0xffffffffu, probe < hi));
        // after the last probe below lo; before the first one past hi (a lane
        // without a probe counts as past, its place is past n)
        const uint32_t c0 = nl ? (nl - 1u) * gap + 1u : 0u;
        const uint32_t c1 = min(nh * gap, n);
        uint32_t e[kNaWave];
#pragma unroll
        for (int h = 0; h < kNaWave; ++h) {
            const uint32_t x = c0 + lane + 32u * (uint32_t)h;
            e[h] = kOut;
            if (x < c1) e[h] = __ldg(row + x);
        }
        const int32_t* wq = s_w + (uint32_t)list.q[i] * kWCodes;
        add(e[0], wq);
#pragma unroll
        for (int h = 1; h < kNaWave; ++h)
            if (c0 + 32u * (uint32_t)h < c1) add(e[h], wq);
        for (uint32_t x = c0 + 32u * kNaWave; x < c1; x += 32u)
            add(x + lane < c1 ? __ldg(row + x + lane) : kOut, wq);
        const bool low = c0 == 0u, high = c1 == n;
        if (low || high) {
            const uint32_t a = list.a[i], len = list.len[i];
            const uint32_t* r = row - a;             // the row's first word
            // no probe below the partition: 32 words at a time towards the
            // row's start, until one lies below it
            for (uint32_t end = low ? a : 0u; end > 0u;) {
                const uint32_t from = end > 32u ? end - 32u : 0u, x = from + lane;
                const uint32_t word = x < end ? __ldg(r + x) : kOut;
                add(word, wq);
                end = from;
                if (__any_sync(0xffffffffu, (word & kTgtMask) < lo)) break;
            }
            // no probe past it: on, until a word lies past it
            for (uint32_t from = high ? a + n : len; from < len; from += 32u) {
                const uint32_t x = from + lane;
                const uint32_t word = x < len ? __ldg(r + x) : 0u;
                add(x < len ? word : kOut, wq);
                if (__any_sync(0xffffffffu, (word & kTgtMask) >= hi)) break;
            }
        }
    }
}

template <int THREADS, int NPT, bool SMEM_RING>
__global__ void __launch_bounds__(THREADS, 1) k_step_noalloc(const __grid_constant__ NaParams p) {
    extern __shared__ __align__(16) unsigned char smem[];
    const NaSmem L = na_smem(p.ncmax, p.w_span, SMEM_RING);
    uint32_t* s_pois = reinterpret_cast<uint32_t*>(smem + L.pois);
    uint32_t* s_warp = reinterpret_cast<uint32_t*>(smem + L.warp);
    // [0], [1] this CTA's spikes of even / odd launch steps, [2] abort, [3], [4]
    // listed rows of lists of even / odd launch steps
    volatile uint32_t* s_misc = reinterpret_cast<uint32_t*>(smem + L.misc);
    const NaList list = {reinterpret_cast<unsigned long long*>(smem + L.rs),
                         reinterpret_cast<uint32_t*>(smem + L.la),
                         reinterpret_cast<uint32_t*>(smem + L.lw),
                         reinterpret_cast<uint32_t*>(smem + L.rl), smem + L.rq};
    float4* s_win = reinterpret_cast<float4*>(smem + L.win);
    int32_t* s_w = reinterpret_cast<int32_t*>(smem + L.w);
    uint16_t* s_popo = reinterpret_cast<uint16_t*>(smem + L.popo);
    const int tid = threadIdx.x, lane = tid & 31;
    const int c = blockIdx.x, P = p.n_part;
    const int32_t lo = (int32_t)(((long long)c * p.n) / P);
    const int32_t hi = (int32_t)(((long long)(c + 1) * p.n) / P);
    const int32_t nc = hi - lo;
    const size_t n = (size_t)p.n;
    int32_t* ring = SMEM_RING ? reinterpret_cast<int32_t*>(smem + L.ring) : p.ring + lo;
    const size_t stride = SMEM_RING ? (size_t)p.ncmax : n;

    for (int k = tid; k < kMaxPop * kPoisTable; k += THREADS)
        s_pois[k] = p.pois_m1[k / kPoisTable][k % kPoisTable];
    if (tid < kMaxPop) s_win[tid] = na_window(p, tid, lo, hi);
    const int p_lo = pop_index(p.pop_start, p.n_pop, lo);
    for (uint32_t k = tid; k < (uint32_t)p.w_span * kPopWords; k += THREADS) {
        const uint32_t gk = (uint32_t)p_lo * kPopWords + k;
        s_w[k] = gk < (uint32_t)kMaxPop * kPopWords ? __ldg(&p.wtab[gk]) : 0;
    }
    for (int i = tid; i < nc; i += THREADS)
        s_popo[i] = (uint16_t)((pop_index(p.pop_start, p.n_pop, lo + i) - p_lo) * (int)kPopWords);
    if (SMEM_RING)
        for (int slot = tid >> 5; slot < kRing; slot += (THREADS / 32))
            for (int i = lane; i < nc; i += 32) ring[slot * p.ncmax + i] = p.ring[slot * n + lo + i];
    if (tid < 32) s_misc[tid] = 0u;

    float u[NPT], isyn[NPT];
    int32_t refr[NPT], pacc[NPT], pop[NPT];
    uint4 rnd[NPT];
    // the neuron's own row: prefetched into L2 when it spikes, and counted
    unsigned long long row[NPT];
    uint32_t row_n[NPT];
    // the raster position of this step's spikes, taken when they are found and
    // used at the end of the step, when it has long arrived
    uint32_t ras_at[NPT], ras_mask[NPT];
#pragma unroll
    for (int k = 0; k < NPT; ++k) {
        const int li = tid + k * THREADS;
        u[k] = 0.f; isyn[k] = 0.f; refr[k] = 0; pop[k] = 0; pacc[k] = 0;
        rnd[k] = make_uint4(0u, 0u, 0u, 0u);
        row[k] = 0ull; row_n[k] = 0u;
        ras_at[k] = 0u; ras_mask[k] = 0u;
        if (li < nc) {
            u[k] = p.u[lo + li];
            isyn[k] = p.i_syn[lo + li];
            refr[k] = p.refr[lo + li];
            pop[k] = pop_index(p.pop_start, p.n_pop, lo + li);
            row[k] = p.row_ptr[lo + li];
            row_n[k] = (uint32_t)(p.row_ptr[lo + li + 1] - row[k]);
        }
    }
    unsigned long long spikes = 0, events = 0;
    bool aborted = false;
    __syncthreads();

    // list position `at`: the row of neuron `id`, with the window its run is
    // expected in
    auto put_row = [&](uint32_t at, uint32_t id, unsigned long long b, uint32_t len) {
        const int q = pop_index(p.pop_start, p.n_pop, (int32_t)id);
        const float4 w = s_win[q];
        const float fl = (float)len, half = w.z * __fsqrt_rn(fl) + 2.f;
        const uint32_t x0 = min((uint32_t)fmaxf(fl * w.x - half, 0.f), len);
        const uint32_t x1 = min(max((uint32_t)(fl * w.y + half), x0), len);
        list.rs[at] = b + x0;
        list.a[at] = x0;
        list.w[at] = x1 - x0;
        list.len[at] = len;
        list.q[at] = (uint8_t)q;
    };
    auto look_up = [&](uint32_t at, uint32_t id) {
        const unsigned long long b = __ldg(&p.row_ptr[id]);
        put_row(at, id, b, (uint32_t)(__ldg(&p.row_ptr[id + 1]) - b));
    };
    // delivery of the spikes of launch step s (step tb); h: the message head
    // of partition tid, loaded by the caller (words polled again when stale)
    auto deliver = [&](int s, uint32_t tb, ulonglong2 (&h)[4]) -> bool {
        const uint32_t tag = ((uint32_t)s >> 2) + 1u;
        const unsigned long long* m_mine = p.msg + ((size_t)(s & 3) * P + tid) * p.msg_stride;
        uint32_t my_cnt = 0u;
        if (tid < P) {
            if (na_poll(p, m_mine, tag, h[0].x)) my_cnt = (uint32_t)h[0].x;
            else s_misc[2] = 1u;
        }
        // spike i of the message into list position at (row 0 if a wait gave up)
        auto list_inline = [&](uint32_t at, int i) {
            unsigned long long x = h[1 + i].x, y = h[1 + i].y;
            if (na_poll(p, m_mine + 2 + 2 * i, tag, x) && na_poll(p, m_mine + 3 + 2 * i, tag, y)) {
                const uint32_t id = (uint32_t)(x >> kNaLenBits) & kTgtMask, len = (uint32_t)x & kNaLong;
                if (len != kNaLong) put_row(at, id, y & kNaValMask, len);
                else look_up(at, id);
            } else {
                s_misc[2] = 1u;
                put_row(at, 0u, 0ull, 0u);
            }
        };
        auto list_other = [&](uint32_t at, uint32_t i) {
            const unsigned long long* mp = m_mine + 8 + (i - (uint32_t)kNaInline);
            unsigned long long x = __ldcg(mp);
            if (na_poll(p, mp, tag, x)) {
                look_up(at, (uint32_t)(x & kNaValMask));
            } else {
                s_misc[2] = 1u;
                put_row(at, 0u, 0ull, 0u);
            }
        };
        if (tid < P && my_cnt > 0u) {
            const uint32_t at = atomicAdd(const_cast<uint32_t*>(&s_misc[3 + (s & 1)]), my_cnt);
            if (at + my_cnt <= (uint32_t)kNaChunk) {
#pragma unroll
                for (int i = 0; i < kNaInline; ++i)
                    if ((uint32_t)i < my_cnt) list_inline(at + (uint32_t)i, i);
                for (uint32_t i = kNaInline; i < my_cnt; ++i) list_other(at + i, i);
            }
        }
        __syncthreads();
        const uint32_t S_fast = s_misc[3 + (s & 1)];
        if (tid == 0) s_misc[3 + ((s + 1) & 1)] = 0u;   // its last readers are past a barrier
        if (s_misc[2]) return false;
        if (S_fast <= (uint32_t)kNaChunk) {
            na_deliver<THREADS, SMEM_RING>(p, list, s_w, s_popo, S_fast, tb, (uint32_t)lo, (uint32_t)hi, ring, stride);
            __syncthreads();
            return true;
        }
        // more than kNaChunk spikes: offsets by a block-wide scan, in chunks
        const uint32_t incl = warp_incl_scan(my_cnt);
        if (lane == 31) s_warp[tid >> 5] = incl;
        __syncthreads();
        uint32_t my_off = incl - my_cnt;
        for (int w = 0; w < (tid >> 5); ++w) my_off += s_warp[w];
        const uint32_t S = S_fast;
        for (uint32_t base = 0; base < S; base += kNaChunk) {
            const uint32_t m = min((uint32_t)kNaChunk, S - base);
            if (tid < P) {
                const uint32_t i0 = base > my_off ? base - my_off : 0u;
                const uint32_t i1 = base + m > my_off ? min(my_cnt, base + m - my_off) : 0u;
#pragma unroll
                for (int i = 0; i < kNaInline; ++i)
                    if ((uint32_t)i >= i0 && (uint32_t)i < i1) list_inline(my_off + (uint32_t)i - base, i);
                for (uint32_t i = max(i0, (uint32_t)kNaInline); i < i1; ++i) list_other(my_off + i - base, i);
            }
            __syncthreads();
            na_deliver<THREADS, SMEM_RING>(p, list, s_w, s_popo, m, tb, (uint32_t)lo, (uint32_t)hi, ring, stride);
            __syncthreads();
        }
        return s_misc[2] == 0u;
    };
    auto load_head = [&](int s, ulonglong2 (&h)[4]) {
#pragma unroll
        for (int q = 0; q < 4; ++q) h[q] = make_ulonglong2(0ull, 0ull);
        if (s >= 0 && tid < P) {
            const ulonglong2* m = reinterpret_cast<const ulonglong2*>(
                p.msg + ((size_t)(s & 3) * P + tid) * p.msg_stride);
#pragma unroll
            for (int q = 0; q < 4; ++q) h[q] = __ldcg(m + q);
        }
    };

    for (int s = 0; s < p.n_steps; ++s) {
        const int64_t t = p.t0 + s;
        const unsigned long long tag = (unsigned long long)(((uint32_t)s >> 2) + 1u) << kNaTagShift;
        unsigned long long* my_msg = p.msg + ((size_t)(s & 3) * P + c) * p.msg_stride;
        ulonglong2 h[4];
        load_head(s - 1, h);
        // ---- A(t): membrane, threshold; the spikes' message words ----
#pragma unroll
        for (int k = 0; k < NPT; ++k) {
            const int li = tid + k * THREADS;
            bool spk = false;
            if (li < nc) {
                if (refr[k] > 0) {
                    refr[k] -= 1;
                    u[k] = 0.f;
                } else {
                    float v = __fadd_rn(__fmul_rn(p.P22, u[k]), __fmul_rn(p.P21, isyn[k]));
                    if (p.mode == 1) v = __fadd_rn(v, p.cdc[pop[k]]);
                    u[k] = v;
                }
                if (u[k] > p.theta) {
                    spk = true;
                    u[k] = 0.f;
                    refr[k] = p.n_ref;
                }
            }
            const unsigned mask = __ballot_sync(0xffffffffu, spk);
            ras_mask[k] = mask;
            if (mask) {
                uint32_t base = 0;
                if (lane == 0) base = atomicAdd(const_cast<uint32_t*>(&s_misc[s & 1]), (uint32_t)__popc(mask));
                base = __shfl_sync(0xffffffffu, base, 0);
                if (spk) {
                    const uint32_t at = base + (uint32_t)__popc(mask & ((1u << lane) - 1u));
                    const uint32_t id = (uint32_t)(lo + li);
                    if (at < (uint32_t)kNaInline) {
                        const bool fits = row_n[k] < kNaLong && row[k] <= kNaValMask;
                        __stcg(&my_msg[2 + 2 * at], tag | (unsigned long long)id << kNaLenBits |
                                                        (fits ? row_n[k] : kNaLong));
                        __stcg(&my_msg[3 + 2 * at], tag | (fits ? row[k] : 0ull));
                    } else {
                        __stcg(&my_msg[8 + at - (uint32_t)kNaInline], tag | id);
                    }
                    if (row_n[k]) {
                        // the row, rounded out to 16 bytes (never past the
                        // 16-byte granule of its first or last word)
                        const unsigned long long a = reinterpret_cast<unsigned long long>(p.words + row[k]);
                        const unsigned long long a0 = a & ~15ull;
                        prefetch_l2(a0, (uint32_t)((a + 4ull * row_n[k] + 15ull - a0) & ~15ull));
                    }
                    events += row_n[k];
                }
                if (lane == 0) ras_at[k] = atomicAdd(p.ras_n, (uint32_t)__popc(mask));
            }
        }
        // the count, published by the last warp once all have arrived here
        if (tid < THREADS - 32) {
            barrier_arrive(1, THREADS);
        } else {
            barrier_wait(1, THREADS);
            if (tid == THREADS - 32) {
                const uint32_t nsp = s_misc[s & 1];
                s_misc[(s + 1) & 1] = 0u;       // read last in step s - 1
                __stcg(&my_msg[0], tag | nsp);
                spikes += nsp;
            }
        }
        // ---- background counts of step t ----
#pragma unroll
        for (int k = 0; k < NPT; ++k) {
            const int li = tid + k * THREADS;
            if (p.mode == 0 && li < nc) {
                if ((t & 3) == 0 || s == 0)
                    rnd[k] = philox(make_uint4((uint32_t)(lo + li), (uint32_t)(t >> 2), kStreamPois,
                                               (uint32_t)(t >> 34)), p.key0, p.key1);
                // k = #{m : x >= T_m} = #{m : x > T_m - 1}; thresholds ascend
                const uint32_t x = lane_of(rnd[k], (int)(t & 3));
                const uint32_t* thr = s_pois + pop[k] * kPoisTable;
                int kk = 0;
#pragma unroll
                for (int mm = 0; mm < 12; ++mm) kk += x > thr[mm] ? 1 : 0;
                if (kk == 12)
                    for (int mm = 12; mm < kPoisTable; ++mm) kk += x > thr[mm] ? 1 : 0;
                pacc[k] = kk * p.wext_q;
            }
        }
        // ---- D: spikes of step t - 1 ----
        if (s == 0) __syncthreads();            // the counter's reset before step 1's adds
        if (s > 0 && !deliver(s - 1, (uint32_t)(t - 1), h)) {
            aborted = true;
            break;
        }
        // ---- C(t): ring slot t, background, synaptic current; raster ----
        const size_t slot = (size_t)((uint32_t)t & (kRing - 1)) * stride;
#pragma unroll
        for (int k = 0; k < NPT; ++k) {
            const int li = tid + k * THREADS;
            if (li < nc) {
                const int32_t acc = (int32_t)((uint32_t)ring[slot + li] + (uint32_t)pacc[k]);
                ring[slot + li] = 0;
                isyn[k] = __fadd_rn(__fmul_rn(p.P11, isyn[k]),
                                    __fmul_rn(__int2float_rn(acc), 0.00390625f));
            }
            if (ras_mask[k]) {
                const uint32_t at = __shfl_sync(0xffffffffu, ras_at[k], 0) +
                                    (uint32_t)__popc(ras_mask[k] & ((1u << lane) - 1u));
                if (((ras_mask[k] >> lane) & 1u) && at < p.ras_cap) {
                    p.ras_step[at] = (uint32_t)t;
                    p.ras_id[at] = (uint32_t)(lo + li);
                }
            }
        }
    }
    if (!aborted) {
        ulonglong2 h[4];
        load_head(p.n_steps - 1, h);
        deliver(p.n_steps - 1, (uint32_t)(p.t0 + p.n_steps - 1), h);
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < NPT; ++k) {
        const int li = tid + k * THREADS;
        if (li < nc) {
            p.u[lo + li] = u[k];
            p.i_syn[lo + li] = isyn[k];
            p.refr[lo + li] = refr[k];
        }
    }
    if (SMEM_RING)
        for (int slot = tid >> 5; slot < kRing; slot += (THREADS / 32))
            for (int i = lane; i < nc; i += 32) p.ring[slot * n + lo + i] = ring[slot * p.ncmax + i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) events += __shfl_xor_sync(0xffffffffu, events, o);
    if (lane == 0 && events) atomicAdd(&p.counters[1], events);
    if (tid == THREADS - 32 && spikes) atomicAdd(&p.counters[0], spikes);
}

// one neuron per thread covers every network on the full GPU; eight take over
// where fewer SMs are visible.  The ring of the few threads' partitions always
// fits in shared memory.
template <bool SMEM_RING>
const void* na_kernel(int threads, int ncmax) {
    if (threads == kNaFewThreads) return reinterpret_cast<const void*>(&k_step_noalloc<kNaFewThreads, 1, true>);
    if (ncmax <= kNaManyThreads) return reinterpret_cast<const void*>(&k_step_noalloc<kNaManyThreads, 1, SMEM_RING>);
    return reinterpret_cast<const void*>(&k_step_noalloc<kNaManyThreads, 8, SMEM_RING>);
}
const void* na_kernel(int threads, int ncmax, bool smem_ring) {
    return smem_ring ? na_kernel<true>(threads, ncmax) : na_kernel<false>(threads, ncmax);
}

// Partitions of n neurons: one CTA per SM at most and at most 512 neurons
// each where that is possible; networks too small for that are spread to
// kNaFew neurons per CTA, where the CTA's own work no longer sets the time of
// a step (a step waits on L2 round trips and barriers, not on the neurons):
// scale 0.1 with 49 partitions of 158 neurons 2.45 us per step, with 16 of
// 482 2.60, both in the version with 64 probes a row.
constexpr int kNaFew = 160;
int na_partitions(long long n, int sms) {
    const long long need = (n + kNaPart - 1) / kNaPart;
    const long long spread = std::min<long long>((n + kNaFew - 1) / kNaFew, 64);
    return (int)std::max<long long>(1, std::min<long long>(std::min(sms, kNaPart), std::max(need, spread)));
}

// set-up of each device, done once by its first call: the scratch array's
// device address, the architecture check, the SM count, the shared memory a
// CTA may take and the kernels' attributes (so that a call only fills
// parameters, clears the scratch and launches)
struct NaDevice {
    uint32_t* scratch;
    cudaError_t err;
    const char* what;                   // the set-up call that failed
    bool arch_ok;
    int sms, optin;
};
std::once_flag g_setup_once[kNaMaxDevices];
NaDevice g_dev[kNaMaxDevices];

void setup_device(int dev) {
    NaDevice& d = g_dev[dev];
    d.what = "cudaGetSymbolAddress(g_noalloc_scratch)";
    d.err = cudaGetSymbolAddress(reinterpret_cast<void**>(&d.scratch), g_noalloc_scratch);
    if (d.err != cudaSuccess) return;
    cudaDeviceProp prop;
    d.what = "cudaGetDeviceProperties";
    d.err = cudaGetDeviceProperties(&prop, dev);
    if (d.err != cudaSuccess) return;
    d.arch_ok = prop.major == 10 && prop.minor == 3;
    d.sms = prop.multiProcessorCount;
    d.what = "shared memory attributes";
    d.err = cudaDeviceGetAttribute(&d.optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    for (bool ring : {true, false})
        for (const void* fn : {na_kernel(kNaFewThreads, 1, ring), na_kernel(kNaManyThreads, 1, ring),
                               na_kernel(kNaManyThreads, 8 * kNaManyThreads, ring)})
            if (d.err == cudaSuccess)
                d.err = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, d.optin);
}

}  // namespace
}  // namespace snn

using namespace snn;

extern "C" int snn_step_noalloc(const snn_config* cfg, uint64_t seed, const snn_noalloc_io* io,
                                int64_t t0, int64_t n_steps, void* stream) {
    if (!cfg || !io) return set_error(SNN_ERR_INVALID, "config and io are required");
    if (n_steps < 0 || n_steps > (1 << 24) || t0 < 0)
        return set_error(SNN_ERR_INVALID, "need 0 <= n_steps <= 2^24 and t0 >= 0");
    long long n = 0;
    if (cfg->n_pop >= 1 && cfg->n_pop <= kMaxPop)
        for (int q = 0; q < cfg->n_pop; ++q) n += cfg->pop_size[q];
    if (n > SNN_NOALLOC_MAX_NEURONS)
        return set_error(SNN_ERR_INVALID,
                         "snn_step_noalloc supports at most SNN_NOALLOC_MAX_NEURONS (131072) "
                         "neurons: its static scratch holds the spike messages of that many");
    NaParams p;
    std::memset(&p, 0, sizeof(p));
    float pr[4];
    uint64_t pois[kMaxPop][kPoisTable];
    int rc = host_step_constants(cfg, pr, p.cdc, pois, &p.wext_q, &p.n_ref);
    if (rc != SNN_OK) return rc;
    for (int q = 0; q < kMaxPop; ++q)
        for (int m = 0; m < kPoisTable; ++m)   // T >= 1 (validation bounds lambda)
            p.pois_m1[q][m] = (uint32_t)(pois[q][m] - 1u);
    p.P22 = pr[0];
    p.P21 = pr[1];
    p.P11 = pr[2];
    if (!io->row_ptr || !io->words || !io->wtab || !io->u || !io->i_syn || !io->refr ||
        !io->ring || !io->ras_step || !io->ras_id || !io->ras_n || !io->counters || !io->status)
        return set_error(SNN_ERR_INVALID, "every io pointer is required");
    if (n_steps == 0) return SNN_OK;

    // once per device, with that device current: device address of the scratch
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return set_cuda_error(e, "cudaGetDevice");
    if (dev < 0 || dev >= kNaMaxDevices) return set_error(SNN_ERR_UNSUPPORTED, "device index too large");
    std::call_once(g_setup_once[dev], setup_device, dev);
    const NaDevice& d = g_dev[dev];
    if (d.err != cudaSuccess) return set_cuda_error(d.err, d.what);
    if (!d.arch_ok)
        return set_error(SNN_ERR_UNSUPPORTED, "this library is built for sm_103 (GB300) GPUs only");
    const int P = na_partitions(n, d.sms);
    int32_t part_lo[kNaPart + 1], pop_start[kMaxPop + 1] = {0};
    int ncmax = 0;
    for (int c = 0; c <= P; ++c) {
        part_lo[c] = (int32_t)(((long long)c * n) / P);
        if (c) ncmax = std::max(ncmax, part_lo[c] - part_lo[c - 1]);
    }
    for (int q = 0; q < kMaxPop; ++q) pop_start[q + 1] = pop_start[q] + (q < cfg->n_pop ? cfg->pop_size[q] : 0);
    p.w_span = partition_pop_span(part_lo, P, pop_start, cfg->n_pop);
    p.ncmax = ncmax;
    for (int q = 0; q < cfg->n_pop; ++q)
        for (int k = 0; k < cfg->n_pop; ++k) p.prob[k][q] = (float)std::min(cfg->conn_prob[k][q], 1.0);
    p.msg_stride = 8 + (ncmax + 7) / 8 * 8;
    const bool smem_ring = na_smem(ncmax, p.w_span, true).total <= (uint32_t)d.optin;
    const size_t smem = na_smem(ncmax, p.w_span, smem_ring).total;
    const int threads = n > kNaWide || ncmax > kNaFewThreads || !smem_ring ? kNaManyThreads : kNaFewThreads;
    const void* fn = na_kernel(threads, ncmax, smem_ring);
    if (ncmax > 8 * kNaManyThreads || smem > (size_t)d.optin) return set_error(SNN_ERR_UNSUPPORTED, "step kernel does not fit an SM");
    const size_t msg_words = (size_t)4 * P * p.msg_stride;
    static_assert(kNaHeader % 2 == 0, "the message words are 8-byte aligned");
    if (msg_words > kNaMsgWords) return set_error(SNN_ERR_UNSUPPORTED, "spike messages exceed the scratch");

    p.n = (int32_t)n;
    p.n_pop = cfg->n_pop;
    p.n_part = P;
    for (int q = 0; q <= kMaxPop; ++q) p.pop_start[q] = pop_start[q];
    p.theta = (float)cfg->theta;
    p.mode = cfg->input_mode;
    p.key0 = (uint32_t)(seed & 0xffffffffu);
    p.key1 = (uint32_t)(seed >> 32);
    p.t0 = t0;
    p.n_steps = (int32_t)n_steps;
    p.timeout_ns = 2000000000ull;
    p.row_ptr = reinterpret_cast<const unsigned long long*>(io->row_ptr);
    p.words = io->words;
    p.wtab = io->wtab;
    p.u = io->u;
    p.i_syn = io->i_syn;
    p.refr = io->refr;
    p.ring = io->ring;
    p.ras_step = io->ras_step;
    p.ras_id = io->ras_id;
    p.ras_n = io->ras_n;
    p.ras_cap = (uint32_t)std::min<int64_t>(std::max<int64_t>(io->ras_cap, 0), 0x7fffffff);
    p.counters = io->counters;
    p.status = io->status;
    p.scratch = d.scratch;
    p.msg = reinterpret_cast<unsigned long long*>(d.scratch + kNaHeader);

    // the shared scratch keeps the previous call's contents: clear the status
    // words and the messages, whose tags count from the start of the launch
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    e = cudaMemsetAsync(p.scratch, 0, sizeof(uint32_t) * kNaHeader + sizeof(unsigned long long) * msg_words, s);
    if (e != cudaSuccess) return set_cuda_error(e, "clearing the scratch");
    void* args[] = {&p};
    e = cudaLaunchCooperativeKernel(fn, dim3(P), dim3(threads), args, smem, s);
    if (e != cudaSuccess) return set_cuda_error(e, "launch of the allocation-free step kernel");
    return SNN_OK;
}

// adjoint_part.cu -- the surrogate-gradient adjoint (the recursion of grad.cu,
// Sec. 2.1 Eq. 1 run backwards) with its row gather done partition by
// partition, for networks whose rows fit in the SMs' shared memory.
//
// The gather of step t is ds_j = gs + sum over row j of (w / 256) lI_{i,t+d},
// d >= 1, and lI_t = P11 lI_{t+1} + m_{t+1} P21 lu_{t+1}: the gather of step
// t - 1 needs lu_{t+1} and so the partials of step t + 1, but not those of
// step t.  A CTA therefore gathers step t - 1 while the grid barrier of step
// t's partials completes, watched by a warp of its own, and only then adds
// them up into lu_t.  It writes step t - 1's partials over step t + 1's after
// that barrier, which every CTA reached after it had read the latter.  The
// entries of delay 1 ("near") are walked after the others ("far") and
// cover the round trip of the partials.  Measured on the 10 % network, us per
// step (backward of 2000 recorded steps): 7.5 with the wait before the
// membrane adjoint and all it needs, 6.4 with the spike flags and partials
// fetched ahead, 5.8 in this order.  What bounds it now: the shared-memory
// wavefronts of the far walk (2.3 us: entry 1, weight and window 2.3 each on
// random banks), then the round trip of freshly written partials (1 us).
//
// Gathered from a global lI ring, it costs one L2 request per synapse and
// step.  Here the targets are split into the network's partitions and the
// sources of each partition into G groups: CTA (c, g) keeps, for the whole
// launch, the lI window of partition c (slots t + 1 .. t + R - 1 of its
// neurons) and the runs of its source group into c (the pre-decoded entries,
// re-packed as weight index and window cell offset) in shared memory.  Its
// share of the gather then reads shared memory only.  Each source's partial
// sum over its run into c goes to a global array; after the step's grid
// barrier every CTA of partition c adds the partials of its partition's
// neurons over all partitions (a fixed order) and runs the membrane adjoint of
// those neurons itself -- redundantly in the G CTAs, identically -- so the
// lI_t it writes into its window needs no second barrier.  The CTA of group 0
// alone writes the outputs (the lI ring, the nu sums and, at the end, the
// adjoint state).
//
// A lane takes one source, or one chunk of a source's run when the run is
// longer than kApChunk entries (up to kApMaxChunks chunks in consecutive
// lanes, added in chunk order by the first): every sum has a fixed order.
// Sources are sorted by chunk length, dealt to the groups in snake order and
// packed 32 lanes to a lane group, their entries stored column by column
// (entry k of lane l at k * 32 + l), so that a warp walks 32 runs of similar
// length with conflict-free entry loads.  A run shorter than its group's longest is padded
// with entries of weight zero (exact: x + 0 * lI = x for the finite lI), so
// the walk has no per-entry test and its loads pipeline.  Lane groups are
// dealt to the warps longest first, each to the least loaded warp.
#include <algorithm>
#include <vector>

#include "snn_internal.cuh"

namespace snn {
namespace {

constexpr int kApThreads = 512;
constexpr int kApWarps = kApThreads / 32;
constexpr int kApLaunch = kApThreads + 32;   // and the warp that watches the grid barrier
constexpr uint32_t kApNone = 0xffffffffu;
constexpr uint32_t kApWBits = 19;            // weight index << 19 | window cell offset
constexpr uint32_t kApOffMask = (1u << kApWBits) - 1u;
constexpr uint32_t kApChunk = 32;           // entries per lane before a run is split
constexpr uint32_t kApMaxChunks = 4;         // lanes one source's run is split over
constexpr int kApPre = 4;                    // neurons per thread in the membrane phase (ncmax <= 2048)
constexpr int kApPart = 16;                  // partials of a neuron in flight
constexpr int kApFlags = 2;                  // spike flags per thread in flight
constexpr int kApHeader = 8;                 // n_lg, nc, p_lo, span, e_off, 0, 0, 0
// header, then for the entries of delay >= 2 ("far") lenmax[n_lg] and
// ebase[n_lg], for those of delay 1 ("near") lenmax[n_lg] and ebase[n_lg],
// src[32 n_lg], chunks[32 n_lg] (m on a source's first lane, else 0),
// warp_first[kApWarps + 1], lg_order[n_lg], then the entries at e_off

// the chunks of a source added in order, on its first lane (m chunks, else 0)
__device__ __forceinline__ float add_chunks(float v, uint32_t m) {
    float tot = v;
#pragma unroll
    for (uint32_t r = 1; r < kApMaxChunks; ++r) {
        const float w = __shfl_down_sync(0xffffffffu, v, r);
        if (r < m) tot = __fadd_rn(tot, w);
    }
    return tot;
}

// The walk of a lane group with a spiking source: its sum as in the plain
// walk, and the spiking lanes' weight partials, one per target population of
// the partition, added into ga.  A CTA with such a group is the last to
// arrive, and nearly every step has some: with PW = 8 sums an entry costs 35
// instructions, with the 2 that a partition usually spans 17, without 9.
template <int PW>
__device__ __forceinline__ void walk_spiking(const uint32_t* ep, uint32_t lm, uint32_t base_t, uint32_t RW,
                                             const float* win, const float* wf, const float* wb, bool spk,
                                             uint32_t m, double* ga, uint32_t span, float& acc) {
    float pa[PW];
#pragma unroll
    for (int k = 0; k < PW; ++k) pa[k] = 0.f;
#pragma unroll 4
    for (uint32_t k = 0; k < lm; ++k) {
        const uint32_t e = ep[k * 32];
        const uint32_t wi = e >> kApWBits;
        const uint32_t a = base_t + (e & kApOffMask);
        const float lv = win[min(a, a - RW)];
        acc = __fadd_rn(acc, __fmul_rn(wf[wi], lv));
        // (lanes without a spike drop their sums)
        const float v = __fmul_rn(wb[wi], lv);
        const uint32_t pr = wi / (kMaxPop * kWCodes);
#pragma unroll
        for (int kk = 0; kk < PW; ++kk) pa[kk] = __fadd_rn(pa[kk], kk == (int)pr ? v : 0.f);
    }
#pragma unroll
    for (int kk = 0; kk < PW; ++kk) {
        const float t2 = add_chunks(pa[kk], m);
        if (m > 0u && spk && (uint32_t)kk < span) atomicAdd(&ga[kk], (double)t2);   // nothing waits for it
    }
}

__global__ void __launch_bounds__(kApLaunch, 1)
k_adjoint_part(const __grid_constant__ AdjPartParams p) {
    extern __shared__ __align__(16) uint32_t s_img[];
    __shared__ volatile uint32_t s_abort;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int c = (int)blockIdx.x / p.groups, g = (int)blockIdx.x % p.groups;
    const uint32_t ncmax = (uint32_t)p.ncmax, R = (uint32_t)p.ring_r;
    // window rows padded to whole 32-word bank rounds: a cell's bank is
    // its target's, whatever the slot (the plan orders entries by it)
    const uint32_t ws = (ncmax + 31u) & ~31u;
    const size_t n = (size_t)p.n;
    // shared memory: the image [img_max], the window [R][ws], the weights
    // of the partition's target populations (forward, pA; base) and the
    // adjoint state of its neurons
    float* win = reinterpret_cast<float*>(s_img + p.img_max);
    float* wf = win + (size_t)R * ws;
    float* wb = wf + (size_t)p.span_max * kMaxPop * kWCodes + 4;
    // one zero past each table: the weight of the padding entries
    const uint32_t w_zero = (uint32_t)p.span_max * kMaxPop * kWCodes;
    float* s_lu = wb + w_zero + 4;
    float* s_lI = s_lu + ncmax;
    float* s_far = s_lI + ncmax;                 // [max_lg][32] far sums of the lanes
    // group 0: the nu sums of the partition's neurons, accumulated here in
    // the order the global ones would be, read in at the start, written at the end
    double* s_gN = reinterpret_cast<double*>(
        (reinterpret_cast<uintptr_t>(s_far + (size_t)p.max_lg * 32) + 7) & ~uintptr_t(7));
    uint8_t* s_mn = reinterpret_cast<uint8_t*>(s_gN + ncmax);

    if (tid == 0) s_abort = 0u;
    {
        const uint32_t o0 = p.img_off[blockIdx.x], words = p.img_off[blockIdx.x + 1] - o0;
        const uint4* src = reinterpret_cast<const uint4*>(p.img + o0);   // offsets are multiples of 4
        uint4* dst = reinterpret_cast<uint4*>(s_img);
        for (uint32_t k = tid; k < words / 4; k += kApLaunch) dst[k] = __ldg(&src[k]);
    }
    __syncthreads();
    const uint32_t n_lg = s_img[0], nc = s_img[1], p_lo = s_img[2], span = s_img[3];
    const uint32_t* lenmax = s_img + kApHeader;      // far columns
    const uint32_t* ebase = lenmax + n_lg;
    const uint32_t* lenmax_n = ebase + n_lg;         // near columns
    const uint32_t* ebase_n = lenmax_n + n_lg;
    const uint32_t* srcs = ebase_n + n_lg;
    // a word per lane slot: its chunks (m on a source's first lane, else 0) and
    // the spike flags of its source in the even and the odd steps, loaded a step
    // ahead, so that no walk waits for them (arrays of their own would take 64
    // bytes per lane group, 1 % of the shared memory: networks near its limit
    // would no longer fit)
    uint8_t* lane_b = reinterpret_cast<uint8_t*>(s_img + kApHeader + 36 * n_lg);
    auto spk_of = [&](uint32_t slot, int64_t tt) -> uint8_t& { return lane_b[4u * slot + 1u + (uint32_t)(tt & 1)]; };
    const uint32_t* warp_first = srcs + 64 * n_lg;
    const uint32_t* lg_order = warp_first + kApWarps + 1;
    const uint32_t* ent = s_img + s_img[4];
    const int32_t lo = p.part_lo[c];
    for (uint32_t k = tid; k < span * kMaxPop * kWCodes; k += kApLaunch) {
        const uint32_t gk = p_lo * kMaxPop * kWCodes + k;
        wf[k] = __fmul_rn(__int2float_rn(__ldg(&p.wtab[gk])), 0.00390625f);
        wb[k] = __ldg(&p.wbase[gk]);
    }
    if (tid < 4) {
        wf[w_zero + tid] = 0.f;
        wb[w_zero + tid] = 0.f;
    }
    for (uint32_t i = tid; i < nc; i += kApLaunch) {
        s_lu[i] = p.lu[lo + i];
        s_lI[i] = p.lI[lo + i];
        s_mn[i] = p.mnext[lo + i];
        if (g == 0) s_gN[i] = p.gN[lo + i];
    }
    // the window of the first step processed, t_top: lI of steps t_top + d
    const int64_t t_top = p.t_first + p.len - 1;
    for (uint32_t k = tid; k < (R - 1) * nc; k += kApLaunch) {
        const uint32_t d = 1 + k / nc, i = k - (d - 1) * nc;
        const int64_t tt = t_top + d;
        win[(uint32_t)(tt % R) * ws + i] = __ldcg(&p.lring[(size_t)(tt & (kRing - 1)) * n + lo + i]);
    }
    __syncthreads();

    const uint32_t RW = R * ws;               // window words
    // The gather of step tt, far (delay >= 2) or near (delay 1: window step
    // tt + 1).  The far sums wait in s_far; the near walk adds them, combines a
    // source's chunks and writes its partial.  Spiking sources' weight
    // partials go to gAc after each walk.
    auto walk = [&](int64_t tt, uint32_t tDt, bool far) {
        const uint32_t base_t = tDt * ws;
        for (uint32_t wl = warp_first[warp]; wl < warp_first[warp + 1]; ++wl) {
            const uint32_t L = lg_order[wl];
            const uint32_t j = srcs[L * 32 + lane];
            const uint32_t lm = far ? lenmax[L] : lenmax_n[L];
            const uint32_t eb = far ? ebase[L] : ebase_n[L];
            const bool spk = (spk_of(L * 32 + lane, tt) & 1u) != 0u;
            const uint32_t m = lane_b[4u * (L * 32 + lane)];
            const uint32_t* ep = ent + eb + lane;
            float acc = 0.f;
            // entry: weight index << 19 | delay * ws + target; the window
            // cell of step tt + delay is that offset plus tt's row, wrapped
            // (a - RW is huge where a < RW).  Few lane groups hold a spiking
            // source: the others walk without its weight partials.
            if (!__any_sync(0xffffffffu, spk)) {
#pragma unroll 8
                for (uint32_t k = 0; k < lm; ++k) {
                    const uint32_t e = ep[k * 32];
                    const uint32_t a = base_t + (e & kApOffMask);
                    acc = __fadd_rn(acc, __fmul_rn(wf[e >> kApWBits], win[min(a, a - RW)]));
                }
            } else if (span <= 2u) {
                walk_spiking<2>(ep, lm, base_t, RW, win, wf, wb, spk, m,
                                p.gAc + ((size_t)c * n + (spk ? j : 0u)) * kMaxPop, span, acc);
            } else {
                walk_spiking<kMaxPop>(ep, lm, base_t, RW, win, wf, wb, spk, m,
                                      p.gAc + ((size_t)c * n + (spk ? j : 0u)) * kMaxPop, span, acc);
            }
            // the chunks of a source sit in consecutive lanes; its first lane
            // (m > 0) adds them in chunk order
            if (far) {
                s_far[L * 32 + lane] = acc;
            } else {
                acc = __fadd_rn(s_far[L * 32 + lane], acc);
                const float tot = add_chunks(acc, m);
                if (m > 0u) {
                    float* pds = p.pds + (size_t)(tt & 1) * p.n_part * n;
                    __stcg(&pds[(size_t)c * n + j], tot);
                }
            }
        }
    };
    // Grid barrier k: the partials of step t_top - k are written.  The last
    // warp watches it while the others gather.
    auto arrive = [&]() {
        __syncthreads();
        // the watching warp waits for the partials' writes, no gathering one
        if (tid == kApThreads) red_release_gpu_add(p.barrier, 1u);
    };
    auto watch = [&](int k) {
        const uint32_t target = ((uint32_t)k + 1u) * gridDim.x;
        const uint64_t t_start = globaltimer_ns();
        uint32_t iter = 0;
        while (ld_acquire_gpu(p.barrier) < target) {
            if ((++iter & 255u) == 0u) {
                if (ld_relaxed_gpu(p.abort_flag) != 0u) { s_abort = 1u; break; }
                if (globaltimer_ns() - t_start > p.timeout_ns) {
                    atomicOr(p.status, kStatusTimeout);
                    atomicExch(p.abort_flag, 1u);
                    s_abort = 1u;
                    break;
                }
            }
        }
    };

    // spike flag of lane slot k (lane group k / 32) in trace row `row`
    uint32_t my_src[kApFlags];
#pragma unroll
    for (int k = 0; k < kApFlags; ++k) {
        const uint32_t i = (uint32_t)tid + (uint32_t)k * kApThreads;
        my_src[k] = i < 32u * n_lg ? srcs[i] : kApNone;
    }
    auto flag_of = [&](uint32_t k, int row) -> uint8_t {
        const uint32_t j = srcs[k];
        uint8_t f = 0;
        if (j != kApNone) f = __ldg(p.tr_f + (size_t)row * n + j);
        return f;
    };
    // the trace of the partition's neurons in row `row`
    float u_pre[kApPre];
    uint8_t f_pre[kApPre];
    auto load_trace = [&](int row) {
#pragma unroll
        for (int k = 0; k < kApPre; ++k) {
            const uint32_t i = (uint32_t)tid + (uint32_t)k * kApThreads;
            u_pre[k] = 0.f;
            f_pre[k] = 0;
            if (tid < kApThreads && i < nc) {
                u_pre[k] = __ldg(p.tr_u + (size_t)row * n + lo + i);
                f_pre[k] = __ldg(p.tr_f + (size_t)row * n + lo + i);
            }
        }
    };
    load_trace(p.len - 1);
    for (uint32_t k = tid; k < 32u * n_lg; k += kApLaunch) {
        spk_of(k, t_top) = flag_of(k, p.len - 1);
        if (p.len > 1) spk_of(k, t_top - 1) = flag_of(k, p.len - 2);
    }
    __syncthreads();
    uint32_t tD = (uint32_t)(t_top % R);      // window slot of step t
    // step t_top's gather, both parts, before the first barrier
    if (warp < kApWarps) {
        walk(t_top, tD, true);
        __syncwarp();
        walk(t_top, tD, false);
    }
    arrive();
    // Step t: lI_t follows from lu_{t+1}; with it the gather of step t - 1 is
    // done while the partials of step t come in, and lu_t last of all.
    for (int s = p.len - 1; s >= 0; --s) {
        const int64_t t = p.t_first + s;
        const int k_bar = p.len - 1 - s;
        if (warp == kApWarps) {                       // the watching warp
            __syncthreads();
            if (lane == 0) watch(k_bar);
            __syncthreads();
            if (s_abort != 0u) break;
            if (s > 0) arrive();
            continue;
        }
        const uint32_t tD1 = tD == 0u ? R - 1u : tD - 1u;     // window slot of step t - 1
        // ---- lI_t and what else of step t needs no partials ----
        float slope[kApPre], keep[kApPre];            // s'(u_t); (1 - s_t) m_{t+1} P22 lu_{t+1}
#pragma unroll
        for (int kp = 0; kp < kApPre; ++kp) {
            const uint32_t i = (uint32_t)tid + (uint32_t)kp * kApThreads;
            slope[kp] = keep[kp] = 0.f;
            if (i < nc) {
                const uint8_t f = f_pre[kp];
                const bool mn = s_mn[i] != 0u;
                const float lu1 = s_lu[i];
                const float lub = mn ? __fmul_rn(p.P22, lu1) : 0.f;
                const float lIt = __fadd_rn(__fmul_rn(p.P11, s_lI[i]), mn ? __fmul_rn(p.P21, lu1) : 0.f);
                const float sv = (f & 1u) ? 1.f : 0.f;
                const float x = __fsub_rn(u_pre[kp], p.theta);
                const float a = __fadd_rn(1.0f, __fmul_rn(10.0f, fabsf(x)));
                slope[kp] = __fdiv_rn(1.0f, __fmul_rn(a, a));
                keep[kp] = __fmul_rn(__fsub_rn(1.f, sv), lub);
                s_lI[i] = lIt;
                s_mn[i] = (uint8_t)((f >> 1) & 1u);
                win[tD * ws + i] = lIt;
                if (g == 0) s_gN[i] += (double)lIt;
            }
        }
        __syncthreads();
        // the trace of step t - 1 and the spike flags of step t - 2 (into step
        // t's place: its walks are done), in flight during the gather
        uint8_t nf[kApFlags];
        if (s > 0) load_trace(s - 1);
        if (s > 1) {
            const uint8_t* fl = p.tr_f + (size_t)(s - 2) * n;
#pragma unroll
            for (int k = 0; k < kApFlags; ++k) {
                nf[k] = 0;
                if (my_src[k] != kApNone) nf[k] = __ldg(fl + my_src[k]);
            }
        }
        if (s > 0) walk(t - 1, tD1, true);
        if (s > 1) {
#pragma unroll
            for (int k = 0; k < kApFlags; ++k) {
                const uint32_t i = (uint32_t)tid + (uint32_t)k * kApThreads;
                if (i < 32u * n_lg) spk_of(i, t) = nf[k];
            }
            for (uint32_t i = (uint32_t)tid + kApFlags * kApThreads; i < 32u * n_lg; i += kApThreads)
                spk_of(i, t) = flag_of(i, s - 2);
        }
        __syncthreads();                              // the partials of step t are there
        if (s_abort != 0u) break;
        const float* pds_t = p.pds + (size_t)(t & 1) * p.n_part * n + lo;
        // a neuron's first kApPart partials, in flight during the near walk
        float v[kApPart];
#pragma unroll
        for (int r = 0; r < kApPart; ++r)
            v[r] = (uint32_t)tid < nc && r < p.n_part ? __ldcg(&pds_t[(size_t)r * n + tid]) : 0.f;
        if (s > 0) walk(t - 1, tD1, false);
        // ---- lu_t: the partials added in the partitions' order ----
#pragma unroll
        for (int kp = 0; kp < kApPre; ++kp) {
            const uint32_t i = (uint32_t)tid + (uint32_t)kp * kApThreads;
            if (i >= nc) break;
            float acc = 0.f;
            for (int c0 = 0; c0 < p.n_part; c0 += kApPart) {
                if (kp > 0 || c0 > 0) {
#pragma unroll
                    for (int r = 0; r < kApPart; ++r)
                        v[r] = c0 + r < p.n_part ? __ldcg(&pds_t[(size_t)(c0 + r) * n + i]) : 0.f;
                }
#pragma unroll
                for (int r = 0; r < kApPart; ++r)
                    if (c0 + r < p.n_part) acc = __fadd_rn(acc, v[r]);
            }
            const float ds = __fadd_rn(p.gs[pop_index(p.pop_start, p.n_pop, lo + (int32_t)i)], acc);
            s_lu[i] = __fadd_rn(__fmul_rn(ds, slope[kp]), keep[kp]);
        }
        if (s > 0) arrive();
        tD = tD1;
    }
    __syncthreads();
    if (g == 0 && s_abort == 0u) {
        for (uint32_t i = tid; i < nc; i += kApLaunch) {
            p.lu[lo + i] = s_lu[i];
            p.lI[lo + i] = s_lI[i];
            p.mnext[lo + i] = s_mn[i];
            p.gN[lo + i] = s_gN[i];
        }
        // the lI ring of the next launch (the segment before): steps t_first
        // .. t_first + R - 2, which the window holds now
        for (uint32_t k = tid; k < (R - 1) * nc; k += kApLaunch) {
            const uint32_t d = k / nc, i = k - d * nc;
            const int64_t tt = p.t_first + d;
            p.lring[(size_t)(tt & (kRing - 1)) * n + lo + i] = win[(uint32_t)(tt % R) * ws + i];
        }
    }
}

// gA[j][p] += the partition partials of source j, partitions in order
__global__ void __launch_bounds__(256) k_adjoint_part_fold(int32_t n, int32_t n_part, int32_t n_pop,
                                                           const int32_t* __restrict__ part_lo,
                                                           const int32_t* __restrict__ pop_start,
                                                           const double* __restrict__ gAc,
                                                           double* __restrict__ gA) {
    const int32_t j = (int32_t)(blockIdx.x * 256u + threadIdx.x);
    if (j >= n) return;
    int32_t ps[kMaxPop + 1];
    for (int k = 0; k <= kMaxPop; ++k) ps[k] = pop_start[k];
    for (int c = 0; c < n_part; ++c) {
        if (part_lo[c + 1] <= part_lo[c]) continue;
        const int p_lo = pop_index(ps, n_pop, part_lo[c]);
        const double* src = gAc + ((size_t)c * n + j) * kMaxPop;
        for (int k = 0; p_lo + k < kMaxPop; ++k) gA[(size_t)j * kMaxPop + p_lo + k] += src[k];
    }
}

}  // namespace

bool adjoint_part_possible(int n_part, int ncmax, uint64_t nnz) {
    int dev = 0, sms = 0, optin = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
        return false;
    const int G = sms / std::max(1, n_part);
    // each CTA's share of the rows must fit next to the window and the tables
    return G >= 1 && ncmax <= kApPre * kApThreads && (double)nnz * 4.0 / ((double)n_part * G) <= (double)optin * 0.7;
}

int adjoint_part_plan(int n, int n_pop, const int32_t* pop_start, int n_part, const int32_t* part_lo,
                      int ncmax, uint64_t nnz, const unsigned long long* d_row_start,
                      const uint32_t* d_pre, const uint32_t* d_seg, AdjPartPlan* plan) {
    *plan = AdjPartPlan();
    int dev = 0, sms = 0, optin = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
        return -1;
    if (n <= 0 || !adjoint_part_possible(n_part, ncmax, nnz)) return 1;
    const int G = sms / n_part;
    std::vector<unsigned long long> rs(n + 1);
    std::vector<uint32_t> pre(nnz), seg((size_t)n * (n_part + 1));
    if (cudaMemcpy(rs.data(), d_row_start, sizeof(unsigned long long) * (n + 1), cudaMemcpyDeviceToHost) != cudaSuccess ||
        (nnz && cudaMemcpy(pre.data(), d_pre, sizeof(uint32_t) * nnz, cudaMemcpyDeviceToHost) != cudaSuccess) ||
        cudaMemcpy(seg.data(), d_seg, sizeof(uint32_t) * seg.size(), cudaMemcpyDeviceToHost) != cudaSuccess)
        return -1;
    auto pop_of = [&](int32_t i) {
        int q = 0;
        for (int k = 1; k < n_pop; ++k) q += i >= pop_start[k] ? 1 : 0;
        return q;
    };
    // target populations per partition; the padding entries index the zero
    // past the widest partition's table, which must fit the 13-bit index
    int span_max = 1;
    for (int c = 0; c < n_part; ++c)
        if (part_lo[c + 1] > part_lo[c])
            span_max = std::max(span_max, pop_of(part_lo[c + 1] - 1) - pop_of(part_lo[c]) + 1);
    const uint32_t w_zero = (uint32_t)span_max * kMaxPop * kWCodes;
    if (w_zero >= (1u << (32 - kApWBits))) return 1;
    // window rows padded to whole bank rounds (as the kernel does)
    const uint32_t wsp = ((uint32_t)ncmax + 31u) & ~31u;
    if ((size_t)kRing * wsp > kApOffMask) return 1;
    const uint32_t e_pad = (w_zero << kApWBits) | wsp;            // delay 1, target 0, weight 0
    const uint32_t e_pad_far = (w_zero << kApWBits) | (2u * wsp);  // delay 2
    std::vector<uint32_t> img;
    std::vector<uint32_t> off(1, 0u);
    int R = 2;
    size_t img_max = 0;
    uint32_t max_lg = 0;
    for (int c = 0; c < n_part; ++c) {
        const int32_t nc = part_lo[c + 1] - part_lo[c];
        const int p_lo = nc > 0 ? pop_of(part_lo[c]) : 0;
        const int span = nc > 0 ? pop_of(part_lo[c + 1] - 1) - p_lo + 1 : 1;
        auto run_len = [&](int32_t j) {
            const uint32_t* sg = seg.data() + (size_t)j * (n_part + 1) + c;
            return sg[1] - sg[0];
        };
        // a source is one unit of m <= kApMaxChunks lanes: its run in chunks
        // of at most kApChunk entries (as equal as possible), one per lane
        struct Unit {
            int32_t j;
            uint32_t m, clen;                 // chunks, entries of the longest chunk
        };
        std::vector<Unit> units(n);
        for (int32_t j = 0; j < n; ++j) {
            const uint32_t len = run_len(j);
            const uint32_t m = std::min<uint32_t>(kApMaxChunks, std::max<uint32_t>(1u, (len + kApChunk - 1) / kApChunk));
            units[j] = Unit{j, m, (len + m - 1) / m};
        }
        // longest chunks first, dealt to the G groups in snake order (0 .. G-1,
        // G-1 .. 0, ...): every group gets the same mix of chunk lengths
        std::stable_sort(units.begin(), units.end(), [](const Unit& x, const Unit& y) { return x.clen > y.clen; });
        std::vector<std::vector<Unit>> groups(G);
        for (int32_t k = 0; k < n; ++k) {
            const int r = k % G, lap = k / G;
            groups[(lap & 1) ? G - 1 - r : r].push_back(units[k]);
        }
        for (int g = 0; g < G; ++g) {
            // lanes: source, chunk, entries; a unit never straddles two lane groups
            struct Lane {
                int32_t j;
                uint32_t m, k0, len;          // m on the unit's first lane only
            };
            std::vector<Lane> lanes;
            for (const Unit& u : groups[g]) {
                if (lanes.size() % 32 + u.m > 32)
                    while (lanes.size() % 32) lanes.push_back(Lane{-1, 0u, 0u, 0u});
                const uint32_t len = run_len(u.j);
                for (uint32_t q = 0; q < u.m; ++q) {
                    const uint32_t k0 = std::min(len, q * u.clen);
                    lanes.push_back(Lane{u.j, q == 0 ? u.m : 0u, k0, std::min(len, k0 + u.clen) - k0});
                }
            }
            const uint32_t n_lg = (uint32_t)((lanes.size() + 31) / 32);
            while (lanes.size() < (size_t)n_lg * 32) lanes.push_back(Lane{-1, 0u, 0u, 0u});
            const size_t o_wf = kApHeader + 4 * (size_t)n_lg + 64 * (size_t)n_lg;
            std::vector<uint32_t> head(o_wf + kApWarps + 1 + n_lg, 0u);
            head[0] = n_lg;
            head[1] = (uint32_t)nc;
            head[2] = (uint32_t)p_lo;
            head[3] = (uint32_t)span;
            std::vector<uint32_t> ents;
            for (uint32_t L = 0; L < n_lg; ++L) {
                // each lane's entries, re-packed, far (delay >= 2) and near (1)
                std::vector<uint32_t> le[2][32];
                for (uint32_t l = 0; l < 32; ++l) {
                    const Lane& ln = lanes[L * 32 + l];
                    for (uint32_t k = 0; ln.j >= 0 && k < ln.len; ++k) {
                        const uint32_t pe = pre[seg[(size_t)ln.j * (n_part + 1) + c] + ln.k0 + k];
                        const uint32_t off_e = pe & kPreOffMask;
                        const uint32_t d = off_e / (uint32_t)ncmax, loc = off_e % (uint32_t)ncmax;
                        const uint32_t wi = (pe >> kPreOffBits) - (uint32_t)p_lo * kMaxPop * kWCodes;
                        if (d < 1 || d >= (uint32_t)kRing || (int32_t)loc >= nc ||
                            wi >= (uint32_t)span * kMaxPop * kWCodes)
                            return -2;
                        R = std::max(R, (int)d + 1);
                        le[d == 1u ? 1 : 0][l].push_back((wi << kApWBits) | (d * wsp + loc));
                    }
                }
                for (int part = 0; part < 2; ++part) {
                    uint32_t lm = 0;
                    for (uint32_t l = 0; l < 32; ++l) lm = std::max(lm, (uint32_t)le[part][l].size());
                    head[kApHeader + 2 * part * n_lg + L] = lm;
                    head[kApHeader + (2 * part + 1) * n_lg + L] = (uint32_t)ents.size();
                    // padding: weight zero, a valid window cell of the part's delays
                    const uint32_t pad = part == 0 ? e_pad_far : e_pad;
                    // The order of a lane's entries is free (its sum has a
                    // fixed order either way): column k takes from each lane
                    // an entry whose weight bank (weight index mod 32) and
                    // window bank (target mod 32) no lane of the column used
                    // yet, if it has one; a lane with spare columns may wait
                    // (a zero-weight entry) rather than collide.  Lanes with
                    // the most entries left choose first.
                    std::vector<uint32_t>* lp = le[part];
                    for (uint32_t k = 0; k < lm; ++k) {
                        uint32_t used_w = 0u, used_l = 0u;
                        uint32_t col[32];
                        int ord[32];
                        for (int l = 0; l < 32; ++l) {
                            col[l] = pad;
                            ord[l] = l;
                        }
                        std::stable_sort(ord, ord + 32, [&](int x, int y) { return lp[x].size() > lp[y].size(); });
                        for (int oi = 0; oi < 32; ++oi) {
                            const int l = ord[oi];
                            if (lp[l].empty()) continue;
                            size_t best = 0;
                            int best_cost = 3;
                            for (size_t q = 0; q < lp[l].size(); ++q) {
                                const uint32_t e = lp[l][q];
                                const int cost = (int)((used_w >> ((e >> kApWBits) & 31u)) & 1u) +
                                                 (int)((used_l >> (e & 31u)) & 1u);
                                if (cost < best_cost) {
                                    best_cost = cost;
                                    best = q;
                                    if (cost == 0) break;
                                }
                            }
                            const bool slack = lp[l].size() < (size_t)(lm - k);
                            if (best_cost > 0 && slack) continue;
                            const uint32_t e = lp[l][best];
                            lp[l][best] = lp[l].back();
                            lp[l].pop_back();
                            used_w |= 1u << ((e >> kApWBits) & 31u);
                            used_l |= 1u << (e & 31u);
                            col[l] = e;
                        }
                        for (int l = 0; l < 32; ++l) ents.push_back(col[l]);
                    }
                }
            }
            for (uint32_t l = 0; l < 32 * n_lg; ++l) {
                head[kApHeader + 4 * n_lg + l] = lanes[l].j >= 0 ? (uint32_t)lanes[l].j : kApNone;
                head[kApHeader + 4 * n_lg + 32 * n_lg + l] = lanes[l].m;
            }
            // lane groups to warps, longest first, each to the least loaded warp
            std::vector<std::vector<uint32_t>> per_warp(kApWarps);
            std::vector<unsigned long long> load(kApWarps, 0ull);
            for (uint32_t L = 0; L < n_lg; ++L) {
                const int w = (int)(std::min_element(load.begin(), load.end()) - load.begin());
                per_warp[w].push_back(L);
                load[w] += head[kApHeader + L] + head[kApHeader + 2 * n_lg + L] + 1ull;
            }
            uint32_t pos = 0;
            for (int w = 0; w < kApWarps; ++w) {
                head[o_wf + w] = pos;
                for (uint32_t L : per_warp[w]) head[o_wf + kApWarps + 1 + pos++] = L;
            }
            head[o_wf + kApWarps] = pos;
            while (head.size() % 4) head.push_back(0u);
            head[4] = (uint32_t)head.size();
            head.insert(head.end(), ents.begin(), ents.end());
            while (head.size() % 4) head.push_back(0u);
            img.insert(img.end(), head.begin(), head.end());
            off.push_back((uint32_t)img.size());
            img_max = std::max(img_max, head.size());
            max_lg = std::max(max_lg, n_lg);
        }
    }
    const size_t ws = ((size_t)ncmax + 31) / 32 * 32;
    const size_t smem = img_max * 4 + (size_t)R * ws * 4 + (size_t)2 * (span_max * kMaxPop * kWCodes + 4) * 4 +
                        (size_t)ncmax * 8 + (size_t)max_lg * 32 * 4 + 8 + (size_t)ncmax * 8 + (size_t)ncmax;
    if (smem > (size_t)optin) return 1;
    plan->grid = n_part * G;
    plan->groups = G;
    plan->ring_r = R;
    plan->span_max = span_max;
    plan->img_max = (int32_t)img_max;
    plan->max_lg = (int32_t)max_lg;
    plan->smem = smem;
    cudaError_t e = cudaMalloc(&plan->d_img, sizeof(uint32_t) * std::max<size_t>(img.size(), 4));
    if (e == cudaSuccess) e = cudaMalloc(&plan->d_img_off, sizeof(uint32_t) * off.size());
    if (e == cudaSuccess) e = cudaMemcpy(plan->d_img, img.data(), sizeof(uint32_t) * img.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = cudaMemcpy(plan->d_img_off, off.data(), sizeof(uint32_t) * off.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = allow_shared(reinterpret_cast<const void*>(&k_adjoint_part));
    int per_sm = 0;
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_adjoint_part, kApLaunch, smem);
    if (e != cudaSuccess || per_sm * sms < plan->grid) {
        adjoint_part_free(plan);
        cudaGetLastError();
        return e != cudaSuccess ? -1 : 1;
    }
    return 0;
}

void adjoint_part_free(AdjPartPlan* plan) {
    if (plan->d_img) cudaFree(plan->d_img);
    if (plan->d_img_off) cudaFree(plan->d_img_off);
    *plan = AdjPartPlan();
}

cudaError_t launch_adjoint_part(const AdjPartPlan& plan, AdjPartParams& ap, cudaStream_t s) {
    ap.groups = plan.groups;
    ap.ring_r = plan.ring_r;
    ap.span_max = plan.span_max;
    ap.img_max = plan.img_max;
    ap.max_lg = plan.max_lg;
    ap.img = plan.d_img;
    ap.img_off = plan.d_img_off;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(plan.grid);
    cfg.blockDim = dim3(kApLaunch);
    cfg.dynamicSmemBytes = plan.smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    void* args[] = {&ap};
    return cudaLaunchKernelExC(&cfg, reinterpret_cast<const void*>(&k_adjoint_part), args);
}

cudaError_t launch_adjoint_part_fold(int n, int n_part, int n_pop, const int32_t* part_lo,
                                     const int32_t* pop_start, const double* gAc, double* gA,
                                     cudaStream_t s) {
    k_adjoint_part_fold<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(n, n_part, n_pop, part_lo, pop_start,
                                                                    gAc, gA);
    return cudaGetLastError();
}

}  // namespace snn

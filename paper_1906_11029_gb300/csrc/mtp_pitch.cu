// Tent pitching on the GPU (mtp_pitch_tents_device, see include/mtp.h): the same rounds and
// the same FP64 arithmetic as the host pitcher, so the tent list is bit-identical.
//
// A round (Sec. 2: vertices that are not neighbours may be advanced independently) selects every
// vertex V with tau_V < T that is a strict local minimum of (tau, id) over its neighbours and moves
// it to tau'_V = min(T, min_W tau_W + b_VW), all from the values at the start of the round.  There are
// thousands of rounds with little work each, so they run inside one cooperative kernel: a block
// owns a contiguous range of vertices, tau is double-buffered by the round's parity, and one grid
// barrier ends a round (its last arriver decides whether the rounds go on).  A block appends its
// tents to a list of its own; after kPitchChunk rounds, or when a list is full, two kernels order the
// lists by (round, block), which is (round, vertex) since blocks own ascending ranges.  (Three kernels a round
// took 37 us a round on a mesh of 4913 vertices, launches and their gaps for the most part;
// now 16 us, the barrier and dependent loads: 62 -> 26 ms for its 1644 rounds.)
//
// Layer = round: if V is selected in round r and no vertex of {V} u N(V) moved in round r - 1, V's
// test gave the same answer in round r - 1 and V would have moved then; so some vertex of the closed
// neighbourhood moved in round r - 1 and layer_V = 1 + max(last layers) = r by induction.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include <cuda_runtime.h>

#include "mtp_internal.h"

namespace mtp {

constexpr int kPitchThreads = 256;
constexpr int kPitchChunk = 128;              // rounds per launch at most
// List entries of a block per vertex it owns.  A round adds at most one a vertex, and the launch ends early when a
// block's list has no room for another round; usual meshes add 2 .. 5 % of the vertices a round, so that
// the lists (two of them, 20 bytes an entry) hold a launch's 128 rounds in 240 bytes a vertex.
constexpr int kPitchList = 6;
constexpr long long kPitchMaxRounds = 50000000;

struct PitchCtl {
    unsigned arrived;           // blocks that reached the barrier, over the whole launch
    unsigned released;          // rounds whose barrier is open
    int selected;               // vertices selected in the round
    int left;                   // vertices with tau < T
    int full;                   // a block's list has no room for another round
    int stop;                   // 1 all at T, 2 a round selected nothing, 3 a barrier wait expired, 4 full
    int rounds;                 // rounds done by the launch
};

struct PitchArgs {
    PitchCtl* ctl;
    int64_t nv;
    int vpb;                    // vertices per block
    int max_rounds;
    double T;
    const int64_t* ptr;
    const int32_t* dst;
    const double* bnd;
    double* tau;                // [2][nv]; the launch starts from half `start`
    int start;
    int64_t cap;                // list entries per block
    int32_t* lv;                // [block][cap]
    double* lb;
    double* lt;
    int* cnt;                   // [round][block]
};

__device__ __forceinline__ unsigned pitch_acquire(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__global__ void __launch_bounds__(kPitchThreads) pitch_rounds_kernel(const PitchArgs p) {
    __shared__ int warp_cnt[kPitchThreads / 32];
    __shared__ int s_stop;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t v0 = (int64_t)blockIdx.x * p.vpb, v1 = v0 + p.vpb < p.nv ? v0 + p.vpb : p.nv;
    int64_t len = 0;   // entries of this block's list
    for (int r = 0; r < p.max_rounds; ++r) {
        const double* cur = p.tau + ((p.start + r) & 1) * p.nv;
        double* nxt = p.tau + ((p.start + r + 1) & 1) * p.nv;
        const int64_t before = len;
        int done = 0;
        for (int64_t b = v0; b < v1; b += kPitchThreads) {
            const int64_t v = b + threadIdx.x;
            bool sel = false;
            double tv = 0, tn = 0;
            if (v < v1) {
                tv = tn = __ldcg(cur + v);
                if (tv < p.T) {
                    sel = true;
                    const int64_t q1 = p.ptr[v + 1];
                    double cm = INFINITY;
                    for (int64_t q = p.ptr[v]; q < q1; ++q) {
                        const int32_t w = p.dst[q];
                        const double tw = __ldcg(cur + w);
                        if (!((tv < tw) || (tv == tw && v < w))) { sel = false; break; }
                        const double x = __dadd_rn(tw, p.bnd[q]);
                        if (x < cm) cm = x;
                    }
                    if (sel) tn = fmin(p.T, cm);
                }
                __stcg(nxt + v, tn);
                if (sel && !(tn < p.T)) ++done;
            }
            const unsigned m = __ballot_sync(0xffffffffu, sel);
            if (lane == 0) warp_cnt[warp] = __popc(m);
            __syncthreads();
            int off = 0, tot = 0;
#pragma unroll
            for (int w = 0; w < kPitchThreads / 32; ++w) {
                if (w < warp) off += warp_cnt[w];
                tot += warp_cnt[w];
            }
            if (sel) {
                const int64_t at = (int64_t)blockIdx.x * p.cap + len + off + __popc(m & ((1u << lane) - 1));
                p.lv[at] = (int32_t)v;
                p.lb[at] = tv;
                p.lt[at] = tn;
            }
            len += tot;
            __syncthreads();
        }
        done = __reduce_add_sync(0xffffffffu, done);
        if (lane == 0 && done) atomicSub(&p.ctl->left, done);
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) {
            const int n = (int)(len - before);
            p.cnt[(int64_t)r * gridDim.x + blockIdx.x] = n;
            if (n) atomicAdd(&p.ctl->selected, n);
            if (len + p.vpb > p.cap) atomicExch(&p.ctl->full, 1);
            __threadfence();
            if (atomicAdd(&p.ctl->arrived, 1u) == (unsigned)(r + 1) * gridDim.x - 1) {
                // all blocks are here: their counts are visible, none runs on before the release
                __threadfence();
                const int left = *(volatile int*)&p.ctl->left, sel = *(volatile int*)&p.ctl->selected;
                if (left == 0) p.ctl->stop = 1;
                else if (sel == 0) p.ctl->stop = 2;
                else if (*(volatile int*)&p.ctl->full) p.ctl->stop = 4;
                p.ctl->selected = 0;
                p.ctl->rounds = r + 1;
                __threadfence();
                atomicExch(&p.ctl->released, (unsigned)(r + 1));
            }
            long long deadline = 0;
            for (int it = 0; pitch_acquire(&p.ctl->released) < (unsigned)(r + 1); ++it) {
                long long now;
                asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
                if (it == 0) deadline = now + 10000000000LL;   // 10 s
                else if (now > deadline) {
                    atomicExch(&p.ctl->stop, 3);
                    break;
                }
            }
            s_stop = *(volatile int*)&p.ctl->stop;
        }
        __syncthreads();
        if (s_stop) return;
    }
}

// exclusive offsets of the (round, block) lists in output order, and within each block's list
__global__ void __launch_bounds__(1024) pitch_offsets_kernel(const PitchCtl* ctl, int nblocks, const int* cnt, int64_t* out_off,
                                                             int64_t* list_off, int64_t* round_end) {
    __shared__ int64_t warp_sum[32];
    const int rounds = ctl->rounds, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t n = (int64_t)rounds * nblocks;
    int64_t carry = 0;
    for (int64_t b = 0; b < n; b += 1024) {
        const int64_t i = b + threadIdx.x;
        const int64_t x = i < n ? cnt[i] : 0;
        int64_t s = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        if (lane == 31) warp_sum[warp] = s;
        __syncthreads();
        int64_t off = carry, tot = 0;
        for (int w = 0; w < 32; ++w) {
            if (w < warp) off += warp_sum[w];
            tot += warp_sum[w];
        }
        if (i < n) {
            out_off[i] = off + s - x;
            if ((i + 1) % nblocks == 0) round_end[i / nblocks] = off + s;
        }
        carry += tot;
        __syncthreads();
    }
    for (int b = threadIdx.x; b < nblocks; b += 1024) {
        int64_t s = 0;
        for (int r = 0; r < rounds; ++r) {
            list_off[(int64_t)r * nblocks + b] = s;
            s += cnt[(int64_t)r * nblocks + b];
        }
    }
}

__global__ void __launch_bounds__(kPitchThreads) pitch_order_kernel(const PitchCtl* ctl, const int* cnt, const int64_t* out_off,
                                                                    const int64_t* list_off, int64_t cap, const int32_t* lv,
                                                                    const double* lb, const double* lt, int32_t* ov, double* ob,
                                                                    double* ot) {
    const int rounds = ctl->rounds, nb = gridDim.x, lane = threadIdx.x & 31;
    for (int r = threadIdx.x >> 5; r < rounds; r += kPitchThreads / 32) {
        const int64_t k = (int64_t)r * nb + blockIdx.x, from = blockIdx.x * cap + list_off[k], to = out_off[k];
        for (int i = lane; i < cnt[k]; i += 32) {
            ov[to + i] = lv[from + i];
            ob[to + i] = lb[from + i];
            ot[to + i] = lt[from + i];
        }
    }
}

#define PITCH_TRY(call)                                                                          \
    do {                                                                                         \
        cudaError_t _e = (call);                                                                 \
        if (_e != cudaSuccess)                                                                   \
            return set_error(_e == cudaErrorMemoryAllocation ? MTP_ENOMEM : MTP_ECUDA,           \
                             std::string(#call) + ": " + cudaGetErrorString(_e));                \
    } while (0)

namespace {

// device buffers of one pitching call, freed on every exit path
struct PitchBuffers {
    std::vector<void*> owned;
    ~PitchBuffers() {
        for (void* p : owned) cudaFree(p);
    }
    template <typename T>
    cudaError_t alloc(T** p, size_t n) {
        *p = nullptr;
        cudaError_t e = cudaMalloc((void**)p, (n ? n : 1) * sizeof(T));
        if (e == cudaSuccess) owned.push_back(*p);
        return e;
    }
};

}  // namespace

int device_pitch(const Mesh& m, const PitchGraph& g, double T, Tents& out, void* stream) {
    cudaStream_t st = (cudaStream_t)stream;
    const int64_t nv = m.nv;
    // blocks: one vertex per thread as long as all blocks are resident together
    int dev = 0, nsm = 0, per_sm = 0;
    PITCH_TRY(cudaGetDevice(&dev));
    PITCH_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    PITCH_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, pitch_rounds_kernel, kPitchThreads, 0));
    const int64_t resident = (int64_t)std::max(1, per_sm) * nsm;
    int64_t vpt = 1;
    while ((nv + vpt * kPitchThreads - 1) / (vpt * kPitchThreads) > resident) ++vpt;
    const int nblocks = (int)((nv + vpt * kPitchThreads - 1) / (vpt * kPitchThreads));
    PitchArgs p{};
    p.nv = nv;
    p.vpb = (int)(vpt * kPitchThreads);
    p.T = T;
    p.max_rounds = kPitchChunk;
    p.cap = (int64_t)p.vpb * kPitchList;
    PitchBuffers B;
    int64_t *d_ptr, *d_out_off, *d_list_off, *d_round_end;
    int32_t *d_dst, *o_v;
    double *d_bnd, *o_b, *o_t;
    const size_t list = (size_t)nblocks * p.cap, cells = (size_t)p.max_rounds * nblocks;
    PITCH_TRY(B.alloc(&p.ctl, 1));
    PITCH_TRY(B.alloc(&d_ptr, g.ptr.size()));
    PITCH_TRY(B.alloc(&d_dst, g.dst.size()));
    PITCH_TRY(B.alloc(&d_bnd, g.bnd.size()));
    PITCH_TRY(B.alloc(&p.tau, 2 * nv));
    PITCH_TRY(B.alloc(&p.lv, list));
    PITCH_TRY(B.alloc(&p.lb, list));
    PITCH_TRY(B.alloc(&p.lt, list));
    PITCH_TRY(B.alloc(&p.cnt, cells));
    PITCH_TRY(B.alloc(&d_out_off, cells));
    PITCH_TRY(B.alloc(&d_list_off, cells));
    PITCH_TRY(B.alloc(&d_round_end, p.max_rounds));
    PITCH_TRY(B.alloc(&o_v, list));
    PITCH_TRY(B.alloc(&o_b, list));
    PITCH_TRY(B.alloc(&o_t, list));
    p.ptr = d_ptr;
    p.dst = d_dst;
    p.bnd = d_bnd;
    PITCH_TRY(cudaMemcpyAsync(d_ptr, g.ptr.data(), g.ptr.size() * sizeof(int64_t), cudaMemcpyHostToDevice, st));
    if (!g.dst.empty()) {
        PITCH_TRY(cudaMemcpyAsync(d_dst, g.dst.data(), g.dst.size() * sizeof(int32_t), cudaMemcpyHostToDevice, st));
        PITCH_TRY(cudaMemcpyAsync(d_bnd, g.bnd.data(), g.bnd.size() * sizeof(double), cudaMemcpyHostToDevice, st));
    }
    PITCH_TRY(cudaMemsetAsync(p.tau, 0, 2 * nv * sizeof(double), st));
    out.layer_ptr.assign(1, 0);
    PitchCtl h{};
    h.left = (int)nv;
    std::vector<int64_t> ends(p.max_rounds);
    long long rounds = 0;
    while (true) {
        h.arrived = h.released = 0;
        h.rounds = h.full = h.stop = 0;
        PITCH_TRY(cudaMemcpyAsync(p.ctl, &h, sizeof(h), cudaMemcpyHostToDevice, st));
        void* args[] = {&p};
        PITCH_TRY(cudaLaunchCooperativeKernel((const void*)pitch_rounds_kernel, dim3(nblocks), dim3(kPitchThreads), args, 0, st));
        pitch_offsets_kernel<<<1, 1024, 0, st>>>(p.ctl, nblocks, p.cnt, d_out_off, d_list_off, d_round_end);
        pitch_order_kernel<<<nblocks, kPitchThreads, 0, st>>>(p.ctl, p.cnt, d_out_off, d_list_off, p.cap, p.lv, p.lb, p.lt, o_v,
                                                              o_b, o_t);
        PITCH_TRY(cudaGetLastError());
        PITCH_TRY(cudaMemcpyAsync(&h, p.ctl, sizeof(h), cudaMemcpyDeviceToHost, st));
        PITCH_TRY(cudaMemcpyAsync(ends.data(), d_round_end, p.max_rounds * sizeof(int64_t), cudaMemcpyDeviceToHost, st));
        PITCH_TRY(cudaStreamSynchronize(st));
        if (h.stop == 3) return set_error(MTP_ETIMEOUT, "device pitcher: a wait between rounds exceeded the limit");
        // a round that selected nothing adds no layer
        const int nr = h.stop == 2 ? h.rounds - 1 : h.rounds;
        const int64_t n0 = (int64_t)out.vertex.size(), n = nr > 0 ? ends[nr - 1] : 0;
        out.vertex.resize(n0 + n);
        out.layer.resize(n0 + n);
        out.t_bot.resize(n0 + n);
        out.t_top.resize(n0 + n);
        if (n) {
            PITCH_TRY(cudaMemcpyAsync(out.vertex.data() + n0, o_v, n * sizeof(int32_t), cudaMemcpyDeviceToHost, st));
            PITCH_TRY(cudaMemcpyAsync(out.t_bot.data() + n0, o_b, n * sizeof(double), cudaMemcpyDeviceToHost, st));
            PITCH_TRY(cudaMemcpyAsync(out.t_top.data() + n0, o_t, n * sizeof(double), cudaMemcpyDeviceToHost, st));
        }
        for (int r = 0; r < nr; ++r) {
            const int64_t from = r ? ends[r - 1] : 0;
            std::fill(out.layer.begin() + n0 + from, out.layer.begin() + n0 + ends[r], (int32_t)(rounds + r));
            out.layer_ptr.push_back(n0 + ends[r]);
        }
        PITCH_TRY(cudaStreamSynchronize(st));
        rounds += nr;
        p.start = (p.start + h.rounds) & 1;
        if (h.stop == 1) break;
        if (h.stop == 2) return set_error(MTP_ECAUSAL, "pitching stalled before reaching T");
        if (rounds > kPitchMaxRounds)
            return set_error(MTP_ECAUSAL, "device pitcher: no end after " + std::to_string(kPitchMaxRounds) +
                                              " rounds (edge bounds below the resolution of tau?)");
    }
    return MTP_OK;
}

}  // namespace mtp

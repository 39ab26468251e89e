// Continuous batching of inference presentations on a frozen network.
//
// A server keeps S slots of per-sample state resident on the device, S chosen
// so the slots' state fits a byte cap.  Requests (one image's rates, a seed
// and a presentation length) wait in a queue; each snn_serve_step call admits
// queued requests into free slots -- resetting only those slots, as an
// episodic run would (Sec. "Episodic vs. continuing simulation") -- runs up
// to k time steps for every active slot, and retires the slots whose
// presentation ended, so the next call backfills them while the others keep
// running.  The batch size therefore changes per slot rather than per run
// (Sec. "Dynamic minibatch size").
//
// Every slot counts its own steps, and the Poisson draw of a slot at its step t
// is the same function of (seed, t, input) as in snn_run; with learning off the
// samples do not interact, and the arithmetic is snn_run's: each request's spike
// counts equal those of running it alone.
//
// The work of a call scales with the live slots, not with the capacity: one
// launch of k_serve_chunk runs up to k steps with one CTA per live slot, and
// the all-but-self inhibition of a slot is a count inside its CTA.  Calls do not
// wait for the device: the host knows each slot's remaining steps, so it retires
// and backfills without reading anything back, and snn_serve_poll hands out the
// requests whose call has finished (an event).
//
// A call is one launch (two when it admits): the kernels read the call's
// admissions and slot list in pinned host memory, and a slot that ends in the
// call writes its counts to a pinned result row itself.  With 512 requests of 50
// to 500 steps, 400 neurons, k = 10, a call took 56 us of host time (copies of
// its lists, a gather launch, a copy per finished row, scans over all slots) and
// its kernel 43 us; now 29 us on average, the one that admits all 512 included,
// and the burst 3.9 ms instead of 5.7.  The pinned per-call buffers rotate, each
// reused only after the call that last used it has finished on the device, which
// also bounds how far the host runs ahead.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <deque>
#include <functional>
#include <string>
#include <vector>

#include "snn_nvtx.cuh"
#include "snn_sample.cuh"

namespace snn {
const snn_spec& net_spec(const snn_net* n);
Bufs net_bufs(const snn_net* n);
int net_device(const snn_net* n);
Consts net_consts(const snn_net* n, int B, float dt);
void net_set_error(snn_net* n, const char* msg);
void set_thread_error(const char* msg);
}  // namespace snn

namespace {

constexpr unsigned FULL = 0xFFFFFFFFu;
constexpr int SC_THREADS = 256;         // threads of a slot's CTA
constexpr int STAGES = 3;               // host staging buffers (calls in flight)

struct SlotBufs {
    const float* W;        // [n_in][N] the network's weights (read only)
    const double* theta;   // [N]
    float* wscale;         // [N] FP8 column scales of the frozen W
    uint32_t* thr;         // [S][n_in]
    uint64_t* seeds;       // [S]
    float* v_e;            // [S][N]
    float* v_i;            // [S][N]
    uint32_t* st;          // [S][N]
    uint32_t* counts;      // [S][N]
    uint32_t* cnt;         // [S] inhibitory spikes of the slot's previous step
    int* t_loc;            // [S] steps taken by the slot's request
    int* t_len;            // [S] its presentation length
    uint32_t* ring;        // [R][N] result rows (pinned host memory)
};

// One call's lists, in pinned host memory that the kernels read.
struct Admission { int slot, len; uint64_t seed; };
struct Live { int slot, row; };         // a slot that steps; its result row if it ends in the call, else -1

// Admitted slot a: thresholds from its rates, state reset, counters.
__global__ void k_serve_admit(snn::Consts c, SlotBufs d, const Admission* adm, const float* rates) {
    const int a = blockIdx.x;
    const Admission ad = adm[a];
    const int s = ad.slot;
    for (int i = threadIdx.x; i < c.n_in; i += blockDim.x)
        d.thr[(size_t)s * c.n_in + i] = snn::poisson_threshold(rates[(size_t)a * c.n_in + i], c.dt);
    for (int j = threadIdx.x; j < c.N; j += blockDim.x) {
        const size_t k = (size_t)s * c.N + j;
        d.v_e[k] = c.e_rest;
        d.v_i[k] = c.i_rest;
        d.st[k] = 0u;
        d.counts[k] = 0u;
    }
    if (threadIdx.x == 0) {
        d.cnt[s] = 0u;
        d.seeds[s] = ad.seed;
        d.t_loc[s] = 0;
        d.t_len[s] = ad.len;
    }
}

// One CTA per live slot runs up to k of its steps (snn_sample.cuh), the state
// in registers between them.
template <int NPT>
__global__ void __launch_bounds__(1024, 1) k_serve_chunk(const __grid_constant__ snn::Consts c,
                                                         const __grid_constant__ SlotBufs d,
                                                         const Live* __restrict__ live, int k) {
    extern __shared__ __align__(16) unsigned char ssm[];
    const Live lv = live[blockIdx.x];
    const int s = lv.slot;
    const int t0 = d.t_loc[s];
    const int steps = min(k, d.t_len[s] - t0);
    if (steps <= 0) return;                             // (uniform over the CTA)
    const size_t sn = (size_t)s * c.N;
    snn::SampleIO io{};
    io.W = d.W;
    io.theta = d.theta;
    io.wscale = d.wscale;
    io.thr = d.thr + (size_t)s * c.n_in;
    io.seed = d.seeds[s];
    io.v_e = d.v_e + sn;
    io.v_i = d.v_i + sn;
    io.st = d.st + sn;
    io.counts = d.counts + sn;
    const int C = snn::run_sample<NPT, false>(c, io, (unsigned long long)t0, steps, (int)d.cnt[s], ssm);
    if (lv.row >= 0)                                    // (each thread's own counts)
        for (int j = threadIdx.x; j < c.N; j += blockDim.x) d.ring[(size_t)lv.row * c.N + j] = io.counts[j];
    if (threadIdx.x == 0) {
        d.t_loc[s] = t0 + steps;
        d.cnt[s] = (uint32_t)C;
    }
}

// Layers too wide for a thread's registers: the same step with the state in
// global memory, a loop over the neurons.
__global__ void __launch_bounds__(SC_THREADS) k_serve_chunk_wide(snn::Consts c, SlotBufs d,
                                                                 const Live* __restrict__ live, int k) {
    extern __shared__ uint32_t sh[];
    uint32_t* words = sh;                               // [Iw] input spike words of the step
    uint16_t* act = (uint16_t*)(sh + c.Iw);             // [n_in] active inputs, ascending
    __shared__ int s_nact;
    __shared__ uint32_t s_cnt[2];
    const Live lv = live[blockIdx.x];
    const int s = lv.slot;
    const int t0 = d.t_loc[s];
    const int steps = min(k, d.t_len[s] - t0);
    if (steps <= 0) return;                             // (uniform over the CTA)
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarp = blockDim.x >> 5;
    const uint64_t seed = d.seeds[s];
    const uint32_t* thr = d.thr + (size_t)s * c.n_in;
    int C = (int)d.cnt[s];
    for (int t = 0; t < steps; ++t) {
        const unsigned long long tt = (unsigned long long)(t0 + t);
        for (int iw = warp; iw < c.Iw; iw += nwarp) {
            const int i = iw * 32 + lane;
            const bool sp = i < c.n_in && snn::poisson_spike(seed, tt, c.n_in, i, thr[i]);
            const uint32_t w = __ballot_sync(FULL, sp);
            if (lane == 0) words[iw] = w;
        }
        if (threadIdx.x == 0) s_cnt[t & 1] = 0u;
        __syncthreads();
        if (warp == 0) {                                // the list, by a scan over the words
            uint32_t running = 0;
            for (int w0 = 0; w0 < c.Iw; w0 += 32) {
                const int w = w0 + lane;
                uint32_t word = w < c.Iw ? words[w] : 0u;
                const uint32_t n = __popc(word);
                uint32_t incl = n;
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(FULL, incl, o);
                    if (lane >= o) incl += y;
                }
                uint32_t off = running + incl - n;
                while (word) {
                    act[off++] = (uint16_t)(w * 32 + __ffs(word) - 1);
                    word &= word - 1;
                }
                running += __shfl_sync(FULL, incl, 31);
            }
            if (lane == 0) s_nact = (int)running;
        }
        __syncthreads();
        const int na = s_nact;
        for (int j0 = 0; j0 < c.N; j0 += blockDim.x) {
            const int j = j0 + threadIdx.x;
            bool si = false;
            if (j < c.N) {
                const float* Wj = d.W + j;
                const float sc = c.wprec == SNN_W_FP8E4M3 ? d.wscale[j] : 1.0f;
                const float inv = __frcp_rn(sc);
                float I = 0.0f;
                for (int a = 0; a < na; ++a) {
                    const float wv = Wj[(size_t)act[a] * c.N];
                    const float r = c.wprec == SNN_W_FP32 ? wv
                                  : c.wprec == SNN_W_BF16 ? snn::w_read_bf16(wv)
                                                          : snn::w_read_e4m3(wv, inv);
                    I = __fadd_rn(I, r);
                }
                if (c.wprec == SNN_W_FP8E4M3) I = __fmul_rn(I, sc);
                const size_t idx = (size_t)s * c.N + j;
                float v = d.v_e[idx], vi = d.v_i[idx];
                const uint32_t st = snn::pair_update(c, v, vi, d.st[idx], I, C,
                                                     __fadd_rn(c.e_thresh, __double2float_rn(d.theta[j])));
                d.v_e[idx] = v;
                d.v_i[idx] = vi;
                d.st[idx] = st;
                if (st & snn::ST_SE) d.counts[idx] += 1u;
                si = (st & snn::ST_SI) != 0u;
            }
            const uint32_t wi = __ballot_sync(FULL, si);
            if (lane == 0 && wi) atomicAdd(&s_cnt[t & 1], (uint32_t)__popc(wi));
        }
        __syncthreads();
        C = (int)s_cnt[t & 1];
    }
    if (lv.row >= 0)                                    // (each thread's own counts)
        for (int j = threadIdx.x; j < c.N; j += blockDim.x) d.ring[(size_t)lv.row * c.N + j] = d.counts[(size_t)s * c.N + j];
    if (threadIdx.x == 0) {
        d.t_loc[s] = t0 + steps;
        d.cnt[s] = (uint32_t)C;
    }
}

__global__ void k_serve_scales(snn::Consts c, SlotBufs d) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= c.N) return;
    float m = 0.0f;
    for (int i = 0; i < c.n_in; ++i) m = fmaxf(m, fabsf(d.W[(size_t)i * c.N + j]));
    d.wscale[j] = snn::e4m3_scale_of(m);
}

struct Request {
    uint64_t id;
    uint64_t seed;
    int T;
    std::vector<float> rates;
};

struct Slot {
    uint64_t id = 0;
    int remaining = 0;   // steps left; 0 = free
};

struct Result {
    uint64_t id;
    std::vector<uint32_t> counts;
};

// Finished requests whose counts are being copied to pinned rows.
struct Pending {
    cudaEvent_t ev = nullptr;
    std::vector<uint64_t> ids;
    std::vector<int> rows;
};

// One call's pinned buffers.
struct Stage {
    float* rates = nullptr;       // [S][n_in] admitted rates
    Admission* adm = nullptr;     // [S]
    Live* live = nullptr;         // [S]
    cudaEvent_t done = nullptr;   // the call that last used this stage has finished
    bool used = false;
};

size_t slot_bytes_of(const snn_spec& sp) {
    const size_t NI = sp.n_in, N = sp.n_exc;
    // thresholds, seed, voltages, packed refractory/spike word, counts, the
    // inhibitory count and step counters on the device; two result rows and one
    // slot's share of each call's lists (rates, slots) in every stage, pinned
    return NI * 4 + 8 + N * 16 + 12 + 2 * N * 4 + STAGES * (NI * 4 + 4 * 7);
}

}  // namespace

struct snn_server {
    snn_net* net = nullptr;
    int device = 0;
    int S = 0, R = 0;
    float dt = 1.0f;
    snn::Consts c{};
    SlotBufs d{};
    std::vector<void*> allocs;
    std::vector<void*> host_allocs;
    Stage stage[STAGES];
    int next_stage = 0;
    std::vector<int> free_rows;
    std::vector<int> free_slots;   // a heap, the lowest first
    std::vector<int> active;       // slots with steps left, ascending
    std::vector<cudaEvent_t> free_events;
    std::deque<Request> queue;
    std::vector<Slot> slots;
    std::deque<Pending> pending;
    std::deque<Result> done;
    uint64_t next_id = 1;
    cudaStream_t last = nullptr;
    std::string err;
};

namespace {

snn_status sfail(snn_server* s, snn_status code, const std::string& msg) {
    if (s) s->err = msg;
    snn::set_thread_error(msg.c_str());
    return code;
}

#define SERVE_CUDA(srv, expr)                                                              \
    do {                                                                                   \
        cudaError_t e_ = (expr);                                                           \
        if (e_ != cudaSuccess)                                                             \
            return sfail(srv, e_ == cudaErrorMemoryAllocation ? SNN_ERR_OOM : SNN_ERR_CUDA, \
                         std::string(#expr) + ": " + cudaGetErrorString(e_));              \
    } while (0)

template <typename T>
cudaError_t salloc(snn_server* s, T** p, size_t count) {
    cudaError_t e = cudaMalloc((void**)p, count * sizeof(T) + 16);
    if (e == cudaSuccess) s->allocs.push_back(*p);
    return e;
}

template <typename T>
cudaError_t halloc(snn_server* s, T** p, size_t count) {
    cudaError_t e = cudaMallocHost((void**)p, count * sizeof(T) + 16);
    if (e == cudaSuccess) s->host_allocs.push_back(*p);
    return e;
}

// Moves every pending batch whose copy has landed (wait: the oldest batch even
// if it has not) into the finished queue and frees its rows.
cudaError_t collect(snn_server* s, bool wait_oldest) {
    const int N = s->c.N;
    while (!s->pending.empty()) {
        Pending& p = s->pending.front();
        cudaError_t e = wait_oldest ? cudaEventSynchronize(p.ev) : cudaEventQuery(p.ev);
        if (e == cudaErrorNotReady) return cudaSuccess;
        if (e != cudaSuccess) return e;
        wait_oldest = false;
        for (size_t f = 0; f < p.ids.size(); ++f) {
            Result r;
            r.id = p.ids[f];
            const uint32_t* row = s->d.ring + (size_t)p.rows[f] * N;
            r.counts.assign(row, row + N);
            s->done.push_back(std::move(r));
            s->free_rows.push_back(p.rows[f]);
        }
        s->free_events.push_back(p.ev);
        s->pending.pop_front();
    }
    return cudaSuccess;
}

}  // namespace

extern "C" {

size_t snn_serve_slot_bytes(const snn_net* net) {
    return net ? slot_bytes_of(snn::net_spec(net)) : 0;
}

snn_status snn_serve_destroy(snn_server* s) {
    if (!s) return SNN_OK;
    cudaSetDevice(s->device);
    cudaDeviceSynchronize();
    for (Pending& p : s->pending) if (p.ev) cudaEventDestroy(p.ev);
    for (cudaEvent_t e : s->free_events) cudaEventDestroy(e);
    for (Stage& st : s->stage) if (st.done) cudaEventDestroy(st.done);
    for (void* p : s->allocs) cudaFree(p);
    for (void* p : s->host_allocs) cudaFreeHost(p);
    delete s;
    return SNN_OK;
}

snn_status snn_serve_create(snn_net* net, int max_slots, size_t state_cap_bytes, float dt_ms,
                            snn_server** out) {
    if (!out) return sfail(nullptr, SNN_ERR_ARG, "snn_serve_create: out is NULL");
    *out = nullptr;
    if (!net) return sfail(nullptr, SNN_ERR_ARG, "snn_serve_create: net is NULL");
    if (max_slots <= 0 || !std::isfinite(dt_ms) || !(dt_ms > 0.0f))
        return sfail(nullptr, SNN_ERR_ARG, "snn_serve_create: max_slots and dt_ms must be > 0");
    const snn_spec& sp = snn::net_spec(net);
    const size_t per = slot_bytes_of(sp);
    const size_t fit = state_cap_bytes / per;
    if (fit == 0)
        return sfail(nullptr, SNN_ERR_CAPACITY,
                     "snn_serve_create: the state cap holds no slot (one slot needs " +
                         std::to_string(per) + " bytes)");
    const int S = (int)(fit < (size_t)max_slots ? fit : (size_t)max_slots);
    snn_server* s = new (std::nothrow) snn_server();
    if (!s) return sfail(nullptr, SNN_ERR_OOM, "snn_serve_create: host allocation failed");
    s->net = net;
    s->device = snn::net_device(net);
    s->S = S;
    s->R = 2 * S;
    s->dt = dt_ms;
    s->c = snn::net_consts(net, S, dt_ms);
    s->slots.resize(S);
    const snn::Bufs nb = snn::net_bufs(net);
    const size_t NI = sp.n_in, N = sp.n_exc;
    SlotBufs& d = s->d;
    d.W = nb.W;
    d.theta = nb.theta;
    cudaError_t e = cudaSetDevice(s->device);
    if (e == cudaSuccess) e = salloc(s, &d.wscale, N);
    if (e == cudaSuccess) e = salloc(s, &d.thr, (size_t)S * NI);
    if (e == cudaSuccess) e = salloc(s, &d.seeds, (size_t)S);
    if (e == cudaSuccess) e = salloc(s, &d.v_e, (size_t)S * N);
    if (e == cudaSuccess) e = salloc(s, &d.v_i, (size_t)S * N);
    if (e == cudaSuccess) e = salloc(s, &d.st, (size_t)S * N);
    if (e == cudaSuccess) e = salloc(s, &d.counts, (size_t)S * N);
    if (e == cudaSuccess) e = salloc(s, &d.cnt, (size_t)S);
    if (e == cudaSuccess) e = salloc(s, &d.t_loc, (size_t)S);
    if (e == cudaSuccess) e = salloc(s, &d.t_len, (size_t)S);
    if (e == cudaSuccess) e = halloc(s, &d.ring, (size_t)s->R * N);
    for (int k = 0; k < STAGES && e == cudaSuccess; ++k) {
        Stage& st = s->stage[k];
        e = halloc(s, &st.rates, (size_t)S * NI);
        if (e == cudaSuccess) e = halloc(s, &st.adm, (size_t)S);
        if (e == cudaSuccess) e = halloc(s, &st.live, (size_t)S);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&st.done, cudaEventDisableTiming);
    }
    for (int r = s->R - 1; r >= 0; --r) s->free_rows.push_back(r);
    for (int k = 0; k < S; ++k) s->free_slots.push_back(k);   // ascending: a heap, the lowest first
    if (e == cudaSuccess) e = cudaMemset(d.t_len, 0, (size_t)S * 4);
    if (e == cudaSuccess) e = cudaMemset(d.t_loc, 0, (size_t)S * 4);
    if (e == cudaSuccess && sp.wprec == SNN_W_FP8E4M3) {   // the frozen W's column scales
        cudaStream_t cs = nullptr;
        e = cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking);
        if (e == cudaSuccess) {
            k_serve_scales<<<((int)N + 255) / 256, 256, 0, cs>>>(s->c, d);
            e = cudaGetLastError();
            if (e == cudaSuccess) e = cudaStreamSynchronize(cs);
            cudaStreamDestroy(cs);
        }
    }
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e != cudaSuccess) {
        const snn_status code = e == cudaErrorMemoryAllocation ? SNN_ERR_OOM : SNN_ERR_CUDA;
        sfail(nullptr, code, std::string("snn_serve_create: ") + cudaGetErrorString(e));
        snn_serve_destroy(s);
        return code;
    }
    *out = s;
    return SNN_OK;
}

snn_status snn_serve_submit(snn_server* s, const float* rates_hz, uint64_t seed, int T,
                            uint64_t* id) {
    if (!s || !rates_hz || !id || T <= 0)
        return sfail(s, SNN_ERR_ARG, "snn_serve_submit: NULL argument or T <= 0");
    Request r;
    r.id = s->next_id++;
    r.seed = seed;
    r.T = T;
    r.rates.assign(rates_hz, rates_hz + s->c.n_in);
    s->queue.push_back(std::move(r));
    *id = s->queue.back().id;
    return SNN_OK;
}

snn_status snn_serve_step(snn_server* s, int k, void* stream_, int* steps_run) {
    const snn::NvtxRange range("snn_serve_step");
    if (!s || k <= 0) return sfail(s, SNN_ERR_ARG, "snn_serve_step: NULL server or k <= 0");
    if (steps_run) *steps_run = 0;
    cudaStream_t st = (cudaStream_t)stream_;
    SERVE_CUDA(s, cudaSetDevice(s->device));
    const int NI = s->c.n_in, N = s->c.N;
    // this call's buffers: free once the call that used them last has finished
    Stage& sg = s->stage[s->next_stage];
    s->next_stage = (s->next_stage + 1) % STAGES;
    if (sg.used) SERVE_CUDA(s, cudaEventSynchronize(sg.done));
    SERVE_CUDA(s, collect(s, false));
    // ---- admit queued requests into free slots, the lowest first
    int na = 0;
    const size_t before = s->active.size();
    while (!s->free_slots.empty() && !s->queue.empty()) {
        std::pop_heap(s->free_slots.begin(), s->free_slots.end(), std::greater<int>());
        const int slot = s->free_slots.back();
        s->free_slots.pop_back();
        Request& r = s->queue.front();
        std::memcpy(sg.rates + (size_t)na * NI, r.rates.data(), (size_t)NI * 4);
        sg.adm[na] = Admission{slot, r.T, r.seed};
        s->slots[slot].id = r.id;
        s->slots[slot].remaining = r.T;
        s->active.push_back(slot);
        s->queue.pop_front();
        ++na;
    }
    std::inplace_merge(s->active.begin(), s->active.begin() + before, s->active.end());
    if (na > 0) {
        k_serve_admit<<<na, 256, 0, st>>>(s->c, s->d, sg.adm, sg.rates);
        SERVE_CUDA(s, cudaGetLastError());
    }
    // ---- up to k steps of every live slot, one CTA per slot; those that end
    // within them are retired, each with a result row
    int longest = 0, nf = 0;
    for (int slot : s->active) longest = s->slots[slot].remaining > longest ? s->slots[slot].remaining : longest;
    const int kk = k < longest ? k : longest;
    for (int slot : s->active) nf += s->slots[slot].remaining <= kk;
    while ((int)s->free_rows.size() < nf) {               // the ring is full: wait for the oldest batch
        if (s->pending.empty()) return sfail(s, SNN_ERR_CUDA, "snn_serve_step: result ring exhausted");
        SERVE_CUDA(s, collect(s, true));
    }
    Pending p;
    int nl = 0, left = 0;
    for (int slot : s->active) {
        Slot& sl = s->slots[slot];
        sl.remaining -= kk;
        Live& lv = sg.live[nl++];
        lv = Live{slot, -1};
        if (sl.remaining > 0) {
            s->active[left++] = slot;
            continue;
        }
        sl.remaining = 0;
        lv.row = s->free_rows.back();
        s->free_rows.pop_back();
        p.ids.push_back(sl.id);
        p.rows.push_back(lv.row);
        s->free_slots.push_back(slot);
        std::push_heap(s->free_slots.begin(), s->free_slots.end(), std::greater<int>());
    }
    s->active.resize(left);
    if (nl > 0) {
        const int npt = NI <= 65535 ? snn::sample_npt(N) : 0;
        const size_t need = snn::sample_smem(NI, s->c.Iw, false, false).bytes;
        if (npt == 0 || need > snn::SAMPLE_SMEM_DEFAULT) {
            const size_t smem = (size_t)s->c.Iw * 4 + (size_t)NI * 2 + 16;
            k_serve_chunk_wide<<<nl, SC_THREADS, smem, st>>>(s->c, s->d, sg.live, kk);
        } else {
            auto kern = npt == 1 ? k_serve_chunk<1> : npt == 2 ? k_serve_chunk<2>
                      : npt == 4 ? k_serve_chunk<4> : k_serve_chunk<8>;
            kern<<<nl, snn::sample_threads(N, npt), need, st>>>(s->c, s->d, sg.live, kk);
        }
        SERVE_CUDA(s, cudaGetLastError());
    }
    if (steps_run) *steps_run = kk;
    if (nf > 0) {
        if (s->free_events.empty()) {
            SERVE_CUDA(s, cudaEventCreateWithFlags(&p.ev, cudaEventDisableTiming));
        } else {
            p.ev = s->free_events.back();
            s->free_events.pop_back();
        }
        SERVE_CUDA(s, cudaEventRecord(p.ev, st));
        s->pending.push_back(std::move(p));
    }
    SERVE_CUDA(s, cudaEventRecord(sg.done, st));
    sg.used = true;
    s->last = st;
    return SNN_OK;
}

snn_status snn_serve_poll(snn_server* s, uint64_t* ids, uint32_t* counts, int max, int* n_out) {
    if (!s || !n_out || max < 0 || (max > 0 && (!ids || !counts)))
        return sfail(s, SNN_ERR_ARG, "snn_serve_poll: NULL argument");
    SERVE_CUDA(s, collect(s, false));
    int n = 0;
    const int N = s->c.N;
    while (n < max && !s->done.empty()) {
        Result& r = s->done.front();
        ids[n] = r.id;
        std::memcpy(counts + (size_t)n * N, r.counts.data(), (size_t)N * 4);
        s->done.pop_front();
        ++n;
    }
    *n_out = n;
    return SNN_OK;
}

snn_status snn_serve_wait(snn_server* s) {
    if (!s) return sfail(nullptr, SNN_ERR_ARG, "snn_serve_wait: NULL server");
    SERVE_CUDA(s, cudaSetDevice(s->device));
    while (!s->pending.empty()) SERVE_CUDA(s, collect(s, true));
    if (s->last) SERVE_CUDA(s, cudaStreamSynchronize(s->last));
    return SNN_OK;
}

snn_status snn_serve_status(const snn_server* s, int* slots, int* active, int* queued, int* done) {
    if (!s) return SNN_ERR_ARG;
    const int a = (int)s->active.size();
    size_t in_flight = 0;
    for (const Pending& p : s->pending) in_flight += p.ids.size();
    if (slots) *slots = s->S;
    if (active) *active = a;
    if (queued) *queued = (int)s->queue.size();
    if (done) *done = (int)(s->done.size() + in_flight);
    return SNN_OK;
}

}  // extern "C"

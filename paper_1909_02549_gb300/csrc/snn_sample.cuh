// Frozen presentations, one sample per CTA: with learning off the samples of a
// batch do not interact, so a CTA runs its sample for many steps with the
// neurons' state in registers and no exchange with other CTAs.  Used by the
// learning-off runs of the persistent mode and by the serving loop.
//
// Inputs whose rate is zero never spike and are left out once, at the start:
// the draws and lists below run over the live inputs, ascending.  Per step:
//   X  the first rows of the step's active-input list are loaded; while they
//      are in flight the next step's inputs are drawn; then the ordered sums, the
//      neuron updates and the count of inhibitory spikes;
//   Y  the next step's list, each warp placing its own words' inputs after a
//      masked sum of the words' counts.
// Two block barriers a step.  What bounds it: the chain of the weight rows' L2
// round trip, the neuron update and the two barriers.
#pragma once

#include "snn_internal.cuh"

namespace snn {

// One sample's buffers.
struct SampleIO {
    const float* W;            // [n_in][N]
    const double* theta;       // [N]
    const float* wscale;       // [N] FP8 column scales (read for FP8 weights only)
    const uint32_t* thr;       // [n_in]
    uint64_t seed;
    float *v_e, *v_i, *x_post; // [N] state, updated in place (x_post with TRACE only)
    uint32_t* st;              // [N]
    uint32_t* counts;          // [N], added to
    const float* x_in;         // [n_in] presynaptic traces before the steps (TRACE only)
    float* x_out;              // [n_in] after them
    uint32_t *raster_e, *raster_i, *raster_in;   // the sample's row of step 0 (recorded runs)
    size_t rs_n, rs_i;         // words between steps of the rasters
};

// Dynamic shared memory that a kernel of run_sample may use without an opt-in: the
// default 48 KB less the static arrays of run_sample (144 bytes), which count too.
constexpr size_t SAMPLE_SMEM_DEFAULT = 48 * 1024 - 256;

struct SampleSmem {
    size_t o_idx, o_act, o_words, o_x, o_rec, bytes;   // after the live inputs' thresholds
};

__host__ __device__ inline SampleSmem sample_smem(int n_in, int Iw, bool trace, bool rec) {
    SampleSmem m{};
    size_t o = (size_t)n_in * 4;
    m.o_words = o; o += (size_t)Iw * 4;
    m.o_x = o;     o += trace ? (size_t)n_in * 4 : 0;
    m.o_rec = o;   o += rec ? (size_t)Iw * 4 : 0;
    o = (o + 15) & ~(size_t)15;
    m.o_act = o;   o += ((size_t)n_in + 16) * 2;
    o = (o + 15) & ~(size_t)15;
    m.o_idx = o;   o += (size_t)n_in * 2;
    m.bytes = (o + 15) & ~(size_t)15;
    return m;
}

// Neurons per thread for a layer of N (0: too wide), and the block's threads.
inline int sample_npt(int N) { return N <= 512 ? 1 : N <= 2048 ? 2 : N <= 4096 ? 4 : N <= 8192 ? 8 : 0; }
inline int sample_threads(int N, int npt) {
    const int t = ((N + npt - 1) / npt + 31) / 32 * 32;
    return t < 256 ? 256 : t;            // (warps without neurons still draw)
}

// `steps` steps from the sample's absolute step t0; C: the previous step's
// inhibitory count, and the returned one the last step's.
template <int NPT, bool TRACE>
__device__ __forceinline__ int run_sample(const Consts& c, const SampleIO& io, unsigned long long t0, int steps,
                                          int C, unsigned char* sm) {
    constexpr unsigned FULL = 0xFFFFFFFFu;
    constexpr int U = NPT <= 1 ? 8 : NPT <= 2 ? 4 : 2;     // list rows whose loads are issued together
    const int tid = threadIdx.x, nth = blockDim.x, warp = tid >> 5, lane = tid & 31, nwarp = nth >> 5;
    const int N = c.N, NI = c.n_in;
    const SampleSmem L = sample_smem(NI, c.Iw, TRACE, c.rec_input != 0);
    uint32_t* const cthr = reinterpret_cast<uint32_t*>(sm);                 // live inputs: thresholds
    uint32_t* const words = reinterpret_cast<uint32_t*>(sm + L.o_words);    // spikes of the drawn step
    float* const xs = reinterpret_cast<float*>(sm + L.o_x);                 // traces of the live inputs
    uint32_t* const rec = reinterpret_cast<uint32_t*>(sm + L.o_rec);        // input word of the raster
    uint16_t* const act = reinterpret_cast<uint16_t*>(sm + L.o_act);        // active inputs, ascending
    uint16_t* const cidx = reinterpret_cast<uint16_t*>(sm + L.o_idx);       // live inputs, ascending
    __shared__ int s_wn[32];
    __shared__ uint32_t s_cnt[2];

    // ---- the live inputs
    int nl = 0;
    for (int i0 = 0; i0 < NI; i0 += nth) {
        const int i = i0 + tid;
        const uint32_t thr = i < NI ? io.thr[i] : 0u;
        const uint32_t m = __ballot_sync(FULL, thr != 0u);
        if (lane == 0) s_wn[warp] = __popc(m);
        __syncthreads();
        const int wn = lane < nwarp ? s_wn[lane] : 0;
        const int at = nl + __reduce_add_sync(FULL, lane < warp ? wn : 0) + __popc(m & ((1u << lane) - 1u));
        if (thr != 0u) {
            cthr[at] = thr;
            cidx[at] = (uint16_t)i;
            if (TRACE) xs[at] = io.x_in[i];
        }
        nl += __reduce_add_sync(FULL, wn);
        __syncthreads();
    }
    for (int k = tid; k < NI + 16; k += nth) act[k] = 0;   // (entries past a list are rows in range)
    if (tid < 2) s_cnt[tid] = 0u;
    const int nw = (nl + 31) / 32;

    // ---- neurons j = tid + k * nth
    float v[NPT], vi[NPT], x[NPT], th[NPT], inv[NPT];      // inv: FP8, the inverse column scale
    uint32_t st[NPT], cnt[NPT];
#pragma unroll
    for (int k = 0; k < NPT; ++k) {
        const int j = tid + k * nth;
        const bool ok = j < N;
        v[k] = ok ? io.v_e[j] : 0.0f;
        vi[k] = ok ? io.v_i[j] : 0.0f;
        x[k] = ok && TRACE ? io.x_post[j] : 0.0f;
        st[k] = ok ? io.st[j] : 0u;
        th[k] = ok ? __fadd_rn(c.e_thresh, __double2float_rn(io.theta[j])) : 0.0f;
        cnt[k] = 0u;
        inv[k] = c.wprec == SNN_W_FP8E4M3 && ok ? __frcp_rn(io.wscale[j]) : 1.0f;   // exact: a power of two
    }

    auto draw = [&](unsigned long long tt) {
        for (int w = warp; w < nw; w += nwarp) {
            const int k = w * 32 + lane;
            bool s = false;
            if (k < nl) {
                s = (uint32_t)(splitmix64(io.seed ^ splitmix64(tt * (uint64_t)NI + (uint64_t)cidx[k])) >> 32) < cthr[k];
                if (TRACE) xs[k] = __fadd_rn(__fmul_rn(xs[k], c.a_x), s ? 1.0f : 0.0f);
            }
            const uint32_t m = __ballot_sync(FULL, s);
            if (lane == 0) words[w] = m;
        }
    };
    // the list from the words; returns its length
    auto list = [&]() {
        int n = 0;
        for (int w0 = 0; w0 < nw; w0 += 32) {
            const uint32_t word = w0 + lane < nw ? words[w0 + lane] : 0u;
            const int pc = __popc(word);
            for (int w = warp; w < 32 && w0 + w < nw; w += nwarp) {
                const uint32_t m = __shfl_sync(FULL, word, w);
                const int at = n + __reduce_add_sync(FULL, lane < w ? pc : 0) + __popc(m & ((1u << lane) - 1u));
                if ((m >> lane) & 1u) act[at] = cidx[(w0 + w) * 32 + lane];
            }
            n += __reduce_add_sync(FULL, pc);
        }
        return n;
    };
    auto wread = [&](float w, float inv) {
        return c.wprec == SNN_W_FP32 ? w : c.wprec == SNN_W_BF16 ? w_read_bf16(w) : w_read_e4m3(w, inv);
    };

    __syncthreads();
    draw(t0);
    __syncthreads();
    int n = list();
    __syncthreads();
    for (int t = 0; t < steps; ++t) {
        // ---- X: currents, the next step's draws inside the first loads' flight
        float I[NPT], w[U][NPT];
#pragma unroll
        for (int k = 0; k < NPT; ++k) I[k] = 0.0f;
        auto load = [&](int a) {
#pragma unroll
            for (int q = 0; q < U; ++q) {
                const float* row = io.W + (size_t)act[a + q] * N + tid;
#pragma unroll
                for (int k = 0; k < NPT; ++k) w[q][k] = row[tid + k * nth < N ? k * nth : -tid];
            }
        };
        auto add = [&](int a) {
#pragma unroll
            for (int q = 0; q < U; ++q)
                if (a + q < n) {
#pragma unroll
                    for (int k = 0; k < NPT; ++k) I[k] = __fadd_rn(I[k], wread(w[q][k], inv[k]));
                }
        };
        load(0);
        if (c.rec_input) {
            for (int k = tid; k < c.Iw; k += nth) rec[k] = 0u;
            __syncthreads();
            for (int a = tid; a < n; a += nth) atomicOr(&rec[act[a] >> 5], 1u << (act[a] & 31));
            __syncthreads();
            for (int k = tid; k < c.Iw; k += nth) io.raster_in[(size_t)t * io.rs_i + k] = rec[k];
        }
        if (t + 1 < steps) draw(t0 + (unsigned long long)(t + 1));
        add(0);
        for (int a = U; a < n; a += U) {
            load(a);
            add(a);
        }
        uint32_t nsi = 0u;
#pragma unroll
        for (int k = 0; k < NPT; ++k) {
            const int j = tid + k * nth;
            if (c.wprec == SNN_W_FP8E4M3) I[k] = __fmul_rn(I[k], __frcp_rn(inv[k]));
            st[k] = pair_update(c, v[k], vi[k], st[k], I[k], C, th[k]);
            if (j >= N) st[k] = 0u;                        // (no neuron: no spikes)
            const bool se = (st[k] & ST_SE) != 0u, si = (st[k] & ST_SI) != 0u;
            if (TRACE) x[k] = __fadd_rn(__fmul_rn(x[k], c.a_x), se ? 1.0f : 0.0f);
            cnt[k] += se ? 1u : 0u;
            const uint32_t wi = __ballot_sync(FULL, si);
            nsi += (uint32_t)__popc(wi);
            if (c.rec_raster) {
                const uint32_t we = __ballot_sync(FULL, se);
                if (lane == 0 && j < N) {                  // (j >> 5: the warp's word)
                    io.raster_e[(size_t)t * io.rs_n + (j >> 5)] = we;
                    io.raster_i[(size_t)t * io.rs_n + (j >> 5)] = wi;
                }
            }
        }
        if (lane == 0 && nsi) atomicAdd(&s_cnt[t & 1], nsi);
        __syncthreads();
        // ---- Y: the count, and the next step's list
        C = (int)s_cnt[t & 1];
        if (tid == 0) s_cnt[(t + 1) & 1] = 0u;
        if (t + 1 < steps) n = list();
        __syncthreads();
    }

    // ---- the state back
#pragma unroll
    for (int k = 0; k < NPT; ++k) {
        const int j = tid + k * nth;
        if (j >= N) continue;
        io.v_e[j] = v[k];
        io.v_i[j] = vi[k];
        if (TRACE) io.x_post[j] = x[k];
        io.st[j] = st[k];
        if (cnt[k]) io.counts[j] += cnt[k];
    }
    if (TRACE) {
        for (int k = tid; k < nl; k += nth) io.x_out[cidx[k]] = xs[k];
        for (int i = tid; i < NI; i += nth) {              // the inputs that never spike: decay alone
            if (io.thr[i] != 0u) continue;
            float y = io.x_in[i];
            if (y != 0.0f)
                for (int t = 0; t < steps; ++t) y = __fadd_rn(__fmul_rn(y, c.a_x), 0.0f);
            io.x_out[i] = y;
        }
    }
    return C;
}

}  // namespace snn

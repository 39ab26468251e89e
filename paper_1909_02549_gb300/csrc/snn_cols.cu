// Column-tile form of one time step, used by the per-step and graph runs: one
// launch per step in which a block owns TC neuron columns for every sample.
//
// The step's neuron update, the batch reduction of the STDP update and the
// thresholds are local to a column, so the block keeps what one hands to the
// next in shared memory: the depression terms e[b][j] = nu_pre x_post[b][j] and
// the step's spike masks.  The weights as the current reads them (converted
// once) are staged there too.  State, 16 bytes a neuron, is read and written
// once.  The first blocks of the grid draw the next step's input spikes, whose
// buffers rotate (Bufs), so that no launch of its own is needed for them.  The
// update's two sums take two lane layouts: the potentiation a row per lane (x_pre
// rows are coalesced), the depression a row and four columns.
//
// What bounds it: the state's bytes against HBM, then issue slots.  Per step at
// 100 -> 10000, B = 1024, learning: 328 MB, 48 us at the copy bandwidth.  The
// separate kernels took 535 us on average (encode 5, neuron 129, the rest the
// update, which gathers x_pre with a sample per lane), this form 150 us: 97 while
// nothing fires, 135 between the bursts in which most columns fire, 180 inside
// them; it issues 52 to 119 M warp instructions a step.  784 -> 6400, B = 1024:
// 1293 us before, 202 now.
//
// The sums are those of k_neuron and k_stdp: currents in ascending input, the
// potentiation and depression sums each in ascending sample.  Samples in which
// a column has not fired have e = +0, which leaves a sum unchanged and gives
// the maximum the 0 that idle samples give it.
#include <cfloat>

#include "snn_internal.cuh"

namespace snn {
namespace {

constexpr unsigned FULL = 0xFFFFFFFFu;
constexpr int CT = 256;                  // threads per block
constexpr int CB = 3;                    // blocks per SM that registers and tile sizes aim at
constexpr int CW = CT / 32;
constexpr int EG = 4;                    // warps that draw one sample (CW / EG samples per block)
constexpr int ES = CW / EG;

struct ColGeom {
    int TC, lgq;                         // columns per block, log2 of its column quads
    int Ip;                              // stride of the active-input lists
    int ntile, nenc;                     // column blocks, drawing blocks
    int pls;                             // stride of the post-sample lists
    size_t o_es, o_q, o_pl, o_th, smem;  // shared memory: staged weights (then the potentiation), e, spike
                                         // masks, post-sample lists, thresholds, FP8 scales, post counts
};

// The input spikes, traces and ascending active-input lists of absolute step te
// (run-local step t_enc): EG warps per sample.
__device__ __forceinline__ void draw_samples(const Consts& c, const Bufs& d, const ColGeom& g,
                                             unsigned long long te, int t_enc, uint32_t* wbuf) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int grp = warp / EG, gw = warp % EG;
    const int b = blockIdx.x * ES + grp;
    if (b >= c.B) return;                                  // (whole groups)
    const size_t nbi = (size_t)c.B * c.n_in;
    const float* xp = d.x_pre + (size_t)((te + XPRE_SLOTS - 1) % XPRE_SLOTS) * nbi + (size_t)b * c.n_in;
    float* xc = d.x_pre + (size_t)(te % XPRE_SLOTS) * nbi + (size_t)b * c.n_in;
    uint32_t* pre = d.preT + (size_t)(te % PRET_SLOTS) * c.n_in * c.Bw + (b >> 5);
    uint32_t* words = wbuf + grp * c.Iw;
    const uint64_t seed = d.seeds[b];
    const int cur = (int)(te & 1ull);
    for (int w = gw; w < c.Iw; w += EG) {
        const int i = w * 32 + lane;
        const int ic = i < c.n_in ? i : c.n_in - 1;
        const uint32_t thr = d.thr[(size_t)b * c.n_in + ic];
        const float xo = xp[ic];
        bool s = false;
        if (i < c.n_in) {
            s = poisson_spike(seed, te, c.n_in, i, thr);
            xc[i] = __fadd_rn(__fmul_rn(xo, c.a_x), s ? 1.0f : 0.0f);
            if (s) atomicOr(&pre[(size_t)i * c.Bw], 1u << (b & 31));
        }
        const uint32_t m = __ballot_sync(FULL, s);
        if (lane == 0) {
            words[w] = m;
            d.inb[((size_t)cur * c.B + b) * c.Iw + w] = m;
            if (c.rec_input) d.raster_in[((size_t)t_enc * c.B + b) * c.Iw + w] = m;
        }
    }
    static_assert(ES == 2, "a named barrier per group, with immediate numbers");
    if (grp == 0) asm volatile("bar.sync 1, 128;" ::: "memory");
    else asm volatile("bar.sync 2, 128;" ::: "memory");
    if (gw != 0) return;
    uint16_t* out = d.act_idx + ((size_t)cur * c.B + b) * g.Ip;
    int run = 0;
    for (int w0 = 0; w0 < c.Iw; w0 += 32) {
        const uint32_t word = w0 + lane < c.Iw ? words[w0 + lane] : 0u;
        const int n = __popc(word);
        int x = n;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(FULL, x, o);
            if (lane >= o) x += y;
        }
        int off = run + x - n;
        for (uint32_t m = word; m; m &= m - 1) out[off++] = (uint16_t)((w0 + lane) * 32 + __ffs(m) - 1);
        run += __shfl_sync(FULL, x, 31);
    }
    if (lane < ((run + 3) & ~3) - run) out[run + lane] = (uint16_t)c.n_in;   // whole groups of four: the zero row
    if (lane == 0) d.act_cnt[(size_t)cur * c.B + b] = (uint32_t)run;
}

// The thresholds after a step in which column j had n spikes over the batch.
template <int RED>
__device__ __forceinline__ double theta_after(const Consts& c, double th, int n) {
    double r;
    if (RED == SNN_REDUCE_SUM) r = (double)n;
    else if (RED == SNN_REDUCE_MEAN)      // n / B; exactly n * 2^-k for B = 2^k
        r = c.B_pow2 ? __dmul_rn((double)n, (double)c.inv_B) : __ddiv_rn((double)n, (double)c.B);
    else r = n > 0 ? 1.0 : 0.0;
    return __dadd_rn(__dmul_rn(th, c.a_th), __dmul_rn(c.theta_plus, r));
}

// Four adjacent elements p[0..3], of which nv are the row's; V4: 16-byte aligned
// and all four inside, one access.
template <bool V4, typename T>
__device__ __forceinline__ void ld4(const T* p, int nv, T (&o)[4]) {
    if (V4) {
        const uint4 q = __ldcg(reinterpret_cast<const uint4*>(p));   // (read once: kept out of L1)
        const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) o[k] = *reinterpret_cast<const T*>(&w[k]);
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) o[k] = p[k < nv ? k : 0];
    }
}
template <bool V4, typename T>
__device__ __forceinline__ void st4(T* p, int nv, const T (&o)[4]) {
    if (V4) {
        uint4 q;
        q.x = *reinterpret_cast<const uint32_t*>(&o[0]);
        q.y = *reinterpret_cast<const uint32_t*>(&o[1]);
        q.z = *reinterpret_cast<const uint32_t*>(&o[2]);
        q.w = *reinterpret_cast<const uint32_t*>(&o[3]);
        __stcg(reinterpret_cast<uint4*>(p), q);
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (k < nv) p[k] = o[k];
    }
}

constexpr int XU = 8;                    // post samples whose x_pre loads are issued together

// Pot[i][j] of the columns that fired: the sum over their post samples,
// ascending, of nu_post x_pre (max: the largest of nu_post x_pre - e, e where the
// input fired too).  A task is (column, 32 R input rows), R adjacent rows per
// lane (one 16-byte load of x_pre where R = 4), XU samples' loads in flight.
template <int RED, int R>
__device__ __forceinline__ void potentiate(const Consts& c, const uint16_t* PL, int pls, const int* npost,
                                           const float* xp, const uint32_t* pre, const float* Es, float* Pot,
                                           int TC, int nc) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, NI = c.n_in;
    const int nch = (NI + 32 * R - 1) / (32 * R);
    for (int u = warp; u < nc * nch; u += CW) {
        const int j = u / nch, i = ((u - j * nch) * 32 + lane) * R, n = npost[j];
        if (n == 0) continue;
        const float* xr = xp + (i < NI ? i : 0);
        const uint16_t* bl = PL + j * pls;                 // (16-byte rows)
        float p[R];
#pragma unroll
        for (int r = 0; r < R; ++r) p[r] = RED == SNN_REDUCE_MAX ? -FLT_MAX : 0.0f;
        auto load = [&](int b, float (&x)[R]) {
            const float* q = xr + (size_t)((uint32_t)b * (uint32_t)NI);   // (B * n_in < 2^31)
            if (R == 4) {
                const float4 v = *reinterpret_cast<const float4*>(q);
                x[0] = v.x; x[1 % R] = v.y; x[2 % R] = v.z; x[3 % R] = v.w;
            } else {
                x[0] = *q;
            }
        };
        auto add = [&](int b, const float (&x)[R]) {
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const float a = __fmul_rn(c.nu_post, x[r]);
                if (RED == SNN_REDUCE_MAX) {
                    const int ir = i + r < NI ? i + r : 0;
                    const bool pr = (pre[(size_t)ir * c.Bw + (b >> 5)] >> (b & 31)) & 1u;
                    p[r] = fmaxf(p[r], __fsub_rn(a, pr ? Es[b * TC + j] : 0.0f));
                } else {
                    p[r] = __fadd_rn(p[r], a);
                }
            }
        };
        constexpr int U = XU;
        int k = 0;
        for (; k + U <= n; k += U) {
            int bs[U];
            float x[U][R];
#pragma unroll
            for (int z = 0; z < U; z += 2) {
                const uint32_t w = *reinterpret_cast<const uint32_t*>(bl + k + z);
                bs[z] = (int)(w & 0xFFFFu);
                bs[z + 1] = (int)(w >> 16);
            }
#pragma unroll
            for (int z = 0; z < U; ++z) load(bs[z], x[z]);
#pragma unroll
            for (int z = 0; z < U; ++z) add(bs[z], x[z]);
        }
        for (; k < n; ++k) {
            float x[R];
            load(bl[k], x);
            add(bl[k], x);
        }
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (i + r < NI) Pot[(i + r) * TC + j] = p[r];
    }
}

// t_local = -1: only the drawing blocks, for the run's first step.
template <int RED, bool V4>
__global__ void __launch_bounds__(CT, CB) k_cols(const __grid_constant__ Consts c, const __grid_constant__ Bufs d,
                                                const __grid_constant__ ColGeom g, const int t_local) {
    extern __shared__ __align__(16) unsigned char csm[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const unsigned long long te = d.step[0] + (unsigned long long)(t_local + 1);   // the step drawn here
    {   // the next step's count accumulator and the input masks of the one after
        // it: their last readers ran in an earlier launch
        const size_t gt = (size_t)blockIdx.x * CT + tid, nth = (size_t)gridDim.x * CT;
        uint32_t* cnt = d.cnt + (size_t)(te % 3ull) * c.B;
        for (size_t k = gt; k < (size_t)c.B; k += nth) cnt[k] = 0u;
        const size_t n_pre = (size_t)c.n_in * c.Bw;
        uint32_t* nxt = d.preT + (size_t)((te + 1ull) % PRET_SLOTS) * n_pre;
        for (size_t k = gt; k < n_pre; k += nth) nxt[k] = 0u;
    }
    if ((int)blockIdx.x < g.nenc) {
        draw_samples(c, d, g, te, t_local + 1, reinterpret_cast<uint32_t*>(csm));
        return;
    }
    if (t_local < 0) return;
    const unsigned long long tt = te - 1ull;
    const int cur = (int)(tt & 1ull), p3 = (int)(tt % 3ull);
    const int B = c.B, N = c.N, NI = c.n_in, Bw = c.Bw, TC = g.TC, lgq = g.lgq, nq = 1 << lgq;
    const int j0 = ((int)blockIdx.x - g.nenc) * TC, nc = min(TC, N - j0);
    float* const Wc = reinterpret_cast<float*>(csm);                 // [NI + 1][TC] as the current reads them
    float* const Es = reinterpret_cast<float*>(csm + g.o_es);        // [B + 1][TC], the last row zero
    uint32_t* const Qm = reinterpret_cast<uint32_t*>(csm + g.o_q);   // [Bw][TC]
    uint16_t* const PL = reinterpret_cast<uint16_t*>(csm + g.o_pl);  // [TC][pls] samples in which a column fired
    float* const thj = reinterpret_cast<float*>(csm + g.o_th);       // [TC] thresholds, [TC] FP8 scales,
    float* const wsc = thj + TC;                                     // [TC] post spikes
    int* const npost = reinterpret_cast<int*>(wsc + TC);
    __shared__ double thS[8];                              // the columns' thresholds (TC <= 8)
    __shared__ int s_any;                                  // a column of the tile has a trace or a spike

    // ---- staged weights, thresholds, cleared masks
    for (int k = tid; k < Bw * TC; k += CT) Qm[k] = 0u;
    if (tid < TC) {
        const double th = tid < nc ? d.theta[j0 + tid] : 0.0;
        thS[tid] = th;
        thj[tid] = __fadd_rn(c.e_thresh, __double2float_rn(th));
    }
    if (tid == 0) s_any = 0;
    if (c.learn && tid < TC) Es[B * TC + tid] = 0.0f;
    if (c.wprec == SNN_W_FP8E4M3) {                        // column scales of this step's weights
        for (int jl = warp; jl < TC; jl += CW) {
            float m = 0.0f;
            if (jl < nc)
                for (int i = lane; i < NI; i += 32) m = fmaxf(m, fabsf(d.W[(size_t)i * N + j0 + jl]));
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(FULL, m, o));
            if (lane == 0) wsc[jl] = e4m3_scale_of(m);
        }
        __syncthreads();
    }
    for (int k = tid; k < (NI + 1) << lgq; k += CT) {
        const int i = k >> lgq, jl = 4 * (k & (nq - 1)), nv = nc - jl;
        float w[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        if (i < NI && nv > 0) {
            ld4<V4>(d.W + (size_t)i * N + j0 + jl, nv, w);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if (c.wprec == SNN_W_BF16) w[q] = w_read_bf16(w[q]);
                else if (c.wprec == SNN_W_FP8E4M3) w[q] = w_read_e4m3(w[q], __frcp_rn(wsc[jl + q]));
            }
        }
        *reinterpret_cast<float4*>(Wc + 4 * k) = make_float4(w[0], w[1], w[2], w[3]);
    }
    __syncthreads();

    // ---- currents and neurons: a thread per (sample, column quad)
    const uint32_t* cnt_prev = d.cnt + (size_t)((p3 + 2) % 3) * B;
    const uint32_t* an = d.act_cnt + (size_t)cur * B;
    const uint16_t* acts = d.act_idx + (size_t)cur * B * g.Ip;
    bool mine = false;
    // the next unit's loads are in flight while one is computed
    struct Unit { float ve[4], vi[4], xq[4]; uint32_t st[4]; int na, C; uint2 i4; };
    const int nu = B << lgq;
    auto load = [&](int u, Unit& x) {
        const int b = u >> lgq, jl = 4 * (u & (nq - 1)), left = nc - jl, nv = V4 ? 4 : left;
        const size_t idx = left > 0 ? (size_t)b * N + j0 + jl : 0;
        ld4<V4>(d.v_e + idx, nv, x.ve);
        ld4<V4>(d.v_i + idx, nv, x.vi);
        ld4<V4>(d.x_post + idx, nv, x.xq);
        ld4<V4>(d.st + idx, nv, x.st);
        x.na = (int)an[b];
        x.C = (int)cnt_prev[b];
        x.i4 = *reinterpret_cast<const uint2*>(acts + (size_t)b * g.Ip);   // (rows of at least 8 entries)
    };
    Unit nx;
    if (tid < nu) load(tid, nx);
    for (int u = tid; u < nu; u += CT) {
        Unit x = nx;
        load(u + CT < nu ? u + CT : u, nx);
        const int b = u >> lgq, jl = 4 * (u & (nq - 1)), left = nc - jl, nv = V4 ? 4 : left;
        if (left <= 0) {
            if (c.learn) *reinterpret_cast<float4*>(Es + b * TC + jl) = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            continue;
        }
        const size_t idx = (size_t)b * N + j0 + jl;
        float (&ve)[4] = x.ve, (&vi)[4] = x.vi, (&xq)[4] = x.xq;
        uint32_t (&st)[4] = x.st;
        const int na = x.na, C = x.C;
        const uint16_t* al = acts + (size_t)b * g.Ip;
        float I[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        for (int a = 0; a < na; a += 4) {                  // four entries a load, the last padded with the
            const uint2 i4 = a == 0 ? x.i4 : *reinterpret_cast<const uint2*>(al + a);   // zero row (never -0)
            const uint32_t r[4] = {i4.x & 0xFFFFu, i4.x >> 16, i4.y & 0xFFFFu, i4.y >> 16};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float4 w = *reinterpret_cast<const float4*>(Wc + r[q] * TC + jl);
                I[0] = __fadd_rn(I[0], w.x);
                I[1] = __fadd_rn(I[1], w.y);
                I[2] = __fadd_rn(I[2], w.z);
                I[3] = __fadd_rn(I[3], w.w);
            }
        }
        float e[4];
        uint32_t fe = 0u, fi = 0u;                         // the quad's spikes
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (c.wprec == SNN_W_FP8E4M3) I[q] = __fmul_rn(I[q], wsc[jl + q]);
            st[q] = pair_update(c, ve[q], vi[q], st[q], I[q], C, thj[jl + q]);
            xq[q] = __fadd_rn(__fmul_rn(xq[q], c.a_x), (st[q] & ST_SE) ? 1.0f : 0.0f);
            e[q] = q < nv ? __fmul_rn(c.nu_pre, xq[q]) : 0.0f;
            mine = mine || (q < nv && xq[q] != 0.0f);
            if (st[q] & ST_SE) fe |= 1u << q;
            if (st[q] & ST_SI) fi |= 1u << q;
        }
        if (nv < 4) { fe &= (1u << nv) - 1u; fi &= (1u << nv) - 1u; }
        for (uint32_t m = fe; m; m &= m - 1) {
            const int q = __ffs(m) - 1;
            const uint32_t bit = 1u << (b & 31);
            atomicAdd(&d.counts[idx + q], 1u);             // (one writer; no value is waited for)
            atomicOr(&Qm[(b >> 5) * TC + jl + q], bit);
            atomicOr(&d.spkT[(size_t)(j0 + jl + q) * Bw + (b >> 5)], bit);
        }
        if (fi) atomicAdd(&d.cnt[(size_t)p3 * B + b], (uint32_t)__popc(fi));
        if (c.rec_raster && (fe | fi)) {                   // (j0 + jl is a multiple of 4: one word)
            const size_t o = ((size_t)t_local * B + b) * c.Nw + ((j0 + jl) >> 5);
            if (fe) atomicOr(&d.raster_e[o], fe << ((j0 + jl) & 31));
            if (fi) atomicOr(&d.raster_i[o], fi << ((j0 + jl) & 31));
        }
        st4<V4>(d.v_e + idx, nv, ve);
        st4<V4>(d.v_i + idx, nv, vi);
        st4<V4>(d.x_post + idx, nv, xq);
        st4<V4>(d.st + idx, nv, st);
        if (c.learn) *reinterpret_cast<float4*>(Es + b * TC + jl) = make_float4(e[0], e[1], e[2], e[3]);
    }
    if (!c.learn) return;
    if (__any_sync(FULL, mine) && lane == 0) s_any = 1;
    __syncthreads();

    // ---- per column: the samples in which it fired, ascending, and its threshold
    for (int j = warp; j < TC; j += CW) {
        uint16_t* out = PL + j * g.pls;
        int run = 0;
        for (int w0 = 0; w0 < Bw; w0 += 32) {
            const uint32_t word = w0 + lane < Bw ? Qm[(w0 + lane) * TC + j] : 0u;
            const int n = __popc(word);
            int x = n;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(FULL, x, o);
                if (lane >= o) x += y;
            }
            int off = run + x - n;
            for (uint32_t m = word; m; m &= m - 1) out[off++] = (uint16_t)((w0 + lane) * 32 + __ffs(m) - 1);
            run += __shfl_sync(FULL, x, 31);
        }
        if (lane == 0) {
            npost[j] = run;
            if (j < nc) d.theta[j0 + j] = theta_after<RED>(c, thS[j], run);
        }
    }
    __syncthreads();
    if (!s_any) return;                                    // no trace, no spike: nothing to update (uniform)

    // ---- potentiation of the columns that fired, into the staged weights' place:
    // a task per (column, 32 input rows), lanes = rows, so each x_pre row is one
    // coalesced load; sum over the post samples, ascending, XU loads in flight
    float* const Pot = Wc;                                 // [NI][TC], read where npost > 0
    const float* const xp = d.x_pre + (size_t)(tt % XPRE_SLOTS) * B * NI;
    const uint32_t* const pre = d.preT + (size_t)(tt % PRET_SLOTS) * NI * Bw;
    if ((NI & 3) == 0) potentiate<RED, 4>(c, PL, g.pls, npost, xp, pre, Es, Pot, TC, nc);
    else potentiate<RED, 1>(c, PL, g.pls, npost, xp, pre, Es, Pot, TC, nc);
    __syncthreads();

    // ---- depression and the update: a lane per (input row, column quad)
    const int RW = 32 >> lgq, jl = 4 * (lane & (nq - 1)), nv = nc - jl;
    const float* const Eq = Es + jl;
    int np[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) np[k] = nv > k ? npost[jl + k] : 0;
    const bool anyp = (np[0] | np[1] | np[2] | np[3]) != 0;
    for (int i = RW * warp + (lane >> lgq); i < NI; i += RW * CW) {
        if (nv <= 0) continue;
        const uint32_t* P = pre + (size_t)i * Bw;
        float dep[4];                                      // max: the running maximum of the idle columns' 0 - e
        int nev = 0;                                       // samples whose input fired
        uint32_t both[4] = {0u, 0u, 0u, 0u};               // max: of them those in which the column fired too
#pragma unroll
        for (int k = 0; k < 4; ++k) dep[k] = RED == SNN_REDUCE_MAX ? -FLT_MAX : 0.0f;
        // the row's weights, in flight during the walk
        const size_t o = (size_t)i * N + j0 + jl;
        float wv[4], wl[4];
        ld4<V4>(d.W + o, nv, wv);
        if (c.wmaster) ld4<V4>(d.W_lo + o, nv, wl);
        // every sample whose input i fired, ascending; PWN words a round trip
        constexpr int PWN = 16;
        for (int w0 = 0; w0 < Bw; w0 += PWN) {
            uint32_t pw[PWN];
            if ((Bw & 3) == 0) {
#pragma unroll
                for (int z = 0; z < PWN; z += 4) {
                    const uint4 q = *reinterpret_cast<const uint4*>(P + (w0 + z < Bw ? w0 + z : 0));
                    pw[z] = q.x; pw[z + 1] = q.y; pw[z + 2] = q.z; pw[z + 3] = q.w;
                }
            } else {
#pragma unroll
                for (int z = 0; z < PWN; ++z) pw[z] = P[w0 + z < Bw ? w0 + z : 0];
            }
#pragma unroll
            for (int z = 0; z < PWN; ++z) {
                if (w0 + z >= Bw) break;
                const int w = w0 + z;
                uint32_t m = pw[z];
                nev += __popc(m);
                uint32_t qk[4] = {0u, 0u, 0u, 0u};
                if (RED == SNN_REDUCE_MAX) {
                    const uint4 q = *reinterpret_cast<const uint4*>(Qm + w * TC + jl);
                    qk[0] = q.x; qk[1] = q.y; qk[2] = q.z; qk[3] = q.w;
#pragma unroll
                    for (int k = 0; k < 4; ++k) both[k] += __popc(m & qk[k]);
                }
                if (RED == SNN_REDUCE_MAX) {
                    for (; m; m &= m - 1) {
                        const int bit = __ffs(m) - 1;
                        const float4 e = *reinterpret_cast<const float4*>(Eq + (w * 32 + bit) * TC);
                        const float ev[4] = {e.x, e.y, e.z, e.w};
#pragma unroll
                        for (int k = 0; k < 4; ++k)        // post samples: above
                            if (!((qk[k] >> bit) & 1u)) dep[k] = fmaxf(dep[k], __fsub_rn(0.0f, ev[k]));
                    }
                } else {
                    while (m) {                            // two samples a turn, the second perhaps the zero row
                        const int ba = w * 32 + __ffs(m) - 1;
                        m &= m - 1;
                        const int bb = m ? w * 32 + __ffs(m) - 1 : B;
                        m &= m - 1;
                        const float4 ea = *reinterpret_cast<const float4*>(Eq + ba * TC);
                        const float4 eb = *reinterpret_cast<const float4*>(Eq + bb * TC);
                        dep[0] = __fadd_rn(__fadd_rn(dep[0], ea.x), eb.x);
                        dep[1] = __fadd_rn(__fadd_rn(dep[1], ea.y), eb.y);
                        dep[2] = __fadd_rn(__fadd_rn(dep[2], ea.z), eb.z);
                        dep[3] = __fadd_rn(__fadd_rn(dep[3], ea.w), eb.w);
                    }
                }
            }
        }
        if (nev == 0 && !anyp) continue;
        const float4 p4 = *reinterpret_cast<const float4*>(Pot + i * TC + jl);
        const float pt[4] = {p4.x, p4.y, p4.z, p4.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            float D;
            if (RED == SNN_REDUCE_MAX) {
                D = np[k] ? fmaxf(pt[k], dep[k]) : dep[k];
                if (nev + np[k] - (int)both[k] < B) D = fmaxf(D, 0.0f);   // idle samples add 0
            } else {
                D = __fsub_rn(np[k] ? pt[k] : 0.0f, dep[k]);
                // 0 / B = 0 with its sign: no division for the columns without a trace
                // (784->2440, B = 20: 22.8 -> 20.0 us a step; separate kernels 21.1)
                if (RED == SNN_REDUCE_MEAN && D != 0.0f) D = batch_mean(c, D);
            }
            if (c.wmaster) master_add(wv[k], wl[k], D, c.w_min, c.w_max);
            else wv[k] = plain_add(wv[k], D, c.w_min, c.w_max);
        }
        st4<V4>(d.W + o, nv, wv);
        if (c.wmaster) st4<V4>(d.W_lo + o, nv, wl);
    }
}

// Columns per block: eight (a 32-byte sector of each state row), unless four let
// CB blocks share an SM's shared memory (their phases overlap: one streams state
// while another updates) or give every SM two blocks and still fit one wave: a few
// blocks left over take a second one (784->2000 at B = 16 and 128, us a step with
// four columns, eight, and the separate kernels: 19.6, 13.4, 17.8 and 28.6, 19.5,
// 33.7; frozen at B = 128: 11.6, 7.5, 11.7).  With the maximum, whose walk has more
// registers and longer rows, two short waves stay faster above 512 samples (784->2200,
// B = 1024: 210 and 275).  TC = 0: no tile fits.
ColGeom col_geom(const Consts& c, int sms, size_t smem_optin) {
    ColGeom g{};
    g.Ip = (c.n_in + 7) & ~7;
    g.nenc = (c.B + ES - 1) / ES;
    const size_t share = (smem_optin + 1024) / CB - 1024;  // (an SM's shared memory is the opt-in limit and 1 KB)
    for (int tc = 8; tc >= 4; tc /= 2) {
        ColGeom t = g;
        auto up = [](size_t x) { return (x + 15) & ~(size_t)15; };
        t.TC = tc;
        t.lgq = tc == 8 ? 1 : 0;
        t.ntile = (c.N + tc - 1) / tc;
        t.o_es = up((size_t)(c.n_in + 1) * tc * 4);
        t.o_q = t.o_es + (c.learn ? up((size_t)(c.B + 1) * tc * 4) : 0);
        t.pls = (c.B + 7) & ~7;
        t.o_pl = t.o_q + up((size_t)c.Bw * tc * 4);
        t.o_th = t.o_pl + (c.learn ? up((size_t)tc * t.pls * 2) : 0);
        t.smem = t.o_th + up((size_t)tc * 12);
        const size_t enc = up((size_t)ES * c.Iw * 4);
        if (t.smem < enc) t.smem = enc;
        if (t.smem + 1024 > smem_optin) continue;
        const bool one_wave = t.ntile <= CB * sms || (c.learn && c.reduce == SNN_REDUCE_MAX && c.B > 512);
        if (g.TC == 0 || g.smem > share || (g.ntile < 2 * sms && one_wave)) g = t;
        else break;
    }
    return g;
}

// Whether the column tiles are faster than the separate kernels.  A block runs all
// samples of its columns, so few columns leave SMs idle when samples are many, and
// it stages its weights before it starts, which few samples do not repay where the
// blocks need several waves.  The separate update grows with n_in, B and the spikes,
// so learning moves the line far out.  Us a step, graph runs of 40 steps, separate
// kernels / this one (784 inputs: digits; 100: 120 Hz):
//   frozen, aligned rows, 100 inputs: 50 columns at B = 128 and 1024: 7.0 / 5.4, 8.1 /
//   27; 600 at 176 and 428 7.7 / 6.3, 8.5 / 11.2; 1800 at 64 and 128 7.4 / 6.7, 8.1 /
//   8.5; 2440 at 512 19.7 / 17.3; 784 inputs: 50 at 256 and 1024 11 / 8.7, 16.8 / 25.7;
//   600 at 428 and 2048 14.2 / 13.1, 44.8 / 51.2; 1600 at 1024 44.0 / 36.6; 32 inputs:
//   1000 at B = 16, 64 and 428: 4.5 / 6.0, 4.8 / 4.2, 7.0 / 10.6;
//   frozen, rows that are not 16-byte aligned, 784 inputs: 1023 at 100 and 128 10.4 /
//   8.3, 10.6 / 13.5; 2999 at 48 and 100 10.2 / 9.6, 12.4 / 14.8;
//   learning, several waves: 10000 columns at B = 33, 64 and 200: 784 inputs 47.8 /
//   54.5, 57.7 / 47.2, 149.7 / 85; 100 inputs 19.0 / 28.9, 24.7 / 20.4, 57 / 43; 225
//   inputs 15.5 / 28, 18.1 / 18.3, 39.0 / 39.4; unaligned, 784->6001 at 33, 64 and 128
//   34.3 / 44.6, 42.8 / 44.9, 65.9 / 58; sum, 225->10000 at 33 and 64 13.9 / 15.7, 17.6 /
//   16.7; max, 784->6400 at 40 64.6 / 54.2;
//   learning, one wave: divided means of a few samples, 1023->2440 at B = 3 and 40 21.4 /
//   24, 33.1 / 29.8; unaligned, 784->1537 at 33, 128 and 256 22.2 / 21, 31.2 / 35.6,
//   52.5 / 49.2; 32 inputs, 1000 at B = 128 and 256 7.0 / 5.6, 7.7 / 9.6;
//   runs of one step, which launch the drawing blocks on their own: 784->6400, B = 64 40.5
//   / 44.6 learning, 35.8 / 38.1 frozen; B = 256 0.78 and 0.85 of the separate kernels'.
bool pays(const Consts& c, const ColGeom& g, int sms, int T) {
    if (T == 1 && c.N > 1024 && c.B < 128) return false;
    const bool aligned = (c.N & 3) == 0, waves = (c.N + 7) / 8 > CB * sms, few_inputs = c.n_in <= 96;
    if (!c.learn) {
        if (few_inputs) return false;
        if (waves) return aligned && c.B >= 64;
        if (g.TC == 8) return aligned ? c.N >= 16 * sms || c.n_in >= 512 || c.B <= 64 * c.Iw : c.B <= 48;
        if (!aligned && c.N > 512) return c.B <= (c.N <= 8 * sms ? 100 : 64);
        if (c.n_in >= 512 && c.N >= 1000) return true;
        return c.B <= (c.N < 64 ? 80 + 12 * c.Iw : c.N <= 8 * sms ? 112 + 16 * c.Iw : 64 + 12 * c.Iw);
    }
    const bool divides = c.reduce == SNN_REDUCE_MEAN && !c.B_pow2;
    if (few_inputs) return !waves && c.B <= (c.reduce == SNN_REDUCE_MAX ? 256 : 128) && (g.TC == 4 || !divides);
    if (waves) return c.B >= (divides ? (c.n_in >= 512 ? 100 : 160) : aligned ? 40 : 128);
    if (g.TC == 8) return !divides || c.n_in <= 128 || c.B > (aligned ? 12 : 31);
    return aligned || c.N <= 8 * sms || c.n_in < 512 || c.B <= 48 || c.B >= 256;
}

}  // namespace

cudaError_t launch_cols_step(const Consts& c, const Bufs& d, int t_local, int T, cudaStream_t s, int* used) {
    *used = 0;
    if (c.rule != SNN_RULE_PAIR || c.n_in > 65534 || c.B > 65535) return cudaSuccess;
    int dev = 0, sms = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    ColGeom g = col_geom(c, sms, (size_t)optin);
    if (g.TC == 0 || !pays(c, g, sms, T)) return cudaSuccess;
    const bool v4 = (c.N & 3) == 0;
    auto kern = c.reduce == SNN_REDUCE_SUM    ? (v4 ? k_cols<SNN_REDUCE_SUM, true> : k_cols<SNN_REDUCE_SUM, false>)
                : c.reduce == SNN_REDUCE_MEAN ? (v4 ? k_cols<SNN_REDUCE_MEAN, true> : k_cols<SNN_REDUCE_MEAN, false>)
                                              : (v4 ? k_cols<SNN_REDUCE_MAX, true> : k_cols<SNN_REDUCE_MAX, false>);
    if (t_local == 0) {   // (the default limit, 48 KB, counts the kernel's static shared memory too)
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - 1024);
        if (e != cudaSuccess) return e;
    }
    if (t_local == 0) {                                    // the first step's input
        kern<<<g.nenc, CT, g.smem, s>>>(c, d, g, -1);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    if (t_local + 1 == T) g.nenc = 0;
    kern<<<g.nenc + g.ntile, CT, g.smem, s>>>(c, d, g, t_local);
    *used = 1;
    return cudaGetLastError();
}

}  // namespace snn

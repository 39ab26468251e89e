// Small-batch learning runs of the persistent mode: one thread-block cluster
// holds the whole network for all steps.
//
// With few samples a step has little work, and the column kernel's step is a
// chain of round trips through L2: the grid barrier, the staged counts, lists
// and masks, the encode's thresholds and traces.  Here CTA r of a cluster of CS owns the
// columns [r*ncc, (r+1)*ncc) of every sample, and all it needs of the others
// reaches its shared memory directly: the input-spike words (each CTA draws a
// share and stores it in every CTA) and the inhibitory counts (a spike adds to
// every CTA's).  Weights, thresholds, presynaptic traces (every CTA keeps all,
// they only change at live inputs) and lists are in shared memory, neuron state
// in registers.  One hardware cluster barrier a step, split around the update:
//   A  from the step's words: traces, each sample's active inputs, ascending, and
//      each input row's mask of samples (a warp per word);
//   B  half the warps: currents and neurons; the other half draw the next step's
//      words.  Arrive at the cluster barrier;
//   C  the update: a warp per 32 input rows, then wait at the cluster barrier.
// What bounds it: the instructions of one warp in turn (some twelve cycles each
// with their stalls, 420 a warp and step at 784->100, B = 1), the cluster barrier
// and three block barriers.  Us a step in the column kernel and here, runs of 60
// steps with their start: 784->100 at B = 1 8.1 and 2.5, 784->400 at B = 16 9.4 and
// 6.4; each further step 7.7 and 2.0, 8.6 and 5.3.
//
// Same sums as the other forms: currents in ascending input, the potentiation
// and depression sums each in ascending sample; terms left out are +0.
#include <cfloat>
#include <mutex>

#include "snn_internal.cuh"
#include "snn_tc.cuh"

namespace snn {
namespace {

constexpr unsigned FULL = 0xFFFFFFFFu;

struct SmallGeom {
    int CS, ncc;                          // CTAs of the cluster, columns per CTA
    int astr;                             // stride of the active-input lists
    size_t o_x, o_es, o_words, o_tab, o_wofs, o_act, o_idx, o_othr, o_oidx, o_rowm, o_q, o_cnt, o_th, smem;
};

__device__ __forceinline__ void red_cluster_add(uint32_t addr, uint32_t v) {
    asm volatile("red.relaxed.cluster.shared::cluster.add.u32 [%0], %1;" :: "r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

// IPT (sample, column) items per neuron thread.  Loops are not unrolled unless
// written out: unrolled, the step's code did not fit the instruction cache, and
// each phase began by fetching it (95 KB; hit rate 92 %).
// The batch mean of an accumulated update; the division out of line (see k_small).
__device__ __noinline__ float divide(float a, float b) { return __fdiv_rn(a, b); }
__device__ __noinline__ double divide(double a, double b) { return __ddiv_rn(a, b); }
__device__ __forceinline__ float mean_of(const Consts& c, float acc) {
    return c.B_pow2 ? __fmul_rn(acc, c.inv_B) : divide(acc, (float)c.B);
}

// ST threads, half of them neuron threads.
template <int ST, int IPT, bool MAX>
__global__ void __launch_bounds__(ST, 1) k_small(const __grid_constant__ Consts c, const __grid_constant__ Bufs d,
                                                 const __grid_constant__ SmallGeom g, const int T) {
    constexpr int SW = ST / 32, NT = ST / 2;
    extern __shared__ __align__(16) unsigned char sm[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int CS = g.CS, ncc = g.ncc, rank = blockIdx.x;
    const int N = c.N, NI = c.n_in, B = c.B;
    const int j0 = rank * ncc, nc = max(0, min(ncc, N - j0));
    float* const Ws = reinterpret_cast<float*>(sm);                        // [NI + 1][ncc], the last row zero
    float* const xs = reinterpret_cast<float*>(sm + g.o_x);                // [B][NI] presynaptic traces
    float* const Es = reinterpret_cast<float*>(sm + g.o_es);               // [B + 1][ncc] nu_pre x_post, the last row zero
    uint32_t* const words = reinterpret_cast<uint32_t*>(sm + g.o_words);   // [2][B * Iw] live-input words
    uint32_t* const tab = reinterpret_cast<uint32_t*>(sm + g.o_tab);       // word -> sample, word of the sample
    int* const wofs = reinterpret_cast<int*>(sm + g.o_wofs);               // [B + 1] first word of a sample
    uint16_t* const act = reinterpret_cast<uint16_t*>(sm + g.o_act);       // [B][astr] active inputs, ascending, whole
                                                                           // groups of four padded with the zero row
    uint16_t* const cidx = reinterpret_cast<uint16_t*>(sm + g.o_idx);      // [B][NI] live inputs, ascending
    uint32_t* const othr = reinterpret_cast<uint32_t*>(sm + g.o_othr);     // the words this CTA draws: thresholds
    uint16_t* const oidx = reinterpret_cast<uint16_t*>(sm + g.o_oidx);     // and inputs, 32 a word
    uint32_t* const rowm = reinterpret_cast<uint32_t*>(sm + g.o_rowm);     // [NI] samples whose input fired
    uint32_t* const Qm = reinterpret_cast<uint32_t*>(sm + g.o_q);          // [2][ncc] samples in which a column fired
    uint32_t* const cnt = reinterpret_cast<uint32_t*>(sm + g.o_cnt);       // [3][B] inhibitory counts, then [B] list lengths
    int* const nact = reinterpret_cast<int*>(cnt + 3 * B);
    double* const thS = reinterpret_cast<double*>(sm + g.o_th);            // [ncc], then the float thresholds
    float* const thj = reinterpret_cast<float*>(thS + ncc);
    __shared__ int s_live[32];
    __shared__ uint64_t s_seed[32];
    if (*reinterpret_cast<volatile uint32_t*>(d.err) != 0u) return;        // an earlier run failed: do nothing
    const unsigned long long base = d.step[0], last = base + (unsigned long long)T - 1ull;
    const size_t nbi = (size_t)B * NI;
    const int WB = B * c.Iw;                                               // words of a buffer

    // ---- set-up: columns, traces, live inputs (a rate, or a trace that still decays)
#pragma unroll 1
    for (int k = tid; k < (NI + 1) * ncc; k += ST) {
        const int i = k / ncc, jl = k - i * ncc;
        Ws[k] = i < NI && jl < nc ? d.W[(size_t)i * N + j0 + jl] : 0.0f;
    }
    const float* x_in = d.x_pre + (size_t)((base + XPRE_SLOTS - 1) % XPRE_SLOTS) * nbi;
#pragma unroll 1
    for (int k = tid; k < B * NI; k += ST) xs[k] = x_in[k];
#pragma unroll 1
    for (int k = tid; k < NI; k += ST) rowm[k] = 0u;
#pragma unroll 1
    for (int k = tid; k < ncc; k += ST) Es[B * ncc + k] = 0.0f;
#pragma unroll 1
    for (int k = tid; k < 2 * ncc; k += ST) Qm[k] = 0u;
#pragma unroll 1
    for (int b = tid; b < B; b += ST) {
        const int p = (int)((base + 2ull) % 3ull);
#pragma unroll 1
        for (int q = 0; q < 3; ++q) cnt[q * B + b] = q == p ? d.cnt[(size_t)p * B + b] : 0u;
    }
#pragma unroll 1
    for (int jl = tid; jl < ncc; jl += ST) {
        thS[jl] = jl < nc ? d.theta[j0 + jl] : 0.0;
        thj[jl] = __fadd_rn(c.e_thresh, __double2float_rn(thS[jl]));
    }
#pragma unroll 1
    for (int b = warp; b < B; b += SW) {
        int n = 0;
#pragma unroll 1
        for (int i0 = 0; i0 < NI; i0 += 32) {
            const int i = i0 + lane;
            const bool live = i < NI && (d.thr[(size_t)b * NI + i] != 0u || x_in[(size_t)b * NI + i] != 0.0f);
            const uint32_t m = __ballot_sync(FULL, live);
            if (live) cidx[b * NI + n + __popc(m & ((1u << lane) - 1u))] = (uint16_t)i;
            n += __popc(m);
        }
        if (lane == 0) {
            s_live[b] = n;
            s_seed[b] = d.seeds[b];
        }
    }
    __syncthreads();
    if (tid == 0) {
        int o = 0;
#pragma unroll 1
        for (int b = 0; b < B; ++b) { wofs[b] = o; o += (s_live[b] + 31) / 32; }
        wofs[B] = o;
    }
    __syncthreads();
    const int TW = wofs[B];
#pragma unroll 1
    for (int b = warp; b < B; b += SW)
#pragma unroll 1
        for (int w = lane; w < wofs[b + 1] - wofs[b]; w += 32) tab[wofs[b] + w] = (uint32_t)b | ((uint32_t)w << 8);
    __syncthreads();
#pragma unroll 1
    for (int q = rank + CS * warp, z = warp; q < TW; q += CS * SW, z += SW) {   // own word z is word rank + CS z
        const int b = (int)(tab[q] & 0xFFu), k = (int)(tab[q] >> 8) * 32 + lane;
        const int i = k < s_live[b] ? cidx[b * NI + k] : 0;
        oidx[z * 32 + lane] = (uint16_t)i;
        othr[z * 32 + lane] = k < s_live[b] ? d.thr[(size_t)b * NI + i] : 0u;
    }
    if (c.rec_input) {                                     // the raster's rows of this CTA's samples, cleared
#pragma unroll 1
        for (int b = rank; b < B; b += CS)
#pragma unroll 1
            for (int k = tid; k < T * c.Iw; k += ST)
                d.raster_in[((size_t)(k / c.Iw) * B + b) * c.Iw + k % c.Iw] = 0u;
    }

    // ---- the neuron threads' items
    float v[IPT], vi[IPT], x[IPT];
    uint32_t st[IPT], ns[IPT];
    int ib[IPT], ij[IPT];                                  // sample (-1: none), column
#pragma unroll
    for (int k = 0; k < IPT; ++k) {
        const int it = tid + k * NT;
        const int b = it / ncc, jl = it - b * ncc;
        const bool ok = tid < NT && b < B && jl < nc;
        ib[k] = ok ? b : -1;
        ij[k] = jl;
        const size_t o = ok ? (size_t)b * N + j0 + jl : 0;
        v[k] = ok ? d.v_e[o] : 0.0f;
        vi[k] = ok ? d.v_i[o] : 0.0f;
        x[k] = ok ? d.x_post[o] : 0.0f;
        st[k] = ok ? d.st[o] : 0u;
        ns[k] = 0u;
    }

    // this CTA's share of the words of local step t, into every CTA
    auto draw = [&](int t, int w0, int dw) {
        const unsigned long long tt = base + (unsigned long long)t;
        uint32_t* out = words + (t & 1) * WB;
#pragma unroll 1
        for (int z = w0, q = rank + CS * w0; q < TW; z += dw, q += CS * dw) {
            const bool s = poisson_spike(s_seed[tab[q] & 0xFFu], tt, NI, oidx[z * 32 + lane], othr[z * 32 + lane]);
            const uint32_t m = __ballot_sync(FULL, s);
            if (lane < CS) tc::st_cluster_u32(tc::cluster_map(tc::su32(out + q), (uint32_t)lane), m);
        }
    };

    tc::cluster_sync();                                    // every CTA runs before its memory is written
    draw(0, warp, SW);
    tc::cluster_sync();

    int p3 = (int)(base % 3ull);                           // the step's count slot
#pragma unroll 1
    for (int t = 0; t < T; ++t, p3 = p3 == 2 ? 0 : p3 + 1) {
        const int pp = p3 == 0 ? 2 : p3 - 1, pn = p3 == 2 ? 0 : p3 + 1;
        const uint32_t* wt = words + (t & 1) * WB;
        uint32_t* const Q = Qm + (t & 1) * ncc;
        // ---- A: traces, lists, row masks (a warp per word)
#pragma unroll 1
        for (int b = tid; b < B; b += ST) cnt[pn * B + b] = 0u;   // the next step's accumulator
#pragma unroll 1
        for (int q = warp; q < TW; q += SW) {
            const uint32_t e = tab[q];
            const int b = (int)(e & 0xFFu), w = (int)(e >> 8), k = w * 32 + lane;
            const uint32_t m = wt[q];
            int at = lane < w ? __popc(wt[q - w + lane]) : 0;
            if (w > 32)                                    // (more than 1024 live inputs)
#pragma unroll 1
                for (int y = 32 + lane; y < w; y += 32) at += __popc(wt[q - w + y]);
            at = __reduce_add_sync(FULL, at);
            const int n = at + __popc(m);
            uint16_t* const al = act + b * g.astr;
            if (k < s_live[b]) {
                const int i = cidx[b * NI + k];
                const bool s = (m >> lane) & 1u;
                float* xp = xs + b * NI + i;
                *xp = __fadd_rn(__fmul_rn(*xp, c.a_x), s ? 1.0f : 0.0f);
                if (s) {
                    al[at + __popc(m & ((1u << lane) - 1u))] = (uint16_t)i;
                    atomicOr(&rowm[i], 1u << b);
                    if (c.rec_input && b % CS == rank)
                        atomicOr(&d.raster_in[((size_t)t * B + b) * c.Iw + (i >> 5)], 1u << (i & 31));
                }
            }
            if (q + 1 == wofs[b + 1]) {                    // the sample's last word: its length and padding
                if (lane == 0) nact[b] = n;
                if (lane < ((n + 3) & ~3) - n) al[n + lane] = (uint16_t)NI;
            }
        }
        __syncthreads();
        // ---- B: neurons, and the next step's words
        if (tid < NT) {
#pragma unroll
            for (int k = 0; k < IPT; ++k) {
                if (ib[k] < 0) continue;
                const int b = ib[k], jl = ij[k];
                const int n = s_live[b] ? nact[b] : 0;
                const uint16_t* al = act + b * g.astr;     // (8-byte rows)
                float I = 0.0f;
#pragma unroll 1
                for (int a = 0; a < n; a += 4) {           // four rows in flight, added in order; the last group
                    const uint2 r4 = *reinterpret_cast<const uint2*>(al + a);   // padded (the sum is never -0)
                    const int r[4] = {(int)(r4.x & 0xFFFFu), (int)(r4.x >> 16), (int)(r4.y & 0xFFFFu), (int)(r4.y >> 16)};
                    float w[4];
#pragma unroll
                    for (int z = 0; z < 4; ++z) w[z] = Ws[r[z] * ncc + jl];
#pragma unroll
                    for (int z = 0; z < 4; ++z) I = __fadd_rn(I, c.wprec == SNN_W_BF16 ? w_read_bf16(w[z]) : w[z]);
                }
                st[k] = pair_update(c, v[k], vi[k], st[k], I, (int)cnt[pp * B + b], thj[jl]);
                const bool se = (st[k] & ST_SE) != 0u, si = (st[k] & ST_SI) != 0u;
                x[k] = __fadd_rn(__fmul_rn(x[k], c.a_x), se ? 1.0f : 0.0f);
                Es[b * ncc + jl] = __fmul_rn(c.nu_pre, x[k]);
                if (se) {
                    ++ns[k];
                    atomicOr(&Q[jl], 1u << b);
                }
                if (si)
#pragma unroll 1
                    for (int r = 0; r < CS; ++r)
                        red_cluster_add(tc::cluster_map(tc::su32(cnt + p3 * B + b), (uint32_t)r), 1u);
                if (c.rec_raster && (se || si)) {
                    const size_t o = ((size_t)t * B + b) * c.Nw + ((j0 + jl) >> 5);
                    const uint32_t bit = 1u << ((j0 + jl) & 31);
                    if (se) atomicOr(&d.raster_e[o], bit);
                    if (si) atomicOr(&d.raster_i[o], bit);
                }
            }
        } else if (t + 1 < T) {
            draw(t + 1, warp - NT / 32, (ST - NT) / 32);
        }
        cluster_arrive();
        __syncthreads();
        // ---- C: thresholds, and the update of each warp's 32 input rows
#pragma unroll 1
        for (int jl = ST - 1 - tid; jl < nc; jl += ST) {   // (the last warps: the first have rows)
            const int n = __popc(Q[jl]);
            double r;
            if (c.reduce == SNN_REDUCE_SUM) r = (double)n;
            else if (c.reduce == SNN_REDUCE_MEAN)          // n / B; exactly n * 2^-k for B = 2^k
                r = c.B_pow2 ? __dmul_rn((double)n, (double)c.inv_B) : divide((double)n, (double)c.B);
            else r = n > 0 ? 1.0 : 0.0;
            thS[jl] = __dadd_rn(__dmul_rn(thS[jl], c.a_th), __dmul_rn(c.theta_plus, r));
            thj[jl] = __fadd_rn(c.e_thresh, __double2float_rn(thS[jl]));
        }
#pragma unroll 1
        for (int jl = tid; jl < ncc; jl += ST) Qm[((t + 1) & 1) * ncc + jl] = 0u;
        const uint32_t all = B < 32 ? (1u << B) - 1u : FULL;
#pragma unroll 1
        for (int i0 = warp * 32; i0 < NI; i0 += SW * 32) {
            const int i = i0 + lane;
            const uint32_t mine = i < NI ? rowm[i] : 0u;   // this lane's row
            uint32_t rows = __ballot_sync(FULL, mine != 0u);
#pragma unroll 1
            for (int jc = 0; jc < nc; jc += 32) {
                const int jl = jc + lane;
                const uint32_t q = jl < nc ? Q[jl] : 0u;
                // columns without a post spike, lanes = columns: the rows that fired,
                // two a turn (past the last: no sample, no store)
#pragma unroll 1
                for (uint32_t rr = rows; rr;) {
                    int r[2];
                    uint32_t m[2], left = 0u;
                    float D[2];
#pragma unroll
                    for (int z = 0; z < 2; ++z) {
                        r[z] = rr ? __ffs(rr) - 1 : -1;
                        rr &= rr - 1;
                        m[z] = __shfl_sync(FULL, mine, r[z] & 31);
                        if (r[z] < 0) m[z] = 0u;
                        left |= m[z];
                        D[z] = MAX ? -FLT_MAX : 0.0f;
                    }
                    if (jl >= nc || q != 0u) continue;
                    float* const wp = Ws + i0 * ncc + jl;
                    float w[2];
#pragma unroll
                    for (int z = 0; z < 2; ++z) w[z] = wp[(r[z] < 0 ? 0 : r[z]) * ncc];
                    uint32_t y[2] = {m[0], m[1]};
#pragma unroll 1
                    while (left) {
                        left = 0u;
#pragma unroll
                        for (int z = 0; z < 2; ++z) {      // (a row without samples left reads the zero row)
                            const float e = Es[(y[z] ? __ffs(y[z]) - 1 : B) * ncc + jl];
                            if (!MAX) D[z] = __fadd_rn(D[z], e);
                            else if (y[z]) D[z] = fmaxf(D[z], __fsub_rn(0.0f, e));
                            y[z] &= y[z] - 1;
                            left |= y[z];
                        }
                    }
#pragma unroll
                    for (int z = 0; z < 2; ++z) {
                        if (r[z] < 0) break;
                        if (!MAX) {
                            D[z] = __fsub_rn(0.0f, D[z]);
                            if (c.reduce == SNN_REDUCE_MEAN) D[z] = mean_of(c, D[z]);
                        } else if (m[z] != all) {
                            D[z] = fmaxf(D[z], 0.0f);      // idle samples add 0
                        }
                        wp[r[z] * ncc] = plain_add(w[z], D[z], c.w_min, c.w_max);
                    }
                }
                // columns with one, lanes = rows
#pragma unroll 1
                for (uint32_t pc = __ballot_sync(FULL, q != 0u); pc; pc &= pc - 1) {
                    const int jq = __ffs(pc) - 1;
                    const uint32_t qm = __shfl_sync(FULL, q, jq);
                    if (i >= NI) continue;
                    float pot = MAX ? -FLT_MAX : 0.0f, dep = 0.0f;
#pragma unroll 1
                    for (uint32_t z = qm; z; z &= z - 1) {
                        const int b = __ffs(z) - 1;
                        const float a = __fmul_rn(c.nu_post, xs[b * NI + i]);
                        if (MAX) pot = fmaxf(pot, __fsub_rn(a, (mine >> b) & 1u ? Es[b * ncc + jc + jq] : 0.0f));
                        else pot = __fadd_rn(pot, a);
                    }
#pragma unroll 1
                    for (uint32_t z = MAX ? mine & ~qm : mine; z; z &= z - 1) {
                        const float e = Es[(__ffs(z) - 1) * ncc + jc + jq];
                        if (MAX) pot = fmaxf(pot, __fsub_rn(0.0f, e));
                        else dep = __fadd_rn(dep, e);
                    }
                    float D = MAX ? pot : __fsub_rn(pot, dep);
                    if (c.reduce == SNN_REDUCE_MEAN) D = mean_of(c, D);
                    if (MAX && (mine | qm) != all) D = fmaxf(D, 0.0f);
                    float* w = Ws + i * ncc + jc + jq;
                    *w = plain_add(*w, D, c.w_min, c.w_max);
                }
            }
            if (i < NI) rowm[i] = 0u;
        }
        cluster_wait();                                    // (every CTA is past its part B)
        __syncthreads();                                   // and this one past its part C
    }

    // ---- everything back
#pragma unroll 1
    for (int k = tid; k < NI * nc; k += ST) {
        const int i = k / nc, jl = k - i * nc;
        d.W[(size_t)i * N + j0 + jl] = Ws[i * ncc + jl];
    }
#pragma unroll 1
    for (int jl = tid; jl < nc; jl += ST) d.theta[j0 + jl] = thS[jl];
#pragma unroll
    for (int k = 0; k < IPT; ++k) {
        if (ib[k] < 0) continue;
        const size_t o = (size_t)ib[k] * N + j0 + ij[k];
        d.v_e[o] = v[k];
        d.v_i[o] = vi[k];
        d.x_post[o] = x[k];
        d.st[o] = st[k];
        if (ns[k]) {
            d.counts[o] += ns[k];
            atomicOr(&d.spkT[(size_t)(j0 + ij[k]) * c.Bw], 1u << ib[k]);   // (B <= 32: one word)
        }
    }
    float* x_out = d.x_pre + (size_t)(last % XPRE_SLOTS) * nbi;
#pragma unroll 1
    for (int b = rank; b < B; b += CS)
#pragma unroll 1
        for (int i = tid; i < NI; i += ST) x_out[(size_t)b * NI + i] = xs[b * NI + i];
    if (rank == 0)
#pragma unroll 1
        for (int b = tid; b < B; b += ST) d.cnt[(size_t)(last % 3ull) * B + b] = cnt[(size_t)(last % 3ull) * B + b];
}

SmallGeom small_geom(const Consts& c, int CS) {
    SmallGeom g{};
    g.CS = CS;
    g.ncc = (c.N + CS - 1) / CS;
    size_t o = 0;
    auto take = [&](size_t bytes) { const size_t at = o; o = (o + bytes + 15) & ~(size_t)15; return at; };
    g.astr = (c.n_in + 7) & ~3;           // a list and its padding, whole groups of four
    take((size_t)(c.n_in + 1) * g.ncc * 4);
    g.o_x = take((size_t)c.B * c.n_in * 4);
    g.o_es = take((size_t)(c.B + 1) * g.ncc * 4);
    g.o_words = take((size_t)2 * c.B * c.Iw * 4);
    g.o_tab = take((size_t)c.B * c.Iw * 4);
    g.o_wofs = take((size_t)(c.B + 1) * 4);
    g.o_act = take((size_t)c.B * g.astr * 2);
    g.o_idx = take((size_t)c.B * c.n_in * 2);
    const size_t own = ((size_t)c.B * c.Iw + CS - 1) / CS * 32;   // lanes of the words a CTA draws
    g.o_othr = take(own * 4);
    g.o_oidx = take(own * 2);
    g.o_rowm = take((size_t)c.n_in * 4);
    g.o_q = take((size_t)2 * g.ncc * 4);
    g.o_cnt = take((size_t)4 * c.B * 4);
    g.o_th = take((size_t)g.ncc * 12);
    g.smem = o;
    return g;
}

}  // namespace

cudaError_t launch_small(const Consts& c, const Bufs& d, int T, cudaStream_t s, int* used) {
    *used = 0;
    if (!c.learn || c.test_timeout || c.rule != SNN_RULE_PAIR || c.wmaster != SNN_WMASTER_FP32 ||
        c.wprec == SNN_W_FP8E4M3 || c.B > 32 || c.n_in > 65534)
        return cudaSuccess;
    // Few samples: half of the threads and the narrowest cluster whose CTAs keep
    // a column per lane: a block barrier costs 212 cycles with 16 warps and 317
    // with 32, the cluster barrier with its stores 865 with 8 CTAs and 1140 to
    // 1240 with 16 (784->100, B = 1: 1024 threads and 16 CTAs 746 us a run of 250
    // steps, 512 and 8 629, 256 and 4 709; 784->400, B = 16: 1024 threads 1441,
    // 512 1915).  Above ITEMS items a CTA the column kernel is faster (us a step there
    // and here, 1000 columns of 100 inputs: B = 4 9.9 and 6.7, B = 8 10.8 and 11.7).
    // Without lateral inhibition the columns fire in bursts, and each that fired costs a
    // warp a pass over its rows, with a division each where the mean takes one: fewer items (100 inputs of 120 Hz: 100->
    // 224, B = 32 9.2 and 10.5, 100->6400, B = 1 9.6 and 12.2, 100->280, B = 24 10.3 and
    // 12.8, 100->144, B = 24 10.3 and 10.8; but 100->100, B = 32 9.1 and 8.8, 100->4000, B
    // = 1 9.3 and 7.8, 100->100, B = 17 10.2 and 9.0).  With inhibition, dense inputs cost
    // the rows' passes too: 784->448, B = 16 at 1 and 6 % active 9.3 and 6.4, 15.8 and 19.8.
    constexpr size_t SMEM = 224 * 1024;
    const bool inhibition = c.w_ei != 0.0f && c.w_ie != 0.0f;
    const bool divides = c.reduce == SNN_REDUCE_MEAN && !c.B_pow2;
    const int ITEMS = inhibition ? 448 : divides && c.B > 16 ? 168 : 288;
    const bool few = c.B <= 4;
    using Kern = void (*)(Consts, Bufs, SmallGeom, int);
    static const Kern kerns[3][2] = {{k_small<1024, 1, false>, k_small<1024, 1, true>},
                                     {k_small<512, 1, false>, k_small<512, 1, true>},
                                     {k_small<512, 2, false>, k_small<512, 2, true>}};
    // The attributes, and whether the device places a cluster of 16 (the portable
    // size is 8), once per device: threads of a process share them under a lock.
    static int widest[64] = {0};
    static std::mutex mu;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    cudaLaunchConfig_t cfg{};
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    {
        std::lock_guard<std::mutex> lock(mu);
        if (widest[dev] == 0) {
            for (const auto& kr : kerns)
                for (const Kern k : kr) {
                    e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM);
                    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
                    if (e != cudaSuccess) return e;
                }
            cfg.blockDim = dim3(1024);
            cfg.gridDim = dim3(16);
            at[0].val.clusterDim.x = 16;
            cfg.dynamicSmemBytes = SMEM;
            int n = 0;
            if (cudaOccupancyMaxActiveClusters(&n, kerns[0][0], &cfg) != cudaSuccess) cudaGetLastError();
            widest[dev] = n > 0 ? 16 : 8;
        }
    }
    SmallGeom g{};
    for (int cs = few ? 8 : widest[dev]; cs <= widest[dev]; cs *= 2) {
        const SmallGeom t = small_geom(c, cs);
        if (t.smem > SMEM || c.B * t.ncc > ITEMS) continue;
        g = t;
        if (t.ncc <= 32) break;
    }
    // A run's start costs more here (a few CTAs load the weights and list the live inputs,
    // a word after the other), which some steps repay: us a run, there and here, at T = 1,
    // 3 and 10: 784->100, B = 1 37 / 43, 51 / 46, 104 / 57; 784->1000, B = 1 43 / 71, 61 /
    // 75, 134 / 91; 784->400, B = 16 40 / 53, 56 / 62, 117 / 102; 3000->50, B = 4 45 / 92,
    // 76 / 118, 181 / 183; 100->4000, B = 1 38 / 52, 54 / 62, 112 / 100.
    if (g.CS == 0 || T < 4 + (c.Iw + g.ncc) / 16) return cudaSuccess;
    cfg.blockDim = dim3(few ? 512 : 1024);                 // half of them neuron threads
    cfg.gridDim = dim3(g.CS);
    at[0].val.clusterDim.x = g.CS;
    cfg.dynamicSmemBytes = g.smem;
    *used = 1;
    return cudaLaunchKernelEx(&cfg, kerns[!few ? 0 : c.B * g.ncc <= 256 ? 1 : 2][c.reduce == SNN_REDUCE_MAX], c, d, g, T);
}

}  // namespace snn

// Learning-off runs of the persistent mode: a CTA per sample, all steps in one
// launch (see snn_sample.cuh).  The column-partitioned kernel crosses a grid
// barrier every step for the input lists and the inhibitory counts, which no
// other sample needs when nothing learns.  Us a step there and here: 784->400
// at B = 1, 256 and 1024: 6.0, 8.0, 14.4 and 1.3, 1.9, 5.9; 784->1600 at B = 256
// 9.2 and 4.8; 100->4000 at B = 1024 61 and 25.
#include "snn_sample.cuh"

namespace snn {

cudaError_t launch_colscale(const Consts& c, const Bufs& d, cudaStream_t s);   // snn_step.cu

namespace {

template <int NPT>
__global__ void __launch_bounds__(1024, 1) k_infer(const __grid_constant__ Consts c, const __grid_constant__ Bufs d,
                                                   const int T) {
    extern __shared__ __align__(16) unsigned char ism[];
    if (*reinterpret_cast<volatile uint32_t*>(d.err) != 0u) return;   // an earlier run failed: do nothing
    const int b = blockIdx.x, B = c.B;
    const unsigned long long base = d.step[0], last = base + (unsigned long long)T - 1ull;
    const size_t bn = (size_t)b * c.N, bi = (size_t)b * c.n_in, nbi = (size_t)B * c.n_in;
    SampleIO io;
    io.W = d.W;
    io.theta = d.theta;
    io.wscale = d.wscale;
    io.thr = d.thr + bi;
    io.seed = d.seeds[b];
    io.v_e = d.v_e + bn;
    io.v_i = d.v_i + bn;
    io.x_post = d.x_post + bn;
    io.st = d.st + bn;
    io.counts = d.counts + bn;
    io.x_in = d.x_pre + (size_t)((base + XPRE_SLOTS - 1) % XPRE_SLOTS) * nbi + bi;
    io.x_out = d.x_pre + (size_t)(last % XPRE_SLOTS) * nbi + bi;
    io.raster_e = d.raster_e + (size_t)b * c.Nw;
    io.raster_i = d.raster_i + (size_t)b * c.Nw;
    io.raster_in = d.raster_in + (size_t)b * c.Iw;
    io.rs_n = (size_t)B * c.Nw;
    io.rs_i = (size_t)B * c.Iw;
    const int C = run_sample<NPT, true>(c, io, base, T, (int)d.cnt[(size_t)((base + 2ull) % 3ull) * B + b], ism);
    if (threadIdx.x == 0) d.cnt[(size_t)(last % 3ull) * B + b] = (uint32_t)C;
    for (int j = threadIdx.x; j < c.N; j += blockDim.x)    // (each thread's own writes above)
        if (d.counts[bn + j]) atomicOr(&d.spkT[(size_t)j * c.Bw + (b >> 5)], 1u << (b & 31));
}

}  // namespace

cudaError_t launch_infer(const Consts& c, const Bufs& d, int T, cudaStream_t s, int* used) {
    *used = 0;
    const int npt = sample_npt(c.N);
    // Above 4096 neurons a CTA's step takes as long as the column kernel's of a whole
    // batch until the samples fill the SMs, one each, and a second wave doubles its time:
    // from 64 samples, and with a last wave at least five eighths full (784->6400, us a
    // step there and here: B = 16, 64, 128, 160 and 256 7.0 / 7.5, 8.6 / 7.8, 11.2 / 8.0,
    // 12.3 / 13.9, 15.3 / 14.7).  Not FP8, whose decoding is repeated by every sample
    // (B = 256: 18.8 and 34).
    // The weight rows come from L2 for each sample, so dense inputs favour the column
    // kernel, more so the wider the layer.  The figures above and those in the header
    // are at image rates (1 % of the inputs active); with an eighth active: 784->1000
    // still faster at every B, 784->3000 B = 1 12.9 / 21.7, B = 64 31.4 / 22.3, 784->6400
    // B = 64 and 128 27.8 / 40.9, 41.3 / 41.1.  The rates are on the device, so the rule
    // does not look at them.
    if (npt == 8) {
        int dev = 0, sms = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        const bool short_wave = c.B > sms && 8 * ((c.B - 1) % sms + 1) < 5 * sms;
        if (c.B < 64 || short_wave || c.wprec == SNN_W_FP8E4M3) return cudaSuccess;
    }
    const size_t smem = sample_smem(c.n_in, c.Iw, true, c.rec_input != 0).bytes;
    if (c.learn || c.test_timeout || npt == 0 || c.n_in > 65535 || smem > 200 * 1024) return cudaSuccess;
    cudaError_t e;
    if (c.wprec == SNN_W_FP8E4M3 && (e = launch_colscale(c, d, s)) != cudaSuccess) return e;
    auto kern = npt == 1 ? k_infer<1> : npt == 2 ? k_infer<2> : npt == 4 ? k_infer<4> : k_infer<8>;
    if (smem > SAMPLE_SMEM_DEFAULT) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
        if (e != cudaSuccess) return e;
    }
    kern<<<c.B, sample_threads(c.N, npt), smem, s>>>(c, d, T);
    *used = 1;
    return cudaGetLastError();
}

}  // namespace snn

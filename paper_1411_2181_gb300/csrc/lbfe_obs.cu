// lbfe_obs.cu -- droplet diagnostics (Sec. 1 and Sec. 3: deformation,
// orientation, projected length, necking and break-up).
//
// One pass over the populations of an instance computes, per x-plane, the
// integer sums over the droplet cells (rho_A > rho_B) of 1, y, z, y^2, z^2
// and yz, and the FP64 component masses.  Membership is decided on
// single-precision densities summed in population order.  The host turns
// the per-plane sums into the centroid, the second-moment tensor, D, theta,
// L_p, necks and break-up.
//
// Bound by reading the populations once.  A block takes 32 x-planes, a lane
// one of them: the sums over the rows its warps visit stay in registers, and
// meet in shared memory once per block, then in global memory by 64-bit
// integer atomics (exact and order-free).  Masses are added in a fixed order
// (rows of a thread, lanes, warps, then blocks by the last block to finish),
// which also completes the record the host reads with one copy:
//   [6 Lx] sums, mass A, mass B (FP64 bits), status word, finished blocks.
// Measured on 192 x 96 x 80 in FP32, call to result: 256 us with one block
// per row of x-planes, shared-memory sums in the loop, a one-thread sum of
// the masses and three copies; 71 to 76 us now, about 50 us of it this kernel
// (floor 33 us).
#include "lbfe_internal.cuh"

namespace lbfe {

constexpr int kObsThreads = 256;
constexpr int kObsWarps = kObsThreads / 32;

template <typename T>
__global__ void __launch_bounds__(kObsThreads)
k_obs(const __grid_constant__ InstDev I, int cur, unsigned *status) {
    const int Lx = I.Lx, Ly = I.Ly;
    const T *f = (const T *)I.f[cur];
    const long long S = I.S;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int x = blockIdx.x * 32 + lane;
    double mA = 0.0, mB = 0.0;
    unsigned long long sum[6] = {0, 0, 0, 0, 0, 0};
    bool bad = false;
    const int rows = Ly * I.Lz;
    for (int row = blockIdx.y * kObsWarps + warp; row < rows; row += gridDim.y * kObsWarps) {
        const long long n = (long long)row * Lx + min(x, Lx - 1);
        const float2 od = offset_dens<T>(I, cur, n);
        float va[Q], vb[Q];
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            va[i] = Store<T>::ld(f + (long long)i * S + n);
            vb[i] = Store<T>::ld(f + (long long)(Q + i) * S + n);
        }
        // every load is issued before the first sum: left alone, the compiler
        // keeps two or three in flight and the kernel reads at 1.4 TB/s
        __syncwarp();
        float ra = 0.f, rb = 0.f;
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            if (Store<T>::offset) { va[i] += wq(i) * od.x; vb[i] += wq(i) * od.y; }
            ra += va[i];
            rb += vb[i];
        }
        if (x >= Lx) continue;
        mA += (double)ra;
        mB += (double)rb;
        bad |= (ra != ra) || (rb != rb);
        if (ra > rb) {
            const unsigned y = (unsigned)(row % Ly), z = (unsigned)(row / Ly);   // below 2^16
            sum[0] += 1;
            sum[1] += y;
            sum[2] += z;
            sum[3] += y * y;
            sum[4] += z * z;
            sum[5] += y * z;
        }
    }
    if (bad) raise_flag(status, I, kFlagDiverged);
    __shared__ unsigned long long sh[6][kObsWarps][32];
    __shared__ double red[2][kObsThreads];
    __shared__ bool last;
#pragma unroll
    for (int q = 0; q < 6; ++q) sh[q][warp][lane] = sum[q];
    red[0][threadIdx.x] = mA;
    red[1][threadIdx.x] = mB;
    __syncthreads();
    if (threadIdx.x < 6 * 32) {
        unsigned long long s = 0;
#pragma unroll
        for (int w = 0; w < kObsWarps; ++w) s += sh[warp][w][lane];
        if (s) atomicAdd(I.prof + warp * Lx + x, s);
    }
    auto tree = [&]() {
        for (int s = kObsThreads / 2; s > 0; s >>= 1) {
            if ((int)threadIdx.x < s) {
                red[0][threadIdx.x] += red[0][threadIdx.x + s];
                red[1][threadIdx.x] += red[1][threadIdx.x + s];
            }
            __syncthreads();
        }
    };
    tree();
    const int blocks = gridDim.x * gridDim.y, block = blockIdx.y * gridDim.x + blockIdx.x;
    unsigned long long *tail = I.prof + 6 * (long long)Lx;
    if (threadIdx.x == 0) {
        I.mpart[block] = red[0][0];
        I.mpart[kObsBlocks + block] = red[1][0];
        __threadfence();
        last = atomicAdd((unsigned *)(tail + 3), 1u) == (unsigned)blocks - 1;
        __threadfence();
    }
    __syncthreads();
    if (!last) return;
    mA = mB = 0.0;
    for (int q = threadIdx.x; q < blocks; q += kObsThreads) {
        mA += __ldcg(I.mpart + q);
        mB += __ldcg(I.mpart + kObsBlocks + q);
    }
    red[0][threadIdx.x] = mA;
    red[1][threadIdx.x] = mB;
    __syncthreads();
    tree();
    if (threadIdx.x == 0) {
        tail[0] = (unsigned long long)__double_as_longlong(red[0][0]);
        tail[1] = (unsigned long long)__double_as_longlong(red[1][0]);
        tail[2] = __ldcg(I.status ? I.status : status);
    }
}

// The record of instance I into I.prof (obs_words(Lx) words).
cudaError_t launch_observables(const InstDev &I, int precision, int cur, unsigned *status, cudaStream_t stream) {
    cudaError_t e = cudaMemsetAsync(I.prof, 0, sizeof(unsigned long long) * obs_words(I.Lx), stream);
    if (e != cudaSuccess) return e;
    const int tiles = (I.Lx + 31) / 32;
    // blocks of eight rows at a time, three blocks on an SM
    const long long rows = (long long)I.Ly * I.Lz;
    const long long most = kObsBlocks / tiles, want = (rows + kObsWarps - 1) / kObsWarps;
    const dim3 grid((unsigned)tiles, (unsigned)(want < most ? want : most));
    switch (precision) {
        case LBFE_FP16_OFFSET: k_obs<__half><<<grid, kObsThreads, 0, stream>>>(I, cur, status); break;
        case LBFE_BF16_OFFSET: k_obs<__nv_bfloat16><<<grid, kObsThreads, 0, stream>>>(I, cur, status); break;
        default: k_obs<float><<<grid, kObsThreads, 0, stream>>>(I, cur, status);
    }
    return cudaGetLastError();
}

}  // namespace lbfe

// Binning entropy estimate of a layer's activations (Bi-GCN Sec. 6.2): per neuron (column) the range
// over the N samples (rows), an M-interval histogram over that range, H_hat = -sum p log2 p, and the
// independent sum over the neurons.  Two streaming passes over the N x d matrix (range, histogram),
// both bound by HBM reads; the histogram of a strip of columns lives in shared memory.
#include <algorithm>

#include "bigcn_internal.cuh"

namespace bigcn {

namespace {

constexpr int kEntThreads = 256;
constexpr int kEntWarps = kEntThreads / kWarp;

// Order-preserving map from float to unsigned (so that integer atomicMin / atomicMax order floats).
__device__ __forceinline__ uint32_t float_key(float x)
{
    const uint32_t b = __float_as_uint(x);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float key_float(uint32_t k)
{
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

// Pass 1.  Block (x, y) scans its share of the rows for columns 32 y .. 32 y + 31: lane = column, the
// warps of a block take rows in turn (each warp load is 128 contiguous bytes), four rows in flight per
// warp.  One atomicMin and one atomicMax per column and block on the order-preserving keys.
__global__ void __launch_bounds__(kEntThreads)
range_kernel(const float* __restrict__ H, int64_t n, int d, int64_t ld, int64_t rows_per_block,
             uint32_t* __restrict__ key_min, uint32_t* __restrict__ key_max)
{
    pdl_enter();
    __shared__ float s_lo[kEntWarps][kWarp], s_hi[kEntWarps][kWarp];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int col = blockIdx.y * 32 + lane;
    const int64_t r0 = (int64_t)blockIdx.x * rows_per_block;
    const int64_t r1 = min(n, r0 + rows_per_block);
    float lo = INFINITY, hi = -INFINITY;
    if (col < d) {
        int64_t r = r0 + warp;
        for (; r + 3 * kEntWarps < r1; r += 4 * kEntWarps) {
            float x[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) x[u] = __ldg(H + (r + u * kEntWarps) * ld + col);
#pragma unroll
            for (int u = 0; u < 4; ++u) { lo = fminf(lo, x[u]); hi = fmaxf(hi, x[u]); }
        }
        for (; r < r1; r += kEntWarps) {
            const float x = __ldg(H + r * ld + col);
            lo = fminf(lo, x);
            hi = fmaxf(hi, x);
        }
    }
    s_lo[warp][lane] = lo;
    s_hi[warp][lane] = hi;
    __syncthreads();
    if (warp == 0 && col < d) {
#pragma unroll
        for (int w = 1; w < kEntWarps; ++w) { lo = fminf(lo, s_lo[w][lane]); hi = fmaxf(hi, s_hi[w][lane]); }
        if (lo <= hi) {                                   // the block saw at least one row
            atomicMin(key_min + col, float_key(lo));
            atomicMax(key_max + col, float_key(hi));
        }
    }
}

// Before pass 1: keys that every value replaces, zero counters, and a zero where the last block of entropy_kernel counts.
__global__ void __launch_bounds__(kEntThreads)
init_kernel(uint32_t* __restrict__ key_min, uint32_t* __restrict__ key_max, int d, uint32_t* __restrict__ counts, int64_t n_counts,
            double* __restrict__ total)
{
    pdl_enter();
    const int64_t i0 = (int64_t)blockIdx.x * kEntThreads + threadIdx.x, step = (int64_t)gridDim.x * kEntThreads;
    for (int64_t i = i0; i < n_counts; i += step) counts[i] = 0u;
    for (int64_t i = i0; i < d; i += step) {
        key_min[i] = 0xffffffffu;
        key_max[i] = 0u;
    }
    if (i0 == 0) *total = 0.0;
}

// Pass 2.  Block (x, y) histograms its share of the rows for the strip of CW columns CW y ..: a warp
// instruction covers 32 / CW rows x CW columns (CW * 4 contiguous bytes per row); the strip's M x CW
// counters sit in shared memory and are added to the global ones once per block.  The counters of a column stay in
// the 32 / CW banks of its own.  (With the counters of a column contiguous the atomic adds of a warp met in random banks,
// about 3.5 of 32 in the fullest, and that bounded the pass: 0.49 ms for 2.4 M x 128 values and 1,000 intervals, now
// 0.25 ms; reading them takes 0.19 ms.)  The rows are taken from the
// last to the first, because pass 1 has just left the last ones of every share in the L2.  The interval of a
// value is decided in fp32 exactly as documented for the entry point: (x - min) * (M / (max - min)),
// truncated, clamped to M - 1; a constant column has scale 0 and lands in interval 0.
constexpr int kHistThreads = 1024;
template <int CW>
__global__ void __launch_bounds__(kHistThreads, 1)
histogram_kernel(const float* __restrict__ H, int64_t n, int d, int64_t ld, int n_bins, int64_t rows_per_block,
                 const uint32_t* __restrict__ key_min, const uint32_t* __restrict__ key_max,
                 float* __restrict__ col_min, float* __restrict__ col_max, uint32_t* __restrict__ counts)
{
    pdl_enter();
    extern __shared__ uint32_t hist[];                    // [n_bins][CW]
    constexpr int RPW = kWarp / CW;                       // rows per warp instruction
    constexpr int RPB = RPW * (kHistThreads / kWarp);     // rows per block step
    constexpr int U = 8;                                  // loads in flight per thread
    for (int i = threadIdx.x; i < CW * n_bins; i += kHistThreads) hist[i] = 0u;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int cl = lane % CW;                             // column inside the strip
    const int col = blockIdx.y * CW + cl;
    const bool col_in = col < d;
    float lo = 0.f, scale = 0.f;
    if (col_in) {
        lo = key_float(key_min[col]);
        const float hi = key_float(key_max[col]);
        scale = hi > lo ? __fdiv_rn((float)n_bins, __fsub_rn(hi, lo)) : 0.f;
        if (blockIdx.x == 0 && threadIdx.x < CW) { col_min[col] = lo; col_max[col] = hi; }
    }
    __syncthreads();
    const int64_t r0 = (int64_t)blockIdx.x * rows_per_block;
    const int64_t r1 = min(n, r0 + rows_per_block);
    uint32_t* my = hist + cl;
    const int last = n_bins - 1;
    if (col_in) {
        int64_t r = r1 - 1 - (warp * RPW + lane / CW);
        const float* src = H + r * ld + col;
        for (; r - (U - 1) * RPB >= r0; r -= U * RPB, src -= (int64_t)U * RPB * ld) {
            float x[U];
#pragma unroll
            for (int u = 0; u < U; ++u) x[u] = __ldg(src - (int64_t)(u * RPB) * ld);
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int m = min((int)__fmul_rn(__fsub_rn(x[u], lo), scale), last);
                atomicAdd(my + m * CW, 1u);
            }
        }
        for (; r >= r0; r -= RPB, src -= (int64_t)RPB * ld) {
            const int m = min((int)__fmul_rn(__fsub_rn(__ldg(src), lo), scale), last);
            atomicAdd(my + m * CW, 1u);
        }
    }
    __syncthreads();
    if (col_in) {
        uint32_t* out = counts + (int64_t)col * n_bins;
        for (int m = warp * RPW + lane / CW; m < n_bins; m += RPB) {
            const uint32_t v = my[m * CW];
            if (v) atomicAdd(out + m, v);
        }
    }
}

// H_hat of one column per block, in double: threads take intervals t, t + 256, ... and the partial sums are combined in a
// fixed order.  (A warp per column left most of the chip idle: 30 us for 128 columns of 1,000 intervals.)  The block that
// finishes last (counted in the place of the total, which is 0 before) adds the columns up, in a fixed order too: H_ind.
__global__ void __launch_bounds__(kEntThreads)
entropy_kernel(const uint32_t* __restrict__ counts, int d, int n_bins, int64_t n, double* entropy, double* total)
{
    pdl_enter();
    __shared__ bool last_block;
    __shared__ double part[kEntWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t* c = counts + (int64_t)blockIdx.x * n_bins;
    const double inv_n = 1.0 / (double)n;
    double h = 0.0;
    for (int m = threadIdx.x; m < n_bins; m += kEntThreads) {
        const uint32_t v = c[m];
        if (v) {
            const double p = (double)v * inv_n;
            h -= p * log2(p);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) h += __shfl_xor_sync(0xffffffffu, h, o);
    if (lane == 0) part[warp] = h;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < kEntWarps; ++w) s += part[w];
        entropy[blockIdx.x] = s;
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) last_block = atomicAdd(reinterpret_cast<unsigned*>(total), 1u) == gridDim.x - 1;
    __syncthreads();
    if (last_block && threadIdx.x < kWarp) {
        __threadfence();
        double s = 0.0;
        for (int j = lane; j < d; j += 32) s += __ldcg(entropy + j);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) *total = s;
    }
}

template <int CW>
cudaError_t launch_histogram(cudaStream_t s, const float* H, int64_t n, int d, int64_t ld, int n_bins,
                             const uint32_t* key_min, const uint32_t* key_max, float* col_min, float* col_max,
                             uint32_t* counts)
{
    const size_t smem = (size_t)CW * n_bins * sizeof(uint32_t);
    cudaError_t e = cudaFuncSetAttribute(histogram_kernel<CW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const unsigned gy = (unsigned)ceil_div(d, CW);
    const int per_sm = smem > 112 * 1024 ? 1 : 2;
    // about one resident wave of blocks over both grid dimensions; every block takes a contiguous range of rows, at least
    // as many as it has counters to add up at the end
    const int64_t gx = std::max<int64_t>(1, std::min<int64_t>(ceil_div(n, std::max(1024, n_bins)), (int64_t)sm_count() * per_sm / gy));
    const int64_t rows_per_block = ceil_div(n, gx);
    launch_kernel(histogram_kernel<CW>, dim3((unsigned)gx, gy), kHistThreads, smem, s, H, n, d, ld, n_bins, rows_per_block, key_min,
                                                                         key_max, col_min, col_max, counts);
    return cudaGetLastError();
}

}  // namespace

size_t entropy_scratch_bytes(int d) { return 2 * (size_t)d * sizeof(uint32_t); }

int entropy_max_bins() { return 8192; }

cudaError_t launch_entropy_bins(cudaStream_t s, const float* H, int64_t n, int d, int64_t ld, int n_bins,
                                float* col_min, float* col_max, uint32_t* counts, double* entropy, double* total,
                                void* scratch, int* launches)
{
    uint32_t* key_min = static_cast<uint32_t*>(scratch);
    uint32_t* key_max = key_min + d;
    const int64_t n_counts = (int64_t)d * n_bins;
    launch_kernel(init_kernel, (unsigned)std::min<int64_t>(ceil_div(n_counts, kEntThreads * 4), (int64_t)sm_count() * 8), kEntThreads, 0, s, key_min, key_max, d, counts, n_counts, total);
    ++*launches;
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    {
        const unsigned gy = (unsigned)ceil_div(d, 32);
        const int64_t gx = std::max<int64_t>(1, std::min<int64_t>(ceil_div(n, 256), ceil_div((int64_t)sm_count() * 8, gy)));
        launch_kernel(range_kernel, dim3((unsigned)gx, gy), kEntThreads, 0, s, H, n, d, ld, ceil_div(n, gx), key_min, key_max);
        ++*launches;
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    // Strips of 16 columns where their counters fit a block's shared memory; of 8 where that leaves fewer lanes past the
    // last of up to 24 columns (beyond, the half as long row pieces cost more).  Strips of 32 have no two lanes in a bank, but
    // twice the counters to clear and to add up, which only the rows of a long matrix that is one such strip make up for.
    // All of the estimate, strips of 32 / 16 / 8: 2.4 M rows, 100 intervals, 8 columns 98 / 77 / 67 us, 24: 138 / 146 / 140, 31:
    // 156 / 171 / 181, 48: 251 / 230 / 258, 128: 452 / 450 / 486; 1,000 intervals, 24: 163 / 157 / 146, 31: 179 / 185 / 187, 128:
    // 469 / 460 / 492; 300,000 rows, 100 intervals, 8: 38 / 28 / 24, 24: 42 / 36 / 31, 48: 58 / 46 / 46, 128: 93 / 85 / 87.
    const bool one = d > 16 && d <= 32 && n >= (int64_t(1) << 20) && n_bins <= (d > 24 ? 1750 : 200);
    const bool narrow = d <= 24 && round_up(d, 8) < round_up(d, 16) && n_bins <= 1750;
    if (one) e = launch_histogram<32>(s, H, n, d, ld, n_bins, key_min, key_max, col_min, col_max, counts);
    else if (n_bins <= 3500 && !narrow) e = launch_histogram<16>(s, H, n, d, ld, n_bins, key_min, key_max, col_min, col_max, counts);
    else if (n_bins <= 7000) e = launch_histogram<8>(s, H, n, d, ld, n_bins, key_min, key_max, col_min, col_max, counts);
    else e = launch_histogram<4>(s, H, n, d, ld, n_bins, key_min, key_max, col_min, col_max, counts);
    ++*launches;
    if (e != cudaSuccess) return e;
    launch_kernel(entropy_kernel, (unsigned)d, kEntThreads, 0, s, counts, d, n_bins, n, entropy, total);
    ++*launches;
    return cudaGetLastError();
}

}  // namespace bigcn

// Back-propagation through one binarized graph convolutional layer (Bi-GCN Algorithm 1, Sec. 4.3):
//   G_zeta = A_tilde^T G'            (the aggregation kernel of the forward pass, fp32 rows)
//   G_W~   = H~^T G_zeta             H~_ik = beta_i F_ik from the packed input bits
//   G_H~   = G_zeta W~^T             W~_kj = alpha_j sign(W_kj)
//   G_H    = G_H~ [|G_H~| < 1]       (Eq. bp-H)
//   G_W_ij = (1/d_in) B_ij sum_k G_W~_kj B_kj + alpha_j G_W~_ij [|W_ij| < 1]   (Eq. bp-W)
// The two dense products have one +-1 operand that is expanded from bits (or from the sign of W) into
// shared memory tile by tile as bf16; the fp32 operand is split into three bf16 terms; the products run
// on the tensor cores with fp32 accumulation.
#include <algorithm>

#include <cuda_bf16.h>

#include "bigcn_internal.cuh"
#include "tc_common.cuh"

namespace bigcn {

namespace {

constexpr int kBwThreads = 256;       // 8 warps per block

// Copies rows of d floats into rows of ld_out floats (ld_out >= d, a multiple of 4), zero-filling the tail.
__global__ void pad_rows_kernel(const float* __restrict__ src, int64_t n, int d, int64_t ld_in,
                                float* __restrict__ dst, int64_t ld_out)
{
    pdl_enter();
    const int64_t total = n * ld_out;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = t / ld_out;
        const int j = (int)(t - i * ld_out);
        dst[t] = j < d ? __ldg(src + i * ld_in + j) : 0.f;
    }
}

// G_W~ = sum of the slabs (double accumulation: the slabs can differ by orders of magnitude), and for Eq. bp-W the sums
// sum_k G_W~_kj sign(W_kj) over four inputs k.  A block takes 32 channels x 4 inputs; of its 1,024 threads eight share
// an element and take every eighth slab each, eight loads in flight; their sums are added in order.  (One thread per element
// walked through all slabs alone: 15 to 28 us whatever the sizes.)
constexpr int kRedRows = 4, kRedGroups = 8;
__global__ void __launch_bounds__(32 * kRedRows * kRedGroups)
grad_wt_reduce_kernel(const float* __restrict__ part, int n_splits, int d_in, int d_out, const float* __restrict__ W, int64_t ldw,
                      float* __restrict__ g_wt, double* __restrict__ col_part /* [ceil(d_in / 4)][d_out] */)
{
    pdl_enter();
    __shared__ double s_sum[kRedGroups][kRedRows][33];
    const int tx = threadIdx.x & 31, r = (threadIdx.x >> 5) % kRedRows, zg = threadIdx.x / (32 * kRedRows);
    const int j = blockIdx.x * 32 + tx, k = blockIdx.y * kRedRows + r;
    const int64_t elems = (int64_t)d_in * d_out;
    double s = 0.0;
    if (j < d_out && k < d_in) {
        const float* src = part + (int64_t)k * d_out + j;
#pragma unroll 8
        for (int z = zg; z < n_splits; z += kRedGroups) s += (double)__ldg(src + z * elems);
    }
    s_sum[zg][r][tx] = s;
    __syncthreads();
    if (zg == 0) {
        for (int q = 1; q < kRedGroups; ++q) s += s_sum[q][r][tx];
        const float g = (float)s;
        double sg = 0.0;
        if (j < d_out && k < d_in) {
            g_wt[(int64_t)k * d_out + j] = g;
            sg = __ldg(W + (int64_t)k * ldw + j) >= 0.f ? (double)g : -(double)g;
        }
        s_sum[0][r][tx] = sg;
    }
    __syncthreads();
    if (threadIdx.x < 32 && j < d_out) {
        double c = 0.0;
        for (int q = 0; q < kRedRows; ++q) c += s_sum[0][q][tx];
        col_part[(int64_t)blockIdx.y * d_out + j] = c;
    }
}

// ---- the two dense products, on the tensor cores ------------------------------------------------------
// Both products have one operand that is exactly +-1 (exact in bf16) and one fp32 operand.  The fp32
// operand x is split into three bf16 terms x = hi + mid + lo (each the rounding of what is left:
// 3 x 8 significant bits cover fp32's 24), so three bf16 tensor-core products with fp32 accumulation
// reproduce the fp32 product to fp32 accuracy.  mma.sync m16n8k16 (row-major A, column-major B):
// with g = lane / 4, t = lane % 4 a thread holds A[g | g+8][2t, 2t+1 | +8], B[2t, 2t+1 | +8][g],
// C[g | g+8][2t, 2t+1].  Tiles are staged in shared memory as bf16 with a row pitch of 40 elements
// (20 words), which makes the fragment reads of a warp hit 32 different banks.
constexpr int kMmaPitch = 40;                    // bf16 elements per staged row (32 + 8 pad)
constexpr int kMmaTile = 128;                    // output tile 128 x 128 per block, 8 warps of 32 x 64
constexpr int kMmaK = 32;                        // reduction elements per staged step

__device__ __forceinline__ void split3(float x, unsigned short& hi, unsigned short& mid, unsigned short& lo)
{
    const __nv_bfloat16 h = __float2bfloat16_rn(x);
    const float r1 = __fsub_rn(x, __bfloat162float(h));
    const __nv_bfloat16 m = __float2bfloat16_rn(r1);
    const float r2 = __fsub_rn(r1, __bfloat162float(m));
    const __nv_bfloat16 l = __float2bfloat16_rn(r2);
    hi = __bfloat16_as_ushort(h);
    mid = __bfloat16_as_ushort(m);
    lo = __bfloat16_as_ushort(l);
}

__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], const uint32_t (&b)[2])
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// One staged step of the block's 128 x 128 tile: As[3][128][pitch] (the three terms of the fp32
// operand, rows = output rows, k contiguous), Bs[128][pitch] (the +-1 operand, rows = output columns,
// k contiguous).  Warp (wr, wc) owns rows 32 wr.., columns 64 wc...
__device__ __forceinline__ void mma_step(const unsigned short* As, const unsigned short* Bs, int wr, int wc, int lane,
                                         float (&acc)[2][8][4])
{
    const int g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int kk = 0; kk < kMmaK; kk += 16) {
        uint32_t b[8][2];
#pragma unroll
        for (int nb = 0; nb < 8; ++nb) {
            const unsigned short* p = Bs + (wc * 64 + nb * 8 + g) * kMmaPitch + kk + 2 * t;
            b[nb][0] = *reinterpret_cast<const uint32_t*>(p);
            b[nb][1] = *reinterpret_cast<const uint32_t*>(p + 8);
        }
#pragma unroll
        for (int sp = 0; sp < 3; ++sp) {
#pragma unroll
            for (int mb = 0; mb < 2; ++mb) {
                const unsigned short* p = As + (sp * kMmaTile + wr * 32 + mb * 16 + g) * kMmaPitch + kk + 2 * t;
                uint32_t a[4];
                a[0] = *reinterpret_cast<const uint32_t*>(p);
                a[1] = *reinterpret_cast<const uint32_t*>(p + 8 * kMmaPitch);
                a[2] = *reinterpret_cast<const uint32_t*>(p + 8);
                a[3] = *reinterpret_cast<const uint32_t*>(p + 8 * kMmaPitch + 8);
#pragma unroll
                for (int nb = 0; nb < 8; ++nb) mma_bf16(acc[mb][nb], a, b[nb]);
            }
        }
    }
}

// G_H = clip(G_zeta W~^T) on the tensor cores.  Block (x, y): rows [128 x, +128) x inputs k in
// [128 y, +128); the reduction runs over the output channels j in steps of 32.  A = G_zeta * alpha_j
// (split in three), B[k][j] = sign(W[k][j]).
__global__ void __launch_bounds__(kBwThreads)
grad_h_mma_kernel(const float* __restrict__ gz, int64_t ldz, const float* __restrict__ alpha,
                  const float* __restrict__ W, int64_t ldw, int64_t n, int d_in, int d_out,
                  float* __restrict__ g_h, int64_t ldh)
{
    pdl_enter();
    __shared__ __align__(16) unsigned short As[3 * kMmaTile * kMmaPitch];
    __shared__ __align__(16) unsigned short Bs[kMmaTile * kMmaPitch];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int wr = warp >> 1, wc = warp & 1;
    const int64_t i0 = (int64_t)blockIdx.x * kMmaTile;
    const int k0 = blockIdx.y * kMmaTile;
    const bool vec_ok = (ldz % 4 == 0) && (reinterpret_cast<uintptr_t>(gz) % 16 == 0);
    float acc[2][8][4];
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 8; ++b)
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[a][b][c] = 0.f;
    for (int j0 = 0; j0 < d_out; j0 += kMmaK) {
        __syncthreads();                                   // the previous step's tiles are consumed
        // stage 128 x 32 of each operand: a thread takes 4 consecutive j of one row (16-byte loads where the
        // row allows it) and writes 8 bytes per term
        for (int t = threadIdx.x; t < kMmaTile * (kMmaK / 4); t += kBwThreads) {
            const int jq = (t & 7) * 4, rr = t >> 3;
            const int j = j0 + jq;
            const int64_t row = i0 + rr;
            float x[4] = {0.f, 0.f, 0.f, 0.f};
            if (row < n) {
                if (j + 3 < d_out && vec_ok) {
                    const float4 v = __ldg(reinterpret_cast<const float4*>(gz + row * ldz + j));
                    x[0] = v.x, x[1] = v.y, x[2] = v.z, x[3] = v.w;
                } else {
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (j + q < d_out) x[q] = __ldg(gz + row * ldz + j + q);
                }
            }
            unsigned short hi[4], mid[4], lo[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) split3(j + q < d_out ? __fmul_rn(x[q], __ldg(alpha + j + q)) : 0.f, hi[q], mid[q], lo[q]);
            auto pack = [](const unsigned short (&h)[4]) { return make_uint2((uint32_t)h[0] | ((uint32_t)h[1] << 16), (uint32_t)h[2] | ((uint32_t)h[3] << 16)); };
            *reinterpret_cast<uint2*>(&As[(0 * kMmaTile + rr) * kMmaPitch + jq]) = pack(hi);
            *reinterpret_cast<uint2*>(&As[(1 * kMmaTile + rr) * kMmaPitch + jq]) = pack(mid);
            *reinterpret_cast<uint2*>(&As[(2 * kMmaTile + rr) * kMmaPitch + jq]) = pack(lo);
            const int k = k0 + rr;
            unsigned short sg[4] = {0, 0, 0, 0};
            if (k < d_in) {
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (j + q < d_out) sg[q] = __ldg(W + (int64_t)k * ldw + j + q) >= 0.f ? 0x3F80 : 0xBF80;
            }
            *reinterpret_cast<uint2*>(&Bs[rr * kMmaPitch + jq]) = pack(sg);
        }
        __syncthreads();
        mma_step(As, Bs, wr, wc, lane, acc);
    }
    const int g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int mb = 0; mb < 2; ++mb)
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            const int64_t row = i0 + wr * 32 + mb * 16 + g + 8 * half;
            if (row >= n) continue;
#pragma unroll
            for (int nb = 0; nb < 8; ++nb)
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const int k = k0 + wc * 64 + nb * 8 + 2 * t + q;
                    const float v = acc[mb][nb][2 * half + q];
                    if (k < d_in) g_h[row * ldh + k] = fabsf(v) < 1.f ? v : 0.f;            // Eq. bp-H
                }
        }
}

// ---- G_H on the 5th-generation tensor cores ---------------------------------------------------------------
// The same product as grad_h_mma_kernel with tcgen05.mma kind::f16 (bf16 operands, fp32 accumulators in tensor memory):
// M = 128 rows, N = 64 / 128 / 256 inputs (blockIdx.y: slices of N), the reduction over the output channels in chunks of 64.
// Both operands are K-major with 128-byte swizzle: 64 channels of a row are 128 contiguous bytes, so a warp reads and stages
// two whole row pieces without bank conflicts.  One block of 16 warps per multiprocessor.  The fp32 operand has two stages of
// its three terms: while one is multiplied the other is filled, and the chunk after that is on its way in registers; two
// accumulators, so that a tile is read back, clipped (Eq. bp-H) and written under the products of the next one.  The signs of
// W stay in shared memory for all tiles where all of their chunks fit (d_out <= 65536 / N); longer ones pass through
// two stages.  (One stage, the signs rebuilt for every chunk of every tile, stores that met in the banks eight at a time:
// 2.4 M nodes, 256 -> 256, 2.8 ms; now 1.37 ms.)
// Needs d_in a multiple of 4 and 16-byte aligned rows of g_h; every mbarrier wait is bounded.
__device__ int g_bw_tc_timeout;

constexpr int kGhThreads = 512, kGhRows = 128, kGhK = 64;
constexpr int kGhTerm = kGhRows * 128;                      // bytes of one term of a chunk
constexpr int kGhStage = 3 * kGhTerm;
__host__ __device__ constexpr int gh_slots(int n) { return 1024 / n; }         // chunks of signs that stay: 128 KB

template <int N>
__global__ void __launch_bounds__(kGhThreads, 1)
grad_h_tc_kernel(const float* __restrict__ gz, int64_t ldz, const float* __restrict__ alpha,
                 const float* __restrict__ W, int64_t ldw, int64_t n, int d_in, int d_out,
                 float* __restrict__ g_h, int64_t ldh)
{
    pdl_enter();
    constexpr int kBChunk = N * 128;
    constexpr int kItems = kGhRows * (kGhK / 4) / kGhThreads, kBItems = N * (kGhK / 4) / kGhThreads;
    constexpr int kCols = 2 * N;                            // two accumulators
    extern __shared__ unsigned char bw_raw[];
    __shared__ __align__(8) uint64_t bar[2];
    __shared__ uint32_t tmem_base_s;
    unsigned char* sm = bw_raw + ((1024u - (tc::smem_u32(bw_raw) & 1023u)) & 1023u);
    unsigned char* Bs = sm + 2 * kGhStage;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp == 0) tc::tmem_alloc(&tmem_base_s, kCols);
    if (threadIdx.x == 0) {
        tc::barrier_init(&bar[0]);
        tc::barrier_init(&bar[1]);
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem_base = tmem_base_s;
    // instruction descriptor: D = f32, A = B = bf16, both K-major, N, M = 128
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(kGhRows >> 4) << 24);
    const bool vec_ok = (ldz % 4 == 0) && (reinterpret_cast<uintptr_t>(gz) % 16 == 0);
    const bool w_vec_ok = (ldw % 4 == 0) && (reinterpret_cast<uintptr_t>(W) % 16 == 0);
    const int k0 = blockIdx.y * N;
    const int n_chunks = (d_out + kGhK - 1) / kGhK;
    const bool resident = n_chunks <= gh_slots(N);
    const int64_t n_tiles = ceil_div(n, kGhRows);
    const int64_t my_tiles = n_tiles > blockIdx.x ? (n_tiles - 1 - blockIdx.x) / gridDim.x + 1 : 0;
    const int64_t total = my_tiles * n_chunks;              // chunks of all tiles of this block, one after the other
    // this thread's pieces of a chunk: channels jq .. jq + 3 of rows threadIdx.x / 16 + 32 it, of both operands
    const int jq = (threadIdx.x & 15) * 4, r0 = threadIdx.x >> 4;
    const uint32_t off = (uint32_t)((r0 >> 3) * 1024 + (r0 & 7) * 128 + (((jq >> 3) ^ (r0 & 7)) << 4) + (jq & 7) * 2);   // + 4096 it
    auto load4 = [](const float* src, bool whole, int left) {                  // the first `left` of four floats
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (whole && left >= 4) return __ldg(reinterpret_cast<const float4*>(src));
        if (left > 0) v.x = __ldg(src);
        if (left > 1) v.y = __ldg(src + 1);
        if (left > 2) v.z = __ldg(src + 2);
        if (left > 3) v.w = __ldg(src + 3);
        return v;
    };
    float4 xv[kItems], av;
    auto load = [&](int64_t tile, int ch) {
        const int j = ch * kGhK + jq;
#pragma unroll
        for (int it = 0; it < kItems; ++it) {
            const int64_t row = tile * kGhRows + r0 + 32 * it;
            xv[it] = load4(gz + row * ldz + j, vec_ok, row < n ? d_out - j : 0);
        }
        av = load4(alpha + j, false, d_out - j);
    };
    auto wait = [&](int64_t c) {                            // until the products of chunk c are done
        const bool in_time = __all_sync(0xffffffffu, tc::wait_barrier(&bar[c & 1], (uint32_t)(c >> 1) & 1u));
        if (!in_time) atomicExch(&g_bw_tc_timeout, 1);
        return in_time;
    };
    // a finished tile: a thread owns row 32 (warp % 4) + lane, its warp a quarter of the columns, 16 at a time, which leave
    // as 64-byte pieces of rows through 2 KB of a free stage
    const int lane_base = 32 * (warp & 3), c_begin = (warp >> 2) * (N / 4);
    auto finish = [&](int64_t tile, int acc, unsigned char* scratch) {
        unsigned char* scr = scratch + warp * 2048;
        const int64_t row0 = tile * kGhRows + lane_base;
#pragma unroll 1
        for (int c0 = c_begin; c0 < c_begin + N / 4; c0 += 16) {
            uint32_t v[16];
            tc::tmem_ld16(tmem_base + ((uint32_t)lane_base << 16) + (uint32_t)(acc * N + c0), v);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                float f[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float g = __uint_as_float(v[4 * u + e]);
                    f[e] = fabsf(g) < 1.f ? g : 0.f;                                      // Eq. bp-H
                }
                *reinterpret_cast<float4*>(scr + lane * 64 + ((u ^ ((lane >> 1) & 3)) << 4)) = make_float4(f[0], f[1], f[2], f[3]);
            }
            __syncwarp();
#pragma unroll
            for (int it = 0; it < 4; ++it) {
                const int r = it * 8 + (lane >> 2), u = lane & 3;
                const float4 val = *reinterpret_cast<const float4*>(scr + r * 64 + ((u ^ ((r >> 1) & 3)) << 4));
                const int col = k0 + c0 + 4 * u;
                if (row0 + r < n && col < d_in) *reinterpret_cast<float4*>(g_h + (row0 + r) * ldh + col) = val;
            }
            __syncwarp();
        }
    };
    bool ok = true;
    int64_t tile = blockIdx.x;
    int ch = 0, acc = 0;
    if (total > 0) load(tile, 0);
    for (int64_t c = 0; c < total; ++c) {
        const int st = (int)(c & 1);
        unsigned char* stage = sm + st * kGhStage;
        unsigned char* signs = Bs + (resident ? ch : st) * kBChunk;
        if (c >= 2) ok = wait(c - 2) && ok;
        const float a4[4] = {av.x, av.y, av.z, av.w};
#pragma unroll
        for (int it = 0; it < kItems; ++it) {
            const float x[4] = {__fmul_rn(xv[it].x, a4[0]), __fmul_rn(xv[it].y, a4[1]), __fmul_rn(xv[it].z, a4[2]), __fmul_rn(xv[it].w, a4[3])};
            unsigned short hi[4], mid[4], lo[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) split3(x[u], hi[u], mid[u], lo[u]);
            auto pack = [](const unsigned short (&h)[4]) { return make_uint2((uint32_t)h[0] | ((uint32_t)h[1] << 16), (uint32_t)h[2] | ((uint32_t)h[3] << 16)); };
            *reinterpret_cast<uint2*>(stage + 0 * kGhTerm + off + 4096 * it) = pack(hi);
            *reinterpret_cast<uint2*>(stage + 1 * kGhTerm + off + 4096 * it) = pack(mid);
            *reinterpret_cast<uint2*>(stage + 2 * kGhTerm + off + 4096 * it) = pack(lo);
        }
        if (!resident || c < n_chunks) {
            const int j = ch * kGhK + jq;
#pragma unroll
            for (int it = 0; it < kBItems; ++it) {
                const int k = k0 + r0 + 32 * it;
                const int left = k < d_in ? d_out - j : 0;
                const float4 wv = load4(W + (int64_t)k * ldw + j, w_vec_ok, left);
                const float w[4] = {wv.x, wv.y, wv.z, wv.w};
                uint32_t sg[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) sg[u] = u < left ? (w[u] >= 0.f ? 0x3F80u : 0xBF80u) : 0u;
                *reinterpret_cast<uint2*>(signs + off + 4096 * it) = make_uint2(sg[0] | (sg[1] << 16), sg[2] | (sg[3] << 16));
            }
        }
        const int64_t cur_tile = tile;
        const int cur_ch = ch;
        if (++ch == n_chunks) {
            ch = 0;
            tile += gridDim.x;
        }
        if (c + 1 < total) load(tile, ch);
        tc::fence_async_smem();
        tc::fence_before_sync();
        if (__syncthreads_or(!ok)) { ok = false; break; }   // operands complete; leave together on a timeout
        tc::fence_after_sync();
        if (threadIdx.x == 0) {
            const uint32_t a_base = tc::smem_u32(stage), b_base = tc::smem_u32(signs);
            for (int ks = 0; ks < kGhK / 16; ++ks) {
                const uint64_t bd = tc::make_desc(b_base + ks * 32, 16, 1024) | ((uint64_t)2 << 61);
#pragma unroll
                for (int sp = 0; sp < 3; ++sp) {
                    const uint64_t ad = tc::make_desc(a_base + sp * kGhTerm + ks * 32, 16, 1024) | ((uint64_t)2 << 61);
                    const uint32_t accum = (cur_ch > 0 || ks > 0 || sp > 0) ? 1u : 0u;
                    asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
                                 ::"r"(tmem_base + (uint32_t)(acc * N)), "l"(ad), "l"(bd), "r"(idesc), "r"(accum) : "memory");
                }
            }
            tc::commit_to(&bar[st]);
        }
        if (cur_ch == 0 && c > 0) {                         // the tile before, from the other accumulator, by way of the other stage
            ok = wait(c - 1) && ok;
            tc::fence_after_sync();
            if (ok) finish(cur_tile - gridDim.x, acc ^ 1, sm + (st ^ 1) * kGhStage);
            tc::fence_before_sync();
            __syncthreads();                                // that stage is filled next
        }
        if (cur_ch == n_chunks - 1) acc ^= 1;
    }
    if (total > 0 && ok) {
        ok = wait(total - 1);
        tc::fence_after_sync();
        if (ok) finish(tile - gridDim.x, acc ^ 1, sm + (total & 1) * kGhStage);
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) tc::tmem_free(tmem_base, kCols);
}

// ---- G_W~ partial sums on the 5th-generation tensor cores -------------------------------------------------
// C^T[j][k] = sum over nodes of (beta_i G_zeta[i][j]) F[i][k] with tcgen05.mma kind::f16: M = 128 channels j, N = 64 / 128 /
// 256 inputs k (blockIdx.z: slices of N), the reduction over the block's nodes, accumulated in fp32 tiles of tensor memory
// that are read back at the end, added and written as slab blockIdx.y of `part` ([k][j]: consecutive lanes write
// consecutive j): one tile for 256 inputs, for fewer two of half the chunks each, which halves the rounding of the long sums
// where a block has twice the nodes (100 K nodes, 64 -> 64: G_W off by 1.1e-6 of its norm with one tile, 6e-7 with two; as
// many blocks more instead of tiles: 127 -> 132 us).  Both operands are node-major in global memory and stay so in shared
// memory: M- and N-major operands
// with 128-byte swizzle (64 channels or inputs of a node are 128 contiguous bytes), so nothing is transposed and every
// store is a vector.  Chunks of 32 nodes, two stages: while one is multiplied the other is filled, and the chunk after
// that is on its way in registers.  (With K-major operands every store was 4 bytes and the stages took turns: 2.4 M nodes,
// 256 -> 256, 2.7 ms.)
constexpr int kWtNodes = 32;                               // nodes per chunk
constexpr int kWtAtom = kWtNodes * 128;                    // bytes of 64 columns of a chunk

template <int N>
__global__ void __launch_bounds__(kBwThreads, 2)
grad_wt_tc_kernel(const uint32_t* __restrict__ bits, int64_t stride, const float* __restrict__ beta,
                  const float* __restrict__ gz, int64_t ldz, int64_t n, int d_in, int d_out,
                  int64_t rows_per_split, float* __restrict__ part)
{
    pdl_enter();
    constexpr int kStage = 6 * kWtAtom + N / 64 * kWtAtom;  // three terms x two atoms of channels, N / 64 atoms of inputs
    constexpr int kItems = kWtNodes * 32 / kBwThreads;      // 16-byte pieces of a chunk per thread
    constexpr int kTiles = N <= 128 ? 2 : 1;                // accumulators
    extern __shared__ unsigned char bw_raw[];
    __shared__ __align__(8) uint64_t bar[2];
    __shared__ uint32_t tmem_base_s;
    unsigned char* sm = bw_raw + ((1024u - (tc::smem_u32(bw_raw) & 1023u)) & 1023u);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp == 0) tc::tmem_alloc(&tmem_base_s, kTiles * N);
    if (threadIdx.x == 0) {
        tc::barrier_init(&bar[0]);
        tc::barrier_init(&bar[1]);
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem_base = tmem_base_s;
    // D = f32, A = B = bf16, A M-major, B N-major, N, M = 128
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
    const bool vec_ok = (ldz % 4 == 0) && (reinterpret_cast<uintptr_t>(gz) % 16 == 0);
    const int j0 = blockIdx.x * 128, k0 = blockIdx.z * N;
    const int64_t r_begin = (int64_t)blockIdx.y * rows_per_split;
    const int64_t r_end = min(n, r_begin + rows_per_split);
    const int n_chunks = r_begin < r_end ? (int)ceil_div(r_end - r_begin, kWtNodes) : 0;
    const int second = kTiles == 2 ? (n_chunks + 1) / 2 : n_chunks;      // first chunk of the second accumulator
    // this thread's pieces: channels j .. j + 3 of nodes warp + 8 it; and word wd of node `lane`
    const int j = j0 + 4 * lane, wd = (k0 >> 5) + warp;
    const bool has_word = warp < N / 32 && wd < stride;
    float4 xv[kItems];
    float bv[kItems];
    uint32_t word = 0u;
    auto load = [&](int c) {
        const int64_t r0 = r_begin + (int64_t)c * kWtNodes;
#pragma unroll
        for (int it = 0; it < kItems; ++it) {
            const int64_t row = r0 + warp + 8 * it;
            xv[it] = make_float4(0.f, 0.f, 0.f, 0.f);
            bv[it] = 0.f;
            if (row < r_end) {
                bv[it] = __ldg(beta + row);
                if (j + 3 < d_out && vec_ok) {
                    xv[it] = __ldg(reinterpret_cast<const float4*>(gz + row * ldz + j));
                } else {
                    if (j < d_out) xv[it].x = __ldg(gz + row * ldz + j);
                    if (j + 1 < d_out) xv[it].y = __ldg(gz + row * ldz + j + 1);
                    if (j + 2 < d_out) xv[it].z = __ldg(gz + row * ldz + j + 2);
                    if (j + 3 < d_out) xv[it].w = __ldg(gz + row * ldz + j + 3);
                }
            }
        }
        if (has_word) word = __ldg(bits + min(r0 + lane, r_end - 1) * stride + wd);   // (past the end: met by zeros)
    };
    // where they go inside a stage
    uint32_t a_off[kItems];
#pragma unroll
    for (int it = 0; it < kItems; ++it) {
        const int node = warp + 8 * it;
        a_off[it] = (uint32_t)((lane >> 4) * kWtAtom + (node >> 3) * 1024 + (node & 7) * 128 + ((((lane & 15) >> 1) ^ (node & 7)) << 4) + (lane & 1) * 8);
    }
    const uint32_t b_off = (uint32_t)(6 * kWtAtom + (warp >> 1) * kWtAtom + (lane >> 3) * 1024 + (lane & 7) * 128);
    bool ok = true;
    if (n_chunks > 0) load(0);
    for (int c = 0; c < n_chunks; ++c) {
        const int st = c & 1;
        unsigned char* stage = sm + st * kStage;
        if (c >= 2 && !tc::wait_barrier(&bar[st], (uint32_t)((c >> 1) + 1) & 1u)) {   // the products of chunk c - 2 are done
            atomicExch(&g_bw_tc_timeout, 1);
            ok = false;
        }
#pragma unroll
        for (int it = 0; it < kItems; ++it) {
            const float x[4] = {xv[it].x * bv[it], xv[it].y * bv[it], xv[it].z * bv[it], xv[it].w * bv[it]};
            unsigned short hi[4], mid[4], lo[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) split3(x[u], hi[u], mid[u], lo[u]);
            auto pack = [](const unsigned short (&h)[4]) { return make_uint2((uint32_t)h[0] | ((uint32_t)h[1] << 16), (uint32_t)h[2] | ((uint32_t)h[3] << 16)); };
            *reinterpret_cast<uint2*>(stage + 0 * kWtAtom + a_off[it]) = pack(hi);
            *reinterpret_cast<uint2*>(stage + 2 * kWtAtom + a_off[it]) = pack(mid);
            *reinterpret_cast<uint2*>(stage + 4 * kWtAtom + a_off[it]) = pack(lo);
        }
        if (warp < N / 32) {
            const uint32_t minus = ~word;                   // bit 0: -1
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                uint32_t o[4];
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const uint32_t two = minus >> (8 * q + 2 * r);
                    o[r] = 0x3F803F80u | ((two & 1u) << 15) | ((two & 2u) << 30);
                }
                *reinterpret_cast<uint4*>(stage + b_off + (((((warp & 1) * 4 + q)) ^ (lane & 7)) << 4)) = make_uint4(o[0], o[1], o[2], o[3]);
            }
        }
        if (c + 1 < n_chunks) load(c + 1);
        tc::fence_async_smem();
        tc::fence_before_sync();
        if (__syncthreads_or(!ok)) { ok = false; break; }   // leave together on a timeout
        tc::fence_after_sync();
        if (threadIdx.x == 0) {
            const uint32_t base = tc::smem_u32(stage), acc = tmem_base + (c >= second ? (uint32_t)N : 0u);
            for (int ks = 0; ks < kWtNodes / 16; ++ks) {
                const uint64_t bd = tc::make_desc(base + 6 * kWtAtom + ks * 2048, kWtAtom, 1024) | ((uint64_t)2 << 61);
#pragma unroll
                for (int sp = 0; sp < 3; ++sp) {
                    const uint64_t ad = tc::make_desc(base + sp * 2 * kWtAtom + ks * 2048, kWtAtom, 1024) | ((uint64_t)2 << 61);
                    const uint32_t accum = ((c > 0 && c != second) || ks > 0 || sp > 0) ? 1u : 0u;
                    asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
                                 ::"r"(acc), "l"(ad), "l"(bd), "r"(idesc), "r"(accum) : "memory");
                }
            }
            tc::commit_to(&bar[st]);
        }
    }
    if (ok && n_chunks > 0 && !tc::wait_barrier(&bar[(n_chunks - 1) & 1], (uint32_t)((n_chunks - 1) >> 1) & 1u)) {
        atomicExch(&g_bw_tc_timeout, 1);
        ok = false;
    }
    tc::fence_after_sync();
    ok = !__syncthreads_or(!ok);
    // ---- the slab: thread = channel j (tensor-memory lane), its warp's half of the inputs k
    if (ok) {
        float* slab = part + (int64_t)blockIdx.y * d_in * d_out;
        const int lane_base = 32 * (warp & 3);
        const int jj = j0 + lane_base + lane;
        const int c_begin = (warp >> 2) * (N / 2);
        for (int c0 = c_begin; c0 < c_begin + N / 2; c0 += 16) {
            uint32_t v[16];
            if (n_chunks > 0) tc::tmem_ld16(tmem_base + ((uint32_t)lane_base << 16) + (uint32_t)c0, v);
            if (second < n_chunks) {
                uint32_t u[16];
                tc::tmem_ld16(tmem_base + ((uint32_t)lane_base << 16) + (uint32_t)(N + c0), u);
#pragma unroll
                for (int e = 0; e < 16; ++e) v[e] = __float_as_uint(__uint_as_float(v[e]) + __uint_as_float(u[e]));
            }
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                const int k = k0 + c0 + e;
                if (jj < d_out && k < d_in) slab[(int64_t)k * d_out + jj] = n_chunks > 0 ? __uint_as_float(v[e]) : 0.f;
            }
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) tc::tmem_free(tmem_base, kTiles * N);
}

template <int N>
cudaError_t launch_grad_wt_tc(cudaStream_t s, const uint32_t* bits, int64_t stride, const float* beta, const float* gz,
                              int64_t ldz, int64_t n, int d_in, int d_out, int n_splits, int64_t rows_per_split, float* part)
{
    const size_t smem = 2 * (6 + N / 64) * (size_t)kWtAtom + 1024;
    cudaError_t e = cudaFuncSetAttribute(grad_wt_tc_kernel<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)ceil_div(d_out, 128), (unsigned)n_splits, (unsigned)ceil_div(d_in, N));
    launch_kernel(grad_wt_tc_kernel<N>, grid, kBwThreads, smem, s, bits, stride, beta, gz, ldz, n, d_in, d_out, rows_per_split, part);
    return cudaGetLastError();
}

template <int N>
cudaError_t launch_grad_h_tc(cudaStream_t s, const float* gz, int64_t ldz, const float* alpha, const float* W, int64_t ldw,
                             int64_t n, int d_in, int d_out, float* g_h, int64_t ldh)
{
    const int chunks = (int)ceil_div(d_out, kGhK);
    const size_t smem = 2 * kGhStage + (size_t)(chunks <= gh_slots(N) ? chunks : 2) * N * 128 + 1024;
    cudaError_t e = cudaFuncSetAttribute(grad_h_tc_kernel<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const unsigned slices = (unsigned)ceil_div(d_in, N);
    const dim3 grid((unsigned)std::min<int64_t>(ceil_div(n, kGhRows), std::max(1, sm_count() / (int)slices)), slices);
    launch_kernel(grad_h_tc_kernel<N>, grid, kGhThreads, smem, s, gz, ldz, alpha, W, ldw, n, d_in, d_out, g_h, ldh);
    return cudaGetLastError();
}

// Eq. bp-W.  A block per 32 channels x 32 inputs: thread (tx, ty) adds the partial column sums ty, ty + 32, ... of channel
// j0 + tx in double, the 32 sums of a channel are added in order, and every element gets
// (1/d_in) B_ij col_j + alpha_j G_W~_ij [|W_ij| < 1].
__global__ void __launch_bounds__(1024)
grad_w_kernel(const float* __restrict__ g_wt, const double* __restrict__ col_part, int n_part, const float* __restrict__ W, int64_t ldw,
              const float* __restrict__ alpha, int d_in, int d_out, float* __restrict__ g_w, int64_t ldgw)
{
    pdl_enter();
    __shared__ double part[32][33];
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int j = blockIdx.x * 32 + tx, i = blockIdx.y * 32 + ty;
    double s = 0.0;
    if (j < d_out) {
#pragma unroll 4
        for (int q = ty; q < n_part; q += 32) s += __ldg(col_part + (int64_t)q * d_out + j);
    }
    part[ty][tx] = s;
    __syncthreads();
    if (j >= d_out || i >= d_in) return;
    double c = 0.0;
    for (int r = 0; r < 32; ++r) c += part[r][tx];
    c /= (double)d_in;
    const float w = __ldg(W + (int64_t)i * ldw + j);
    double g = w >= 0.f ? c : -c;
    if (fabsf(w) < 1.f) g += (double)__ldg(alpha + j) * (double)__ldg(g_wt + (int64_t)i * d_out + j);
    g_w[(int64_t)i * ldgw + j] = (float)g;
}

int64_t pad4(int64_t d) { return (d + 3) / 4 * 4; }

// Parts that the sum over the nodes is split into: two blocks per multiprocessor in all, at least 128 nodes each.  Twice as many
// where an odd number of 128 inputs above 256 would leave fewer than four per multiprocessor and 128 x 128 weights: a part
// is one fp32 accumulation, whose rounding grows with its length (100 K nodes, 300 -> 200: G_W off by 3.3e-6 of its norm with
// 74 parts, by 2.4e-6 with 98).
int wt_splits(int64_t n, int d_in, int d_out)
{
    const int64_t tiles = ceil_div(d_in, 256) * ceil_div(d_out, 128), squares = ceil_div(d_in, 128) * ceil_div(d_out, 128);
    const int64_t wave = std::max<int64_t>(1, sm_count() * 2 / tiles);
    const int64_t want = d_in > 256 && sm_count() * 4 / squares > wave ? 2 * wave : wave;
    return (int)std::max<int64_t>(1, std::min<int64_t>(want, ceil_div(n, 128)));
}

}  // namespace

int backward_tc_timeouts()
{
    int v = 0;
    if (cudaMemcpyFromSymbol(&v, g_bw_tc_timeout, sizeof(int)) != cudaSuccess) return -1;
    return v;
}

size_t backward_scratch_bytes(int64_t n, int d_in, int d_out)
{
    const size_t a = 256;
    auto up = [&](size_t b) { return (b + a - 1) / a * a; };
    size_t total = up((size_t)n * pad4(d_out) * 4);                              // G' with rows padded to 16 bytes
    total += up((size_t)n * pad4(d_out) * 4);                                    // G_zeta
    total += up((size_t)wt_splits(n, d_in, d_out) * d_in * d_out * 4);           // slabs of G_W~
    total += up((size_t)d_in * d_out * 4);                                       // G_W~
    total += up((size_t)ceil_div(d_in, kRedRows) * d_out * 8);                   // column sums of Eq. bp-W
    total += up(spmm_scratch_bytes(n, 0, 0));
    return total;
}

cudaError_t launch_layer_backward(cudaStream_t s, int64_t n, const int64_t* rowptr, const int32_t* colidx,
                                  const float* val, int d_in, int d_out, const float* W, int64_t ldw,
                                  const float* alpha, const uint32_t* in_bits, int64_t stride_in,
                                  const float* in_beta, const float* g_out, int64_t ldg, float* g_in,
                                  int64_t ldgi, float* g_w, int64_t ldgw, int64_t long_row, void* scratch,
                                  int* launches)
{
    const size_t a = 256;
    auto up = [&](size_t b) { return (b + a - 1) / a * a; };
    char* base = static_cast<char*>(scratch);
    const int64_t ldz = pad4(d_out);
    float* g_pad = reinterpret_cast<float*>(base);
    base += up((size_t)n * ldz * 4);
    float* gz = reinterpret_cast<float*>(base);
    base += up((size_t)n * ldz * 4);
    int n_splits = wt_splits(n, d_in, d_out);
    float* part = reinterpret_cast<float*>(base);
    base += up((size_t)n_splits * d_in * d_out * 4);
    float* g_wt = reinterpret_cast<float*>(base);
    base += up((size_t)d_in * d_out * 4);
    const int n_part = (int)ceil_div(d_in, kRedRows);
    double* col_part = reinterpret_cast<double*>(base);
    base += up((size_t)n_part * d_out * 8);
    void* counter = base;

    // step 1a: G_zeta = A_tilde^T G' (A_tilde is symmetric: the forward aggregation on fp32 rows)
    const float* g_src = g_out;
    if (ldg != ldz || reinterpret_cast<uintptr_t>(g_out) % 16 != 0) {            // rows must be 16-byte vectors
        launch_kernel(pad_rows_kernel, (unsigned)std::min<int64_t>(ceil_div(n * ldz, 256), sm_count() * 16), 256, 0, s, g_out, n, d_out, ldg, g_pad, ldz);
        ++*launches;
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        g_src = g_pad;
    }
    SpmmArgs sa;
    sa.n = n;
    sa.rowptr = rowptr;
    sa.colidx = colidx;
    sa.val = val;
    sa.fmt = kZetaF32;
    sa.zeta = g_src;
    sa.ldz = ldz;
    sa.d_out = d_out;
    sa.node_w = nullptr;
    sa.col_w = nullptr;
    sa.add = nullptr;
    sa.ld_add = 0;
    sa.h_out = gz;
    sa.ldh = ldz;
    sa.next_bits = nullptr;
    sa.next_stride = 0;
    sa.next_beta = nullptr;
    sa.next_shift = nullptr;
    sa.next_scale = nullptr;
    sa.long_row = long_row;
    sa.scratch = counter;
    sa.scratch_bytes = spmm_scratch_bytes(n, 0, 0);
    sa.any_order = true;
    cudaError_t e = launch_spmm(s, sa, launches);
    if (e != cudaSuccess) return e;

    // step 1b: G_W~ = H~^T G_zeta, split over the rows, slabs added in a fixed order
    {
        // whole pairs of chunks; of few nodes whole chunks, and no part without nodes (19,717 nodes, 500 -> 64: 103 parts of 192 nodes and
        // 45 empty ones, now 124 of 160)
        const int64_t each = ceil_div(n, n_splits), unit = each <= 8 * kWtNodes ? kWtNodes : 2 * kWtNodes;
        const int64_t rows_per_split = std::max<int64_t>(1, ceil_div(each, unit)) * unit;
        n_splits = (int)std::max<int64_t>(1, ceil_div(n, rows_per_split));
        ++*launches;
        if (d_in <= 64) e = launch_grad_wt_tc<64>(s, in_bits, stride_in, in_beta, gz, ldz, n, d_in, d_out, n_splits, rows_per_split, part);
        else if (d_in <= 128) e = launch_grad_wt_tc<128>(s, in_bits, stride_in, in_beta, gz, ldz, n, d_in, d_out, n_splits, rows_per_split, part);
        else e = launch_grad_wt_tc<256>(s, in_bits, stride_in, in_beta, gz, ldz, n, d_in, d_out, n_splits, rows_per_split, part);
        if (e != cudaSuccess) return e;
        launch_kernel(grad_wt_reduce_kernel, dim3((unsigned)ceil_div(d_out, 32), (unsigned)n_part), 32 * kRedRows * kRedGroups, 0, s, part, n_splits, d_in, d_out, W, ldw, g_wt, col_part);
        ++*launches;
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    // step 1c + 2: G_H = clip(G_zeta W~^T)
    if (g_in) {
        ++*launches;
        if (d_in % 4 == 0 && ldgi % 4 == 0 && reinterpret_cast<uintptr_t>(g_in) % 16 == 0) {   // tcgen05 version
            if (d_in <= 64) e = launch_grad_h_tc<64>(s, gz, ldz, alpha, W, ldw, n, d_in, d_out, g_in, ldgi);
            else if (d_in <= 128) e = launch_grad_h_tc<128>(s, gz, ldz, alpha, W, ldw, n, d_in, d_out, g_in, ldgi);
            else e = launch_grad_h_tc<256>(s, gz, ldz, alpha, W, ldw, n, d_in, d_out, g_in, ldgi);
            if (e != cudaSuccess) return e;
        } else {
            const dim3 grid((unsigned)ceil_div(n, kMmaTile), (unsigned)ceil_div(d_in, kMmaTile));
            launch_kernel(grad_h_mma_kernel, grid, kBwThreads, 0, s, gz, ldz, alpha, W, ldw, n, d_in, d_out, g_in, ldgi);
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
        }
    }
    // step 3: Eq. bp-W
    launch_kernel(grad_w_kernel, dim3((unsigned)ceil_div(d_out, 32), (unsigned)ceil_div(d_in, 32)), dim3(32, 32), 0, s, g_wt, col_part, n_part, W, ldw, alpha, d_in, d_out, g_w, ldgw);
    ++*launches;
    return cudaGetLastError();
}

}  // namespace bigcn

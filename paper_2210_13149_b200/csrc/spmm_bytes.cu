// Aggregation H' = A_tilde zeta (Bi-GCN, last equation of Sec. 4.2.3) of rows of 33..64 signed bytes as exact integer products,
// optionally with the re-binarization of H' for the next layer (Sec. 4.2.2) in its epilogue.
//
// A warp takes the groups of stored entries of its units of work (spmm_groups.cuh: two rows where they fit 128 entries, else one, or a
// piece of one).  The byte rows of a group are copied to shared memory as they are (cp.async) and read transposed by ldmatrix, 32
// entries x 16 columns at a time, as the A operand of mma.sync m16n8k32; the B operand holds the entries' weights w = A_tilde_ie
// beta_e in fixed point against a power of two of the row's largest (|q| <= 2^30), split into four balanced base-256 digits: columns
// 0..3 for the first row, 4..7 for the second.  The digit sums are exact in 32 bits; a lane pair recombines them at a row's end, and
// a lane holds the row's columns 16 m + g + 8 odd.  Pieces of a row share a scale (with 3 bits to spare) and the accumulators until one
// has a larger weight or 480 entries are summed; what there is then moves to an fp32 sum.  A weight is off by at most 2^-30 of the
// largest of its row, in rows of more than 128 entries 2^-27 of the largest of the piece that set its scale; the fp32 sums that this
// replaces rounded every addition to 2^-24.
//
// Half-dot bytes (kHalf): zeta holds s = (dot' - 1) / 2 and the node factor carries the first feature sign f; sum w dot = 2 sum w s +
// sum w + b0_j sum w f.  The two sums over the weights are two columns of one more A operand, all ones and the signs.
//
// Weights that have no fixed point (a piece's largest not finite, or outside 2^-87 .. 2^104) meet their dots one by one in fp32, from the
// byte rows in shared memory, while their digits are 0: the other pieces of a row are summed like any, so that such a weight beside a
// hub row costs what its 128 entries do.  (Summed from memory by the warp that ends it, a row of 100,000 entries with one NaN took
// 49 ms, with 0.22 for the launch now.)
#include <algorithm>
#include <type_traits>

#include "bigcn_internal.cuh"
#include "spmm_dev.cuh"
#include "spmm_groups.cuh"
#include "tc_common.cuh"

namespace bigcn {

namespace {

using namespace groups;
using tc::smem_u32;

constexpr int kWarps = 8, kThreads = 32 * kWarps, kBlocks = 2;
constexpr int kRowBytes = 64, kWindowBytes = 32 * kRowBytes;
constexpr int kRing = 5;                            // windows of 32 entries: a group's up to four, and the first of the next
constexpr int kChain = 480;                         // entries under one scale: |digit byte| <= 2^14 each, times 256, fit 32 bits

template <int MT>                                   // 16-column products
struct Slot {                                       // of a warp
    uint8_t rows[kRing][kWindowBytes];              // byte rows of the windows of the group at hand and of the next; 16-byte pieces of entry e exchanged by (e / 2) % 4
    uint2 q[2][32][2];                              // [window / 2][entry][window % 2]: digits of the entry's weight under the group's two rows (0 under the other)
    uint8_t sign[kGroup];                           // first feature signs, +-1
    float sums[2][16 * MT];                         // an open row's sums; of a direct group, what its rows sum in fp32
};

struct BytesDev {
    SpmmDev p;
    GraphPlan plan;
    float* parts;                                   // [chunks][2][16 MT]: pieces of rows cut by a unit's end
    unsigned* counters;                             // [chunks] pieces done; zeroed before
};

__device__ __forceinline__ void imma(int (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0,%1,%2,%3},{%4,%5,%6,%7},{%8,%9},{%0,%1,%2,%3};\n"
        : "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// kTail: a byte row is 64 bytes and carries its node factor in the last four.  kAdd: rows of p.add are added.
template <int MT, bool kHalf, bool kTail, bool kAdd>
__global__ void __launch_bounds__(kThreads, kBlocks) agg_bytes_kernel(const __grid_constant__ BytesDev d)
{
    pdl_enter();
    const SpmmDev& p = d.p;
    extern __shared__ __align__(128) unsigned char bytes_smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = lane >> 2, t = lane & 3;
    const bool odd = t & 1;
    Slot<MT>* const slot = reinterpret_cast<Slot<MT>*>(bytes_smem) + warp;
    float4* const tab = reinterpret_cast<float4*>(reinterpret_cast<Slot<MT>*>(bytes_smem) + kWarps);   // per column: alpha, first weight sign, next shift, next scale
    const uint32_t rows0 = smem_u32(slot->rows), q0 = smem_u32(slot->q) + (uint32_t)(lane * 16);
    for (int j = threadIdx.x; j < 16 * MT; j += kThreads) {
        const bool in = j < p.d_out;
        tab[j] = make_float4(in ? (p.col_w ? __ldg(p.col_w + j) : 1.f) : 0.f, in && kHalf ? __ldg(p.col_b0 + j) : 0.f,
                             in && p.next_shift ? __ldg(p.next_shift + j) : 0.f, in ? (p.next_shift ? __ldg(p.next_scale + j) : 1.f) : 0.f);
    }
    __syncthreads();
    const int my_col = g + 8 * odd;                 // this lane's columns are 16 m + my_col
    const uint32_t my_ld = (uint32_t)(lane * kRowBytes + (((lane >> 1) & 3) << 4));   // piece m of entry 32 i + lane at 2048 i + (my_ld ^ (m << 4))
    const int my_e = lane >> 2;                     // copies: an instruction takes 8 rows, four lanes each
    const uint32_t my_dst = (uint32_t)(my_e * kRowBytes + (((lane & 3) ^ ((my_e >> 1) & 3)) << 4));

    // Three groups in flight: one (a) is computed, with everything it needs loaded in the turn before; the rows (and node factors) of
    // the next (b) are on their way, and the column indices and values of the one after (c).
    Stream c_group((int)(blockIdx.x * kWarps) + uniform(warp), (int)(gridDim.x * kWarps));
    int b_row = 0, b_meta = 0, b_place = 0;
    float b_val[4] = {}, b_fac[4] = {};
    int b_col[4] = {};
    int at_a = 0, at_b = 0, win_a = 0;              // ring positions of the first windows of a and b; windows of a
    auto ring = [](int i) { return i >= kRing ? i - kRing : i; };
    // rows of b's windows [from, to)
    auto copy = [&](int from, int to) {
        const int cnt = b_meta & 255;
        const char* src = reinterpret_cast<const char*>(p.zeta) + 16 * (lane & 3);
        const int mine = (lane & 3) < p.nv ? cnt - my_e : 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (i < from || i >= to) continue;
            const uint32_t dst = rows0 + (uint32_t)(ring(at_b + i) * kWindowBytes) + my_dst;
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const uint32_t c = (uint32_t)__shfl_sync(0xffffffffu, b_col[i], 8 * h + my_e);
                if (32 * i + 8 * h < mine)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n"
                                 ::"r"(dst + (uint32_t)(8 * h * kRowBytes)), "l"(src + (uint64_t)c * (uint32_t)(16 * p.nv)) : "memory");
            }
        }
    };
    // c becomes b
    auto take = [&]() {
        b_row = c_group.row;
        b_meta = c_group.meta;
        b_place = c_group.place;
        at_b = ring(at_a + win_a);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            b_val[i] = c_group.val[i];
            b_col[i] = c_group.col[i];
            if constexpr (!kTail) {
                if (32 * i < (b_meta & 255)) b_fac[i] = __ldg(p.node_w + b_col[i]);
            }
        }
    };

    int c[MT][4], cx[4];
    auto clear = [&]() {
#pragma unroll
        for (int m = 0; m < MT; ++m) c[m][0] = c[m][1] = c[m][2] = c[m][3] = 0;
        cx[0] = cx[1] = cx[2] = cx[3] = 0;
    };
    // the digit sums of this lane's row as numbers
    auto read_back = [&](float sc, float (&x)[MT]) {
        auto number = [&](int lo, int hi) { return fmaf((float)hi, 65536.f, (float)lo) * sc; };
        float ws = 0.f, wg = 0.f;
        if constexpr (kHalf) {
            const int part = cx[1] * 256 + cx[0];
            const int lo = __shfl_sync(0xffffffffu, part, t & 2), hi = __shfl_sync(0xffffffffu, part, (t & 2) + 1);
            const int lo2 = __shfl_sync(0xffffffffu, part, 4 + (t & 2)), hi2 = __shfl_sync(0xffffffffu, part, 4 + (t & 2) + 1);
            ws = number(lo, hi);
            wg = number(lo2, hi2);
        }
#pragma unroll
        for (int m = 0; m < MT; ++m) {
            const int a = c[m][1] * 256 + c[m][0], b = c[m][3] * 256 + c[m][2];   // columns g and g + 8: of the low digits, or (odd) of the high ones
            const int got = __shfl_xor_sync(0xffffffffu, odd ? a : b, 1);
            x[m] = number(odd ? got : a, odd ? b : got);
            if constexpr (kHalf) x[m] = fmaf(2.f, x[m], fmaf(tab[16 * m + my_col].y, wg, ws));
        }
    };
    bool row_open = false;                          // slot->sums holds sums of the row that the pieces belong to
    uint32_t chain_x = 0;                           // the scale of the pieces summed in the accumulators, and their entries
    int chain = 0;
    auto move = [&]() {
        float x[MT];
        read_back(__uint_as_float((chain_x - 29u) << 23), x);
        if (t < 2) {
#pragma unroll
            for (int m = 0; m < MT; ++m) {
                float* f = slot->sums[0] + 16 * m + my_col;
                *f = row_open ? *f + x[m] : x[m];
            }
        }
        row_open = true;
        clear();
    };
    // row `row` and, in the lanes t >= 2 where there are two, row + 1: column factor, the added rows, H' and the next layer's bits
    auto finish = [&](float (&x)[MT], const float (&own)[MT], int row, bool two) {
        const int64_t rw = row + (t >> 1);
        const bool on = two || t < 2;
        float l1 = 0.f;
        uint32_t word = 0u;
#pragma unroll
        for (int m = 0; m < MT; ++m) {
            const int col = 16 * m + my_col;
            const float4 k = tab[col];
            const bool in = col < p.d_out;
            float v = x[m] * k.x;
            if constexpr (kAdd) v += own[m];
            if (p.h_out && on && in) p.h_out[rw * p.ldh + col] = v;
            if (p.next_bits) {
                const float xh = __fmul_rn(__fsub_rn(v, k.z), k.w);
                const uint32_t b = __ballot_sync(0xffffffffu, in && xh >= 0.f);
                if ((lane >> 1) == m) word = b;
                l1 += in ? fabsf(xh) : 0.f;
            }
        }
        if (p.next_bits) {
            // lane 2 m + h of the first ones: byte 2 m + h of a row, its bits 4 apart in the ballot
            auto pick = [](uint32_t v) {
                v &= 0x11111111u;
                v = (v | v >> 3) & 0x03030303u;
                v = (v | v >> 6) & 0x000f000fu;
                return (unsigned char)(v | v >> 12);
            };
            unsigned char* dst = reinterpret_cast<unsigned char*>(p.next_bits + (int64_t)row * p.next_stride) + lane;
            if (lane < 4 * p.next_stride) {
                dst[0] = pick(word >> (lane & 1));
                if (two) dst[4 * p.next_stride] = pick(word >> (2 + (lane & 1)));
            }
            l1 += __shfl_xor_sync(0xffffffffu, l1, 1);
#pragma unroll
            for (int o = 4; o < 32; o <<= 1) l1 += __shfl_xor_sync(0xffffffffu, l1, o);
            if (g == 0 && !odd && on) p.next_beta[rw] = l1 * p.inv_d_out;
        }
    };
    auto no_fixed_point = [](uint32_t most) { return most != 0u && ((most >> 23) < kExpLow || (most >> 23) > kExpHigh); };
    auto exponent = [](uint32_t most) { return min(max(most >> 23, kExpLow), kExpHigh + 1u); };

    // adds sum_e w_e dot_ej over entries [from, to) of the group whose windows lie at `at`, in fp32, to (or, fresh, as) sums[h].
    // slot->q holds the weights, slot->sign the signs
    auto sum_written = [&](int at, int from, int to, int h, bool fresh) {
#pragma unroll 1
        for (int j = lane; j < 16 * MT; j += 32) {
            float s = 0.f;
#pragma unroll 4
            for (int e = from; e < to; ++e) {
                const int i = e >> 5, r = e & 31;
                const float b = (float)(signed char)slot->rows[ring(at + i)][r * kRowBytes + (((j >> 4) ^ ((r >> 1) & 3)) << 4) + (j & 15)];
                float dot = b;
                if constexpr (kHalf) dot = 2.f * b + 1.f + ((slot->sign[e] & 0x80) ? -tab[j].y : tab[j].y);
                s = fmaf(__uint_as_float(slot->q[i >> 1][r][i & 1].x), dot, s);
            }
            slot->sums[h][j] = fresh ? s : slot->sums[h][j] + s;
        }
    };
    bool have_a = false, have_b = false, have_c = c_group.next(d.plan);
    if (have_c) c_group.load(p.colidx, p.val, lane);
    for (;;) {
        have_a = have_b;
        const int row = b_row, meta = b_meta, place = b_place;
        at_a = at_b;
        win_a = have_a ? ((meta & 255) + 31) >> 5 : 0;
        float w[4], fac[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            w[i] = b_val[i];
            fac[i] = b_fac[i];
        }
        have_b = have_c;
        const int early = kRing - win_a;
        if (have_b) {
            take();
            copy(0, min(early, 4));
            have_c = c_group.next(d.plan);
            if (have_c) c_group.load(p.colidx, p.val, lane);
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
        if (have_a) {
            const int cnt = meta & 255, mid = (meta >> 8) & 255, flags = meta >> 16;
            float own[MT] = {};                     // what is added to the rows, asked for before their products
            if (kAdd && (flags & (kDirect | kLast)) && (t < 2 || (flags & kPair))) {
                const float* src = p.add + (int64_t)(row + (t >> 1)) * p.ld_add + my_col;
#pragma unroll
                for (int m = 0; m < MT; ++m) own[m] = 16 * m + my_col < p.d_out ? __ldg(src + 16 * m) : 0.f;
            }
            asm volatile("cp.async.wait_group 1;\n" ::: "memory");
            __syncwarp();
            uint32_t rows[4];                       // this lane's row of each window
#pragma unroll
            for (int i = 0; i < 4; ++i) rows[i] = rows0 + (uint32_t)(ring(at_a + i) * kWindowBytes) + my_ld;
            uint32_t m0 = 0u, m1 = 0u;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (32 * i >= cnt) {
                    w[i] = 0.f;
                    continue;
                }
                if constexpr (kTail) asm volatile("ld.shared.f32 %0, [%1];\n" : "=f"(fac[i]) : "r"((rows[i] ^ 48u) + 12u) : "memory");
                w[i] = 32 * i + lane < cnt ? w[i] * (kHalf ? fabsf(fac[i]) : fac[i]) : 0.f;
                const uint32_t mag = __float_as_uint(w[i]) & 0x7fffffffu;      // (as integers, NaN is the largest of all)
                if (32 * i + lane < mid) m0 = max(m0, mag);
                else m1 = max(m1, mag);
            }
            m0 = __reduce_max_sync(0xffffffffu, m0);
            m1 = flags & kPair ? __reduce_max_sync(0xffffffffu, m1) : 0u;
            const bool written0 = no_fixed_point(m0), written1 = no_fixed_point(m1);
            uint32_t x0 = written0 ? kExpLow : exponent(m0);
            const uint32_t x1 = exponent(m1);
            if (flags & (kDirect | kFirst)) {
                clear();
                row_open = false;
                if (!(flags & (kDirect | kLast))) x0 += 3;
                chain_x = x0;
                chain = cnt;
            } else if (x0 <= chain_x && chain + cnt <= kChain) {
                x0 = chain_x;
                chain += cnt;
            } else {
                move();
                if (!(flags & kLast)) x0 += 3;
                chain_x = x0;
                chain = cnt;
            }
            if (written0 || written1) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    slot->q[i >> 1][lane][i & 1].x = __float_as_uint(w[i]);
                    if constexpr (kHalf) slot->sign[32 * i + lane] = signbit(fac[i]) ? 0xffu : 1u;
                }
                __syncwarp();
                if (written0) {
                    sum_written(at_a, 0, mid, 0, !row_open);
                    row_open = !(flags & kDirect);
                }
                if (written1) sum_written(at_a, mid, cnt, 1, true);
                __syncwarp();
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (32 * i + lane < mid ? written0 : written1) w[i] = 0.f;
            }
            const float f0 = __uint_as_float((283u - x0) << 23), f1 = __uint_as_float((283u - x1) << 23);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (32 * i >= cnt) break;
                const bool a = 32 * i + lane < mid;
                const uint32_t dg = ((uint32_t)__float2int_rn(w[i] * (a ? f0 : f1)) + kFlip) ^ kFlip;
                slot->q[i >> 1][lane][i & 1] = make_uint2(a ? dg : 0u, a ? 0u : dg);
                if constexpr (kHalf) slot->sign[32 * i + lane] = signbit(fac[i]) ? 0xffu : 1u;
            }
            __syncwarp();
            auto window = [&](uint32_t at, int i, uint32_t b0, uint32_t b1) {
#pragma unroll
                for (int m = 0; m < MT; ++m) {
                    uint32_t a[4];
                    ldmatrix_bytes(at ^ (uint32_t)(m << 4), a);
                    imma(c[m], a[0], a[1], a[2], a[3], b0, b1);
                }
                if constexpr (kHalf) {
                    const uint32_t* s = reinterpret_cast<const uint32_t*>(slot->sign + 32 * i) + t;
                    const uint32_t s0 = s[0], s1 = s[4];
                    imma(cx, g == 0 ? 0x01010101u : (g == 1 ? s0 : 0u), 0u, g == 0 ? 0x01010101u : (g == 1 ? s1 : 0u), 0u, b0, b1);
                }
            };
            auto windows = [&](int i, uint32_t at0, uint32_t at1) {
                uint32_t b[4];
                ldmatrix_bytes(q0 + (uint32_t)(i * 256), b);
                window(at0, i, b[0], b[2]);
                if (32 * (i + 1) < cnt) window(at1, i + 1, b[1], b[3]);
            };
            if (cnt > 0) windows(0, rows[0], rows[1]);
            if (cnt > 64) windows(2, rows[2], rows[3]);
            if (have_b && early < 4) {              // the rows that had to wait for a's places
                __syncwarp();
                copy(early, 4);
            }
            asm volatile("cp.async.commit_group;\n" ::: "memory");
            if (flags & (kDirect | kLast)) {
                float x[MT];
                bool done = true;
                if (flags & kDirect) {
                    read_back(__uint_as_float(((t < 2 ? x0 : x1) - 29u) << 23), x);
                    if (t < 2 ? written0 : written1) {
#pragma unroll
                        for (int m = 0; m < MT; ++m) x[m] = slot->sums[t >> 1][16 * m + my_col];
                    }
                } else {
                    move();
                    done = flags & kWhole;
                    __syncwarp();
                    if (!done) {
                        // the row reaches over several units: leave this one's sums; whoever comes last adds them up in order
                        constexpr int kPart = 16 * MT;
                        const int u0 = ((int)__ldg(p.rowptr + row) + kRowCost * row) >> d.plan.chunk_log2;
                        const int u1 = ((int)__ldg(p.rowptr + row + 1) + kRowCost * (row + 1) - 1) >> d.plan.chunk_log2;
                        float* part = d.parts + ((int64_t)place * 2 + ((flags & kStarts) ? 1 : 0)) * kPart;
#pragma unroll 1
                        for (int i = lane; i < kPart; i += 32) part[i] = slot->sums[0][i];
                        __threadfence();
                        __syncwarp();
                        unsigned before = 0;
                        if (lane == 0) before = atomicAdd(d.counters + u0, 1u);
                        done = __shfl_sync(0xffffffffu, before, 0) == (unsigned)(u1 - u0);
                        if (done) {
                            __threadfence();
#pragma unroll 1
                            for (int i = lane; i < kPart; i += 32) {
                                float s = __ldcg(d.parts + ((int64_t)u0 * 2 + 1) * kPart + i);
                                for (int u = u0 + 1; u <= u1; ++u) s += __ldcg(d.parts + (int64_t)u * 2 * kPart + i);
                                slot->sums[0][i] = s;
                            }
                            __syncwarp();
                        }
                    }
#pragma unroll
                    for (int m = 0; m < MT; ++m) x[m] = slot->sums[0][16 * m + my_col];
                }
                if (done) finish(x, own, row, flags & kPair);
            }
        } else if (!have_b) {
            break;
        } else {
            asm volatile("cp.async.commit_group;\n" ::: "memory");
        }
        __syncwarp();                               // the rows and digits just read are written again
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");
}

size_t up256(size_t x) { return (x + 255) / 256 * 256; }
size_t parts_bytes(int chunks) { return up256((size_t)chunks * 2 * 64 * 4); }

template <int MT, bool kHalf, bool kTail, bool kAdd>
cudaError_t launch_inst(cudaStream_t s, const BytesDev& d)
{
    constexpr int smem = kWarps * (int)sizeof(Slot<MT>) + 16 * MT * 16;
    cudaError_t e = cudaFuncSetAttribute(agg_bytes_kernel<MT, kHalf, kTail, kAdd>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    e = cudaMemsetAsync(d.counters, 0, (size_t)d.plan.chunks * 4, s);
    if (e != cudaSuccess) return e;
    const unsigned grid = (unsigned)std::min<int64_t>(ceil_div(d.plan.chunks, kWarps), (int64_t)sm_count() * kBlocks);
    launch_kernel(agg_bytes_kernel<MT, kHalf, kTail, kAdd>, grid, kThreads, smem, s, d);
    return cudaGetLastError();
}
template <int MT>
cudaError_t launch_mt(cudaStream_t s, const BytesDev& d)
{
    auto inst = [&](auto half, auto tail) {
        return d.p.add ? launch_inst<MT, half(), tail(), true>(s, d) : launch_inst<MT, half(), tail(), false>(s, d);
    };
    const std::true_type yes;
    const std::false_type no;
    if (d.p.row_tail) return d.p.half_dots ? inst(yes, yes) : inst(no, yes);
    return d.p.half_dots ? inst(yes, no) : inst(no, no);
}

}  // namespace

bool spmm_bytes_covers(int64_t n, int64_t nnz, int d_in, int d_out)
{
    return d_in <= 256 && d_out > 32 && d_out <= 64 && n > 0 && nnz + kRowCost * (n + 2) < (int64_t(1) << 31) - 4096;
}

// Where these products take the place of the lane-per-entry stream: on rows long enough to fill groups, and where the plan, which the
// layer may have to make for itself, is small beside the launch.  256 inputs, the aggregation alone (and the plan) against the
// stream: 2.4 M rows of 51, 47 columns 2.19 (0.06) / 2.59 ms, 64 columns 2.38 / 3.25; 800,000 of 30, 40 columns 569 (63) / 642 us;
// 200,000 of 60, 40 columns 232 (23) / 270, of 30 189 (21) / 196; 30,000 of 200 117 (12) / 154, of 60 65 (12) / 74; 169,343 of
// 15 140 (19) / 121.  Whole layers, stream / products with the plan, power-law graphs in rows of 42 and 60: 4.3 M entries, 40 columns 137 /
// 153 and 122 / 140, 64 columns 164 / 169 and 153 / 155; 6 M entries, 40 columns 180 / 178 and 164 / 159, 64 columns 219 / 195 and 188 /
// 165; so rows of three products, which the stream takes with fewer registers, need 5 Mi entries, and rows of four 4 Mi.
bool spmm_bytes_pays(int64_t n, int64_t nnz, int d_in, int d_out)
{
    return spmm_bytes_covers(n, nnz, d_in, d_out) && nnz >= 40 * n && nnz >= (int64_t(d_out <= 48 ? 5 : 4) << 20);
}

size_t spmm_bytes_scratch_bytes(int64_t n, int64_t nnz)
{
    const int chunks = spmm_bits_plan_at(n, nnz, nullptr).chunks;
    return parts_bytes(chunks) + up256((size_t)chunks * 4);
}

cudaError_t launch_spmm_bytes(cudaStream_t s, const SpmmDev& p, int64_t nnz, const void* plan, void* scratch)
{
    BytesDev d = {};
    d.p = p;
    d.plan = spmm_bits_plan_at(p.n, nnz, plan);
    d.parts = static_cast<float*>(scratch);
    d.counters = reinterpret_cast<unsigned*>(static_cast<char*>(scratch) + parts_bytes(d.plan.chunks));
    return p.d_out <= 48 ? launch_mt<3>(s, d) : launch_mt<4>(s, d);
}

}  // namespace bigcn

// One layer of Bi-GCN (Sec. 4.2.3) with the aggregation taken before the contraction, on the packed sign bits:
//
//     H' = A_tilde (diag(beta) F B diag(alpha)) = ((A_tilde diag(beta)) F) B diag(alpha) = P B diag(alpha),
//
// P_ik = sum_e w_e F_ek over the stored entries e of row i, w_e = A_tilde_ie beta_e, F_ek = +-1.  The gather then reads one
// bit per source column -- 16 or 32 bytes per stored entry of a matrix that stays in the L2 -- where aggregating contracted
// rows reads 1 to 4 bytes per output column.  Both products run on the tensor cores with exact integers.
//
// plan_kernel: the split of the stored entries into units and groups, a property of the graph, made once per forward.
//
// agg_bits_kernel: P.  The weights of a row are written in fixed point against a power of two of the row (sum |q| <= 2^30)
// and split into four balanced base-256 digits.  A warp takes groups of up to 128 consecutive stored entries (two rows where
// they fit, else one row or a piece of one) in windows of 32: mma.sync m16n8k32 multiplies the window's bits (A operand,
// 16 columns x 32 entries) by its digits (B operand, 32 entries x two rows' four digits).  The packed rows of a group are
// copied to shared memory as they are and read transposed by ldmatrix, a lane getting one byte of four entries in a register;
// (bytes & 0x01010101 << j) IS the operand of column j scaled by 2^j, which the read-back removes: one logic instruction per
// four bits.  The mma.sync form is taken because it alone lets the operand be built in registers; tcgen05 wants it in shared
// memory, where the expanded bytes would cost two passes over 256 bytes per entry.  P leaves as its four digit bytes, in the
// layout the next kernel reads.  Bound: instructions at the few warps that the accumulators leave room for (53 to 58 % of the issue
// slots, the logic pipe 57 %, the tensor pipe 18 %; 256 columns, 31.5 M entries 0.79 ms).
//
// bits_gemm_kernel: H' = P B diag(alpha) as tcgen05.mma.kind::i8.  The digits of 32 rows are one operand of N = 128 (row,
// digit) columns, K-major with 128-byte swizzle, fetched by bulk copies; the other is the weights expanded to +-1 bytes
// (M = 128 output columns, resident).  The epilogue combines a row's four digit sums (exact int32), scales by the row's power
// of two and alpha, and stores H' and / or packs it for the next layer.
//
// Rows whose weights have no common fixed point -- a non-finite one, or magnitudes outside 2^-87 .. 2^104 -- carry a mark for
// their scale, and the second kernel sums them as they are written, in fp32 (literal_row).
//
// Two kernels and not one: with both in one kernel the code of all roles did not stay in the instruction cache, and
// tiles waited for their longest row; P costs one write and one read of 4 bytes per input column and node, which the first
// kernel's arithmetic hides and the second is bound by.
//
// Measured, hidden layers of 2.45 M nodes and 126 M stored entries, all kernels of a layer: 100 -> 256 columns 5.0 -> 2.7 ms,
// 256 -> 256 columns 5.5 -> 4.0 ms (aggregation 2.0 and 3.1, contraction 0.7 and 0.85), against the contraction first and
// byte rows gathered.
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

__device__ int g_bits_timeout;                      // set when a bounded wait ran out

// ---- P -------------------------------------------------------------------------------------------------------------

// Entries of a row under one scale: their sum of |q| >> kMagShift fits 32 bits.  From kChainAny on, pieces whose largest weight is
// less than a quarter of the scale's start another, so that they are not rounded more coarsely for it.  (Up to three pieces
// whatever the row: 60,000 nodes in rows of 470, 256 inputs, one read-back for three pieces 506 us, 488 now.)
constexpr int kChain = 2048, kChainAny = 384, kMagShift = 10;
constexpr int kTileRows = 32;                       // rows of a tile of P
constexpr int kTileChunk = 128 * 128;               // bytes of 128 input columns of a tile: 32 rows x 4 digits x 128

struct AggDev {
    int n;                                          // n and entries + kRowCost n below 2^31
    const int64_t* rowptr;
    const int32_t* colidx;
    const float* val;
    const float* beta;
    const uint8_t* bits;                            // packed input rows
    uint32_t row_bytes;
    int first_byte;                                 // of the first slice of columns in a row
    int slices;                                     // slices of K columns
    int chunk_log2;                                 // entries + kRowCost per row and unit of work
    int chunks;                                     // units
    const int4* groups;                             // of all units: first entry, first row, entries | those of the first row << 8 | Flags << 16
    const int2* units;                              // per unit: its first group, how many
    uint8_t* p;                                     // tiles of [n_kc][32 rows x 4 digits][128 bytes], swizzled
    int n_kc, first_kc;
    float* row_scale;                               // what a row's integers stand for (the same for all of its slices)
    float* parts;                                   // [slices][chunks][2][K + 4]: pieces of rows cut by a unit's end, and their sum |w|
    unsigned* counters;                             // [slices][chunks] pieces done; zeroed before
};

constexpr int kMore = 64;                           // beside Flags, of a group in a slot: the next one adds to its products

// A row without a fixed point (by the exponent of its largest weight, of a whole row: of the largest of the lanes' sums) gets a scale
// whose exponent is zero, all ones or beyond, which marks it for literal_row(); what its integers are is of no account then.
__device__ __forceinline__ bool is_literal(float scale) { return __float_as_uint(scale) - 1u >= 0x7f7fffffu; }
__device__ __forceinline__ float max_nan(float a, float b)   // NaN if either is
{
    float r;
    asm("max.NaN.f32 %0, %1, %2;\n" : "=f"(r) : "f"(a), "f"(b));
    return r;
}

// Warps per block and resident blocks per multiprocessor: what the registers leave room for beside 64, 32 or 16 accumulators
// per lane.
__host__ __device__ constexpr int agg_warps(int k) { return k == 128 ? 10 : 8; }
__host__ __device__ constexpr int agg_blocks(int k) { return k > 64 ? 2 : 3; }

template <int K>
struct Slot {
    static constexpr int kRowBytes = K > 128 ? 32 : 16;
    uint8_t rows[kGroup * kRowBytes];               // the entries' packed rows; 32-byte rows: halves exchanged in every other four
    uint2 q[2][32][2];                              // [window / 2][entry][window % 2]: digits of the entry's weight under the group's two rows (0 under the other)
    int windows, flags, row, unit;
    int w0, w1;                                     // sums of q per row; a piece of a row: of the low and of the high digits of q
    uint32_t x0, x1;                                // what an integer stands for: 2^(x - 127); a piece: x1 = sum (|q| >> 8) + 1
};

__device__ __forceinline__ void imma(int (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k32.row.col.s32.u8.s8.s32 {%0,%1,%2,%3},{%4,%5,%6,%7},{%8,%9},{%0,%1,%2,%3};\n"
                 : "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// byte d of four words, for d = 0..3
__device__ __forceinline__ void transpose4(const uint32_t (&u)[4], uint32_t (&o)[4])
{
    const uint32_t a = __byte_perm(u[0], u[1], 0x5140), b = __byte_perm(u[2], u[3], 0x5140);
    const uint32_t c = __byte_perm(u[0], u[1], 0x7362), e = __byte_perm(u[2], u[3], 0x7362);
    o[0] = __byte_perm(a, b, 0x5410);
    o[1] = __byte_perm(a, b, 0x7632);
    o[2] = __byte_perm(c, e, 0x5410);
    o[3] = __byte_perm(c, e, 0x7632);
}

// ---- the split of the work: a property of the graph alone, made once per forward and shared by its layers.  A thread walks
// the rows of one unit -- positions [u, u + 1) << chunk_log2, where a row takes kRowCost positions and its entries -- and
// cuts them into groups: two whole rows where both fit a group, else one, else pieces of a row.  (Inside agg_bits_kernel
// the same walk took a quarter of its time: all 32 lanes of a warp on one chain of dependent steps.)
struct Walk {
    const int64_t* rowptr;
    int n, mb, me;
    int r, pos, hi;
    bool in_row, starts, ends;
    __device__ __forceinline__ int offset(int row) const { return (int)__ldg(rowptr + min(row, n)); }
    __device__ void begin(int unit, int chunk_log2)
    {
        mb = unit << chunk_log2;
        me = mb + min(1 << chunk_log2, 0x7fffffff - mb);
        int lo = 0, up = n;                         // the first row whose position is not before the unit's
        while (lo < up) {
            const int mid = lo + (up - lo) / 2;
            if (offset(mid) + kRowCost * mid >= mb) up = mid;
            else lo = mid + 1;
        }
        r = lo;
        if (lo > 0 && offset(lo) + kRowCost * lo > mb) r = lo - 1;   // the row before reaches into the unit
        in_row = false;
    }
    __device__ bool next(int4& g)
    {
        int flags = 0;
        if (!in_row) {
            if (r >= n) return false;
            const int a = offset(r), b = offset(r + 1), b2 = offset(r + 2);
            if (a + kRowCost * r >= me) return false;
            starts = a + kRowCost * r >= mb;
            ends = b + kRowCost * (r + 1) <= me;
            if (starts && ends && b - a <= kGroup) {
                const bool two = r + 1 < n && b2 - a <= kGroup && b2 + kRowCost * (r + 2) <= me;
                const int cnt = (two ? b2 : b) - a;
                g = make_int4(a, r, cnt | ((b - a) << 8) | ((kDirect | (two ? kPair : 0)) << 16), 0);
                r += two ? 2 : 1;
                return true;
            }
            pos = starts ? a : max(a, mb - kRowCost * (r + 1));
            hi = max(pos, ends ? b : min(b, me - kRowCost * (r + 1)));
            flags = kFirst;
        }
        const int cnt = min(kGroup, hi - pos);
        if (starts) flags |= kStarts;
        if (starts && ends) flags |= kWhole;
        in_row = pos + cnt < hi;
        if (!in_row) flags |= kLast;
        g = make_int4(pos, r, cnt | (cnt << 8) | (flags << 16), 0);
        pos += cnt;
        if (!in_row) r = ends ? r + 1 : n;          // the rest of the row belongs to later units
        return true;
    }
};

__global__ void __launch_bounds__(128) plan_kernel(const int64_t* __restrict__ rowptr, int n, int chunk_log2, int chunks,
                                                   int4* __restrict__ groups, int2* __restrict__ units, unsigned* __restrict__ used)
{
    pdl_enter();
    const int u = (int)(blockIdx.x * blockDim.x + threadIdx.x);
    if (u >= chunks) return;
    Walk w{rowptr, n};
    int4 g;
    int count = 0;
    w.begin(u, chunk_log2);
    const int r0 = w.r;
    while (w.next(g)) ++count;
    const int at = (int)atomicAdd(used, (unsigned)count);
    units[u] = make_int2(at, count);
    w.r = r0;
    w.in_row = false;
    for (int i = 0; i < count && w.next(g); ++i) groups[at + i] = g;
}

// Inside 128 columns P keeps the eight columns of byte c of the packed row at positions 16 (c % 8) + 8 (c / 8) + 0..7: what a
// lane holds after the products is then one run of bytes.  (bits_gemm_kernel orders the weights alike.)
template <int K>
__global__ void __launch_bounds__(32 * agg_warps(K), agg_blocks(K)) agg_bits_kernel(const AggDev d)
{
    pdl_enter();
    constexpr int kLaneBytes = K / 64;              // byte columns of a row that a lane takes: g, g + 8, ...
    constexpr int MT = K / 16;                      // 16-column products per window, and values per lane after the read-back
    constexpr int kAggWarps = agg_warps(K);
    constexpr int kRB = Slot<K>::kRowBytes, kHalves = kRB / 16;
    extern __shared__ __align__(128) unsigned char agg_smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = lane >> 2, t = lane & 3;
    const bool odd = t & 1;
    Slot<K>* const slots = reinterpret_cast<Slot<K>*>(agg_smem) + 2 * warp;
    float* const facc = reinterpret_cast<float*>(reinterpret_cast<Slot<K>*>(agg_smem) + 2 * kAggWarps) + K * warp;   // an open row's sums: value i of lane 4 g + odd at 16 i + 2 g + odd
    const uint32_t slot0 = smem_u32(slots);
    const uint32_t my_ld = kHalves == 2 ? (uint32_t)(lane * 32 + (((lane >> 2) & 1) << 4)) : (uint32_t)(lane * 16);

    // ---- this warp's units of work, group after group; a group is asked for one ahead
    int unit = (int)(blockIdx.x * kAggWarps + warp), where = 0;      // the unit after the one at hand; chunk | slice << 24 of that
    const int4* at = d.groups;                      // the group after the one asked for
    int left = 0;                                   // groups of the unit from the one asked for on
    int4 asked = make_int4(0, 0, 0, 0);
    auto offset = [&](int row) { return (int)__ldg(d.rowptr + row); };
    int g_s = 0, g_row = 0, g_meta = 0, g_where = 0;   // the group at hand: first entry, first row, entries | those of the first row << 8 | Flags << 16
    auto gen = [&]() -> bool {
        while (left == 0) {
            if (unit >= d.chunks * d.slices) return false;
            where = (unit / d.chunks) << 24 | unit % d.chunks;
            const int2 u = __ldg(d.units + (where & 0xffffff));
            at = d.groups + u.x;
            left = u.y;
            if (left > 0) asked = __ldg(at++);
            unit += (int)(gridDim.x * kAggWarps);
        }
        g_s = asked.x;
        g_row = asked.y;
        g_meta = asked.z;
        g_where = where;
        if (--left > 0) asked = __ldg(at++);
        return true;
    };

    int col[4];
    float w[4], bt[4];
    auto load = [&]() {
        const int g_cnt = g_meta & 255;
        // (lanes past the group's end take its last entry with weight 0: a column of their own choice, node 0 say, would send
        // every warp of the GPU to one sector of the L2)
        const int32_t* pc = d.colidx + g_s;
        const float* pv = d.val + g_s + lane;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            col[i] = 0;
            w[i] = 0.f;
            if (32 * i < g_cnt) col[i] = __ldg(pc + min(32 * i + lane, g_cnt - 1));
            if (32 * i + lane < g_cnt) w[i] = __ldg(pv + 32 * i);
        }
    };
    auto load_beta = [&]() {
#pragma unroll
        for (int i = 0; i < 4; ++i) bt[i] = __ldg(d.beta + col[i]);
    };
    int chain = 0;                                  // pieces of a long row: entries taken under one scale, and its exponent
    uint32_t chain_x = 0;
    // digits and copies of the rows of the group at hand, into slot k & 1
    auto publish = [&](int k) {
        Slot<K>* sl = slots + (k & 1);
        const int g_cnt = g_meta & 255, g_mid = (g_meta >> 8) & 255, g_flags = g_meta >> 16;
        // an instruction copies 16 rows of 32 bytes, two lanes each, or 32 rows of 16
        const int my_e = lane / kHalves;
        const uint32_t my_dst = kHalves == 2 ? (uint32_t)(my_e * 32 + (((lane & 1) ^ ((my_e >> 2) & 1)) << 4)) : (uint32_t)(lane * 16);
        const uint32_t my_src = kHalves == 2 ? (uint32_t)((lane & 1) << 4) : 0u;
        const uint32_t dst = slot0 + (uint32_t)((k & 1) * sizeof(Slot<K>)) + my_dst;
        const uint8_t* src = d.bits + min((uint32_t)(d.first_byte + (g_where >> 24) * (K / 8)) + my_src, d.row_bytes - 16u);   // (columns past the row's end have weight 0)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (32 * i >= g_cnt) break;
#pragma unroll
            for (int h = 0; h < kHalves; ++h) {
                const uint32_t c = (uint32_t)__shfl_sync(0xffffffffu, col[i], h * (32 / kHalves) + my_e);
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n"
                             ::"r"(dst + (uint32_t)((32 * i + h * (32 / kHalves)) * kRB)), "l"(src + (uint64_t)c * d.row_bytes) : "memory");
            }
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
#pragma unroll
        for (int i = 0; i < 4; ++i) w[i] *= bt[i];
        uint32_t x0, x1 = kExpLow, s0, s1 = 0;      // s: exponents of what an integer stands for
        int lc0 = 0, lc1 = 0;
        int flags = g_flags;
        if (flags & kDirect) {
            // Whole rows: q = round(w 2^(156 - lc - x)) with sum |w| <= 2^(x + lc - 126), so that sum |q| <= 2^30 (and a half per
            // entry) and a weight is off by 2^-30 of sum |w| at most, whatever share of it the largest has.  (A scale of
            // entries times the largest weight was off by 2^-24 of that.)  x is the exponent of the largest of the lanes' sums;
            // these are added up in units of 2^(x - 146), rounded up.
            float m0 = 0.f, m1 = 0.f;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (32 * i + lane < g_mid) m0 += fabsf(w[i]);
                else m1 += fabsf(w[i]);
            }
            auto scale = [](float m, uint32_t& x, uint32_t& s) {
                const uint32_t most = __reduce_max_sync(0xffffffffu, __float_as_uint(m));   // (as integers, NaN is the largest of all)
                x = max(most >> 23, kExpLow);
                if (x > kExpHigh) x = 320u;          // s from 271 on
                const unsigned t = __reduce_add_sync(0xffffffffu, (unsigned)__float2int_ru(m * __uint_as_float((273u - x) << 23)));
                const int lc = 12 - __clz((int)t - 1);   // -20 to 12 (a row of zeros); below -10, sum |w| < 2^-96, s is 0 or less
                s = x + lc - 29u;
                return lc;
            };
            lc0 = scale(m0, x0, s0);
            if (flags & kPair) lc1 = scale(m1, x1, s1);
        } else {
            // a piece of a row: |q| <= 2^30 by its largest weight.  The pieces of a unit share a scale (with 3 bits to spare for
            // larger weights) and one read-back, as long as none has a larger weight, or from kChainAny entries on much smaller ones
            // (weights too small for a fixed point count only where the whole row has no larger ones: finish())
            float m0 = 0.f;
#pragma unroll
            for (int i = 0; i < 4; ++i) m0 = max_nan(m0, fabsf(w[i]));
            x0 = max(__reduce_max_sync(0xffffffffu, __float_as_uint(m0)) >> 23, kExpLow);
            if (x0 > kExpHigh) x0 = 281u;           // bound infinite or NaN, also with 3 bits to spare
            if (!(flags & kFirst) && x0 <= chain_x && (chain + g_cnt <= kChainAny || (chain + g_cnt <= kChain && x0 + 5u >= chain_x))) {
                x0 = chain_x;
                chain += g_cnt;
                if (lane == 0) slots[(k & 1) ^ 1].flags |= kMore;
            } else {
                if (!(flags & kLast)) x0 += 3;
                chain_x = x0;
                chain = g_cnt;
            }
            s0 = x0 - 29u;
        }
        const float f0 = __uint_as_float((283u - lc0 - x0) << 23), f1 = __uint_as_float((283u - lc1 - x1) << 23);
        int w0 = 0, w1 = 0, mag = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (32 * i >= g_cnt) break;
            const bool a = 32 * i + lane < g_mid;
            const int q = __float2int_rn(w[i] * (a ? f0 : f1));
            const uint32_t dg = ((uint32_t)q + kFlip) ^ kFlip;
            sl->q[i >> 1][lane][i & 1] = make_uint2(a ? dg : 0u, a ? 0u : dg);
            if (flags & kDirect) {
                if (a) w0 += q;
                else w1 += q;
            } else {                                // q = 65536 hi + lo, lo its two low digits
                const int hi = (q + 0x8080) >> 16;
                w0 += q - hi * 65536;
                w1 += hi;
                mag += (abs(q) >> kMagShift) + 1;
            }
        }
        w0 = __reduce_add_sync(0xffffffffu, w0);
        if ((flags & (kDirect | kPair)) != kDirect) w1 = __reduce_add_sync(0xffffffffu, w1);
        if (!(flags & kDirect)) mag = __reduce_add_sync(0xffffffffu, mag);
        if (lane == 0) {
            *reinterpret_cast<int4*>(&sl->windows) = make_int4((g_cnt + 31) >> 5, flags, g_row, g_where);
            *reinterpret_cast<int4*>(&sl->w0) = make_int4(w0, w1, (int)s0, flags & kDirect ? (int)s1 : mag);
        }
    };
    auto tile_of = [&](int row, int pb) { return d.p + (int64_t)(row >> 5) * d.n_kc * kTileChunk + (d.first_kc + (pb >> 7)) * kTileChunk; };
    // facc -> digits of one row
    auto finish = [&](int row, int sli, float bound) {        // bound >= sum |w| of the row: the same for all slices
        __syncwarp();
        const uint32_t b = __float_as_uint(bound * 1.0009765625f), x = max(b >> 23, kExpLow);
        const float up = __uint_as_float((283u - x) << 23);   // |f| < 2^(x - 126): q = round(f 2^(156 - x))
        // values i .. i + V - 1 of lane 4 g' + odd', V = K / 32 of its MT
        constexpr int V = K / 32;
        const int go = lane >> 1, i0 = (lane & 1) * V;
        uint32_t o[4][(V + 3) / 4];
#pragma unroll
        for (int q4 = 0; q4 < (V + 3) / 4; ++q4) {
            uint32_t u[4], tr[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) u[i] = 4 * q4 + i < V ? ((uint32_t)__float2int_rn(facc[(i0 + (4 * q4 + i) % V) * 16 + go] * up) + kFlip) ^ kFlip : 0u;
            transpose4(u, tr);
#pragma unroll
            for (int i = 0; i < 4; ++i) o[i][q4] = tr[i];
        }
        const int pb = sli * K + (K == 256 ? (go & 1) * 128 : (go & 1) * MT) + (go >> 1) * 16 + i0;
        uint8_t* tile = tile_of(row, pb);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int nr = (row & 31) * 4 + i;
            uint8_t* dst = tile + nr * 128 + ((((pb & 127) >> 4) ^ (nr & 7)) << 4) + (pb & 15);
            if constexpr (V == 8) *reinterpret_cast<uint2*>(dst) = make_uint2(o[i][0], o[i][1]);
            else if constexpr (V == 4) *reinterpret_cast<uint32_t*>(dst) = o[i][0];
            else *reinterpret_cast<uint16_t*>(dst) = (uint16_t)o[i][0];
        }
        if (lane == 0) d.row_scale[row] = __uint_as_float((b < (kExpLow << 23) || b >= ((kExpHigh + 1) << 23) ? 0u : x - 29u) << 23);
        __syncwarp();
    };

    int c[MT][4];
    // one window: its rows at `rows`, b0 and b1 its digits
    auto compute = [&](uint32_t rows, uint32_t b0, uint32_t b1) {
#pragma unroll
        for (int h = 0; h < kHalves; ++h) {
            uint32_t a[4];
            ldmatrix_bytes(rows ^ (h ? 16u : 0u), a);
#pragma unroll
            for (int b = 0; b < (kLaneBytes > 1 ? 2 : 1); ++b)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const uint32_t ma = 0x01010101u << (2 * j), mb_ = 0x01010101u << (2 * j + 1);
                    imma(c[(h * 2 + b) * 4 + j], a[b] & ma, a[b] & mb_, a[2 + b] & ma, a[2 + b] & mb_, b0, b1);
                }
        }
    };

    // Three groups in flight: one is computed while the rows of the next are copied and the column indices and values of the
    // one after are loaded.
    bool have = gen();                              // the group at hand (in col, w, bt)
    if (have) {
        load();
        load_beta();
    }
    bool row_open = false;                          // facc holds sums of the row that the pieces belong to
    bool filled = false, more_of_row = false;       // the slot to compute holds a group; it adds to the products so far
    float bound = 0.f;                              // sum |w| of the open row
    int wlo = 0, whi = 0, wmag = 0;                 // of the pieces since the last read-back
    for (int k = 0;; ++k) {
        const bool more = have;
        if (have) {
            publish(k);
            have = gen();
            if (have) load();
        } else {
            asm volatile("cp.async.commit_group;\n" ::: "memory");
        }
        if (filled) {
            const Slot<K>* sl = slots + ((k - 1) & 1);
            const uint32_t sbase = slot0 + (uint32_t)(((k - 1) & 1) * sizeof(Slot<K>));
            asm volatile("cp.async.wait_group 1;\n" ::: "memory");
            __syncwarp();
            const int4 hd = *reinterpret_cast<const int4*>(&sl->windows), hw = *reinterpret_cast<const int4*>(&sl->w0);
            const int nw = hd.x, flags = hd.y;
            if (!more_of_row) {
#pragma unroll
                for (int i = 0; i < MT; ++i) c[i][0] = c[i][1] = c[i][2] = c[i][3] = 0;
                wlo = whi = wmag = 0;
            }
            uint32_t rows = sbase + my_ld, qs = sbase + (uint32_t)(kGroup * kRB) + (uint32_t)(lane * 16);
#pragma unroll 1
            for (int i = 0; i < nw; i += 2) {
                uint32_t b[4];
                ldmatrix_bytes(qs, b);
                compute(rows, b[0], b[2]);
                if (i + 1 < nw) compute(rows + 32 * kRB, b[1], b[3]);
                rows += 64 * kRB;
                qs += 512;
            }
            if (have) load_beta();
            more_of_row = flags & kMore;
            if (!(flags & kPair)) {
                wlo += hw.x;
                whi += hw.y;
                wmag += hw.w;
            }
            if (!more_of_row) {
                // read-back: a lane pair holds the low and the high digits of one row; each keeps half of the columns
                auto halves = [&](int i, int q, int& low, int& high) {           // sums over the entries whose bit is set
                    const int lo = c[i][2 * q + 1] * 256 + c[i][2 * q], up = c[i + MT / 2][2 * q + 1] * 256 + c[i + MT / 2][2 * q];
                    const int got = __shfl_xor_sync(0xffffffffu, odd ? lo : up, 1);
                    low = odd ? got : lo;
                    high = odd ? up : got;
                };
                const int row = hd.z + (t >> 1);
                const int sli = hd.w >> 24;
                if (flags & kDirect) {
                    // v = 2 sum_{bit = 1} q - sum q, biased by kFlip
                    const int base = (int)kFlip - (t >> 1 ? hw.y : hw.x);
                    uint32_t v[MT];
#pragma unroll
                    for (int i = 0; i < MT / 2; ++i) {
#pragma unroll
                        for (int q = 0; q < 2; ++q) {
                            int low, high, s;
                            halves(i, q, low, high);
                            if constexpr (K > 64) s = (low >> (2 * (i & 3) + q)) + high * (65536 >> (2 * (i & 3) + q));
                            else s = (low >> (2 * i + q + (odd ? 4 : 0))) + high * (odd ? 65536 >> (2 * i + q + 4) : 65536 >> (2 * i + q));
                            v[2 * i + q] = (uint32_t)(2 * s + base);
                        }
                    }
                    if ((flags & kPair) || t < 2) {
                        const int pb = sli * K + (K == 256 ? (odd ? 128 : 0) : (odd ? MT : 0)) + g * 16;
                        uint8_t* tile = tile_of(row, pb) + (pb & 15);
                        uint32_t o[4][MT / 4];
#pragma unroll
                        for (int q4 = 0; q4 < MT / 4; ++q4) {
                            uint32_t u[4], tr[4];
#pragma unroll
                            for (int i = 0; i < 4; ++i) u[i] = v[4 * q4 + i] ^ kFlip;
                            transpose4(u, tr);
#pragma unroll
                            for (int i = 0; i < 4; ++i) o[i][q4] = tr[i];
                        }
                        const int nr = (row & 31) * 4;
                        tile += nr * 128;
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            uint8_t* dst = tile + i * 128 + ((g ^ ((nr & 7) + i)) << 4);
                            if constexpr (MT == 16) *reinterpret_cast<uint4*>(dst) = make_uint4(o[i][0], o[i][1], o[i][2], o[i][3]);
                            else if constexpr (MT == 8) *reinterpret_cast<uint2*>(dst) = make_uint2(o[i][0], o[i][1]);
                            else *reinterpret_cast<uint32_t*>(dst) = o[i][0];
                        }
                        if (g == 0 && !odd) d.row_scale[row] = __uint_as_float((uint32_t)(t >> 1 ? hw.w : hw.z) << 23);
                    }
                } else {
                    // pieces of a row: added up in fp32
                    const float sc = __uint_as_float((uint32_t)hw.z << 23);
                    const bool first = !row_open;
                    row_open = true;
                    constexpr float kMag = (float)(1 << kMagShift);
                    bound = first ? (float)(unsigned)wmag * (kMag * sc) : fmaf((float)(unsigned)wmag, kMag * sc, bound);
                    float* f = facc + 2 * g + (odd ? 1 : 0);
#pragma unroll
                    for (int i = 0; i < MT / 2; ++i) {
#pragma unroll
                        for (int q = 0; q < 2; ++q) {
                            // (shifted before the digits are put together, so that kChain entries fit)
                            const int bit = K > 64 ? 2 * (i & 3) + q : 2 * i + q, bit_up = K > 64 ? bit : bit + 4;
                            const int lo = (c[i][2 * q + 1] >> bit) * 256 + (c[i][2 * q] >> bit);
                            const int up = (c[i + MT / 2][2 * q + 1] >> bit_up) * 256 + (c[i + MT / 2][2 * q] >> bit_up);
                            const int got = __shfl_xor_sync(0xffffffffu, odd ? lo : up, 1);
                            const float x = fmaf((float)(2 * (odd ? up : got) - whi), 65536.f, (float)(2 * (odd ? got : lo) - wlo)) * sc;
                            if (t < 2) f[16 * (2 * i + q)] = first ? x : x + f[16 * (2 * i + q)];
                        }
                    }
                    if (flags & kLast) {
                        row_open = false;
                        bool done = flags & kWhole;
                        const int rw = hd.z;
                        if (!done) {
                            // the row reaches over several units: leave this one's sums; whoever comes last adds them up in order
                            __syncwarp();
                            const int u0 = sli * d.chunks + ((offset(rw) + kRowCost * rw) >> d.chunk_log2);
                            const int u1 = sli * d.chunks + ((offset(rw + 1) + kRowCost * (rw + 1) - 1) >> d.chunk_log2);
                            float* part = d.parts + ((int64_t)(sli * d.chunks + (hd.w & 0xffffff)) * 2 + ((flags & kStarts) ? 1 : 0)) * (K + 4);
                            if (lane == 0) part[K] = bound;
#pragma unroll 1
                            for (int i = lane; i < K; i += 32) part[i] = facc[i];
                            __threadfence();
                            __syncwarp();
                            unsigned before = 0;
                            if (lane == 0) before = atomicAdd(d.counters + u0, 1u);
                            before = __shfl_sync(0xffffffffu, before, 0);
                            done = before == (unsigned)(u1 - u0);
                            if (done) {
                                __threadfence();
#pragma unroll 1
                                for (int i = lane; i < K + 32; i += 32) {
                                    const int j = min(i, K);
                                    float s = __ldcg(d.parts + ((int64_t)u0 * 2 + 1) * (K + 4) + j);
                                    for (int u = u0 + 1; u <= u1; ++u) s += __ldcg(d.parts + (int64_t)u * 2 * (K + 4) + j);
                                    if (j < K) facc[j] = s;
                                    else bound = s;
                                }
                            }
                        }
                        if (done) finish(rw, sli, bound);
                    }
                }
            }
        } else if (have) {
            load_beta();
        }
        if (!more) break;
        filled = true;
        __syncwarp();                               // the slot just read is filled next
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");
}

// ---- P B diag(alpha) -----------------------------------------------------------------------------------------------

constexpr int kGemmStages = 3;
constexpr int kOwnElts = 2 * kTileRows * 256;       // two tiles of up to 256 columns or four of up to 128
constexpr int kEpiGroups = 4;                       // warpgroups that read accumulators back
constexpr int kGemmThreads = 128 * kEpiGroups + 64; // + a copying and an issuing warp
constexpr int kTries = 1 << 20;                     // bound of a wait: tries of up to 1 us (a single one does not linger)

struct GemmMisc {
    uint64_t full[kGemmStages], empty[kGemmStages];
    uint64_t acc_full[4], acc_empty[4], own_full[4];
    alignas(16) float rows[16][2][kTileRows];       // per epilogue warp: row scales of the tile, and the nodes' own factors
    uint32_t tmem;
    int abort;
    alignas(16) uint32_t words[2][4][kTileRows][4]; // by turn, warpgroup: packed words of 32 rows, one per warp
    float l1[2][4][4][kTileRows];                   // sums of |x| likewise
};

__device__ __forceinline__ void mbar_init(uint64_t* bar, int count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar)
{
    asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(bar)) : "memory");
}
// false when the block gives up, which threads that wait for the same barrier may learn differently: one sees it complete,
// another the end of its tries
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, volatile int* abort, int tries)
{
    for (int it = 0; it < tries; ++it) {
        uint32_t done;
        asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.acquire.cta.shared::cta.b64 p, [%1], %2, %3;\nselp.u32 %0, 1, 0, p;\n}\n"
                     : "=r"(done) : "r"(smem_u32(bar)), "r"(parity), "r"(tries > 1 ? 1000u : 0u) : "memory");
        if (done) return true;
        if (*abort) return false;
    }
    atomicExch(&g_bits_timeout, 1);
    *abort = 1;
    return false;
}

// Waits for a copy or product of this thread's own before the block ends (bounded; at once unless the block gave up).
__device__ __forceinline__ void wait_landed(uint64_t* bar, uint32_t parity)
{
    uint32_t done = 0;
    for (int it = 0; it < kTries && !done; ++it)
        asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.acquire.cta.shared::cta.b64 p, [%1], %2, 1000;\nselp.u32 %0, 1, 0, p;\n}\n"
                     : "=r"(done) : "r"(smem_u32(bar)), "r"(parity) : "memory");
}
// A named barrier of `threads` threads that tells each whether all of them were ok.
__device__ __forceinline__ bool meet(int id, int threads, bool ok)
{
    uint32_t all;
    asm volatile("{\n.reg .pred p, q;\nsetp.ne.b32 p, %3, 0;\nbarrier.cta.red.and.aligned.pred q, %1, %2, p;\nselp.u32 %0, 1, 0, q;\n}\n"
                 : "=r"(all) : "r"(id), "r"(threads), "r"(ok ? 1u : 0u) : "memory");
    return all != 0;
}
__device__ __forceinline__ void copy_bulk(uint32_t dst, const void* src, uint32_t bytes, uint64_t* bar)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}

struct GemmDev {
    const uint8_t* p;
    int n_kc, d_in;
    const float* row_scale;
    const uint32_t* w_bits;
    int w_stride;
    int tiles;
    int tries;                                      // bound of the waits between the block's roles
    const int16_t* own;                             // kOwn: the nodes' own dots, rows of own_ld
    int own_ld;
    const float* own_alpha;
    const float* own_beta;
    const uint32_t* bits;                           // packed input rows of w_stride words
};

// One row by one warp, as it is written: every entry's integer dot with every channel times its weight, in fp32, then alpha, the
// node's own term, and what the epilogue does with a row.  For rows without a fixed point; speed does not matter.
__device__ __noinline__ void literal_row(const SpmmDev& p, const GemmDev& d, int64_t row, int lane)
{
    float acc[8];                                   // channels 32 t + lane
#pragma unroll
    for (int t = 0; t < 8; ++t) acc[t] = 0.f;
    const int kw = (d.d_in + 31) >> 5;
    const uint32_t last = 0xffffffffu >> (32 * kw - d.d_in);
    const int64_t end = __ldg(p.rowptr + row + 1);
    for (int64_t e = __ldg(p.rowptr + row); e < end; ++e) {
        const int c = __ldg(p.colidx + e);
        const float w = __ldg(p.val + e) * __ldg(p.node_w + c);
        const uint32_t* f = d.bits + (int64_t)c * d.w_stride;
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            const int ch = 32 * t + lane;
            if (ch >= p.d_out) break;
            int differ = 0;
            for (int k = 0; k < kw; ++k) differ += __popc((__ldg(f + k) ^ __ldg(d.w_bits + (int64_t)ch * d.w_stride + k)) & (k == kw - 1 ? last : 0xffffffffu));
            acc[t] = fmaf(w, (float)(d.d_in - 2 * differ), acc[t]);
        }
    }
    float l1 = 0.f;
#pragma unroll
    for (int t = 0; t < 8; ++t) {
        const int ch = 32 * t + lane;
        const bool in = ch < p.d_out;
        float x = 0.f, xh = 0.f;
        if (in) {
            x = acc[t] * __ldg(p.col_w + ch);
            if (d.own) x += __fmul_rn(__fmul_rn(__ldg(d.own_beta + row), __ldg(d.own_alpha + ch)), (float)d.own[row * d.own_ld + ch]);
            if (p.h_out) p.h_out[row * p.ldh + ch] = x;
            xh = p.next_shift ? __fmul_rn(__fsub_rn(x, __ldg(p.next_shift + ch)), __ldg(p.next_scale + ch)) : x;
            l1 += fabsf(xh);
        }
        if (p.next_bits && t < p.next_stride) {
            const uint32_t word = __ballot_sync(0xffffffffu, in && xh >= 0.f);
            if (lane == 0) p.next_bits[row * p.next_stride + t] = word;
        }
    }
    if (p.next_bits) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) l1 += __shfl_xor_sync(0xffffffffu, l1, o);
        if (lane == 0) p.next_beta[row] = l1 * p.inv_d_out;
    }
}

// NM: blocks of 128 output columns.  Accumulators: 4 / NM tiles in tensor memory, each with a warpgroup per block of columns.
// kOwn (Bi-GraphSAGE): the node's own term, beta_i alpha_j dot_ij, is added to the row.  Its dots come as 16-bit integers by bulk
// copies, a tile ahead of their use; read from fp32 rows by the epilogue itself, the latency of each read bounded the
// kernel (2.4 M rows of 256 columns: 4.9 ms against 0.9 ms without the term).
template <int NM, bool kBitsOnly, bool kOwn>
__global__ void __launch_bounds__(kGemmThreads, 1) bits_gemm_kernel(const SpmmDev p, const GemmDev d)
{
    pdl_enter();
    constexpr int kAcc = 4 / NM;
    extern __shared__ unsigned char gemm_raw[];
    unsigned char* sm = gemm_raw + ((1024u - (smem_u32(gemm_raw) & 1023u)) & 1023u);
    unsigned char* stages = sm;                                       // kGemmStages x kTileChunk
    unsigned char* a_op = stages + kGemmStages * kTileChunk;          // NM x [128 x 128 n_kc]
    int16_t* own_s = reinterpret_cast<int16_t*>(a_op + NM * 128 * 128 * d.n_kc);      // kAcc x [32 x own_ld]
    GemmMisc* m = reinterpret_cast<GemmMisc*>(own_s + (kOwn ? kOwnElts : 0));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    volatile int* abort = &m->abort;
    if (warp == 0) tc::tmem_alloc(&m->tmem, 512);
    if (threadIdx.x == 32) {
        for (int i = 0; i < kGemmStages; ++i) {
            mbar_init(&m->full[i], 1);
            mbar_init(&m->empty[i], 1);
        }
        for (int i = 0; i < 4; ++i) {
            mbar_init(&m->acc_full[i], 1);
            mbar_init(&m->acc_empty[i], 4 * NM);
            mbar_init(&m->own_full[i], 1);
        }
        m->abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    // the weights as +-1 bytes in the order of P's columns, 0 past d_in and d_out (the digits there are not written): positions
    // 16 c .. 16 c + 15 of 128 are the columns of bytes c and c + 8
    for (int it = threadIdx.x; it < NM * 128 * 8 * d.n_kc; it += kGemmThreads) {
        const int j = it % (NM * 128), kc = it / (NM * 128);
        uint32_t o[4] = {0u, 0u, 0u, 0u};
        if (j < p.d_out) {
            const int byte = (kc >> 3) * 16 + (kc & 7);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int cols = d.d_in - 8 * (byte + (q >> 1) * 8) - 4 * (q & 1);                  // columns left from this group of four on
                if (cols > 0) {
                    const uint32_t bits = reinterpret_cast<const uint8_t*>(d.w_bits + (int64_t)j * d.w_stride)[byte + (q >> 1) * 8] >> (4 * (q & 1));
                    const uint32_t set = ((bits & 15u) * 0x00204081u) & 0x01010101u;                // bit b -> byte b
                    o[q] = (0xffffffffu ^ (set * 0xfeu)) & (cols >= 4 ? 0xffffffffu : (1u << (8 * cols)) - 1u);   // 1 -> 0x01, 0 -> 0xff
                }
            }
        }
        *reinterpret_cast<uint4*>(a_op + (j >> 7) * (128 * 128 * d.n_kc) + tc::canon_off(128, j & 127, kc)) = make_uint4(o[0], o[1], o[2], o[3]);
    }
    tc::fence_async_smem();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = m->tmem;
    bool literal = false;                                             // a row of this warp's tiles is to be summed as it is written
    const int my_tiles = (int)blockIdx.x < d.tiles ? (d.tiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;

    if (warp == 4 * kEpiGroups) {                                     // copies
        if (lane == 0) {
            int s = 0;
            for (int i = 0; i < my_tiles; ++i) {
                const uint8_t* src = d.p + (int64_t)(blockIdx.x + i * gridDim.x) * d.n_kc * kTileChunk;
                bool ok = true;
                for (int kc = 0; kc < d.n_kc && ok; ++kc, ++s) {
                    const int st = s % kGemmStages;
                    if (s >= kGemmStages) ok = mbar_wait(&m->empty[st], (uint32_t)(s / kGemmStages + 1) & 1u, abort, d.tries);
                    if (!ok) break;
                    copy_bulk(smem_u32(stages + st * kTileChunk), src + (int64_t)kc * kTileChunk, kTileChunk, &m->full[st]);
                }
                if (!ok) break;
            }
            for (int q = max(0, s - kGemmStages); q < s; ++q) wait_landed(&m->full[q % kGemmStages], (uint32_t)(q / kGemmStages) & 1u);
        }
    } else if (warp == 4 * kEpiGroups + 1) {                          // products
        if (lane == 0) {
            // D = s32, A = B = s8, both K-major, N = 128, M = 128
            const uint32_t idesc = (2u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(128 >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
            const uint32_t a_base = smem_u32(a_op), s_base = smem_u32(stages);
            int s = 0, i = 0, owns = 0;
            for (; i < my_tiles; ++i) {
                const int acc = i % kAcc;
                if (i >= kAcc && !mbar_wait(&m->acc_empty[acc], (uint32_t)(i / kAcc + 1) & 1u, abort, d.tries)) break;
                if constexpr (kOwn) {
                    const int64_t r0 = (int64_t)(blockIdx.x + i * gridDim.x) * kTileRows;
                    const uint32_t bytes = (uint32_t)min((int64_t)kTileRows, p.n - r0) * (uint32_t)(2 * d.own_ld);
                    copy_bulk(smem_u32(own_s + acc * kTileRows * d.own_ld), d.own + r0 * d.own_ld, bytes, &m->own_full[acc]);
                    ++owns;
                }
                bool ok = true;
                for (int kc = 0; kc < d.n_kc; ++kc, ++s) {
                    const int st = s % kGemmStages;
                    ok = mbar_wait(&m->full[st], (uint32_t)(s / kGemmStages) & 1u, abort, d.tries);
                    if (!ok) break;
                    tc::fence_after_sync();
                    for (int h = 0; h < NM; ++h)
                        for (int ks = 0; ks < 4; ++ks) {
                            const uint64_t ad = tc::make_desc(a_base + h * (128 * 128 * d.n_kc) + (8 * kc + 2 * ks) * 2048, 2048, 128);
                            const uint64_t bd = tc::make_desc(s_base + st * kTileChunk + ks * 32, 16, 1024) | ((uint64_t)2 << 61);
                            asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n}\n"
                                         ::"r"(tmem + (uint32_t)((acc * NM + h) * 128)), "l"(ad), "l"(bd), "r"(idesc), "r"(kc + ks > 0 ? 1u : 0u) : "memory");
                        }
                    tc::commit_to(&m->empty[st]);
                }
                if (!ok) break;
                tc::commit_to(&m->acc_full[acc]);
            }
            // what was issued is done before the block frees its memory, also where the block gave up
            if (s > 0) wait_landed(&m->empty[(s - 1) % kGemmStages], (uint32_t)((s - 1) / kGemmStages) & 1u);
            for (int q = max(0, owns - kAcc); q < owns; ++q) wait_landed(&m->own_full[q % kAcc], (uint32_t)(q / kAcc) & 1u);
        }
    } else {                                                          // epilogue
        const int wg = warp >> 2, wq = warp & 3, h = wg % NM, acc = wg / NM;
        const int ch = 128 * h + 32 * wq + lane;
        const bool in = ch < p.d_out;
        const float alpha = in ? __ldg(p.col_w + ch) : 0.f;
        const float own_alpha = kOwn && in ? __ldg(d.own_alpha + ch) : 0.f;
        const float shift = (in && p.next_shift) ? __ldg(p.next_shift + ch) : 0.f;
        const float scale = in ? (p.next_shift ? __ldg(p.next_scale + ch) : 1.f) : 0.f;   // 0: columns that do not exist add nothing to beta
        const uint32_t t_addr = tmem + ((uint32_t)(32 * wq) << 16) + (uint32_t)((acc * NM + h) * 128);
        for (int i = acc; i < my_tiles; i += kAcc) {
            const int row0 = (int)(blockIdx.x + i * gridDim.x) * kTileRows, turn = (i / kAcc) & 1;
            const int my_row = (int)min((int64_t)row0 + lane, p.n - 1);
            const float scale_row = __ldg(d.row_scale + my_row);
            literal = literal || is_literal(scale_row);
            m->rows[warp][0][lane] = scale_row;
            if constexpr (kOwn) m->rows[warp][1][lane] = __ldg(d.own_beta + my_row);
            __syncwarp();
            bool ok = mbar_wait(&m->acc_full[acc], (uint32_t)(i / kAcc) & 1u, abort, d.tries);
            if constexpr (kOwn) ok = ok && mbar_wait(&m->own_full[acc], (uint32_t)(i / kAcc) & 1u, abort, d.tries);
            ok = __all_sync(0xffffffffu, ok);
            const int16_t* own = own_s + acc * kTileRows * d.own_ld + ch;
            uint32_t word = 0u;
            float l1_row = 0.f;                                       // lane r: the warp's sum of |x| over row r
            if (ok) {
                tc::fence_after_sync();
                auto four = [&](int rb, const uint32_t (&v)[16]) {        // four rows
                    float l1[4];
                    const float4 rs4 = *reinterpret_cast<const float4*>(&m->rows[warp][0][4 * rb]);
                    const float rs[4] = {rs4.x, rs4.y, rs4.z, rs4.w};
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        const int lo = (int)v[4 * r] + ((int)v[4 * r + 1] << 8), hi = (int)v[4 * r + 2] + ((int)v[4 * r + 3] << 8);
                        float x = fmaf((float)hi, 65536.f, (float)lo) * rs[r] * alpha;
                        if constexpr (kOwn) {
                            if (in) x += __fmul_rn(__fmul_rn(m->rows[warp][1][4 * rb + r], own_alpha), (float)own[(4 * rb + r) * d.own_ld]);
                        }
                        if constexpr (!kBitsOnly) {
                            const int row = row0 + 4 * rb + r;
                            if (row < p.n && in && p.h_out) p.h_out[(int64_t)row * p.ldh + ch] = x;
                        }
                        const float xh = __fmul_rn(__fsub_rn(x, shift), scale);
                        const uint32_t b = __ballot_sync(0xffffffffu, in && xh >= 0.f);
                        if (lane == 4 * rb + r) word = b;
                        l1[r] = fabsf(xh);
                    }
                    if (kBitsOnly || p.next_bits) {                       // four sums over the warp: lanes 4 q + r end with row r's
                        const bool b0 = lane & 1, b1 = lane & 2;
                        const float s0 = (b0 ? l1[1] : l1[0]) + __shfl_xor_sync(0xffffffffu, b0 ? l1[0] : l1[1], 1);
                        const float s1 = (b0 ? l1[3] : l1[2]) + __shfl_xor_sync(0xffffffffu, b0 ? l1[2] : l1[3], 1);
                        float s = (b1 ? s1 : s0) + __shfl_xor_sync(0xffffffffu, b1 ? s0 : s1, 2);
#pragma unroll
                        for (int o = 4; o < 32; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
                        if ((lane >> 2) == rb) l1_row = s;
                    }
                };
                // the next four's sums are on their way under the arithmetic of these, by loads without a condition: between a load and its
                // wait the registers must not pass a merge of control flow, where they may be copied (100 -> 256, 2.4 M rows: 681 -> 629 us; with 256
                // inputs the copies of P bound the kernel: 827 / 836, more of them in flight 852)
                uint32_t v[2][16];
                tc::tmem_ld16_nowait(t_addr, v[0]);
                tc::tmem_wait16(v[0]);
#pragma unroll 1
                for (int rb = 0; rb < kTileRows / 4; rb += 2) {
                    tc::tmem_ld16_nowait(t_addr + (uint32_t)(rb * 16 + 16), v[1]);
                    four(rb, v[0]);
                    tc::tmem_wait16(v[1]);
                    tc::tmem_ld16_nowait(t_addr + (uint32_t)(min(rb + 2, kTileRows / 4 - 2) * 16), v[0]);   // (the last one again)
                    four(rb + 1, v[1]);
                    tc::tmem_wait16(v[0]);
                }
                tc::fence_before_sync();
                __syncwarp();                                         // (also: rows[] is written again for the next tile)
                if (lane == 0) mbar_arrive(&m->acc_empty[acc]);
            }
            if (kBitsOnly || p.next_bits) {
                m->words[turn][wg][lane][wq] = word;
                m->l1[turn][wg][wq][lane] = l1_row;
                // the warps of an accumulator leave together: one that went on alone would wait here for the others
                if (!meet(1 + acc, 128 * NM, ok)) break;
                const int tid = 32 * wq + lane;
                if (tid < kTileRows && row0 + tid < p.n)              // this warpgroup's 128 columns of row tid
                    *reinterpret_cast<uint4*>(p.next_bits + (int64_t)(row0 + tid) * p.next_stride + 4 * h) = *reinterpret_cast<const uint4*>(m->words[turn][wg][tid]);
                if (h == 0 && tid >= 96 && row0 + lane < p.n) {
                    float s = (m->l1[turn][wg][0][lane] + m->l1[turn][wg][1][lane]) + (m->l1[turn][wg][2][lane] + m->l1[turn][wg][3][lane]);
                    if constexpr (NM == 2) s += (m->l1[turn][wg + 1][0][lane] + m->l1[turn][wg + 1][1][lane]) + (m->l1[turn][wg + 1][2][lane] + m->l1[turn][wg + 1][3][lane]);
                    p.next_beta[row0 + lane] = s * p.inv_d_out;
                }
            } else if (!ok) {
                break;
            }
        }
    }
    tc::fence_before_sync();
    literal = __syncthreads_or(literal) && !*abort;
    if (warp == 0) tc::tmem_free(m->tmem, 512);
    if (literal) {
        for (int i = warp; i < my_tiles; i += kGemmThreads / 32) {
            const int row0 = (int)(blockIdx.x + i * gridDim.x) * kTileRows;
            const bool mine = row0 + lane < p.n && is_literal(__ldg(d.row_scale + row0 + lane));
            for (unsigned todo = __ballot_sync(0xffffffffu, mine); todo; todo &= todo - 1) literal_row(p, d, row0 + __ffs(todo) - 1, lane);
        }
    }
}

int gemm_smem(int nm, int n_kc, bool own) { return kGemmStages * kTileChunk + nm * 128 * 128 * n_kc + (own ? kOwnElts * 2 : 0) + (int)sizeof(GemmMisc) + 1024; }

// How the work of agg_bits_kernel is split, and the scratch of a layer.
constexpr int kUnitsWanted = 4 * 16 * 148;           // four units for every warp that a B200 holds
struct Plan {
    int n_kc, chunk_log2, chunks, full;              // full: slices of 256 columns; rest: columns of a narrower last one (0: none)
    int rest;
    size_t groups_bytes, units_bytes;                // of the graph
    size_t p_bytes, scale_bytes, parts_bytes, counter_bytes;   // of a layer
    size_t graph_bytes() const { return groups_bytes + units_bytes; }
    size_t layer_bytes() const { return p_bytes + scale_bytes + parts_bytes + counter_bytes; }
};
size_t up256(size_t x) { return (x + 255) / 256 * 256; }
Plan make_plan(int64_t n, int64_t nnz, int d_in)
{
    Plan pl;
    pl.full = d_in / 256;
    pl.rest = d_in % 256;
    if (pl.rest > 128) {
        ++pl.full;
        pl.rest = 0;
    }
    pl.n_kc = (int)ceil_div(d_in, 128);
    // units of 256 to 2,048 positions: enough of them for four per resident warp where the graph is large enough, so that
    // dense rows and the last units do not leave warps idle; no larger, because a cut row costs two passes over its sums
    const int64_t positions = nnz + kRowCost * n;
    pl.chunk_log2 = 8;
    while (pl.chunk_log2 < 11 && (positions >> (pl.chunk_log2 + 1)) >= kUnitsWanted) ++pl.chunk_log2;
    pl.chunks = (int)std::max<int64_t>(1, ceil_div(positions, int64_t(1) << pl.chunk_log2));
    const int64_t units = (int64_t)pl.chunks * std::max(1, pl.full);
    pl.groups_bytes = up256((size_t)(n + nnz / kGroup + 2 * pl.chunks + 1) * sizeof(int4));
    pl.units_bytes = up256((size_t)pl.chunks * sizeof(int2) + 16);
    pl.p_bytes = up256((size_t)ceil_div(n, kTileRows) * pl.n_kc * kTileChunk);
    pl.scale_bytes = up256((size_t)round_up(n, kTileRows) * 4);
    pl.parts_bytes = up256((size_t)units * 2 * (256 + 4) * 4);
    pl.counter_bytes = up256((size_t)(units + pl.chunks) * 4);
    return pl;
}

}  // namespace

bool spmm_bits_covers(int64_t n, int64_t nnz, int d_in, int d_out, bool own)
{
    const int64_t row_bytes = round_up(ceil_div(d_in, 32), 4) * 4;
    return d_out <= 256 && n * row_bytes < (int64_t(1) << 32) && nnz + kRowCost * (n + 2) < (int64_t(1) << 31) - 4096 &&
           gemm_smem(d_out > 128 ? 2 : 1, (int)ceil_div(d_in, 128), own) <= 227 * 1024;
}

// Predicted picoseconds on one B200, fitted to hidden layers (bits and beta wanted) of d_in 64..602, d_out 16..256 on graphs of
// 20,000 to 2,400,000 nodes with 4 to 490 entries a row; the model is within 15 % of nearly all of them.  This order pays
// per stored entry and input column and, above all, per row (the read-back of P and the second kernel); the other per
// stored entry and output column.  So this one is the better for long rows and wide outputs (256 -> 256, 28 M entries in
// rows of 490: 0.56 against 1.12 ms), the other for short rows (256 -> 256, 2.6 M entries in rows of 15: 0.30 against 0.21 ms).
bool spmm_bits_pays(int64_t n, int64_t nnz, int d_in, int d_out)
{
    if (d_out <= 32) return false;                   // level at best
    const int full = d_in / 256 + (d_in % 256 > 128 ? 1 : 0), rest = d_in % 256 > 128 ? 0 : d_in % 256;
    const double here_entry = 15.0 * full + (rest == 0 ? 0.0 : (rest > 64 ? 10.0 : 8.0));
    const double here_row = 800.0 * full + (rest == 0 ? 0.0 : 520.0) + (d_out > 128 ? 230.0 : 0.0);
    double there_entry, there_row;
    if (d_out > 128 && d_in > 256) {                 // fp16 rows, in the L2 or not
        there_entry = (double)n * d_out * 2 <= 125e6 ? 48.0 : 63.0;
        there_row = 1100.0;
    } else if (d_out > 128) {
        there_entry = 32.0;
        there_row = nnz >= 8 * n ? 550.0 : 800.0;
    } else if (d_out > 64) {
        there_entry = 36.0;
        there_row = d_in > 256 ? 720.0 : 290.0;
    } else {
        there_entry = d_in > 256 ? 24.0 : 15.0;
        there_row = d_in > 256 ? 500.0 : 680.0;
    }
    return 65e6 + here_entry * nnz + here_row * n < 0.95 * (10e6 + there_entry * nnz + there_row * n);
}

groups::GraphPlan spmm_bits_plan_at(int64_t n, int64_t nnz, const void* plan)
{
    const Plan pl = make_plan(n, nnz, 1);
    return {pl.chunk_log2, pl.chunks, static_cast<const int4*>(plan), reinterpret_cast<const int2*>(static_cast<const char*>(plan) + pl.groups_bytes)};
}
size_t spmm_bits_plan_bytes(int64_t n, int64_t nnz) { return make_plan(n, nnz, 1).graph_bytes(); }
size_t spmm_bits_scratch_bytes(int64_t n, int64_t nnz, int d_in) { return make_plan(n, nnz, d_in).layer_bytes(); }

cudaError_t launch_spmm_bits_plan(cudaStream_t s, int64_t n, int64_t nnz, const int64_t* rowptr, void* plan, int* launches)
{
    if (n == 0) return cudaSuccess;
    const Plan pl = make_plan(n, nnz, 1);
    char* base = static_cast<char*>(plan);
    int2* units = reinterpret_cast<int2*>(base + pl.groups_bytes);
    unsigned* used = reinterpret_cast<unsigned*>(base + pl.graph_bytes() - 16);
    const cudaError_t e = cudaMemsetAsync(used, 0, 4, s);
    if (e != cudaSuccess) return e;
    launch_kernel(plan_kernel, (unsigned)ceil_div(pl.chunks, 128), 128, 0, s, rowptr, (int)n, pl.chunk_log2, pl.chunks, reinterpret_cast<int4*>(base), units, used);
    if (launches) ++*launches;
    return cudaGetLastError();
}

cudaError_t launch_spmm_bits(cudaStream_t s, const SpmmArgs& a, const void* plan, const uint32_t* bits, int64_t stride, int d_in,
                             const uint32_t* w_bits, const OwnTerm* own, int* launches, cudaEvent_t between)
{
    if (a.n == 0) return cudaSuccess;
    const Plan pl = make_plan(a.n, a.nnz, d_in);
    char* base = static_cast<char*>(a.scratch);
    AggDev g = {};
    g.n = (int)a.n;
    g.rowptr = a.rowptr;
    g.colidx = a.colidx;
    g.val = a.val;
    g.beta = a.node_w;
    g.bits = reinterpret_cast<const uint8_t*>(bits);
    g.row_bytes = (uint32_t)(stride * 4);
    g.chunk_log2 = pl.chunk_log2;
    g.chunks = pl.chunks;
    g.groups = static_cast<const int4*>(plan);
    g.units = reinterpret_cast<const int2*>(static_cast<const char*>(plan) + pl.groups_bytes);
    g.p = reinterpret_cast<uint8_t*>(base);
    g.n_kc = pl.n_kc;
    g.row_scale = reinterpret_cast<float*>(base + pl.p_bytes);
    g.parts = reinterpret_cast<float*>(base + pl.p_bytes + pl.scale_bytes);
    unsigned* counters = reinterpret_cast<unsigned*>(base + pl.p_bytes + pl.scale_bytes + pl.parts_bytes);
    cudaError_t e = cudaMemsetAsync(counters, 0, pl.counter_bytes, s);
    if (e != cudaSuccess) return e;
    auto agg = [&](auto k) -> cudaError_t {
        constexpr int K = decltype(k)::value;
        constexpr int kAggWarps = agg_warps(K);
        const int smem = kAggWarps * (2 * (int)sizeof(Slot<K>) + K * 4);
        cudaError_t err = cudaFuncSetAttribute(agg_bits_kernel<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (err != cudaSuccess) return err;
        const unsigned grid = (unsigned)std::min<int64_t>(ceil_div((int64_t)g.chunks * g.slices, kAggWarps), (int64_t)sm_count() * agg_blocks(K));
        launch_kernel(agg_bits_kernel<K>, grid, 32 * kAggWarps, smem, s, g);
        if (launches) ++*launches;
        return cudaGetLastError();
    };
    if (pl.full) {
        g.slices = pl.full;
        g.counters = counters;
        if ((e = agg(std::integral_constant<int, 256>())) != cudaSuccess) return e;
    }
    if (pl.rest) {
        g.slices = 1;
        g.first_byte = 32 * pl.full;
        g.first_kc = 2 * pl.full;
        g.counters = counters + (size_t)pl.chunks * pl.full;
        if ((e = pl.rest > 64 ? agg(std::integral_constant<int, 128>()) : agg(std::integral_constant<int, 64>())) != cudaSuccess) return e;
    }
    if (between && (e = cudaEventRecord(between, s)) != cudaSuccess) return e;

    SpmmDev p = {};
    p.n = a.n;
    p.rowptr = a.rowptr;
    p.colidx = a.colidx;
    p.val = a.val;
    p.node_w = a.node_w;
    p.d_out = a.d_out;
    p.col_w = a.col_w;
    p.h_out = a.h_out;
    p.ldh = a.ldh;
    p.next_bits = a.next_bits;
    p.next_stride = a.next_stride;
    p.next_beta = a.next_beta;
    p.next_shift = a.next_shift;
    p.next_scale = a.next_scale;
    p.inv_d_out = 1.f / (float)a.d_out;
    GemmDev d = {};
    d.p = g.p;
    d.n_kc = pl.n_kc;
    d.d_in = d_in;
    d.row_scale = g.row_scale;
    d.w_bits = w_bits;
    d.w_stride = (int)stride;
    d.tiles = (int)ceil_div(a.n, kTileRows);
    d.tries = a.wait_tries > 0 ? std::min(a.wait_tries, kTries) : kTries;
    d.own = own ? own->dots : nullptr;
    d.own_ld = own ? (int)own->ld : 0;
    d.own_alpha = own ? own->alpha : nullptr;
    d.own_beta = a.node_w;
    d.bits = bits;
    const int nm = a.d_out > 128 ? 2 : 1;
    const int smem = gemm_smem(nm, pl.n_kc, own != nullptr);
    const bool bits_only = p.next_bits && !p.h_out;
    auto gemm = [&](auto kernel) -> cudaError_t {
        cudaError_t err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (err != cudaSuccess) return err;
        launch_kernel(kernel, (unsigned)std::min(d.tiles, sm_count()), kGemmThreads, smem, s, p, d);
        if (launches) ++*launches;
        return cudaGetLastError();
    };
    if (own) {
        if (nm == 2) return bits_only ? gemm(bits_gemm_kernel<2, true, true>) : gemm(bits_gemm_kernel<2, false, true>);
        return bits_only ? gemm(bits_gemm_kernel<1, true, true>) : gemm(bits_gemm_kernel<1, false, true>);
    }
    if (nm == 2) return bits_only ? gemm(bits_gemm_kernel<2, true, false>) : gemm(bits_gemm_kernel<2, false, false>);
    return bits_only ? gemm(bits_gemm_kernel<1, true, false>) : gemm(bits_gemm_kernel<1, false, false>);
}

int spmm_bits_timeouts()
{
    int v = 0;
    if (cudaMemcpyFromSymbol(&v, g_bits_timeout, sizeof(int)) != cudaSuccess) return -1;
    return v;
}

}  // namespace bigcn

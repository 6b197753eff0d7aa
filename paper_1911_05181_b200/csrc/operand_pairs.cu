// A caller's fp32 operands as fp16 pairs (common.cuh), for products whose operands may mix magnitudes along the sum.
//
// A TF32 pair keeps 22 bits of any value; an fp16 pair keeps them of a scaled value x' = s*x with 2^-3 <= |x'| < 65504 and is off by
// at most 2^-25 below.  One scale serves a row of op(A), or a column of op(B): all that stands in one sum.  So a value that is faint beside
// the rest of its row may lose bits, and whether that matters depends on what the other operand multiplies it with.  The conversion counts,
// for every row of op(A) and column of op(B),
//     faint   values not 0 with |x'| < 2^-3
//     low     values with |x'| < 2^7, zeros among them
// and the product may be formed from the pairs if for the largest counts of both operands (rows and columns without a value do not count)
//     4 (faint_A + faint_B) <= K - low_A - low_B   or   faint_A + faint_B = 0,
// and every value is finite and below 65504.  For then, of any entry of the product, what the faint values lose is at most
// 2^-25 2^16 (faint_A + faint_B), while at least K - low_A - low_B of its terms are 2^14 or more: the loss is below 2^-25 of the sum of the
// terms' magnitudes, an eighth of the rounding of a pair itself and half of what one addition in 32 bits may round.  Where the test fails (values of very different size along a sum, mostly zeros on
// both sides, infinities, not-a-numbers) the product is formed from TF32 pairs as before.  Both ways are launched; the
// verdict stays on the device, and the kernels of the way not taken return at once.
//
// Operands that fail should not pay for a conversion that nobody reads (480 x 3203 x 65536: 380 us).  So the first blocks to run leave what they have
// counted of whole rows, or expect of columns from the sample that these are scaled after, and all blocks stop as soon as the test above cannot be met
// by that, or a value has been found that decides it.  The verdict is "no" wherever these expectations miss the test, whether or not a
// block was late enough to stop for it: it depends on the operands alone.  Calls whose operands fail, over the same without the conversion,
// before and after (half zeros, log-normal, one infinity): 480 x 3203 x 65536 1.35-1.37 / 1.05-1.10, 4096^3 1.16 / 1.06-1.09, 2304^3 1.32 / 1.20-1.23, 16000 x 480 x 3203
// 1.42 / 1.11-1.12, 8192^3 1.05 / 0.99-1.01; operands that pass 0.92-1.02 of the time before, as the operands' blocks run in turn.
//
// Bound by memory: every value is read once and written once as four bytes (rows whose scale needs their own largest value: read
// twice beyond the first 8192, the second time from L2).  Where the sums run across the stored rows, the scale of a column comes
// from up to 64 of its rows, spread evenly, with three bits to spare: its largest value over all rows would take a pass of its own.
#include "common.cuh"

namespace ulsnn {

namespace {

constexpr int STRIP = 256;                  // columns of a strip: eight per lane
constexpr int MOST_ROWS = 512;
constexpr int SAMPLE = 64;                  // rows
constexpr int EARLY = 64;                   // blocks that leave the counts of their first rows
constexpr int RESIDENT = 148 * 3;           // blocks that run from the start
constexpr uint32_t SPARE_BITS = 2;          // a sampled maximum is scaled to 2^12 .. 2^13 instead of 2^14 .. 2^15
constexpr float OVER = 65504.f, FAINT_VALUE = 0.125f, LOW_VALUE = 128.f;

__device__ __forceinline__ uint32_t magnitude(float x) { return __float_as_uint(x) & 0x7FFFFFFFu; }

struct Params {
    OperandPair m[2];
    int blocks[2];
    int rows_per_block[2];                  // conversion across stored rows
    int warps_per_row[2];                   // conversion along stored rows: 1, 2, 4 or 8
    uint64_t sample_step[2];                // rows from one sampled row to the next, times 65536
    uint32_t* state;                        // OPERAND_PAIR_WORDS words
    int64_t K;
};
// words of `state`: the verdict, a ticket, then for each operand that is scaled by its rows the largest counts of faint and of low values,
// eight words for the parts of a row, for each that is scaled by its columns the same two counts as the sample has them, and whether to go on
enum : int { VERDICT = 0, TICKET = 1, LARGEST = 2, EXPECTED = 34, OUTLOOK = 38 };
static_assert(OUTLOOK + 1 == OPERAND_PAIR_WORDS, "words");
enum : uint32_t { GO_ON = 0, ANY_FAINT_DECIDES = 1, STOP = 2 };     // values of OUTLOOK

// What the counts left so far allow: they only grow, and so does this.
__device__ uint32_t outlook(const Params& p) {
    const volatile uint32_t* state = p.state;
    int64_t faint = 0, low = 0;
    for (int w = 0; w < 2; ++w) {
        if (!p.m[w].per_row) { faint += state[EXPECTED + 2 * w]; low += state[EXPECTED + 2 * w + 1]; continue; }
#pragma unroll
        for (int i = 0; i < 8; ++i) { faint += state[LARGEST + 16 * w + i]; low += state[LARGEST + 16 * w + 8 + i]; }
    }
    if (faint > 0 && 4 * faint > p.K - low) return STOP;
    return p.K <= low ? ANY_FAINT_DECIDES : GO_ON;
}
__device__ void look_out(const Params& p) {        // by one thread, after its block's counts
    __threadfence();
    const uint32_t o = outlook(p);
    if (o != GO_ON) atomicMax(p.state + OUTLOOK, o);
}
__device__ __forceinline__ uint32_t current_outlook(const Params& p) { return *(const volatile uint32_t*)(p.state + OUTLOOK); }

// Everything that the conversion counts in set to 0
__global__ void __launch_bounds__(256) operand_start_kernel(const Params p) {
    chain_wait();
    if (blockIdx.x == 0 && threadIdx.x < OPERAND_PAIR_WORDS) p.state[threadIdx.x] = 0u;
    for (int w = 0; w < 2; ++w)
        if (!p.m[w].per_row)
            for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < 3 * p.m[w].cols; i += (int64_t)gridDim.x * 256) p.m[w].counts[i] = 0u;
}

// eight consecutive values of a row from column c0 on, zeros behind the row
__device__ __forceinline__ void load8(const float* s, int64_t c0, int64_t cols, bool vec, float (&v)[8]) {
    if (vec && c0 + 8 <= cols) {
        const float4 a = chain_ld(reinterpret_cast<const float4*>(s)), b = chain_ld(reinterpret_cast<const float4*>(s + 4));
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
    } else {
#pragma unroll
        for (int t = 0; t < 8; ++t) v[t] = c0 + t < cols ? chain_ld(s + t) : 0.f;
    }
}
__device__ __forceinline__ void store8(__half* dst, int64_t plane, const float (&v)[8]) {
    uint32_t h[4], l[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) split_pair(v[2 * t], v[2 * t + 1], h[t], l[t]);
    *reinterpret_cast<uint4*>(dst) = make_uint4(h[0], h[1], h[2], h[3]);
    *reinterpret_cast<uint4*>(dst + plane) = make_uint4(l[0], l[1], l[2], l[3]);
}

// Rows that are summed along: G warps take a row, once for its largest value and once to write it.  The counts of a row are bounded by the
// sum, over its G parts, of the largest count of any row's such part.
template <int G>
__device__ void convert_rows(const Params& p, const OperandPair& m, int which, int block) {
    __shared__ uint32_t red[2][8], counts[2][8], seen[2];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, part = warp % G;
    const bool vec = (((uintptr_t)m.src) & 15) == 0 && (m.lds & 3) == 0;
    constexpr int HELD = 4;
    uint32_t faint_most = 0, low_most = 0, unfit = 0, turn = 0;
    const int64_t step = (int64_t)p.blocks[which] * (8 / G);
    auto leave_counts = [&] {           // a word per part, operand and count
        if (lane == 0) { counts[0][warp] = faint_most; counts[1][warp] = low_most; }
        __syncthreads();
        if (threadIdx.x < 2 * G) {
            const int kind = threadIdx.x / G, of = threadIdx.x % G;
            uint32_t most = 0;
#pragma unroll
            for (int w = of; w < 8; w += G) most = max(most, counts[kind][w]);
            if (most) atomicMax(p.state + LARGEST + 16 * which + 8 * kind + of, most);
        }
    };
    for (int64_t r0 = (int64_t)block * (8 / G); r0 < m.rows; r0 += step, turn ^= 1u) {
        uint32_t go = (G > 1 ? threadIdx.x : lane) == 0 ? current_outlook(p) : 0u;
        const int64_t r = r0 + warp / G;
        const int64_t width = r < m.rows ? (m.cols + 7) / 8 * 8 : 0;
        const float* s = m.src + r * m.lds;
        const int64_t first = 8 * (lane + 32 * part), stride = 256 * G;
        float held[HELD][8];
        uint32_t mx = 0;
        auto largest = [&](const float (&x)[8]) {
#pragma unroll
            for (int t = 0; t < 8; ++t) mx = finite_max(mx, magnitude(x[t]));
        };
#pragma unroll
        for (int k = 0; k < HELD; ++k) { const int64_t c0 = first + stride * k; if (c0 < width) load8(s + c0, c0, m.cols, vec, held[k]); }
#pragma unroll
        for (int k = 0; k < HELD; ++k) if (first + stride * k < width) largest(held[k]);
#pragma unroll 2
        for (int64_t c0 = first + stride * HELD; c0 < width; c0 += stride) {
            float v[8];
            load8(s + c0, c0, m.cols, vec, v);
            largest(v);
        }
        mx = __reduce_max_sync(0xffffffffu, mx);
        if (G > 1) {
            if (lane == 0) red[turn][warp] = mx;
            if (threadIdx.x == 0) seen[turn] = go;
            __syncthreads();
#pragma unroll
            for (int w = 0; w < G; ++w) mx = max(mx, red[turn][warp / G * G + w]);
            go = seen[turn];
        } else {
            go = __shfl_sync(0xffffffffu, go, 0);
        }
        if (go == STOP && r0 >= step) break;        // all warps of a block write their first rows: they meet after them
        uint32_t faint = 0, low = 0;
        const float scale = pair_scale(mx);
        auto write = [&](int64_t c0, const float (&x)[8]) {
            float v[8];
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                v[t] = x[t] * scale;
                const float a = fabsf(v[t]);
                unfit |= !(a < OVER) ? 1u : 0u;
                low += a < LOW_VALUE && c0 + t < m.cols ? 1u : 0u;
                faint += a < FAINT_VALUE && magnitude(x[t]) != 0u ? 1u : 0u;
            }
            store8(m.dst + r * m.ld + c0, m.plane, v);
        };
#pragma unroll
        for (int k = 0; k < HELD; ++k) { const int64_t c0 = first + stride * k; if (c0 < width) write(c0, held[k]); }
#pragma unroll 2
        for (int64_t c0 = first + stride * HELD; c0 < width; c0 += stride) {
            float v[8];
            load8(s + c0, c0, m.cols, vec, v);
            write(c0, v);
        }
        if (lane == 0 && part == 0 && r < m.rows) m.max_bits[r] = mx;
        faint = __reduce_add_sync(0xffffffffu, faint); low = __reduce_add_sync(0xffffffffu, low);
        if (mx != 0u) { faint_most = max(faint_most, faint); low_most = max(low_most, low); }
        if (__any_sync(0xffffffffu, unfit != 0u || (go == ANY_FAINT_DECIDES && faint != 0u)) && lane == 0) atomicMax(p.state + OUTLOOK, (uint32_t)STOP);
        if (block < EARLY && r0 < step) {       // its first rows
            leave_counts();
            __syncthreads();
            if (threadIdx.x == 0) look_out(p);
        }
    }
    __syncthreads();
    leave_counts();
}

// Rows that are summed across: a block takes a strip of columns through a run of the rows, a warp every eighth of them.  A lane has eight
// neighbouring columns where the rows can be read 16 bytes at a time, else every 32nd: eight reads of single values that are neighbours in
// a lane take 70 cycles of the load unit per KB, and 16 when they are neighbours across the warp.
struct Strip {
    uint32_t counts[8][STRIP];              // low values in the lower half, faint ones in the upper; runs are at most MOST_ROWS rows
    uint32_t any[STRIP];
    uint32_t exponents[2][8][STRIP];        // of the sampled values, four of a column to a word
    uint32_t low[8], faint[8], columns[8], told;
};
template <bool VEC>
__device__ void convert_columns(const Params& p, const OperandPair& m, int which, int block, Strip& strip) {
    auto& counts = strip.counts;
    auto& any = strip.any;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int strips = (int)((m.cols + STRIP - 1) / STRIP);
    const int64_t c0 = (int64_t)(block % strips) * STRIP + (VEC ? 8 * lane : lane);
    const int64_t r0 = (int64_t)(block / strips) * p.rows_per_block[which], r1 = min(m.rows, r0 + p.rows_per_block[which]);
    const int64_t width = (m.cols + 7) / 8 * 8;
    constexpr int APART = VEC ? 1 : 32;             // from one of a lane's columns to the next
    any[threadIdx.x] = 0u;
    if (threadIdx.x == 0) strip.told = 0u;
    uint32_t count[8] = {0, 0, 0, 0, 0, 0, 0, 0}, unfit = 0, some = 0;
    auto load = [&](int64_t r, float (&x)[8]) {
        const float* s = m.src + r * m.lds + c0;
        if (VEC) load8(s, c0, m.cols, true, x);
        else {
#pragma unroll
            for (int t = 0; t < 8; ++t) x[t] = c0 + 32 * t < m.cols ? chain_ld(s + 32 * t) : 0.f;
        }
    };
    // the columns' scales, from the sample: every block of the strip comes to the same ones
    const int first = VEC ? 8 * lane : lane;
    {
        const int sample = m.rows < SAMPLE ? (int)m.rows : SAMPLE;
        uint32_t mx[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll 1
        for (int part = 0; part < 2; ++part) {
            const int i = warp + 32 * part;
            uint32_t e[8];
#pragma unroll
            for (int t = 0; t < 8; ++t) e[t] = 0xFEFEFEFEu;        // neither faint nor low: no value
            if (i < sample) {
                float x[4][8];
#pragma unroll
                for (int k = 0; k < 4; ++k) load((int64_t)((uint64_t)min(i + 8 * k, sample - 1) * p.sample_step[which] >> 16), x[k]);
#pragma unroll
                for (int k = 0; k < 4; ++k)
#pragma unroll
                    for (int t = 0; t < 8; ++t) {
                        const uint32_t a = magnitude(x[k][t]);
                        mx[t] = finite_max(mx[t], a);
                        if (i + 8 * k < sample) e[t] = __byte_perm(e[t], a >> 23, k == 0 ? 0x3214 : k == 1 ? 0x3240 : k == 2 ? 0x3410 : 0x4210);
                    }
            }
            if (block < strips)
#pragma unroll
                for (int t = 0; t < 8; ++t) strip.exponents[part][warp][first + APART * t] = e[t];
        }
#pragma unroll
        for (int t = 0; t < 8; ++t) counts[warp][first + APART * t] = mx[t];
        __syncthreads();
        uint32_t most = 0;
#pragma unroll
        for (int w = 0; w < 8; ++w) most = max(most, counts[w][threadIdx.x]);
        if (block < strips) {       // what to expect of the strip's columns: scaled values are below 2^(e - (most + SPARE_BITS) + 15)
            uint32_t low = 0, faint = 0;
            const uint32_t field = (most >> 23) + SPARE_BITS;
            const uint32_t below_low = 0x01010101u * (field > 7 ? min(field - 7, 253u) : 0u), below_faint = 0x01010101u * (field > 17 ? min(field - 17, 253u) : 0u);
            if (most)
#pragma unroll
                for (int part = 0; part < 2; ++part)
#pragma unroll
                    for (int w = 0; w < 8; ++w) {
                        const uint32_t e = strip.exponents[part][w][threadIdx.x];
                        low += __popc(__vcmpltu4(e, below_low)) >> 3;
                        faint += __popc(__vcmpltu4(e, below_faint) & __vcmpne4(e, 0u)) >> 3;
                    }
            const uint32_t columns = __reduce_add_sync(0xffffffffu, most ? 1u : 0u);
            low = __reduce_add_sync(0xffffffffu, low); faint = __reduce_add_sync(0xffffffffu, faint);
            if (lane == 0) { strip.low[warp] = low; strip.faint[warp] = faint; strip.columns[warp] = columns; }
        }
        most = (most ? min((most >> 23) + SPARE_BITS, 254u) : 127u) << 23;      // nothing but zeros seen: as if the largest were 1
        __syncthreads();
        if (block < strips && threadIdx.x == 0) {
            uint64_t low = 0, faint = 0, columns = 0;
#pragma unroll
            for (int w = 0; w < 8; ++w) { low += strip.low[w]; faint += strip.faint[w]; columns += strip.columns[w]; }
            if (columns) {
                const uint64_t of = columns * (uint64_t)sample;
                if (faint) atomicMax(p.state + EXPECTED + 2 * which, (uint32_t)((uint64_t)m.rows * faint / of));
                if (low) atomicMax(p.state + EXPECTED + 2 * which + 1, (uint32_t)((uint64_t)m.rows * low / of));
            }
            look_out(p);
        }
        counts[0][threadIdx.x] = most;
        const int64_t c = (int64_t)(block % strips) * STRIP + threadIdx.x;
        if (block < strips && c < m.cols) m.max_bits[c] = most;
        __syncthreads();
    }
    float scale[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) scale[t] = pair_scale(counts[0][first + APART * t]);
    __syncthreads();
    auto write = [&](int64_t r, const float (&x)[8]) {
        float v[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            v[t] = x[t] * scale[t];
            const float a = fabsf(v[t]);
            const bool nz = magnitude(x[t]) != 0u;
            unfit |= !(a < OVER) ? 1u : 0u;
            some |= nz ? 1u << t : 0u;
            count[t] += (a < LOW_VALUE ? 1u : 0u) + (a < FAINT_VALUE && nz ? 0x10000u : 0u);
        }
        __half* dst = m.dst + r * m.ld + c0;
        if (VEC) {
            if (c0 < width) store8(dst, m.plane, v);
        } else {
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                if (c0 + 32 * t >= width) break;
                const __half h = __float2half_rn(v[t]);
                dst[32 * t] = h;
                dst[m.plane + 32 * t] = __float2half_rn(v[t] - __half2float(h));
            }
        }
    };
    constexpr int AHEAD = 4;
    for (int64_t r = r0 + warp; r < r1; r += 8 * AHEAD) {
        uint32_t go = lane == 0 ? current_outlook(p) : 0u;
        float x[AHEAD][8];
#pragma unroll
        for (int k = 0; k < AHEAD; ++k) if (r + 8 * k < r1) load(r + 8 * k, x[k]);
#pragma unroll
        for (int k = 0; k < AHEAD; ++k) if (r + 8 * k < r1) write(r + 8 * k, x[k]);
        go = __shfl_sync(0xffffffffu, go, 0);
        if (go == STOP) break;
        uint32_t counted = 0;
        if (go == ANY_FAINT_DECIDES) {
#pragma unroll
            for (int t = 0; t < 8; ++t) counted |= count[t];
        }
        // a value that decides: one warp of the block tells the others
        if (__any_sync(0xffffffffu, unfit != 0u || counted >> 16 != 0u) && lane == 0 && atomicExch(&strip.told, 1u) == 0u) atomicMax(p.state + OUTLOOK, (uint32_t)STOP);
    }
#pragma unroll
    for (int t = 0; t < 8; ++t) counts[warp][first + APART * t] = count[t];
    __syncthreads();
#pragma unroll
    for (int t = 0; t < 8; ++t) if ((some >> t) & 1u) any[first + APART * t] = 1u;
    __syncthreads();
    const int64_t c = (int64_t)(block % strips) * STRIP + threadIdx.x;
    if (c < m.cols) {
        uint32_t low = 0, faint = 0;
#pragma unroll
        for (int w = 0; w < 8; ++w) { low += counts[w][threadIdx.x] & 0xFFFFu; faint += counts[w][threadIdx.x] >> 16; }
        if (faint) atomicAdd(m.counts + c, faint);
        if (low) atomicAdd(m.counts + m.cols + c, low);
        if (any[threadIdx.x]) m.counts[2 * m.cols + c] = 1u;
    }
}

__global__ void __launch_bounds__(256, 3) operand_pairs_kernel(const Params p) {
    chain_wait();
    __shared__ uint32_t ticket, most[8][2];
    __shared__ Strip strip;
    // the operands' blocks in turn, so that the first of both run early
    const int in_turn = 2 * min(p.blocks[0], p.blocks[1]), b = (int)blockIdx.x;
    const int which = b < in_turn ? b & 1 : p.blocks[1] > p.blocks[0] ? 1 : 0, block = b < in_turn ? b >> 1 : b - in_turn / 2;
    const OperandPair& m = p.m[which];
    bool stopped = false;
    if (b >= RESIDENT) {
        if (threadIdx.x == 0) ticket = current_outlook(p);
        __syncthreads();
        stopped = ticket == STOP;
        __syncthreads();
    }
    if (stopped) {
    } else if (!m.per_row) {
        if ((((uintptr_t)m.src) & 15) == 0 && (m.lds & 3) == 0) convert_columns<true>(p, m, which, block, strip);
        else convert_columns<false>(p, m, which, block, strip);
    }
    else if (p.warps_per_row[which] == 8) convert_rows<8>(p, m, which, block);
    else if (p.warps_per_row[which] == 4) convert_rows<4>(p, m, which, block);
    else if (p.warps_per_row[which] == 2) convert_rows<2>(p, m, which, block);
    else convert_rows<1>(p, m, which, block);
    // the last block that is through looks the counts over
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) ticket = atomicAdd(p.state + TICKET, 1u);
    __syncthreads();
    if (ticket != gridDim.x - 1) return;
    __threadfence();
    const volatile uint32_t* state = p.state;
    int64_t faint = 0, low = 0;
    for (int w = 0; w < 2; ++w) {
        const OperandPair& o = p.m[w];
        uint32_t f = 0, l = 0;
        if (o.per_row) {
            for (int i = 0; i < 8; ++i) { f += state[LARGEST + 16 * w + i]; l += state[LARGEST + 16 * w + 8 + i]; }
        } else {
            const volatile uint32_t* counts = o.counts;
            for (int64_t c = threadIdx.x; c < o.cols; c += blockDim.x)
                if (counts[2 * o.cols + c]) { f = max(f, counts[c]); l = max(l, counts[o.cols + c]); }
        }
        f = __reduce_max_sync(0xffffffffu, f); l = __reduce_max_sync(0xffffffffu, l);
        __syncthreads();
        if ((threadIdx.x & 31) == 0) { most[threadIdx.x >> 5][0] = f; most[threadIdx.x >> 5][1] = l; }
        __syncthreads();
        for (int i = 0; i < 8; ++i) { f = max(f, most[i][0]); l = max(l, most[i][1]); }
        faint += f; low += l;
    }
    if (threadIdx.x == 0) {
        // blocks that stopped have left no counts, but then their reason is in what the others left
        const uint32_t o = max(outlook(p), state[OUTLOOK]);
        const bool holds = faint == 0 || 4 * faint <= p.K - low;
        p.state[VERDICT] = o != STOP && !(o == ANY_FAINT_DECIDES && faint > 0) && holds ? 1u : 0u;
    }
}

}  // namespace

ulsnn_status_t launch_operand_pairs(const OperandPair& a, const OperandPair& b, int64_t K, uint32_t* state, cudaStream_t stream) {
    Params p{};
    p.m[0] = a; p.m[1] = b; p.state = state; p.K = K;
    int strips[2];
    for (int w = 0; w < 2; ++w) {
        const OperandPair& m = p.m[w];
        if (m.rows <= 0 || m.cols <= 0 || (m.ld & 7) != 0 || (m.plane & 7) != 0 || (((uintptr_t)m.dst) & 15) != 0 || (!m.per_row && !m.counts)) return ULSNN_ERR_INVALID_ARG;
        strips[w] = (int)((m.cols + STRIP - 1) / STRIP);
    }
    int64_t counted = 0;
    for (int w = 0; w < 2; ++w) if (!p.m[w].per_row && p.m[w].cols > counted) counted = p.m[w].cols;
    const int64_t zeroing = (3 * counted + 1023) / 1024 < 1 ? 1 : (3 * counted + 1023) / 1024;
    launch_chained(operand_start_kernel, (unsigned)(zeroing < 148 ? zeroing : 148), 256, stream, p);
    count_launch(2);
    if (cudaGetLastError() != cudaSuccess) return ULSNN_ERR_CUDA;
    for (int w = 0; w < 2; ++w) {
        const OperandPair& m = p.m[w];
        int64_t blocks;
        if (m.per_row) {
            p.warps_per_row[w] = m.cols <= 1024 ? 1 : m.cols <= 2048 ? 2 : m.cols <= 4096 ? 4 : 8;      // up to 8192 columns are read once
            blocks = (m.rows * p.warps_per_row[w] + 7) / 8;
            if (blocks > 148 * 12) blocks = 148 * 12;
        } else {
            // runs of rows that give every SM some blocks
            p.sample_step[w] = ((uint64_t)m.rows << 16) / (uint64_t)(m.rows < SAMPLE ? m.rows : SAMPLE);
            int64_t run = (m.rows * strips[w] / (148 * 4) + 31) / 32 * 32;
            run = run < 128 ? 128 : run > MOST_ROWS ? MOST_ROWS : run;
            p.rows_per_block[w] = (int)run;
            blocks = (m.rows + run - 1) / run * strips[w];
        }
        if (blocks > 0x3fffffff) return ULSNN_ERR_TOO_LARGE;
        p.blocks[w] = (int)blocks;
    }
    launch_chained(operand_pairs_kernel, (unsigned)(p.blocks[0] + p.blocks[1]), 256, stream, p);
    count_launch(2);
    return cuda_ok(cudaGetLastError());
}

}  // namespace ulsnn

// Token-delta Rice codecs (codec ids 5 and 6): quantise-then-encode for the delivery module (paper Sec. 3.2
// "KV-cache delivery" cites a scheme that quantises a KV cache and encodes it into binary strings, and Sec. 3.1 has
// the delivery module decompress on the GPU; the bitstream itself is this library's own, see kdn.h).
//
// Every (layer, K|V, 64-token group) is a SEGMENT of row_elems channels; a channel's n <= 64 codes are one
// SUB-STREAM: zigzag of the codes (mode 0) or of their token-to-token differences (mode 1), Rice-coded with a
// parameter k, bits filling bytes from the top.  A CTA works on one slice of `cols` channels of one segment:
//   store    plan   (kdn_td_plan_kernel):   quantise, pick (mode, k) per channel from bit planes, write scales / lens / params
//            scan   (kdn_td_scan_kernel):   segment sizes -> seg_off (one CTA per op)
//            encode (kdn_td_encode_kernel): quantise again, write every sub-stream at its final place
//   retrieve / compose (kdn_td_decode_kernel): bulk-copy the slice's bytes into shared memory; a thread undoes Rice,
//            zigzag and the delta of two channels, scales (and rotates) the values and writes them into bf16 rows that
//            128-bit stores scatter to the pool blocks.
// The store reads the pool twice instead of keeping codes in scratch memory: no kernel here uses memory beyond the
// pool and the chunk.  Every wait is bounded as in the tile pipeline.
#pragma once

#include "kdn_kernels.cuh"

namespace kdn {

__host__ __device__ inline int td_qmax(int codec) { return codec == 5 ? 127 : 7; }
__host__ __device__ inline int td_raw_bits(int codec) { return codec == 5 ? 9 : 5; }
__host__ __device__ inline unsigned td_max_len(int codec) { return codec == 5 ? 72u : 40u; }

// Byte offsets of the regions of a chunk of T tokens (see kdn.h).
struct TdLayout {
    unsigned long long S, scales, lens, params, streams, capacity;
};
__host__ __device__ inline TdLayout td_layout(int L, unsigned row_elems, int T, int codec)
{
    TdLayout t;
    const unsigned long long G = ((unsigned long long)T + 63ull) >> 6;
    t.S = 2ull * (unsigned long long)L * G;
    t.scales = (8ull * (t.S + 1ull) + 15ull) & ~15ull;
    t.lens = t.scales + 4ull * t.S * row_elems;
    t.params = t.lens + t.S * row_elems;
    t.streams = t.params + t.S * row_elems;
    t.capacity = t.streams + t.S * (((unsigned long long)row_elems * td_max_len(codec) + 15ull) & ~15ull);
    return t;
}

struct TdLaunch {
    int n_ops;
    void *const *k_layers;
    void *const *v_layers;
    long long n_blocks;
    int bs;
    int D;
    int L;                    // layers of the pool = layers of every chunk
    unsigned row_elems;
    unsigned cols;            // channels per CTA
    unsigned n_split;         // row_elems / cols, a power of two
    unsigned split_shift;     // log2(n_split)
    int bs_shift;             // log2(bs), -1 where bs is not a power of two
    int minus_one;            // -1 as a launch parameter: see TdStream
    float fone;               // 1.0f (see Launch::one)
    unsigned pow2[12];        // 1 << i: multiply-adds by these stay on the multiplier's pipe (as literals they become shifts)
    unsigned word_row;        // decode: bytes of one row of interleaved words (4 * cols), for the same reason
    const float2 *rope;
    int *status;
    unsigned long long wait_limit_ns;   // a wait for a slice's bytes gives up after this long
    TdLayout layout[kInlineOps];        // of each op's chunk
    DevOp inline_ops[kInlineOps];
};

// Shared memory of the encoder: the rows' addresses, a little scratch, the stream staging area.
// Behind the encoder's staging area: room for the longest thing a channel could write from the last planned byte on (64
// appends, a word each, and the last word), so that a sub-stream that came out longer than planned -- the pool changed under the store --
// garbles the chunk's bytes, which the caller has then forfeited, but never leaves the area.
constexpr unsigned kTdStageSlack = 288u;
constexpr unsigned kTdEncodeHead = 66u * 8u + 32u * 4u + 112u;      // a multiple of 128
// Shared memory of the decode kernel: the sub-streams interleaved word by word (so that the 32 lanes of a warp, each
// somewhere else in its stream, read 32 different banks), half of the group's bf16 rows, the sub-streams' offsets, the
// rows' addresses.  The slice's stream bytes as they lie in the chunk share the rows' place: they are interleaved before
// the first row is written.  The interleaved words come first: a damaged stream may look a few rows past them, which is
// then still inside the CTA's memory, and garbage either way.
constexpr unsigned kTdHalf = 32;                            // rows between two write-outs
__host__ __device__ inline unsigned td_words(int codec) { return td_max_len(codec) / 4u + 1u; }   // the longest sub-stream, and the word after
__host__ __device__ inline size_t td_stage_bytes(unsigned cols, unsigned words) { return (size_t)cols * (words - 1u) * 4u + 32u + kTdStageSlack; }
__host__ __device__ inline size_t td_encode_smem_bytes(unsigned cols, unsigned words) { return kTdEncodeHead + td_stage_bytes(cols, words); }
__host__ __device__ inline size_t td_decode_words_bytes(unsigned cols, unsigned words) { return (size_t)words * cols * 4u; }
__host__ __device__ inline size_t td_decode_rows_bytes(unsigned cols, unsigned words)
{
    const size_t a = (size_t)kTdHalf * cols * 2u, s = ((size_t)cols * (words - 1u) * 4u + 256u + 127u) & ~(size_t)127u;
    return a > s ? a : s;
}
__host__ __device__ inline size_t td_decode_smem_bytes(unsigned cols, unsigned words)
{
    return td_decode_words_bytes(cols, words) + td_decode_rows_bytes(cols, words) + (size_t)cols * 4u + 64u * 8u + 256u + 16u;
}

// Big-endian view of a little-endian word: the stream's first byte in the top bits.
__device__ __forceinline__ uint32_t td_be(uint32_t w) { return __byte_perm(w, 0u, 0x0123); }

// The code of one bf16 value, given its channel's reciprocal: round_half_even(x * inv), formed as two separately rounded fp32 operations.
// What is not finite (a NaN; an infinity, whose channel's reciprocal is zero) has the code -1: the planner and the encoder, which work
// on several values at once, put it in where they meet one, so that it spoils no more than its own channel.
__device__ __forceinline__ int td_code(uint32_t x_bf16, float inv)
{
    const float p = __fmul_rn(__uint_as_float(x_bf16 << 16), inv);
    return p == p ? (int)(signed char)(__float_as_uint(__fadd_rn(p, 12582912.0f)) & 0xffu) : -1;
}

// Exclusive prefix sum of one value per thread over the block (blockDim.x a multiple of 32, at most 1024);
// *total receives the sum.  `scratch` is 33 words of shared memory.  (64 bits: the segments that a step adds up may take more than 4 GiB.)
__device__ __forceinline__ unsigned long long td_block_scan(unsigned long long v, unsigned long long *scratch, unsigned long long *total)
{
    const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    unsigned long long inc = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned long long o = __shfl_up_sync(0xffffffffu, inc, d);
        if (lane >= (unsigned)d) inc += o;
    }
    if (lane == 31u) scratch[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        unsigned long long w = lane < nwarps ? scratch[lane] : 0ull, winc = w;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned long long o = __shfl_up_sync(0xffffffffu, winc, d);
            if (lane >= (unsigned)d) winc += o;
        }
        scratch[lane] = winc - w;
        if (lane == 31u) scratch[32] = winc;
    }
    __syncthreads();
    const unsigned long long r = scratch[warp] + inc - v;
    *total = scratch[32];
    __syncthreads();
    return r;
}

// First index of the increasing list whose entry is >= key (n when there is none).  At most 32 steps.
__device__ __forceinline__ unsigned td_lower_bound(const int32_t *list, unsigned n, long long key)
{
    unsigned lo = 0, hi = n;
    while (lo < hi) {
        const unsigned mid = (lo + hi) >> 1;
        if ((long long)list[mid] < key) lo = mid + 1u; else hi = mid;
    }
    return lo;
}

struct TdSlice {              // what a CTA of the store and decode kernels works on
    DevOp op;
    unsigned g, part, plane, li, kv, n_tok, c0, seg;
    unsigned long long G;
    bool valid;
};
__device__ __forceinline__ TdSlice td_slice(const TdLaunch &P)
{
    TdSlice s;
    s.op = P.inline_ops[blockIdx.z];
    s.g = blockIdx.x >> P.split_shift;
    s.part = blockIdx.x & (P.n_split - 1u);
    s.plane = blockIdx.y;                                      // index into the op's layer range: li * 2 + kv
    s.li = s.plane >> 1;
    s.kv = s.plane & 1u;
    s.G = ((unsigned long long)s.op.T + 63ull) >> 6;
    s.valid = s.op.codec >= 5 && s.g < s.G && s.li < (unsigned)s.op.nl;
    const unsigned t0 = s.g << 6;
    s.n_tok = s.valid ? ((unsigned)s.op.T - t0 < 64u ? (unsigned)s.op.T - t0 : 64u) : 0u;
    s.c0 = s.part * P.cols;
    s.seg = (unsigned)(((unsigned long long)(s.op.l0 + (int)s.li) * 2ull + s.kv) * s.G + s.g);
    return s;
}

// Where a slice's sub-streams lie: two channels a thread, 2 tid and 2 tid + 1 of the slice.  `scratch`: 32 words of shared memory.
// All threads of the block call this (one barrier).
struct TdOffsets {
    unsigned pair;                // lengths of the thread's two sub-streams, one byte each (0 past the slice's end)
    unsigned off;                 // byte offset of the first of them inside the slice
    unsigned slice, before;       // bytes of the slice, and of the segment's slices before it
};
__device__ __forceinline__ TdOffsets td_offsets(const unsigned char *lens, unsigned c0, unsigned C, unsigned nthreads, unsigned *scratch)
{
    const unsigned tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5, nwarps = nthreads >> 5;
    TdOffsets o;
    // channels before the slice: 16 lengths a load (the table's rows and c0 are multiples of 16)
    unsigned before = 0;
    for (unsigned i = tid; i < (c0 >> 4); i += nthreads) {
        const uint4 v = *reinterpret_cast<const uint4 *>(lens + 16u * i);
        before = __dp4a(v.x, 0x01010101u, before); before = __dp4a(v.y, 0x01010101u, before);
        before = __dp4a(v.z, 0x01010101u, before); before = __dp4a(v.w, 0x01010101u, before);
    }
    o.pair = 2u * tid < C ? *reinterpret_cast<const unsigned short *>(lens + c0 + 2u * tid) : 0u;
    const unsigned both = (o.pair & 0xffu) + (o.pair >> 8);
    unsigned inc = both;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned v = __shfl_up_sync(0xffffffffu, inc, d);
        if (lane >= (unsigned)d) inc += v;
    }
    before = __reduce_add_sync(0xffffffffu, before);
    if (lane == 31u) { scratch[warp] = inc; scratch[16u + warp] = before; }
    __syncthreads();
    o.off = inc - both;
    o.slice = 0u;
    o.before = 0u;
    for (unsigned w = 0; w < nwarps; ++w) {
        if (w == warp) o.off += o.slice;
        o.slice += scratch[w];
        o.before += scratch[16u + w];
    }
    return o;
}

// Pool addresses of the slice in the token rows of the group, row t at rows[t + t / 32], or, without kGap, rows[t] (0 for rows past the chunk's end).  Threads
// t = first, first + step, ... of those who fill one table call this; true when one of the thread's rows lies outside the pool or the table.
// kAhead: before the wait for the kernel in front (see ld_ahead).
template <bool kAhead, bool kGap>
__device__ __forceinline__ bool td_row_addresses(const TdLaunch &P, const TdSlice &s, unsigned long long *rows, unsigned first, unsigned step)
{
    const unsigned char *base = reinterpret_cast<const unsigned char *>((s.kv ? P.v_layers : P.k_layers)[s.op.l0 + (int)s.li]);
    bool bad = false;
    for (unsigned t = first; t < 64u; t += step) {
        unsigned long long a = 0ull;
        if (t < s.n_tok) {
            const long long pos = group_row_pos<kAhead>(s.op, s.g, t);
            long long id = -1;
            const long long blk = P.bs_shift >= 0 ? pos >> P.bs_shift : pos / P.bs;
            if (pos >= 0) id = kAhead ? ld_ahead(s.op.table + blk) : s.op.table[blk];
            if (id < 0 || id >= P.n_blocks) bad = true;
            else a = (unsigned long long)(base + ((unsigned long long)(id * P.bs + (pos - blk * P.bs)) * P.row_elems + s.c0) * 2ull);
        }
        rows[kGap ? t + (t >> 5) : t] = a;
    }
    return bad;
}

// ------------------------------------------------------------------------------------------ store: plan --

// The planner works on bit planes: plane i of a channel's 32 tokens is one 32-bit word, bit t of it bit i of token t's
// code, so one logic operation handles 32 symbols and counting is popc.
//
// From codes to planes.  A thread holds two neighbouring channels of 32 tokens; their codes, biased to be positive, are
// gathered in the floating-point pipe (see gather2), a word of four tokens t, t + 8, t + 16, t + 24 (8-bit codes) or of eight
// tokens t, t + 4, .. (4-bit codes).  Transposing 8 x 8 (4 x 4) bits inside every byte (nibble) lane across the eight (four)
// words then leaves the planes in the tokens' own order.
template <int kN> __device__ __forceinline__ void td_transpose(const TdLaunch &P, uint32_t (&w)[kN])
{
#pragma unroll
    for (int d = kN / 2; d >= 1; d >>= 1) {
        const uint32_t m = d == 4 ? 0x0f0f0f0fu : d == 2 ? 0x33333333u : 0x55555555u;
#pragma unroll
        for (int j = 0; j < kN; ++j) {
            if (j & d) continue;
            const uint32_t a = w[j], b = w[j + d];
            w[j] = (a & m) | ((b * P.pow2[d]) & ~m);
            w[j + d] = ((a >> d) & m) | (b & ~m);
        }
    }
}

// The sum over 64 symbols of what a code word takes beyond its k + 1 bits, times 16, for a k at which a symbol may escape: u >> k for the unary part, or
// kEsc - 1 - k for an escape (u >> k >= 15).  lo and hi are the planes of u for tokens 0-31 and 32-63; the two halves' numbers are added
// plane by plane first, which leaves one count per plane of the sum: popc runs at an eighth of the rate of the logic.
template <int kPlanes, int kMax, int kEsc, int kK>
__device__ __forceinline__ unsigned td_plan_sum(const TdLaunch &P, const uint32_t (&lo)[kPlanes], const uint32_t (&hi)[kPlanes])
{
    constexpr int v = kEsc - 1 - kK;
    static_assert((kMax >> kK) >= 15, "nothing escapes at this k");
    static_assert(v >= 16 && v < 32, "the planes of an escape's cost");
    uint32_t x[2][5];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const uint32_t (&b)[kPlanes] = h ? hi : lo;
        uint32_t over = 0u;                                  // bits above the four that a short quotient has
#pragma unroll
        for (int i = kK + 4; i < kPlanes; ++i) over |= b[i];
        const uint32_t esc = (b[kK] & b[kK + 1] & b[kK + 2] & b[kK + 3]) | over;
#pragma unroll
        for (int i = 0; i < 4; ++i) x[h][i] = ((v >> i) & 1) ? b[kK + i] | esc : b[kK + i] & ~esc;
        x[h][4] = esc;
    }
    unsigned sum = 0u;
    uint32_t carry = 0u;
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const uint32_t p = x[0][i], q = x[1][i];
        sum += (unsigned)__popc(p ^ q ^ carry) * P.pow2[4 + i];
        carry = (p & q) | (carry & (p | q));
    }
    return sum + (unsigned)__popc(carry) * P.pow2[9];
}
// The smallest (bits * 16 + mode * 8 + k) over the parameters of one mode, and `best`, for n symbols.  With c_i symbols that have bit i, the sum of
// u >> k is c_k + 2 c_(k+1) + 4 c_(k+2) + ..: two popc a plane serve every k at which nothing can escape.  Where something can, the
// same sum with its large weights cut down bounds the bits from below: weights of at most 2^(i-k) that add up to no more than
// kEsc - 1 - k count neither a unary part nor an escape for more than it takes.  Only a k that could then still win for a channel of the warp is
// looked at closely, and its escapes' planes are counted only where there is an escape.  (The k of kPlanes and more cannot win: at kPlanes - 1
// a code word takes no more bits, and the smaller k goes first.)  8B shape, 16 chunks of 512 tokens, the whole store, with every k counted by itself
// and this way, us: 8-bit codes, uncorrelated 852 / 795, correlation 0.9 860 / 810, 0.99 907 / 853; 4-bit 719 / 698, 714 / 693, 711 / 689.
template <int kK> struct TdConst { static constexpr int value = kK; };
template <int kMode, int kPlanes, int kMax, int kEsc>
__device__ __forceinline__ unsigned td_plan_mode(const TdLaunch &P, unsigned best, const uint32_t (&lo)[kPlanes], const uint32_t (&hi)[kPlanes],
                                                 unsigned n, bool act)
{
    constexpr int kTop = kPlanes < 8 ? kPlanes - 1 : 7;
    constexpr int kFree = kMax < 15 ? 0 : kMax < 30 ? 1 : kMax < 60 ? 2 : kMax < 120 ? 3 : kMax < 240 ? 4 : kMax < 480 ? 5 : 6;   // the least k at which nothing escapes
    const unsigned n16 = n * 16u;
    unsigned c[kPlanes], all[kPlanes];                       // all[k]: the sum of u >> k
#pragma unroll
    for (int i = kPlanes - 1; i >= 0; --i) {
        c[i] = (unsigned)__popc(lo[i]) + (unsigned)__popc(hi[i]);
        all[i] = i == kPlanes - 1 ? c[i] : all[i + 1] * P.pow2[1] + c[i];
    }
#pragma unroll
    for (int k = kTop; k >= kFree; --k) best = min(best, all[k] * P.pow2[4] + n16 * (unsigned)(k + 1) + (unsigned)(kMode * 8 + k));
    // what `all` counts too much for k: the weights above 8 cut down to kEsc - 1 - k - 15 in all
    auto bound = [&](int k) {
        unsigned b = all[k];
        int left = kEsc - 1 - k - 15;
#pragma unroll
        for (int i = kPlanes - 1; i >= k + 4; --i) {
            const int planes = i - (k + 4) + 1, w = left / planes < (1 << (i - k)) ? left / planes : 1 << (i - k);
            b -= c[i] * (unsigned)((1 << (i - k)) - w);
            left -= w;
        }
        return b * 16u;
    };
    // most often none of them can win
    unsigned least = 0xffffffffu;
#pragma unroll
    for (int k = kFree - 1; k >= 0; --k) least = min(least, bound(k) + n16 * (unsigned)(k + 1) + (unsigned)(kMode * 8 + k));
    if (!__any_sync(0xffffffffu, act && least < best)) return best;
    // one of the k at which a symbol could escape; does one?
    auto look = [&](auto which) {
        constexpr int k = decltype(which)::value;
        if (!__any_sync(0xffffffffu, act && bound(k) + n16 * (k + 1u) + (kMode * 8u + k) < best)) return;
        uint32_t esc = (lo[k] & lo[k + 1] & lo[k + 2] & lo[k + 3]) | (hi[k] & hi[k + 1] & hi[k + 2] & hi[k + 3]);
#pragma unroll
        for (int i = k + 4; i < kPlanes; ++i) esc |= lo[i] | hi[i];
        const unsigned sum = __any_sync(0xffffffffu, esc != 0u) ? td_plan_sum<kPlanes, kMax, kEsc, k>(P, lo, hi) : all[k] * 16u;
        best = min(best, sum + n16 * (k + 1u) + (kMode * 8u + k));
    };
    if constexpr (kFree > 5) look(TdConst<5>());
    if constexpr (kFree > 4) look(TdConst<4>());
    if constexpr (kFree > 3) look(TdConst<3>());
    if constexpr (kFree > 2) look(TdConst<2>());
    if constexpr (kFree > 1) look(TdConst<1>());
    if constexpr (kFree > 0) look(TdConst<0>());
    return best;
}

// Two channels of 32 tokens (x: bf16 pairs) -> bits * 16 + parameters of the one channel this thread answers for (lane 16 + l
// has tokens 32-63 of the channels lane l has 0-31 of; lane l answers for the first of the two).  n: tokens of the group.
// kFull: n = 64, known when the code is made.  odd (one value for the warp): some of the tokens are not finite, those of the masks odd_a and odd_b.
template <bool kInt4, bool kFull>
__device__ __forceinline__ unsigned td_plan_channel(const TdLaunch &P, const uint32_t (&x)[32], float inv_a, float inv_b, unsigned n, bool act,
                                                    bool odd, uint32_t odd_a, uint32_t odd_b)
{
    constexpr int kW = kInt4 ? 4 : 8;                       // words per channel before, planes after transposing
    const f32x2 inv2 = pack2(inv_a, inv_b), one2 = pack2(P.fone, P.fone);
    const float magic = 12582912.0f + (kInt4 ? 8.0f : 128.0f);
    const f32x2 magic2 = pack2(magic, magic), minus_m2 = pack2(-12582912.0f, -12582912.0f);
    auto code = [&](int t) { return add2_unfused(mul2(bf16x2_widen(x[t]), inv2), magic2, one2); };      // 1.5 * 2^23 + bias + code
    uint32_t wa[kW], wb[kW];
#pragma unroll
    for (int j = 0; j < kW; ++j) {
        f32x2 g[2];
        if (kInt4) {
            const f32x2 k16 = pack2(16.0f, 16.0f), k256 = pack2(256.0f, 256.0f), k4096 = pack2(4096.0f, 4096.0f);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                g[h] = gather2(code(j + 16 * h), code(j + 16 * h + 4), minus_m2, k16);
                g[h] = gather2(g[h], code(j + 16 * h + 8), minus_m2, k256);
                g[h] = gather2(g[h], code(j + 16 * h + 12), minus_m2, k4096);
            }
        } else {
            const f32x2 k256 = pack2(256.0f, 256.0f);
            g[0] = gather2(code(j), code(j + 8), minus_m2, k256);
            g[1] = gather2(code(j + 16), code(j + 24), minus_m2, k256);
        }
        uint32_t a0, b0, a1, b1;
        unpack2_bits(g[0], a0, b0);
        unpack2_bits(g[1], a1, b1);
        wa[j] = __byte_perm(a0, a1, 0x5410);
        wb[j] = __byte_perm(b0, b1, 0x5410);
    }
    td_transpose<kW>(P, wa);
    td_transpose<kW>(P, wb);
    if (__builtin_expect(odd, 0)) {
#pragma unroll
        for (int i = 0; i < kW; ++i) {                       // bias - 1: ones below the top plane
            wa[i] = i < kW - 1 ? wa[i] | odd_a : wa[i] & ~odd_a;
            wb[i] = i < kW - 1 ? wb[i] | odd_b : wb[i] & ~odd_b;
        }
    }
    // each of the two lanes that share a pair of channels takes one of them over whole
    const bool upper = (threadIdx.x & 16u) != 0u;
    uint32_t lo[kW], hi[kW];
#pragma unroll
    for (int i = 0; i < kW; ++i) {
        const uint32_t got = __shfl_xor_sync(0xffffffffu, upper ? wa[i] : wb[i], 16);
        lo[i] = upper ? got : wa[i];
        hi[i] = upper ? wb[i] : got;
    }
    // mode 0: the biased code's top plane is the complement of the sign; u = 2 q or 2 ~q + 1
    unsigned best;
    {
        uint32_t ul[kW], uh[kW];
        ul[0] = ~lo[kW - 1]; uh[0] = ~hi[kW - 1];
#pragma unroll
        for (int i = 1; i < kW; ++i) { ul[i] = lo[i - 1] ^ ul[0]; uh[i] = hi[i - 1] ^ uh[0]; }
        best = td_plan_mode<0, kW, kInt4 ? 14 : 254, kInt4 ? 20 : 24>(P, 0xffffffffu, ul, uh, n, act);
    }
    // mode 1: e = code - code of the token before (the bias falls out; before the first token stands the bias itself)
    {
        uint32_t dl[kW + 1], dh[kW + 1];
        const uint32_t vl = n >= 32u ? 0xffffffffu : (1u << n) - 1u, vh = n >= 64u ? 0xffffffffu : n > 32u ? (1u << (n - 32u)) - 1u : 0u;
        uint32_t bl = 0u, bh = 0u;                           // borrows
#pragma unroll
        for (int i = 0; i < kW; ++i) {
            uint32_t pl = lo[i] * P.pow2[1] + (i == kW - 1 ? 1u : 0u), ph = __funnelshift_l(lo[i], hi[i], 1);
            if (!kFull) {                                   // tokens that are not there: no difference
                pl = (pl & vl) | (lo[i] & ~vl);
                ph = (ph & vh) | (hi[i] & ~vh);
            }
            dl[i + 1] = lo[i] ^ pl ^ bl;
            dh[i + 1] = hi[i] ^ ph ^ bh;
            bl = (~lo[i] & pl) | (bl & (~lo[i] | pl));
            bh = (~hi[i] & ph) | (bh & (~hi[i] | ph));
        }
        dl[0] = bl; dh[0] = bh;                              // the last borrow is the sign
#pragma unroll
        for (int i = 1; i <= kW; ++i) { dl[i] ^= bl; dh[i] ^= bh; }
        best = td_plan_mode<1, kW + 1, kInt4 ? 28 : 508, kInt4 ? 20 : 24>(P, best, dl, dh, n, act);
    }
    return best;
}

// A warp takes 32 channels: lanes l and l + 16 hold the same two channels, tokens 0-31 and 32-63, straight from the pool in
// registers (no shared tile: every value is used once, and a thread has 32 loads in flight).  Bound by instruction issue, as far as 24 warps an SM, whose
// loads come in one burst each, can fill it: 71 % of the slots, the pipe of logic and shifts 56 % (4-bit codes 67 and 39 %).  8B shape, 8 chunks of 512
// tokens, under the profiler: 537 us with a table of code-word lengths looked up per symbol, 168 us this way (uncorrelated; correlation 0.9: 178), 4-bit
// codes 141.  Six CTAs of 128 threads an SM (78 registers); seven or eight spill and are 2 % slower.
// kThreads: 128 is the usual slice of 128 channels, 512 stands for any other.
template <unsigned kThreads>
__global__ void __launch_bounds__(kThreads, kThreads == 128u ? 6 : 1) kdn_td_plan_kernel(const __grid_constant__ TdLaunch P)
{
    // pool addresses of the group's token rows (0: past the chunk's end), row t at index t + t / 32: the two that a warp reads at once in
    // different banks.  A table a warp: no barrier in this kernel, a warp computes while others load.
    __shared__ unsigned long long all_rows[kThreads / 32u][66];
    dependency_wait();
    release_dependents();
    const TdSlice s = td_slice(P);
    if (!s.valid) return;
    const unsigned C = P.cols, RE = P.row_elems, tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    const int codec = s.op.codec;
    const TdLayout &lay = P.layout[blockIdx.z];
    const unsigned long long row = (unsigned long long)s.seg * RE + s.c0;
    unsigned long long *rows = all_rows[warp];
    const bool bad = td_row_addresses<false, true>(P, s, rows, lane, 32u);
    __syncwarp();
    const unsigned half = lane >> 4, pair = warp * 16u + (lane & 15u), ch = 2u * pair + half;      // ch: the channel the thread answers for
    const bool act = 2u * pair < C;                         // (C is a multiple of 16)
    unsigned *warp_bytes = reinterpret_cast<unsigned *>(s.op.data + lay.streams) + ((size_t)s.seg * P.n_split + s.part) * ((C + 31u) >> 5) + warp;
    if (__any_sync(0xffffffffu, bad)) {
        // channels that are given up leave lengths of zero behind: the scan and the encoder then see a consistent, if
        // incomplete, chunk instead of whatever the buffer held before
        if (act) {
            s.op.data[lay.lens + row + ch] = 0;
            s.op.data[lay.params + row + ch] = 0;
        }
        if (lane == 0) {
            atomicCAS(P.status, 0, kStatusRange);
            *warp_bytes = 0u;
        }
        return;
    }
    uint32_t x[32];
    const unsigned long long *my_rows = rows + 33u * half;
    const bool full = s.n_tok == 64u;
    const unsigned n_mine = !act ? 0u : s.n_tok < 32u * half ? 0u : s.n_tok - 32u * half;
    if (full && act) {
#pragma unroll
        for (int t = 0; t < 32; ++t) x[t] = __ldcg(reinterpret_cast<const uint32_t *>(my_rows[t] + (unsigned long long)(2u * pair) * P.pow2[1]));
    } else {
#pragma unroll
        for (int t = 0; t < 32; ++t) x[t] = (unsigned)t < n_mine ? __ldcg(reinterpret_cast<const uint32_t *>(my_rows[t]) + pair) : 0u;
    }
    uint32_t m0 = maxabs_nan_bf16x2(x[0], x[1]), m1 = maxabs_nan_bf16x2(x[2], x[3]);
#pragma unroll
    for (int t = 4; t < 32; t += 2) { m0 = maxabs_nan_bf16x2(m0, x[t]); m1 = maxabs_nan_bf16x2(m1, x[t + 1]); }
    m0 = maxabs_nan_bf16x2(m0, m1);
    m0 = maxabs_nan_bf16x2(m0, __shfl_xor_sync(0xffffffffu, m0, 16));
    // Values that are not finite would spoil the codes of the tokens that share a word with theirs: noted, and zeroed.  A channel's
    // largest magnitude is that of its numbers, infinities included.
    const bool odd = __any_sync(0xffffffffu, (m0 & 0x7f80u) == 0x7f80u || (m0 & 0x7f800000u) == 0x7f800000u);
    uint32_t odd_a = 0u, odd_b = 0u;
    if (__builtin_expect(odd, 0)) {
        m0 = 0u;
#pragma unroll
        for (int t = 0; t < 32; ++t) {
            m0 = maxabs_bf16x2(m0, x[t]);
            if ((x[t] & 0x7f80u) == 0x7f80u) { odd_a |= 1u << t; x[t] &= 0xffff0000u; }
            if ((x[t] & 0x7f800000u) == 0x7f800000u) { odd_b |= 1u << t; x[t] &= 0x0000ffffu; }
        }
        m0 = maxabs_bf16x2(m0, __shfl_xor_sync(0xffffffffu, m0, 16));
    }
    // scale and reciprocal of the thread's own channel, the other channel's reciprocal from its partner
    const float qmax = (float)td_qmax(codec);
    const float a = __uint_as_float(half ? m0 & 0x7fff0000u : (m0 & 0x7fffu) << 16);
    const float sc = __fdiv_rn(a, qmax);
    const bool ok = sc >= 1.17549435e-38f;                  // smallest normal fp32; false for NaN too
    const float inv = ok ? __fdiv_rn(qmax, a) : 0.0f;
    const float other = __shfl_xor_sync(0xffffffffu, inv, 16);
    const float inv_a = half ? other : inv, inv_b = half ? inv : other;
    unsigned best;
    if (codec == 5) best = full ? td_plan_channel<false, true>(P, x, inv_a, inv_b, 64u, act, odd, odd_a, odd_b) : td_plan_channel<false, false>(P, x, inv_a, inv_b, s.n_tok, act, odd, odd_a, odd_b);
    else best = full ? td_plan_channel<true, true>(P, x, inv_a, inv_b, 64u, act, odd, odd_a, odd_b) : td_plan_channel<true, false>(P, x, inv_a, inv_b, s.n_tok, act, odd, odd_a, odd_b);
    const unsigned len = act ? (best + 7u * 16u) >> 7 : 0u;                   // bytes of the sub-stream
    if (act) {
        reinterpret_cast<float *>(s.op.data + lay.scales)[row + ch] = ok ? sc : 0.0f;
        s.op.data[lay.lens + row + ch] = (unsigned char)len;
        s.op.data[lay.params + row + ch] = (unsigned char)(best & 15u);
    }
    // The warp's bytes are left for the scan at the start of the streams, four bytes a warp: the encoder overwrites them, as
    // every sub-stream takes at least a byte.
    const unsigned sum = __reduce_add_sync(0xffffffffu, len);
    if (lane == 0) *warp_bytes = sum;
}

// ------------------------------------------------------------------------------------------ store: scan --

// One CTA per op: seg_off[s + 1] = seg_off[s] + the segment's sub-stream bytes rounded up to 16, 1024 segments at a time.
// Latency is all that counts here: 512 tokens at the 8B shape took 58 us when the lengths were added up here, and take 5 now
// that the planner leaves sums behind.
constexpr unsigned kTdScanThreads = 1024;
__global__ void __launch_bounds__(kTdScanThreads) kdn_td_scan_kernel(const __grid_constant__ TdLaunch P)
{
    __shared__ unsigned long long scratch[33];
    dependency_wait();
    release_dependents();
    const DevOp op = P.inline_ops[blockIdx.x];
    if (op.codec < 5 || op.T <= 0) return;
    const TdLayout &lay = P.layout[blockIdx.x];
    unsigned long long *seg_off = reinterpret_cast<unsigned long long *>(op.data);
    const unsigned *warp_bytes = reinterpret_cast<const unsigned *>(op.data + lay.streams);
    const unsigned tid = threadIdx.x, per_seg = P.n_split * ((P.cols + 31u) >> 5);
    unsigned long long run = lay.streams;
    if (tid == 0) {
        seg_off[0] = run;
        if ((lay.S + 1ull) & 1ull) seg_off[lay.S + 1ull] = 0ull;             // the table is padded to 16 bytes with zeros
    }
    for (unsigned long long base = 0; base < lay.S; base += kTdScanThreads) {
        const unsigned long long sidx = base + tid;
        unsigned size = 0;
        if (sidx < lay.S) {
            if ((per_seg & 3u) == 0u) {
                const uint4 *mine = reinterpret_cast<const uint4 *>(warp_bytes + sidx * per_seg);
#pragma unroll 8
                for (unsigned p = 0; p < (per_seg >> 2); ++p) {
                    const uint4 v = mine[p];
                    size += v.x + v.y + v.z + v.w;
                }
            } else {
                for (unsigned p = 0; p < per_seg; ++p) size += warp_bytes[sidx * per_seg + p];
            }
        }
        size = (size + 15u) & ~15u;                          // (of one segment: at most 72 bytes for each of 2^24 channels)
        unsigned long long total;
        const unsigned long long before = td_block_scan(size, scratch, &total);
        if (sidx < lay.S) seg_off[sidx + 1ull] = run + before + size;
        run += total;
    }
}

// ---------------------------------------------------------------------------------------- store: encode --

// One sub-stream on its way out.  As in the decoder the bits are kept complemented, so that unary parts are zeros: a symbol u
// is the number 2^(k+1) - 1 - (u mod 2^k) in (u >> k) + k + 1 bits.  u itself comes out of the floating-point pipe as
// |2 e + 1/2| - 1/2 (2 e for e >= 0, else -2 e - 1), in the low bits of 2^23 + u; and from there the length, for two channels at once: a
// multiply-add by -2^-k that rounds up gives kTdLenZero - (u >> k) - (k + 1), minus the length in the low bits of its representation.  (k = 0: the
// summand would take 25 bits, so u - 1 stands for u, whose low bits are of no interest then.)
struct TdOut {
    uint32_t acc;          // the bits not yet written, in the low (bits mod 32) bits; garbage above them
    unsigned bits;         // bits so far, those of the first word that are not the sub-stream's own included, modulo 64
    uint32_t wp;           // shared address of the word being filled
    unsigned k;            // Rice parameter
    uint32_t kmask, kbit;  // 2^k - 1, 2^k
    float limit;           // kTdLenZero - (k + 16): code words this long are escapes
};
constexpr unsigned kTdLoad = 8;                              // tokens loaded ahead
constexpr uint32_t kTdUZero = 0x4B000000u;                   // bits of 2^23
constexpr float kTdLenZero = 12582912.0f;                    // 1.5 * 2^23
constexpr uint32_t kTdLenBits = 0x4B400000u;                 // its bits, a multiple of 64

// addr: where the sub-stream goes in the staging area
__device__ __forceinline__ void td_out_init(TdOut &o, uint32_t addr, unsigned param)
{
    o.k = param & 7u;
    o.kbit = 1u << o.k;
    o.kmask = o.kbit - 1u;
    o.limit = kTdLenZero - (float)(o.k + 16u);
    o.acc = 0u;
    o.bits = (addr & 3u) * 8u;
    o.wp = addr & ~3u;
}
// Append the low `len` bits of w (1 <= len <= 32, nothing above them; nlen = -len, give or take a multiple of 64).  (Shifts take their count modulo 32.)
// Words go out with plain predicated stores: the first one too, with zeros where its neighbour's last bits belong, which are ORed in at the
// end.  (An OR into the staging area for every word cost a branch round the instruction: store of 16 chunks 923 -> 898 us.)
__device__ __forceinline__ void td_append(TdOut &o, uint32_t w, unsigned nlen)
{
    const uint32_t left = __funnelshift_l(0u, w, nlen);                     // left-aligned
    const uint32_t word = __funnelshift_r(left, o.acc, o.bits);
    const unsigned bits = o.bits - nlen;
    o.acc = __funnelshift_r(left, o.acc, nlen);
    asm volatile("{ .reg .pred p; setp.ne.u32 p, %2, 0; @p st.shared.u32 [%0], %1; @p add.u32 %0, %0, 4; }"
                 : "+r"(o.wp) : "r"(word), "r"((o.bits ^ bits) & 32u) : "memory");
    o.bits = bits;
}
// One symbol, escapes included; ub: bits of 2^23 + u (- 1 for k = 0), n: kTdLenZero minus its length, were it none.  (Length and escape out of the
// multiply-add that the joined symbols take them from: with integers from u, store of 8 chunks of 512 tokens with 8-bit codes, small values and 2 % large
// ones: 726 us, this way 674; uncorrelated 420 -> 406, 4-bit codes 355 -> 338.)
__device__ __forceinline__ void td_append_any(TdOut &o, uint32_t ub, float n, unsigned raw_bits)
{
    const bool escape = n <= o.limit;
    td_append(o, escape ? ~(ub + (o.kbit & 1u)) & ((1u << raw_bits) - 1u) : (~ub & o.kmask) | o.kbit, escape ? 0u - (15u + raw_bits) : __float_as_uint(n));
}
__device__ __forceinline__ float td_fma_up(float a, float b, float c)
{
    float d;
    asm("fma.rp.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
__device__ __forceinline__ float td_min3_nan(float a, float b, float c)
{
    float d;
    asm("min.NaN.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
__device__ __forceinline__ f32x2 td_fma2_up(f32x2 a, f32x2 b, f32x2 c)        // rounded towards +infinity
{
    f32x2 d;
    asm("fma.rp.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
// Four symbols of two sub-streams (ux, uy, and nx, ny: kTdLenZero minus their lengths), kJoin of them joined before they are appended (4-bit codes:
// four, 8-bit codes: two).  Where one is an escape, or the joined ones are longer than a word, one at a time.  A NaN goes the same way:
// again(i, a, b) then forms symbol i of both sub-streams with care, and leaves behind what the next one needs.
template <unsigned kN> struct TdJoin { static constexpr unsigned value = kN; };
template <unsigned kJoin, typename Again>
__device__ __forceinline__ void td_append4(TdOut &x, TdOut &y, const uint32_t (&ux)[4], const uint32_t (&uy)[4], const float (&nx)[4], const float (&ny)[4],
                                           float px, float py, float lx, float ly, unsigned raw_bits, Again again)
{
    uint32_t zx[4], zy[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        zx[i] = (~ux[i] & x.kmask) | x.kbit;
        zy[i] = (~uy[i] & y.kmask) | y.kbit;
    }
    const float mx = td_min3_nan(td_min3_nan(nx[0], nx[1], nx[2]), nx[3], nx[3]), my = td_min3_nan(td_min3_nan(ny[0], ny[1], ny[2]), ny[3], ny[3]);
    int jx[4], jy[4], longest = 0x7fffffff;                  // joined: minus the lengths, plus kJoin times kTdLenBits
#pragma unroll
    for (int i = 0; i < 4; i += (int)kJoin) {
        jx[i] = __float_as_int(nx[i]); jy[i] = __float_as_int(ny[i]);
#pragma unroll
        for (int j = 1; j < (int)kJoin; ++j) {
            zx[i] = __funnelshift_r(0u, zx[i], __float_as_uint(nx[i + j])) + zx[i + j];       // shifted left by the length
            zy[i] = __funnelshift_r(0u, zy[i], __float_as_uint(ny[i + j])) + zy[i + j];
            jx[i] = (int)((unsigned)jx[i] + __float_as_uint(nx[i + j]));
            jy[i] = (int)((unsigned)jy[i] + __float_as_uint(ny[i + j]));
        }
        longest = __vimin3_s32(longest, jx[i], jy[i]);
    }
    if (__builtin_expect(!(mx > x.limit) || !(my > y.limit) || longest < (int)(kJoin * kTdLenBits - 32u), 0)) {
        uint32_t a[4], b[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) { a[i] = ux[i]; b[i] = uy[i]; }
        if (__builtin_expect(mx != mx || my != my, 0)) {
#pragma unroll 1
            for (int i = 0; i < 4; ++i) {
                a[0] = a[1]; a[1] = a[2]; a[2] = a[3];
                b[0] = b[1]; b[1] = b[2]; b[2] = b[3];
                again((unsigned)i, a[3], b[3]);
            }
        }
#pragma unroll 1
        for (int i = 0; i < 4; ++i) {                        // (rolled up: instruction fetch is felt in this kernel)
            td_append_any(x, a[0], td_fma_up(__uint_as_float(a[0]), px, lx), raw_bits);
            td_append_any(y, b[0], td_fma_up(__uint_as_float(b[0]), py, ly), raw_bits);
            a[0] = a[1]; a[1] = a[2]; a[2] = a[3];
            b[0] = b[1]; b[1] = b[2]; b[2] = b[3];
        }
    } else {
#pragma unroll
        for (int i = 0; i < 4; i += (int)kJoin) {
            td_append(x, zx[i], (unsigned)jx[i]);
            td_append(y, zy[i], (unsigned)jy[i]);
        }
    }
}
// The end of a sub-stream: zero bits (ones, complemented) up to the byte; and, when all of the slice's whole words are out, the bits of its last
// word, which neighbours may share.
__device__ __forceinline__ void td_out_pad(TdOut &o)
{
    const unsigned pad = (0u - o.bits) & 7u;
    if (pad) td_append(o, (1u << pad) - 1u, 0u - pad);
}
__device__ __forceinline__ void td_out_last(const TdOut &o)
{
    if (o.bits & 31u) {
        const uint32_t word = o.acc << (32u - (o.bits & 31u));
        asm volatile("red.shared.or.b32 [%0], %1;" :: "r"(o.wp), "r"(word) : "memory");
    }
}

// A thread quantises and codes two neighbouring channels side by side, token by token, straight from the pool: the planner's scale
// says what the largest magnitude was (a bf16 number: scale * qmax rounded to bf16 is that number again), so there is no pass
// for it and no tile.  The staging area holds the slice's bits complemented, as big-endian words.  Bound by instruction issue and by its loads (73 %
// of the slots, 31 warps an SM, 21.5 warp instructions per 32 symbols, 4-bit codes 19.1).  8B shape, 8 chunks of 512 tokens, under the profiler: 495 us with a
// tile, a pass over it for the magnitudes and every symbol appended by itself, 222 us this way; 4-bit codes 196.  The whole store of 16 chunks takes
// 765 us with 8-bit codes (uncorrelated; correlation 0.9: 780, 0.99: 824), 660, 656 and 654 us with 4-bit ones.  Sixteen CTAs of 64 threads an SM
// (64 registers) with eight tokens loaded ahead; twelve CTAs, four or sixteen tokens were 1-7 % slower.
// (Other slices: at most 256 threads, 96 registers; at 104 a slice of 192 channels loses a CTA an SM and 10 %.)
template <unsigned kCols>
__global__ void __launch_bounds__(kCols ? kCols / 2u : 320u, kCols ? 16 : 2) kdn_td_encode_kernel(const __grid_constant__ TdLaunch P)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const TdSlice s = td_slice(P);
    if (!s.valid) return;
    const unsigned C = kCols ? kCols : P.cols, RE = P.row_elems;
    const unsigned nthreads = kCols ? kCols / 2u : blockDim.x, tid = threadIdx.x;
    const int codec = s.op.codec;
    const unsigned raw_bits = (unsigned)td_raw_bits(codec);
    unsigned long long *rows = reinterpret_cast<unsigned long long *>(smem_raw);            // [64], and two to spare
    unsigned *scratch = reinterpret_cast<unsigned *>(rows + 66);                             // 32 words
    unsigned char *stage = smem_raw + kTdEncodeHead;
    const TdLayout &lay = P.layout[blockIdx.z];
    const unsigned long long row = (unsigned long long)s.seg * RE;
    const bool act = 2u * tid < C;
    // this kernel may start as soon as the scan's CTAs have seen the planner end: the row addresses are what it can have ready
    const bool bad = td_row_addresses<true, false>(P, s, rows, tid, nthreads);
    dependency_wait();
    release_dependents();
    const TdOffsets o = td_offsets(s.op.data + lay.lens + row, s.c0, C, nthreads, scratch);
    const unsigned long long seg_begin = reinterpret_cast<const unsigned long long *>(s.op.data)[s.seg];
    unsigned char *dst = s.op.data + seg_begin + o.before;
    const unsigned shift = (unsigned)((unsigned long long)dst & 15ull);                      // staging mirrors the destination's alignment
    // the lengths are the planner's, but a planner CTA may have given up: nothing may leave the staging area or the chunk
    // (the capacity ends on a 16-byte boundary, so the padding of a segment's last slice fits whenever its bytes do)
    const bool sane = o.slice <= C * td_max_len(codec) && seg_begin >= lay.streams && seg_begin + o.before + o.slice <= lay.capacity;
    for (unsigned i = tid; i < (shift + (sane ? o.slice : 0u) + 31u) / 16u; i += nthreads) sts128(stage + (size_t)i * 16u, make_uint4(0u, 0u, 0u, 0u));
    if (__syncthreads_or(bad || !sane)) {                                                     // (also publishes the zeros and the rows)
        if (tid == 0) atomicCAS(P.status, 0, kStatusRange);
        return;
    }
    const unsigned len_x = o.pair & 0xffu, len_y = o.pair >> 8;
    // (a length of zero: the planner gave this slice up)
    const bool coding = act && len_x != 0u && len_y != 0u && len_x <= td_max_len(codec) && len_y <= td_max_len(codec);
    TdOut x, y;
    if (coding) {
        const unsigned long long at = row + s.c0 + 2u * tid;
        const unsigned params = *reinterpret_cast<const unsigned short *>(s.op.data + lay.params + at);
        const float2 sc = *reinterpret_cast<const float2 *>(s.op.data + lay.scales + 4ull * at);
        const float qmax = (float)td_qmax(codec);
        const float inv_x = sc.x != 0.0f ? __fdiv_rn(qmax, __bfloat162float(__float2bfloat16_rn(__fmul_rn(sc.x, qmax)))) : 0.0f;
        const float inv_y = sc.y != 0.0f ? __fdiv_rn(qmax, __bfloat162float(__float2bfloat16_rn(__fmul_rn(sc.y, qmax)))) : 0.0f;
        const uint32_t addr_x = smem_u32(stage) + shift + o.off;
        td_out_init(x, addr_x, params & 0xffu);
        td_out_init(y, addr_x + len_x, params >> 8);
        // per token: m + code (m = 1.5 * 2^23), minus m or the token before (delta mode), all exact
        const float m = 12582912.0f;
        const f32x2 inv2 = pack2(inv_x, inv_y), m2 = pack2(m, m), one2 = pack2(P.fone, P.fone), two2 = pack2(2.0f, 2.0f), half2 = pack2(0.5f, 0.5f);
        const bool dx = (params & 8u) != 0u, dy = (params & 0x800u) != 0u;
        const f32x2 nd2 = pack2(dx ? -1.0f : 0.0f, dy ? -1.0f : 0.0f), nc2 = pack2(dx ? 0.0f : -m, dy ? 0.0f : -m);
        f32x2 base = pack2(-m, -m);
        const float zero_x = x.k ? 8388607.5f : 8388606.5f, zero_y = y.k ? 8388607.5f : 8388606.5f;
        auto per_len = [&](unsigned k) { return __uint_as_float((127u - k) << 23); };           // 2^-k
        const f32x2 per2 = pack2(-per_len(x.k), -per_len(y.k));
        auto len_zero = [&](unsigned k) { return k ? kTdLenZero + 8388608.0f * per_len(k) - (float)(k + 1u) : kTdLenZero + 8388606.0f; };
        const f32x2 len2 = pack2(len_zero(x.k), len_zero(y.k));
        float px, py, lx, ly;
        unpack2(per2, px, py);
        unpack2(len2, lx, ly);
        auto symbol = [&](uint32_t v, uint32_t &a, uint32_t &b) {
            const f32x2 r = add2_unfused(mul2(bf16x2_widen(v), inv2), m2, one2);
            const f32x2 f = fma2(add2(r, base), two2, half2);
            base = fma2(r, nd2, nc2);
            float fa, fb;
            unpack2(f, fa, fb);
            a = __float_as_uint(__fadd_rn(fabsf(fa), zero_x));
            b = __float_as_uint(__fadd_rn(fabsf(fb), zero_y));
        };
        // the same of token t, whatever it is (one that is not finite also spoils `base`)
        auto again = [&](unsigned t, uint32_t &a, uint32_t &b) {
            const uint32_t v = __ldcg(reinterpret_cast<const uint32_t *>(rows[t]) + tid);
            const uint32_t u = t ? __ldcg(reinterpret_cast<const uint32_t *>(rows[t - 1u]) + tid) : 0u;
            const int qx = td_code(v & 0xffffu, inv_x), qy = td_code(v >> 16, inv_y);
            const int ex = dx ? qx - td_code(u & 0xffffu, inv_x) : qx, ey = dy ? qy - td_code(u >> 16, inv_y) : qy;
            a = __float_as_uint((float)((x.k ? 8388608 : 8388607) + ((ex << 1) ^ (ex >> 31))));
            b = __float_as_uint((float)((y.k ? 8388608 : 8388607) + ((ey << 1) ^ (ey >> 31))));
            base = fma2(pack2(m + (float)qx, m + (float)qy), nd2, nc2);
        };
        // kTdLoad tokens at a time, the next ones already on their way
        auto load = [&](unsigned t0, uint32_t (&v)[kTdLoad]) {
            const ulonglong2 *r = reinterpret_cast<const ulonglong2 *>(rows + t0);
#pragma unroll
            for (int i = 0; i < (int)kTdLoad; i += 2) {
                const ulonglong2 d = r[i / 2];
                v[i] = __ldcg(reinterpret_cast<const uint32_t *>(d.x + (unsigned long long)(2u * tid) * P.pow2[1]));
                v[i + 1] = __ldcg(reinterpret_cast<const uint32_t *>(d.y + (unsigned long long)(2u * tid) * P.pow2[1]));
            }
        };
        auto code = [&](auto join) -> unsigned {
            unsigned t0 = 0;
            uint32_t v[kTdLoad], next[kTdLoad];
            if (kTdLoad <= s.n_tok) load(0u, next);
#pragma unroll 1
            for (; t0 + kTdLoad <= s.n_tok; t0 += kTdLoad) {
#pragma unroll
                for (int i = 0; i < (int)kTdLoad; ++i) v[i] = next[i];
                if (t0 + 2u * kTdLoad <= s.n_tok) load(t0 + kTdLoad, next);
#pragma unroll
                for (int i = 0; i < (int)kTdLoad; i += 4) {
                    uint32_t ux[4], uy[4];
                    float nx[4], ny[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        symbol(v[i + j], ux[j], uy[j]);
                        unpack2(td_fma2_up(pack2_bits(ux[j], uy[j]), per2, len2), nx[j], ny[j]);
                    }
                    td_append4<decltype(join)::value>(x, y, ux, uy, nx, ny, px, py, lx, ly, raw_bits, [&](unsigned j, uint32_t &a, uint32_t &b) { again(t0 + (unsigned)i + j, a, b); });
                }
            }
            return t0;
        };
        unsigned t0 = codec == 6 ? code(TdJoin<4>()) : code(TdJoin<2>());
#pragma unroll 1
        for (; t0 < s.n_tok; ++t0) {
            uint32_t ux, uy;
            symbol(__ldcg(reinterpret_cast<const uint32_t *>(rows[t0]) + tid), ux, uy);
            if (max(ux, uy) > 0x7f800000u) again(t0, ux, uy);
            td_append_any(x, ux, td_fma_up(__uint_as_float(ux), px, lx), raw_bits);
            td_append_any(y, uy, td_fma_up(__uint_as_float(uy), py, ly), raw_bits);
        }
        td_out_pad(x);
        td_out_pad(y);
    }
    __syncthreads();                                         // the whole words of all sub-streams are out
    if (coding) {
        td_out_last(x);
        td_out_last(y);
    }
    // the last slice of a segment also writes the zero bytes that pad the segment to 16
    unsigned pad = 0;
    if (s.part == P.n_split - 1u) {
        pad = (16u - ((shift + o.slice) & 15u)) & 15u;
        if (tid < pad) {
            const unsigned i = shift + o.slice + tid;
            const uint32_t word = 0xff000000u >> (8u * (i & 3u));
            asm volatile("red.shared.or.b32 [%0], %1;" :: "r"(smem_u32(stage) + (i & ~3u)), "r"(word) : "memory");
        }
    }
    __syncthreads();
    const unsigned n_out = o.slice + pad;
    // staging -> chunk, words turned to little-endian and complemented: bytes up to the first 16-byte boundary, 16-byte vectors,
    // bytes after the last boundary
    const unsigned head = shift ? (16u - shift < n_out ? 16u - shift : n_out) : 0u;
    const unsigned vecs = (n_out - head) >> 4, tail = (n_out - head) & 15u;
    auto byte_at = [&](unsigned i) { return (unsigned char)~(*reinterpret_cast<const uint32_t *>(stage + (i & ~3u)) >> (24u - 8u * (i & 3u))); };
    if (tid < head) dst[tid] = byte_at(shift + tid);
    for (unsigned v = tid; v < vecs; v += nthreads) {
        const uint4 w = lds128(stage + shift + head + (size_t)v * 16u);
        *reinterpret_cast<uint4 *>(dst + head + (size_t)v * 16u) = make_uint4(~td_be(w.x), ~td_be(w.y), ~td_be(w.z), ~td_be(w.w));
    }
    if (tid < tail) dst[head + vecs * 16u + tid] = byte_at(shift + head + vecs * 16u + tid);
}

// ----------------------------------------------------------------------------------- retrieve / compose --

// One sub-stream on its way through the decoder.  Everything is kept in the form that takes the fewest operations of the
// pipe that shifts, compares and logic share (it issues every other cycle and is what bounds this kernel):
//  * the words hold the complement of the stream, so the ones of the unary part are leading zeros.  With h the next 32
//    bits, n = clz(h) and len = n + k + 1, z = h >> (32 - len) = 2^(k+1) - 1 - rem, and v = z - n 2^k = c - u with
//    c = 2^(k+1) - 1, the symbol u never appears itself;
//  * 2 e (e = the signed code or code difference) is u for even u and -(u + 1) for odd u, i.e. v - c - 1, or, where v is odd,
//    2 c + 1 - v - c - 1: one predicated multiply-add (it runs on the other integer pipe; its constant factors arrive as launch
//    parameters: known ones would be turned back into shifts and adds);
//  * the running code is kept as the bits of the fp32 number 2^22 + 512 + q, whose unit in the last place is 1/2: adding
//    2 e to the bits adds e to the number, and one subtraction gives q exactly.
struct TdStream {
    uint32_t col;          // shared address of word 0 of the sub-stream
    unsigned bp;           // bits consumed
    unsigned nk1;          // -(k + 1)
    int kneg;              // -2^k
    int c21;               // 2 c + 1
    int d, c2;             // next = acc * d + c2 + ...: d = 1 in delta mode, else 0 and c2 holds the fresh start
    int acc;
};
constexpr int kTdCodeBits = 0x4A800000 + 1024;             // 2^22 + 512 as fp32 bits
constexpr float kTdCodeZero = 4194304.0f + 512.0f;

__device__ __forceinline__ void td_stream_init(TdStream &s, uint32_t col, unsigned param)
{
    const unsigned k = param & 7u;
    const int c = (int)((2u << k) - 1u);
    s.col = col;
    s.bp = 0u;
    s.nk1 = 0u - (k + 1u);
    s.kneg = -(int)(1u << k);
    s.c21 = 2 * c + 1;
    s.d = (param & 8u) ? 1 : 0;
    s.c2 = -(c + 1) + ((param & 8u) ? 0 : kTdCodeBits);
    s.acc = kTdCodeBits;
}
template <unsigned kCols>
__device__ __forceinline__ uint32_t td_window(const TdStream &s, unsigned row_b)
{
    const uint32_t a = (s.bp >> 5) * row_b + s.col;
    uint32_t w0, w1;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(w0) : "r"(a));
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(w1) : "r"(a + (kCols ? kCols * 4u : row_b)));
    return __funnelshift_l(w1, w0, s.bp);
}
// The next symbol out of the window h, taken not to be an escape; returns the length of its unary part (15 and more: it was one)
// and, in nlen, minus the length of the code word (shifts take their count modulo 32: by nlen means by 32 - len).
__device__ __forceinline__ unsigned td_symbol(const TdLaunch &P, TdStream &s, uint32_t h, unsigned &nlen)
{
    unsigned n;
    asm("bfind.shiftamt.u32 %0, %1;" : "=r"(n) : "r"(h));
    nlen = s.nk1 - n;
    int v = (int)n * s.kneg + (int)__funnelshift_r(h, 0u, nlen);
    asm("{ .reg .pred p; .reg .b32 t; and.b32 t, %0, 1; setp.ne.s32 p, t, 0; @p mad.lo.s32 %0, %0, %1, %2; }" : "+r"(v) : "r"(P.minus_one), "r"(s.c21));
    s.acc = v + (s.acc * s.d + s.c2);
    return n;
}
// The same with escapes.
__device__ __forceinline__ void td_symbol_any(const TdLaunch &P, TdStream &s, uint32_t h, unsigned raw_bits)
{
    if ((h >> 17) != 0u) {                                  // fewer than fifteen ones
        unsigned nlen;
        td_symbol(P, s, h, nlen);
        s.bp -= nlen;
        return;
    }
    const int u = (int)((~h << 15) >> (32u - raw_bits));
    s.bp += 15u + raw_bits;
    s.acc = (u ^ -(u & 1)) + (s.d ? s.acc : kTdCodeBits);
}

// kStep symbols of two streams side by side, kWin of them out of one 32-bit window. Taken to be no escapes and to fit their windows; where that was
// wrong, once more with care, which takes about three times as long, and one lane's escape holds up its warp: so a step is no longer than
// it has to be.
template <unsigned kCols, unsigned kWin, unsigned kStep>
__device__ __forceinline__ void td_step(const TdLaunch &P, TdStream &x, TdStream &y, unsigned row_b, unsigned raw_bits, int (&vx)[kStep], int (&vy)[kStep])
{
    const unsigned bp_x = x.bp, bp_y = y.bp;
    const int acc_x = x.acc, acc_y = y.acc;
    unsigned longest = 0, most = 0;
#pragma unroll
    for (unsigned i = 0; i < kStep; i += kWin) {
        uint32_t hx = td_window<kCols>(x, row_b), hy = td_window<kCols>(y, row_b);
        unsigned bx = 0u, by = 0u;                          // minus the bits taken out of the window
#pragma unroll
        for (unsigned j = 0; j < kWin; ++j) {
            unsigned lx, ly;
            const unsigned nx = td_symbol(P, x, hx, lx), ny = td_symbol(P, y, hy, ly);
            longest = __vimax3_u32(longest, nx, ny);
            bx += lx; by += ly;
            hx = __funnelshift_r(0u, hx, lx);               // hx << length
            hy = __funnelshift_r(0u, hy, ly);
            vx[i + j] = x.acc; vy[i + j] = y.acc;
        }
        x.bp -= bx; y.bp -= by;
        most = __vimax3_u32(most, 0u - bx, 0u - by);
    }
    if (__builtin_expect(longest >= 15u || most > 32u, 0)) {
        x.bp = bp_x; y.bp = bp_y; x.acc = acc_x; y.acc = acc_y;
#pragma unroll
        for (unsigned i = 0; i < kStep; ++i) {
            td_symbol_any(P, x, td_window<kCols>(x, row_b), raw_bits);
            td_symbol_any(P, y, td_window<kCols>(y, row_b), raw_bits);
            vx[i] = x.acc; vy[i] = y.acc;
        }
    }
}

// Bound by instruction issue and the integer pipes (8B shape, 4-bit codes: issue slots 81 %, logic 57 %, DRAM 37 %, 19.8 warp instructions per 32
// symbols; 8-bit codes 73 %, 49 %, 39 %, 22.3, with ten CTAs an SM where 4-bit codes have fourteen); what was done about it is at TdStream and td_step.  A
// thread decodes two channels side by side -- neighbours, whose bf16 values make one word, or, where keys are re-rotated, the two channels of a rotation pair --
// so that one stream's chain of dependent operations hides the other's, and writes finished values into the rows: no pass over codes.  Half
// of the rows at a time keeps a CTA of 64 threads at 15 KiB of shared memory (8-bit codes: 20); all rows at a time were
// 15 % slower.  The rows leave with 128-bit stores, sixteen lanes to a 256-byte piece of a token row.  8B shape, 32 chunks of 512
// tokens, correlation 0.9: 4-bit codes 1728 us with one thread per channel, a code tile and a separate pass that multiplied, 696 us this way; 8-bit
// codes 1765 -> 873 us.
// kCols: channels per CTA when known at compile time (the usual slice; every stride in the decoding loop is then an
// immediate), 0: taken from the launch record.
// kCodec: the codec of the launch's chunks, 0 where it has chunks of both.  (A kernel per codec takes fewer instructions, but a launch for each
// half of such a call leaves the SMs to half a call at a time and pays for one more.  8B shape, us a retrieve, two launches / one: a chunk of each codec,
// 64 tokens 16.2 / 13.5, 512 tokens 65.2 / 59.5, sixteen of each 1064 / 1008; compose, eight of each, 331 tokens, 70B shape with two heads 269 / 252.  Two
// whole bodies behind one branch were no good: 1145 and 288.)
template <bool kCompose, unsigned kCols, int kCodec>
__global__ void __launch_bounds__(kCols ? kCols / 2u : 512u, kCols ? 12 : 1) kdn_td_decode_kernel(const __grid_constant__ TdLaunch P)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    dependency_wait();
    release_dependents();
    const TdSlice s = td_slice(P);
    if (!s.valid) return;
    const int codec = kCodec ? kCodec : s.op.codec;
    const unsigned kWords = td_words(codec), raw_bits = (unsigned)td_raw_bits(codec);
    const unsigned C = kCols ? kCols : P.cols, RE = P.row_elems;
    const unsigned nthreads = kCols ? kCols / 2u : blockDim.x;

    uint32_t *I = reinterpret_cast<uint32_t *>(smem_raw);                // interleaved sub-streams [word][C]
    unsigned char *A = smem_raw + td_decode_words_bytes(C, kWords);     // the slice's stream bytes, then bf16 rows [kTdHalf][C]
    unsigned *offs = reinterpret_cast<unsigned *>(A + td_decode_rows_bytes(C, kWords));   // where each channel's sub-stream starts
    unsigned long long *rows = reinterpret_cast<unsigned long long *>(offs + C);     // pool address of each token row's slice, 0: not written
    unsigned *scratch = reinterpret_cast<unsigned *>(rows + 64);         // 64 words
    unsigned long long *bar_mem = reinterpret_cast<unsigned long long *>(reinterpret_cast<unsigned char *>(scratch) + 256u);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(bar_mem + 1);
    const uint32_t bar = smem_u32(bar_mem);
    const unsigned tid = threadIdx.x;
    if (tid == 0) {
        mbar_init(bar, 1u);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_async_smem();
    }
    // a select-list (compose): which of its entries fall into this group?  Two threads look; none: nothing to do here
    const bool selecting = kCompose && s.op.list_mode == 2;
    if (selecting && tid < 2u) scratch[40u + tid] = td_lower_bound(s.op.list, (unsigned)s.op.n_list, ((long long)s.g + tid) << 6);
    const TdLayout &lay = P.layout[blockIdx.z];
    const unsigned long long row = (unsigned long long)s.seg * RE;
    const unsigned char *lens = s.op.data + lay.lens + row;
    const bool act = 2u * tid < C;
    const TdOffsets o = td_offsets(lens, s.c0, C, nthreads, scratch);     // (its barrier also publishes the mbarrier and the two indices)
    if (selecting && scratch[40] >= scratch[41]) return;                  // every thread alike, and no copy has been started
    const unsigned total_before = o.before, total_slice = o.slice, my_off = o.off, pair = o.pair;
    const unsigned long long seg_begin = reinterpret_cast<const unsigned long long *>(s.op.data)[s.seg];
    const unsigned long long src = seg_begin + total_before;
    const unsigned shift = (unsigned)(((unsigned long long)s.op.data + src) & 15ull);
    const unsigned bytes_al = (shift + total_slice + 15u) & ~15u;
    // a damaged chunk must not send a copy outside the chunk or outside the staging area
    // (op.scales, which these codecs have no other use for, points behind the bytes of the chunk that exist at op.data:
    // its capacity, or what a staging slab holds of it)
    const unsigned long long exist = (unsigned long long)(s.op.scales - s.op.data);
    const unsigned long long have = exist < lay.capacity ? exist : lay.capacity;
    const bool sane = total_slice <= C * td_max_len(codec) && src >= lay.streams && src <= have && src - shift + bytes_al <= have;
    if (tid == 0) {
        if (!sane) {
            atomicCAS(P.status, 0, kStatusRange);
            *abort_flag = 1;
        } else if (bytes_al != 0u) {
            mbar_arrive_expect_tx(bar, bytes_al);
            const unsigned char *g = s.op.data + src - shift;
            for (unsigned o = 0; o < bytes_al; o += 32768u)
                bulk_g2s(smem_u32(A + o), g + o, bytes_al - o < 32768u ? bytes_al - o : 32768u, bar);
        } else {
            mbar_arrive(bar);
        }
    }
    // while the bytes are on their way: the thread's two channels, and where the rows go
    const bool rotating = kCompose && s.kv == 0u && s.op.rope >= 0;
    const unsigned half = (unsigned)P.D >> 1;
    const unsigned head = rotating ? tid / half : 0u;
    const unsigned ca = rotating ? head * (unsigned)P.D + (tid - head * half) : 2u * tid;   // first channel, inside the slice
    const unsigned cb = rotating ? ca + half : ca + 1u;
    unsigned param_a = 0, param_b = 0;
    float sc_a = 0.0f, sc_b = 0.0f;
    if (act) {
        const unsigned char *params = s.op.data + lay.params + row + s.c0;
        const float *scales = reinterpret_cast<const float *>(s.op.data + lay.scales) + row + s.c0;
        param_a = params[ca]; param_b = params[cb];
        sc_a = scales[ca]; sc_b = scales[cb];
        offs[2u * tid] = my_off | ((pair & 0xffu) << 24);                 // (a slice holds fewer than 2^24 bytes)
        offs[2u * tid + 1u] = (my_off + (pair & 0xffu)) | ((pair >> 8) << 24);
    }
    {
        unsigned char *base = reinterpret_cast<unsigned char *>((s.kv ? P.v_layers : P.k_layers)[s.op.l0 + (int)s.li]);
        if (selecting) {
            for (unsigned r = tid; r < 64u; r += nthreads) rows[r] = 0ull;
            __syncthreads();
        }
        // the rows of the group, or its listed ones
        const unsigned first = selecting ? scratch[40] : 0u, last = selecting ? scratch[41] : s.n_tok;
        for (unsigned i = first + tid; i < last; i += nthreads) {
            bool bad = false;
            unsigned r = i;
            if (selecting) {
                const long long c = (long long)s.op.list[i] - ((long long)s.g << 6);
                bad = c < 0 || c >= (long long)s.n_tok;                   // (a list that is not increasing)
                r = (unsigned)c;
            }
            if (!bad) {
                const long long pos = group_row_pos(s.op, s.g, r);
                bad = pos < 0;
                if (!bad) {
                    const long long blk = P.bs_shift >= 0 ? pos >> P.bs_shift : pos / P.bs;
                    const long long id = s.op.table[blk];
                    bad = id < 0 || id >= P.n_blocks;
                    if (!bad) rows[r] = (unsigned long long)(base + ((unsigned long long)(id * P.bs + (pos - blk * P.bs)) * RE + s.c0) * 2ull);
                }
            }
            if (bad) {
                atomicCAS(P.status, 0, kStatusRange);
                *abort_flag = 2;                                          // nothing of this slice is written
            }
        }
    }
    const bool landed = mbar_wait(bar, 0u, abort_flag, P.wait_limit_ns);
    if (!__syncthreads_and(landed)) {                                     // all threads leave together
        if (tid == 0 && sane) {
            if (*abort_flag != 2) atomicCAS(P.status, 0, kStatusTimeout);
            // the CTA does not leave while a copy into its shared memory is in flight
            const unsigned long long t0 = global_timer_ns();
            while (!mbar_try_wait(bar, 0u))
                if (global_timer_ns() - t0 > kWaitLimitNs) break;
        }
        return;
    }
    if (*abort_flag) return;
    TdStream x, y;
    if (act) {
        // the sub-streams, as complemented big-endian words, into two columns of the interleaved area (the first streams
        // of all threads, then the second ones): word j of every channel sits in one row, so a warp's loads below never
        // meet in a bank wherever each lane is in its stream
        const unsigned oa = offs[ca], ob = offs[cb];
        unsigned len_a = oa >> 24, len_b = ob >> 24;
        // (a length no sub-stream can have means a damaged chunk: reported, and clamped so that nothing leaves the area)
        if (len_a > td_max_len(codec) || len_b > td_max_len(codec)) atomicCAS(P.status, 0, kStatusRange);
        len_a = len_a < td_max_len(codec) ? len_a : td_max_len(codec);
        len_b = len_b < td_max_len(codec) ? len_b : td_max_len(codec);
        const uint32_t addr_a = smem_u32(A) + shift + (oa & 0xffffffu), addr_b = smem_u32(A) + shift + (ob & 0xffffffu);
        const uint32_t al_a = addr_a & ~3u, al_b = addr_b & ~3u;
        const uint32_t sel_a = 0x0123u + (addr_a & 3u) * 0x1111u, sel_b = 0x0123u + (addr_b & 3u) * 0x1111u;   // realign and swap bytes
        const unsigned nw = (((len_a > len_b ? len_a : len_b) + 3u) >> 2) + 1u;     // the window looks one word past the last bit
        uint32_t a0, a1, b0, b1;
        asm volatile("ld.shared.u32 %0, [%1];" : "=r"(a0) : "r"(al_a));
        asm volatile("ld.shared.u32 %0, [%1];" : "=r"(b0) : "r"(al_b));
        uint32_t *col_a = I + tid, *col_b = I + (C >> 1) + tid;
#pragma unroll 2
        for (unsigned j = 0; j < nw; ++j) {
            asm volatile("ld.shared.u32 %0, [%1];" : "=r"(a1) : "r"(al_a + 4u * (j + 1u)));
            asm volatile("ld.shared.u32 %0, [%1];" : "=r"(b1) : "r"(al_b + 4u * (j + 1u)));
            col_a[(size_t)j * C] = ~__byte_perm(a0, a1, sel_a);
            col_b[(size_t)j * C] = ~__byte_perm(b0, b1, sel_b);
            a0 = a1; b0 = b1;
        }
        td_stream_init(x, smem_u32(col_a), param_a);
        td_stream_init(y, smem_u32(col_b), param_b);
    }
    __syncthreads();                                                      // stream bytes no longer read: the rows may be written
    const unsigned row_b = P.word_row, max_bits = (kWords - 1u) * 32u;   // a sub-stream's last symbol starts before that bit
    const f32x2 sc2 = pack2(sc_a, sc_b), zero2 = pack2(-kTdCodeZero, -kTdCodeZero);
    f32x2 cc = 0ull, ss = 0ull;
    if (rotating && act) {
        const float2 cs = *(P.rope + (size_t)s.op.rope * half + (tid - head * half));
        cc = pack2(cs.x, cs.x);
        ss = pack2(-cs.y, cs.y);
    }
    const uint32_t out = smem_u32(A) + ca * 2u;
    auto put = [&](unsigned t, int acc_x, int acc_y) {
        const f32x2 val = mul2(add2(pack2(__int_as_float(acc_x), __int_as_float(acc_y)), zero2), sc2);
        const uint32_t o = out + t * (C * 2u);
        if (kCompose && rotating) {
            float u, w;
            unpack2(val, u, w);
            const uint32_t r = pack_bf16x2(fma2(val, cc, mul2(pack2(w, u), ss)));         // u cos - w sin, w cos + u sin
            asm volatile("st.shared.u16 [%0], %1;" :: "r"(o), "h"((unsigned short)r) : "memory");
            asm volatile("st.shared.u16 [%0], %1;" :: "r"(o + half * 2u), "h"((unsigned short)(r >> 16)) : "memory");
        } else {
            asm volatile("st.shared.u32 [%0], %1;" :: "r"(o), "r"(pack_bf16x2(val)) : "memory");
        }
    };
    const unsigned vecs = C >> 3;                                          // 16-byte vectors per row
#pragma unroll 1
    for (unsigned t0 = 0; t0 < s.n_tok; t0 += kTdHalf) {
        const unsigned nt = s.n_tok - t0 < kTdHalf ? s.n_tok - t0 : kTdHalf;
        if (act) {
            unsigned t = 0;
            auto clamp = [&]() {                             // (a damaged stream cannot run off the area: at most eight symbols between two of these)
                x.bp = x.bp < max_bits ? x.bp : max_bits;
                y.bp = y.bp < max_bits ? y.bp : max_bits;
            };
            // steps of step symbols, win to a window, in rounds of times steps; whole: no round that would end past nt
            auto steps = [&](auto win, auto step, auto times, auto whole) {
                constexpr unsigned kStep = (unsigned)decltype(step)::value, kTimes = (unsigned)decltype(times)::value;
                constexpr bool kWhole = decltype(whole)::value != 0;
#pragma unroll 1
                for (; t + (kWhole ? kTimes * kStep : kStep) <= nt; t += kWhole ? kTimes * kStep : 0u) {
                    clamp();
#pragma unroll
                    for (unsigned i = 0; i < kTimes; ++i) {
                        if (!kWhole && i && t + kStep > nt) break;
                        int vx[kStep], vy[kStep];
                        td_step<kCols, (unsigned)decltype(win)::value, kStep>(P, x, y, row_b, raw_bits, vx, vy);
#pragma unroll
                        for (unsigned j = 0; j < kStep; ++j) put(t + (kWhole ? i * kStep : 0u) + j, vx[j], vy[j]);
                        if (!kWhole) t += kStep;
                    }
                }
            };
            // A look for escapes after every window of 4-bit codes (four to one) and every second one of 8-bit codes, two steps a round, and a last half-round
            // before single symbols.  Against a look every six or eight symbols and up to seven single ones at the end, 8B shape, us a retrieve: sixteen
            // chunks of 512 tokens with heavy tails (t distribution, three degrees) 727 -> 659, thirty-two with a jump every 16 tokens 1127 -> 1042 and (4-bit)
            // 940 -> 817, thirty-two of 7 tokens (4-bit) 33.3 -> 30.2, one of 61 tokens 9.5 -> 7.9, of 29 (4-bit) 6.1 -> 5.25; without any of that the same
            // (878 -> 874, 700 -> 698).  8-bit codes in compose keep three to a window, which the code of a rotation makes worth while (70B shape, two heads,
            // 219 -> 216, with jumps 268 -> 240; pairs 226 and 258); in a short launch a window that overflows costs more than that gives, so retrieves take
            // pairs.  Rounds that may end in the middle share their code with the end of a half: better where a rotation has made the code long (4-bit
            // codes in compose 184 -> 178, with jumps 227 -> 201), worse elsewhere (698 -> 721).
            const TdConst<0> part;
            const TdConst<1> one, whole;
            const TdConst<2> two;
            const TdConst<3> three;
            const TdConst<4> four;
            if (codec == 6) {
                if constexpr (!kCompose && kCodec) { steps(four, four, two, whole); steps(four, four, one, whole); }
                else if constexpr (kCols || !kCodec) steps(four, four, two, part);
                else steps(four, four, one, whole);
            } else {
                if constexpr (!kCompose && kCodec) { steps(two, four, two, whole); steps(two, four, one, whole); }
                else if constexpr (kCompose && kCodec && kCols) { steps(three, three, two, whole); steps(two, two, one, whole); }
                else if constexpr (!kCompose) steps(two, four, two, part);
                else if constexpr (!kCodec) steps(two, two, two, part);
                else steps(two, four, one, whole);
            }
#pragma unroll 1
            for (; t < nt; ++t) {
                clamp();
                td_symbol_any(P, x, td_window<kCols>(x, row_b), raw_bits);
                td_symbol_any(P, y, td_window<kCols>(y, row_b), raw_bits);
                put(t, x.acc, y.acc);
            }
        }
        __syncthreads();
        // rows -> pool blocks, sixteen bytes a lane
        if (kCols && nt == kTdHalf) {
            constexpr unsigned kLanes = kCols ? kCols / 8u : 1u, kStep = kCols ? kCols / 2u / kLanes : 1u;      // lanes a row, rows a pass
            const unsigned c = tid & (kLanes - 1u), r = tid / kLanes;
#pragma unroll
            for (unsigned i = 0; i < kTdHalf; i += kStep) {
                const unsigned long long d = rows[t0 + i + r];
                if (d) *reinterpret_cast<uint4 *>(d + 16ull * c) = lds128(A + (size_t)((i + r) * kLanes + c) * 16u);
            }
        } else {
            for (unsigned v = tid; v < nt * vecs; v += nthreads) {
                const unsigned t = v / vecs, c = v - t * vecs;
                const unsigned long long d = rows[t0 + t];
                if (d) *reinterpret_cast<uint4 *>(d + 16ull * c) = lds128(A + (size_t)v * 16u);
            }
        }
        __syncthreads();
    }
}

}  // namespace kdn

// Store and retrieve one token row at a time, without the tile pipeline: for keep-lists over short rows, which sit anywhere in the
// pool, and for pool blocks so small that a block is no more than a row or two.  There the tile pipeline is bound by the two threads
// of a CTA that issue its bulk copies (one a row: about 0.16 us each), not by memory.  Here every thread moves vectors between the
// chunk and the pool by itself, coding or decoding them on the way: sixteen elements (or eight, where bf16 may have to be
// retrieved).  Loads are 16 bytes a lane, contiguous over the warp: 16-byte loads 32 bytes apart cost 40 %.
//
// A CTA takes a set of rows of one op, kJ vectors a thread, and goes through some of the op's planes with them.  The rows' places in the
// pool are looked up once.  Per plane each thread's vectors come in through asynchronous copies into shared-memory
// slots that only this thread uses -- a deeper queue than registers would hold -- kStages planes ahead, counted on an mbarrier
// per stage (bounded waits, as in the tile pipeline); nothing else is synchronised.  On the chunk side a CTA's vectors are
// contiguous whatever the rows do; on the pool side a row is.  Bound by memory and, when coding, by the latency of a plane: 8B shape with
// two heads, half of 16 x 1024 tokens kept, int8: retrieve 76 us (5.4 TB/s), store 78 us (5.3 TB/s).  Loads into registers instead of
// slots: 92 and 87 us.  (The retrieve of vectors of sixteen elements spills 24 bytes at the 64 registers that four CTAs an SM leave.)
#pragma once

#include "kdn_kernels.cuh"

namespace kdn {

constexpr unsigned kRowsThreads = 256;
constexpr int kRowsStages = 2;             // planes in flight a CTA (of four CTAs an SM: 64 KiB of bf16, or of codes; three or four lose 10 %)
constexpr int kRowsVectors = 4;            // slots a thread fills for a plane
constexpr unsigned kRowsPerCta = 256;      // rows a CTA takes at most (one look-up a thread)

struct RowsLaunch {
    const DevOp *ops;         // device array, or nullptr: inline_ops.  tile_begin counts CTAs.
    int n_ops;
    void *const *k_layers;
    void *const *v_layers;
    long long n_blocks;
    int bs;
    int bs_shift;             // log2(bs), -1 where bs is not a power of two
    unsigned row_elems;
    unsigned vpr;             // vectors per row
    unsigned vpr_magic;       // v / vpr = the high word of v * vpr_magic for every vector of a CTA (0: one row per CTA, or vpr = 1)
    unsigned rows;            // token rows per CTA
    unsigned planes;          // planes a CTA goes through
    unsigned unit;            // rows that are given up together when one of them has no place
    int *status;
    unsigned long long wait_limit_ns;
    float one;                // 1.0f (see Launch::one)
    DevOp inline_ops[kInlineOps];
};

__host__ __device__ constexpr size_t rows_smem_bytes(int kJ)
{
    // slots, scales, places, barriers and the abort word
    return (size_t)kRowsStages * kJ * kRowsThreads * (16u + 4u) + kRowsPerCta * 8u + 8u * kRowsStages + 16u;
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src) { asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory"); }
__device__ __forceinline__ void cp_async8(uint32_t dst, const void *src) { asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory"); }
__device__ __forceinline__ void cp_async4(uint32_t dst, const void *src) { asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory"); }
// One of the barrier's expected arrivals, made when all of the thread's copies so far have landed.
__device__ __forceinline__ void cp_async_arrive(uint32_t bar) { asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(bar) : "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0u;
}
// Bounded wait, `since` = when the CTA started.  A limit shorter than a thread may be parked for is kept by looking at the clock.
__device__ __forceinline__ bool rows_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag, unsigned long long limit_ns, unsigned long long since)
{
    if (mbar_test(bar, parity)) return true;
    if (limit_ns >= 20000ull) return mbar_wait_slow(bar, parity, abort_flag, limit_ns);
    while (!mbar_test(bar, parity))
        if (*abort_flag || global_timer_ns() - since > limit_ns) { *abort_flag = 1; return false; }
    return true;
}

// Sixteen bf16 elements of a group of 64 that four neighbouring lanes hold -> codes (int8: four words, int4: two) and the group's
// scale: the arithmetic of quantise_tile.
template <bool kInt4>
__device__ __forceinline__ uint4 rows_quantise(uint4 a, uint4 b, float one, float &scale)
{
    uint32_t m = maxabs_bf16x2(maxabs_bf16x2(maxabs_bf16x2(a.x, a.y), maxabs_bf16x2(a.z, a.w)), maxabs_bf16x2(maxabs_bf16x2(b.x, b.y), maxabs_bf16x2(b.z, b.w)));
    m = maxabs_bf16x2(m, __shfl_xor_sync(0xffffffffu, m, 1));
    m = maxabs_bf16x2(m, __shfl_xor_sync(0xffffffffu, m, 2));
    const float qmax = kInt4 ? 7.0f : 127.0f;
    const float top = fmaxf(__uint_as_float((m << 16) & 0x7fffffffu), __uint_as_float(m & 0x7fff0000u));
    const bool odd = (threadIdx.x & 1u) != 0u;             // the two divides are made by the even and the odd lanes
    const float mine = __fdiv_rn(odd ? qmax : top, odd ? top : qmax);
    const float other = __shfl_xor_sync(0xffffffffu, mine, 1);
    scale = odd ? other : mine;
    const bool ok = scale >= 1.17549435e-38f;              // smallest normal fp32; false for NaN too
    const float inv = ok ? (odd ? mine : other) : 0.0f;
    scale = ok ? scale : 0.0f;
    const f32x2 inv2 = pack2(inv, inv), one2 = pack2(one, one);
    const float magic = 12582912.0f + (kInt4 ? 8.0f : 128.0f);
    const f32x2 magic2 = pack2(magic, magic), minus_m2 = pack2(-12582912.0f, -12582912.0f), k256 = pack2(256.0f, 256.0f);
    auto code = [&](uint32_t w) { return add2_unfused(mul2(bf16x2_widen(w), inv2), magic2, one2); };
    const f32x2 t0 = gather2(code(a.x), code(a.y), minus_m2, k256), t1 = gather2(code(a.z), code(a.w), minus_m2, k256);
    const f32x2 t2 = gather2(code(b.x), code(b.y), minus_m2, k256), t3 = gather2(code(b.z), code(b.w), minus_m2, k256);
    if (kInt4)
        return make_uint4(__byte_perm(nibbles4_from(t0), nibbles4_from(t1), 0x5410) ^ 0x88888888u,
                          __byte_perm(nibbles4_from(t2), nibbles4_from(t3), 0x5410) ^ 0x88888888u, 0u, 0u);
    return make_uint4(codes4_from(t0), codes4_from(t1), codes4_from(t2), codes4_from(t3));
}

// One plane's share of a CTA: where its chunk memory, its scales and its pool plane are.
struct RowsPlane {
    unsigned char *pool, *chunk;
    float *scales;            // of the CTA's first group of 64; key planes of a per-channel key codec: of chunk token 0
    int kind;                 // 0 bf16, 1 int8, 2 int4, 3 / 4 the same with a scale per channel
};

template <int OP>
__device__ __forceinline__ RowsPlane rows_plane(const RowsLaunch &P, const DevOp &op, unsigned plane, unsigned i0)
{
    const unsigned kv = op.kv_sel ? (unsigned)op.kv_sel - 1u : plane & 1u, li = op.kv_sel ? plane : plane >> 1;
    RowsPlane pl;
    pl.pool = reinterpret_cast<unsigned char *>(__ldg(reinterpret_cast<const unsigned long long *>(kv ? P.v_layers : P.k_layers) + op.l0 + (int)li));
    const unsigned long long in_plane = (unsigned long long)i0 * P.row_elems;
    const unsigned long long ce = ((unsigned long long)li * 2ull + kv) * (unsigned long long)op.T * P.row_elems + in_plane;
    const bool int4 = op.codec == 2 || op.codec == 4;
    pl.kind = op.codec == 0 ? 0 : int4 ? 2 : 1;
    pl.chunk = op.data + (op.codec == 0 ? 2ull * ce : int4 ? ce >> 1 : ce);
    pl.scales = reinterpret_cast<float *>(op.scales);
    if (op.codec >= 3) {
        // per layer: key scales [ceil(T / 64)][row_elems], then value scales [T][row_elems / 64]
        const unsigned long long n_groups = ((unsigned long long)op.T + 63ull) >> 6;
        pl.scales += li * (n_groups * P.row_elems + (((unsigned long long)op.T * P.row_elems) >> 6));
        if (kv == 0u) pl.kind += 2;
        else pl.scales += n_groups * P.row_elems + (in_plane >> 6);
    } else {
        pl.scales += ce >> 6;
    }
    return pl;
}

// kVec: elements of a vector.  A slot holds 16 bytes.  In a store a vector is two slots: a lane fetches slots lane and 32 + lane of its
// warp's 64 and codes slots 2 lane and 2 lane + 1, which other lanes may have fetched.
template <int OP, int kJ, int kVec>
__device__ __forceinline__ void rows_move(const RowsLaunch &P)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    uint4 *slots = reinterpret_cast<uint4 *>(smem_raw);                                                   // [stage][j][thread]
    float *slot_scales = reinterpret_cast<float *>(slots + (size_t)kRowsStages * kJ * kRowsThreads);      // [stage][j][thread]
    unsigned long long *place = reinterpret_cast<unsigned long long *>(slot_scales + (size_t)kRowsStages * kJ * kRowsThreads);
    const uint32_t bars = smem_u32(place + kRowsPerCta);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(reinterpret_cast<unsigned char *>(place + kRowsPerCta) + 8u * kRowsStages);
    const unsigned tid = threadIdx.x;
    const unsigned long long since = global_timer_ns();
    if (tid == 0) {
        for (int s = 0; s < kRowsStages; ++s) mbar_init(bars + 8u * (uint32_t)s, kRowsThreads);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // (waiting first: a kernel behind this one starts when the one before it is known to be over)
    dependency_wait();
    release_dependents();
    const DevOp *ops = P.ops ? P.ops : P.inline_ops;
    int lo = 0, hi = P.n_ops - 1;
    while (lo < hi) {                                       // last op with tile_begin <= this CTA
        const int mid = (lo + hi + 1) >> 1;
        if (ops[mid].tile_begin <= blockIdx.x) lo = mid; else hi = mid - 1;
    }
    const DevOp &op = ops[lo];
    const unsigned n_rows = (unsigned)(op.list_mode ? op.n_list : op.T);
    const unsigned row_tiles = (n_rows + P.rows - 1u) / P.rows;
    const unsigned gl = blockIdx.x - op.tile_begin, pc = gl / row_tiles, i0 = (gl - pc * row_tiles) * P.rows;
    const unsigned nr = n_rows - i0 < P.rows ? n_rows - i0 : P.rows;
    bool bad = false;
    if (tid < nr) {
        const unsigned i = i0 + tid;
        const long long rel = op.list_mode == 1 ? (long long)__ldcg(op.list + i) : (long long)i;
        const long long p = op.off + rel;
        unsigned long long a = ~0ull;                       // byte offset of the row in a pool plane; all ones: no place
        if (rel >= 0 && p < op.pos_end) {
            const long long b = P.bs_shift >= 0 ? p >> P.bs_shift : p / P.bs;
            const long long id = __ldcg(op.table + b);
            if (id >= 0 && id < P.n_blocks) a = (unsigned long long)(id * P.bs + (p - b * P.bs)) * P.row_elems * 2ull;
        }
        place[tid] = a;
        bad = a == ~0ull;
    }
    if (__syncthreads_or(bad)) {
        // a row without a place takes the rows of its unit with it
        if (bad) atomicCAS(P.status, 0, kStatusRange);
        bool out = false;
        if (tid < nr) {
            const unsigned u0 = (i0 + tid) / P.unit * P.unit;
            for (unsigned i = u0 > i0 ? u0 - i0 : 0u; i < nr && i0 + i < u0 + P.unit; ++i) out |= place[i] == ~0ull;
        }
        __syncthreads();
        if (out) place[tid] = ~0ull;
        __syncthreads();
    }
    // the thread's vectors: tid, tid + 256, ...
    constexpr int kSlots = OP == OP_STORE ? kJ / 2 * 2 : kJ, kVecs = OP == OP_STORE ? kJ / 2 : kJ;
    unsigned long long at[kSlots];                          // byte offset in a pool plane of what a slot is for; all ones: nothing
    unsigned there = 0u;                                    // store: bit j = vector j exists
    const unsigned n_vec = nr * P.vpr;
#pragma unroll
    for (int j = 0; j < kVecs; ++j) {
        const unsigned v = tid + (unsigned)j * kRowsThreads;
        const unsigned r = P.vpr == 1u ? v : __umulhi(v, P.vpr_magic);
        if (OP == OP_STORE) {
            if (v < n_vec && place[r] != ~0ull) there |= 1u << j;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const unsigned s16 = 2u * (v & ~31u) + 32u * (unsigned)h + (v & 31u), w = s16 >> 1;       // slot, and the vector it belongs to
                const unsigned q = P.vpr == 1u ? w : __umulhi(w, P.vpr_magic);
                at[2 * j + h] = w < n_vec ? place[q] : ~0ull;
                if (at[2 * j + h] != ~0ull) at[2 * j + h] += 32ull * (w - q * P.vpr) + 16ull * (s16 & 1u);
            }
        } else {
            at[j] = v < n_vec ? place[r] : ~0ull;
            if (at[j] != ~0ull) at[j] += (2ull * kVec) * (v - r * P.vpr);
        }
    }
    const unsigned n_planes = (unsigned)op.nl * (op.kv_sel ? 1u : 2u);
    const unsigned p0 = pc * P.planes, p1 = p0 + P.planes < n_planes ? p0 + P.planes : n_planes;

    auto fetch = [&](unsigned plane, unsigned stage) {
        const RowsPlane pl = rows_plane<OP>(P, op, plane, i0);
#pragma unroll
        for (int j = 0; j < kSlots; ++j) {
            if (at[j] == ~0ull) continue;
            const unsigned v = tid + (unsigned)j * kRowsThreads;
            const uint32_t dst = smem_u32(slots + (stage * kJ + (unsigned)j) * kRowsThreads + tid);
            if (OP == OP_STORE) {
                cp_async16(smem_u32(slots + (stage * kJ + 2u * ((unsigned)j >> 1)) * kRowsThreads + 2u * (tid & ~31u) + 32u * ((unsigned)j & 1u) + (tid & 31u)),
                           pl.pool + at[j]);
            } else if (kVec == 8 && pl.kind == 0) {
                cp_async16(dst, pl.chunk + 16ull * v);
            } else {
                constexpr unsigned kBytes = kVec;           // of int8 codes
                if (pl.kind & 1) { if (kBytes == 16u) cp_async16(dst, pl.chunk + 16ull * v); else cp_async8(dst, pl.chunk + 8ull * v); }
                else { if (kBytes == 16u) cp_async8(dst, pl.chunk + 8ull * v); else cp_async4(dst, pl.chunk + 4ull * v); }
                if (pl.kind < 3) cp_async4(smem_u32(slot_scales + (stage * kJ + (unsigned)j) * kRowsThreads + tid), pl.scales + v / (64u / kVec));
            }
        }
        cp_async_arrive(bars + 8u * stage);
    };
    auto finish = [&](unsigned plane, unsigned stage) {
        const RowsPlane pl = rows_plane<OP>(P, op, plane, i0);
        const bool wide = (((unsigned long long)pl.pool | (2ull * P.row_elems)) & 31ull) == 0ull;      // 32-byte stores
#pragma unroll
        for (int j = 0; j < kVecs; ++j) {
            const unsigned v = tid + (unsigned)j * kRowsThreads;
            if (OP == OP_STORE) {
                const uint4 *block = slots + (stage * kJ + 2u * (unsigned)j) * kRowsThreads + 2u * (tid & ~31u);       // the warp's 64 slots
                const unsigned lane = tid & 31u;
                if (pl.kind == 0) {
                    uint4 *dst = reinterpret_cast<uint4 *>(pl.chunk) + 2u * (v & ~31u) + lane;
                    if (at[2 * j] != ~0ull) dst[0] = block[lane];
                    if (at[2 * j + 1] != ~0ull) dst[32] = block[32u + lane];
                } else {
                    float scale;                            // (all lanes: the group's lanes shuffle)
                    const uint4 a = block[2u * lane], b = block[2u * lane + 1u];
                    const uint4 q = pl.kind == 2 ? rows_quantise<true>(a, b, P.one, scale) : rows_quantise<false>(a, b, P.one, scale);
                    if ((there >> j) & 1u) {
                        if (pl.kind == 2) reinterpret_cast<uint2 *>(pl.chunk)[v] = make_uint2(q.x, q.y);
                        else reinterpret_cast<uint4 *>(pl.chunk)[v] = q;
                        if ((v & 3u) == 0u) pl.scales[v >> 2] = scale;
                    }
                }
                continue;
            }
            const uint4 x = slots[(stage * kJ + (unsigned)j) * kRowsThreads + tid];
            if (at[j] != ~0ull) {
                if (kVec == 8 && pl.kind == 0) {
                    *reinterpret_cast<uint4 *>(pl.pool + at[j]) = x;
                    continue;
                }
                f32x2 f[kVec / 2];
                if (pl.kind & 1) {
                    const f32x2 minus_bias = pack2(-8388736.0f, -8388736.0f);
                    const uint32_t w[4] = { x.x ^ 0x80808080u, x.y ^ 0x80808080u, x.z ^ 0x80808080u, x.w ^ 0x80808080u };
#pragma unroll
                    for (int k = 0; k < kVec / 4; ++k) { f[2 * k] = codes_to_f32x2<0>(w[k], minus_bias); f[2 * k + 1] = codes_to_f32x2<2>(w[k], minus_bias); }
                } else {
                    const f32x2 minus_bias4 = pack2(-8388616.0f, -8388616.0f);
                    nibbles_to_f32x2(x.x, minus_bias4, f);
                    if (kVec == 16) nibbles_to_f32x2(x.y, minus_bias4, f + (kVec / 2 - 4));
                }
                if (pl.kind >= 3) {
                    // a scale per channel (they start at any multiple of four bytes, and are the same for up to 64 rows: L1 has them)
                    const unsigned r = P.vpr == 1u ? v : __umulhi(v, P.vpr_magic);
                    const float *sp = pl.scales + (unsigned long long)((i0 + r) >> 6) * P.row_elems + (unsigned)kVec * (v - r * P.vpr);
#pragma unroll
                    for (int k = 0; k < kVec / 2; ++k) f[k] = mul2(f[k], pack2(sp[2 * k], sp[2 * k + 1]));
                } else {
                    const float sc = slot_scales[(stage * kJ + (unsigned)j) * kRowsThreads + tid];
                    const f32x2 sc2 = pack2(sc, sc);
#pragma unroll
                    for (int k = 0; k < kVec / 2; ++k) f[k] = mul2(f[k], sc2);
                }
                const uint4 a = make_uint4(pack_bf16x2(f[0]), pack_bf16x2(f[1]), pack_bf16x2(f[2]), pack_bf16x2(f[3]));
                unsigned char *dst = pl.pool + at[j];
                if (kVec == 16) {
                    const uint4 b = make_uint4(pack_bf16x2(f[kVec / 2 - 4]), pack_bf16x2(f[kVec / 2 - 3]), pack_bf16x2(f[kVec / 2 - 2]), pack_bf16x2(f[kVec / 2 - 1]));
                    if (wide) {
                        asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w),
                                     "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w) : "memory");
                        continue;
                    }
                    reinterpret_cast<uint4 *>(dst)[1] = b;
                }
                *reinterpret_cast<uint4 *>(dst) = a;
            }
        }
    };
    unsigned ahead = p0;
    for (int s = 0; s < kRowsStages - 1; ++s, ++ahead)
        if (ahead < p1) fetch(ahead, (unsigned)s);
    unsigned stage = 0, fill = kRowsStages - 1;
    uint32_t phase = 0;
    for (unsigned plane = p0; plane < p1; ++plane) {
        if (OP == OP_STORE) __syncwarp();                   // the stage's slots have been read by the whole warp
        if (ahead < p1) { fetch(ahead, fill); ++ahead; }
        if (++fill == (unsigned)kRowsStages) fill = 0;
        if (!rows_wait(bars + 8u * stage, phase, abort_flag, P.wait_limit_ns, since)) {
            atomicCAS(P.status, 0, kStatusTimeout);
            cp_async_wait_all();
            return;
        }
        finish(plane, stage);
        if (++stage == (unsigned)kRowsStages) { stage = 0; phase ^= 1u; }
    }
}

// kJ slots a thread, vectors of kVec elements.
template <int kJ, int kVec>
__global__ void __launch_bounds__(kRowsThreads, 4) kdn_store_rows_kernel(const __grid_constant__ RowsLaunch P) { rows_move<OP_STORE, kJ, kVec>(P); }
template <int kJ, int kVec>
__global__ void __launch_bounds__(kRowsThreads, 4) kdn_retrieve_rows_kernel(const __grid_constant__ RowsLaunch P) { rows_move<OP_RETRIEVE, kJ, kVec>(P); }

}  // namespace kdn

// attn_decode.cu -- split-K grouped-query decode attention over the paged cache,
// on the tensor cores (mma.sync m16n8k16).
//
// One new token per request attends over its whole context, so the kernel is
// bound by the stream of cached keys and values (long contexts) or by its own
// latency (short ones).  The G query heads that share a kv head are the eight
// columns of an MMA: scores S^T = K q^T with keys as rows, outputs O^T = V^T P^T
// with dims as rows.  On fp32 FMAs the same work, two multiply-adds per cached
// value and head fed from shared memory, ran at a fifth of the HBM rate.
//
// Precision.  Queries and probabilities are fp32 and enter the MMAs as three
// bf16 parts (truncations of eight bits each, all 24 in the end), keys and values
// are the cache's bf16 values; products are exact.  The first parts' products
// start from zero for every 16 summed terms and are added in fp32 (the tensor
// core's own accumulation truncates); the small parts share an accumulator.
//
// Split.  A block of four warps takes a run of pages of one (request, kv head);
// warp w takes keys 16 w .. 16 w + 15 of each page, with a ring of `stages` tiles
// of its own filled by 16-byte asynchronous copies, an online softmax of its own,
// and no barrier.  The warps' states meet in shared memory at the end.  The grid
// has at most kSlots blocks; a request with more pages than its share of them
// gives each block several.  With one block for the (request, kv head) its result
// is final; otherwise the states go to scratch, and the last block to arrive
// (completion ticket) merges them in order.  Lengths, the page table and all but
// the newest position were written before this step's first launch, so the first
// tiles are on their way before the wait for the kernel ahead.
//
// Measured (a block per page on fp32 FMAs in brackets), 70B heads: contexts 16383,
// 16000, 9001 and 12345 together 54 us, 4.1 TB/s (154); eight of 128 to 4041 30 us
// (50); error against fp64 2.1e-7 (3.5e-7).  Each block costs a fixed 4 to 5 us
// of first loads and of meeting at the end, so one wave of blocks is best: 912 or
// 1216 blocks took 58 and 65 us, eight warps a block on two pages 68 to 76.
// Short launches stay with the block per page (launch_attention).
#include <math.h>

#include "gemv.cuh"

namespace loip {
namespace {

constexpr int kAW = 4;  // warps per block: 16 keys of a page each
constexpr int kAThreads = kAW * 32;
constexpr int kPage = 64;
constexpr int kMaxParts = 256;  // blocks per (request, kv head) that the merge holds weights for
constexpr int kSlots = 456;     // blocks of a launch: one wave, three per SM
constexpr int kRing = 2;        // tiles of a warp's ring when a block takes several pages

struct AttnDecodeParams {
    const float* q;  // [B, Hq * D]
    KvView kv;
    const int32_t* ctx_lens;
    const int32_t* positions;  // used when ctx_lens is null: ctx = position + 1
    const int32_t* row_req;
    int B, Hq, Hkv, max_chunks, stages;
    float scale;
    float* scratch;  // [B][Hq][max_chunks][D + 2] partial states (output, maximum, sum)
    int* counters;   // [B][Hq]
    float* o;        // [B, Hq * D]
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
// 16-byte copy; n = 0 reads nothing and zero-fills
__device__ __forceinline__ void cp_async16z(uint32_t dst, const void* src, uint32_t n) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ uint4 lds128(uint32_t a) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "r"(a)
                 : "memory");
    return v;
}
// four 8 x 8 blocks, transposed (lane l gives a row address of block l / 8)
__device__ __forceinline__ void ldmatrix4_t(uint32_t (&r)[4], uint32_t a) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(a)
                 : "memory");
}
// transpose of an 8 x 8 block of 16-bit values held as an MMA fragment
__device__ __forceinline__ uint32_t transpose8(uint32_t v) {
    uint32_t r;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(r) : "r"(v));
    return r;
}
__device__ __forceinline__ void mma(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma0(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%10,%10,%10,%10};"
        : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}
// the three bf16 parts of two values, packed (first value in the low half)
__device__ __forceinline__ void split3(float a, float b, uint32_t& hi, uint32_t& mid, uint32_t& lo) {
    const uint32_t ua = __float_as_uint(a), ub = __float_as_uint(b);
    hi = __byte_perm(ua, ub, 0x7632);
    const float ra = a - __uint_as_float(ua & 0xffff0000u), rb = b - __uint_as_float(ub & 0xffff0000u);
    const uint32_t va = __float_as_uint(ra), vb = __float_as_uint(rb);
    mid = __byte_perm(va, vb, 0x7632);
    lo = __byte_perm(__float_as_uint(ra - __uint_as_float(va & 0xffff0000u)),
                     __float_as_uint(rb - __uint_as_float(vb & 0xffff0000u)), 0x7632);
}

// A warp's state in the merge: [head][D + 4] outputs, then maxima and sums
template <int G, int D>
struct Merge {
    static constexpr int OP = D + 4;  // pitch of a head's outputs, against bank conflicts
    static constexpr int WARP = G * OP + 2 * G;
    static constexpr int BYTES = kAW * WARP * 4;
};
template <int G, int D>
constexpr int attn_decode_smem(int stages) {
    const int ring = kAW * stages * 2 * 16 * D * 2, weights = 2 * G * kMaxParts * 4;
    return ring > weights ? (ring > Merge<G, D>::BYTES ? ring : Merge<G, D>::BYTES)
                          : (weights > Merge<G, D>::BYTES ? weights : Merge<G, D>::BYTES);
}

// This warp's state over its keys of pages [pg0, pg1) in plain fp32, for a state
// that came out NaN: an infinite key, value or query meets the zero parts of a
// split operand, where the fp32 product stays infinite (and an infinitely low
// score has weight zero).
template <int G, int D>
__device__ __noinline__ void warp_state_fp32(const AttnDecodeParams& p, int row, int kvh, int req, int ctx, int pg0,
                                             int pg1, int warp, float* state) {
    const int lane = threadIdx.x & 31;
    float* m_out = state + G * Merge<G, D>::OP;
    for (int g = 0; g < G; ++g) {
        const float* q = p.q + (size_t)row * p.Hq * D + (size_t)(kvh * G + g) * D;
        float m = -INFINITY, l = 0.f, o[D / 32];
        for (int i = 0; i < D / 32; ++i) o[i] = 0.f;
        for (int pg = pg0; pg < pg1; ++pg) {
            const uint16_t* K = reinterpret_cast<const uint16_t*>(
                                    p.kv.base + p.kv.page_offsets[(int64_t)req * p.kv.max_pages + pg] +
                                    (uint64_t)p.kv.layer * p.kv.layer_page_bytes) +
                                (size_t)kvh * kPage * D;
            const uint16_t* V = K + (size_t)p.Hkv * kPage * D;
            for (int t = warp * 16; t < warp * 16 + 16 && pg * kPage + t < ctx; ++t) {
                float s = 0.f;
                for (int i = 0; i < D / 32; ++i) s = fmaf(q[lane + 32 * i], bf2f(K[(size_t)t * D + lane + 32 * i]), s);
                for (int x = 16; x; x >>= 1) s += __shfl_xor_sync(0xffffffffu, s, x);
                s *= p.scale;
                const float mn = fmaxf(m, s), c = m == -INFINITY ? 0.f : expf(m - mn);
                const float w = s == -INFINITY && mn == -INFINITY ? 0.f : expf(s - mn);
                l = l * c + w;
                for (int i = 0; i < D / 32; ++i) o[i] = fmaf(w, bf2f(V[(size_t)t * D + lane + 32 * i]), o[i] * c);
                m = mn;
            }
        }
        for (int i = 0; i < D / 32; ++i) state[g * Merge<G, D>::OP + lane + 32 * i] = o[i];
        if (lane == 0) {
            m_out[g] = m;
            m_out[G + g] = l;
        }
    }
}

template <int G, int D>
__global__ void __launch_bounds__(kAThreads) attn_decode_kernel(const __grid_constant__ AttnDecodeParams p) {
    constexpr int CH = D / 8;  // 16-byte pieces of a key's row
    constexpr int TILE = 16 * D * 2;
    using M = Merge<G, D>;
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ int s_last;
    __shared__ float s_c[G][kAW], s_ml[G][2];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int g = lane >> 2, t4 = lane & 3;
    const int part = blockIdx.x, kvh = blockIdx.y, row = blockIdx.z;
    pdl_trigger();
    const int ctx = p.ctx_lens ? p.ctx_lens[row] : p.positions[row] + 1;
    const int npages = (ctx + kPage - 1) / kPage;
    const int ppb = (npages + gridDim.x - 1) / gridDim.x;  // pages per block
    const int nparts = ppb ? (npages + ppb - 1) / ppb : 0;
    if (part >= nparts) {
        pdl_wait();
        return;
    }
    const int req = p.row_req ? p.row_req[row] : row;
    const int pg0 = part * ppb, pg1 = min(npages, pg0 + ppb);
    const int64_t* table = p.kv.page_offsets + (int64_t)req * p.kv.max_pages;
    const char* layer = p.kv.base + (uint64_t)p.kv.layer * p.kv.layer_page_bytes + (size_t)kvh * kPage * D * 2;
    const uint32_t ring = smem_u32(smem) + (uint32_t)(warp * p.stages) * (2 * TILE);
    // Keys 16 warp .. + 15 of page pg -> ring slot; rows past the context are
    // zero-filled.  skip: a row (of the tile) left for later.  In a tile, piece c of
    // key t sits at c ^ 4 (t & 1) for K and c ^ (t & 7) for V: no bank conflicts.
    auto copy_row = [&](const char* src, uint32_t dst, int t, int c, uint32_t n) {
        cp_async16z(dst + (uint32_t)((t * CH + (c ^ ((t & 1) << 2))) * 16), src + (size_t)t * (D * 2) + c * 16, n);
        cp_async16z(dst + TILE + (uint32_t)((t * CH + (c ^ (t & 7))) * 16),
                    src + (size_t)p.Hkv * kPage * D * 2 + (size_t)t * (D * 2) + c * 16, n);
    };
    auto fetch = [&](int pg, int slot, int skip) {
        if (pg < pg1) {
            const char* src = layer + table[pg] + (size_t)warp * 16 * D * 2;
            const int nv = ctx - pg * kPage - warp * 16;
#pragma unroll
            for (int i = 0; i < 16 * CH / 32; ++i) {
                const int t = (i * 32 + lane) / CH, c = lane & (CH - 1);
                if (t != skip) copy_row(src, ring + (uint32_t)slot * (2 * TILE), t, c, t < nv ? 16u : 0u);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // the newest position's row comes from the kernel ahead of this one
    const int new_pg = (ctx - 1) / kPage, new_t = (ctx - 1) % kPage - warp * 16;
    const bool has_new = new_t >= 0 && new_t < 16;
    for (int s = 0; s < p.stages; ++s) fetch(pg0 + s, s, has_new && pg0 + s == new_pg ? new_t : -1);
    pdl_wait();
    if (has_new && new_pg >= pg0 && new_pg < min(pg1, pg0 + p.stages) && lane < CH)
        copy_row(layer + table[new_pg] + (size_t)warp * 16 * D * 2, ring + (uint32_t)(new_pg - pg0) * (2 * TILE), new_t,
                 lane, 16u);
    asm volatile("cp.async.commit_group;" ::: "memory");
    // queries as the B operand: lane (head g, t4) holds dims 32 j + 8 t4 .. + 7 (K of
    // the products is permuted so that a lane's 16-byte pieces are two MMAs' operands)
    uint32_t qh[D / 32][4], qm[D / 32][4], ql[D / 32][4];
    {
        const float* q = p.q + (size_t)row * p.Hq * D + (size_t)(kvh * G + (g < G ? g : 0)) * D + t4 * 8;
#pragma unroll
        for (int j = 0; j < D / 32; ++j) {
            float4 a = *reinterpret_cast<const float4*>(q + 32 * j), b = *reinterpret_cast<const float4*>(q + 32 * j + 4);
            if (g >= G) a = b = make_float4(0.f, 0.f, 0.f, 0.f);
            split3(a.x, a.y, qh[j][0], qm[j][0], ql[j][0]);
            split3(a.z, a.w, qh[j][1], qm[j][1], ql[j][1]);
            split3(b.x, b.y, qh[j][2], qm[j][2], ql[j][2]);
            split3(b.z, b.w, qh[j][3], qm[j][3], ql[j][3]);
        }
    }
    float o[D / 16][4];  // dims 16 i + g and + 8, heads 2 t4 and + 1
#pragma unroll
    for (int i = 0; i < D / 16; ++i) o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f;
    float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};  // heads 2 t4 and + 1 (l: this lane's keys)
    const uint32_t k_off = (uint32_t)((g * CH + (t4 ^ ((g & 1) << 2))) * 16);  // piece 4 j + t4 follows from piece t4
    const int v_key = (lane & 7) + ((lane >> 4) << 3), v_c = (lane >> 3) & 1;
    const uint32_t v_off = (uint32_t)(TILE + v_key * CH * 16);
    int slot = 0;
#pragma unroll 1
    for (int pg = pg0; pg < pg1; ++pg) {
        // the tile's group, and the newest row's behind the first `stages` groups
        if (pg + 1 < pg1 && pg0 + p.stages < pg1 && p.stages == kRing)
            asm volatile("cp.async.wait_group %0;" ::"n"(kRing - 1) : "memory");
        else
            asm volatile("cp.async.wait_all;" ::: "memory");
        __syncwarp();
        const int nv = ctx - pg * kPage - warp * 16;
        if (nv > 0) {
            const uint32_t tile = ring + (uint32_t)slot * (2 * TILE);
            float s[4] = {0.f, 0.f, 0.f, 0.f}, em[4], el[4];
#pragma unroll
            for (int j = 0; j < D / 32; ++j) {
                const uint32_t at = tile + (k_off ^ (64u * (j & 1))) + 128u * (j >> 1);
                const uint4 r0 = lds128(at), r1 = lds128(at + 8 * CH * 16);  // keys g and g + 8
                const uint32_t a0[4] = {r0.x, r1.x, r0.y, r1.y}, a1[4] = {r0.z, r1.z, r0.w, r1.w};
                float h0[4], h1[4];
                mma0(h0, a0, qh[j][0], qh[j][1]);
                mma0(h1, a1, qh[j][2], qh[j][3]);
                if (j == 0) {
                    mma0(em, a0, qm[j][0], qm[j][1]);
                    mma0(el, a0, ql[j][0], ql[j][1]);
                } else {
                    mma(em, a0, qm[j][0], qm[j][1]);
                    mma(el, a0, ql[j][0], ql[j][1]);
                }
                mma(em, a1, qm[j][2], qm[j][3]);
                mma(el, a1, ql[j][2], ql[j][3]);
#pragma unroll
                for (int i = 0; i < 4; ++i) s[i] += h0[i] + h1[i];
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                s[i] = (s[i] + (em[i] + el[i])) * p.scale;
                if (g + (i >> 1) * 8 >= nv) s[i] = -INFINITY;
            }
            float corr[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                float mx = fmaxf(s[e], s[e + 2]);
#pragma unroll
                for (int x = 4; x < 32; x <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, x));
                const float mn = fmaxf(m[e], mx);
                corr[e] = m[e] == -INFINITY ? 0.f : expf(m[e] - mn);
                m[e] = mn;
                s[e] = expf(s[e] - mn);
                s[e + 2] = expf(s[e + 2] - mn);
                l[e] = l[e] * corr[e] + (s[e] + s[e + 2]);
            }
            // probabilities as the B operand: keys along K, heads as columns
            uint32_t b[3][2];
            split3(s[0], s[1], b[0][0], b[1][0], b[2][0]);
            split3(s[2], s[3], b[0][1], b[1][1], b[2][1]);
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                b[i][0] = transpose8(b[i][0]);
                b[i][1] = transpose8(b[i][1]);
            }
#pragma unroll
            for (int i = 0; i < D / 16; ++i) {
                uint32_t a[4];
                ldmatrix4_t(a, tile + v_off + (uint32_t)(((2 * i + v_c) ^ (v_key & 7)) * 16));
                // blocks: (keys 0-7, dims 0-7), (keys 0-7, dims 8-15), (keys 8-15, ...)
                float h[4], e[4];
                mma0(e, a, b[2][0], b[2][1]);
                mma(e, a, b[1][0], b[1][1]);
                mma0(h, a, b[0][0], b[0][1]);
#pragma unroll
                for (int x = 0; x < 4; ++x) o[i][x] = fmaf(o[i][x], corr[x & 1], h[x] + e[x]);
            }
        }
        __syncwarp();  // every lane is done with the slot
        fetch(pg + p.stages, slot, -1);
        slot = slot + 1 == p.stages ? 0 : slot + 1;
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
#pragma unroll
    for (int e = 0; e < 2; ++e)
#pragma unroll
        for (int x = 4; x < 32; x <<= 1) l[e] += __shfl_xor_sync(0xffffffffu, l[e], x);
    // ---- the warps' states meet (the rings are done)
    float* state = reinterpret_cast<float*>(smem) + warp * M::WARP;
    __syncthreads();
    bool bad = false;
#pragma unroll
    for (int i = 0; i < D / 16; ++i)
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            const int head = 2 * t4 + (x & 1);
            if (head < G) {
                state[head * M::OP + 16 * i + g + (x >> 1) * 8] = o[i][x];
                bad |= o[i][x] != o[i][x];
            }
        }
#pragma unroll
    for (int e = 0; e < 2; ++e)
        if (2 * t4 + e < G) {
            bad |= l[e] != l[e];
            if (g == 0) {
                state[G * M::OP + 2 * t4 + e] = m[e];
                state[G * M::OP + G + 2 * t4 + e] = l[e];
            }
        }
    if (__any_sync(0xffffffffu, bad)) warp_state_fp32<G, D>(p, row, kvh, req, ctx, pg0, pg1, warp, state);
    __syncthreads();
    const float* st = reinterpret_cast<const float*>(smem);
    const size_t hstride = (size_t)p.max_chunks * (D + 2);
    float* base = p.scratch + ((size_t)row * p.Hq + (size_t)kvh * G) * hstride;
    float* out = p.o + (size_t)row * p.Hq * D + (size_t)kvh * G * D;
    if (tid < kAW * G) {  // the warps' weights, the maximum and the sum of each head
        const int head = tid / kAW, w = tid % kAW;
        const float mw = st[w * M::WARP + G * M::OP + head];
        const unsigned lanes = 0xfu << (lane & 28);
        float mx = fmaxf(mw, __shfl_xor_sync(lanes, mw, 1));
        mx = fmaxf(mx, __shfl_xor_sync(lanes, mx, 2));
        const float c = mw == -INFINITY ? 0.f : expf(mw - mx);  // 0: a warp without keys
        float lsum = mw == -INFINITY ? 0.f : st[w * M::WARP + G * M::OP + G + head] * c;
        lsum += __shfl_xor_sync(lanes, lsum, 1);
        lsum += __shfl_xor_sync(lanes, lsum, 2);
        s_c[head][w] = c;
        if (w == 0) {
            s_ml[head][0] = mx;
            s_ml[head][1] = lsum;
        }
    }
    __syncthreads();
#pragma unroll
    for (int i = tid; i < G * D; i += kAThreads) {
        const int head = i / D, j = i - head * D;
        float v = 0.f;
#pragma unroll
        for (int w = 0; w < kAW; ++w) v = fmaf(st[w * M::WARP + head * M::OP + j], s_c[head][w], v);
        if (nparts == 1) {
            out[i] = v / s_ml[head][1];
        } else {
            float* ps = base + head * hstride + (size_t)part * (D + 2);
            ps[j] = v;
            if (j < 2) ps[D + j] = s_ml[head][j];
        }
    }
    if (nparts == 1) return;
    // ---- the last block of this (request, kv head) merges the parts
    __threadfence();
    __syncthreads();
    if (tid == 0) {
        int* cnt = p.counters + (size_t)row * p.Hq + kvh;
        const int ticket = atomicAdd(cnt, 1);
        s_last = ticket == nparts - 1;
        if (s_last) atomicExch(cnt, 0);  // every part has arrived: reset for the next launch
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    constexpr int NOUT = (G * D + kAThreads - 1) / kAThreads, PB = 8;
    // the first parts' outputs do not depend on the weights: their loads go out
    // together with those of the maxima and sums
    float v[PB][NOUT];
    auto load_parts = [&](int c0) {
#pragma unroll
        for (int u = 0; u < PB; ++u)
#pragma unroll
            for (int k = 0; k < NOUT; ++k) {
                const int e = tid + kAThreads * k, head = e / D, j = e - head * D;
                v[u][k] = (e < G * D && c0 + u < nparts) ? __ldcg(base + head * hstride + (size_t)(c0 + u) * (D + 2) + j)
                                                         : 0.f;
            }
    };
    load_parts(0);
    float* s_w = reinterpret_cast<float*>(smem);  // [G][kMaxParts] weights
    float* s_l = s_w + G * kMaxParts;
    for (int i = tid; i < G * nparts; i += kAThreads) {
        const int head = i / nparts, c = i - head * nparts;
        const float* pc = base + head * hstride + (size_t)c * (D + 2);
        s_w[head * kMaxParts + c] = __ldcg(pc + D);
        s_l[head * kMaxParts + c] = __ldcg(pc + D + 1);
    }
    __syncthreads();
    for (int head = warp; head < G; head += kAW) {
        float* w = s_w + head * kMaxParts;
        float mx = -INFINITY, lsum = 0.f;
        for (int c = lane; c < nparts; c += 32) mx = fmaxf(mx, w[c]);
#pragma unroll
        for (int x = 16; x; x >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, x));
        for (int c = lane; c < nparts; c += 32) {
            const float e = expf(w[c] - mx);
            w[c] = e;
            lsum = fmaf(s_l[head * kMaxParts + c], e, lsum);
        }
#pragma unroll
        for (int x = 16; x; x >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, x);
        const float inv = 1.0f / lsum;
        for (int c = lane; c < nparts; c += 32) w[c] *= inv;
    }
    __syncthreads();
    float acc[NOUT];
#pragma unroll
    for (int k = 0; k < NOUT; ++k) acc[k] = 0.f;
    for (int c0 = 0; c0 < nparts; c0 += PB) {
        if (c0 > 0) load_parts(c0);
#pragma unroll
        for (int u = 0; u < PB; ++u)
#pragma unroll
            for (int k = 0; k < NOUT; ++k) {
                const int e = tid + kAThreads * k;
                if (e < G * D && c0 + u < nparts) acc[k] = fmaf(v[u][k], s_w[e / D * kMaxParts + c0 + u], acc[k]);
            }
    }
#pragma unroll
    for (int k = 0; k < NOUT; ++k)
        if (tid + kAThreads * k < G * D) out[tid + kAThreads * k] = acc[k];
}

template <int G, int D>
cudaError_t launch_t(AttnDecodeParams& p, cudaStream_t st, bool pdl) {
    // blocks per (request, kv head): a page each up to kSlots in all, at most what
    // the merge holds; a ring of kRing tiles once a block may take several pages
    int parts = kSlots / (p.Hkv * p.B);
    parts = parts < 1 ? 1 : parts > kMaxParts ? kMaxParts : parts;
    if (parts > p.max_chunks) parts = p.max_chunks;
    p.stages = parts < p.max_chunks ? kRing : 1;
    const int smem = attn_decode_smem<G, D>(p.stages);
    cudaError_t e = cudaFuncSetAttribute(attn_decode_kernel<G, D>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         attn_decode_smem<G, D>(kRing));
    if (e != cudaSuccess) return e;
    return launch_k(attn_decode_kernel<G, D>, dim3(parts, p.Hkv, p.B), dim3(kAThreads), smem, st, pdl, p);
}

}  // namespace

cudaError_t launch_attention_decode(const float* q, KvView kv, const int32_t* ctx_lens, const int32_t* positions,
                                    const int32_t* row_req, int B, int Hq, int Hkv, int d, int max_chunks,
                                    float* scratch, int* counters, float* o, cudaStream_t st, bool pdl) {
    AttnDecodeParams p{};
    p.q = q;
    p.kv = kv;
    p.ctx_lens = ctx_lens;
    p.positions = positions;
    p.row_req = row_req;
    p.B = B;
    p.Hq = Hq;
    p.Hkv = Hkv;
    p.max_chunks = max_chunks;
    p.scale = 1.0f / sqrtf((float)d);
    p.scratch = scratch;
    p.counters = counters;
    p.o = o;
    const int G = Hq / Hkv;
    if (d == 128) {
        switch (G) {
            case 1: return launch_t<1, 128>(p, st, pdl);
            case 2: return launch_t<2, 128>(p, st, pdl);
            case 4: return launch_t<4, 128>(p, st, pdl);
            case 8: return launch_t<8, 128>(p, st, pdl);
        }
    } else if (d == 64) {
        switch (G) {
            case 1: return launch_t<1, 64>(p, st, pdl);
            case 2: return launch_t<2, 64>(p, st, pdl);
            case 4: return launch_t<4, 64>(p, st, pdl);
            case 8: return launch_t<8, 64>(p, st, pdl);
        }
    }
    return cudaErrorInvalidValue;
}

}  // namespace loip

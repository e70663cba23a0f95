// attn_tc.cu -- causal prefill attention on the 5th-generation tensor cores.
//
// The prefill's attention (every prompt token against the cached keys and
// values of its request up to its own position: grouped-query attention with a
// causal mask) is a dense contraction over 128-row query tiles, so it runs as
// tcgen05 MMAs: S = Q K^T into tensor memory, the softmax on the CUDA cores,
// O_blk = P V into tensor memory, one key page (64 positions) at a time.
//
// Tile.  One CTA per (query tile, kv head).  A query tile is up to 256 / G
// consecutive positions of one request (G = Hq / Hkv query heads share the kv
// head): two halves of 128 MMA rows, row = pi * G + gi of (position, query head)
// pairs, that attend over the same key pages, read once per CTA.  Blocks are
// launched longest tile first.
//
// Roles (12 warps of 168 registers at launch; setmaxnreg makes that 224 for the
// eight softmax warps and 56 for the others, 64512 in all as before):
//   warps 0-3, 4-7  the softmax of half 0 and half 1, a thread to a row: S from
//                   tensor memory, the online softmax, P to tensor memory, each
//                   page's O_blk added to fp32 registers;
//   warps 8, 9      one lane each issues the MMAs of half 0 and half 1: S of page
//                   kb + 1 as soon as S of kb has been read (it runs under that
//                   page's softmax), P V of kb when P is in place;
//   warps 10, 11    load the key and the value pages (cp.async), two buffers each.
// The halves meet only at the shared pages.
//
// Precision.  The operands of kind::f16 are bf16; the queries (fp32) and the
// probabilities P (fp32) are each given as a split pair hi = bf16(v), lo =
// bf16(v - hi), two MMAs per K step, so the products carry ~16 significant
// bits; keys and values are the cache's bf16 values exactly.  The tensor core
// sums at most one page per MMA group (its truncating accumulation stays
// short); each page's O_blk is added to fp32 registers with the online-softmax
// rescale (round to nearest).  The output is written as the next projection's
// split operand.
//
// Shared memory (bf16, 128-byte swizzle: 16-byte chunk c of row r at r * 128 +
// ((c ^ (r & 7)) * 16), 8-row atoms of 1024 bytes):
//   Q_hi, Q_lo   [128 rows][D] per half   D/64 slabs of 16 KB each
//   K, V         [64 keys][D]             D/64 slabs of 8 KB, two buffers each
// K is the K-major B operand of S, V the MN-major B operand of P V: both lie as
// the cache has them.
// Tensor memory, per half h: S [128 x 64] fp32 at column 64 h; P_hi and P_lo
// [128 x 64] bf16 (two per column) at 128 + 64 h, the A operand of P V; O_blk
// [128 x D] fp32 at 256 + 128 h.
//
// Barriers, one completion per page (per two pages for the page buffers), each
// waited for by every party before any of them can take part in its next one:
// s_full (S computed), s_free (S read, 128 threads), p_ready (P stored and the
// last O_blk read, 128 threads), pv_full (O_blk computed) per half; k_full, v_full
// (landed, 32 threads), k_empty, v_empty (read by both halves) per buffer.
//
// Measured, one prompt of 4001 positions at the 8B heads: 263 us, against 800 for
// one half per CTA with every warp also loading pages, transposing V and waiting
// at block-wide barriers, one chain per page. The tensor pipe needs about 110 us
// of it; the rest is the softmax warps' chain (two warps to a scheduler).
//
// Every wait is bounded (2 s of %globaltimer); on timeout the CTA records an
// error code, every role leaves, copies and MMAs in flight finish, the tensor
// memory is freed and the kernel returns.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "internal.h"

namespace loip {

__device__ int g_attn_tc_error;  // first failure code of any tensor-core attention launch (0 = none)

namespace {

constexpr int kAttnThreads = 384;
constexpr int kKeys = 64;  // keys per block (one KV page)
constexpr uint32_t kTmemCols = 512, kPCol = 128, kOCol = 256;

template <int D>
struct AttnTcSmem {
    static constexpr int SLABS = D / 64;
    static constexpr int Q_SLAB = 128 * 128;  // bytes: 128 rows x 64 bf16
    static constexpr int K_SLAB = 64 * 128;
    static constexpr int QHALF = 2 * SLABS * Q_SLAB;  // Q_hi, then Q_lo, of one half
    static constexpr int QLO = SLABS * Q_SLAB;
    static constexpr int KB = 2 * QHALF;  // two K buffers
    static constexpr int KBUF = SLABS * K_SLAB;
    static constexpr int VB = KB + 2 * KBUF;  // two V buffers
    static constexpr int BAR = VB + 2 * KBUF;
    static constexpr int BYTES = BAR + 192;
    // + alignment of the dynamic window; over half of an SM's shared memory, so
    // that one CTA has the SM's tensor memory to itself
    static constexpr int ALLOC = BYTES + 1024 > 120 * 1024 ? BYTES + 1024 : 120 * 1024;
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t swz(int r, int c) { return (uint32_t)(r * 128 + ((c ^ (r & 7)) << 4)); }

__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// Waits at most 2 s, or until another thread of the CTA has given up (*abort).
__device__ __forceinline__ void mbar_wait_slow(uint32_t bar, uint32_t parity, volatile int* abort) {
    const uint64_t t0 = global_ns();
    while (!mbar_try_wait(bar, parity) && !*abort)
        if (global_ns() - t0 > 2000000000ull) {
            *abort = 1;
            atomicCAS(&g_attn_tc_error, 0, 1);
        }
}
__device__ __forceinline__ void mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort) {
    if (!mbar_try_wait(bar, parity)) mbar_wait_slow(bar, parity, abort);
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// kind::f16 instruction descriptor: fp32 accumulator, bf16 A and B, A K-major, B
// K-major or MN-major, M = 128, N = n
__host__ __device__ constexpr uint32_t idesc(int n, bool b_mn = false) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((b_mn ? 1u : 0u) << 16) | ((uint32_t)(n >> 3) << 17) |
           ((uint32_t)(128 >> 4) << 24);
}
__device__ __forceinline__ void umma(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t id, uint32_t acc) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(
            tmem_d),
        "l"(adesc), "l"(bdesc), "r"(id), "r"(acc)
        : "memory");
}
// the A operand in tensor memory (rows = lanes, two bf16 per column)
__device__ __forceinline__ void umma_ta(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t id, uint32_t acc) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(
            tmem_d),
        "r"(tmem_a), "l"(bdesc), "r"(id), "r"(acc)
        : "memory");
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// Shared-memory matrix descriptor, 128-byte rows with the 128-byte swizzle in
// 8-row atoms 1024 bytes apart.  K-major: rows are M or N, a row holds 64 of K
// (`lead` unused).  MN-major: rows are K, a row holds 64 of N, the next 64 of N
// `lead` bytes further on.
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr, uint32_t lead = 16) {
    uint64_t d = (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)(lead >> 4) << 16;
    d |= (uint64_t)(1024 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float* v) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%"
        "19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\ntcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, "
        "[%16];\ntcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&r)[8]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr), "r"(r[0]),
                 "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
                 : "memory");
}
__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// two fp32 -> their bf16 roundings (hi) and the bf16 roundings of what is left
// (lo), packed with the first value in the low half
__device__ __forceinline__ void split2(float a, float b, uint32_t& hi, uint32_t& lo) {
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(hi) : "f"(b), "f"(a));
    const float ra = a - __uint_as_float(hi << 16), rb = b - __uint_as_float(hi & 0xffff0000u);
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(lo) : "f"(rb), "f"(ra));
}
// 16-byte copy; with n = 0 nothing is read and the destination is zero-filled
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, uint32_t n) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}

struct AttnTcParams {
    const float* q;      // [M, Hq * D] fp32
    KvView kv;
    const int4* tiles;   // {row0, n_rows, request, pos0}
    int Hq, Hkv, M, n_tiles;
    float scale_log2;    // log2(e) / sqrt(d): scores in base 2
    uint16_t* o;         // split pair [2][M][Hq * D]
};

template <int G, int D>
__global__ void __launch_bounds__(kAttnThreads, 1) attn_tc_kernel(const __grid_constant__ AttnTcParams p) {
    using S = AttnTcSmem<D>;
    constexpr int PT = 128 / G;  // positions per half
    extern __shared__ uint8_t smem_raw[];
    __shared__ int s_abort;
    uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    volatile int* abort = &s_abort;
    const uint32_t sbase = smem_u32(sm), bar = sbase + S::BAR;
    // pairs of barriers: per half, then per page buffer
    const uint32_t s_full = bar, s_free = bar + 16, p_ready = bar + 32, pv_full = bar + 48, k_full = bar + 64,
                   v_full = bar + 80, k_empty = bar + 96, v_empty = bar + 112, end_bar = bar + 128, q_full = bar + 144;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(sm + S::BAR + 152);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int4 tile = p.tiles[p.n_tiles - 1 - (int)(blockIdx.x / p.Hkv)];
    const int g = blockIdx.x % p.Hkv;  // kv head
    const int req = tile.z, pos0 = tile.w, last_pos = pos0 + tile.y - 1;
    const int qd = p.Hq * D;
    // pages of the tile and of each half
    const int nkb = last_pos / kKeys + 1;
    const int pages0 = (pos0 + min(PT, tile.y) - 1) / kKeys + 1, pages1 = tile.y > PT ? nkb : 0;

    if (tid == 0) {
        auto init = [](uint32_t at, uint32_t count) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(at), "r"(count) : "memory");
        };
        for (int i = 0; i < 2; ++i) {
            init(s_full + 8 * i, 1);
            init(s_free + 8 * i, 128);
            init(p_ready + 8 * i, 128);
            init(pv_full + 8 * i, 1);
            init(k_full + 8 * i, 32);
            init(v_full + 8 * i, 32);
            init(k_empty + 8 * i, 2);
            init(v_empty + 8 * i, 2);
            init(end_bar + 8 * i, 1);
        }
        init(q_full, 256);
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;

    if (warp >= 8) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
        if (warp >= 10) {
            // ---- loaders: warp 10 the keys, warp 11 the values.  Positions past the
            // tile's last one hold no key yet (the page may keep anything there): their
            // K and V are zero-filled, so that their zero weights in P meet finite
            // values (0 x NaN would spoil the row).  A page is under way while the one
            // before it is used; it has about a page's time to land.
            const bool is_v = warp == 11;
            const char* src0 = p.kv.base + (uint64_t)p.kv.layer * p.kv.layer_page_bytes +
                               (size_t)((is_v ? p.Hkv : 0) + g) * kKeys * D * 2;
            const uint32_t buf0 = sbase + (is_v ? S::VB : S::KB), full = is_v ? v_full : k_full,
                           empty = is_v ? v_empty : k_empty;
            constexpr int CH = D / 8;  // 16-byte chunks of a key's row
            const int c = lane & (CH - 1), key0 = lane / CH;
            for (int kb = 0; kb < nkb && !*abort; ++kb) {
                const uint32_t b = kb & 1;
                const char* src = src0 + p.kv.page_offsets[(int64_t)req * p.kv.max_pages + kb];
                const int n_keys = last_pos - kb * kKeys + 1;  // valid keys in this page (>= 1)
                const uint32_t dst = buf0 + b * S::KBUF + (uint32_t)((c >> 3) * S::K_SLAB);
                if (kb >= 2) mbar_wait(empty + 8 * b, (uint32_t)((kb >> 1) - 1) & 1u, abort);
                __syncwarp();
#pragma unroll 8
                for (int key = key0; key < kKeys; key += 32 / CH)
                    cp_async16(dst + swz(key, c & 7), src + (size_t)key * (D * 2) + c * 16, key < n_keys ? 16u : 0u);
                asm volatile("cp.async.wait_all;" ::: "memory");
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // generic-proxy writes -> the tensor core
                mbar_arrive(full + 8 * b);
            }
        } else if (lane == 0) {
            // ---- MMAs of half h
            const int h = warp - 8, n = h ? pages1 : pages0;
            const uint32_t t_s = tmem + 64u * h, t_p = tmem + kPCol + 64u * h, t_o = tmem + kOCol + 128u * h;
            auto page_parity = [](int kb) { return (uint32_t)(kb >> 1) & 1u; };
            // S = (Q_hi + Q_lo) K^T of page kb; a half without that page only passes its keys on
            auto s_step = [&](int kb) {
                const uint32_t b = kb & 1;
                mbar_wait(k_full + 8 * b, page_parity(kb), abort);
                if (kb >= n) {
                    mbar_arrive(k_empty + 8 * b);
                    return;
                }
                if (kb > 0) mbar_wait(s_free + 8 * h, (kb - 1) & 1, abort);
                if (*abort) return;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t qb = sbase + h * S::QHALF, kbuf = sbase + S::KB + b * S::KBUF;
#pragma unroll
                for (int k = 0; k < D / 16; ++k) {
                    const uint32_t qo = qb + (uint32_t)((k >> 2) * S::Q_SLAB);
                    const uint64_t bd = sdesc(kbuf + (uint32_t)((k >> 2) * S::K_SLAB)) + 2 * (k & 3);
                    umma(t_s, sdesc(qo) + 2 * (k & 3), bd, idesc(kKeys), k != 0);
                    umma(t_s, sdesc(qo + S::QLO) + 2 * (k & 3), bd, idesc(kKeys), 1u);
                }
                umma_commit(s_full + 8 * h);
                umma_commit(k_empty + 8 * b);
            };
            // O_blk = (P_hi + P_lo) V of page kb
            auto pv_step = [&](int kb) {
                const uint32_t b = kb & 1;
                mbar_wait(v_full + 8 * b, page_parity(kb), abort);
                if (kb >= n) {
                    mbar_arrive(v_empty + 8 * b);
                    return;
                }
                mbar_wait(p_ready + 8 * h, kb & 1, abort);
                if (*abort) return;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint64_t vd = sdesc(sbase + S::VB + b * S::KBUF, S::K_SLAB);
#pragma unroll
                for (int k = 0; k < kKeys / 16; ++k) {  // 16 keys: two atoms
                    umma_ta(t_o, t_p + 8 * k, vd + (2048 >> 4) * k, idesc(D, true), k != 0);
                    umma_ta(t_o, t_p + 32 + 8 * k, vd + (2048 >> 4) * k, idesc(D, true), 1u);
                }
                umma_commit(pv_full + 8 * h);
                umma_commit(v_empty + 8 * b);
            };
            mbar_wait(q_full, 0, abort);
            s_step(0);
            for (int kb = 0; kb < nkb && !*abort; ++kb) {
                if (kb + 1 < nkb) s_step(kb + 1);
                pv_step(kb);
            }
            if (*abort) {  // what was issued completes before the tensor memory is released
                int never = 0;
                umma_commit(end_bar + 8 * h);
                mbar_wait(end_bar + 8 * h, 0, &never);
            }
        }
        __syncwarp();
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 224;");
        // ---- softmax.  My row: position pi of the tile, query head gi of the kv head
        const int h = warp >> 2, r = (warp & 3) * 32 + lane;
        const int pi = h * PT + r / G, gi = r % G;
        const bool live = pi < tile.y;
        const int my_pos = pos0 + (live ? pi : 0), n = h ? pages1 : pages0;
        const int full_pos = pos0 + h * PT;  // pages that end at or before it need no mask in my half
        {  // Q rows -> split pair, swizzled
            const float* qr = p.q + (size_t)(tile.x + (live ? pi : 0)) * qd + (size_t)(g * G + gi) * D;
            uint8_t* qs = sm + h * S::QHALF;
#pragma unroll 4
            for (int c8 = 0; c8 < D / 8; ++c8) {  // 8 elements = one 16-byte chunk
                float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
                if (live) {
                    a = *reinterpret_cast<const float4*>(qr + 8 * c8);
                    b = *reinterpret_cast<const float4*>(qr + 8 * c8 + 4);
                }
                uint4 hi, lo;
                split2(a.x, a.y, hi.x, lo.x);
                split2(a.z, a.w, hi.y, lo.y);
                split2(b.x, b.y, hi.z, lo.z);
                split2(b.z, b.w, hi.w, lo.w);
                const uint32_t off = (uint32_t)((c8 >> 3) * S::Q_SLAB) + swz(r, c8 & 7);
                *reinterpret_cast<uint4*>(qs + off) = hi;
                *reinterpret_cast<uint4*>(qs + S::QLO + off) = lo;
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            mbar_arrive(q_full);
        }
        const uint32_t t_row = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        const uint32_t t_s = t_row + 64u * h, t_p = t_row + kPCol + 64u * h, t_o = t_row + kOCol + 128u * h;
        float o[D];
#pragma unroll
        for (int j = 0; j < D; ++j) o[j] = 0.f;
        float m_run = -INFINITY, l_run = 0.f, alpha = 0.f;  // row maximum (base 2) and sum; rescale of the last page
        // O = O * alpha + O_blk of page kb (in fp32 registers); false after an abort,
        // when products may still be running
        auto add_o = [&](int kb) {
            mbar_wait(pv_full + 8 * h, kb & 1, abort);
            if (__any_sync(0xffffffffu, *abort)) return false;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
            for (int j0 = 0; j0 < D; j0 += 16) {
                float v[16];
                tmem_ld16(t_o + j0, v);
#pragma unroll
                for (int j = 0; j < 16; ++j) o[j0 + j] = fmaf(o[j0 + j], alpha, v[j]);
            }
            return true;
        };
        bool ok = true;
#pragma unroll 1
        for (int kb = 0; kb < n; ++kb) {
            mbar_wait(s_full + 8 * h, kb & 1, abort);
            ok = !__any_sync(0xffffffffu, *abort);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            float s[kKeys];
            tmem_ld32(t_s, s);
            tmem_ld32(t_s + 32, s + 32);
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            mbar_arrive(s_free + 8 * h);
            if (kb * kKeys + kKeys - 1 > full_pos) {
#pragma unroll
                for (int j = 0; j < kKeys; ++j) s[j] = kb * kKeys + j <= my_pos ? s[j] : -INFINITY;
            }
            float mq[4] = {s[0], s[1], s[2], s[3]};
#pragma unroll
            for (int j = 4; j < kKeys; ++j) mq[j & 3] = fmaxf(mq[j & 3], s[j]);
            const float mx = fmaxf(fmaxf(mq[0], mq[1]), fmaxf(mq[2], mq[3]));
            // a row has its key 0 in page 0, so m_new is finite from the first page on
            const float m_new = fmaxf(m_run, mx * p.scale_log2);
            const float next_alpha = ex2(m_run - m_new);
            float lsum[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int j = 0; j < kKeys; ++j) {
                s[j] = ex2(fmaf(s[j], p.scale_log2, -m_new));
                lsum[j & 3] += s[j];
            }
            m_run = m_new;
            l_run = fmaf(l_run, next_alpha, (lsum[0] + lsum[1]) + (lsum[2] + lsum[3]));
            // the previous page's output; then P's place is free
            if (kb > 0) {
                ok = add_o(kb - 1);
                if (!ok) break;
            }
            alpha = next_alpha;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                uint32_t hi[8], lo[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) split2(s[16 * q + 2 * j], s[16 * q + 2 * j + 1], hi[j], lo[j]);
                tmem_st8(t_p + 8 * q, hi);
                tmem_st8(t_p + 32 + 8 * q, lo);
            }
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            mbar_arrive(p_ready + 8 * h);
        }
        if (n > 0 && ok) ok = add_o(n - 1);
        if (live && ok) {
            const float inv = 1.0f / l_run;
            const size_t plane = (size_t)p.M * qd;
            uint16_t* orow = p.o + (size_t)(tile.x + pi) * qd + (size_t)(g * G + gi) * D;
#pragma unroll
            for (int j = 0; j < D; j += 8) {
                uint4 hi, lo;
                split2(o[j] * inv, o[j + 1] * inv, hi.x, lo.x);
                split2(o[j + 2] * inv, o[j + 3] * inv, hi.y, lo.y);
                split2(o[j + 4] * inv, o[j + 5] * inv, hi.z, lo.z);
                split2(o[j + 6] * inv, o[j + 7] * inv, hi.w, lo.w);
                *reinterpret_cast<uint4*>(orow + j) = hi;
                *reinterpret_cast<uint4*>(orow + plane + j) = lo;
            }
        }
        __syncwarp();
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
    }
}

template <int G, int D>
cudaError_t launch_t(const AttnTcParams& p, cudaStream_t st) {
    constexpr int SMEM = AttnTcSmem<D>::ALLOC;
    cudaError_t e = cudaFuncSetAttribute(attn_tc_kernel<G, D>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM);
    if (e != cudaSuccess) return e;
    attn_tc_kernel<G, D><<<p.n_tiles * p.Hkv, kAttnThreads, SMEM, st>>>(p);
    return cudaGetLastError();
}

}  // namespace

// Both halves of a tile share its pages, which halves the loads and overlaps the
// halves' chains; but a pass whose tiles of one half fit the chip at once (152
// CTAs) is as long as its longest chain, and that is shorter with one half.
int attention_tc_tile_positions(int rows, int Hq, int Hkv) {
    if (Hkv < 1 || Hq < Hkv) return 0;
    const int half = 128 / (Hq / Hkv);
    return (int64_t)((rows + half - 1) / half) * Hkv <= 152 ? half : 2 * half;
}

cudaError_t launch_attention_tc(const float* q, KvView kv, const int4* tiles, int n_tiles, int M, int Hq, int Hkv,
                                int d, uint16_t* o, cudaStream_t st) {
    if (n_tiles <= 0) return cudaSuccess;
    if (kv.page_tokens != kKeys || Hkv < 1 || Hq % Hkv) return cudaErrorInvalidValue;
    AttnTcParams p{};
    p.q = q;
    p.kv = kv;
    p.tiles = tiles;
    p.Hq = Hq;
    p.Hkv = Hkv;
    p.M = M;
    p.n_tiles = n_tiles;
    p.scale_log2 = 1.4426950408889634f / sqrtf((float)d);
    p.o = o;
    const int G = Hq / Hkv;
    if (d == 128) {
        switch (G) {
            case 1: return launch_t<1, 128>(p, st);
            case 2: return launch_t<2, 128>(p, st);
            case 4: return launch_t<4, 128>(p, st);
            case 8: return launch_t<8, 128>(p, st);
        }
    } else if (d == 64) {
        switch (G) {
            case 1: return launch_t<1, 64>(p, st);
            case 2: return launch_t<2, 64>(p, st);
            case 4: return launch_t<4, 64>(p, st);
            case 8: return launch_t<8, 64>(p, st);
        }
    }
    return cudaErrorInvalidValue;
}

cudaError_t attention_tc_error(int* code) { return cudaMemcpyFromSymbol(code, g_attn_tc_error, sizeof(int)); }

}  // namespace loip

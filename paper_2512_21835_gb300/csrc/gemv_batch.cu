// gemv_batch.cu -- the decode projections on a ring of bulk copies: for batches of
// 2 to 8 rows on the tensor cores (mma.sync m16n8k16), for batch 1 with fp32 FMAs
// (further down).
//
// The product is bound by the weight stream, so the kernel is a deep ring of
// bulk copies with just enough arithmetic behind it.  Eight fp32 activation
// rows per weight are too much for the CUDA cores (70B gate/up at batch 8 ran
// at 0.29 of the copy peak), while one m16n8k16 MMA takes a 16 x 16 weight tile
// against all eight rows.
//
// Precision.  The MMA takes bf16 operands; the weights are bf16, and an fp32
// activation is cut into three bf16 parts that together hold all of its 24
// significant bits: x = hi + mid + lo, each part the next eight bits (by
// truncation, so every difference is exact).  All products are exact in fp32.
// The tensor core's own accumulation truncates, so a hi product sums 16 columns
// from zero and everything else is added in fp32; the small lo and mid parts
// share one accumulator.  Relative error against fp64, random data (in brackets
// the fp32 FMA kernel this one replaced): 6.9e-8 (8.1e-8) at K = 256, 1.0e-7
// (2.1e-7) at K = 4096, 1.7e-7 (5.4e-7) at K = 28672.
//
// Split.  One block per SM owns a contiguous range of output units (rows; RoPE
// pairs; gate/up pairs), cut evenly to a single unit, since what counts is the
// bytes per SM.  K goes in chunks of 512.  A producer warp fills a ring of 16 KB
// stages, one tile (16 rows x 512 columns) each, up to kStages tiles ahead,
// across chunk and pass ends, starting before the wait for the previous kernel.
// A tile is two 3-D TMA boxes of 8 rows x 8 blocks of 64 columns: large boxes
// matter, a TMA operation costs its issuing thread about 100 ns whatever its
// size (1 KB boxes stream 1.7 TB/s, 8 KB boxes 6.5 TB/s).  Sixteen warps
// consume: a warp takes half the 16-byte pieces of one 64-column block of every
// tile, so each activation is read, normalised and split by exactly one lane of
// the block and stays in its registers for all tiles of the chunk -- K is
// permuted so that the eight consecutive elements a lane reads are its operand
// of two MMAs -- and the activations need no shared stage.  Blocks with more
// than T tiles take several passes over K.  At the end of a pass the 16 warps'
// partial sums meet in shared memory and are added in warp order (the result
// does not depend on scheduling), and the fused epilogue runs on them.
//
// Measured, batch 8, back-to-back launches (before, with fp32 FMAs from shared
// memory, in brackets): 70B gate/up 144 us, 6.5 TB/s (487), down 82 (478), O 31
// (154), QKV 38 (146), LM head 348 (570 at batch 4).  Batch 2 takes the same time.
// Tried: cp.async by the consuming warps in 64- or 128-byte row pieces or whole
// kilobyte rows (5.0-5.4 TB/s: two to four times the instructions), 1 KB bulk
// copies (3.3 TB/s, the issue cost above).
#include <cuda.h>
#include <cudaTypedefs.h>
#include <math.h>

#include "gemv.cuh"

namespace loip {

__device__ int g_gemv_error;  // first failure code of any launch (0 = none)

namespace {

constexpr int kBW = 16;                  // consumer warps per block
constexpr int kBThreads = kBW * 32 + 32;  // and the producer warp
constexpr int kBChunk = 32 * kBW;        // columns per chunk
constexpr int kTileFloats = 16 * 8;      // one tile's outputs: 16 rows x 8 batch rows
// A stage: two groups of 8 rows, each [8 blocks of 64 columns][8 rows][128 bytes]
// with the 128-byte swizzle (16-byte piece c of row r sits at c ^ r)
constexpr uint32_t kGroupBytes = 8192, kStageBytes = 2 * kGroupBytes;
constexpr int kStages = 11;
constexpr int kRound = 4;  // tiles whose partial sums meet at a time
constexpr int kBatchSmem = 1024 + kStages * (int)kStageBytes + kRound * kBW * kTileFloats * 4;

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
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
// Waits at most 2 s of %globaltimer, or until another warp of the block has
// given up (*abort).
__device__ __noinline__ void mbar_wait_slow(uint32_t bar, uint32_t parity, volatile int* abort) {
    uint64_t t0, t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    while (!mbar_try_wait(bar, parity) && !*abort) {
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        if (t - t0 > 2000000000ull) {
            *abort = 1;
            atomicCAS(&g_gemv_error, 0, 1);
        }
    }
}
__device__ __forceinline__ void mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort) {
    if (!mbar_try_wait(bar, parity)) mbar_wait_slow(bar, parity, abort);
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int x, int y, int z, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(
            dst),
        "l"((uint64_t)map), "r"(x), "r"(y), "r"(z), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_bf16_zero(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%10,%10,%10,%10};"
        : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}
__device__ __forceinline__ uint4 lds128(uint32_t a) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "r"(a)
                 : "memory");
    return v;
}

// A tile's 16 rows are 16 outputs, or 8 pairs with the first elements in rows
// 0..7 and the second ones in rows 8..15 (a lane's accumulator then holds both
// elements of its pair).
template <int EPI>
struct TileUnits {
    static constexpr bool PAIRS = EPI == EPI_QKV || EPI == EPI_SWIGLU;
    static constexpr int U = PAIRS ? 8 : 16;
};

// First weight row of unit u, and the distance (elements) from it to the row
// half a tile further down: the pair's second row, or the row 8 units on.
template <int EPI>
__device__ __forceinline__ int unit_row0(const GemvParams& p, int u) {
    return EPI == EPI_QKV ? u + (u & ~((p.d >> 1) - 1)) : u;  // d/2 is a power of two: head * d + i
}
template <int EPI>
__device__ __forceinline__ int64_t half_step(const GemvParams& p) {
    if (EPI == EPI_QKV) return (int64_t)(p.d >> 1) * p.K;
    if (EPI == EPI_SWIGLU) return p.w1 - p.w0;
    return (int64_t)8 * p.K;
}

// The same output in plain fp32, for a sum that came out NaN: an infinite
// weight or activation meets the zero or undefined parts of a split, where the
// fp32 product may be infinite instead.  (A NaN operand ends it at once.)
__device__ __noinline__ float dot_fp32(const float* x, const uint16_t* g, const uint16_t* w, int K) {
    float a = 0.f;
    for (int k = 0; k < K && a == a; ++k) a = fmaf(bf2f(w[k]), g ? x[k] * bf2f(g[k]) : x[k], a);
    return a;
}

// TMA: the weights come by tensor map (device memory, K % 64 == 0); otherwise the
// producer warp copies them 16 bytes at a time into the same layout.
template <int EPI, int T, bool TMA>
__global__ void __launch_bounds__(kBThreads, 1)
    gemv_batch_kernel(const __grid_constant__ CUtensorMap tm0, const __grid_constant__ CUtensorMap tm1,
                      const __grid_constant__ GemvParams p) {
    constexpr int UPT = TileUnits<EPI>::U;
    constexpr bool PAIRS = TileUnits<EPI>::PAIRS;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    __shared__ uint64_t s_full[kStages], s_empty[kStages];
    __shared__ float s_ss[kBW][8];
    __shared__ uint64_t s_key[kBW][8];
    __shared__ int s_abort;
    float* red = reinterpret_cast<float*>(smem + kStages * kStageBytes);
    volatile int* abort = &s_abort;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int K = p.K;
    const uint32_t ring = smem_u32(smem), full0 = smem_u32(s_full), empty0 = smem_u32(s_empty);

    const int u_begin = (int)((int64_t)p.n_units * blockIdx.x / gridDim.x);
    const int u_end = (int)((int64_t)p.n_units * (blockIdx.x + 1) / gridDim.x);
    // first unit of the first tile: a QKV tile's eight rows must not cross a head
    const int u_first = EPI == EPI_QKV ? u_begin & ~7 : u_begin;
    const int n_tiles = (u_end - u_first + UPT - 1) / UPT;
    const int n_pass = (n_tiles + T - 1) / T;
    const int tpp = n_pass ? (n_tiles + n_pass - 1) / n_pass : 0;  // tiles per pass
    const int n_chunks = (K + kBChunk - 1) / kBChunk;
    const int64_t step = half_step<EPI>(p);

    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(full0 + 8 * s, TMA ? 1 : 32);
            mbar_init(empty0 + 8 * s, kBW);
        }
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (!TMA && K % kBChunk)  // the columns past K meet zero activations: nothing undefined may sit there
        for (uint32_t i = tid; i < kStages * kStageBytes / 16; i += kBThreads)
            reinterpret_cast<uint4*>(smem)[i] = make_uint4(0, 0, 0, 0);
    __syncthreads();

    if (warp == kBW) {  // ---- producer: tiles in the order (pass, chunk, tile)
        int s = 0, n = 0;    // stage, tiles copied
        uint32_t phase = 1;  // the first wait for each stage passes at once
        if (!TMA || lane == 0)
            for (int first = 0; first < n_tiles; first += tpp) {
                const int nt = min(tpp, n_tiles - first);
                for (int c = 0; c < n_chunks; ++c)
                    for (int t = 0; t < nt; ++t, ++n) {
                        mbar_wait(empty0 + 8 * s, phase, abort);
                        if (*abort) goto done;
                        const int u0 = u_first + (first + t) * UPT;
                        const uint32_t bar = full0 + 8 * s, dst = ring + (uint32_t)s * kStageBytes;
                        if (TMA) {
                            const int row = unit_row0<EPI>(p, u0);
                            const bool two = PAIRS || u0 + 8 < u_end;
                            mbar_expect_tx(bar, two ? kStageBytes : kGroupBytes);
                            tma_load_3d(dst, &tm0, 0, row, c * (kBChunk / 64), bar);
                            if (two)
                                tma_load_3d(dst + kGroupBytes, EPI == EPI_SWIGLU ? &tm1 : &tm0, 0,
                                            EPI == EPI_SWIGLU ? row : EPI == EPI_QKV ? row + (p.d >> 1) : row + 8,
                                            c * (kBChunk / 64), bar);
                        } else {
                            const int pieces = min(kBChunk, K - c * kBChunk) / 8;
                            for (int i = 0; i < 16; ++i) {
                                const int u = u0 + (PAIRS ? i & 7 : i);
                                if (u >= u_end) continue;
                                const uint16_t* src = p.w0 + (int64_t)unit_row0<EPI>(p, u) * K +
                                                      (PAIRS && i >= 8 ? step : 0) + c * kBChunk;
                                const uint32_t d = dst + (i >> 3) * kGroupBytes + (i & 7) * 128;
                                for (int j = lane; j < pieces; j += 32)
                                    cp_async16(d + (j >> 3) * 1024 + (((j ^ i) & 7) << 4), src + 8 * j);
                            }
                            asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
                        }
                        if (++s == kStages) {
                            s = 0;
                            phase ^= 1;
                        }
                    }
            }
        pdl_trigger();
    done:
        if (*abort) {  // given up: the copies in flight land before the block's shared memory is released
            if (!TMA) asm volatile("cp.async.wait_all;" ::: "memory");
            int never = 0;
            if (!TMA || lane == 0)
                for (int k = max(0, n - kStages); k < n; ++k)
                    mbar_wait(full0 + 8 * (k % kStages), (k / kStages) & 1, &never);
        }
        return;
    }

    // ---- consumers
    const int g = lane >> 2, t4 = lane & 3;
    const bool norm = p.g != nullptr;
    const int piece = 2 * t4 + (warp & 1);             // of the warp's block of 64 columns
    const int kw = (warp >> 1) * 64 + piece * 8;       // this lane's eight columns inside a chunk
    pdl_wait();

    // activations: this lane's eight columns of batch row g
    float4 xa, xb;
    uint4 gv;
    const float* xrow = p.in + (size_t)(g < p.B ? g : 0) * K;
    auto load_x = [&](int c) {
        const int k = c * kBChunk + kw;
        xa = xb = make_float4(0.f, 0.f, 0.f, 0.f);
        gv = make_uint4(0, 0, 0, 0);
        if (g < p.B && k < K) {
            xa = *reinterpret_cast<const float4*>(xrow + k);
            xb = *reinterpret_cast<const float4*>(xrow + k + 4);
            if (norm) gv = *reinterpret_cast<const uint4*>(p.g + k);
        }
    };
    auto sync_consumers = [&]() { asm volatile("bar.sync 1, %0;" ::"n"(kBW * 32) : "memory"); };
    float ss = 0.f, inv = 1.f;
    uint64_t best = 0;
    int s = 0;
    uint32_t phase = 0;
    const uint32_t lane_off = (uint32_t)((warp >> 1) * 1024 + g * 128 + ((piece ^ g) << 4));
    const int b = tid & 7;  // batch row of this thread's outputs

    // one output pair of a tile: the 16 partial sums in warp order, then the
    // epilogue (round slot t, row group rg)
    auto outputs = [&](int t, int rg, int tile) {
        const float* r = red + t * kBW * kTileFloats + rg * 8 + b;
        float v[2] = {0.f, 0.f};
#pragma unroll
        for (int w = 0; w < kBW; ++w) {
            v[0] += r[w * kTileFloats];
            v[1] += r[w * kTileFloats + 64];
        }
        const int u = u_first + tile * UPT + rg;
        if (EPI == EPI_QKV && u < u_begin) return;  // the previous block's
#pragma unroll
        for (int half = 0; half < 2; ++half)
            if (v[half] != v[half] && (PAIRS ? u : u + 8 * half) < u_end)
                v[half] = dot_fp32(p.in + (size_t)b * K, p.g,
                                   p.w0 + (int64_t)unit_row0<EPI>(p, u) * K + half * step, K);
        if (EPI == EPI_QKV) {
            if (u >= u_end) return;
            const int hd = p.d >> 1, h = u / hd, j = u - h * hd;
            float v0 = v[0] * inv, v1 = v[1] * inv;
            const int pos = p.positions[b];
            if (p.qk_raw && h < p.Hq + p.Hkv) {  // normalised and rotated by qk_norm_rope_kernel
                float* raw = p.qk_raw + (size_t)b * (p.Hq + 2 * p.Hkv) * p.d + (size_t)h * p.d;
                raw[j] = v0;
                raw[j + hd] = v1;
                return;
            }
            if (h < p.Hq + p.Hkv) {
                float cf, sf;
                rope_cos_sin(pos, p.rope.inv_freq[j], &cf, &sf);
                const float r0 = v0 * cf - v1 * sf, r1 = v1 * cf + v0 * sf;
                v0 = r0;
                v1 = r1;
            }
            if (h < p.Hq) {
                float* q = p.out + (size_t)b * p.Hq * p.d + (size_t)h * p.d;
                q[j] = v0;
                q[j + hd] = v1;
            } else {
                const int req = p.row_req ? p.row_req[b] : b;
                const bool is_v = h >= p.Hq + p.Hkv;
                const int kh = h - p.Hq - (is_v ? p.Hkv : 0);
                uint16_t* row =
                    reinterpret_cast<uint16_t*>(kv_row(p.kv, req, pos, is_v ? 1 : 0, kh, p.Hkv, p.d));
                row[j] = f2bf(v0);
                row[j + hd] = f2bf(v1);
            }
        } else if (EPI == EPI_SWIGLU) {
            if (u >= u_end) return;
            const float gt = v[0] * inv, ut = v[1] * inv;
            p.out[(size_t)b * p.N + u] = gt / (1.0f + expf(-gt)) * ut;
        } else {
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                const int row = u + 8 * half;
                if (row >= u_end) continue;
                float* o = p.out ? p.out + (size_t)b * p.N + row : nullptr;
                if (EPI == EPI_RESID) {
                    *o += v[half];
                } else {
                    const float lg = v[half] * inv;
                    if (o) *o = lg;
                    const uint64_t key = argmax_key(lg, (uint32_t)row);
                    best = key > best ? key : best;
                }
            }
        }
    };

    load_x(0);
    for (int first = 0; first < n_tiles; first += tpp) {
        const int nt = min(tpp, n_tiles - first);
        float acc[T][4];
#pragma unroll
        for (int t = 0; t < T; ++t) acc[t][0] = acc[t][1] = acc[t][2] = acc[t][3] = 0.f;
#pragma unroll 1
        for (int c = 0; c < n_chunks; ++c) {
            // split into three bf16 parts, packed as the MMA's B operand: words
            // 0 and 1 are the first MMA's k pairs, 2 and 3 the second's
            uint32_t hi[4], mid[4], lo[4];
            {
                float x[8] = {xa.x, xa.y, xa.z, xa.w, xb.x, xb.y, xb.z, xb.w};
                if (norm) {
                    const float gf[8] = {bf_lo(gv.x), bf_hi(gv.x), bf_lo(gv.y), bf_hi(gv.y),
                                         bf_lo(gv.z), bf_hi(gv.z), bf_lo(gv.w), bf_hi(gv.w)};
                    if (first == 0)
#pragma unroll
                        for (int e = 0; e < 8; ++e) ss = fmaf(x[e], x[e], ss);
#pragma unroll
                    for (int e = 0; e < 8; ++e) x[e] *= gf[e];
                }
#pragma unroll
                for (int e = 0; e < 8; e += 2) {
                    const uint32_t u0 = __float_as_uint(x[e]), u1 = __float_as_uint(x[e + 1]);
                    hi[e / 2] = __byte_perm(u0, u1, 0x7632);
                    const float r0 = x[e] - __uint_as_float(u0 & 0xffff0000u);
                    const float r1 = x[e + 1] - __uint_as_float(u1 & 0xffff0000u);
                    const uint32_t v0 = __float_as_uint(r0), v1 = __float_as_uint(r1);
                    mid[e / 2] = __byte_perm(v0, v1, 0x7632);
                    const uint32_t w0 = __float_as_uint(r0 - __uint_as_float(v0 & 0xffff0000u));
                    const uint32_t w1 = __float_as_uint(r1 - __uint_as_float(v1 & 0xffff0000u));
                    lo[e / 2] = __byte_perm(w0, w1, 0x7632);
                }
            }
            load_x(c + 1 < n_chunks ? c + 1 : 0);  // the next chunk's, or the next pass's first
#pragma unroll
            for (int t = 0; t < T; ++t) {
                if (t >= nt) break;
                mbar_wait(full0 + 8 * s, phase, abort);
                __syncwarp();
                const uint32_t src = ring + (uint32_t)s * kStageBytes + lane_off;
                const uint4 r0 = lds128(src), r1 = lds128(src + kGroupBytes);  // rows g and g + 8
                const uint32_t a0[4] = {r0.x, r1.x, r0.y, r1.y}, a1[4] = {r0.z, r1.z, r0.w, r1.w};
                float e[4], h0[4], h1[4];
                mma_bf16_zero(e, a0, lo[0], lo[1]);
                // every lane has read the stage: the MMA above is warp-wide and uses the data
                if (lane == 0) mbar_arrive(empty0 + 8 * s);
                mma_bf16(e, a1, lo[2], lo[3]);
                mma_bf16(e, a0, mid[0], mid[1]);
                mma_bf16(e, a1, mid[2], mid[3]);
                mma_bf16_zero(h0, a0, hi[0], hi[1]);
                mma_bf16_zero(h1, a1, hi[2], hi[3]);
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[t][i] += h0[i] + (h1[i] + e[i]);
                if (++s == kStages) {
                    s = 0;
                    phase ^= 1;
                }
            }
        }
        if (first == 0) {
            float q = ss + __shfl_xor_sync(0xffffffffu, ss, 1);
            q += __shfl_xor_sync(0xffffffffu, q, 2);
            if (t4 == 0) s_ss[warp][g] = q;
        }
        // ---- the warps' partial sums meet, kRound tiles at a time
#pragma unroll
        for (int r0 = 0; r0 < T; r0 += kRound) {
            if (r0 >= nt) break;
#pragma unroll
            for (int t = r0; t < r0 + kRound && t < T; ++t) {
                float* r = red + ((t - r0) * kBW + warp) * kTileFloats + g * 8 + 2 * t4;
                *reinterpret_cast<float2*>(r) = make_float2(acc[t][0], acc[t][1]);
                *reinterpret_cast<float2*>(r + 64) = make_float2(acc[t][2], acc[t][3]);
            }
            sync_consumers();
            if (first == 0 && r0 == 0 && norm) {
                float q = 0.f;
                for (int w = 0; w < kBW; ++w) q += s_ss[w][b];
                inv = 1.0f / sqrtf(q / (float)K + p.eps);
            }
            const int n = min(kRound, nt - r0);
            if (b < p.B && !*abort)
                for (int i = tid; i < n * 64; i += kBW * 32) outputs(i >> 6, (i >> 3) & 7, first + r0 + (i >> 6));
            sync_consumers();  // the partial sums are rewritten by the next round
        }
    }
    if (EPI == EPI_LOGITS) {
        // a thread holds the best of batch row tid & 7
#pragma unroll
        for (int o = 8; o < 32; o <<= 1) {
            const uint64_t k = __shfl_xor_sync(0xffffffffu, best, o);
            best = k > best ? k : best;
        }
        if (lane < 8) s_key[warp][lane] = best;
        sync_consumers();
        if (tid < 8) {
            uint64_t k = 0;
            for (int w = 0; w < kBW; ++w) k = s_key[w][tid] > k ? s_key[w][tid] : k;
            p.keys[(size_t)blockIdx.x * 8 + tid] = k;
        }
        // final hidden z = RMSNorm(x) * g, written once
        if (blockIdx.x == 0 && p.z) {
            for (int i = tid; i < 8 * K; i += kBW * 32) {
                const int k = i >> 3;  // batch row i & 7 = b
                if (b < p.B) p.z[(size_t)b * K + k] = p.in[(size_t)b * K + k] * inv * bf2f(p.g[k]);
            }
        }
    }
}

// ----------------------------------------------------------------------------
// Batch 1: the same ring and tiles, fp32 FMAs.  Eight consumer warps take one
// 64-column block of a chunk each; a lane holds one 16-byte piece of it for four
// rows of every tile, and the eight activations that meet it stay in registers
// for all tiles of the chunk.  Eight products are summed from zero and then added
// to the row's sum, so a chain of additions is K / 512 + 8 long.
//
// A step runs these kernels back to back, each bound by the weight stream, so
// what is left to gain lies between them: the wait for the previous kernel, the
// first activation loads and the last sums take about 2 us per launch, in which
// nothing streams if the ring is already full.  So the next kernel is triggered
// when a block has issued its last copy, and the ring takes most of the shared
// memory: a block of the next launch then starts where one has ended, and fills
// its ring during the gap.  8B step of 32 layers: 2967 -> 2780 us, 70B layer 254 ->
// 239 (before: loads to registers, by blocks of eight rows for QKV, O and down and by
// persistent warps for gate/up).  In one sweep: 2806 us; triggered at the start 2845;
// with 6 stages, so that two launches share an SM and the ring fills long before the
// gap, 3114 and 3470; with 16 more tiles copied ahead into L2 2804.
// ----------------------------------------------------------------------------
constexpr int kRW = 8;                   // consumer warps per block
constexpr int kRThreads = kRW * 32 + 32;  // and the producer warp
constexpr int kRT = 8;                   // tiles per pass
constexpr int kRingSmem = 1024 + kStages * (int)kStageBytes;

template <int EPI>
__global__ void __launch_bounds__(kRThreads, 1)
    gemv_ring_kernel(const __grid_constant__ CUtensorMap tm0, const __grid_constant__ CUtensorMap tm1,
                     const __grid_constant__ GemvParams p) {
    constexpr int UPT = TileUnits<EPI>::U;
    constexpr bool PAIRS = TileUnits<EPI>::PAIRS;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    __shared__ uint64_t s_full[kStages], s_empty[kStages];
    __shared__ float s_red[kRW][kRT * 16];
    __shared__ float s_ss[kRW];
    __shared__ int s_abort;
    volatile int* abort = &s_abort;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int K = p.K;
    const uint32_t ring = smem_u32(smem), full0 = smem_u32(s_full), empty0 = smem_u32(s_empty);
    const int all = (p.n_units + UPT - 1) / UPT;
    const int tile0 = (int)((int64_t)all * blockIdx.x / gridDim.x);
    const int n_tiles = (int)((int64_t)all * (blockIdx.x + 1) / gridDim.x) - tile0;
    const int n_pass = (n_tiles + kRT - 1) / kRT;
    const int tpp = (n_tiles + n_pass - 1) / n_pass;  // tiles per pass
    const int n_chunks = (K + kBChunk - 1) / kBChunk;

    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(full0 + 8 * s, 1);
            mbar_init(empty0 + 8 * s, kRW);
        }
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();

    if (warp == kRW) {  // ---- producer: tiles in the order (pass, chunk, tile)
        if (lane != 0) return;
        int s = 0, n = 0;
        uint32_t phase = 1;  // the first wait for each stage passes at once
        for (int first = 0; first < n_tiles; first += tpp) {
            const int nt = min(tpp, n_tiles - first);
            for (int c = 0; c < n_chunks; ++c)
                for (int t = 0; t < nt; ++t, ++n) {
                    mbar_wait(empty0 + 8 * s, phase, abort);
                    if (*abort) goto done;
                    const int u0 = (tile0 + first + t) * UPT;
                    const int row = unit_row0<EPI>(p, u0);
                    const bool two = PAIRS || u0 + 8 < p.n_units;
                    const uint32_t bar = full0 + 8 * s, dst = ring + (uint32_t)s * kStageBytes;
                    mbar_expect_tx(bar, two ? kStageBytes : kGroupBytes);
                    tma_load_3d(dst, &tm0, 0, row, c * (kBChunk / 64), bar);
                    if (two)
                        tma_load_3d(dst + kGroupBytes, EPI == EPI_SWIGLU ? &tm1 : &tm0, 0,
                                    EPI == EPI_SWIGLU ? row : EPI == EPI_QKV ? row + (p.d >> 1) : row + 8,
                                    c * (kBChunk / 64), bar);
                    if (++s == kStages) {
                        s = 0;
                        phase ^= 1;
                    }
                }
        }
        pdl_trigger();
    done:
        if (*abort) {  // given up: the copies in flight land before the block's shared memory is released
            int never = 0;
            for (int k = max(0, n - kStages); k < n; ++k)
                mbar_wait(full0 + 8 * (k % kStages), (k / kStages) & 1, &never);
        }
        return;
    }

    // ---- consumers: a lane holds eight columns (16-byte piece `piece` of the
    // warp's 64) and takes rows r, r + 4, r + 8, r + 12 of every tile
    const int piece = lane & 7, r = lane >> 3;
    const bool norm = p.g != nullptr;
    const int kw = warp * 64 + piece * 8;
    uint32_t off[2];
    off[0] = (uint32_t)(warp * 1024 + r * 128 + ((piece ^ r) << 4));
    off[1] = (uint32_t)(warp * 1024 + (r + 4) * 128 + ((piece ^ (r + 4)) << 4));
    pdl_wait();

    float4 xa, xb;
    uint4 gv;
    auto load_x = [&](int c) {
        const int k = c * kBChunk + kw;
        xa = xb = make_float4(0.f, 0.f, 0.f, 0.f);
        gv = make_uint4(0, 0, 0, 0);
        if (k < K) {
            xa = *reinterpret_cast<const float4*>(p.in + k);
            xb = *reinterpret_cast<const float4*>(p.in + k + 4);
            if (norm) gv = *reinterpret_cast<const uint4*>(p.g + k);
        }
    };
    auto sync_consumers = [&]() { asm volatile("bar.sync 1, %0;" ::"n"(kRW * 32) : "memory"); };
    float ss = 0.f, inv = 1.f;
    int s = 0;
    uint32_t phase = 0;
    load_x(0);
    for (int first = 0; first < n_tiles; first += tpp) {
        const int nt = min(tpp, n_tiles - first);
        // what the epilogue needs from memory, early
        const int n_out = nt * UPT, u = (tile0 + first) * UPT + tid;
        const bool mine = tid < n_out && u < p.n_units;
        float ea = 0.f, eb = 0.f;
        int pos = 0, head = 0, j = 0;
        if (EPI == EPI_RESID && mine) ea = p.out[u];
        if (EPI == EPI_QKV && mine) {
            pos = p.positions[0];
            head = u / (p.d >> 1);
            j = u - head * (p.d >> 1);
            if (!p.qk_raw && head < p.Hq + p.Hkv) rope_cos_sin(pos, p.rope.inv_freq[j], &ea, &eb);
        }
        float acc[kRT][4];
#pragma unroll
        for (int t = 0; t < kRT; ++t) acc[t][0] = acc[t][1] = acc[t][2] = acc[t][3] = 0.f;
#pragma unroll 1
        for (int c = 0; c < n_chunks; ++c) {
            float x[8] = {xa.x, xa.y, xa.z, xa.w, xb.x, xb.y, xb.z, xb.w};
            if (norm) {
                const float gf[8] = {bf_lo(gv.x), bf_hi(gv.x), bf_lo(gv.y), bf_hi(gv.y),
                                     bf_lo(gv.z), bf_hi(gv.z), bf_lo(gv.w), bf_hi(gv.w)};
                if (first == 0)
#pragma unroll
                    for (int e = 0; e < 8; ++e) ss = fmaf(x[e], x[e], ss);
#pragma unroll
                for (int e = 0; e < 8; ++e) x[e] *= gf[e];
            }
            load_x(c + 1 < n_chunks ? c + 1 : 0);  // the next chunk's, or the next pass's first
#pragma unroll
            for (int t = 0; t < kRT; ++t) {
                if (t >= nt) break;
                mbar_wait(full0 + 8 * s, phase, abort);
                const uint32_t src = ring + (uint32_t)s * kStageBytes;
                uint4 w[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) w[i] = lds128(src + (i >> 1) * kGroupBytes + off[i & 1]);
                __syncwarp();
                if (lane == 0) mbar_arrive(empty0 + 8 * s);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    float a = bf_lo(w[i].x) * x[0];
                    a = fmaf(bf_hi(w[i].x), x[1], a);
                    a = fmaf(bf_lo(w[i].y), x[2], a);
                    a = fmaf(bf_hi(w[i].y), x[3], a);
                    a = fmaf(bf_lo(w[i].z), x[4], a);
                    a = fmaf(bf_hi(w[i].z), x[5], a);
                    a = fmaf(bf_lo(w[i].w), x[6], a);
                    a = fmaf(bf_hi(w[i].w), x[7], a);
                    acc[t][i] += a;
                }
                if (++s == kStages) {
                    s = 0;
                    phase ^= 1;
                }
            }
        }
        // the eight lanes of a row, then the warps in order
#pragma unroll
        for (int t = 0; t < kRT; ++t) {
            if (t >= nt) break;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                float v = acc[t][i];
#pragma unroll
                for (int o = 4; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                if (piece == 0) s_red[warp][t * 16 + r + 4 * i] = v;
            }
        }
        if (first == 0 && norm) {
            float q = ss;
#pragma unroll
            for (int o = 4; o; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
            if (lane == 0) s_ss[warp] = q;
        }
        sync_consumers();
        if (first == 0 && norm) {
            float q = 0.f;
            for (int w = 0; w < kRW; ++w) q += s_ss[w];
            inv = 1.0f / sqrtf(q / (float)K + p.eps);
        }
        if (mine && !*abort) {
            const int slot = PAIRS ? (tid >> 3) * 16 + (tid & 7) : tid;
            float v0 = 0.f, v1 = 0.f;
#pragma unroll
            for (int w = 0; w < kRW; ++w) {
                v0 += s_red[w][slot];
                if (PAIRS) v1 += s_red[w][slot + 8];
            }
            v0 *= inv;
            v1 *= inv;
            if (EPI == EPI_RESID) {
                p.out[u] = ea + v0;
            } else if (EPI == EPI_SWIGLU) {
                p.out[u] = v0 / (1.0f + expf(-v0)) * v1;
            } else {
                const int hd = p.d >> 1;
                if (p.qk_raw && head < p.Hq + p.Hkv) {  // normalised and rotated by qk_norm_rope_kernel
                    p.qk_raw[(size_t)head * p.d + j] = v0;
                    p.qk_raw[(size_t)head * p.d + j + hd] = v1;
                } else {
                    if (head < p.Hq + p.Hkv) {
                        const float r0 = v0 * ea - v1 * eb, r1 = v1 * ea + v0 * eb;
                        v0 = r0;
                        v1 = r1;
                    }
                    if (head < p.Hq) {
                        p.out[(size_t)head * p.d + j] = v0;
                        p.out[(size_t)head * p.d + j + hd] = v1;
                    } else {
                        const int req = p.row_req ? p.row_req[0] : 0;
                        const bool is_v = head >= p.Hq + p.Hkv;
                        const int kh = head - p.Hq - (is_v ? p.Hkv : 0);
                        uint16_t* row =
                            reinterpret_cast<uint16_t*>(kv_row(p.kv, req, pos, is_v ? 1 : 0, kh, p.Hkv, p.d));
                        row[j] = f2bf(v0);
                        row[j + hd] = f2bf(v1);
                    }
                }
            }
        }
        if (first + tpp < n_tiles) sync_consumers();  // the partial sums are rewritten by the next pass
    }
}

PFN_cuTensorMapEncodeTiled_v12000 encoder() {
    static const PFN_cuTensorMapEncodeTiled_v12000 fn = [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            f = nullptr;
        return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(f);
    }();
    return fn;
}

// A row-major [rows, K] bf16 matrix as {64 columns, rows, K / 64}; box: 8 rows of
// 8 column blocks.
cudaError_t make_map(CUtensorMap* m, const uint16_t* w, uint64_t rows, uint64_t K) {
    const auto encode = encoder();
    if (!encode) return cudaErrorNotSupported;
    cuuint64_t dims[3] = {64, rows, K / 64}, strides[2] = {K * 2, 128};
    cuuint32_t box[3] = {64, 8, kBChunk / 64}, es[3] = {1, 1, 1};
    const CUresult r = encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<uint16_t*>(w), dims, strides, box, es,
                              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

template <int EPI, int T, bool TMA>
cudaError_t launch_batch_t(const CUtensorMap& m0, const CUtensorMap& m1, const GemvParams& p, int blocks,
                           cudaStream_t st, bool pdl) {
    cudaError_t e =
        cudaFuncSetAttribute(gemv_batch_kernel<EPI, T, TMA>, cudaFuncAttributeMaxDynamicSharedMemorySize, kBatchSmem);
    if (e != cudaSuccess) return e;
    return launch_k(gemv_batch_kernel<EPI, T, TMA>, dim3(blocks), dim3(kBThreads), kBatchSmem, st, pdl, m0, m1, p);
}

template <int EPI>
cudaError_t launch_batch(const GemvParams& p, cudaStream_t st, bool pdl, int* nblocks_out) {
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    constexpr int UPT = TileUnits<EPI>::U;
    const int tiles = (p.n_units + UPT - 1) / UPT;
    const int blocks = tiles < sms ? tiles : sms;
    if (nblocks_out) *nblocks_out = blocks;
    CUtensorMap m0{}, m1{};
    const bool tma = !p.w_host && p.K % 64 == 0;
    if (tma) {
        const uint64_t rows = EPI == EPI_QKV ? 2ull * p.n_units : (uint64_t)p.n_units;
        e = make_map(&m0, p.w0, rows, p.K);
        if (e == cudaSuccess && EPI == EPI_SWIGLU) e = make_map(&m1, p.w1, rows, p.K);
        if (e != cudaSuccess) return e;
    }
    // at most four tiles a block: the variant with fewer accumulators
    const bool few = ((p.n_units + blocks - 1) / blocks + UPT - 1) / UPT + (EPI == EPI_QKV) <= 4;
    if (tma)
        return few ? launch_batch_t<EPI, 4, true>(m0, m1, p, blocks, st, pdl)
                   : launch_batch_t<EPI, 8, true>(m0, m1, p, blocks, st, pdl);
    return few ? launch_batch_t<EPI, 4, false>(m0, m1, p, blocks, st, pdl)
               : launch_batch_t<EPI, 8, false>(m0, m1, p, blocks, st, pdl);
}

template <int EPI>
cudaError_t launch_ring(const GemvParams& p, cudaStream_t st, bool pdl) {
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    constexpr int UPT = TileUnits<EPI>::U;
    const int tiles = (p.n_units + UPT - 1) / UPT, per = (tiles + sms - 1) / sms;
    const int blocks = (tiles + per - 1) / per;
    const uint64_t rows = EPI == EPI_QKV ? 2ull * p.n_units : (uint64_t)p.n_units;
    CUtensorMap m0{}, m1{};
    e = make_map(&m0, p.w0, rows, p.K);
    if (e == cudaSuccess && EPI == EPI_SWIGLU) e = make_map(&m1, p.w1, rows, p.K);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(gemv_ring_kernel<EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, kRingSmem);
    if (e != cudaSuccess) return e;
    return launch_k(gemv_ring_kernel<EPI>, dim3(blocks), dim3(kRThreads), kRingSmem, st, pdl, m0, m1, p);
}

}  // namespace

cudaError_t launch_gemv_ring(int epi, const GemvParams& p, cudaStream_t st, bool pdl) {
    switch (epi) {
        case EPI_QKV: return launch_ring<EPI_QKV>(p, st, pdl);
        case EPI_RESID: return launch_ring<EPI_RESID>(p, st, pdl);
        case EPI_SWIGLU: return launch_ring<EPI_SWIGLU>(p, st, pdl);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_gemv_batch(int epi, const GemvParams& p, cudaStream_t st, bool pdl, int* nblocks_out) {
    switch (epi) {
        case EPI_QKV: return launch_batch<EPI_QKV>(p, st, pdl, nblocks_out);
        case EPI_RESID: return launch_batch<EPI_RESID>(p, st, pdl, nblocks_out);
        case EPI_SWIGLU: return launch_batch<EPI_SWIGLU>(p, st, pdl, nblocks_out);
        default: return launch_batch<EPI_LOGITS>(p, st, pdl, nblocks_out);
    }
}

cudaError_t gemv_batch_error(int* code) { return cudaMemcpyFromSymbol(code, g_gemv_error, sizeof(int)); }
cudaError_t gemv_batch_error_word(const int** dev) {
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_gemv_error);
    *dev = static_cast<const int*>(p);
    return e;
}

}  // namespace loip

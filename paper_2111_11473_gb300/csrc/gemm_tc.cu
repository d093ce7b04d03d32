// Tensor-core (tcgen05) matrix product for the mixed-precision path.
//
// C = alpha * A B + beta * C with float32 operands and output.  Each operand
// is split into bf16 hi/lo parts (x = hi + lo to 2^-17 relative) by a pack
// pass that also makes it K-major.  The product kernel runs
// hi*hi + hi*lo + lo*hi (or hi*hi only) as tcgen05.mma kind::f16 with a
// float32 accumulator in tensor memory:
//   - TMA (cp.async.bulk.tensor, 128-byte swizzle) stages 128 x 64 tiles of
//     one operand and bn x 64 tiles of the other through a shared-memory ring
//     on mbarriers and fills what lies outside the operands with zeros;
//   - one elected lane of a converged warp issues the MMAs and commits each
//     stage back to the producer; a final commit releases the epilogue;
//   - eight warps read the 128 x bn accumulator with tcgen05.ld and write C.
// Every mbarrier wait is bounded: on expiry the kernel raises an error flag
// that the host turns into THC_ERR_TIMEOUT, and frees its tensor memory.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cmath>
#include <mutex>

#include "common.cuh"
#include "gemm_tc.cuh"

namespace thc {
namespace {

constexpr int BM = 128;          // UMMA M (rows of the accumulator)
constexpr int BK = 64;           // K per stage: one 128-byte swizzle atom of bf16
constexpr int UK = 16;           // K per tcgen05.mma for 16-bit inputs
constexpr long long kWaitCycles = 4000000000LL;   // about 2 s at 2 GHz

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(count));
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(bar)),
                 "r"(bytes));
}

// Parity wait bounded by a clock64 budget; returns false if it expired.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
    const uint32_t a = smem_u32(bar);
    const long long t0 = clock64();
    for (;;) {
        uint32_t done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
            " selp.b32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(a), "r"(parity));
        if (done) return true;
        if (clock64() - t0 > kWaitCycles) return false;
    }
}

__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, uint64_t* bar,
                                            int c0, int c1, int c2) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4}], [%5];\n" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(smem_u32(bar))
        : "memory");
}

// tcgen05 shared-memory matrix descriptor: K-major, 128-byte swizzle, rows of
// 128 bytes, 8-row groups 1024 bytes apart.
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)1 << 16;                 // leading byte offset (unused for this layout)
    d |= (uint64_t)(1024 >> 4) << 32;       // stride byte offset
    d |= (uint64_t)1 << 46;                 // descriptor version for tcgen05
    d |= (uint64_t)2 << 61;                 // 128-byte swizzle
    return d;
}

// Instruction descriptor of kind::f16: bf16 A and B, float32 D, both K-major.
__host__ __device__ constexpr uint32_t instr_desc(int m, int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) |
           ((uint32_t)(m >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc,
                                         uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate));
}

__device__ __forceinline__ void mma_commit(uint64_t* bar) {
    asm volatile(
        "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
            smem_u32(bar))
        : "memory");
}

// One lane of a converged warp.
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile(
        "{\n .reg .pred q;\n elect.sync _|q, 0xffffffff;\n selp.b32 %0, 1, 0, q;\n}\n"
        : "=r"(p));
    return p != 0;
}

// Tile: 128 rows x bn columns, bn a multiple of 16 up to 256 chosen per
// product.  What bounds a product is either the write of C (short K) or the
// operand tiles' way from L2 to shared memory (a 128 x 128 tile takes 64 KB
// per 64-wide K step for 384 cycles of MMAs, a 128 x 256 tile 96 KB for 768),
// hence the widest tile that the columns fill, two accumulators of up to 256
// columns so that the epilogue of one tile overlaps the main loop of the next,
// and eight epilogue warps (four took 5.5 us per 128 x 128 tile, which made
// the products of K = 40 take 347 us where C is written in 57).
constexpr int kMaxBN = 256;
constexpr int kMaxStages = 8;
constexpr int kEpiWarps = 8;
constexpr int kTcThreads = 64 + 32 * kEpiWarps;   // producer, MMA issuer, epilogue
constexpr int kEpiCols = 16;                      // columns staged at once
constexpr int kRingBytes = 208 * 1024;            // ring space within the 227 KB of an SM

// Control block, after the operand ring in shared memory.
struct TcCtl {
    uint64_t full[kMaxStages];
    uint64_t empty[kMaxStages];
    uint64_t acc_full[2];     // accumulator buffer b holds a finished tile
    uint64_t acc_empty[2];    // the epilogue has drained accumulator buffer b
    uint64_t drain;
    uint32_t tmem;
    int fail;
    float epi[kEpiWarps][32 * (kEpiCols + 1)];   // per epilogue warp: 32 rows, padded
};

struct TcArgs {
    int M, N;              // real accumulator rows (UMMA M side, all batches of a
                           // collapsed product) and columns
    int Mb;                // rows per batch: row i is row i % Mb of batch bo + i / Mb
    int bn;                // tile columns
    int stages;            // ring depth
    int nbo;               // output batches
    int Ktot;              // packed K per output batch
    int ksteps;            // 64-wide K steps per output batch
    int splits;
    int mblocks, nblocks;
    long long ntiles;      // mblocks * nblocks * nbo * splits
    float* C;              // output (or partials when splits > 1)
    long long crs, ccs, cbs;   // C(i, j) of batch b at C[b*cbs + i*crs + j*ccs]
    long long split_stride;    // partials of one split
    float alpha, beta;     // alpha 1 when splits > 1
    int nprod;
    int vec;               // C rows take 32-byte stores
    int a_bcast, b_bcast;  // operand shared by every batch: packed once, batch coord 0
    int* err;
};

struct TileCoord {
    int m0, n0, bo, split, k_lo, nk;
};

__device__ __forceinline__ TileCoord tile_coord(const TcArgs& a, long long t) {
    TileCoord c;
    const int splits = a.splits, ksteps = a.ksteps;
    const int nbk = (int)(t % a.nblocks);
    long long r = t / a.nblocks;
    const int mbk = (int)(r % a.mblocks);
    r /= a.mblocks;
    c.bo = (int)(r / splits);
    c.split = (int)(r % splits);
    c.m0 = mbk * BM;
    c.n0 = nbk * a.bn;
    const int chunk = (ksteps + splits - 1) / splits;
    c.k_lo = c.split * chunk;
    c.nk = max(0, min(ksteps, c.k_lo + chunk) - c.k_lo);
    return c;
}

// One test of a phase, without waiting (true: completed).
__device__ __forceinline__ bool mbar_test(uint64_t* bar, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.b32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return done != 0;
}

// Bounded wait that also gives up once another role has failed.
__device__ __forceinline__ bool mbar_wait_or_fail(uint64_t* bar, uint32_t parity,
                                                  volatile int* fail) {
    if (mbar_test(bar, parity)) return true;
    const uint32_t a = smem_u32(bar);
    const long long t0 = clock64();
    for (;;) {
        uint32_t done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
            " selp.b32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(a), "r"(parity));
        if (done) return true;
        if (*fail) return false;
        if (clock64() - t0 > kWaitCycles) {
            atomicExch((int*)fail, 1);
            return false;
        }
    }
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(bar)) : "memory");
}

// Eight floats of a row: one 32-byte access (a full sector) per lane.
__device__ __forceinline__ void st8(float* p, const float* v) {
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};\n" ::"l"(p), "f"(v[0]),
                 "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
                 : "memory");
}
__device__ __forceinline__ void ld8(const float* p, float* v) {
    asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]),
                   "=f"(v[6]), "=f"(v[7])
                 : "l"(p)
                 : "memory");
}

// Persistent warp-specialised product: warp 0 streams operand tiles with TMA,
// warp 1 issues the MMAs into one of two tensor-memory accumulators, and
// warps 2-9 drain the other accumulator to C, so that the epilogue of one
// tile overlaps the main loop of the next.  Tiles are taken round-robin.
template <bool RMW>
__global__ void __launch_bounds__(kTcThreads, 1)
    k_gemm_tc(const __grid_constant__ CUtensorMap ta_hi, const __grid_constant__ CUtensorMap ta_lo,
              const __grid_constant__ CUtensorMap tb_hi, const __grid_constant__ CUtensorMap tb_lo,
              const TcArgs args) {
    grid_wait();
    extern __shared__ __align__(1024) unsigned char tc_raw[];
    // 1024-byte alignment of the tile ring (required by the 128-byte swizzle)
    unsigned char* ring = reinterpret_cast<unsigned char*>(
        (reinterpret_cast<uintptr_t>(tc_raw) + 1023) & ~uintptr_t(1023));
    const bool three = args.nprod == 3;
    const uint32_t a_bytes = BM * BK * 2, b_bytes = (uint32_t)args.bn * BK * 2;
    const uint32_t stage_bytes = (three ? 2 : 1) * (a_bytes + b_bytes);
    const int ST = args.stages;
    // stage: [A hi | B hi | A lo | B lo]
    TcCtl& sm = *reinterpret_cast<TcCtl*>(ring + (size_t)ST * stage_bytes);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr uint32_t kCols = 2 * kMaxBN;
    volatile int* fail = &sm.fail;

    if (threadIdx.x == 0) {
        for (int s = 0; s < ST; ++s) {
            mbar_init(&sm.full[s], 1);
            mbar_init(&sm.empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&sm.acc_full[b], 1);
            mbar_init(&sm.acc_empty[b], kEpiWarps);
        }
        mbar_init(&sm.drain, 1);
        sm.fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                         smem_u32(&sm.tmem)),
                     "r"(kCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
    }
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = sm.tmem;

    if (warp == 0) {
        if (lane == 0) {
            // TMA producer
            int s = 0, issued = 0;
            uint32_t par = 0;           // parity of the pass over the ring
            bool wrapped = false, ok = true;
            for (long long t = blockIdx.x; t < args.ntiles && ok && !*fail; t += gridDim.x) {
                const TileCoord c = tile_coord(args, t);
                const int ba = args.a_bcast ? 0 : c.bo, bb = args.b_bcast ? 0 : c.bo;
                for (int i = 0; i < c.nk; ++i) {
                    if (wrapped && !mbar_wait_or_fail(&sm.empty[s], par ^ 1u, fail)) {
                        ok = false;
                        break;
                    }
                    const int kc = (c.k_lo + i) * BK;
                    unsigned char* st = ring + (size_t)s * stage_bytes;
                    mbar_expect_tx(&sm.full[s], stage_bytes);
                    tma_load_3d(st, &ta_hi, &sm.full[s], kc, c.m0, ba);
                    tma_load_3d(st + a_bytes, &tb_hi, &sm.full[s], kc, c.n0, bb);
                    if (three) {
                        tma_load_3d(st + a_bytes + b_bytes, &ta_lo, &sm.full[s], kc, c.m0, ba);
                        tma_load_3d(st + 2 * a_bytes + b_bytes, &tb_lo, &sm.full[s], kc, c.n0, bb);
                    }
                    issued = max(issued, s + 1);
                    if (++s == ST) {
                        s = 0;
                        par ^= 1u;
                        wrapped = true;
                    }
                }
            }
            // Every load this thread issued has landed before the CTA exits
            // (immediate unless a wait above gave up): stages below s were
            // last filled in this pass over the ring, the others in the one before.
            for (int e = 0; e < issued; ++e) mbar_wait(&sm.full[e], e < s ? par : par ^ 1u);
        }
    } else if (warp == 1) {
        // MMA issuer: the whole warp runs the loop and one elected lane
        // issues, so that the descriptors stay in uniform registers.
        const uint32_t idesc = instr_desc(BM, args.bn);
        const uint64_t base = smem_desc(smem_u32(ring));
        const uint64_t dstage = stage_bytes >> 4, dbh = a_bytes >> 4,
                       dal = (a_bytes + b_bytes) >> 4, dbl = (2 * a_bytes + b_bytes) >> 4;
        constexpr uint64_t dk = (uint64_t)(UK * 2) >> 4;   // along K inside the swizzle atom
        auto wait_all = [&](uint64_t* bar, uint32_t parity) {
            return __all_sync(0xffffffffu, mbar_wait_or_fail(bar, parity, fail)) != 0;
        };
        int s = 0, tl = 0;
        uint32_t par = 0;
        bool ok = true;
        for (long long t = blockIdx.x; t < args.ntiles && ok; t += gridDim.x, ++tl) {
            const TileCoord c = tile_coord(args, t);
            const int buf = tl & 1;
            if (tl >= 2 && !wait_all(&sm.acc_empty[buf], (uint32_t)(((tl >> 1) - 1) & 1))) break;
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            const uint32_t dst = tmem + (uint32_t)(buf * kMaxBN);
            for (int i = 0; i < c.nk; ++i) {
                if (!wait_all(&sm.full[s], par)) {
                    ok = false;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                const uint64_t d0 = base + (uint64_t)s * dstage;
                // 16-wide steps that hold data (Ktot is a multiple of 16)
                const int kks = min(BK / UK, (args.Ktot - (c.k_lo + i) * BK) / UK);
                if (elect_one()) {
#pragma unroll
                    for (int kk = 0; kk < BK / UK; ++kk) {
                        if (kk < kks) {
                            const uint64_t a = d0 + kk * dk;
                            mma_bf16(dst, a, a + dbh, idesc, (i > 0 || kk > 0) ? 1u : 0u);
                            if (three) {
                                mma_bf16(dst, a, a + dbl, idesc, 1u);
                                mma_bf16(dst, a + dal, a + dbh, idesc, 1u);
                            }
                        }
                    }
                    mma_commit(&sm.empty[s]);
                }
                __syncwarp();
                if (++s == ST) {
                    s = 0;
                    par ^= 1u;
                }
            }
            if (ok && elect_one()) mma_commit(&sm.acc_full[buf]);
            __syncwarp();
        }
        // All MMAs this warp issued have completed before TMEM is freed.
        if (elect_one()) mma_commit(&sm.drain);
        __syncwarp();
        mbar_wait(&sm.drain, 0);
    } else {
        // Epilogue: warp w reads accumulator lanes 32 (w % 4) .. + 31 (one row
        // per lane) in 32-column chunks, every second chunk.  Rows of C that
        // take it are written by 32-byte stores straight from the registers;
        // other row-major outputs go through a shared-memory transpose, so that
        // a store instruction covers two runs of 16 columns; outputs with
        // contiguous rows need neither.
        const int q = warp & 3;
        const int ew = warp - 2;
        float* stg = sm.epi[ew];
        int tl = 0;
        for (long long t = blockIdx.x; t < args.ntiles; t += gridDim.x, ++tl) {
            const TileCoord c = tile_coord(args, t);
            const int buf = tl & 1;
            if (!mbar_wait_or_fail(&sm.acc_full[buf], (uint32_t)((tl >> 1) & 1), fail)) break;
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            const int i = c.m0 + q * 32 + lane;
            const bool iok = i < args.M;
            long long roff = 0;
            if (iok) {
                const int b = i / args.Mb;
                roff = (long long)(c.bo + b) * args.cbs + (long long)(i - b * args.Mb) * args.crs +
                       (long long)c.split * args.split_stride;
            }
            const int jend = min(args.N, c.n0 + args.bn);
#pragma unroll 1
            for (int c0 = 32 * (ew >> 2); c.n0 + c0 < jend; c0 += 64) {
                uint32_t r[32];
                const uint32_t taddr =
                    tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * kMaxBN + c0);
                asm volatile(
                    "tcgen05.ld.sync.aligned.32x32b.x32.b32"
                    " {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
                    "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
                    : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                      "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]),
                      "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
                      "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
                      "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]),
                      "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                    : "r"(taddr));
                asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
                float val[32];
#pragma unroll
                for (int j = 0; j < 32; ++j)
                    val[j] = c.nk > 0 ? args.alpha * __uint_as_float(r[j]) : 0.f;
                const int j0 = c.n0 + c0;
                // RMW (beta != 0, no split): the old values of C are loaded
                // before any is used, so that their latencies overlap.
                if (args.vec) {
                    if (iok) {
                        float* p = args.C + roff + j0;
                        if constexpr (RMW) {
                            float old[32];
#pragma unroll
                            for (int g = 0; g < 4; ++g)
                                if (j0 + 8 * g < jend) ld8(p + 8 * g, old + 8 * g);
#pragma unroll
                            for (int j = 0; j < 32; ++j) val[j] = fmaf(args.beta, old[j], val[j]);
                        }
#pragma unroll
                        for (int g = 0; g < 4; ++g)
                            if (j0 + 8 * g < jend) st8(p + 8 * g, val + 8 * g);
                    }
                } else if (args.ccs == 1) {
#pragma unroll
                    for (int h = 0; h < 32 / kEpiCols; ++h) {
#pragma unroll
                        for (int j = 0; j < kEpiCols; ++j)
                            stg[lane * (kEpiCols + 1) + j] = val[h * kEpiCols + j];
                        __syncwarp();
                        const int jc = lane & (kEpiCols - 1), j = j0 + h * kEpiCols + jc;
                        const int rsub = lane / kEpiCols;
                        float old[kEpiCols];
#pragma unroll
                        for (int rr = 0; rr < 16; ++rr) {
                            const int row = 2 * rr + rsub;
                            const long long off = __shfl_sync(0xffffffffu, roff, row) + j;
                            const bool ok = c.m0 + q * 32 + row < args.M && j < jend;
                            if constexpr (RMW) old[rr] = ok ? args.C[off] : 0.f;
                            else if (ok) args.C[off] = stg[row * (kEpiCols + 1) + jc];
                        }
                        if constexpr (RMW) {
#pragma unroll
                            for (int rr = 0; rr < 16; ++rr) {
                                const int row = 2 * rr + rsub;
                                const long long off = __shfl_sync(0xffffffffu, roff, row) + j;
                                if (c.m0 + q * 32 + row < args.M && j < jend)
                                    args.C[off] = fmaf(args.beta, old[rr],
                                                       stg[row * (kEpiCols + 1) + jc]);
                            }
                        }
                        __syncwarp();
                    }
                } else if (iok) {
                    float* p = args.C + roff + (long long)j0 * args.ccs;
                    if constexpr (RMW) {
                        float old[32];
#pragma unroll
                        for (int j = 0; j < 32; ++j)
                            old[j] = j0 + j < jend ? p[(long long)j * args.ccs] : 0.f;
#pragma unroll
                        for (int j = 0; j < 32; ++j) val[j] = fmaf(args.beta, old[j], val[j]);
                    }
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        if (j0 + j < jend) p[(long long)j * args.ccs] = val[j];
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&sm.acc_empty[buf]);
        }
    }
    __syncthreads();
    if (sm.fail && threadIdx.x == 0) atomicExch(args.err, 1);
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem),
                     "r"(kCols));
}

// A strided float32 operand to pack into bf16 hi/lo, K-major:
// out[b][r][k] = split(src(b, r, k)), r < R, k < Kp (Kd rounded up to 16, so
// that rows start on 32-byte sectors), or out[r][b*Kp + k] for batch-reduced
// products.  Nothing is padded to tiles: the product's TMA loads read zeros
// beyond the operand.
struct PackOp {
    const float* src;
    long long rs, ks, bs;
    int R, Kd, Kp, nb, reduce;
    int vec;               // 16-byte loads along k
    long long units;       // blocks' worth of work
    __nv_bfloat16* hi;
    __nv_bfloat16* lo;     // null: hi only
};
constexpr int PK_R = 32, PK_K = 64;    // tiles of strided float64 sources
constexpr int PT_R = 64;               // rows of a tile of strided float32 sources
constexpr int PK_U = 4;                // contiguous sources: octets of k per thread

__device__ __forceinline__ void pack_octet(const PackOp& op, long long row, int b, int r, int k,
                                           const float* v) {
    union { __nv_bfloat16 b[8]; uint4 u; } vh, vl;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        const __nv_bfloat16 hh = __float2bfloat16_rn(v[e]);
        vh.b[e] = hh;
        vl.b[e] = __float2bfloat16_rn(v[e] - __bfloat162float(hh));
    }
    const long long o = op.reduce ? (long long)r * op.nb * op.Kp + (long long)b * op.Kp + k
                                  : row * op.Kp + k;
    *reinterpret_cast<uint4*>(op.hi + o) = vh.u;
    if (op.lo) *reinterpret_cast<uint4*>(op.lo + o) = vl.u;
}

// One block's unit of a source that is contiguous along k: 1024 octets of k,
// four per thread, their loads issued together (HBM bound: 8 bytes per element).
__device__ __forceinline__ void pack_contiguous(const PackOp& op, long long u) {
    const unsigned oc = (unsigned)op.Kp >> 3;
    const long long rows = (long long)op.nb * op.R, base = u * (256 * PK_U);
    const long long row0 = base / oc;
    const unsigned rem = (unsigned)(base - row0 * oc);
    float4 x[PK_U][2];
    long long row[PK_U];
    int b[PK_U], r[PK_U], k[PK_U];
#pragma unroll
    for (int h = 0; h < PK_U; ++h) {
        const unsigned l = rem + h * 256 + threadIdx.x;
        row[h] = row0 + l / oc;
        k[h] = (int)(l % oc) * 8;
        b[h] = (int)((unsigned)row[h] / (unsigned)op.R);
        r[h] = (int)row[h] - b[h] * op.R;
        const float* s = op.src + b[h] * op.bs + r[h] * op.rs + k[h];
        const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
        x[h][0] = row[h] < rows && k[h] < op.Kd ? *reinterpret_cast<const float4*>(s) : z;
        x[h][1] = row[h] < rows && k[h] + 4 < op.Kd ? *reinterpret_cast<const float4*>(s + 4) : z;
    }
#pragma unroll
    for (int h = 0; h < PK_U; ++h) {
        if (row[h] < rows) {
            const float v[8] = {x[h][0].x, x[h][0].y, x[h][0].z, x[h][0].w,
                                x[h][1].x, x[h][1].y, x[h][1].z, x[h][1].w};
            pack_octet(op, row[h], b[h], r[h], k[h], v);
        }
    }
}

// One block's unit of any other source: a 64 (r) x 64 (k) tile goes through
// shared memory so that the global reads run along whichever index of the
// source is contiguous, and every thread then writes 8 consecutive k of a row
// as one 16-byte store of hi and lo.  16 loads per thread are in flight (with
// 32 rows and 8 loads, 600 x 400 x 400 took 228 us, of which its bytes take 114).
__device__ __forceinline__ void pack_tile(const PackOp& op, long long u,
                                          float (*tile)[PK_K + 1]) {
    const int tk = (op.Kp + PK_K - 1) / PK_K, tr = (op.R + PT_R - 1) / PT_R;
    const int k0 = (int)(u % tk) * PK_K;
    const long long v = u / tk;
    const int r0 = (int)(v % tr) * PT_R, b = (int)(v / tr);
    const float* s = op.src + (long long)b * op.bs;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    float x[16];
    if (op.ks <= op.rs) {
        // warp w reads rows w, w + 8, ...; lanes run along k (two halves of 32)
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            const int r = r0 + warp + 8 * (e >> 1), k = k0 + (e & 1) * 32 + lane;
            x[e] = (r < op.R && k < op.Kd) ? s[(long long)r * op.rs + (long long)k * op.ks] : 0.f;
        }
#pragma unroll
        for (int e = 0; e < 16; ++e) tile[warp + 8 * (e >> 1)][(e & 1) * 32 + lane] = x[e];
    } else {
        // warp w reads columns w, w + 8, ...; lanes run along r (two halves of 32)
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            const int r = r0 + (e & 1) * 32 + lane, k = k0 + warp + 8 * (e >> 1);
            x[e] = (r < op.R && k < op.Kd) ? s[(long long)r * op.rs + (long long)k * op.ks] : 0.f;
        }
#pragma unroll
        for (int e = 0; e < 16; ++e) tile[(e & 1) * 32 + lane][warp + 8 * (e >> 1)] = x[e];
    }
    __syncthreads();
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        // 32 rows x 8 octets of k
        const int rr = (t >> 3) + 32 * h, r = r0 + rr, k = k0 + (t & 7) * 8;
        if (r < op.R && k < op.Kp) {
            float w[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) w[e] = tile[rr][(t & 7) * 8 + e];
            pack_octet(op, (long long)b * op.R + r, b, r, k, w);
        }
    }
    __syncthreads();
}

// Both operands of a product in one launch (one launch each cost 2 to 3 us
// more per product, and most operands are packed in 4 to 10).
__global__ void __launch_bounds__(256) k_pack(const PackOp a, const PackOp b) {
    grid_wait();
    __shared__ float tile[PT_R][PK_K + 1];
    for (long long u = blockIdx.x; u < a.units + b.units; u += gridDim.x) {
        if (u < a.units) {
            if (a.vec) pack_contiguous(a, u);
            else pack_tile(a, u, tile);
        } else {
            if (b.vec) pack_contiguous(b, u - a.units);
            else pack_tile(b, u - a.units, tile);
        }
    }
}

__global__ void k_splitk_sum(const float* part, int splits, int nbo, int M, int N,
                             long long pcbs, float* C, long long crs, long long ccs,
                             long long cbs, float alpha, float beta) {
    grid_wait();
    const long long MN = (long long)M * N, total = MN * nbo;
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
         idx += (long long)gridDim.x * blockDim.x) {
        const int b = (int)(idx / MN);
        const long long e = idx % MN;
        const int i = (int)(e / N), j = (int)(e % N);
        float acc = 0.f;
        for (int s = 0; s < splits; ++s)
            acc += part[((long long)s * nbo + b) * pcbs + (long long)i * N + j];
        float* c = C + (long long)b * cbs + (long long)i * crs + (long long)j * ccs;
        *c = beta != 0.f ? fmaf(beta, *c, alpha * acc) : alpha * acc;
    }
}

PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;
std::once_flag g_encode_once;

cudaError_t get_encode() {
    std::call_once(g_encode_once, [] {
        cudaDriverEntryPointQueryResult q;
        void* fn = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000,
                                             cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            g_encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    });
    return g_encode ? cudaSuccess : cudaErrorNotSupported;
}

// 3-D map over bf16 data [nbo][rows][Ktot] with boxes of 64 (K) x box_rows.
cudaError_t make_map(CUtensorMap* map, const __nv_bfloat16* base, long long Ktot, long long rows,
                     int nbo, int box_rows) {
    cuuint64_t dims[3] = {(cuuint64_t)Ktot, (cuuint64_t)rows, (cuuint64_t)nbo};
    cuuint64_t strides[2] = {(cuuint64_t)(Ktot * 2), (cuuint64_t)(Ktot * 2 * rows)};
    cuuint32_t box[3] = {(cuuint32_t)BK, (cuuint32_t)box_rows, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = g_encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, (void*)base, dims, strides, box,
                          estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

cudaError_t launch_tc(const CUtensorMap* maps, const TcArgs& a, cudaStream_t s) {
    const int stage = (a.nprod == 3 ? 2 : 1) * (BM + a.bn) * BK * 2;
    const int smem = a.stages * stage + (int)sizeof(TcCtl) + 1024;
    constexpr int kMost = kRingBytes + (int)sizeof(TcCtl) + 1024;
    static_assert(kMost <= 227 * 1024, "ring and control block exceed an SM's shared memory");
    cudaError_t e = smem_optin((const void*)k_gemm_tc<false>, kMost);
    if (e == cudaSuccess) e = smem_optin((const void*)k_gemm_tc<true>, kMost);
    if (e != cudaSuccess) return e;
    const long long sms = device_sms();
    const unsigned grid = (unsigned)std::min<long long>(a.ntiles, sms);
    if (a.splits == 1 && a.beta != 0.f)
        launch_chained(k_gemm_tc<true>, grid, kTcThreads, smem, s, maps[0], maps[1], maps[2],
                       maps[3], a);
    else
        launch_chained(k_gemm_tc<false>, grid, kTcThreads, smem, s, maps[0], maps[1], maps[2],
                       maps[3], a);
    count_launches(1);
    return cudaGetLastError();
}

long long rup(long long x, long long m) { return (x + m - 1) / m * m; }

// Self-test of the bounded-wait path: thread 0 waits on an mbarrier that is
// completed only if `complete` is set, with a budget of `cycles`; on expiry
// it raises *flag, as every production wait does, and returns.
__global__ void k_wait_selftest(int complete, long long cycles, int* flag) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x != 0) return;
    mbar_init(&bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    if (complete) mbar_arrive(&bar);
    const uint32_t a = smem_u32(&bar);
    const long long t0 = clock64();
    for (;;) {
        uint32_t done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
            " selp.b32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(a), "r"(0u));
        if (done) return;
        if (clock64() - t0 > cycles) {
            atomicExch(flag, 1);
            return;
        }
    }
}

}  // namespace

cudaError_t wait_selftest(int complete, long long cycles, int* flag, cudaStream_t s) {
    k_wait_selftest<<<1, 32, 0, s>>>(complete, cycles, flag);
    count_launches(1);
    return cudaGetLastError();
}

size_t gemm_tc_pack_elems(int M, int N, int K, int batch, bool reduce) {
    // Worst case over the two orientations (both sides padded to 128).
    const long long Kp = rup(std::max(K, 1), BK);
    const long long Rm = rup(M, 128), Rn = rup(N, 128);
    return (size_t)(2 * (Rm + Rn) * Kp * batch);
}

void PackCache::release() {
    for (Entry& e : entries) cudaFree(e.hi);
    entries.clear();
    constant.clear();
    bytes = 0;
}

namespace {

// Packed K of one batch: rows of packed operands start on 32-byte sectors.
long long pack_k(int K) { return rup(std::max(K, 1), UK); }

// Units of work of packing one operand (nb batches of R rows).
PackOp pack_op(const float* p, long long rs, long long ks, long long bs, int R, int Kd, int nb,
               int Kp, int reduce, __nv_bfloat16* hi, __nv_bfloat16* lo) {
    PackOp op{p, rs, ks, bs, R, Kd, Kp, nb, reduce, 0, 0, hi, lo};
    const long long rows = (long long)nb * R;
    op.vec = ks == 1 && Kd % 4 == 0 && rs % 4 == 0 && (nb == 1 || bs % 4 == 0) &&
             reinterpret_cast<uintptr_t>(p) % 16 == 0 && rows < INT32_MAX;
    op.units = op.vec ? (rows * (Kp / 8) + 256 * PK_U - 1) / (256 * PK_U)
                      : (long long)cdiv(Kp, PK_K) * cdiv(R, PT_R) * nb;
    return op;
}

// Where one operand's packed form goes: the workspace, or (use_cache) the
// cache of constant packs, where a form made before is taken as it is (units
// = 0) and a new one gets its own buffer (*made).  A cached operand that
// cannot be stored (budget or allocation) is an error, never a workspace
// write: the workspace was sized without it.
cudaError_t pack_target(const float* p, long long rs, long long cs, long long bs, int R, int Kd,
                        int nb, int nb_packed, int Kp, int reduce, int nprod,
                        __nv_bfloat16* ws_hi, __nv_bfloat16* ws_lo, bool use_cache,
                        PackCache* cache, PackOp* op, PackCache::Entry* made) {
    made->hi = nullptr;
    if (!use_cache) {
        *op = pack_op(p, rs, cs, bs, R, Kd, nb_packed, Kp, reduce, ws_hi, ws_lo);
        return cudaSuccess;
    }
    for (const PackCache::Entry& e : cache->entries)
        if (e.p == p && e.rs == rs && e.cs == cs && e.bs == bs && e.R == R && e.Kd == Kd &&
            e.nb == nb && e.Kp == Kp && e.reduce == reduce && e.nprod == nprod) {
            *op = PackOp{};
            op->hi = e.hi;
            op->lo = e.lo;
            return cudaSuccess;
        }
    const size_t elems = (size_t)R * Kp * nb_packed;
    const size_t bytes = elems * 2 * (nprod == 3 ? 2 : 1);
    if (cache->bytes + bytes > cache->budget) return cudaErrorMemoryAllocation;
    __nv_bfloat16* buf = nullptr;
    if (cudaMalloc(&buf, bytes) != cudaSuccess) {
        cudaGetLastError();
        return cudaErrorMemoryAllocation;
    }
    *made = PackCache::Entry{p, rs, cs, bs, R, Kd, nb, Kp, reduce, nprod, buf,
                             nprod == 3 ? buf + elems : nullptr};
    *op = pack_op(p, rs, cs, bs, R, Kd, nb_packed, Kp, reduce, made->hi, made->lo);
    return cudaSuccess;
}

}  // namespace

cudaError_t gemm_tc(const Gemm<float>& g, const TcWorkspace& ws, int nprod, cudaStream_t s,
                    PackCache* cache) {
    if (g.M <= 0 || g.N <= 0 || g.batch <= 0) return cudaSuccess;
    cudaError_t e = get_encode();
    if (e != cudaSuccess) return e;
    const int nb = g.batch;
    const int nbo = g.reduce ? 1 : nb;
    const bool bc = !g.reduce && nb > 1;
    const bool m_bc = bc && g.sAb == 0, n_bc = bc && g.sBb == 0;
    // Orientation: the UMMA M side (128-row tiles) takes the larger of M, N;
    // if one operand is shared by every batch, the rows of the other one's
    // batches (packed one after the other), so that a batch leaves no ragged
    // row tile of its own (400 rows fill 4 tiles of 128 to 78 %).
    bool swap = g.N > g.M, collapse = false;
    if (m_bc != n_bc && (long long)nb * (m_bc ? g.N : g.M) < INT32_MAX - BM) {
        swap = m_bc;
        collapse = true;
    }
    const int Mr = swap ? g.N : g.M, Nr = swap ? g.M : g.N;
    const int Kp = (int)pack_k(g.K);
    const long long Ktot = g.reduce ? (long long)Kp * nb : Kp;
    if (Ktot > INT32_MAX) return cudaErrorMemoryAllocation;
    // Operand views: UMMA-A rows r, K index k.
    // Unswapped: A side = A(m, k), B side = B(k, n) read as (n, k).
    View<float> va = g.A, vb{g.B.p, g.B.cs, g.B.rs};
    long long sa = g.sAb, sb = g.sBb;
    if (swap) {
        std::swap(va, vb);
        std::swap(sa, sb);
    }
    const bool a_bc = swap ? n_bc : m_bc, b_bc = swap ? m_bc : n_bc;
    const int nba = a_bc ? 1 : nbo, nbb = b_bc ? 1 : nbo;
    const size_t needA = (size_t)(Mr * Ktot * nba), needB = (size_t)(Nr * Ktot * nbb);
    // Operands served from the cache of constant packs take no workspace.
    const int red = g.reduce ? 1 : 0;
    const size_t bytesA = needA * 2 * (nprod == 3 ? 2 : 1);
    const size_t bytesB = needB * 2 * (nprod == 3 ? 2 : 1);
    const bool a_cached =
        cache && cache->serves(va.p, bytesA, va.rs, va.cs, sa, Mr, g.K, nb, Kp, red, nprod);
    // B is checked against the budget left after A's (possibly new) entry.
    bool b_cached = false;
    if (cache) {
        const size_t held = cache->bytes;
        if (a_cached) cache->bytes += bytesA;
        b_cached = cache->serves(vb.p, bytesB, vb.rs, vb.cs, sb, Nr, g.K, nb, Kp, red, nprod);
        cache->bytes = held;
    }
    const size_t need = (nprod == 3 ? 2 : 1) * ((a_cached ? 0 : needA) + (b_cached ? 0 : needB));
    if (need > ws.elems) return cudaErrorMemoryAllocation;
    // Workspace layout [A hi | B hi | A lo | B lo], cached operands omitted.
    const size_t wsA = a_cached ? 0 : needA, wsB = b_cached ? 0 : needB;
    __nv_bfloat16* a_hi = ws.buf;
    __nv_bfloat16* b_hi = a_hi + wsA;
    __nv_bfloat16* a_lo = nprod == 3 ? b_hi + wsB : nullptr;
    __nv_bfloat16* b_lo = nprod == 3 ? a_lo + wsA : nullptr;
    PackOp pa{}, pb{};
    PackCache::Entry made[2];
    made[1].hi = nullptr;
    e = pack_target(va.p, va.rs, va.cs, sa, Mr, g.K, nb, a_bc ? 1 : nb, Kp, red, nprod, a_hi, a_lo,
                    a_cached, cache, &pa, &made[0]);
    if (e == cudaSuccess) {
        // the second operand sees the budget that the first one's new form leaves
        const size_t held = cache ? cache->bytes : 0;
        if (made[0].hi) cache->bytes += bytesA;
        e = pack_target(vb.p, vb.rs, vb.cs, sb, Nr, g.K, nb, b_bc ? 1 : nb, Kp, red, nprod, b_hi,
                        b_lo, b_cached, cache, &pb, &made[1]);
        if (cache) cache->bytes = held;
    }
    if (e == cudaSuccess && pa.units + pb.units > 0) {
        const unsigned grid = (unsigned)std::min<long long>(pa.units + pb.units, 1 << 30);
        launch_chained(k_pack, grid, 256, 0, s, pa, pb);
        count_launches(1);
        e = cudaGetLastError();
    }
    for (int i = 0; i < 2; ++i) {
        if (!made[i].hi) continue;
        if (e != cudaSuccess) {
            cudaFree(made[i].hi);
        } else {
            cache->entries.push_back(made[i]);
            cache->bytes += i ? bytesB : bytesA;
        }
    }
    if (e != cudaSuccess) return e;

    TcArgs a{};
    a.M = collapse ? nb * Mr : Mr;
    a.N = Nr;
    a.Mb = Mr;
    a.nbo = collapse ? 1 : nbo;
    a.Ktot = (int)Ktot;
    a.ksteps = (int)((Ktot + BK - 1) / BK);
    a.nprod = nprod;
    a.a_bcast = a_bc ? 1 : 0;
    a.b_bcast = b_bc ? 1 : 0;
    a.err = ws.err;
    a.alpha = (float)g.alpha;
    a.beta = (float)g.beta;
    a.mblocks = (int)cdiv(a.M, BM);
    // Columns: as few tiles as 256 columns allow, of equal width; narrower
    // ones (down to 64) where the product would leave SMs idle and K is too
    // short to be split instead.
    const long long sms = device_sms(), rowtiles = (long long)a.mblocks * a.nbo;
    int nblocks = (int)cdiv(Nr, kMaxBN);
    if (a.ksteps < 16)
        while (rowtiles * nblocks < sms && Nr > 64 * nblocks) ++nblocks;
    a.bn = (int)rup(cdiv(Nr, nblocks), 16);
    a.nblocks = (int)cdiv(Nr, a.bn);
    const long long tiles = rowtiles * a.nblocks;
    // K splits: the count with the fewest K steps on the busiest SM.
    int splits = 1;
    if (tiles < sms && a.ksteps >= 8 && ws.partial) {
        const long long per = (long long)Mr * Nr * nbo;
        const int most = (int)std::min<long long>(
            {2 * sms / tiles, a.ksteps / 4, 32, per > 0 ? (long long)ws.partial_elems / per : 1});
        long long best = a.ksteps;
        for (int t = 2; t <= most; ++t) {
            const long long steps =
                (tiles * t + sms - 1) / sms * (((long long)a.ksteps + t - 1) / t);
            if (steps < best) {
                best = steps;
                splits = t;
            }
        }
    }
    a.splits = splits;
    a.ntiles = tiles * splits;
    const int stage = (nprod == 3 ? 2 : 1) * (BM + a.bn) * BK * 2;
    a.stages = std::min(kMaxStages, kRingBytes / stage);
    // C(m, n) = g.C[b*sCb + m*ldc + n]; accumulator (i, j) is (m, n) or (n, m).
    const long long crs = swap ? 1 : g.ldc, ccs = swap ? g.ldc : 1;
    if (splits > 1) {
        a.C = ws.partial;
        a.crs = Nr;
        a.ccs = 1;
        a.cbs = (long long)Mr * Nr;
        a.split_stride = a.cbs * nbo;
        a.alpha = 1.f;
    } else {
        a.C = g.C;
        a.crs = crs;
        a.ccs = ccs;
        a.cbs = g.reduce ? 0 : g.sCb;
    }
    a.vec = a.ccs == 1 && a.crs % 8 == 0 && (nbo == 1 || a.cbs % 8 == 0) && Nr % 8 == 0 &&
            reinterpret_cast<uintptr_t>(a.C) % 32 == 0;
    CUtensorMap maps[4];
    // a collapsed operand is one list of rows
    const long long rowsA = a.M, rowsB = Nr;
    const int mba = collapse ? 1 : nba, mbb = nbb;
    if ((e = make_map(&maps[0], pa.hi, Ktot, rowsA, mba, BM)) != cudaSuccess) return e;
    if ((e = make_map(&maps[1], nprod == 3 ? pa.lo : pa.hi, Ktot, rowsA, mba, BM)) != cudaSuccess)
        return e;
    if ((e = make_map(&maps[2], pb.hi, Ktot, rowsB, mbb, a.bn)) != cudaSuccess) return e;
    if ((e = make_map(&maps[3], nprod == 3 ? pb.lo : pb.hi, Ktot, rowsB, mbb, a.bn)) != cudaSuccess)
        return e;
    e = launch_tc(maps, a, s);
    if (e != cudaSuccess) return e;
    if (splits > 1) {
        const long long total = (long long)Mr * Nr * nbo;
        const unsigned blocks = (unsigned)std::min<long long>((total + 255) / 256, 152 * 16);
        launch_chained(k_splitk_sum, blocks, 256, 0, s, ws.partial, splits, nbo, Mr, Nr,
                       (long long)Mr * Nr, g.C, crs, ccs, g.reduce ? 0 : g.sCb, (float)g.alpha,
                       (float)g.beta);
        count_launches(1);
        e = cudaGetLastError();
    }
    return e;
}

// ---------------------------------------------------------------------------
// Float64 products on the tensor cores by integer slices (the splitting
// scheme of Ozaki et al.).  Every row r of an operand (UMMA orientation, K
// along the row; in a batch-reduced product the row runs over all batches) is
// scaled by 2^-e_r, e_r the binary exponent of its largest entry, so that its
// entries lie in (-1, 1), rounded to 55 fractional bits and cut into
// kSlices = 7 balanced digits of 8 bits (7 bits for the first):
//   x = 2^e_r (sum_t a_t 2^(1-8t) + r_x),   a_t in [-128, 128], |r_x| <= 2^-56,
// read straight from the IEEE-754 fields (integer operations only).
// A slice is exact in bf16, a product of two is an integer of at most 2^14,
// and a float32 sum of at most 1024 of them an integer of at most 2^24: the
// tensor cores' float32 accumulation is exact.  The pairs (t, u) with
// t + u = l form level l, S_l = sum a_t b_u, and
//   C = 2^(e_r + e_c) sum_{l=2..8} 2^(2-8l) S_l   (28 pairs).
// Balanced digits are why 28 pairs suffice: the digits left out (l >= 9) have
// random signs and change a product term by about 2^-56 of 2^(e_r + e_c)
// (rms), where 8 slices of 7 unsigned bits and 36 pairs, the form used before,
// lost 2^-55 with the product's own sign.  Against 64-bit-mantissa sums over
// K = 40, 400 and 4000 the error is 0.45 times the old one on Gaussian
// entries and 0.47 to 0.57 times on entries spread over 2^-40 .. 1.  (Six
// 9-bit digits and 26 pairs are as accurate, but products of such digits leave
// room for 256 of them only, so that two levels would be drained in every K
// step, where these digits drain one level every second step.)
namespace {

constexpr int kSlices = 7;
constexpr int kLevels = 7;                 // l = 2 .. 8 (q = l - 2)

// Biased exponent field of |x| (0 for zero; subnormals count as field 1).
__device__ __forceinline__ int f64_field(double x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffULL;
    const int f = (int)(b >> 52);
    return f == 0 ? (b != 0 ? 1 : 0) : f;
}

// Load a PK_R x PK_K tile of a strided float64 operand (zeros outside) the way
// k_pack does: reads run along whichever index is contiguous.
__device__ __forceinline__ void f64_tile(double (*tile)[PK_K + 1], const double* s, long long rs,
                                         long long ks, int R, int Kd, int r0, int k0) {
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    if (ks <= rs) {
        for (int rr = warp; rr < PK_R; rr += 8) {
            const int r = r0 + rr;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int k = k0 + h * 32 + lane;
                tile[rr][h * 32 + lane] =
                    (r < R && k < Kd) ? s[(long long)r * rs + (long long)k * ks] : 0.0;
            }
        }
    } else {
        for (int kk = warp; kk < PK_K; kk += 8) {
            const int r = r0 + lane, k = k0 + kk;
            tile[lane][kk] = (r < R && k < Kd) ? s[(long long)r * rs + (long long)k * ks] : 0.0;
        }
    }
}

// One operand of a product: rows r < R, K indices k < Kd of batches b < nb at
// src[b bs + r rs + k ks]; its slices and row exponents.  A launch covers both
// operands of a product: blocks 0 .. nblk(A) - 1 and the rest.
struct SliceOp {
    const double* src;
    long long rs, ks, bs;
    int R, nb;
    int flat;            // the batches' rows form one list (b R + r) of the slices
    __nv_bfloat16* out;
    int* expo;
};
struct SlicePair {
    SliceOp op[2];
    long long blocks0;   // blocks of op[0]
    int Kd, Kp, reduce;
    long long Ktot;
};

// The tile of this block of 64 K indices x 32 rows: k tile fastest, then row
// tile, then batch.
struct SliceTile {
    int k0, r0, b;
};
__device__ __forceinline__ SliceTile slice_tile(const SlicePair& p, const SliceOp& op, long long blk) {
    const int kt = (p.Kp + PK_K - 1) / PK_K, rt = (op.R + PK_R - 1) / PK_R;
    SliceTile t;
    t.k0 = (int)(blk % kt) * PK_K;
    blk /= kt;
    t.r0 = (int)(blk % rt) * PK_R;
    t.b = (int)(blk / rt);
    return t;
}

// expo[bo * R + r] = max over the row of the biased exponent field (atomic
// over the K tiles; the array starts at zero = all-zero row).
__global__ void __launch_bounds__(256) k_row_exp(const __grid_constant__ SlicePair p) {
    grid_wait();
    __shared__ double tile[PK_R][PK_K + 1];
    const bool second = blockIdx.x >= p.blocks0;
    const SliceOp& op = p.op[second];
    const SliceTile c = slice_tile(p, op, blockIdx.x - (second ? p.blocks0 : 0));
    const int t = threadIdx.x;
    f64_tile(tile, op.src + c.b * op.bs, op.rs, op.ks, op.R, p.Kd, c.r0, c.k0);
    __syncthreads();
    const int rr = t >> 3, oct = t & 7;
    int m = 0;
#pragma unroll
    for (int e = 0; e < 8; ++e) m = max(m, f64_field(tile[rr][oct * 8 + e]));
    // the 8 threads of a row are consecutive lanes of one warp
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) m = max(m, __shfl_down_sync(0xffffffffu, m, o, 8));
    const int r = c.r0 + rr;
    if (oct == 0 && r < op.R && m > 0)
        atomicMax(&op.expo[(p.reduce ? 0 : (long long)c.b * op.R) + r], m);
}

// Bits of the float32 whose upper half is the bf16 digit (byte n of w) - 128:
// 2^23 + byte is exact in float32, the subtraction leaves the digit, and a
// float32 of at most 8 significant bits is its bf16 in the upper 16 bits.
__device__ __forceinline__ unsigned digit_bits(unsigned w, int n) {
    const unsigned f = __byte_perm(w, 0x4B000000u, 0x7440u | (unsigned)n);
    return __float_as_uint(__uint_as_float(f) - 8388736.0f);
}

// The 7 digits of x as such float32 bits, d[t - 1] = digit t, for a row of
// exponent field fe (x below 2^(fe - 1022)).  V = x 2^(55 - e) rounded to an
// integer, |V| <= 2^55; adding 128 to each of its six low bytes turns the
// balanced base-256 digits into unsigned ones (and 256 the first, on top).
__device__ __forceinline__ void f64_digits(double x, int fe, unsigned (&d)[kSlices]) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
    const int f = (int)((bits >> 52) & 0x7ff);
    const unsigned long long mant =
        ((bits & 0xfffffffffffffULL) | (f ? (1ULL << 52) : 0ULL)) << 2;
    const int sh = fe - (f ? f : 1);       // >= 0 (an all-zero row has fe = 0 and mant = 0)
    // round half up at the shifted-out bit; mant has two spare low bits
    unsigned long long V = 0;
    if (sh <= 2) V = mant >> max(sh, 0);
    else if (sh < 56) V = (mant + (1ULL << (sh - 1))) >> sh;
    const unsigned long long W = ((bits >> 63) ? 0ULL - V : V) + 0x0100808080808080ULL;
    const unsigned lo = (unsigned)W, hi = (unsigned)(W >> 32);
    d[6] = digit_bits(lo, 0);
    d[5] = digit_bits(lo, 1);
    d[4] = digit_bits(lo, 2);
    d[3] = digit_bits(lo, 3);
    d[2] = digit_bits(hi, 0);
    d[1] = digit_bits(hi, 1);
    d[0] = __float_as_uint(__uint_as_float(0x4B000000u | (hi >> 16)) - 8388864.0f);
}

// Slices of one operand, 64 K indices at a time: element (bo, k, slice q, r)
// at ((bo nkb + k / 64) kSlices + q) R + r) 64 + k % 64, so that what a K step
// of the product reads lies together (with K running along whole rows, a step
// of a 400 x 240000 operand touched 2800 lines 3.4 MB apart: 7800 cycles per
// K step instead of 6000).  A reduced product's batches follow one another
// along k (Kp indices each, Kp a multiple of 8).  Written up to the next
// multiple of 16, which is as far as the product reads.
__device__ __forceinline__ void slice_store(const SlicePair& p, const SliceOp& op, int b, int r, int k,
                                            const double* x, int fe) {
    unsigned v[kSlices][4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        unsigned d0[kSlices], d1[kSlices];
        f64_digits(x[2 * j], fe, d0);
        f64_digits(x[2 * j + 1], fe, d1);
#pragma unroll
        for (int q = 0; q < kSlices; ++q) v[q][j] = __byte_perm(d0[q], d1[q], 0x7632);
    }
    const long long nkb = (p.Ktot + BK - 1) / BK;
    const long long kg = (p.reduce ? (long long)b * p.Kp : 0) + k;
    const long long bo = p.reduce || op.flat ? 0 : b;
    const long long rows = op.flat ? (long long)op.nb * op.R : op.R;
    const long long row = op.flat ? (long long)b * op.R + r : r;
    __nv_bfloat16* o = op.out + ((bo * nkb + kg / BK) * kSlices * rows + row) * BK + kg % BK;
    const long long plane = rows * BK;
#pragma unroll
    for (int q = 0; q < kSlices; ++q)
        *reinterpret_cast<uint4*>(o + q * plane) = make_uint4(v[q][0], v[q][1], v[q][2], v[q][3]);
}

// True for the 8 K indices from k on that have to be written: the batch's own
// and, after the last one, the zeros up to a multiple of 16.
__device__ __forceinline__ bool slice_written(const SlicePair& p, int b, int nb, int k) {
    if (k < p.Kp) return true;
    return (!p.reduce || b == nb - 1) &&
           (p.reduce ? (long long)b * p.Kp : 0) + k < (p.Ktot + 15) / 16 * 16;
}

__global__ void __launch_bounds__(256, 5) k_slice64(const __grid_constant__ SlicePair p) {
    grid_wait();
    __shared__ double tile[PK_R][PK_K + 1];
    const bool second = blockIdx.x >= p.blocks0;
    const SliceOp& op = p.op[second];
    const SliceTile c = slice_tile(p, op, blockIdx.x - (second ? p.blocks0 : 0));
    f64_tile(tile, op.src + c.b * op.bs, op.rs, op.ks, op.R, p.Kd, c.r0, c.k0);
    __syncthreads();
    const int rr = threadIdx.x >> 3, oct = threadIdx.x & 7;
    const int r = c.r0 + rr, k = c.k0 + oct * 8;
    if (r < op.R && slice_written(p, c.b, op.nb, k))
        slice_store(p, op, c.b, r, k, &tile[rr][oct * 8],
                    op.expo[(p.reduce ? 0 : (long long)c.b * op.R) + r]);
}

// Exponents and slices in one pass for rows that fit shared memory (separate
// batches, K <= kFusedK): a block holds SR rows with all their K indices, so
// that the operand is read once and no exponent array has to be cleared.
constexpr int SR = 16;            // rows per block
constexpr int kFusedK = 512;      // at most 75 KB of shared memory: three blocks per SM

// Place of K index k in a row (8 threads read 8 groups of 8 at once), and the
// odd number of doubles of a row of Kw (a multiple of 16).
__host__ __device__ __forceinline__ int row_at(int k) { return k + (k >> 3); }
__host__ __device__ __forceinline__ int row_pitch(int Kw) { return Kw / 8 * 9 + 1; }

__global__ void __launch_bounds__(256) k_slice_rows(const __grid_constant__ SlicePair p) {
    grid_wait();
    extern __shared__ __align__(16) double rows[];   // [SR][pitch]
    __shared__ int fe[SR];
    const bool second = blockIdx.x >= p.blocks0;
    const SliceOp& op = p.op[second];
    const long long blk = blockIdx.x - (second ? p.blocks0 : 0);
    const int rt = (op.R + SR - 1) / SR;
    const int r0 = (int)(blk % rt) * SR, b = (int)(blk / rt);
    const double* s = op.src + b * op.bs;
    // K indices held: the written ones
    const int Kw = (p.Kp + 15) / 16 * 16, pitch = row_pitch(Kw);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (op.ks <= op.rs) {
        for (int rr = warp; rr < SR; rr += 8) {
            const int r = r0 + rr;
#pragma unroll 4
            for (int k = lane; k < Kw; k += 32)
                rows[rr * pitch + row_at(k)] = (r < op.R && k < p.Kd) ? s[(long long)r * op.rs + (long long)k * op.ks] : 0.0;
        }
    } else {
        // half a warp along the rows
        const int rr = threadIdx.x & (SR - 1), r = r0 + rr;
#pragma unroll 4
        for (int k = threadIdx.x / SR; k < Kw; k += 256 / SR)
            rows[rr * pitch + row_at(k)] = (r < op.R && k < p.Kd) ? s[(long long)r * op.rs + (long long)k * op.ks] : 0.0;
    }
    __syncthreads();
    for (int rr = warp; rr < SR; rr += 8) {
        int m = 0;
        for (int k = lane; k < Kw; k += 32) m = max(m, f64_field(rows[rr * pitch + row_at(k)]));
        m = __reduce_max_sync(0xffffffffu, m);
        if (lane == 0) {
            fe[rr] = m;
            if (r0 + rr < op.R) op.expo[(long long)b * op.R + r0 + rr] = m;
        }
    }
    __syncthreads();
    // 8 K indices per thread: 8 threads write 128 contiguous bytes of a slice
    const int octs = Kw / 8;
    for (int e = threadIdx.x; e < SR * ((octs + 7) / 8) * 8; e += 256) {
        const int oct = e / (8 * SR) * 8 + (e & 7), rr = (e >> 3) & (SR - 1);
        if (oct < octs && r0 + rr < op.R) {
            double x[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) x[j] = rows[rr * pitch + oct * 9 + j];
            slice_store(p, op, b, r0 + rr, oct * 8, x, fe[rr]);
        }
    }
}

// Lists the outputs (i, j) of a single product with
//   sum_k |a_ik b_jk| < 2^(e_i + e_j)          (e: the exponents of the slices);
// redo[0] counts them (the list ends at `cap`).
// A product by slices is off by at most K 2^-53 2^(e_i + e_j) (rounding of the
// operands and digit pairs left out, 8 units of 2^-56 per term), float64 sums
// by K 2^-53 sum_k |a_ik b_jk| and more: where the sum reaches the scale, the
// slices' bound is no larger.  It does not where the large entries of a row meet
// the small ones of a column, and at a few outputs of heavy-tailed rows.  The sum
// is bounded from below by the first digits, |a| >= (|a_1| - 0.502) 2^(e - 7): as 8-bit
// integers 2 |a_1| - 1 (0.4 % above that at most, which kEnough allows for), four
// products per instruction, and only until every output of the tile has enough: 60
// of 300 K indices for Gaussian entries.  Zero rows are exact; those with a
// non-finite entry and results outside 2^-700 .. 2^800 are left to float64 sums.
// Tile of 32 x 32 outputs, 2 x 2 per thread: 12 us for 8000 x 200 x 300, 29 for
// 300 x 200 x 8000 (few tiles, 10 K blocks each), 25 for 8000 x 300 x 200; with
// float32 products 26, 46 and 59.
constexpr unsigned kEnough = 66200u;     // (2 2^7)^2 and a hundredth
__global__ void __launch_bounds__(256)
    k_slices_even(const __nv_bfloat16* A, const __nv_bfloat16* B, int M, int N, int K,
                  const int* eA, const int* eB, int* redo, int2* list, int cap) {
    grid_wait();
    __shared__ unsigned a[BK / 4][33], b[BK / 4][33];      // four K indices per word
    const int nt = (N + 31) / 32;
    const int m0 = (int)(blockIdx.x / (unsigned)nt) * 32, n0 = (int)(blockIdx.x % (unsigned)nt) * 32;
    const int lr = threadIdx.x >> 3, lk = (threadIdx.x & 7) * 8;     // row and K octet loaded
    const int tr = threadIdx.x >> 4, tc = threadIdx.x & 15;
    unsigned sum[2][2] = {};
    bool need[2][2], bad[2][2];   // a sum to look at; an output that is not for slices
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int m = m0 + tr + 16 * i, n = n0 + tc + 16 * j;
            const bool in = m < M && n < N;
            const int ea = in ? eA[m] : 0, eb = in ? eB[n] : 0, e = ea + eb;
            const bool zero = ea == 0 || eb == 0;
            bad[i][j] = max(ea, eb) == 2047 || (!zero && (e <= 2044 - 700 || e >= 2044 + 800));
            need[i][j] = !zero && !bad[i][j];
        }
    // 2 |d| - 1 or 0 in the low byte of the float's bits
    auto lower = [](unsigned half) {
        return __float_as_uint(fmaxf(fmaf(2.f, fabsf(__uint_as_float(half << 16)), 8388607.f), 8388608.f)) &
               0xFFu;
    };
    for (int k0 = 0;; k0 += BK) {
        bool enough = true;
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 2; ++j) enough = enough && (!need[i][j] || sum[i][j] >= kEnough);
        // (also the barrier between the reads of a K block and its successor's writes)
        if (__syncthreads_and(enough) || k0 >= K) break;
        const uint4 z = make_uint4(0u, 0u, 0u, 0u);
        const long long at = (long long)(k0 / BK) * kSlices;
        const uint4 va = m0 + lr < M
            ? *reinterpret_cast<const uint4*>(A + (at * M + m0 + lr) * BK + lk) : z;
        const uint4 vb = n0 + lr < N
            ? *reinterpret_cast<const uint4*>(B + (at * N + n0 + lr) * BK + lk) : z;
        const unsigned ua[4] = {va.x, va.y, va.z, va.w}, ub[4] = {vb.x, vb.y, vb.z, vb.w};
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            unsigned wa = 0u, wb = 0u;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int e = 4 * h + j;
                if (k0 + lk + e < K) {            // (what follows is not written)
                    wa |= lower(ua[e / 2] >> (16 * (e & 1)) & 0xFFFFu) << (8 * j);
                    wb |= lower(ub[e / 2] >> (16 * (e & 1)) & 0xFFFFu) << (8 * j);
                }
            }
            a[lk / 4 + h][lr] = wa;
            b[lk / 4 + h][lr] = wb;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < BK / 4; ++k) {
            const unsigned a0 = a[k][tr], a1 = a[k][tr + 16], b0 = b[k][tc], b1 = b[k][tc + 16];
            sum[0][0] = __dp4a(a0, b0, sum[0][0]);
            sum[0][1] = __dp4a(a0, b1, sum[0][1]);
            sum[1][0] = __dp4a(a1, b0, sum[1][0]);
            sum[1][1] = __dp4a(a1, b1, sum[1][1]);
        }
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 2; ++j) sum[i][j] = min(sum[i][j], 1u << 24);   // (no wrap)
    }
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j)
            if ((bad[i][j] || (need[i][j] && sum[i][j] < kEnough)) &&
                *(volatile int*)redo <= cap) {       // (more need not be counted)
                const int at = atomicAdd(redo, 1);
                if (at < cap) list[at] = make_int2(m0 + tr + 16 * i, n0 + tc + 16 * j);
            }
}

// The listed outputs as float64 sums, a warp each; if there are more than `cap` of
// them, or C's old values were needed, only says so in redo[1].
__global__ void __launch_bounds__(256)
    k_redo64(const double* A, long long ars, long long aks, const double* B, long long brs,
             long long bks, int K, double alpha, double* C, long long crs, long long ccs, int* redo,
             const int2* list, int cap) {
    grid_wait();
    const int n = redo[0], lane = threadIdx.x & 31;
    if (n > cap) {
        if (blockIdx.x == 0 && threadIdx.x == 0) redo[1] = 1;
        return;
    }
    for (int e = blockIdx.x * 8 + (threadIdx.x >> 5); e < n; e += gridDim.x * 8) {
        const int2 ij = list[e];
        const double *a = A + ij.x * ars, *b = B + ij.y * brs;
        double s = 0.0;
#pragma unroll 4
        for (int k = lane; k < K; k += 32) s = fma(a[k * aks], b[k * bks], s);
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if (lane == 0) C[ij.x * crs + ij.y * ccs] = alpha * s;
    }
}

__device__ __forceinline__ double pow2(int k) {
    return (k >= -1022 && k <= 1023) ? __longlong_as_double((long long)(k + 1023) << 52)
                                     : scalbn(1.0, k);
}

// 5-D map over the slices (K index in its block, row, slice, block, batch)
// with boxes of 64 x box_rows x box_slices; rows outside read zero.
cudaError_t make_map_slices(CUtensorMap* map, const __nv_bfloat16* base, long long nkb,
                            long long rows, int nbo, int box_rows, int box_slices) {
    cuuint64_t dims[5] = {(cuuint64_t)BK, (cuuint64_t)rows, (cuuint64_t)kSlices, (cuuint64_t)nkb,
                          (cuuint64_t)nbo};
    const cuuint64_t row = BK * 2, plane = row * (cuuint64_t)rows, block = plane * kSlices;
    cuuint64_t strides[4] = {row, plane, block, block * (cuuint64_t)nkb};
    cuuint32_t box[5] = {(cuuint32_t)BK, (cuuint32_t)box_rows, (cuuint32_t)box_slices, 1, 1};
    cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    CUresult r = g_encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, (void*)base, dims, strides, box,
                          estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

constexpr int FN = 64;                    // tile columns (B rows)
constexpr int kMaxSteps = 1024;           // 64-wide K steps of one tile (range of the int64 sums)

// K indices of a slice: K rounded up to a 16-byte store, batches of a reduced
// product one after another.
long long f64_ktot(int K, int batch, bool reduce) {
    const long long Kp = rup(std::max(K, 1), 8);
    return reduce ? Kp * batch : Kp;
}

// Split-K count: items = tiles x splits fill waves of SMs, each item takes its
// K steps (1.9 us each at the tensor pipe's rate) and about one step more for
// its first loads and its last drains, and the float64 partials are written
// and read once.  At least 4 K steps per split, at most 32 splits.
int f64_splits(long long tiles, long long ksteps, long long outputs, size_t part_elems,
               long long sms) {
    auto cost = [&](long long sp) {
        const double waves = (double)((tiles * sp + sms - 1) / sms);
        const double sum = sp > 1 ? (2.0 + outputs * sp * 16.0 / 4e6) / 1.9 : 0.0;
        return waves * ((double)((ksteps + sp - 1) / sp) + 1.0) + sum;
    };
    const int lo = (int)((ksteps + kMaxSteps - 1) / kMaxSteps);
    int best = lo;
    for (int sp = lo + 1; sp <= 32 && ksteps / sp >= 4; ++sp) {
        if ((size_t)(outputs * sp) > part_elems / 2) break;
        if (cost(sp) < 0.98 * cost(best)) best = sp;
    }
    return best;
}

}  // namespace

void gemm_f64_tc_sizes(int M, int N, int K, int batch, bool reduce, size_t* slice_elems,
                       size_t* part_elems, size_t* expo_elems) {
    const long long Ktot = f64_ktot(K, batch, reduce);
    const long long nbo = reduce ? 1 : batch;
    *slice_elems = (size_t)(kSlices * ((long long)M + N) * rup(Ktot, BK) * nbo);
    // float64 split-K partials, counted in floats: only products of few tiles
    // or of a K above one tile's range are split
    const long long tiles = (long long)cdiv(std::max(M, N), BM) * cdiv(std::min(M, N), FN) * nbo;
    const long long steps = (Ktot + BK - 1) / BK;
    const long long sp = tiles < 2 * 152 || steps > kMaxSteps
                             ? std::max<long long>(1, std::min<long long>(32, steps / 4)) : 0;
    *part_elems = (size_t)(2 * sp * nbo * (long long)M * N);
    *expo_elems = (size_t)(((long long)M + N) * nbo);
}

// ---------------------------------------------------------------------------
// Fused float64 product: one persistent kernel per product.  For every
// 64-wide K step it loads the 7 slices of a 128-row A tile and of a 64-row B
// tile once and forms the 28 digit pairs (t, u), t + u <= 8, in seven level
// accumulators in tensor memory (level q = t + u - 2 at columns 64 q ..
// 64 q + 63).  The B slices lie one after another in shared memory and the
// levels of A slice t one after another in tensor memory, so one MMA of
// N = 64 m forms m pairs at once: A is read from shared memory 10 times per
// 16-deep sub-step instead of 28 (an MMA of N = 64 reads 6 KB in the 32 cycles
// it computes, above the 128 bytes per cycle shared memory delivers; the
// merged ones average 110), and 40 MMAs are issued per K step.
// A level is drained before its sum can pass 2^24: (q + 1) pairs x 64 x 2^14
// per step, every 16, 8, 4, 4 and 2 steps for q = 0 .. 4 (exact); q = 5 and 6
// weigh 2^-54 and 2^-62 and are drained every 4 and 8 steps: digits of one sign
// near the largest ones take their sums to 1.5 and 3.5 times 2^24, and each MMA
// beyond 2^24 rounds the sum by one or two units, 2^-57 per term in all.
// Measured with slicing and exponents (8 unsigned slices, one MMA per pair ->
// this kernel): 4096^3 5.78 -> 2.65 ms (52 TFLOP/s of float64, 0.77 of the
// measured bf16 peak on its 28 products), 400 x 400 x 240000 6.54 -> 3.27 ms,
// 240000 x 400 x 400 6.43 -> 2.45 ms, 160000 x 1200 x 200 5.17 -> 2.03 ms and
// x 40 3.22 -> 1.12 ms (there the epilogue's integer operations bound it).
// The epilogue warps combine drains in registers: int64 for q <= 4, float32
// for the rest with its integer part carried into the int64 after each drain
// of q = 6.  The tile is written once, converted to float64 by integer
// operations: assembled on the FP64 pipe (2 lanes per SM and cycle), a tile's
// 8192 results take 4100 cycles per operation, whether it is predicated off
// or not, against 2700 cycles of MMA at K = 40; so that products with a
// general alpha or beta, which need that pipe, take a loop of their own.
// Roles: warp 0 streams slices with TMA (B slices of a K step double-
// buffered, A slices through a ring), warp 1 issues the MMAs, warps 2-17
// drain: warp w reads TMEM lanes 32 (w % 4) .. + 31 and columns
// 16 ((w - 2) / 4) .. + 15 of a level (16 warps: the conversions to int64 and
// the TMEM reads are latency chains that eight did not hide).  A level's
// drain is requested as soon as its last pair of the step is issued (q after
// A slice q + 1), so that it overlaps the remaining pairs.  Every wait is
// bounded.
namespace {

constexpr int FA = 6;                     // A-slice ring depth
constexpr int kF64EpiWarps = 16;
constexpr int kF64Threads = 64 + 32 * kF64EpiWarps;
constexpr int FC = 16;                    // columns of a level per epilogue warp

struct F64Smem {
    __nv_bfloat16 b[2][kSlices * FN * BK];  // B slices of one K step, slice after slice
    __nv_bfloat16 a[FA][BM * BK];           // A slices, one per ring entry
    alignas(16) int eb[kF64EpiWarps][FC];   // exponent fields of each warp's columns
    uint64_t bfull[2], bempty[2], afull[FA], aempty[FA];
    uint64_t lfull[kLevels], lempty[kLevels];
    uint64_t drain;
    uint32_t tmem;
    int fail;
};

struct F64Args {
    int M, N;                // real accumulator rows (A side, all batches of a
                             // collapsed product) and columns (B side)
    int Mb;                  // rows per batch: row i is row i % Mb of batch bo + i / Mb
    int nbo, mblocks, nblocks, ksteps, splits;
    int last_kk;             // 16-deep sub-steps of the last K step
    long long ntiles;        // mblocks * nblocks * nbo * splits
    int a_bcast, b_bcast;
    const int* eA;           // row exponent fields [bo][M], [bo][N]
    const int* eB;
    double* C;               // output, or float64 partials when splits > 1
    long long crs, ccs, cbs;
    long long split_stride;  // partials of one split
    double alpha, beta;
    int alpha_exp;           // alpha = +-2^alpha_exp, or kNoPow2
    int hshift;              // fractional bits below the int64 sums' unit
    int* err;
};
constexpr int kNoPow2 = 1 << 20;

struct F64Coord {
    int m0, n0, bo, split, k_lo, nk;
};

__device__ __forceinline__ F64Coord f64_coord(const F64Args& a, long long t) {
    F64Coord c;
    const int nbk = (int)(t % a.nblocks);
    long long r = t / a.nblocks;
    const int mbk = (int)(r % a.mblocks);
    r /= a.mblocks;
    c.bo = (int)(r / a.splits);
    c.split = (int)(r % a.splits);
    c.m0 = mbk * BM;
    c.n0 = nbk * FN;
    const int chunk = (a.ksteps + a.splits - 1) / a.splits;
    c.k_lo = c.split * chunk;
    c.nk = max(0, min(a.ksteps, c.k_lo + chunk) - c.k_lo);
    return c;
}

// Levels (bit q) that K step i starts afresh: every 16, 8, 4, 4, 2, 4, 8 steps
// for q = 0 .. 6, so none at odd steps, {4} at 2 mod 4, {2 .. 5} at 4 mod 8,
// {1 .. 6} at 8 mod 16, all at 0 mod 16.  Step i drains what step i + 1 starts.
__device__ __forceinline__ unsigned f64_fresh(int i) {
    return (unsigned)(0x7F7E3C1000ULL >> (8 * (__ffs(i | 16) - 1))) & 0x7fu;
}
__device__ __forceinline__ unsigned f64_drained(int i, int nk) {
    return i == nk - 1 ? 0x7fu : f64_fresh(i + 1);
}

// Slices sl .. of rows row .. in K block kb of batch b.
__device__ __forceinline__ void tma_load_slices(void* dst, const CUtensorMap* map, uint64_t* bar,
                                                int row, int sl, int kb, int b) {
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4, %5, %6}], [%7];\n" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(0), "r"(row), "r"(sl), "r"(kb), "r"(b),
        "r"(smem_u32(bar))
        : "memory");
}

// F 2^e (|F| < 2^62) for the whole range: all-zero rows, values near the ends
// of the float64 range, rows with a non-finite entry, small F.
__device__ __noinline__ double f64_scaled(long long F, int fa, int fb, int e) {
    if (fa == 2047 || fb == 2047) return __longlong_as_double(0x7ff8000000000000LL);
    if (F == 0) return 0.0;
    return (double)F * pow2(e);
}

// Bits of the same by integer operations, rounded to nearest, for |F| >= 2^32
// and a result inside the normal range.
__device__ __forceinline__ long long f64_bits(long long F, int e, unsigned neg) {
    const int s = (int)(F >> 63);
    const unsigned long long a = (unsigned long long)((F ^ (long long)s) - s);
    // leading one at bit 62, rounded to 53 bits with it at bit 52, where it
    // adds itself to the exponent
    const int lz1 = __clz((int)(a >> 32)) - 1;
    const unsigned long long m = ((a << lz1) + 0x200ULL) >> 10;
    const unsigned hi = (unsigned)(m >> 32) + ((unsigned)(1084 + e - lz1) << 20);
    return (long long)(((unsigned long long)(hi | (((unsigned)s ^ neg) & 0x80000000u)) << 32) |
                       (unsigned)m);
}

// Turn the FC sums of one accumulator row into the bits of their float64
// values 2^(fa + eb[j] + ebase) F, in place (neg: all ones to negate).
__device__ __forceinline__ void f64_finish(long long (&H)[FC], const float (&T)[FC], const int* eb,
                                           int hs, int fa, int ebase, unsigned neg, bool range_ok,
                                           int ncols) {
    const float ts = __uint_as_float((unsigned)(127 + hs) << 23);
    unsigned slow = range_ok ? 0u : 0xffffffffu;
    int e[FC];
#pragma unroll
    for (int j = 0; j < FC; j += 4) {
        const int4 v = *reinterpret_cast<const int4*>(eb + j);
        e[j] = v.x;
        e[j + 1] = v.y;
        e[j + 2] = v.z;
        e[j + 3] = v.w;
    }
#pragma unroll
    for (int j = 0; j < FC; ++j) {
        const float m = fmaf(T[j], ts, 12582912.f);
        H[j] = (H[j] << hs) + (int)(__float_as_uint(m) - 0x4B400000u);
        // |F| < 2^32: the high word is 0 or all ones (a few of 2^62)
        const int h = (int)(H[j] >> 32);
        if ((h ^ (h >> 31)) == 0) slow |= 1u << j;
    }
    slow &= (1u << ncols) - 1u;   // (columns outside are not stored)
    if (slow == 0) {
#pragma unroll
        for (int j = 0; j < FC; ++j) H[j] = f64_bits(H[j], fa + ebase + e[j], neg);
    } else {
#pragma unroll
        for (int j = 0; j < FC; ++j) {
            const double v = f64_scaled(neg ? -H[j] : H[j], fa, e[j], fa + ebase + e[j]);
            H[j] = __double_as_longlong(v);
        }
    }
}

__global__ void __launch_bounds__(kF64Threads, 1)
    k_gemm_f64s(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                const F64Args args) {
    grid_wait();
    extern __shared__ __align__(1024) unsigned char f64_raw[];
    F64Smem& sm = *reinterpret_cast<F64Smem*>((reinterpret_cast<uintptr_t>(f64_raw) + 1023) &
                                              ~uintptr_t(1023));
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    volatile int* fail = &sm.fail;
    if (threadIdx.x == 0) {
        for (int s = 0; s < 2; ++s) {
            mbar_init(&sm.bfull[s], 1);
            mbar_init(&sm.bempty[s], 1);
        }
        for (int s = 0; s < FA; ++s) {
            mbar_init(&sm.afull[s], 1);
            mbar_init(&sm.aempty[s], 1);
        }
        for (int q = 0; q < kLevels; ++q) {
            mbar_init(&sm.lfull[q], 1);
            mbar_init(&sm.lempty[q], kF64EpiWarps);
        }
        mbar_init(&sm.drain, 1);
        sm.fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                         smem_u32(&sm.tmem)),
                     "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
    }
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = sm.tmem;

    if (warp == 0) {
        if (lane == 0) {
            // TMA producer
            long long bit = 0, ait = 0;
            long long blast[2] = {-1, -1};
            int as = 0;              // ring slot and parity of the next A slice
            uint32_t apar = 1;       // (the first pass over the ring does not wait)
            bool ok = true;
            for (long long t = blockIdx.x; t < args.ntiles && ok && !*fail; t += gridDim.x) {
                const F64Coord c = f64_coord(args, t);
                const int ba = args.a_bcast ? 0 : c.bo, bb = args.b_bcast ? 0 : c.bo;
                for (int i = 0; i < c.nk && ok; ++i) {
                    const int kb = c.k_lo + i;
                    const int bs = (int)(bit & 1);
                    if (bit >= 2 && !mbar_wait_or_fail(&sm.bempty[bs], (uint32_t)(((bit >> 1) - 1) & 1), fail)) {
                        ok = false;
                        break;
                    }
                    mbar_expect_tx(&sm.bfull[bs], (uint32_t)(kSlices * FN * BK * 2));
                    tma_load_slices(sm.b[bs], &tmB, &sm.bfull[bs], c.n0, 0, kb, bb);
                    blast[bs] = bit++;
                    for (int ts = 0; ts < kSlices; ++ts) {
                        if (ait >= FA && !mbar_wait_or_fail(&sm.aempty[as], apar, fail)) {
                            ok = false;
                            break;
                        }
                        mbar_expect_tx(&sm.afull[as], (uint32_t)(BM * BK * 2));
                        tma_load_slices(sm.a[as], &tmA, &sm.afull[as], c.m0, ts, kb, ba);
                        ++ait;
                        if (++as == FA) {
                            as = 0;
                            apar ^= 1u;
                        }
                    }
                }
            }
            // Every load issued has landed before the CTA exits.
            for (int s = 0; s < 2; ++s)
                if (blast[s] >= 0) mbar_wait(&sm.bfull[s], (uint32_t)((blast[s] >> 1) & 1));
            for (int s = 0; s < FA; ++s) {
                // last load into slot s: number (ait - 1 - s) / FA of that slot
                if (ait > s) mbar_wait(&sm.afull[s], (uint32_t)(((ait - 1 - s) / FA) & 1));
            }
        }
    } else if (warp == 1) {
        // MMA issuer.  The whole warp runs the loop and one elected lane
        // issues, so that the descriptors stay in uniform registers (issued
        // from a one-lane branch, every MMA first moved its operands there:
        // 7700 cycles per K step at 4096^3 instead of 6000; testing barriers
        // ahead took it to 5260, of which the tensor pipe works 3580).  Descriptors are stepped by constants (the start-address
        // field counts 16-byte units).
        const uint64_t a0 = smem_desc(smem_u32(sm.a[0]));
        const uint64_t b0 = smem_desc(smem_u32(sm.b[0]));
        constexpr uint64_t kAStep = (uint64_t)(BM * BK * 2) >> 4;
        constexpr uint64_t kBSlice = (uint64_t)(FN * BK * 2) >> 4;
        constexpr uint64_t kKStep = (uint64_t)(UK * 2) >> 4;
        int bs = 0, as = 0;
        uint32_t bpar = 0, apar = 0;
        // usedm bit q: level q has been started before (its next restart
        // waits for the drain), parm = parity of that wait.
        unsigned usedm = 0, parm = 0;
        // Whole-warp wait.  The barrier of the next A slice and of the next
        // B buffer is tested before the MMAs of the current slice are issued
        // (ready), so that a test's latency does not leave the tensor pipe,
        // whose queue holds a few MMAs, without work.
        auto wait_all = [&](bool ready, uint64_t* bar, uint32_t par) {
            if (__all_sync(0xffffffffu, ready)) return true;
            return __all_sync(0xffffffffu, mbar_wait_or_fail(bar, par, fail)) != 0;
        };
        auto wait_levels = [&](unsigned m) {
            bool good = true;
#pragma unroll
            for (int q = 0; q < kLevels; ++q)
                if (good && (m >> q & 1u)) good = wait_all(false, &sm.lempty[q], (parm >> q) & 1u);
            return good;
        };
        bool ok = true, a_ready = false, b_ready = false;
        for (long long t = blockIdx.x; t < args.ntiles && ok; t += gridDim.x) {
            const F64Coord c = f64_coord(args, t);
            for (int i = 0; i < c.nk && ok; ++i) {
                ok = wait_all(b_ready, &sm.bfull[bs], bpar);
                if (!ok) break;
                const unsigned fresh = f64_fresh(i), wait = fresh & usedm;
                usedm |= fresh;
                const int nkk = c.k_lo + i == args.ksteps - 1 ? args.last_kk : BK / UK;
                const uint64_t bbase = b0 + (uint64_t)bs * (kSlices * kBSlice);
                const unsigned drained = f64_drained(i, c.nk);
                b_ready = mbar_test(&sm.bfull[bs ^ 1], bpar ^ (uint32_t)bs);
#pragma unroll
                for (int ts = 1; ts <= kSlices; ++ts) {
                    ok = wait_all(a_ready, &sm.afull[as], apar);
                    if (!ok) break;
                    const int as2 = as + 1 == FA ? 0 : as + 1;
                    const uint32_t apar2 = as + 1 == FA ? apar ^ 1u : apar;
                    const uint64_t ad = a0 + (uint64_t)as * kAStep;
                    // n levels from level q on: B slices u = q + 2 - ts ...
                    auto mma = [&](int kk, int q, int n, uint32_t acc) {
                        mma_bf16(tmem + (uint32_t)(q * FN), ad + kk * kKStep,
                                 bbase + (uint64_t)(q + 1 - ts) * kBSlice + kk * kKStep,
                                 instr_desc(BM, n * FN), acc);
                    };
                    if (ts == 1) {
                        // Every level is first touched by the first slice, and
                        // sub-step 0 restarts the fresh ones (accumulate off).
                        // Levels 4 - 6, drained last in the step before, come
                        // after all of levels 0 - 3 (512 cycles of MMA).
                        ok = wait_levels(wait & 0x0fu);
                        if (!ok) break;
                        a_ready = mbar_test(&sm.afull[as2], apar2);
                        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                        if (elect_one()) {
                            if (i & 3) {              // none of 0 - 3
                                mma(0, 0, 4, 1u);
                            } else if (i & 4) {       // 2, 3
                                mma(0, 0, 2, 1u);
                                mma(0, 2, 2, 0u);
                            } else if (i & 8) {       // 1 - 3
                                mma(0, 0, 1, 1u);
                                mma(0, 1, 3, 0u);
                            } else {                  // all
                                mma(0, 0, 4, 0u);
                            }
#pragma unroll
                            for (int kk = 1; kk < BK / UK; ++kk) {
                                if (kk >= nkk) break;
                                mma(kk, 0, 4, 1u);
                            }
                            if (drained & 1u) mma_commit(&sm.lfull[0]);
                        }
                        __syncwarp();
                        ok = wait_levels(wait & 0x70u);
                        parm ^= wait;
                        if (!ok) break;
                        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                        if (elect_one()) {
                            if (i & 1) {              // none of 4 - 6
                                mma(0, 4, 3, 1u);
                            } else if (i & 2) {       // 4
                                mma(0, 4, 1, 0u);
                                mma(0, 5, 2, 1u);
                            } else if (i & 4) {       // 4, 5
                                mma(0, 4, 2, 0u);
                                mma(0, 6, 1, 1u);
                            } else {                  // all
                                mma(0, 4, 3, 0u);
                            }
#pragma unroll
                            for (int kk = 1; kk < BK / UK; ++kk) {
                                if (kk >= nkk) break;
                                mma(kk, 4, 3, 1u);
                            }
                            mma_commit(&sm.aempty[as]);
                        }
                    } else {
                        a_ready = mbar_test(&sm.afull[as2], apar2);
                        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                        if (elect_one()) {
#pragma unroll
                            for (int kk = 0; kk < BK / UK; ++kk) {
                                if (kk >= nkk) break;
                                if (ts == 2) {
                                    mma(kk, 1, 3, 1u);
                                    mma(kk, 4, 3, 1u);
                                } else if (ts == 3) {
                                    mma(kk, 2, 3, 1u);
                                    mma(kk, 5, 2, 1u);
                                } else {
                                    mma(kk, ts - 1, 8 - ts, 1u);
                                }
                            }
                            mma_commit(&sm.aempty[as]);
                            // level q is complete after slice q + 1
                            if (drained >> (ts - 1) & 1u) mma_commit(&sm.lfull[ts - 1]);
                            if (ts == kSlices) mma_commit(&sm.bempty[bs]);
                        }
                    }
                    __syncwarp();
                    as = as2;
                    apar = apar2;
                }
                if (!ok) break;
                bpar ^= (uint32_t)bs;
                bs ^= 1;
            }
            if (__any_sync(0xffffffffu, *fail != 0)) break;
        }
        // All MMAs issued have completed before TMEM is freed.
        __syncwarp();
        if (elect_one()) {
            mma_commit(&sm.drain);
            mbar_wait(&sm.drain, 0);
        }
        __syncwarp();
    } else {
        // Epilogue: drains and the float64 combination of the tile.
        const int q4 = warp & 3, quarter = (warp - 2) >> 2;
        int* eb = sm.eb[warp - 2];
        unsigned dpar = 0;   // bit q: parity of the next lfull wait of level q
        const bool partial = args.splits > 1;
        // alpha = +-2^k goes into the exponent and the sign
        const bool apow = !partial && args.alpha_exp != kNoPow2;
        const bool general = !partial && (args.beta != 0.0 || !apow);
        const int ebase = (apow ? args.alpha_exp : 0) - 2044 - 46 - args.hshift;
        const unsigned aneg = apow && args.alpha < 0.0 ? 0xffffffffu : 0u;
        for (long long t = blockIdx.x; t < args.ntiles; t += gridDim.x) {
            const F64Coord c = f64_coord(args, t);
            // sums in units of 2^-46 of the product's scale: H + T
            long long H[FC];
            float T[FC];
#pragma unroll
            for (int j = 0; j < FC; ++j) {
                H[j] = 0;
                T[j] = 0.f;
            }
            bool ok = true;
            // K indices that a level collects at most (short products)
            const int kmax = c.k_lo + c.nk == args.ksteps
                                 ? (c.nk - 1) * BK + args.last_kk * UK : c.nk * BK;
            for (int i = 0; i < c.nk && ok; ++i) {
#pragma unroll 1
                for (unsigned todo = f64_drained(i, c.nk); todo != 0; todo &= todo - 1) {
                    const int q = __ffs(todo) - 1;
                    if (!mbar_wait_or_fail(&sm.lfull[q], (dpar >> q) & 1u, fail)) {
                        ok = false;
                        break;
                    }
                    dpar ^= 1u << q;
                    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                    uint32_t r[FC];
                    const uint32_t taddr = tmem + ((uint32_t)(q4 * 32) << 16) +
                                           (uint32_t)(q * FN + quarter * FC);
                    asm volatile(
                        "tcgen05.ld.sync.aligned.32x32b.x16.b32"
                        " {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
                        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                          "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]),
                          "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                        : "r"(taddr));
                    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
                    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&sm.lempty[q]);
                    if (q <= 4 && (q + 1) * kmax <= 256) {
                        // sums of at most 2^22: their integers are the low bits
                        // of S + 1.5 2^23 (the conversion instruction runs on a
                        // pipe of 16 lanes per SM)
                        const long long w = 1LL << (8 * (4 - q));
#pragma unroll
                        for (int j = 0; j < FC; ++j) {
                            const float m = __uint_as_float(r[j]) + 12582912.f;
                            H[j] += (long long)(int)(__float_as_uint(m) - 0x4B400000u) * w;
                        }
                    } else if (q == 0) {
                        // weight 2^32
#pragma unroll
                        for (int j = 0; j < FC; ++j)
                            H[j] += (long long)((unsigned long long)(unsigned)__float2int_rn(
                                                    __uint_as_float(r[j])) << 32);
                    } else if (q <= 4) {
                        const int w = 1 << (8 * (4 - q));
#pragma unroll
                        for (int j = 0; j < FC; ++j)
                            H[j] += (long long)__float2int_rn(__uint_as_float(r[j])) * w;
                    } else {
                        const float w = q == 5 ? 0.00390625f : 0.0000152587890625f;
#pragma unroll
                        for (int j = 0; j < FC; ++j) T[j] = fmaf(__uint_as_float(r[j]), w, T[j]);
                        if (q == 6) {
                            // carry the integer part (|T| < 2^19)
#pragma unroll
                            for (int j = 0; j < FC; ++j) {
                                const float m = T[j] + 12582912.f;
                                H[j] += (int)(__float_as_uint(m) - 0x4B400000u);
                                T[j] -= m - 12582912.f;
                            }
                        }
                    }
                }
            }
            if (!ok) break;
            // C(i, j) = alpha 2^(e_r + e_c - 46) (H + T) [+ beta C]
            const int i = c.m0 + q4 * 32 + lane;
            const int col0 = c.n0 + quarter * FC;
            const int ncols = min(FC, args.N - col0);
            const int fa = i < args.M ? args.eA[(long long)(args.a_bcast ? 0 : c.bo) * args.M + i] : 1;
            const int fb = lane < ncols
                         ? args.eB[(long long)(args.b_bcast ? 0 : c.bo) * args.N + col0 + lane] : 0;
            __syncwarp();
            if (lane < FC) eb[lane] = fb;
            // exponents for which every result is a normal number (all-zero
            // columns and rows give F = 0 and do not count)
            int fmx = fb, fmn = fb > 0 ? fb : 4096;
#pragma unroll
            for (int off = 8; off > 0; off >>= 1) {
                fmx = max(fmx, __shfl_xor_sync(0xffffffffu, fmx, off));
                fmn = min(fmn, __shfl_xor_sync(0xffffffffu, fmn, off));
            }
            fmx = __shfl_sync(0xffffffffu, fmx, 0);
            fmn = __shfl_sync(0xffffffffu, fmn, 0);
            const bool range_ok = fa < 2047 && fmx < 2047 && fa + fmn > 2044 - 700 && fa + fmx < 2044 + 800;
            __syncwarp();
            if (i >= args.M || ncols <= 0) continue;
            f64_finish(H, T, eb, args.hshift, fa, ebase, aneg, range_ok, ncols);
            const int ib = i / args.Mb;
            double* Cr = args.C + (long long)(c.bo + ib) * args.cbs +
                         (partial ? (long long)c.split * args.split_stride : 0) +
                         (long long)(i - ib * args.Mb) * args.crs + (long long)col0 * args.ccs;
            if (general) {
#pragma unroll
                for (int j = 0; j < FC; ++j) {
                    if (j >= ncols) continue;
                    double v = __longlong_as_double(H[j]);
                    if (args.alpha_exp == kNoPow2) v *= args.alpha;
                    double* p = Cr + (long long)j * args.ccs;
                    *p = args.beta != 0.0 ? fma(args.beta, *p, v) : v;
                }
            } else if (args.ccs == 1 && ncols == FC && (reinterpret_cast<uintptr_t>(Cr) & 15) == 0) {
#pragma unroll
                for (int j = 0; j < FC; j += 2)
                    *reinterpret_cast<longlong2*>(Cr + j) = make_longlong2(H[j], H[j + 1]);
            } else if (ncols == FC) {
#pragma unroll
                for (int j = 0; j < FC; ++j) Cr[(long long)j * args.ccs] = __longlong_as_double(H[j]);
            } else {
#pragma unroll
                for (int j = 0; j < FC; ++j)
                    if (j < ncols) Cr[(long long)j * args.ccs] = __longlong_as_double(H[j]);
            }
        }
    }
    __syncthreads();
    if (sm.fail && threadIdx.x == 0) atomicExch(args.err, 1);
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem),
                     "r"(512));
}

// C = beta C + alpha sum_split part[split] (float64 split-K partials of the
// fused kernel; element (b, i, j) at part[(split nbo + b) M N + e], e = i N + j
// or, i_fast, j M + i: the index that runs along C's rows).
__global__ void k_f64_splitsum(const double* part, int splits, int nbo, int M, int N, int i_fast,
                               double* C, long long crs, long long ccs, long long cbs,
                               double alpha, double beta) {
    grid_wait();
    const long long MN = (long long)M * N, tot = MN * nbo;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < tot;
         e += (long long)gridDim.x * blockDim.x) {
        const int b = (int)(e / MN);
        const long long r = e % MN;
        const int i = (int)(i_fast ? r % M : r / N), j = (int)(i_fast ? r / M : r % N);
        double s = 0.0;
        for (int sp = 0; sp < splits; ++sp) s += part[(long long)sp * tot + e];
        double* p = C + (long long)b * cbs + (long long)i * crs + (long long)j * ccs;
        *p = (beta != 0.0 ? beta * *p : 0.0) + alpha * s;
    }
}

// Workspace a product takes in one piece.
struct F64Need {
    long long slices, expo, Ktot;
};

F64Need f64_need(const Gemm<double>& g) {
    const long long nbo = g.reduce ? 1 : g.batch;
    const long long Ktot = f64_ktot(g.K, g.batch, g.reduce);
    const long long nba = !g.reduce && g.batch > 1 && g.sAb == 0 ? 1 : nbo;
    const long long nbb = !g.reduce && g.batch > 1 && g.sBb == 0 ? 1 : nbo;
    const long long rows = g.M * nba + g.N * nbb;
    return F64Need{rows * kSlices * rup(Ktot, BK), rows, Ktot};
}

// A K above kMaxSteps steps has to be split, which takes partials.
bool f64_k_fits(const Gemm<double>& g, const F64TcWorkspace& ws) {
    const long long steps = (f64_need(g).Ktot + BK - 1) / BK;
    const long long sp = (steps + kMaxSteps - 1) / kMaxSteps;
    const long long outputs = (long long)g.M * g.N * (g.reduce ? 1 : g.batch);
    return sp <= 1 || (sp <= 32 && (size_t)(outputs * sp) <= ws.part_elems / 2);
}

bool f64_fits(const Gemm<double>& g, const F64TcWorkspace& ws) {
    const F64Need n = f64_need(g);
    return (size_t)n.slices <= ws.slice_elems && (size_t)n.expo <= ws.expo_elems &&
           n.Ktot <= INT32_MAX - BK;
}

cudaError_t gemm_f64_tc_one(const Gemm<double>& g, const F64TcWorkspace& ws, cudaStream_t s);

}  // namespace

// A product whose slices do not fit the workspace is cut into pieces that
// do: batches first (a batch-reduced product accumulates its later pieces
// into C with beta = 1), then the rows or the columns of C, whichever are
// more, in halves rounded to the 128-row tile.  A K too long for one tile's
// sums is cut in halves too when its split-K partials do not fit.
cudaError_t gemm_f64_tc(const Gemm<double>& g, const F64TcWorkspace& ws, cudaStream_t s) {
    if (g.M <= 0 || g.N <= 0 || g.batch <= 0) return cudaSuccess;
    const bool k_fits = f64_k_fits(g, ws);
    if (k_fits && f64_fits(g, ws)) return gemm_f64_tc_one(g, ws, s);
    Gemm<double> g1 = g, g2 = g;
    if (g.batch > 1 && (g.reduce || !f64_fits(g, ws))) {
        const int b1 = g.batch / 2;
        g1.batch = b1;
        g2.batch = g.batch - b1;
        g2.A.p = g.A.p + (long long)b1 * g.sAb;
        g2.B.p = g.B.p + (long long)b1 * g.sBb;
        if (g.reduce) {
            g2.beta = 1.0;
        } else {
            g2.C = g.C + (long long)b1 * g.sCb;
        }
    } else if (!k_fits && g.K > 2 * BK) {
        const int k1 = (int)rup((g.K + 1) / 2, BK);
        g1.K = k1;
        g2.K = g.K - k1;
        g2.A.p = g.A.p + (long long)k1 * g.A.cs;
        g2.B.p = g.B.p + (long long)k1 * g.B.rs;
        g2.beta = 1.0;
    } else if (g.M >= g.N && g.M > BM) {
        const int m1 = (int)rup((g.M + 1) / 2, BM);
        g1.M = m1;
        g2.M = g.M - m1;
        g2.A.p = g.A.p + (long long)m1 * g.A.rs;
        g2.C = g.C + (long long)m1 * g.ldc;
    } else if (g.N > BM) {
        const int n1 = (int)rup((g.N + 1) / 2, BM);
        g1.N = n1;
        g2.N = g.N - n1;
        g2.B.p = g.B.p + (long long)n1 * g.B.cs;
        g2.C = g.C + n1;
    } else {
        return cudaErrorMemoryAllocation;   // a single tile row and column do not fit
    }
    cudaError_t e = gemm_f64_tc(g1, ws, s);
    if (e != cudaSuccess) return e;
    return gemm_f64_tc(g2, ws, s);
}

namespace {

cudaError_t gemm_f64_tc_one(const Gemm<double>& g, const F64TcWorkspace& ws, cudaStream_t s) {
    cudaError_t e = get_encode();
    if (e != cudaSuccess) return e;
    const int nb = g.batch;
    const int nbo = g.reduce ? 1 : nb;
    // The larger side takes the 128-row tiles; if one operand is shared by
    // every batch, the rows of all batches of the other one, as one list:
    // otherwise every batch has a ragged tile (131 rows fill two tiles of 128
    // to a half, 200 and 400 rows 0.78 of theirs).
    const bool m_bc = !g.reduce && nb > 1 && g.sAb == 0, n_bc = !g.reduce && nb > 1 && g.sBb == 0;
    const bool flat = m_bc != n_bc && (long long)nb * (m_bc ? g.N : g.M) < INT32_MAX - BM;
    const bool swap = flat ? m_bc : g.N > g.M;
    const int Mr = swap ? g.N : g.M, Nr = swap ? g.M : g.N;
    const long long Kp = rup(std::max(g.K, 1), 8);
    const long long Ktot = f64_ktot(g.K, nb, g.reduce);
    View<double> va = g.A, vb{g.B.p, g.B.cs, g.B.rs};
    long long sa = g.sAb, sb = g.sBb;
    if (swap) {
        std::swap(va, vb);
        std::swap(sa, sb);
    }
    const bool a_bc = !g.reduce && nb > 1 && sa == 0;
    const bool b_bc = !g.reduce && nb > 1 && sb == 0;
    const int nba = a_bc ? 1 : nbo, nbb = b_bc ? 1 : nbo;
    const long long sliceA = (long long)Mr * kSlices * rup(Ktot, BK) * nba;
    const int rowsA = flat ? nb * Mr : Mr, tilesets = flat ? 1 : nbo;
    const int mblocks = (int)cdiv(rowsA, BM), nblocks = (int)cdiv(Nr, FN);
    const long long tiles = (long long)mblocks * nblocks * tilesets;
    const int ksteps = (int)((Ktot + BK - 1) / BK);
    const long long sms = device_sms();
    const int splits = f64_splits(tiles, ksteps, (long long)Mr * Nr * nbo, ws.part_elems, sms);

    __nv_bfloat16* slA = ws.slices;
    __nv_bfloat16* slB = ws.slices + sliceA;
    int* eA = ws.expo;
    int* eB = ws.expo + (long long)Mr * nba;
    // Row exponents and slices of both operands.
    SlicePair p{};
    p.op[0] = SliceOp{va.p, va.rs, va.cs, sa, Mr, a_bc ? 1 : nb, flat ? 1 : 0, slA, eA};
    p.op[1] = SliceOp{vb.p, vb.rs, vb.cs, sb, Nr, b_bc ? 1 : nb, 0, slB, eB};
    p.Kd = g.K;
    p.Kp = (int)Kp;
    p.Ktot = Ktot;
    p.reduce = g.reduce ? 1 : 0;
    const bool fused = !g.reduce && g.K <= kFusedK;
    const long long kt = fused ? 1 : cdiv(Kp, PK_K);
    long long blocks[2];
    for (int i = 0; i < 2; ++i)
        blocks[i] = kt * cdiv(p.op[i].R, fused ? SR : PK_R) * p.op[i].nb;
    if (blocks[0] + blocks[1] > INT32_MAX) return cudaErrorInvalidValue;
    p.blocks0 = blocks[0];
    const unsigned sgrid = (unsigned)(blocks[0] + blocks[1]);
    if (fused) {
        const int sbytes = SR * row_pitch((int)rup(Kp, 16)) * (int)sizeof(double);
        if ((e = smem_optin((const void*)k_slice_rows, SR * row_pitch(kFusedK) * (int)sizeof(double))) !=
            cudaSuccess)
            return e;
        launch_chained(k_slice_rows, sgrid, 256, sbytes, s, p);
        count_launches(1);
    } else {
        if ((e = cudaMemsetAsync(ws.expo, 0,
                                 sizeof(int) * ((long long)Mr * nba + (long long)Nr * nbb), s)) !=
            cudaSuccess)
            return e;
        launch_chained(k_row_exp, sgrid, 256, 0, s, p);
        launch_chained(k_slice64, sgrid, 256, 0, s, p);
        count_launches(2);
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const bool redo = ws.redo && nb == 1;
    // (a sixteenth of the outputs at most: the rest of the product is then worth it)
    const int redo_cap = g.beta != 0.0 ? 0
                       : (int)std::min<long long>(ws.redo_cap, (long long)Mr * Nr / 16);
    if (redo) {
        const long long grid = (long long)cdiv(Mr, 32) * cdiv(Nr, 32);
        if (grid > INT32_MAX) return cudaErrorInvalidValue;
        if ((e = cudaMemsetAsync(ws.redo, 0, sizeof(int), s)) != cudaSuccess) return e;
        launch_chained(k_slices_even, (unsigned)grid, 256, 0, s, slA, slB, Mr, Nr, g.K, eA, eB,
                       ws.redo, ws.redo_list, redo_cap);
        count_launches(1);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    CUtensorMap mA, mB;
    if ((e = make_map_slices(&mA, slA, ksteps, rowsA, flat ? 1 : nba, BM, 1)) != cudaSuccess) return e;
    if ((e = make_map_slices(&mB, slB, ksteps, Nr, nbb, FN, kSlices)) != cudaSuccess) return e;
    F64Args a{};
    a.M = rowsA;
    a.N = Nr;
    a.Mb = Mr;
    a.nbo = tilesets;
    a.mblocks = mblocks;
    a.nblocks = nblocks;
    a.ksteps = ksteps;
    a.last_kk = (int)((Ktot - (long long)(ksteps - 1) * BK + UK - 1) / UK);
    a.splits = splits;
    a.ntiles = tiles * splits;
    a.a_bcast = a_bc ? 1 : 0;
    a.b_bcast = b_bc ? 1 : 0;
    a.eA = eA;
    a.eB = eB;
    a.alpha = g.alpha;
    a.beta = g.beta;
    {
        int k = 0;
        const double m = std::frexp(std::fabs(g.alpha), &k);   // 0.5 for a power of two
        a.alpha_exp = m == 0.5 && k > -60 && k < 60 ? k - 1 : kNoPow2;
    }
    {
        // |H| <= 2^46 per K index: as many fractional bits as leave |F| < 2^62
        const long long kmax = (long long)((ksteps + splits - 1) / splits) * BK;
        int lg = 0;
        while ((1LL << lg) < kmax) ++lg;
        a.hshift = std::max(0, std::min(16, 16 - lg));
    }
    a.err = ws.err;
    // accumulator (i, j) is C's (m, n), or (n, m) when the operands were swapped
    const long long crs = swap ? 1 : g.ldc, ccs = swap ? g.ldc : 1;
    const long long cbs = g.reduce ? 0 : g.sCb;
    double* part = reinterpret_cast<double*>(ws.part);
    if (splits > 1) {
        a.C = part;
        a.crs = swap ? 1 : Nr;
        a.ccs = swap ? Mr : 1;
        a.cbs = (long long)Mr * Nr;
        a.split_stride = a.cbs * nbo;
    } else {
        a.C = g.C;
        a.crs = crs;
        a.ccs = ccs;
        a.cbs = cbs;
    }
    const int smem = (int)sizeof(F64Smem) + 1024;
    if ((e = smem_optin((const void*)k_gemm_f64s, smem)) != cudaSuccess) return e;
    const unsigned grid = (unsigned)std::min<long long>(a.ntiles, sms);
    launch_chained(k_gemm_f64s, grid, kF64Threads, smem, s, mA, mB, a);
    count_launches(1);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (splits > 1) {
        const long long tot = (long long)Mr * Nr * nbo;
        const unsigned blocks = (unsigned)std::min<long long>((tot + 255) / 256, sms * 16);
        launch_chained(k_f64_splitsum, blocks, 256, 0, s, part, splits, nbo, Mr, Nr, swap ? 1 : 0,
                       g.C, crs, ccs, cbs, g.alpha, g.beta);
        count_launches(1);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    if (redo) {
        launch_chained(k_redo64, (unsigned)sms, 256, 0, s, va.p, va.rs, va.cs, vb.p, vb.rs, vb.cs,
                       g.K, g.alpha, g.C, crs, ccs, ws.redo, ws.redo_list, redo_cap);
        count_launches(1);
        e = cudaGetLastError();
    }
    return e;
}

}  // namespace

// ---------------------------------------------------------------------------
// Randomised self-test: tensor-core products against the CUDA-core products
// of the same float32 operands over random shapes, orientations, batch modes
// (separate, shared operand, batch-reduced), split-K and beta.
namespace {

unsigned long long st_next(unsigned long long& s) {
    s ^= s << 13;
    s ^= s >> 7;
    s ^= s << 17;
    return s;
}

__global__ void k_fill_uniform(float* p, long long n, unsigned long long seed) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        unsigned long long z = seed + 0x9E3779B97F4A7C15ULL * (unsigned long long)(i + 1);
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
        z ^= z >> 31;
        p[i] = (float)((double)(z >> 11) * (1.0 / 9007199254740992.0)) - 0.5f;
    }
}

__global__ void k_max_abs_diff(const float* a, const float* b, long long n, float* out) {
    float m = 0.f, s = 0.f;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        m = fmaxf(m, fabsf(a[i] - b[i]));
        s = fmaxf(s, fabsf(b[i]));
    }
    for (int o = 16; o > 0; o >>= 1) {
        m = fmaxf(m, __shfl_down_sync(0xffffffffu, m, o));
        s = fmaxf(s, __shfl_down_sync(0xffffffffu, s, o));
    }
    if ((threadIdx.x & 31) == 0) {
        atomicMax(reinterpret_cast<int*>(out), __float_as_int(m));
        atomicMax(reinterpret_cast<int*>(out + 1), __float_as_int(s));
    }
}

}  // namespace

cudaError_t gemm_tc_selftest(int cases, unsigned long long seed, double* max_rel,
                             int* failures, cudaStream_t st) {
    *max_rel = 0;
    *failures = 0;
    const long long cap = 1LL << 22;   // elements per operand buffer
    float *A = nullptr, *B = nullptr, *C1 = nullptr, *C2 = nullptr, *red = nullptr, *simt = nullptr;
    TcWorkspace ws{};
    cudaError_t e = cudaSuccess;
    auto al = [&](void** p, size_t bytes) {
        if (e == cudaSuccess) e = cudaMalloc(p, bytes);
    };
    al((void**)&A, cap * 4);
    al((void**)&B, cap * 4);
    al((void**)&C1, cap * 4);
    al((void**)&C2, cap * 4);
    al((void**)&red, 8);
    al((void**)&simt, cap * 4);
    ws.elems = (size_t)1 << 25;
    al((void**)&ws.buf, ws.elems * 2);
    ws.partial_elems = (size_t)1 << 24;
    al((void**)&ws.partial, ws.partial_elems * 4);
    al((void**)&ws.err, 4);
    if (e == cudaSuccess) e = cudaMemsetAsync(ws.err, 0, 4, st);
    unsigned long long s = seed * 2654435761ULL + 1;
    for (int c = 0; c < cases && e == cudaSuccess; ++c) {
        Gemm<float> g;
        g.M = 1 + (int)(st_next(s) % 700);
        g.N = 1 + (int)(st_next(s) % 700);
        g.K = 1 + (int)(st_next(s) % 900);
        g.batch = 1 + (int)(st_next(s) % 4);
        const int mode = (int)(st_next(s) % 4);   // 0 separate, 1 shared A, 2 shared B, 3 reduce
        if (c % 3 == 2) {   // rows that take wide loads and stores
            g.M = (g.M + 7) / 8 * 8;
            g.N = (g.N + 7) / 8 * 8;
            g.K = (g.K + 3) / 4 * 4;
        }
        g.reduce = mode == 3 && g.batch > 1;
        const bool ta = st_next(s) & 1, tb = st_next(s) & 1;
        const int nprod = (st_next(s) % 3 == 0) ? 1 : 3;
        g.beta = (st_next(s) & 1) ? 0.5 : 0.0;
        // a general alpha and powers of two
        g.alpha = (c & 1) ? 1.25 : ((c & 2) ? -0.5 : 2.0);
        while ((long long)g.batch * g.M * g.K > cap || (long long)g.batch * g.K * g.N > cap ||
               (long long)g.batch * g.M * g.N > cap)
            g.K = std::max(1, g.K / 2), g.M = std::max(1, g.M * 3 / 4);
        const long long sa = (long long)g.M * g.K, sb = (long long)g.K * g.N,
                        sc = (long long)g.M * g.N;
        g.A = ta ? View<float>{A, 1, g.M} : View<float>{A, g.K, 1};
        g.B = tb ? View<float>{B, 1, g.K} : View<float>{B, g.N, 1};
        g.sAb = mode == 1 ? 0 : sa;
        g.sBb = mode == 2 ? 0 : sb;
        g.ldc = g.N;
        g.sCb = sc;
        const long long nC = (g.reduce ? 1 : g.batch) * sc;
        k_fill_uniform<<<256, 256, 0, st>>>(A, g.batch * sa, st_next(s));
        k_fill_uniform<<<256, 256, 0, st>>>(B, g.batch * sb, st_next(s));
        k_fill_uniform<<<256, 256, 0, st>>>(C1, nC, st_next(s));
        count_launches(3);
        if ((e = cudaMemcpyAsync(C2, C1, nC * 4, cudaMemcpyDeviceToDevice, st))) break;
        Gemm<float> h = g;
        g.C = C1;
        h.C = C2;
        h.ws = simt;
        h.ws_elems = cap;
        if ((e = gemm_tc(g, ws, nprod, st))) break;
        if ((e = gemm_simt(h, st))) break;
        if ((e = cudaMemsetAsync(red, 0, 8, st))) break;
        k_max_abs_diff<<<256, 256, 0, st>>>(C1, C2, nC, red);
        count_launches(1);
        float hr[2] = {0, 0};
        int herr = 0;
        if ((e = cudaMemcpyAsync(hr, red, 8, cudaMemcpyDeviceToHost, st))) break;
        if ((e = cudaMemcpyAsync(&herr, ws.err, 4, cudaMemcpyDeviceToHost, st))) break;
        if ((e = cudaStreamSynchronize(st))) break;
        // bf16x3: about 3 x 2^-17 per product, float32 sums over K terms;
        // bf16x1: 2^-8 per factor
        const double scale = std::max(1.0f, hr[1]);
        const double rel = hr[0] / scale;
        const double bound = (nprod == 3 ? 2e-5 : 2e-2) * std::sqrt((double)g.K + 1) *
                             (g.reduce ? std::sqrt((double)g.batch) : 1.0);
        *max_rel = std::max(*max_rel, nprod == 3 ? rel : 0.0);
        if (herr || !(rel <= bound)) ++*failures;
    }
    for (void* p : {(void*)A, (void*)B, (void*)C1, (void*)C2, (void*)red, (void*)simt,
                    (void*)ws.buf, (void*)ws.partial, (void*)ws.err})
        if (p) cudaFree(p);
    return e;
}

namespace {

__global__ void k_fill_uniform64(double* p, long long n, unsigned long long seed, int spread) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        unsigned long long z = seed + 0x9E3779B97F4A7C15ULL * (unsigned long long)(i + 1);
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
        z ^= z >> 31;
        double v = (double)(z >> 11) * (1.0 / 9007199254740992.0) - 0.5;
        // spread > 0: magnitudes over 2^-spread .. 1 (rows with a wide range)
        if (spread > 0) v = scalbn(v, -(int)((z >> 3) % (unsigned long long)(spread + 1)));
        p[i] = v;
    }
}

__global__ void k_max_abs_diff64(const double* a, const double* b, long long n, double* out) {
    double m = 0.0, s = 0.0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        m = fmax(m, fabs(a[i] - b[i]));
        s = fmax(s, fabs(b[i]));
    }
    for (int o = 16; o > 0; o >>= 1) {
        m = fmax(m, __shfl_down_sync(0xffffffffu, m, o));
        s = fmax(s, __shfl_down_sync(0xffffffffu, s, o));
    }
    if ((threadIdx.x & 31) == 0) {
        // non-negative doubles order like their bit patterns
        atomicMax(reinterpret_cast<unsigned long long*>(out), (unsigned long long)__double_as_longlong(m));
        atomicMax(reinterpret_cast<unsigned long long*>(out + 1), (unsigned long long)__double_as_longlong(s));
    }
}

}  // namespace

cudaError_t gemm_f64_tc_selftest(int cases, unsigned long long seed, double* max_rel,
                                 int* failures, cudaStream_t st) {
    *max_rel = 0;
    *failures = 0;
    const long long cap = 1LL << 21;   // elements per operand buffer
    double *A = nullptr, *B = nullptr, *C1 = nullptr, *C2 = nullptr, *red = nullptr, *simt = nullptr;
    F64TcWorkspace ws{};
    cudaError_t e = cudaSuccess;
    auto al = [&](void** p, size_t bytes) {
        if (e == cudaSuccess) e = cudaMalloc(p, bytes);
    };
    al((void**)&A, cap * 8);
    al((void**)&B, cap * 8);
    al((void**)&C1, cap * 8);
    al((void**)&C2, cap * 8);
    al((void**)&red, 16);
    al((void**)&simt, cap * 8);
    ws.slice_elems = (size_t)1 << 26;
    al((void**)&ws.slices, ws.slice_elems * 2);
    ws.part_elems = (size_t)64 * cap;   // 32 float64 split-K sums of the largest output
    al((void**)&ws.part, ws.part_elems * 4);
    ws.expo_elems = (size_t)1 << 16;
    al((void**)&ws.expo, ws.expo_elems * 4);
    al((void**)&ws.err, 4);
    if (e == cudaSuccess) e = cudaMemsetAsync(ws.err, 0, 4, st);
    unsigned long long s = seed * 2654435761ULL + 7;
    for (int c = 0; c < cases && e == cudaSuccess; ++c) {
        Gemm<double> g;
        g.M = 1 + (int)(st_next(s) % 600);
        g.N = 1 + (int)(st_next(s) % 600);
        g.K = 1 + (int)(st_next(s) % 2600);    // up to three exact K chunks
        // every fourth case at the edges of the tiles, K steps and sub-steps
        // and of the levels' drain periods
        if (c % 4 == 3) {
            const int mn[8] = {1, 16, 17, 63, 64, 65, 128, 129};
            const int kk[10] = {1, 8, 16, 17, 48, 64, 65, 129, 1024, 1025};
            g.M = mn[st_next(s) % 8] + (int)(st_next(s) % 2) * 128;
            g.N = mn[st_next(s) % 8];
            g.K = kk[st_next(s) % 10];
        }
        g.batch = 1 + (int)(st_next(s) % 4);
        const int mode = (int)(st_next(s) % 4);   // 0 separate, 1 shared A, 2 shared B, 3 reduce
        g.reduce = mode == 3 && g.batch > 1;
        const bool ta = st_next(s) & 1, tb = st_next(s) & 1;
        const int spread = (st_next(s) % 3 == 0) ? 40 : 0;
        g.beta = (st_next(s) & 1) ? 0.5 : 0.0;
        // a general alpha and powers of two
        g.alpha = (c & 1) ? 1.25 : ((c & 2) ? -0.5 : 2.0);
        while ((long long)g.batch * g.M * g.K > cap || (long long)g.batch * g.K * g.N > cap ||
               (long long)g.batch * g.M * g.N > cap)
            g.K = std::max(1, g.K / 2), g.M = std::max(1, g.M * 3 / 4);
        const long long sa = (long long)g.M * g.K, sb = (long long)g.K * g.N,
                        sc = (long long)g.M * g.N;
        g.A = ta ? View<double>{A, 1, g.M} : View<double>{A, g.K, 1};
        g.B = tb ? View<double>{B, 1, g.K} : View<double>{B, g.N, 1};
        g.sAb = mode == 1 ? 0 : sa;
        g.sBb = mode == 2 ? 0 : sb;
        g.ldc = g.N;
        g.sCb = sc;
        const long long nC = (g.reduce ? 1 : g.batch) * sc;
        k_fill_uniform64<<<256, 256, 0, st>>>(A, g.batch * sa, st_next(s), spread);
        k_fill_uniform64<<<256, 256, 0, st>>>(B, g.batch * sb, st_next(s), spread);
        k_fill_uniform64<<<256, 256, 0, st>>>(C1, nC, st_next(s), 0);
        count_launches(3);
        if ((e = cudaMemcpyAsync(C2, C1, nC * 8, cudaMemcpyDeviceToDevice, st))) break;
        Gemm<double> h = g;
        g.C = C1;
        h.C = C2;
        h.ws = simt;
        h.ws_elems = cap;
        // Every third case gets a third of the slice workspace it needs, so
        // that the product is cut into pieces.
        F64TcWorkspace wsc = ws;
        if (c % 3 == 2) {
            const long long Kp = rup(std::max(g.K, 1), BK);
            wsc.slice_elems = (size_t)std::max<long long>(f64_need(g).slices / 3,
                                                          2LL * BM * kSlices * Kp);
        }
        if ((e = gemm_f64_tc(g, wsc, st))) break;
        if ((e = gemm_simt(h, st))) break;
        if ((e = cudaMemsetAsync(red, 0, 16, st))) break;
        k_max_abs_diff64<<<256, 256, 0, st>>>(C1, C2, nC, red);
        count_launches(1);
        double hr[2] = {0, 0};
        int herr = 0;
        if ((e = cudaMemcpyAsync(hr, red, 16, cudaMemcpyDeviceToHost, st))) break;
        if ((e = cudaMemcpyAsync(&herr, ws.err, 4, cudaMemcpyDeviceToHost, st))) break;
        if ((e = cudaStreamSynchronize(st))) break;
        // Both sides are float64-accurate: a few units of 2^-53 times the
        // size of the sums (K terms of up to 1/4, and beta C).
        const double scale = std::max(1.0, hr[1]);
        const double rel = hr[0] / scale;
        const double bound = 1e-15 * ((double)g.K * (g.reduce ? g.batch : 1) + 1);
        *max_rel = std::max(*max_rel, rel);
        if (herr || !(rel <= bound)) ++*failures;
    }
    for (void* p : {(void*)A, (void*)B, (void*)C1, (void*)C2, (void*)red, (void*)simt,
                    (void*)ws.slices, (void*)ws.part, (void*)ws.expo, (void*)ws.err})
        if (p) cudaFree(p);
    return e;
}

}  // namespace thc

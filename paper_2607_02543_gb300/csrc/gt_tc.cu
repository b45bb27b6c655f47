// Exact k nearest live nodes with a tensor-core candidate pass.
//
// Recall@10 (Sec. 5.2) needs the exact top-k over the live set; for the
// 1M x 128 churn workload that is a 10k x 1M x 128 dense contraction per
// round.  The contraction runs on the 5th-generation tensor cores:
//
//   1. gt_prep_rows / gt_prep_queries write bf16 copies of the live rows and
//      the queries (x = hi + lo + e with hi, lo bf16; both as [hi | lo], each
//      segment padded to 64) and the norms an error bound needs.  When every
//      lo is zero (data exactly representable in bf16, e.g. integers up to
//      256) K runs over hi.hi only, otherwise over hi.hi + hi.lo + lo.hi.
//   2. gt_tc_kernel: persistent CTAs; TMA (cp.async.bulk.tensor, 128-byte
//      swizzle) streams 256-row boxes of the row copy through a shared
//      memory ring while the query tile stays resident (or, when the query
//      tile's K does not fit shared memory, travels through the ring beside
//      each row box, one 64-column block at a time); one thread issues
//      tcgen05.mma (M = 128, N = 256, bf16 -> fp32) into a double-buffered TMEM
//      accumulator; eight epilogue warps read it with tcgen05.ld and write,
//      per query and per block of 32 rows, the smallest approximate key
//      key = |x|^2 - 2 q.x (L2) or -q.x (IP); dead rows have key +inf.
//      For few wide rows it writes every key too.
//   3. gt_rerank_kernel: every row of the k blocks with the smallest minima
//      is scored with the canonical fp32 distance (the same definition the
//      rest of the index uses).  The k-th of these distances bounds the
//      answer: an a-priori bound E on |approximate - canonical| turns it into
//      a threshold T on approximate keys that no row of the top k can exceed,
//      and the rows of the remaining blocks with a minimum <= T are scored
//      too (where every key is at hand, only the rows with a key that passes).  So the result is always the exact top-k with canonical
//      distances, ties by smaller id.  Queries without a finite threshold
//      (infinities or NaN in the data), or whose T admits more than half of
//      all blocks, go to the CUDA-core exact kernel.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>

#include <mutex>

#include "common.cuh"
#include "internal.h"

namespace etale {
namespace {

constexpr int TC_ROWS = 128;                      // MMA M: queries per query sub-tile
constexpr int TC_ACC = 256;                       // TMEM columns per accumulator buffer
constexpr int TC_KBOX = 64;                       // bf16 per 128-byte swizzle row
constexpr u32 TC_BOX = TC_ROWS * TC_KBOX * 2;     // 16 KB per 128-row TMA box
// Tile shape: 128 queries against 256 rows, one 256-column accumulator: 96 B of
// operands from shared memory per MMA cycle of the SM's 128.  Two query tiles
// against 128 rows read half as many rows from L2, but 128 B: 2,050 against
// 1,690 cycles a tile (300k x 128 rows, 10k queries).
constexpr int TC_MAX_STAGES = 12;
constexpr int TC_XS = 4;                          // key-base ring slots (one tile's bases each)
constexpr u32 TC_STATIC = 5 * 1024;               // static shared memory of the kernel, rounded up
constexpr int TC_EPI_WARPS = 8;
constexpr int TC_THREADS = (2 + TC_EPI_WARPS) * 32;
constexpr u32 ORD_INF = 0xFF800000u;              // f2ord(+inf)
// kind::f16 instruction descriptor: fp32 accumulator (bits 4-5 = 1), A and B
// bf16 (bits 7-9 = 1, 10-12 = 1), both K-major, N >> 3 at bit 17, M >> 4 at 24
__host__ __device__ constexpr u32 tc_idesc(u32 n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((n >> 3) << 17) | ((u32)(TC_ROWS >> 4) << 24);
}

struct TcArgs {
    u32 nq, n_tiles, kblocks, bn, m_tiles, chunks, tiles_per_chunk, stages;
    u32 seg;              // column blocks of one segment: K runs over hi.hi, hi.lo, lo.hi (see a_col, b_col)
    u32 all_keys;         // 0: smallest key per block of 32 rows; 1: every key; 2: both, the keys in `keys`
    u32 stream_a;         // 1: the query boxes travel through the ring (selects gt_tc_kernel<true>)
    const u32 *nq_dev;    // when set, the batch size is read here (nq is its cap); later query tiles are skipped
    u32 ld;               // row length of the output (blocks or keys)
    float s;              // -2 (L2) or -1 (IP)
    const float *xn;      // n_tiles * bn key bases (+inf for dead rows and padding)
    float *out;           // nq x ld
    float *keys;          // all_keys 2: (n_tiles * bn / 32) x nq x 32, a block's keys for a query on one line
    u32 *err;
};

// ---- PTX wrappers -----------------------------------------------------------
__device__ __forceinline__ void mbar_arrive(u64 *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, int x, int y, u64 *bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(smem_addr(dst)), "l"(map), "r"(x), "r"(y), "r"(smem_addr(bar))
        : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// Shared-memory matrix descriptor of a K-major operand in the 128-byte swizzle
// layout: rows of 128 bytes, 8-row groups 1024 bytes apart (stride byte
// offset), descriptor version 1 (bit 46), swizzle mode 2 (bits 61-63).
__device__ __forceinline__ u64 sw128_desc(u32 saddr) {
    return (u64)((saddr & 0x3FFFFu) >> 4) | ((u64)1 << 16) | ((u64)(1024 >> 4) << 32) | ((u64)1 << 46) |
           ((u64)2 << 61);
}
// mbar_wait by a whole warp, converged afterwards: no lane may run ahead of the
// others' waits (a lane two phases behind would wait for a phase that is over),
// and the issuing instructions read their operands for the warp.
__device__ __forceinline__ bool warp_wait(u64 *bar, u32 parity) {
    return __all_sync(FULL, mbar_wait(bar, parity, WAIT_LIMIT));
}
// One lane of a converged warp (the same one at every call).
__device__ __forceinline__ u32 elect_one() {
    u32 p;
    asm volatile("{\n .reg .pred q;\n elect.sync _|q, 0xffffffff;\n selp.u32 %0, 1, 0, q;\n}" : "=r"(p));
    return p;
}
// Run by a whole warp, issued by the lane with `leader` set.
__device__ __forceinline__ void tc_mma(u32 d, u64 a, u64 b, u32 idesc, u32 acc, u32 leader) {
    asm volatile(
        "{\n .reg .pred p, e;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 e, %5, 0;\n"
        " @e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc), "r"(leader)
        : "memory");
}
__device__ __forceinline__ void tc_commit(u64 *bar, u32 leader) {
    asm volatile(
        "{\n .reg .pred e;\n setp.ne.b32 e, %1, 0;\n"
        " @e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}" ::"r"(smem_addr(bar)),
        "r"(leader)
        : "memory");
}
// 64 consecutive TMEM columns of this warp's 32 lanes; completes at tmem_wait().
__device__ __forceinline__ void tmem_ld64(u32 taddr, u32 *r) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x64.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32, %33, %34, %35, %36, %37, %38, %39, %40, %41, %42, %43, %44, %45, %46, %47, %48, %49, %50, %51, %52, %53, %54, %55, %56, %57, %58, %59, %60, %61, %62, %63}, [%64];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31]), "=r"(r[32]), "=r"(r[33]), "=r"(r[34]), "=r"(r[35]), "=r"(r[36]), "=r"(r[37]), "=r"(r[38]), "=r"(r[39]), "=r"(r[40]), "=r"(r[41]), "=r"(r[42]), "=r"(r[43]), "=r"(r[44]), "=r"(r[45]), "=r"(r[46]), "=r"(r[47]), "=r"(r[48]), "=r"(r[49]), "=r"(r[50]), "=r"(r[51]), "=r"(r[52]), "=r"(r[53]), "=r"(r[54]), "=r"(r[55]), "=r"(r[56]), "=r"(r[57]), "=r"(r[58]), "=r"(r[59]), "=r"(r[60]), "=r"(r[61]), "=r"(r[62]), "=r"(r[63])
                 : "r"(taddr));
}
// Both halves of a register pair at once (the same roundings as two fmaf),
// and the smallest of three.
__device__ __forceinline__ u64 pair32(u32 lo, u32 hi) { return ((u64)hi << 32) | lo; }
__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c) {
    u64 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ float min3(float a, float b, float c) {
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
// 32 bytes, one sector a lane
__device__ __forceinline__ void st_global32(float *p, u64 a, u64 b, u64 c, u64 d) {
    asm volatile("st.global.v4.b64 [%0], {%1, %2, %3, %4};" ::"l"(p), "l"(a), "l"(b), "l"(c), "l"(d) : "memory");
}
__device__ __forceinline__ float pair_lo(u64 v) { return __uint_as_float((u32)v); }
__device__ __forceinline__ float pair_hi(u64 v) { return __uint_as_float((u32)(v >> 32)); }
__device__ __forceinline__ void tmem_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Column block of the query copy [hi | lo] and of the row copy [hi | lo] at step
// kb of K: hi hi lo against hi lo hi.
__device__ __forceinline__ u32 a_col(u32 kb, u32 seg) { return kb < seg ? kb : kb - seg; }
__device__ __forceinline__ u32 b_col(u32 kb, u32 seg) { return kb < 2 * seg ? kb : kb - 2 * seg; }

// ---- candidate pass ---------------------------------------------------------
// Bound by the issue of the MMAs and their waits, then by the row boxes from L2
// (a tile's 64 KB per 128 queries): 300k x 128 integer rows, 10k queries, 1.09
// -> 0.57 ms, 0.69 of the measured bf16 rate.  The epilogue does two keys per
// fma and takes two at a time into the running minimum.
// STREAM_A: the query boxes travel through the ring with the row boxes (a
// compile-time choice, so the resident form's MMA issue loop carries no test).
// KEYS: the keys are written beside the minima (all_keys 2).
template <bool STREAM_A, bool KEYS>
__global__ void __launch_bounds__(TC_THREADS, 1)
    gt_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, TcArgs a) {
    extern __shared__ unsigned char tc_raw[];
    __shared__ __align__(8) u64 full[TC_MAX_STAGES], empty[TC_MAX_STAGES];
    __shared__ __align__(8) u64 a_full, a_empty, t_full[2], t_empty[2], drain, x_full[TC_XS], x_empty[TC_XS];
    __shared__ __align__(16) float xs[TC_XS][TC_ACC];    // ring of the tiles' key bases
    __shared__ u32 tmem_base;
    __shared__ volatile int abort_flag;
    unsigned char *sm = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(tc_raw) + 1023) & ~(uintptr_t)1023);
    const int warp = threadIdx.x >> 5, lane = lane_id();
    const u32 items = a.m_tiles * a.chunks;
    const u32 bbox = a.bn * TC_KBOX * 2;            // bytes of one row box
    // query tiles past the batch size in device memory are skipped, the same
    // items by every role
    const u32 nq_eff = a.nq_dev ? min(*a.nq_dev, a.nq) : a.nq;
    const u32 mt_eff = (nq_eff + TC_ROWS - 1) / TC_ROWS;
    // resident: sA holds the query tile (one or two segments), then the ring of row
    // boxes; streamed: each ring stage is a row box followed by the query box
    // of the same 64 columns
    const u32 sbytes = bbox + (STREAM_A ? TC_BOX : 0u);
    unsigned char *sA = sm;
    const u32 aboxes = min(a.kblocks, 2 * a.seg);
    unsigned char *sB = sm + (STREAM_A ? 0u : (size_t)aboxes * TC_BOX);

    if (threadIdx.x == 0) {
        for (u32 i = 0; i < a.stages; i++) {
            mbar_init(&full[i], 1);
            mbar_init(&empty[i], 1);
        }
        mbar_init(&a_full, 1);
        mbar_init(&a_empty, 1);
        for (int b = 0; b < 2; b++) {
            mbar_init(&t_full[b], 1);
            mbar_init(&t_empty[b], TC_EPI_WARPS);
        }
        for (int i = 0; i < TC_XS; i++) {
            mbar_init(&x_full[i], 1);
            mbar_init(&x_empty[i], TC_EPI_WARPS);
        }
        mbar_init(&drain, 1);
        abort_flag = 0;
        asm volatile("prefetch.tensormap [%0];" ::"l"(&tmA) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&tmB) : "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&tmem_base)),
                     "r"(2 * TC_ACC)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const u32 tmem = tmem_base;

    auto fail = [&]() {
        abort_flag = 1;
        atomicOr(a.err, ERR_TIMEOUT);
    };

    if (warp == 0) {
        // ---- producer: the warp runs the loop together, one elected lane issues every copy ----
        u32 stage = 0, ph = 0, issued = 0, lastpar = 0, a_issued = 0, a_ph = 0, xcount = 0;
        bool first = true, ok = true;
        const bool leader = elect_one();
        for (u32 it = blockIdx.x; it < items && ok && !abort_flag; it += gridDim.x) {
            const u32 mt = it % a.m_tiles, ch = it / a.m_tiles;
            const u32 t0 = ch * a.tiles_per_chunk, t1 = min(a.n_tiles, t0 + a.tiles_per_chunk);
            if (mt >= mt_eff) continue;
            if (!STREAM_A) {
                if (!first) {
                    if (!warp_wait(&a_empty, a_ph)) { ok = false; break; }
                    a_ph ^= 1;
                }
                first = false;
                if (leader) {
                    mbar_expect_tx(&a_full, aboxes * TC_BOX);
                    for (u32 kb = 0; kb < aboxes; kb++)
                        tma_load_2d(sA + (size_t)kb * TC_BOX, &tmA, (int)(kb * TC_KBOX), (int)(mt * TC_ROWS), &a_full);
                }
                __syncwarp();
                a_issued++;
            }
            for (u32 t = t0; t < t1 && ok; t++) {
                // the tile's key bases, up to TC_XS tiles ahead of the epilogue
                // (issued with the accumulator's buffer they cost each tile one
                // copy latency)
                const u32 xi = xcount % TC_XS;
                if (!warp_wait(&x_empty[xi], ((xcount / TC_XS) & 1) ^ 1)) { ok = false; break; }
                if (leader) {
                    mbar_expect_tx(&x_full[xi], a.bn * 4);
                    bulk_g2s(xs[xi], a.xn + (size_t)t * a.bn, a.bn * 4, &x_full[xi]);
                }
                __syncwarp();
                xcount++;
                for (u32 kb = 0; kb < a.kblocks; kb++) {
                    if (!warp_wait(&empty[stage], ph ^ 1)) { ok = false; break; }
                    unsigned char *sb = sB + (size_t)stage * sbytes;
                    if (leader) {
                        mbar_expect_tx(&full[stage], sbytes);
                        tma_load_2d(sb, &tmB, (int)(b_col(kb, a.seg) * TC_KBOX), (int)(t * a.bn), &full[stage]);
                        if (STREAM_A)
                            tma_load_2d(sb + bbox, &tmA, (int)(a_col(kb, a.seg) * TC_KBOX), (int)(mt * TC_ROWS),
                                        &full[stage]);
                    }
                    __syncwarp();
                    issued |= 1u << stage;
                    lastpar = (lastpar & ~(1u << stage)) | (ph << stage);
                    if (++stage == a.stages) {
                        stage = 0;
                        ph ^= 1;
                    }
                }
            }
        }
        if (!ok && lane == 0) fail();
        // every copy this warp issued has landed before the CTA exits
        for (u32 i = 0; i < a.stages; i++)
            if (issued >> i & 1) mbar_wait(&full[i], lastpar >> i & 1, WAIT_LIMIT);
        if (a_issued) mbar_wait(&a_full, (a_issued - 1) & 1, WAIT_LIMIT);
        for (u32 i = 0; i < TC_XS && i < xcount; i++)
            mbar_wait(&x_full[i], ((xcount - 1 - i) / TC_XS) & 1, WAIT_LIMIT);
    } else if (warp == 1) {
        // ---- MMA issuer: the warp runs the loop together, one elected lane issues.
        // With a branch on the lane around the whole loop each tcgen05.mma took
        // about 330 cycles to issue (its operands must be in uniform registers):
        // 3,170 cycles a tile of 128 x 256 x 128 against 1,024 of tensor work.
        {
            u32 stage = 0, ph = 0, a_ph = 0, tcount = 0;
            const u32 leader = elect_one();
            const u32 idesc = tc_idesc(a.bn);
            const u64 dA = sw128_desc(smem_addr(sA)), dB = sw128_desc(smem_addr(sB));
            bool ok = true;
            for (u32 it = blockIdx.x; it < items && ok; it += gridDim.x) {
                const u32 ch = it / a.m_tiles;
                const u32 t0 = ch * a.tiles_per_chunk, t1 = min(a.n_tiles, t0 + a.tiles_per_chunk);
                if (it % a.m_tiles >= mt_eff) continue;
                if (!STREAM_A) {
                    if (!warp_wait(&a_full, a_ph)) { ok = false; break; }
                    a_ph ^= 1;
                    tc_fence_after();
                }
                for (u32 t = t0; t < t1; t++, tcount++) {
                    const u32 b = tcount & 1;
                    if (!warp_wait(&t_empty[b], ((tcount >> 1) & 1) ^ 1)) { ok = false; break; }
                    tc_fence_after();
                    const u32 acol = tmem + b * TC_ACC;
                    for (u32 kb = 0; kb < a.kblocks; kb++) {
                        if (!warp_wait(&full[stage], ph)) { ok = false; break; }
                        tc_fence_after();
                        const u64 bd = dB + (u64)(stage * sbytes >> 4);
                        const u64 ad = STREAM_A ? bd + (bbox >> 4) : dA + (u64)(a_col(kb, a.seg) * (TC_BOX >> 4));
#pragma unroll
                        for (u32 k = 0; k < TC_KBOX / 16; k++)
                            tc_mma(acol, ad + 2 * k, bd + 2 * k, idesc, (kb | k) != 0, leader);
                        tc_commit(&empty[stage], leader);
                        if (++stage == a.stages) {
                            stage = 0;
                            ph ^= 1;
                        }
                    }
                    if (!ok) break;
                    tc_commit(&t_full[b], leader);
                }
                if (!STREAM_A) tc_commit(&a_empty, leader);
            }
            if (!ok && lane == 0) fail();
            // all MMAs issued by this warp are complete before TMEM and
            // shared memory are released
            tc_commit(&drain, leader);
            mbar_wait(&drain, 0, WAIT_LIMIT);
        }
    } else {
        // ---- epilogue: warp w reads TMEM lanes 32 (w % 4) .. + 31; lane = one query ----
        // each group of four warps takes one half of the tile's rows
        const int half = (warp - 2) >> 2, quarter = warp & 3;
        {
            const int row = quarter * 32 + lane;
            u32 tcount = 0;
            bool ok = true;
            for (u32 it = blockIdx.x; it < items && ok; it += gridDim.x) {
                const u32 mt = it % a.m_tiles, ch = it / a.m_tiles;
                const u32 t0 = ch * a.tiles_per_chunk, t1 = min(a.n_tiles, t0 + a.tiles_per_chunk);
                if (mt >= mt_eff) continue;
                const u32 q = mt * TC_ROWS + row;
                const bool valid = q < nq_eff;
                float4 *dst = reinterpret_cast<float4 *>(a.out + (size_t)(valid ? q : 0) * a.ld);
                for (u32 t = t0; t < t1; t++, tcount++) {
                    const u32 b = tcount & 1;
                    const u32 xi = tcount % TC_XS;
                    // every lane waits; the warp goes on together (tcgen05.ld is .sync.aligned)
                    const bool got = !abort_flag && mbar_wait(&t_full[b], (tcount >> 1) & 1, WAIT_LIMIT) &&
                                     mbar_wait(&x_full[xi], (tcount / TC_XS) & 1, WAIT_LIMIT);
                    if (!__all_sync(FULL, got)) { ok = false; break; }
                    tc_fence_after();
                    const u32 tbase = tmem + ((u32)(quarter * 32) << 16) + b * TC_ACC + half * TC_ROWS;
                    u32 r[TC_ROWS];
                    tmem_ld64(tbase, r);
                    tmem_ld64(tbase + 64, r + 64);
                    tmem_wait();
#pragma unroll
                    for (int i = 0; i < TC_ROWS; i++) asm volatile("" : "+r"(r[i]));   // no use moves before the wait
                    // TMEM buffer b and the key bases are refilled after this: only once
                    // every loaded value has been used (given up right after the wait,
                    // the next tile's MMAs overwrote columns still being read)
                    auto release = [&]() {
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) {
                            mbar_arrive(&t_empty[b]);
                            mbar_arrive(&x_empty[xi]);
                        }
                    };
                    const ulonglong2 *x2 = reinterpret_cast<const ulonglong2 *>(xs[xi] + half * TC_ROWS);
                    const u64 s2 = pair32(__float_as_uint(a.s), __float_as_uint(a.s));
                    if (a.all_keys == 1) {
                        float *o = a.out + (size_t)(valid ? q : 0) * a.ld + t * a.bn + half * TC_ROWS;
#pragma unroll
                        for (int j8 = 0; j8 < TC_ROWS / 8; j8++) {
                            const ulonglong2 v = x2[2 * j8], w = x2[2 * j8 + 1];
                            const u32 *rr = r + 8 * j8;
                            const u64 k0 = fma2(s2, pair32(rr[0], rr[1]), v.x), k1 = fma2(s2, pair32(rr[2], rr[3]), v.y);
                            const u64 k2 = fma2(s2, pair32(rr[4], rr[5]), w.x), k3 = fma2(s2, pair32(rr[6], rr[7]), w.y);
                            if (valid) st_global32(o + 8 * j8, k0, k1, k2, k3);
                        }
                        release();
                        continue;
                    }
                    float bm[TC_ROWS / 32];
#pragma unroll
                    for (int c = 0; c < TC_ROWS / 32; c++) {
                        float m0 = __int_as_float(0x7f800000), m1 = m0;
                        float *o = KEYS ? a.keys + ((size_t)(t * (a.bn / 32) + half * (TC_ROWS / 32) + c) * a.nq +
                                                    (valid ? q : 0)) * 32
                                        : nullptr;
#pragma unroll
                        for (int j8 = 0; j8 < 4; j8++) {
                            const ulonglong2 v = x2[c * 8 + 2 * j8], w = x2[c * 8 + 2 * j8 + 1];
                            const u32 *rr = r + c * 32 + 8 * j8;
                            const u64 k0 = fma2(s2, pair32(rr[0], rr[1]), v.x), k1 = fma2(s2, pair32(rr[2], rr[3]), v.y);
                            const u64 k2 = fma2(s2, pair32(rr[4], rr[5]), w.x), k3 = fma2(s2, pair32(rr[6], rr[7]), w.y);
                            m0 = min3(m0, pair_lo(k0), pair_hi(k0));
                            m1 = min3(m1, pair_lo(k1), pair_hi(k1));
                            m0 = min3(m0, pair_lo(k2), pair_hi(k2));
                            m1 = min3(m1, pair_lo(k3), pair_hi(k3));
                            if (KEYS && valid) st_global32(o + 8 * j8, k0, k1, k2, k3);
                        }
                        bm[c] = fminf(m0, m1);
                    }
                    release();
                    if (valid) dst[t * (a.bn / TC_ROWS) + half] = make_float4(bm[0], bm[1], bm[2], bm[3]);
                }
            }
            if (!ok && !abort_flag) fail();
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * TC_ACC)
                     : "memory");
    }
}

// ---- bf16 copies and norms ------------------------------------------------
__device__ __forceinline__ float bf16_round(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }

// Four consecutive elements: hi, lo and residual, with the sums an error bound needs.
struct Split4 {
    uint2 hi, lo;
    float sq, lo2, e2;
    bool anylo;
};
__device__ __forceinline__ uint2 pack_bf16x4(float a, float b, float c, float d) {
    const __nv_bfloat162 x = __floats2bfloat162_rn(a, b), y = __floats2bfloat162_rn(c, d);
    return make_uint2(*reinterpret_cast<const u32 *>(&x), *reinterpret_cast<const u32 *>(&y));
}
__device__ __forceinline__ Split4 split4(float4 v) {
    Split4 o;
    const float h0 = bf16_round(v.x), h1 = bf16_round(v.y), h2 = bf16_round(v.z), h3 = bf16_round(v.w);
    const float l0 = bf16_round(v.x - h0), l1 = bf16_round(v.y - h1), l2 = bf16_round(v.z - h2),
                l3 = bf16_round(v.w - h3);
    const float e0 = (v.x - h0) - l0, e1 = (v.y - h1) - l1, e2 = (v.z - h2) - l2, e3 = (v.w - h3) - l3;
    o.hi = pack_bf16x4(h0, h1, h2, h3);
    o.lo = pack_bf16x4(l0, l1, l2, l3);
    o.sq = fmaf(v.w, v.w, fmaf(v.z, v.z, fmaf(v.y, v.y, v.x * v.x)));
    o.lo2 = fmaf(l3, l3, fmaf(l2, l2, fmaf(l1, l1, l0 * l0)));
    o.e2 = fmaf(e3, e3, fmaf(e2, e2, fmaf(e1, e1, e0 * e0)));
    o.anylo = (l0 != 0.0f) | (l1 != 0.0f) | (l2 != 0.0f) | (l3 != 0.0f);
    return o;
}
// c (optional): subtracted from every element
__device__ __forceinline__ float4 load_row4(const float *r, u32 i, u32 dim, bool on, const float *c) {
    if (!on || i >= dim) return make_float4(0.f, 0.f, 0.f, 0.f);
    float4 v = *reinterpret_cast<const float4 *>(r + i);   // rows are padded to a multiple of 4
    if (c) {
        const float4 m = *reinterpret_cast<const float4 *>(c + i);
        v = make_float4(__fsub_rn(v.x, m.x), __fsub_rn(v.y, m.y), __fsub_rn(v.z, m.z), __fsub_rn(v.w, m.w));
    }
    if (i + 1 >= dim) v.y = 0.f;
    if (i + 2 >= dim) v.z = 0.f;
    if (i + 3 >= dim) v.w = 0.f;
    return v;
}

// A common vector near the rows' mean.  Squared L2 distances do not change
// when it is taken from rows and queries alike, but the norms that the error
// bound grows with do: on the 960-d non-negative mixture the bound falls to a
// third and with it the blocks a query has to score (40k rows, 2,003 queries:
// 21.5 -> 5.4 ms of scoring).
// The sample is CR rows spread over the ids.  gstat[6] is set when one of its
// elements is not exact in bf16: only then do the copies subtract the vector,
// so that data for which one bf16 segment is enough stay so.  A column whose
// mean is no ordinary number keeps 0.
constexpr int CR = 256;
__global__ void __launch_bounds__(1024) gt_center_kernel(Dev d, u64 next_id, float *center, u32 *gstat) {
    __shared__ float part[32][33];
    const u32 col = blockIdx.x * 32 + threadIdx.x, ry = threadIdx.y;   // 32 columns x 32 row groups
    const u32 n = (u32)min((u64)CR, next_id);
    const u64 stride = next_id / n * d.mp;
    float sum = 0.0f;
    bool inexact = false;
    if (col < d.mp)
#pragma unroll 8
        for (u32 j = ry; j < n; j += 32) {
            const float v = d.x[j * stride + col];
            sum += v;
            inexact |= bf16_round(v) != v;
        }
    if (__any_sync(FULL, inexact) && threadIdx.x == 0) atomicOr(gstat + 6, 1u);
    part[ry][threadIdx.x] = sum;
    __syncthreads();
    if (ry == 0 && col < d.mp) {
        float s = 0.0f;
        for (int j = 0; j < 32; j++) s += part[j][threadIdx.x];
        const float c = rintf(s / (float)n);
        center[col] = fabsf(c) <= 1048576.0f ? c : 0.0f;
    }
}

// gstat: [0] max |x|^2, [1] max |lo_x|, [2] max |e_x| (fp32 bits), [3] any lo != 0.
// A warp per row, grid-stride; maxima are kept per warp and published per block.
// ids (optional): row c is node ids[c]; check_live: rows of deleted or
// never-inserted nodes get key base +inf and a zero copy.
// Bound by the rows' bytes (4 m read, 4 m written; 3.5 and 4.3 TB/s).  Publishing
// per warp was 80k atomics on one sector, a row's loads waited for its reference
// word, and the copies held a third segment [hi | lo | hi]: 40k x 960 with queries
// 119 -> 91 us, 300k x 128 105 -> 95.  The blocks that are resident, on rows that
// lie together: four waves of blocks 97 and 105, a warp's four rows apart 133.
// U rows of a warp in flight (4 for rows of one column block, each lane 16 bytes
// of each; 1 else, with four column blocks in flight).
constexpr int PREP_WARPS = 8;
// Sums over the warp of U = 1 value (in every lane) or of U = 4 values (value
// lane >> 3; a lane passes on half of what it still holds), the same additions.
template <int U>
__device__ __forceinline__ float row_sums(const float (&v)[U], int lane) {
    float t = v[0];
    if (U == 4) {
        const bool hi = lane & 16, mid = lane & 8;
        const float a0 = (hi ? v[2 % U] : v[0]) + __shfl_xor_sync(FULL, hi ? v[0] : v[2 % U], 16);
        const float a1 = (hi ? v[3 % U] : v[1 % U]) + __shfl_xor_sync(FULL, hi ? v[1 % U] : v[3 % U], 16);
        t = (mid ? a1 : a0) + __shfl_xor_sync(FULL, mid ? a0 : a1, 8);
    }
#pragma unroll
    for (int h = U == 4 ? 4 : 16; h >= 1; h >>= 1) t += __shfl_xor_sync(FULL, t, h);
    return t;
}
template <int U>
__global__ void __launch_bounds__(PREP_WARPS * 32)
    gt_prep_rows(Dev d, const u32 *ids, u64 next_id, u32 n_pad, bool check_live, u32 kp1, u32 kb, u32 *B, float *xn,
                 u32 *gstat, const float *center) {
    __shared__ float red[3][PREP_WARPS];
    const int lane = lane_id(), warp = threadIdx.x >> 5;
    if (center && !gstat[6]) center = nullptr;
    const u32 nwarps = gridDim.x * PREP_WARPS;
    constexpr int V = 4 / U;   // column blocks of a row in flight
    float mx_sq = 0.0f, mx_lo = 0.0f, mx_e = 0.0f;
    bool any_lo = false;
    for (u32 c0 = (blockIdx.x * PREP_WARPS + warp) * U; c0 < n_pad; c0 += U * nwarps) {
        u32 id[U];
        u64 rf[U];
        bool live[U];
        float sq[U], lo2[U], e2[U];
#pragma unroll
        for (int r = 0; r < U; r++) {
            const u32 c = c0 + r;
            live[r] = c < next_id;
            id[r] = live[r] ? (ids ? ids[c] : c) : 0u;
            rf[r] = check_live && live[r] ? d.ref[id[r]] : 0;
            sq[r] = lo2[r] = e2[r] = 0.0f;
        }
        bool anylo = false;
        for (u32 i0 = 4 * lane; i0 < kp1; i0 += 128 * V) {
            float4 v[U][V];
#pragma unroll
            for (int r = 0; r < U; r++)
#pragma unroll
                for (int u = 0; u < V; u++) {
                    const u32 i = i0 + 128 * u;
                    v[r][u] = load_row4(d.x + (size_t)id[r] * d.mp, i, d.dim, i < kp1 && c0 + r < next_id, center);
                }
#pragma unroll
            for (int r = 0; r < U; r++) {
                const u32 c = c0 + r;
                if (c >= next_id) break;
                const bool on = !check_live || (!ref_del(rf[r]) && ref_slab(rf[r]) != NIL);
                uint2 *br = reinterpret_cast<uint2 *>(B + (size_t)c * (kb / 2));
#pragma unroll
                for (int u = 0; u < V; u++) {
                    const u32 i = i0 + 128 * u;
                    if (i >= kp1) break;
                    const Split4 w = split4(on ? v[r][u] : make_float4(0.f, 0.f, 0.f, 0.f));
                    br[i / 4] = w.hi;
                    br[(kp1 + i) / 4] = w.lo;
                    sq[r] += w.sq;
                    lo2[r] += w.lo2;
                    e2[r] += w.e2;
                    anylo |= w.anylo;
                }
            }
        }
        u32 live_bits = 0;
#pragma unroll
        for (int r = 0; r < U; r++)
            live_bits |= (live[r] && (!check_live || (!ref_del(rf[r]) && ref_slab(rf[r]) != NIL)) ? 1u : 0u) << r;
        const u32 mine = U == 4 ? lane >> 3 : 0;
        const bool on = live_bits >> mine & 1;
        const float n2 = row_sums<U>(sq, lane);
        const u32 c = c0 + mine;
        if ((U == 4 ? lane & 7 : lane) == 0 && c < n_pad) xn[c] = on ? (d.metric == 0 ? n2 : 0.0f) : __int_as_float(0x7f800000);
        if (on) mx_sq = fmaxf(mx_sq, n2);
        // the copy of a row that is not live is zero; without low parts the
        // remainders are zero too
        if (__any_sync(FULL, anylo)) {
            any_lo = true;
            mx_lo = fmaxf(mx_lo, row_sums<U>(lo2, lane));
            mx_e = fmaxf(mx_e, row_sums<U>(e2, lane));
        }
    }
    // of values >= 0 (no NaN passes fmaxf) the bits are ordered as the values are
    const u32 m_sq = __reduce_max_sync(FULL, __float_as_uint(mx_sq)), m_lo = __reduce_max_sync(FULL, __float_as_uint(mx_lo));
    const u32 m_e = __reduce_max_sync(FULL, __float_as_uint(mx_e));
    if (lane == 0) {
        red[0][warp] = __uint_as_float(m_sq);
        red[1][warp] = sqrtf(__uint_as_float(m_lo));
        red[2][warp] = sqrtf(__uint_as_float(m_e));
    }
    any_lo = __syncthreads_or(any_lo);
    if (threadIdx.x < 3) {
        float m = 0.0f;
        for (int w = 0; w < PREP_WARPS; w++) m = fmaxf(m, red[threadIdx.x][w]);
        if (m > 0.0f) atomicMax(gstat + threadIdx.x, __float_as_uint(m));
    }
    if (threadIdx.x == 3 && any_lo) atomicOr(gstat + 3, 1u);
}

// qstat per query: |q|^2, |q|, |lo_q|, |e_q|; copy as [hi | lo]
__global__ void gt_prep_queries(const float *q, u32 mp, u32 dim, u32 nq, u32 kp1, u32 kb, u32 *A, float *qstat,
                                u32 *gstat, const float *center, const u32 *nq_dev) {
    const u32 r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = lane_id();
    if (r >= (nq_dev ? min(*nq_dev, nq) : nq)) return;
    if (center && !gstat[6]) center = nullptr;
    const float *qr = q + (size_t)r * mp;
    uint2 *ar = reinterpret_cast<uint2 *>(A + (size_t)r * (kb / 2));
    float sq = 0.0f, lo2 = 0.0f, e2 = 0.0f;
    bool anylo = false;
    for (u32 i = 4 * lane; i < kp1; i += 128) {
        const Split4 v = split4(load_row4(qr, i, dim, true, center));
        ar[i / 4] = v.hi;
        ar[(kp1 + i) / 4] = v.lo;
        sq += v.sq;
        lo2 += v.lo2;
        e2 += v.e2;
        anylo |= v.anylo;
    }
#pragma unroll
    for (int h = 16; h >= 1; h >>= 1) {
        sq += __shfl_xor_sync(FULL, sq, h);
        lo2 += __shfl_xor_sync(FULL, lo2, h);
        e2 += __shfl_xor_sync(FULL, e2, h);
    }
    anylo = __any_sync(FULL, anylo);
    if (lane == 0) {
        qstat[4 * (size_t)r + 0] = sq;
        qstat[4 * (size_t)r + 1] = sqrtf(sq);
        qstat[4 * (size_t)r + 2] = sqrtf(lo2);
        qstat[4 * (size_t)r + 3] = sqrtf(e2);
        if (anylo && !*reinterpret_cast<volatile u32 *>(gstat + 3)) atomicOr(gstat + 3, 1u);
    }
}

// ---- the error bound ----------------------------------------------------------
// E, the most by which an approximate key can differ from |canonical distance
// - |q|^2| (L2) or from canonical distance - 1 (IP), doubled for safety, up to
// the factor 1 - 2 (m + 4) u of the L2 form below.  qs: |q|^2, |q|, |lo_q|,
// |e_q| of the query; gs: max |x|^2, max |lo_x|, max |e_x| over the rows (fp32
// bits).  K = contracted length.  Every operation rounds up (in fp32: double
// arithmetic cost a warp 3,000 cycles and more).
__device__ float key_error(int metric, float m, float K, bool split, const float *qs, const u32 *gs) {
    auto mul = [](float x, float y) { return __fmul_ru(x, y); };
    auto add = [](float x, float y) { return __fadd_ru(x, y); };
    const float u = 1.0f / 16777216.0f;
    const float qn = qs[0], qa = mul(qs[1], 1.011f), loq = mul(qs[2], 1.011f), eq = mul(qs[3], 1.011f);
    const float X2 = __uint_as_float(gs[0]), X1 = mul(__fsqrt_ru(X2), 1.011f);
    const float Lx = mul(__uint_as_float(gs[1]), 1.011f), Ex = mul(__uint_as_float(gs[2]), 1.011f);
    // |computed dot - q.x|: the terms the split leaves out, plus fp32 accumulation
    const float qx = mul(qa, X1);
    float dot_err = mul(mul(mul(add(K, 2.0f), 2.0f * u), 1.03f), qx);
    if (split) dot_err = add(dot_err, add(add(mul(loq, Lx), mul(add(qa, eq), Ex)), mul(eq, add(X1, Ex))));
    const float mu = mul(add(m, 2.0f), u);
    if (metric == 0) {   // taking the centre off, norms (fp32 sums of squares), 2 x dot error, rounding of the key
        const float s = add(qa, X1);
        float e = add(mul(2.1f * u, mul(s, s)), add(mul(mul(mu, qn), 1.01f), mul(mu, X2)));
        e = add(e, add(2.0f * dot_err, mul(2.0f * u, add(X2, mul(2.1f, qx)))));
        return 2.0f * e;
    }
    return 2.0f * add(add(dot_err, mul(mu, qx)), mul(u, add(1.0f, qx)));
}
// No row with a canonical distance <= dk has an approximate key above the
// returned value (the canonical fp32 distance is within (m + 4) u of the exact
// one, and 1 / (1 - x) <= 1 + 2 x).
__device__ float key_upper_bound(int metric, float m, float qn, float E, float dk) {
    if (metric != 0) return __fadd_ru(__fadd_ru(dk, -1.0f), E);
    const float f = __fadd_ru(1.0f, __fmul_ru(__fadd_ru(m, 4.0f), 4.0f / 16777216.0f));
    return __fadd_ru(__fadd_ru(__fmul_ru(dk, f), -qn), E);
}
// The canonical distance of a row with an approximate key <= key is at most the
// returned value.
__device__ float dist_upper_bound(int metric, float m, float qn, float E, float key) {
    if (metric != 0) return __fadd_ru(__fadd_ru(1.0f, key), E);
    const float f = __fadd_ru(1.0f, __fmul_ru(__fadd_ru(m, 4.0f), 4.0f / 16777216.0f));
    return fmaxf(0.0f, __fmul_ru(__fadd_ru(__fadd_ru(qn, key), E), f));
}

// ---- threshold and exact rerank -----------------------------------------------
__host__ __device__ constexpr int rr_warps(int W) { return W == 1 ? 8 : W; }   // a block's warps
constexpr int RR_LIST = 256;      // candidate blocks a warp collects before it scores them

struct RerankArgs {
    u32 nq, q0, k, nblk, m, kprime, split;
    u64 n_rows;
    const float *q;       // all queries, nq_total x mp fp32
    const float *bmin;    // this group: nq x nblk
    const float *keys;    // KEYS: this group, nblk x nq x 32
    const float *qstat;   // all queries
    const u32 *gstat;
    u32 *out_ids;         // all queries, x k
    float *out_dist;
    u32 *fb;              // queries left to the exact CUDA-core kernel (global indices)
    u32 *fb_count;
    const u32 *err;       // candidate pass error word: nonzero = minima incomplete
};

// canon_dist<8> of two rows against one query row (global memory), the column
// blocks outermost: eight row loads in flight, the query's read once for both.
// The same operations in the same order as canon_dist<8>.
__device__ __forceinline__ void canon_dist_wide2(const float *__restrict__ q, const float *__restrict__ r0,
                                                 const float *__restrict__ r1, int mp, int metric, int g, float &d0,
                                                 float &d1) {
    float p0[4], p1[4];
#pragma unroll
    for (int t = 0; t < 4; t++) p0[t] = p1[t] = 0.0f;
    auto fold = [&](float acc, const float4 &u, const float4 &v) {
        if (metric == 0) {
            const float e0 = __fsub_rn(u.x, v.x), e1 = __fsub_rn(u.y, v.y);
            const float e2 = __fsub_rn(u.z, v.z), e3 = __fsub_rn(u.w, v.w);
            return __fmaf_rn(e3, e3, __fmaf_rn(e2, e2, __fmaf_rn(e1, e1, __fmaf_rn(e0, e0, acc))));
        }
        return __fmaf_rn(u.w, v.w, __fmaf_rn(u.z, v.z, __fmaf_rn(u.y, v.y, __fmaf_rn(u.x, v.x, acc))));
    };
    for (int base = 0; base < mp; base += 128) {
        float4 u[4], v[4], w[4];
#pragma unroll
        for (int t = 0; t < 4; t++) {
            const int i = base + 4 * (g + 8 * t);
            if (i < mp) {
                v[t] = *reinterpret_cast<const float4 *>(r0 + i);
                w[t] = *reinterpret_cast<const float4 *>(r1 + i);
                u[t] = *reinterpret_cast<const float4 *>(q + i);
            }
        }
#pragma unroll
        for (int t = 0; t < 4; t++)
            if (base + 4 * (g + 8 * t) < mp) {
                p0[t] = fold(p0[t], u[t], v[t]);
                p1[t] = fold(p1[t], u[t], w[t]);
            }
    }
    float s0 = __fadd_rn(__fadd_rn(p0[0], p0[2]), __fadd_rn(p0[1], p0[3]));
    float s1 = __fadd_rn(__fadd_rn(p1[0], p1[2]), __fadd_rn(p1[1], p1[3]));
#pragma unroll
    for (int h = 4; h >= 1; h >>= 1) {
        s0 = __fadd_rn(s0, __shfl_xor_sync(FULL, s0, h));
        s1 = __fadd_rn(s1, __shfl_xor_sync(FULL, s1, h));
    }
    d0 = metric == 0 ? s0 : __fsub_rn(1.0f, s0);
    d1 = metric == 0 ? s1 : __fsub_rn(1.0f, s1);
}

// The canonical keys of the rows rl[0 .. n - 1] for the query qv, by one warp.
__device__ __noinline__ void score_rows(const float *x, u32 mp, u32 metric, const float *qv, const u32 *rl, u32 n,
                                        u64 *out) {
    const int lane = lane_id(), grp = lane >> 3, g = lane & 7;
    if (mp <= 128) {
        float4 q[4];
        canon_row_q8(qv, (int)mp, g, q);
        for (u32 r0 = 0; r0 < n; r0 += 8) {
            const u32 ia = rl[min(r0 + grp, n - 1)], ib = rl[min(r0 + 4 + grp, n - 1)];
            float4 va[4], vb[4];
            canon_row_q8(x + (size_t)ia * mp, (int)mp, g, va);
            canon_row_q8(x + (size_t)ib * mp, (int)mp, g, vb);
            const float da = canon_dist_q8v(q, va, (int)mp, (int)metric, g);
            const float db = canon_dist_q8v(q, vb, (int)mp, (int)metric, g);
            if (g == 0) {
                out[r0 + grp] = mkkey(da, ia);
                out[r0 + 4 + grp] = mkkey(db, ib);
            }
        }
    } else {
        const float one[4] = {1.0f, 1.0f, 1.0f, 1.0f};
        for (u32 r0 = 0; r0 < n; r0 += 4) {
            const void *row[4];
#pragma unroll
            for (int c = 0; c < 4; c++) row[c] = x + (size_t)rl[min(r0 + c, n - 1)] * mp;
            const float dd = warp_dists<0, 4, 2>(qv, row, one, (int)mp, (int)metric);
            if (g == 0) out[r0 + grp] = mkkey(dd, rl[min(r0 + grp, n - 1)]);
        }
    }
    __syncwarp();
}

// Bound by the row reads (L2) and their latency.  Scoring what the k-th
// distance leaves open, instead of a fixed 32 blocks with a certificate and a
// full scan by gt_kernel where it fails, and two blocks of 8 warps per SM:
// 10k queries x 300k x 128 integer rows 0.97 -> 0.50 ms; 2,003 queries x 40k x
// 960 real-valued rows, all of which failed the certificate, 53.5 -> 2.9 ms
// (21.5 before gt_center_kernel).
// W warps per query (1, 2, 4 or 8), as many as the SMs hold for all queries at
// once: 2,003 queries x 40k x 960 with 1, 2, 4, 8 warps 88, 98, 140, 237 us, 300
// queries 57, 42, 39, 42.
// KEYS: the candidate pass left every key, and of a candidate block only the rows
// below the threshold are scored: the 960-d batch 866 -> 88 us, the same sizes of
// the non-negative mixture 2.9 -> 0.2 ms.
// Each lane keeps the four smallest minima of the blocks it reads, with their
// numbers, so that a threshold met by at most four blocks of any lane needs no
// second pass over the minima.
template <int W, bool KEYS>
__global__ void __launch_bounds__(rr_warps(W) * 32, 16 / rr_warps(W)) gt_rerank_kernel(Dev d, RerankArgs a) {
    constexpr int RR_WARPS = rr_warps(W);
    __shared__ u32 clist[RR_WARPS][RR_LIST];
    __shared__ u64 ckey[RR_WARPS][32];
    __shared__ u64 xbest[RR_WARPS][32];
    __shared__ u32 xsum[2][RR_WARPS];
    __shared__ u32 rlist[KEYS ? RR_WARPS : 1][64];   // rows to score
    const int warp = threadIdx.x >> 5, lane = lane_id();
    const int tw = warp % W;                         // this warp's place among the query's warps
    const u32 li = blockIdx.x * (RR_WARPS / W) + warp / W;
    if (li >= a.nq || *a.err) return;                // the same for every warp of a query
    const u32 qi = a.q0 + li;
    const float *row = a.bmin + (size_t)li * a.nblk; // nblk is a multiple of 8
    u32 parity = 0;
    auto team_sum = [&](u32 v) -> u32 {
        v = __reduce_add_sync(FULL, v);
        if (W == 1) return v;
        if (lane == 0) xsum[parity][warp] = v;
        __syncthreads();
        u32 s = 0;
#pragma unroll
        for (int w = 0; w < RR_WARPS; w++) s += xsum[parity][w];
        parity ^= 1;
        return s;
    };
    // 1. the four smallest minima of this lane's blocks
    u32 t0 = ~0u, t1 = ~0u, t2 = ~0u, t3 = ~0u, b0 = 0, b1 = 0, b2 = 0, b3 = 0;
    auto keep = [&](float f, u32 b) {
        const u32 v = f2ord(f);
        if (v < t3) {
            if (v < t2) {
                t3 = t2; b3 = b2;
                if (v < t1) {
                    t2 = t1; b2 = b1;
                    if (v < t0) { t1 = t0; b1 = b0; t0 = v; b0 = b; } else { t1 = v; b1 = b; }
                } else { t2 = v; b2 = b; }
            } else { t3 = v; b3 = b; }
        }
    };
    const u32 step = W * 128;
    const float4 none = make_float4(__int_as_float(0x7fffffff), __int_as_float(0x7fffffff), __int_as_float(0x7fffffff),
                                    __int_as_float(0x7fffffff));
    for (u32 b = (u32)(tw * 32 + lane) * 4; b < a.nblk; b += 4 * step) {
        float4 v[4];
#pragma unroll
        for (int u = 0; u < 4; u++)
            v[u] = b + u * step < a.nblk ? __ldg(reinterpret_cast<const float4 *>(row + b + u * step)) : none;
#pragma unroll
        for (int u = 0; u < 4; u++) {
            const u32 bb = b + u * step;
            keep(v[u].x, bb);
            keep(v[u].y, bb + 1);
            keep(v[u].z, bb + 2);
            keep(v[u].w, bb + 3);
        }
    }
    // 2. tau = the k-th smallest kept minimum (bitwise search on the
    //    order-preserving integer image): at least k blocks are <= tau, and
    //    each holds a live row
    u32 tau = 0;
    for (int bit = 31; bit >= 0; bit--) {
        const u32 tr = tau | (1u << bit);
        if (team_sum((u32)(t0 < tr) + (u32)(t1 < tr) + (u32)(t2 < tr) + (u32)(t3 < tr)) < a.k) tau = tr;
    }
    const float *qv = a.q + (size_t)qi * d.mp;
    const int grp = lane >> 3, g = lane & 7;
    float4 qr[4];
    if (d.mp <= 128) canon_row_q8(qv, (int)d.mp, g, qr);
    u64 top = KEY_INF;    // the query's 32 smallest keys, sorted across lanes
    u64 bound = KEY_INF;  // keys above it cannot be in the top k
    bool cert = true;     // the rows not scored cannot be either
    // 3. phase 0: the blocks with a minimum <= tau (dead-only blocks have
    //    +inf); phase 1: those that the k-th distance found does not exclude
    u32 lo = 0, hi = min(tau, ORD_INF - 1);
    // KEYS: of those blocks only the rows whose own key passes are scored, and
    // phase 1 takes the rest of phase 0's blocks too.  (A key that passes is
    // finite, its row live.)  With fewer than k blocks every live row is scored.
    const bool by_rows = KEYS && tau < ORD_INF;
    for (int phase = 0; phase < 2; phase++) {
        auto in = [&](u32 v) { return (by_rows || v > lo) && v <= hi; };
        const bool kept = !__any_sync(FULL, t3 <= hi);   // every block in (lo, hi] is among the kept ones
        if (phase == 1) {
            u32 cnt = 0;
            if (kept) {
                cnt = (u32)in(t0) + (u32)in(t1) + (u32)in(t2) + (u32)in(t3);
            } else {
                for (u32 b = (u32)(tw * 32 + lane) * 4; b < a.nblk; b += step) {
                    const float4 v = __ldg(reinterpret_cast<const float4 *>(row + b));
                    cnt += (u32)in(f2ord(v.x)) + (u32)in(f2ord(v.y)) + (u32)in(f2ord(v.z)) + (u32)in(f2ord(v.w));
                }
            }
            const u32 all = team_sum(cnt);
            if (all == 0) break;
            cert = all <= max(64u, a.nblk / 2);
            if (!cert) break;
        }
        u64 best = KEY_INF;   // this warp's 32 smallest keys of the phase
        // cand, a key a lane, into best: only when one can still enter the top k
        auto merge = [&](u64 cand) {
            const u64 kth = __shfl_sync(FULL, best, (int)a.k - 1);
            if (!__any_sync(FULL, cand < kth && cand < bound)) return;
            cand = warp_sort32(cand);
            const u64 rev = __shfl_sync(FULL, cand, 31 - lane);
            best = warp_sort32(best < rev ? best : rev);
        };
        u32 nrow = 0;         // rows in rlist
        // the first n <= 32 rows of the list
        auto score = [&](u32 n) {
            score_rows(d.x, d.mp, d.metric, qv, rlist[KEYS ? warp : 0], n, ckey[warp]);
            const u64 cand = lane < (int)n ? ckey[warp][lane] : KEY_INF;
            __syncwarp();
            merge(cand);
        };
        u32 cur = (u32)tw * 128;
        for (bool more = true; more;) {
            u32 pend = 0;
            auto collect = [&](u32 v, u32 b) {
                const bool c = in(v);
                const u32 m = __ballot_sync(FULL, c);
                if (c) clist[warp][pend + __popc(m & lanemask_lt())] = b;
                pend += __popc(m);
            };
            if (kept) {
                collect(t0, b0);
                collect(t1, b1);
                collect(t2, b2);
                collect(t3, b3);
                more = false;
            } else {
                for (; cur < a.nblk && pend <= RR_LIST - 128; cur += step) {
                    const u32 b = cur + 4 * lane;
                    const float4 v = b < a.nblk ? __ldg(reinterpret_cast<const float4 *>(row + b)) : none;
                    collect(f2ord(v.x), b);
                    collect(f2ord(v.y), b + 1);
                    collect(f2ord(v.z), b + 2);
                    collect(f2ord(v.w), b + 3);
                }
                more = cur < a.nblk;
            }
            __syncwarp();
            if (by_rows) {
                // keys of eight blocks in flight
                for (u32 i0 = 0; i0 < pend; i0 += 8) {
                    u32 v[8];
#pragma unroll
                    for (int c = 0; c < 8; c++)
                        v[c] = i0 + c < pend ? f2ord(__ldg(a.keys + ((size_t)clist[warp][i0 + c] * a.nq + li) * 32 + lane)) : ~0u;
#pragma unroll
                    for (int c = 0; c < 8; c++) {
                        const bool pass = v[c] > lo && v[c] <= hi;
                        const u32 m = __ballot_sync(FULL, pass);
                        if (m == 0) continue;
                        if (pass) rlist[warp][nrow + __popc(m & lanemask_lt())] = clist[warp][i0 + c] * 32u + lane;
                        nrow += __popc(m);
                        __syncwarp();
                        if (nrow >= 32) {
                            score(32);
                            const u32 rest = lane + 32 < (int)nrow ? rlist[warp][lane + 32] : 0u;
                            __syncwarp();
                            rlist[warp][lane] = rest;
                            __syncwarp();
                            nrow -= 32;
                        }
                    }
                }
                continue;
            }
            for (u32 i = 0; i < pend; i++) {
                const u32 id0 = clist[warp][i] * 32u;
                if (lane == 0 && i + 1 < pend) {
                    // the next candidate block's rows on their way to L2
                    const u64 r0 = (u64)clist[warp][i + 1] * 32u;
                    bulk_prefetch_l2(d.x + r0 * d.mp, (u32)(min((u64)32, a.n_rows - r0) * d.mp * 4u));
                }
                const int nr = (int)min((u64)32, a.n_rows - id0);
                bool live = false;
                if (lane < nr) {
                    const u64 rf = d.ref[id0 + lane];
                    live = !ref_del(rf) && ref_slab(rf) != NIL;
                }
                for (int r0 = 0; r0 < nr; r0 += 8) {
                    // every lane computes (the distance shuffles over the full warp)
                    const int ra = min(r0 + grp, nr - 1), rb = min(r0 + 4 + grp, nr - 1);
                    const float *xa = d.x + (size_t)(id0 + ra) * d.mp, *xb = d.x + (size_t)(id0 + rb) * d.mp;
                    float da, db;
                    if (d.mp <= 128) {
                        float4 va[4], vb[4];
                        canon_row_q8(xa, (int)d.mp, g, va);
                        canon_row_q8(xb, (int)d.mp, g, vb);
                        da = canon_dist_q8v(qr, va, (int)d.mp, (int)d.metric, g);
                        db = canon_dist_q8v(qr, vb, (int)d.mp, (int)d.metric, g);
                    } else {
                        canon_dist_wide2(qv, xa, xb, (int)d.mp, (int)d.metric, g, da, db);
                    }
                    if (g == 0) {
                        ckey[warp][r0 + grp] = mkkey(da, id0 + ra);
                        ckey[warp][r0 + 4 + grp] = mkkey(db, id0 + rb);
                    }
                }
                __syncwarp();
                const u64 cand = live ? ckey[warp][lane] : KEY_INF;
                __syncwarp();
                merge(cand);
            }
            __syncwarp();
        }
        if (KEYS && nrow) score(nrow);
        // join the warps' lists
        if (W > 1) {
            xbest[warp][lane] = best;
            __syncthreads();
        }
        for (int w = 0; w < W; w++) {
            const u64 o = W > 1 ? xbest[w][31 - lane] : __shfl_sync(FULL, best, 31 - lane);
            top = warp_sort32(top < o ? top : o);
        }
        if (W > 1) __syncthreads();
        if (phase == 1 || tau >= ORD_INF) break;     // tau: every live row was scored
        bound = __shfl_sync(FULL, top, (int)a.k - 1);
        float T = __int_as_float(0x7f800000);
        if (bound != KEY_INF) {
            const float *qs = a.qstat + 4 * (size_t)qi;
            T = key_upper_bound((int)d.metric, (float)a.m, qs[0],
                                key_error((int)d.metric, (float)a.m, (float)a.kprime, a.split != 0, qs, a.gstat),
                                key_rho(bound));
        }
        T = __fadd_rn(T, 0.0f);   // +0 for -0: a minimum of +0 is not above it
        cert = isfinite(T);
        lo = hi;
        hi = cert ? f2ord(T) : 0u;
        if (!cert || hi <= lo) break;
    }
    if (W > 1 && tw != 0) return;
    if (cert) {
        if (lane < (int)a.k) {
            a.out_ids[(size_t)qi * a.k + lane] = top == KEY_INF ? NIL : key_id(top);
            a.out_dist[(size_t)qi * a.k + lane] = top == KEY_INF ? __int_as_float(0x7f800000) : key_rho(top);
        }
    } else if (lane == 0) {
        a.fb[atomicAdd(a.fb_count, 1u)] = qi;
    }
}

// ---- seeding: exact top-L of the entry set ---------------------------------
constexpr int SS_CAP = 512;       // candidates a query may keep
constexpr int SS_WARPS = 4;

struct SeedSelArgs {
    u32 nq, L, S, ld, m, kprime;
    const float *q;       // nq x mp fp32
    const float *keys;    // nq x ld approximate keys (entry order)
    const float *qstat;
    const u32 *estat;     // maxima over the entry rows
    u64 *seed;            // nq x L
    u32 *fb;              // queries left to the CUDA-core seed kernel
    u32 *ctr;             // [0] their count, [1] error word of the candidate pass
    const u32 *nq_dev;    // when set, the batch size (nq is its cap)
};

// Canonical distances of the candidates [c0, c1) of one query into key.
__device__ __forceinline__ void seed_score(const Dev &d, const float *qv, const u32 *cidx, u32 c0, u32 c1, u64 *key) {
    const int lane = lane_id(), grp = lane >> 3, g = lane & 7;
    if (d.mp <= 128) {
        // the query's elements in registers; four rows per group in flight
        float4 qr[4];
        canon_row_q8(qv, (int)d.mp, g, qr);
        for (u32 r0 = c0; r0 < c1; r0 += 16) {
            u32 id[4];
#pragma unroll
            for (int u = 0; u < 4; u++) id[u] = d.entries[cidx[min(r0 + grp + 4 * u, c1 - 1)]];
            float4 v[4][4];
#pragma unroll
            for (int u = 0; u < 4; u++) canon_row_q8(d.x + (size_t)id[u] * d.mp, (int)d.mp, g, v[u]);
#pragma unroll
            for (int u = 0; u < 4; u++) {
                const float dd = canon_dist_q8v(qr, v[u], (int)d.mp, (int)d.metric, g);
                const u32 i = r0 + grp + 4 * u;
                if (i < c1 && g == 0) key[i] = mkkey(dd, id[u]);
            }
        }
    } else {
        const float sc[4] = {1.0f, 1.0f, 1.0f, 1.0f};
        for (u32 r0 = c0; r0 < c1; r0 += 4) {
            const void *row[4];
#pragma unroll
            for (int u = 0; u < 4; u++) row[u] = d.x + (size_t)d.entries[cidx[min(r0 + u, c1 - 1)]] * d.mp;
            const float dd = warp_dists<0, 4, 2>(qv, row, sc, (int)d.mp, (int)d.metric);
            const u32 i = r0 + (lane >> 3);
            if (i < c1 && g == 0) key[i] = mkkey(dd, d.entries[cidx[i]]);
        }
    }
    __syncwarp();
}

// A warp per query.  A threshold from a sample of the approximate keys collects
// a few more than L entries; the L-th smallest key among them bounds, by the
// error bound, the L-th canonical distance and with it the approximate key of
// every entry that can be a seed.  Those entries, and no others, are scored
// with the canonical distance and sorted.  Queries with more than SS_CAP of
// them, or without a finite bound, go to the CUDA-core kernel.  Bound by the
// row reads (L2) and, in small batches, by one warp's chain.
__global__ void __launch_bounds__(SS_WARPS * 32, 4) seed_select_kernel(Dev d, SeedSelArgs a) {
    __shared__ u32 cidx_s[SS_WARPS][SS_CAP];
    __shared__ u32 cord_s[SS_WARPS][SS_CAP];   // the candidates' approximate keys, ordered image
    __shared__ u64 ckey_s[SS_WARPS][SS_CAP];
    const int warp = threadIdx.x >> 5, lane = lane_id();
    const u32 qi = blockIdx.x * SS_WARPS + warp;
    if (qi >= (a.nq_dev ? min(*a.nq_dev, a.nq) : a.nq) || a.ctr[1]) return;
    u32 *cidx = cidx_s[warp], *cord = cord_s[warp];
    u64 *ckey = ckey_s[warp];
    const float *row = a.keys + (size_t)qi * a.ld;   // a.ld is a multiple of 256
    // the r-th smallest of n values, value(i) for i < n
    auto nth = [&](u32 r, u32 n, auto value) {
        u32 t = 0;
        for (int bit = 31; bit >= 0; bit--) {
            const u32 tr = t | (1u << bit);
            u32 c = 0;
            for (u32 i = lane; i < n; i += 32) c += (u32)(value(i) < tr);
            if (__reduce_add_sync(FULL, c) < r) t = tr;
        }
        return t;
    };
    // entries with a key in (lo, hi] (all up to hi when !from), appended to the
    // n candidates there are; returns their number with these (more than
    // SS_CAP: not all stored)
    auto collect = [&](u32 lo, bool from, u32 hi, u32 n) {
        for (u32 e0 = 0; e0 < a.S; e0 += 512) {
            float4 v[4];
#pragma unroll
            for (int u = 0; u < 4; u++) {
                const u32 e = e0 + 128 * u + 4 * lane;
                if (e < a.S) v[u] = *reinterpret_cast<const float4 *>(row + e);
            }
#pragma unroll
            for (int u = 0; u < 4; u++) {
                const u32 e = e0 + 128 * u + 4 * lane;
                const u32 o[4] = {f2ord(v[u].x), f2ord(v[u].y), f2ord(v[u].z), f2ord(v[u].w)};
                u32 in = 0;
#pragma unroll
                for (int c = 0; c < 4; c++)
                    if (e + c < a.S && o[c] <= hi && (!from || o[c] > lo)) in |= 1u << c;
                if (!__any_sync(FULL, in != 0)) continue;
#pragma unroll
                for (int c = 0; c < 4; c++) {
                    const u32 m = __ballot_sync(FULL, in >> c & 1u);
                    const u32 pos = n + __popc(m & lanemask_lt());
                    if ((in >> c & 1u) && pos < SS_CAP) {
                        cidx[pos] = e + c;
                        cord[pos] = o[c];
                    }
                    n += __popc(m);
                }
            }
        }
        __syncwarp();
        return n;
    };
    u32 tau = ~0u, cnt = 0;                          // all entries when S <= L
    if (a.S > a.L) {
        // a threshold from every 8th key (16 per lane), kept when the count of
        // keys at or below it lands in [L, SS_CAP]; raised when it falls short
        // (one query in twenty: the exact search over all keys that follows at
        // last takes a warp 80 us and would hold up the whole batch)
        u32 smp[16];
#pragma unroll
        for (int j = 0; j < 16; j++) {
            const u32 e = 8u * (lane + 32u * j);
            smp[j] = e < a.S ? f2ord(row[e]) : ~0u;
        }
        u32 rs = a.L / 8 + 8;
        for (int attempt = 0; attempt < 3; attempt++, rs += rs / 2 + 4) {
            tau = 0;
            for (int bit = 31; bit >= 0; bit--) {
                const u32 tr = tau | (1u << bit);
                u32 c = 0;
#pragma unroll
                for (int j = 0; j < 16; j++) c += (u32)(smp[j] < tr);
                if (__reduce_add_sync(FULL, c) < rs) tau = tr;
            }
            if (tau == ~0u) break;                   // fewer samples than rs
            cnt = collect(0u, false, tau, 0);
            if (cnt >= a.L) break;
        }
        if (tau == ~0u || cnt < a.L || cnt > (u32)SS_CAP) {
            tau = nth(a.L, a.S, [&](u32 e) { return f2ord(row[e]); });
            cnt = collect(0u, false, tau, 0);
        }
    } else {
        cnt = collect(0u, false, tau, 0);
    }
    const float *qs = a.qstat + 4 * (size_t)qi;
    bool cert = cnt <= (u32)SS_CAP;
    if (cert && tau != ~0u) {
        // keep the candidates that the bound does not exclude
        const u32 kth = nth(a.L, cnt, [&](u32 i) { return cord[i]; });
        const float E = key_error((int)d.metric, (float)a.m, (float)a.kprime, true, qs, a.estat);
        const float D = dist_upper_bound((int)d.metric, (float)a.m, qs[0], E, ord2f(kth));
        const float T = __fadd_rn(key_upper_bound((int)d.metric, (float)a.m, qs[0], E, D), 0.0f);
        cert = isfinite(T);
        const u32 hi = f2ord(T);
        if (cert && hi > tau) {
            cnt = collect(tau, true, hi, cnt);
            cert = cnt <= (u32)SS_CAP;
        } else if (cert) {
            u32 n = 0;
            for (u32 i0 = 0; i0 < cnt; i0 += 32) {
                const u32 i = i0 + lane;
                const bool in = i < cnt && cord[i] <= hi;
                const u32 e = in ? cidx[i] : 0u, m = __ballot_sync(FULL, in);
                if (in) cidx[n + __popc(m & lanemask_lt())] = e;   // at or below i: already read
                n += __popc(m);
            }
            cnt = n;
        }
        __syncwarp();
    }
    if (cert) {
        seed_score(d, a.q + (size_t)qi * d.mp, cidx, 0, cnt, ckey);
        // a key's place is the number of smaller ones (they are distinct): a short
        // loop with no dependent step, where the stages of a bitonic sort wait for
        // one another, or, unrolled, for their instructions
        u64 *out = a.seed + (size_t)qi * a.L;
        for (u32 b0 = 0; b0 < cnt; b0 += 128) {
            u64 v[4];
            u32 rank[4];
#pragma unroll
            for (int r = 0; r < 4; r++) {
                const u32 i = b0 + 32 * r + lane;
                v[r] = i < cnt ? ckey[i] : KEY_INF;
                rank[r] = 0;
            }
#pragma unroll 4
            for (u32 j = 0; j < cnt; j++) {
                const u64 o = ckey[j];
#pragma unroll
                for (int r = 0; r < 4; r++) rank[r] += (u32)(o < v[r]);
            }
#pragma unroll
            for (int r = 0; r < 4; r++)
                if (b0 + 32 * r + lane < cnt && rank[r] < a.L) out[rank[r]] = v[r];
        }
        for (u32 i = cnt + lane; i < a.L; i += 32) out[i] = KEY_INF;
    } else if (lane == 0) {
        a.fb[atomicAdd(a.ctr, 1u)] = qi;
    }
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    });
    return fn;
}

bool encode_bf16(CUtensorMap *m, const void *base, u64 rows, u32 cols, u32 box_rows) {
    auto fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[2] = {cols, rows};
    cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
    cuuint32_t box[2] = {TC_KBOX, box_rows};
    cuuint32_t es[2] = {1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, es,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

void prep_rows(const Dev &d, const u32 *ids, u64 next_id, u32 n_pad, bool check_live, u32 kp1, u32 kb, u32 *B, float *xn,
               u32 *gstat, const float *center, cudaStream_t st) {
    const u32 U = kp1 <= 128 ? 4 : 1;
    const u32 grid = std::min<u32>((n_pad + PREP_WARPS * U - 1) / (PREP_WARPS * U), 152 * (U == 4 ? 3 : 4));   // resident blocks
    auto *fn = U == 4 ? gt_prep_rows<4> : gt_prep_rows<1>;
    fn<<<grid, PREP_WARPS * 32, 0, st>>>(d, ids, next_id, n_pad, check_live, kp1, kb, B, xn, gstat, center);
}

}  // namespace

GtTcPlan gt_tc_plan(u32 dim, u64 next_id, u32 nq) {
    GtTcPlan p{};
    p.kp1 = (dim + TC_KBOX - 1) / TC_KBOX * TC_KBOX;
    p.kb = 2 * p.kp1;
    p.n_pad = (next_id + TC_ACC - 1) / TC_ACC * TC_ACC;
    p.bytes_B = (size_t)next_id * p.kb * 2;
    p.bytes_A = (size_t)nq * p.kb * 2;
    return p;
}

cudaError_t launch_gt_tc_prep(const Dev &d, u64 next_id, const float *q, u32 nq, const GtTcPlan &p,
                              const GtTcBufs &b, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(b.gstat, 0, 8 * sizeof(u32), st);
    if (e != cudaSuccess) return e;
    const float *center = d.metric == 0 && next_id ? b.center : nullptr;
    if (center) gt_center_kernel<<<(d.mp + 31) / 32, dim3(32, 32), 0, st>>>(d, next_id, b.center, b.gstat);
    if (p.n_pad)
        prep_rows(d, nullptr, next_id, (u32)p.n_pad, true, p.kp1, p.kb, reinterpret_cast<u32 *>(b.B), b.xn, b.gstat,
                  center, st);
    gt_prep_queries<<<(unsigned)(((size_t)nq * 32 + 255) / 256), 256, 0, st>>>(
        q, d.mp, d.dim, nq, p.kp1, p.kb, reinterpret_cast<u32 *>(b.A), b.qstat, b.gstat, center, nullptr);
    return cudaGetLastError();
}

void gt_tc_configure(GtTcPlan &p, u32 nq, u32 k, u32 mp, bool split, bool keys) {
    p.kprime = split ? 3 * p.kp1 : p.kp1;
    p.split = split;
    p.kblocks = p.kprime / TC_KBOX;
    const u32 abytes = (split ? 2 : 1) * (p.kp1 / TC_KBOX) * TC_BOX;
    const u32 smem_max = 227 * 1024 - 1024 - TC_STATIC;   // alignment slack, static shared memory
    p.bn = TC_ACC;
    const u32 bbox = p.bn * TC_KBOX * 2;
    if (p.n_pad == 0) {
        p.usable = false;
        return;
    }
    // the query tile stays resident when it fits beside two ring stages;
    // otherwise its boxes travel through the ring with the row boxes
    p.stream_a = (u64)abytes + 2ull * bbox > smem_max;
    if (p.stream_a) {
        p.stages = std::min<u32>(TC_MAX_STAGES, smem_max / (bbox + TC_BOX));
        p.smem = p.stages * (bbox + TC_BOX) + 1024;
    } else {
        p.stages = std::min<u32>(TC_MAX_STAGES, (smem_max - abytes) / bbox);
        p.smem = abytes + p.stages * bbox + 1024;
    }
    p.n_tiles = (u32)(p.n_pad / p.bn);
    p.nblk = (u32)(p.n_pad / 32);
    // queries per pass: the block-minimum buffer stays under 4 GiB
    const u64 cap = std::max<u64>(256, ((4ull << 30) / ((u64)p.nblk * 4)) / 256 * 256);
    p.qgroup = (u32)std::min<u64>(nq, cap);
    // Every key written costs 0.7 ns per 1000 rows and query (0.4 beside the
    // longer K of a split); what the rerank then leaves out are 31 of 32 rows in
    // at least k blocks, 4 mp bytes each: 960-d, 40k rows, 2,003 queries, k 10
    // (split) tensor + rerank 1,140 -> 400 us; at 128-d, k 10, even at 20k rows
    // (10k queries: 320 and 332 us), behind at 40k (2,003 queries: 96 and 127).
    p.keys = keys && p.n_pad <= (u64)k * mp * (split ? 24 : 16);
    if (p.keys) {
        const u64 room = (4ull << 30) / (p.n_pad * 4) / TC_ROWS * TC_ROWS;   // queries in 4 GiB
        p.keys = room > 0;
        if (p.keys) p.qgroup = (u32)std::min<u64>(p.qgroup, room);
    }
    p.bytes_keys = p.keys ? (size_t)p.qgroup * p.n_pad * 4 : 0;
    p.bytes_bmin = (size_t)p.qgroup * p.nblk * 4;
    p.usable = true;
}

cudaError_t launch_gt_tc(const Dev &d, u32 q0, u32 nq, const GtTcPlan &p, const GtTcBufs &b, u64 next_id,
                         int num_sms, cudaStream_t st) {
    CUtensorMap ta, tb;
    const void *abase = static_cast<const char *>(b.A) + (size_t)q0 * p.kb * 2;
    if (!encode_bf16(&ta, abase, nq, p.kb, TC_ROWS) || !encode_bf16(&tb, b.B, next_id, p.kb, p.bn))
        return cudaErrorInvalidValue;
    TcArgs a{};
    a.nq = nq;
    a.n_tiles = p.n_tiles;
    a.kblocks = p.kblocks;
    a.seg = p.kp1 / TC_KBOX;
    a.bn = p.bn;
    a.m_tiles = (nq + TC_ROWS - 1) / TC_ROWS;
    // chunks of rows: enough work items to fill every SM, with the fewest
    // idle SMs in the last wave
    u32 best_c = 1;
    double best_score = -1e9;
    const u32 cmax = std::max<u32>(1, std::min<u32>(p.n_tiles, 256));
    for (u32 c = 1; c <= cmax; c++) {
        const u64 items = (u64)a.m_tiles * c;
        const u64 waves = (items + num_sms - 1) / num_sms;
        const double eff = (double)items / (double)(waves * num_sms);
        const double score = eff - (items < (u64)num_sms ? 0.5 : 0.0) - 0.002 * c;
        if (score > best_score) {
            best_score = score;
            best_c = c;
        }
    }
    a.tiles_per_chunk = (p.n_tiles + best_c - 1) / best_c;
    a.chunks = (p.n_tiles + a.tiles_per_chunk - 1) / a.tiles_per_chunk;
    a.stages = p.stages;
    a.stream_a = p.stream_a ? 1u : 0u;
    a.all_keys = p.keys ? 2u : 0u;
    a.ld = p.nblk;
    a.s = d.metric == 0 ? -2.0f : -1.0f;
    a.xn = b.xn;
    a.out = b.bmin;
    a.keys = b.keys;
    a.err = b.err;
    auto *fn = p.stream_a ? (p.keys ? gt_tc_kernel<true, true> : gt_tc_kernel<true, false>)
                          : (p.keys ? gt_tc_kernel<false, true> : gt_tc_kernel<false, false>);
    cudaError_t e = smem_at_least((const void *)fn, p.smem);
    if (e != cudaSuccess) return e;
    const u32 items = a.m_tiles * a.chunks;
    fn<<<std::min<u32>(items, (u32)num_sms), TC_THREADS, p.smem, st>>>(ta, tb, a);
    return cudaGetLastError();
}

cudaError_t launch_gt_rerank(const Dev &d, const float *q, u32 q0, u32 nq, u32 k, const GtTcPlan &p,
                             const GtTcBufs &b, u64 next_id, u32 *out_ids, float *out_dist, int num_sms, cudaStream_t st) {
    RerankArgs r{};
    r.nq = nq;
    r.q0 = q0;
    r.k = k;
    r.nblk = p.nblk;
    r.m = d.dim;
    r.kprime = p.kprime;
    r.split = p.split;
    r.n_rows = next_id;
    r.q = q;
    r.bmin = b.bmin;
    r.keys = b.keys;
    r.qstat = b.qstat;
    r.gstat = b.gstat;
    r.out_ids = out_ids;
    r.out_dist = out_dist;
    r.fb = b.fb;
    r.fb_count = b.gstat + 4;
    r.err = b.err;
    // the most warps per query that the SMs hold at once
    u32 W = 1;
    while (W < 8 && (u64)nq * 2 * W <= (u64)num_sms * 16) W *= 2;
    const u32 grid = W == 1 ? (nq + rr_warps(1) - 1) / rr_warps(1) : nq;
    auto go = [&](auto *fn) { fn<<<grid, rr_warps(W) * 32, 0, st>>>(d, r); };
    if (W == 1) p.keys ? go(gt_rerank_kernel<1, true>) : go(gt_rerank_kernel<1, false>);
    else if (W == 2) p.keys ? go(gt_rerank_kernel<2, true>) : go(gt_rerank_kernel<2, false>);
    else if (W == 4) p.keys ? go(gt_rerank_kernel<4, true>) : go(gt_rerank_kernel<4, false>);
    else p.keys ? go(gt_rerank_kernel<8, true>) : go(gt_rerank_kernel<8, false>);
    return cudaGetLastError();
}

// ---- seeding on tensor cores ----------------------------------------------
SeedTcPlan seed_tc_plan(u32 dim, u32 n_entry, u32 nq) {
    SeedTcPlan p{};
    p.kp1 = (dim + TC_KBOX - 1) / TC_KBOX * TC_KBOX;
    p.kb = 2 * p.kp1;
    p.s_pad = (n_entry + TC_ACC - 1) / TC_ACC * TC_ACC;
    const u32 smem_max = 227 * 1024 - 1024 - TC_STATIC;
    const u32 bbox = TC_ACC * TC_KBOX * 2;
    const u32 abytes = (p.kb / TC_KBOX) * TC_BOX;
    p.usable = n_entry > 0;
    // the query tile resident when it fits beside two ring stages, else streamed
    p.stream_a = abytes + 2 * bbox > smem_max;
    if (p.stream_a) {
        p.stages = std::min<u32>(TC_MAX_STAGES, smem_max / (bbox + TC_BOX));
        p.smem = p.stages * (bbox + TC_BOX) + 1024;
    } else {
        p.stages = std::min<u32>(TC_MAX_STAGES, (smem_max - abytes) / bbox);
        p.smem = abytes + p.stages * bbox + 1024;
    }
    p.bytes_E = (size_t)n_entry * p.kb * 2;
    p.bytes_A = (size_t)nq * p.kb * 2;
    p.bytes_keys = (size_t)nq * p.s_pad * 4;
    return p;
}

cudaError_t launch_seed_tc_entries(const Dev &d, u32 S, const SeedTcPlan &p, const SeedTcBufs &b, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(b.estat, 0, 8 * sizeof(u32), st);
    if (e != cudaSuccess || p.s_pad == 0) return e;
    prep_rows(d, d.entries, S, p.s_pad, false, p.kp1, p.kb, reinterpret_cast<u32 *>(b.E), b.en, b.estat, nullptr, st);
    return cudaGetLastError();
}

cudaError_t launch_seed_tc(const Dev &d, const float *q, u32 nq, u32 S, u32 L, u64 *seed, const SeedTcPlan &p,
                           const SeedTcBufs &b, int num_sms, cudaStream_t st, const u32 *nq_dev) {
    if (nq == 0 || S == 0) return cudaSuccess;
    cudaError_t e = cudaMemsetAsync(b.ctr, 0, 8 * sizeof(u32), st);
    if (e != cudaSuccess) return e;
    gt_prep_queries<<<(unsigned)(((size_t)nq * 32 + 255) / 256), 256, 0, st>>>(
        q, d.mp, d.dim, nq, p.kp1, p.kb, reinterpret_cast<u32 *>(b.A), b.qstat, b.ctr + 4, nullptr, nq_dev);
    CUtensorMap ta, tb;
    if (!encode_bf16(&ta, b.A, nq, p.kb, TC_ROWS) || !encode_bf16(&tb, b.E, S, p.kb, TC_ACC))
        return cudaErrorInvalidValue;
    TcArgs a{};
    a.nq = nq;
    a.n_tiles = p.s_pad / TC_ACC;
    a.seg = p.kp1 / TC_KBOX;
    a.kblocks = 3 * a.seg;
    a.bn = TC_ACC;
    a.m_tiles = (nq + TC_ROWS - 1) / TC_ROWS;
    u32 best_c = 1;
    double best_score = -1e9;
    for (u32 c = 1; c <= a.n_tiles; c++) {
        const u64 items = (u64)a.m_tiles * c;
        const u64 waves = (items + num_sms - 1) / num_sms;
        const double score = (double)items / (double)(waves * num_sms) - 0.02 * c;
        if (score > best_score) {
            best_score = score;
            best_c = c;
        }
    }
    a.tiles_per_chunk = (a.n_tiles + best_c - 1) / best_c;
    a.chunks = (a.n_tiles + a.tiles_per_chunk - 1) / a.tiles_per_chunk;
    a.stages = p.stages;
    a.stream_a = p.stream_a ? 1u : 0u;
    a.nq_dev = nq_dev;
    a.all_keys = 1;
    a.ld = p.s_pad;
    a.s = d.metric == 0 ? -2.0f : -1.0f;
    a.xn = b.en;
    a.out = b.keys;
    a.err = b.ctr + 1;
    auto *fn = p.stream_a ? gt_tc_kernel<true, false> : gt_tc_kernel<false, false>;
    e = smem_at_least((const void *)fn, p.smem);
    if (e != cudaSuccess) return e;
    const u32 items = a.m_tiles * a.chunks;
    fn<<<std::min<u32>(items, (u32)num_sms), TC_THREADS, p.smem, st>>>(ta, tb, a);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    SeedSelArgs r{};
    r.nq = nq;
    r.L = L;
    r.S = S;
    r.ld = p.s_pad;
    r.m = d.dim;
    r.kprime = 3 * p.kp1;
    r.q = q;
    r.keys = b.keys;
    r.qstat = b.qstat;
    r.estat = b.estat;
    r.seed = seed;
    r.fb = b.fb;
    r.ctr = b.ctr;
    r.nq_dev = nq_dev;
    seed_select_kernel<<<(nq + SS_WARPS - 1) / SS_WARPS, SS_WARPS * 32, 0, st>>>(d, r);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    // queries the certificate did not cover: the exact CUDA-core seed, with
    // the count read on the device
    return launch_seed(d, q, nq, L, seed, st, 0, b.ctr, b.fb);
}

}  // namespace etale

// update.cu — RobustPrune, Publish-based update kernels: forward edges and
// own slab (Algorithm 2), reverse-edge offers, the refine pass, tombstoning
// and repair (Algorithm 3), compaction and reclaim (Algorithm 4).
//
// Deterministic mode groups offers by target (a stable radix sort by target
// id keeps sources ascending) and lets one warp fold a target's offers in
// order and publish once.  Lock-free mode gives each offer its own warp,
// which snapshots the target, builds the new list and publishes it with a
// compare-and-swap, retrying up to the attempt budget (Algorithm 1).
#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "internal.h"

namespace etale {

__host__ __device__ inline size_t al16(size_t x) { return (x + 15) / 16 * 16; }

// ---------------------------------------------------------------------------
// Row staging: the rows of the first `ns` candidates are copied into shared
// memory by bulk (TMA) copies completing on the warp's mbarrier; later
// candidates are read from global memory.
// ---------------------------------------------------------------------------
struct Stage {
    float *rows;     // ns_cap x mp floats, 16-byte aligned (nullptr: no staging)
    int ns_cap;
    u64 *bar;        // this warp's mbarrier
    u32 phase;
    bool timeout;
    char *gram;      // gram_bytes(gram_rows, mp) for the tensor-core Gram path (nullptr: canonical path)
    u32 gram_tag;    // its rows as the launch gave them (CANON_ROWS: variant 3)
    int gram_rows;   // candidates the Gram buffer holds (a multiple of 16, <= GRAM_NL)
    struct GramReq *req;     // the block's request slot (cooperative variants)
    u64 wk_rows, wk_state;   // this warp's work tallies (see WK_*), added by stage_done
};

// Tensor-core Gram tile: up to 64 candidates, K staged 128 columns at a time
// as bf16 rows of 256 bytes with no pad; the 16-byte chunk c of row r sits at
// chunk c ^ (r & 7), so the eight rows an ldmatrix phase reads at one column
// fall in eight distinct bank groups.
constexpr int GRAM_N = 64;
constexpr int GRAM_RB = 256;   // bytes per staged row (128 bf16 columns)
// The cooperative path (more than GRAM_N rows, or rows of more than one
// 128-column block; see gram_masks) pads its rows to GRAM_RS_CO bf16 (a 16-byte
// pad: conflict-free ldmatrix without a swizzle) and keeps two blocks of them.
constexpr int GRAM_RS_CO = 136;
constexpr int GRAM_NL = 128;   // candidates of the cooperative path
constexpr int COOP_WARPS = 4;
__host__ __device__ inline u32 gram_xoff(int r, int chunk) { return (u32)(r * GRAM_RB + ((chunk ^ (r & 7)) << 4)); }
// The Gram variant (see warp_prune) of a kernel whose buffer holds gram_rows rows of mp columns.
__host__ __device__ inline int gram_variant(u32 gram_rows, u32 mp) {
    return gram_rows >> 31 ? 3 : gram_rows > (u32)GRAM_N ? 1 : (gram_rows && mp > 128 ? 2 : 0);
}
__host__ __device__ constexpr bool coop_variant(int GV) { return GV >= 1 && GV <= 3; }
// Variant 3, canonical distances on the cooperative path, keeps masks only: its
// buffer is that of CANON_ROWS "rows".
constexpr u32 CANON_ROWS = 0x80000000u | GRAM_NL;
// Bytes of a Gram buffer's rows, and of the whole
// buffer: a (norm, rho) pair per candidate follows, and on the cooperative path
// its domination mask (two words).  rows is a multiple of 16; 0 = no buffer.
__host__ __device__ inline size_t gram_row_bytes(u32 rows, u32 mp) {
    if (rows >> 31) return 0;
    return gram_variant(rows, mp) ? (size_t)(mp > 128 ? 2 : 1) * rows * GRAM_RS_CO * 2 : (size_t)rows * GRAM_RB;
}
__host__ __device__ inline size_t gram_bytes(u32 rows, u32 mp) {
    return gram_row_bytes(rows, mp) + (size_t)(rows & 0x7FFFFFFFu) * (gram_variant(rows, mp) ? 8 + 16 : 8);
}
// Gram rows for a kernel whose prunes see at most max_n candidates (0: the
// Gram path is off or cannot hold them).
inline u32 gram_rows_for(u32 on, u32 max_n) { return on && max_n <= (u32)GRAM_NL ? (max_n + 15) / 16 * 16 : 0; }
// Scratch that is dead whenever the Gram buffer is live (list compaction before
// a prune, the canonical prune's arrays, a prune's output, written after its
// last read of the buffer) lives inside the Gram buffer's row bytes if it fits.
__host__ __device__ inline bool gram_alias(u32 gram, size_t scratch) { return gram && !(gram >> 31) && scratch <= (size_t)gram * GRAM_RB; }

// Shared-memory bytes for a stage of ns rows plus its mbarrier.
__host__ __device__ inline size_t stage_bytes(u32 ns, u32 mp) { return al16((size_t)ns * mp * 4) + 16; }

// Carve a stage at p (16-byte aligned) and initialise the warp's mbarrier.
__device__ __forceinline__ Stage stage_init(char *p, u32 ns, u32 mp, char *gram = nullptr, u32 gram_rows = 0,
                                            GramReq *req = nullptr) {
    Stage st;
    st.rows = ns ? reinterpret_cast<float *>(p) : nullptr;
    st.ns_cap = (int)ns;
    st.bar = reinterpret_cast<u64 *>(p + al16((size_t)ns * mp * 4));
    st.phase = 0;
    st.timeout = false;
    st.gram = gram;
    st.gram_tag = gram_rows;
    st.gram_rows = (int)(gram_rows & 0x7FFFFFFFu);
    st.req = req;
    st.wk_rows = st.wk_state = 0;
    if (lane_id() == 0) mbar_init(st.bar, 1);
    __syncwarp();
    return st;
}

__device__ __forceinline__ void stage_done(const Dev &d, const Stage &st, int kind) {
    if (lane_id() != 0) return;
    if (st.timeout) atomicOr(&d.ctr[C_ERR], (u64)ERR_TIMEOUT);
    if (st.wk_rows) atomicAdd(&d.ctr[C_WK + 2 * kind], st.wk_rows);
    if (st.wk_state) atomicAdd(&d.ctr[C_WK + 2 * kind + 1], st.wk_state);
}

// Row bytes a prune of n candidates gathers: the bf16 copy on the Gram path
// when the index keeps one, else the fp32 rows.
__device__ __forceinline__ u64 prune_row_bytes(const Dev &d, const Stage &st, int n) {
    const bool b16 = st.gram && !(st.gram_tag >> 31) && n <= st.gram_rows && d.xb;
    return (u64)n * (b16 ? 2ull * d.mb : 4ull * d.mp);
}

// Threads per block of the persistent update kernels: one warp, or one with its
// helpers on the cooperative path.  Their shared memory is per item (up to ~20
// KB with the Gram tile), so one-warp blocks pack the SM by the warp instead of
// by four (11 warps instead of 8 at 19 KB).
inline int block_threads(u32 gram_rows, u32 mp) { return gram_variant(gram_rows, mp) ? 32 * COOP_WARPS : 32; }

// Rows that fit a per-warp stage of `budget` bytes, capped at `want`.
inline u32 stage_cap(u32 mp, u32 want, u32 budget) {
    u32 cap = budget / (mp * 4u);
    return cap < want ? cap : want;
}

template <class IdOf>
__device__ __forceinline__ void stage_rows_by(const Dev &d, Stage &st, int ns, IdOf id_of) {
    const int lane = lane_id();
    if (ns <= 0) return;
    const u32 rowb = d.mp * 4;
    if (lane == 0) {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_expect_tx(st.bar, (u32)ns * rowb);
    }
    __syncwarp();
    for (int i = lane; i < ns; i += 32)
        bulk_g2s(st.rows + (size_t)i * d.mp, d.x + (size_t)id_of(i) * d.mp, rowb, st.bar);
    if (!mbar_wait(st.bar, st.phase, WAIT_LIMIT)) {
        st.timeout = true;
        mbar_wait(st.bar, st.phase, WAIT_LIMIT);
    }
    st.phase ^= 1u;
    __syncwarp();
}

__device__ __forceinline__ void stage_rows(const Dev &d, Stage &st, const u64 *ck, int ns) {
    stage_rows_by(d, st, ns, [&](int i) { return key_id(ck[i]); });
}


// ---------------------------------------------------------------------------
// Candidate Gram tile on the tensor cores (mma.sync m16n8k16, bf16 inputs,
// fp32 accumulation): G = X X^T for the n <= 64 candidate rows X, one warp.
// Squared L2 follows as (G_ii - G_ij) + (G_jj - G_ij), inner product as
// 1 - G_ij.  Inputs rounded to bf16 are exact for integer-valued data of
// magnitude <= 256, and so is every product and partial sum while the norms
// stay below 2^24; then each distance equals the canonical one bit for bit.
// ---------------------------------------------------------------------------

// ldmatrix row addresses in the swizzled tile: lane l reads (row, chunk
// 2 ks + (l >> 4)) with row & 7 = l & 7, so the chunk's byte offset in its row
// is (32 ks) ^ c0 with c0 = 16 ((l >> 4) ^ (l & 7)), shared by every row.
__device__ __forceinline__ u32 gram_c0(int lane) { return (u32)(((lane >> 4) ^ (lane & 7)) << 4); }

__device__ __forceinline__ void cp_async16(u32 dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Stage columns [128 kb, 128 kb + 128) of candidate rows [r_lo, r_hi) into the
// swizzled tile at xs, a lane per row and a 16-byte copy per chunk; chunks past
// the row's end are zeroed.  From the bf16 copy when there is one (the same
// round-to-nearest-even values), else converted from the fp32 rows.
__device__ __forceinline__ void gram_stage_rows(const Dev &d, const u64 *ck, int r_lo, int r_hi, int kb, u32 xs) {
    __syncwarp();   // earlier reads of these bytes are done
    const int lane = lane_id();
    const int cols = min(128, (int)d.mb - 128 * kb);   // d.mb is a multiple of 8
    const int nch = cols >> 3;
    for (int r = r_lo + lane; r < r_hi; r += 32) {
        const u32 id = key_id(ck[r]);
        if (d.xb) {
            const auto *src = d.xb + (size_t)id * d.mb + 128 * kb;
#pragma unroll 4
            for (int c = 0; c < 16; c++) {
                if (c < nch) cp_async16(xs + gram_xoff(r, c), src + 8 * c);
                else asm volatile("st.shared.v4.u32 [%0], {%1, %1, %1, %1};" ::"r"(xs + gram_xoff(r, c)), "r"(0u) : "memory");
            }
        } else {
            const float *src = d.x + (size_t)id * d.mp + 128 * kb;
            const int pc = min(128, (int)d.mp - 128 * kb) >> 2;   // float4 columns (d.mp is a multiple of 4)
#pragma unroll 1
            for (int c = 0; c < 16; c++) {
                float4 v0 = make_float4(0.f, 0.f, 0.f, 0.f), v1 = v0;
                if (2 * c < pc) v0 = *reinterpret_cast<const float4 *>(src + 8 * c);
                if (2 * c + 1 < pc) v1 = *reinterpret_cast<const float4 *>(src + 8 * c + 4);
                asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(xs + gram_xoff(r, c)),
                             "r"(pack_bf16(v0.x, v0.y)), "r"(pack_bf16(v0.z, v0.w)), "r"(pack_bf16(v1.x, v1.y)),
                             "r"(pack_bf16(v1.z, v1.w))
                             : "memory");
            }
        }
    }
    cp_async_wait_all();
    __syncwarp();
}

// RobustPrune on the Gram of rows of one 128-column block: same rule and order
// as warp_prune.  First the domination masks: row i's mask holds the later
// candidates j > i that i would drop (alpha^2 * d(i, j) <= rho(j)).  The 16-row
// stripes go from the last to the first, so that a stripe finds every norm it
// needs (the diagonal of its own and of later stripes) and turns its sums into
// mask bits where they are, in registers; a quad's lanes hold the columns of two
// rows, and lane k of it ends with one word of them.  The greedy pass is a
// warp-uniform walk over a 64-bit alive mask, from one candidate that drops
// something to the next; of what is left the first R are the result (a
// candidate drops only later ones, so those after the R-th change nothing).
// Bound by the instructions of one warp (12 to 16 warps an SM, each issuing every
// 7 to 9 cycles).  With the sums stored as a table that each lane then walked a
// row of, and a step of the walk per kept candidate, 300k repairs took 2.02 ms
// against 1.71, the offers of 10k inserts 1.13 against 1.06.
__device__ int warp_prune_gram(const Dev &d, const u64 *ck, int n, u32 *out_id, float *out_rho, Stage &st) {
    const int lane = lane_id();
    float2 *nr2 = reinterpret_cast<float2 *>(st.gram + (size_t)st.gram_rows * GRAM_RB);   // .x: the norms, .y: rho
    const int nm = (n + 15) >> 4, nn = (n + 7) >> 3;
    const u32 xs = smem_addr(st.gram), c0 = gram_c0(lane);
    const float alpha2 = d.alpha2;
    const bool l2 = d.metric == 0;
    const int cq = 2 * (lane & 3), rq = lane >> 2;
    const u64 in_n = n < 64 ? (1ull << n) - 1 : ~0ull;
    u32 mw[4] = {0u, 0u, 0u, 0u};
    for (int i = lane; i < n; i += 32) nr2[i].y = key_rho(ck[i]);
    gram_stage_rows(d, ck, 0, n, 0, xs);
    for (int mt = nm - 1; mt >= 0; mt--) {
        // tile t: rows 16 mt + .., columns 16 mt + 8 t + ..; rows past n hold
        // whatever the buffer held, and their bits are cleared below
        float acc[8][4];
#pragma unroll
        for (int b = 0; b < 8; b++)
#pragma unroll
            for (int c = 0; c < 4; c++) acc[b][c] = 0.f;
        const u32 xm = xs + (u32)(16 * mt + (lane & 7) + 8 * ((lane >> 3) & 1)) * GRAM_RB;
#pragma unroll
        for (int ks = 0; ks < 8; ks++) {
            u32 a0, a1, a2, a3;
            const u32 ko = (u32)(32 * ks) ^ c0;
            ldsm_x4(a0, a1, a2, a3, xm + ko);
#pragma unroll
            for (int t = 0; t < 8; t += 2) {
                if (2 * mt + t >= nn) continue;
                // matrices: (t, k 0-7), (t + 1, k 0-7), (t, k 8-15), (t + 1, k 8-15)
                u32 b0, b1, b2, b3;
                ldsm_x4(b0, b1, b2, b3, xm + (u32)(8 * t) * GRAM_RB + ko);
                mma_bf16_16816(acc[t], a0, a1, a2, a3, b0, b2);
                mma_bf16_16816(acc[t + 1], a0, a1, a2, a3, b1, b3);
            }
        }
        // the diagonal: entry (r, r) of rows rq in tile 0, of rows rq + 8 in tile 1
        const int r0 = 16 * mt + rq;
        if (cq == rq || cq + 1 == rq) {
            nr2[r0].x = cq == rq ? acc[0][0] : acc[0][1];
            nr2[r0 + 8].x = cq == rq ? acc[1][2] : acc[1][3];
        }
        __syncwarp();
        const float n0 = nr2[r0].x, n1 = nr2[r0 + 8].x;
        u32 m[2][2] = {{0u, 0u}, {0u, 0u}};   // row rq, row rq + 8: bits 8 t + h
#pragma unroll
        for (int t = 0; t < 8; t++) {
            if (2 * mt + t >= nn) continue;
            const float4 v = *reinterpret_cast<const float4 *>(nr2 + 16 * mt + 8 * t + cq);
            // (n_i - g) + (n_j - g): every intermediate stays as small as the result
            auto hit = [&](float ni, float g, float nj, float rho) {
                const float dd = l2 ? __fadd_rn(__fsub_rn(ni, g), __fsub_rn(nj, g)) : __fsub_rn(1.0f, g);
                return __fmul_rn(alpha2, dd) <= rho;
            };
            const u32 b = 1u << (8 * (t & 3));
            if (hit(n0, acc[t][0], v.x, v.y)) m[0][t >> 2] |= b;
            if (hit(n0, acc[t][1], v.z, v.w)) m[0][t >> 2] |= 2u * b;
            if (hit(n1, acc[t][2], v.x, v.y)) m[1][t >> 2] |= b;
            if (hit(n1, acc[t][3], v.z, v.w)) m[1][t >> 2] |= 2u * b;
        }
        // to columns of the whole list, then words (row rq + 8 (lane & 1), half
        // (lane >> 1) & 1)
        const u64 w0 = (((u64)m[0][1] << 32) | m[0][0]) << cq << (16 * mt);
        const u64 w1 = (((u64)m[1][1] << 32) | m[1][0]) << cq << (16 * mt);
        const bool odd = lane & 1, up = lane & 2;
        const u64 p = (odd ? w1 : w0) | __shfl_xor_sync(FULL, odd ? w0 : w1, 1);
        const u32 w = (u32)(up ? p >> 32 : p) | __shfl_xor_sync(FULL, (u32)(up ? p : p >> 32), 2);
        const u64 later = (~0ull << (r0 + 8 * (lane & 1)) << 1) & in_n;
        const u32 word = w & (u32)(up ? later >> 32 : later);
#pragma unroll
        for (int k = 0; k < 4; k++)
            if (k == mt) mw[k] = word;
    }
    __syncwarp();   // the rows are read: their last bytes take the masks
    u64 *dom = reinterpret_cast<u64 *>(st.gram + (size_t)st.gram_rows * GRAM_RB - GRAM_N * 8);
#pragma unroll
    for (int k = 0; k < 4; k++)
        if (k < nm) reinterpret_cast<u32 *>(dom + 16 * k + rq + 8 * (lane & 1))[(lane >> 1) & 1] = mw[k];
    __syncwarp();
    // equal adjacent keys collapse to one
    u64 live = 0ull, act = 0ull;
    for (int i0 = 0; i0 < n; i0 += 32) {
        const int i = i0 + lane;
        const u32 b = __ballot_sync(FULL, i < n && (i == 0 || ck[i] != ck[i - 1]));
        const u32 a = __ballot_sync(FULL, i < n && dom[i] != 0);
        live |= (u64)b << i0;
        act |= (u64)a << i0;
    }
    for (u64 todo = live & act; todo;) {
        const int head = __ffsll((long long)todo) - 1;
        todo &= todo - 1;
        const u64 m = ~dom[head];
        live &= m;
        todo &= m;
    }
    const int nout = min(__popcll(live), (int)d.R);
    for (int i0 = 0; i0 < n; i0 += 32) {
        const int i = i0 + lane;
        if (i < n && (live >> i & 1)) {
            const int pos = __popcll(live & ((1ull << i) - 1));
            const u64 hk = ck[i];
            if (pos < nout) {
                out_id[pos] = key_id(hk);
                out_rho[pos] = key_rho(hk);
            }
        }
    }
    __syncwarp();
    return nout;
}
// ---------------------------------------------------------------------------
// The cooperative Gram: the domination masks of up to GRAM_NL candidates with
// rows of any length, by the block's four warps.  The first warp runs the
// kernel; the others wait for its requests.  The rows are staged once, 128
// columns at a time and the next block while this one is multiplied; the
// upper triangle's 16-row stripes are split over the warps (stripes w and nm -
// 1 - w together hold about as many tiles for every w) and their sums stay in
// registers.  Each entry (i, j), j > i, then becomes bit j of row i's mask
// (alpha^2 * d(i, j) <= rho(j)); squared L2 is (G_ii - G_ij) + (G_jj - G_ij),
// inner product 1 - G_ij.  BLOCKSUM: each column block's products are summed
// from zero and added to the total (the form of candidate lists of up to
// GRAM_N), else one chain runs over all columns.
// Bound by the row reads (L2) and the mma.sync chains.  A warp per item that
// restaged every column block for each stripe, or kept its sums in shared
// memory, held 5 warps per SM: 500 deletes of 768-d with R = 64 (32,000 pairs)
// took 6.7 ms against 2.4, the offers of 500 inserts 2.3 against 1.5.
// ---------------------------------------------------------------------------
struct GramReq {
    const u64 *ck;
    int n;
};
__device__ __forceinline__ void coop_bar() { asm volatile("bar.sync 1, 128;" ::: "memory"); }   // 32 COOP_WARPS
// The (norm, rho) pairs and masks of a buffer of `rows` candidates.
__device__ __forceinline__ char *gram_tail(char *buf, u32 rows, u32 mp) { return buf + gram_row_bytes(rows, mp); }

template <bool BLOCKSUM>
__device__ __forceinline__ void gram_masks(const Dev &d, const u64 *ck, int n, char *buf, u32 rows) {
    constexpr int T0 = BLOCKSUM ? 8 : 16, T1 = BLOCKSUM ? 1 : 8;   // tiles of a warp's first and second stripe
    const int tid = threadIdx.x, warp = tid >> 5, lane = lane_id();
    float2 *nr2 = reinterpret_cast<float2 *>(gram_tail(buf, rows, d.mp));   // .x: the norms, .y: rho
    u64 *dom = reinterpret_cast<u64 *>(nr2 + rows);
    const int nm = (n + 15) >> 4, nn = 2 * nm, nkb = ((int)d.mp + 127) >> 7;
    // BLOCKSUM: at most four stripes, one a warp
    const int s0 = warp, s1 = nm - 1 - warp;
    const bool has0 = BLOCKSUM ? s0 < nm : s0 <= s1, has1 = !BLOCKSUM && s0 < s1;
    const u32 blk = (u32)rows * GRAM_RS_CO * 2;
    auto stage = [&](int kb) {
        const u32 xs = smem_addr(buf) + (kb & 1) * blk;
        const int c = tid & 15;
        const bool in = 128 * kb + 8 * c < (int)d.mb;   // d.mb is a multiple of 8
        for (int r = tid >> 4; r < n; r += 2 * COOP_WARPS) {
            const u32 dst = xs + (u32)(r * GRAM_RS_CO * 2 + 16 * c);
            if (in) cp_async16(dst, d.xb + (size_t)key_id(ck[r]) * d.mb + 128 * kb + 8 * c);
            else asm volatile("st.shared.v4.u32 [%0], {%1, %1, %1, %1};" ::"r"(dst), "r"(0u) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float a0[T0][4], a1[T1][4], t0[BLOCKSUM ? T0 : 1][4];
#pragma unroll
    for (int t = 0; t < T0; t++)
#pragma unroll
        for (int c = 0; c < 4; c++) a0[t][c] = 0.f;
#pragma unroll
    for (int t = 0; t < T1; t++)
#pragma unroll
        for (int c = 0; c < 4; c++) a1[t][c] = 0.f;
    if (tid < n) nr2[tid].y = key_rho(ck[tid]);
    stage(0);
    for (int kb = 0; kb < nkb; kb++) {
        if (kb + 1 < nkb) {
            stage(kb + 1);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        coop_bar();
        const u32 xs = smem_addr(buf) + (kb & 1) * blk;
        // one stripe: tiles 2 mt + t, t < NT (two at a time), rows past n hold anything
        auto stripe = [&](auto &acc, auto nt_c, int mt) {
            constexpr int NT = decltype(nt_c)::value;
#pragma unroll
            for (int ks = 0; ks < 8; ks++) {
                u32 x0, x1, x2, x3;
                const int ar = 16 * mt + (lane & 7) + 8 * ((lane >> 3) & 1), ac = 16 * ks + 8 * (lane >> 4);
                ldsm_x4(x0, x1, x2, x3, xs + (u32)((ar * GRAM_RS_CO + ac) * 2));
#pragma unroll
                for (int t = 0; t < NT; t += 2) {
                    if (2 * mt + t >= nn) continue;
                    u32 b0, b1, b2, b3;
                    const int br = 8 * (2 * mt + t) + (lane & 7) + 8 * (lane >> 4);
                    const int bc = 16 * ks + 8 * ((lane >> 3) & 1);
                    ldsm_x4(b0, b1, b2, b3, xs + (u32)((br * GRAM_RS_CO + bc) * 2));
                    mma_bf16_16816(acc[t], x0, x1, x2, x3, b0, b1);
                    mma_bf16_16816(acc[t + 1], x0, x1, x2, x3, b2, b3);
                }
            }
        };
        if (BLOCKSUM) {
            if (has0) {
#pragma unroll
                for (int t = 0; t < T0; t++)
#pragma unroll
                    for (int c = 0; c < 4; c++) t0[BLOCKSUM ? t : 0][c] = 0.f;
                stripe(t0, std::integral_constant<int, BLOCKSUM ? T0 : 0>{}, s0);
#pragma unroll
                for (int t = 0; t < T0; t++)
#pragma unroll
                    for (int c = 0; c < 4; c++)
                        a0[t][c] = kb == 0 ? t0[BLOCKSUM ? t : 0][c] : __fadd_rn(a0[t][c], t0[BLOCKSUM ? t : 0][c]);
            }
        } else {
            if (has0) stripe(a0, std::integral_constant<int, T0>{}, s0);
            if (has1) stripe(a1, std::integral_constant<int, BLOCKSUM ? 0 : T1>{}, s1);
        }
        coop_bar();   // this half is read
    }
    // the diagonal: entry (r, r) sits in tile 2 mt (rows r0) or 2 mt + 1 (rows r0 + 8)
    const int cq = 2 * (lane & 3), rq = lane >> 2;
    auto diag = [&](auto &acc, int mt) {
        const int r0 = 16 * mt + rq, r1 = r0 + 8;
        if (cq == rq || cq + 1 == rq) {
            if (r0 < n) nr2[r0].x = cq == rq ? acc[0][0] : acc[0][1];
            if (r1 < n) nr2[r1].x = cq == rq ? acc[1][2] : acc[1][3];
        }
    };
    if (has0) diag(a0, s0);
    if constexpr (!BLOCKSUM)
        if (has1) diag(a1, s1);
    coop_bar();
    auto masks = [&](auto &acc, auto nt_c, int mt) {
        constexpr int NT = decltype(nt_c)::value;
        const int r0 = 16 * mt + rq, r1 = r0 + 8;
        const float n0 = r0 < n ? nr2[r0].x : 0.f, n1 = r1 < n ? nr2[r1].x : 0.f;
        u64 m0l = 0, m0h = 0, m1l = 0, m1h = 0;
#pragma unroll
        for (int t = 0; t < NT; t++) {
            const int nt = 2 * mt + t;
            if (nt >= nn) continue;
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const int c = 8 * nt + cq + h;
                if (c >= n) continue;
                const float2 v = nr2[c];
                auto hit = [&](float nr, float g) {
                    const float dd = d.metric == 0 ? __fadd_rn(__fsub_rn(nr, g), __fsub_rn(v.x, g)) : __fsub_rn(1.0f, g);
                    return __fmul_rn(d.alpha2, dd) <= v.y;
                };
                const u64 bit = 1ull << (c & 63);
                if (c > r0 && hit(n0, acc[t][h])) { if (c < 64) m0l |= bit; else m0h |= bit; }
                if (c > r1 && hit(n1, acc[t][2 + h])) { if (c < 64) m1l |= bit; else m1h |= bit; }
            }
        }
        // the four lanes of a quad hold the columns of a row
#pragma unroll
        for (int o = 1; o <= 2; o <<= 1) {
            m0l |= __shfl_xor_sync(FULL, m0l, o);
            m0h |= __shfl_xor_sync(FULL, m0h, o);
            m1l |= __shfl_xor_sync(FULL, m1l, o);
            m1h |= __shfl_xor_sync(FULL, m1h, o);
        }
        if ((lane & 3) == 0) {
            if (r0 < n) { dom[2 * r0] = m0l; dom[2 * r0 + 1] = m0h; }
            if (r1 < n) { dom[2 * r1] = m1l; dom[2 * r1 + 1] = m1h; }
        }
    };
    if (has0) masks(a0, std::integral_constant<int, T0>{}, s0);
    if constexpr (!BLOCKSUM)
        if (has1) masks(a1, std::integral_constant<int, T1>{}, s1);
    coop_bar();
}

// The canonical sums of 64 values a lane holds as partials (value p in v[p]):
// the tree of canon_dist over the 32 lanes, where at each level a lane keeps
// half of the values it still has and passes the other half on.  Lane l ends
// with values 2 l and 2 l + 1 in v[0] and v[1].
__device__ __forceinline__ void warp_tree64(float (&v)[64]) {
    const int lane = lane_id();
#pragma unroll
    for (int h = 16, n = 32; h >= 1; h >>= 1, n >>= 1) {
        const bool up = lane & h;
#pragma unroll
        for (int i = 0; i < n; i++)
            v[i] = __fadd_rn(up ? v[i + n] : v[i], __shfl_xor_sync(FULL, up ? v[i] : v[i + n], h));
    }
}

// Canonical distances of the 64 pairs of 8 rows and 8 rows, by one warp: lane j
// sums partial j of every pair.  Lane l returns pairs 2 l and 2 l + 1 (pair 8 i
// + j: rows xr[i], yr[j]).
__device__ __forceinline__ void pair_tile(u32 mp, u32 metric, const float *const (&xr)[8], const float *const (&yr)[8],
                                          float (&dd)[2]) {
    float acc[64];
#pragma unroll
    for (int q = 0; q < 64; q++) acc[q] = 0.0f;
    for (u32 e = 4 * lane_id(); e < mp; e += 128) {
        float4 x[8], y[8];
#pragma unroll
        for (int c = 0; c < 8; c++) {
            x[c] = *reinterpret_cast<const float4 *>(xr[c] + e);
            y[c] = *reinterpret_cast<const float4 *>(yr[c] + e);
        }
        if (metric == 0) {
#pragma unroll
            for (int q = 0; q < 64; q++) {
                const float4 u = x[q >> 3], v = y[q & 7];
                const float d0 = __fsub_rn(u.x, v.x), d1 = __fsub_rn(u.y, v.y);
                const float d2 = __fsub_rn(u.z, v.z), d3 = __fsub_rn(u.w, v.w);
                acc[q] = __fmaf_rn(d3, d3, __fmaf_rn(d2, d2, __fmaf_rn(d1, d1, __fmaf_rn(d0, d0, acc[q]))));
            }
        } else {
#pragma unroll
            for (int q = 0; q < 64; q++) {
                const float4 u = x[q >> 3], v = y[q & 7];
                acc[q] = __fmaf_rn(u.w, v.w, __fmaf_rn(u.z, v.z, __fmaf_rn(u.y, v.y, __fmaf_rn(u.x, v.x, acc[q]))));
            }
        }
    }
    __syncwarp();
    warp_tree64(acc);
#pragma unroll
    for (int k = 0; k < 2; k++) dd[k] = metric == 0 ? acc[k] : __fsub_rn(1.0f, acc[k]);
}
// Tile t of the upper triangle, rows of tiles: t = ty (ty + 1) / 2 + tx, tx <= ty.
__device__ __forceinline__ void tile_of(int t, int &tx, int &ty) {
    for (ty = 0, tx = t; tx > ty;) tx -= ++ty;
}

// The same masks from canonical fp32 distances (variant 3), in 8 x 8 tiles of
// pairs, a warp per tile.  Every pair's distance, where a greedy walk computes
// only those of the heads it keeps: but at a third of the instructions each and
// with no head waiting for the one before.
__device__ __noinline__ void canon_masks(const float *x0, u32 mp, u32 metric, float alpha2, const u64 *ck, int n,
                                         u64 *dom) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = lane_id();
    unsigned char *dom8 = reinterpret_cast<unsigned char *>(dom);   // byte 16 x + ty: columns 8 ty .. of row x
    for (int i = tid; i < 2 * n; i += 32 * COOP_WARPS) dom[i] = 0ull;
    coop_bar();
    const int nt = (n + 7) >> 3;
    for (int t = warp; t < nt * (nt + 1) / 2; t += COOP_WARPS) {
        int tx, ty;
        tile_of(t, tx, ty);
        const float *xr[8], *yr[8];
#pragma unroll
        for (int c = 0; c < 8; c++) {   // past the list: a valid row again
            xr[c] = x0 + (size_t)key_id(ck[min(8 * tx + c, n - 1)]) * mp;
            yr[c] = x0 + (size_t)key_id(ck[min(8 * ty + c, n - 1)]) * mp;
        }
        float dd[2];
        pair_tile(mp, metric, xr, yr, dd);
        u32 bits = 0;
        const int x = 8 * tx + (lane >> 2);   // pairs 2 lane, 2 lane + 1 share a row
#pragma unroll
        for (int k = 0; k < 2; k++) {
            const int j = 2 * (lane & 3) + k, y = 8 * ty + j;
            if (x < y && y < n && __fmul_rn(alpha2, dd[k]) <= key_rho(ck[y])) bits |= 1u << j;
        }
        bits |= __shfl_xor_sync(FULL, bits, 1);
        bits |= __shfl_xor_sync(FULL, bits, 2);
        if ((lane & 3) == 0 && x < n) dom8[16 * x + ty] = (unsigned char)bits;
    }
    coop_bar();
}

// The domination masks of variant GV, by the whole block.
template <int GV>
__device__ __forceinline__ void coop_masks(const Dev &d, const u64 *ck, int n, char *buf, u32 rows) {
    if constexpr (GV == 3) canon_masks(d.x, d.mp, d.metric, d.alpha2, ck, n, reinterpret_cast<u64 *>(buf + GRAM_NL * 8));
    else gram_masks<GV == 2>(d, ck, n, buf, rows);
}

// The helper warps of a block: serve requests until one has n < 0.
template <int GV>
__device__ __noinline__ void gram_helper(const Dev d, char *buf, u32 rows, const GramReq *req) {
    for (;;) {
        coop_bar();
        const int n = *reinterpret_cast<const volatile int *>(&req->n);
        if (n < 0) return;
        coop_masks<GV>(d, *reinterpret_cast<const u64 *const volatile *>(&req->ck), n, buf, rows);
    }
}
__device__ __forceinline__ void gram_release(GramReq *req) {
    if (lane_id() == 0) req->n = -1;
    __syncwarp();
    coop_bar();
}

// RobustPrune from the masks (first warp): a walk over a 128-bit alive mask.
template <int GV>
__device__ int warp_prune_masks(const Dev &d, const u64 *ck, int n, u32 *out_id, float *out_rho, Stage &st) {
    const int lane = lane_id();
    __syncwarp();
    if (lane == 0) {
        st.req->ck = ck;
        st.req->n = n;
    }
    __syncwarp();
    coop_bar();
    coop_masks<GV>(d, ck, n, st.gram, st.gram_tag);
    const u64 *dom = reinterpret_cast<const u64 *>(gram_tail(st.gram, st.gram_tag, d.mp) + (size_t)st.gram_rows * 8);
    // equal adjacent keys collapse to one
    u64 lo = 0, hi = 0;
    for (int i0 = 0; i0 < n; i0 += 32) {
        const int i = i0 + lane;
        const u64 b = __ballot_sync(FULL, i < n && (i == 0 || ck[i] != ck[i - 1]));
        if (i0 < 64) lo |= b << i0; else hi |= b << (i0 - 64);
    }
    int nout = 0;
    const int R = (int)d.R;
    while (nout < R && (lo | hi)) {
        const int head = lo ? __ffsll((long long)lo) - 1 : 64 + __ffsll((long long)hi) - 1;
        if (head < 64) lo &= lo - 1; else hi &= hi - 1;
        if (lane == 0) {
            const u64 hk = ck[head];
            out_id[nout] = key_id(hk);
            out_rho[nout] = key_rho(hk);
        }
        nout++;
        lo &= ~dom[2 * head];
        hi &= ~dom[2 * head + 1];
    }
    __syncwarp();
    return nout;
}

// ---------------------------------------------------------------------------
// RobustPrune over n candidates whose keys ck[0..n) are sorted ascending
// (rho = distance to the owner).  Equal adjacent keys collapse to one.  The
// head is kept; every later candidate p' with alpha^2 * d(head, p') <= rho(p')
// is dropped; stop at R.  Distances between candidates are canonical
// distances, 8 lanes per distance, rows taken from the stage when staged.
// Scratch: alive[n], idx[n].
// ---------------------------------------------------------------------------
// GV, the Gram variant of a kernel: 0, a buffer of at most GRAM_N rows with
// rows of one 128-column block, a warp per item; 1, more than GRAM_N rows, and
// 2, at most GRAM_N rows spanning several blocks: the block's four warps on one
// item (see gram_masks); 3, the same on canonical distances (see canon_masks); 4,
// canonical distances by a warp per item, in a kernel without the Gram's code.
template <int GV>
__device__ int warp_prune(const Dev &d, const u64 *ck, int n, unsigned char *alive, u32 *idx, u32 *out_id,
                          float *out_rho, Stage &st) {
    if (GV != 4 && st.gram && n <= st.gram_rows) {
        if constexpr (coop_variant(GV)) return warp_prune_masks<GV>(d, ck, n, out_id, out_rho, st);
        else return warp_prune_gram(d, ck, n, out_id, out_rho, st);
    }
    const int lane = lane_id();
    const int grp = lane >> 3, g = lane & 7;
    const int ns = st.rows ? min(n, st.ns_cap) : 0;
    stage_rows(d, st, ck, ns);
    for (int i = lane; i < n; i += 32) alive[i] = (i == 0 || ck[i] != ck[i - 1]) ? 1 : 0;
    __syncwarp();
    auto row = [&](int i) -> const float * {
        return i < ns ? st.rows + (size_t)i * d.mp : d.x + (size_t)key_id(ck[i]) * d.mp;
    };
    int nout = 0, start = 0;
    const int R = (int)d.R;
    while (nout < R) {
        int head = -1;
        for (int i0 = start; i0 < n; i0 += 32) {
            int i = i0 + lane;
            u32 m = __ballot_sync(FULL, i < n && alive[i]);
            if (m) { head = i0 + __ffs(m) - 1; break; }
        }
        if (head < 0) break;
        const u64 hk = ck[head];
        if (lane == 0) { out_id[nout] = key_id(hk); out_rho[nout] = key_rho(hk); }
        nout++;
        if (nout == R) break;
        int m_cnt = 0;
        for (int i0 = head + 1; i0 < n; i0 += 32) {
            int i = i0 + lane;
            bool ok = i < n && alive[i];
            u32 m = __ballot_sync(FULL, ok);
            if (ok) idx[m_cnt + __popc(m & lanemask_lt())] = (u32)i;
            m_cnt += __popc(m);
        }
        __syncwarp();
        const float *hrow = row(head);
        if (d.mp <= 128) {
            // the head's four float4 per lane stay in registers
            float4 hr[4];
            canon_row_q8(hrow, (int)d.mp, g, hr);
            for (int r0 = 0; r0 < m_cnt; r0 += 4) {
                const int c = r0 + grp;
                const int cc = c < m_cnt ? c : m_cnt - 1;
                const u32 j = idx[cc];
                const u64 kj = ck[j];
                float4 v[4];
                canon_row_q8(row((int)j), (int)d.mp, g, v);
                const float dd = canon_dist_q8v(hr, v, (int)d.mp, (int)d.metric, g);
                if (c < m_cnt && g == 0 && __fmul_rn(d.alpha2, dd) <= key_rho(kj)) alive[j] = 0;
            }
        } else {
            for (int r0 = 0; r0 < m_cnt; r0 += 4) {
                const int c = r0 + grp;
                const int cc = c < m_cnt ? c : m_cnt - 1;
                const u32 j = idx[cc];
                const u64 kj = ck[j];
                float dd = canon_dist<8>(hrow, row((int)j), (int)d.mp, (int)d.metric, g);
                if (c < m_cnt && g == 0 && __fmul_rn(d.alpha2, dd) <= key_rho(kj)) alive[j] = 0;
            }
        }
        __syncwarp();
        start = head + 1;
    }
    __syncwarp();
    return nout;
}

// Load N(u) into shared memory; returns the degree and the snapshot word.
__device__ __forceinline__ int load_list(const Dev &d, u32 u, u32 *ids, float *rho, u64 &snap) {
    const int lane = lane_id();
    u64 r = 0;
    if (lane == 0) r = ld_ref(d, u);
    r = __shfl_sync(FULL, r, 0);
    snap = r;
    const u32 s = ref_slab(r);
    const int n = s == NIL ? 0 : (int)ref_deg(r);
    for (int j = lane; j < n; j += 32) {
        uint2 e = d.slab[(size_t)s * d.R + j];
        ids[j] = e.x;
        rho[j] = __uint_as_float(e.y);
    }
    __syncwarp();
    return n;
}

__device__ __forceinline__ bool warp_same_list(const u32 *a, const float *ar, int na, const u32 *b,
                                               const float *br, int nb) {
    if (na != nb) return false;
    const int lane = lane_id();
    bool diff = false;
    for (int j = lane; j < na; j += 32)
        diff |= (a[j] != b[j]) || (__float_as_uint(ar[j]) != __float_as_uint(br[j]));
    return __ballot_sync(FULL, diff) == 0;
}

__device__ __forceinline__ bool warp_contains(const u32 *ids, int n, u32 v) {
    bool hit = false;
    for (int j = lane_id(); j < n; j += 32) hit |= ids[j] == v;
    return __ballot_sync(FULL, hit) != 0;
}

// Canonical distances of row v to the nl rows keys[i + (i >= below)], into dv.
__device__ __noinline__ void canon_row_dists(const float *x0, u32 mp, u32 metric, const u64 *keys, int nl, int below,
                                             u32 v, float *dv) {
    const int lane = lane_id(), grp = lane >> 3, g = lane & 7;
    const float *xv = x0 + (size_t)v * mp;
    auto row_of = [&](int i) {
        i = min(i, nl - 1);
        return x0 + (size_t)key_id(keys[i + (i >= below)]) * mp;
    };
    if (mp <= 128) {
        float4 q[4];
        canon_row_q8(xv, (int)mp, g, q);
        for (int r0 = 0; r0 < nl; r0 += 8) {
            float4 x[4], y[4];
            canon_row_q8(row_of(r0 + grp), (int)mp, g, x);
            canon_row_q8(row_of(r0 + 4 + grp), (int)mp, g, y);
            const float da = canon_dist_q8v(q, x, (int)mp, (int)metric, g);
            const float db = canon_dist_q8v(q, y, (int)mp, (int)metric, g);
            if (g == 0 && r0 + grp < nl) dv[r0 + grp] = da;
            if (g == 0 && r0 + 4 + grp < nl) dv[r0 + 4 + grp] = db;
        }
    } else {
        const float one[4] = {1.0f, 1.0f, 1.0f, 1.0f};
        for (int r0 = 0; r0 < nl; r0 += 4) {
            const void *row[4];
#pragma unroll
            for (int c = 0; c < 4; c++) row[c] = row_of(r0 + c);
            const float dd = warp_dists<0, 4, 2>(xv, row, one, (int)mp, (int)metric);
            if (g == 0 && r0 + grp < nl) dv[r0 + grp] = dd;
        }
    }
    __syncwarp();
}

// Apply one offer (v, rho) to the list in place (Algorithm 2, reverse edge):
// a present id is a no-op; below R the entry is inserted in (rho, id) order;
// at R the list is RobustPrune(list + v) about the owner (tombstones drop).
// Scratch: keys[np], alive[np], idx[np] with np >= R + 1 (power of two).
template <int GV>
// pruned: in, whether the list is a RobustPrune output (no entry dropped by
// an earlier one, see ref_pruned); out, the same for the returned list.
__device__ int apply_offer(const Dev &d, u32 *ids, float *rho, int n, u32 v, float vr, u64 *keys,
                           unsigned char *alive, u32 *idx, int np, u32 *oid, float *orho, Stage &st, bool &pruned) {
    const int lane = lane_id();
    if (warp_contains(ids, n, v)) return n;
    const u64 kv = mkkey(vr, v);
    if (n < (int)d.R) {
        pruned = false;   // a plain insertion: v is not checked against the entries
        int pos = 0;
        for (int j0 = 0; j0 < n; j0 += 32) {
            int j = j0 + lane;
            pos += __popc(__ballot_sync(FULL, j < n && mkkey(rho[j], ids[j]) < kv));
        }
        u32 tid[2];
        float tr[2];
        int c = 0;
        for (int j = pos + lane; j < n; j += 32, c++) { tid[c] = ids[j]; tr[c] = rho[j]; }
        __syncwarp();
        c = 0;
        for (int j = pos + lane; j < n; j += 32, c++) { ids[j + 1] = tid[c]; rho[j + 1] = tr[c]; }
        if (lane == 0) { ids[pos] = v; rho[pos] = vr; }
        __syncwarp();
        return n + 1;
    }
    // the list is sorted by (rho, id) and holds no v: the candidates in order
    // are its live entries with v placed at its rank
    int nl = 0, below = 0;
    for (int i0 = 0; i0 < n; i0 += 32) {
        const int i = i0 + lane;
        u64 k = KEY_INF;
        bool live = false;
        if (i < n) {
            k = mkkey(rho[i], ids[i]);
            live = !ref_del(ld_ref(d, ids[i]));
        }
        const u32 lm = __ballot_sync(FULL, live);
        const int pos = nl + __popc(lm & lanemask_lt()) + (k > kv ? 1 : 0);
        if (live) keys[pos] = k;
        below += __popc(__ballot_sync(FULL, live && k < kv));
        nl += __popc(lm);
    }
    // A full list of live entries that no earlier entry drops, with v after
    // all of them: the prune keeps the R entries in order and stops before v.
    st.wk_state += 8ull * n;                 // the entries' reference words
    if (pruned && nl == n && below == nl) return n;
    if (lane == 0) keys[below] = kv;
    __syncwarp();
    const int cn = nl + 1;
    st.wk_rows += prune_row_bytes(d, st, cn);
    // No entry of a pruned list drops a later one: only v's tests are open.
    // The entries before it may drop it, else it may drop those after it.
    // Canonical variants only: 32 distances where the greedy walk computes 528
    // (rounds of 100 + 100 on 10k x 128, deterministic: the offers 258 -> 76 us).
    // On the Gram tile the same short cut was no faster: what bounds an offer
    // there is its chain of loads, fence and compare-and-swap; and in variant 0
    // the code alone costs the lock-free folds a quarter (128 -> 161 registers),
    // so larger canonical launches have variant 4 (deterministic loads of 44k x
    // 120 and 125k x 42 rows 126 -> 75 and 189 -> 120 ms).
    if (GV >= 3 && pruned && d.same_tests) {
        float *dv = reinterpret_cast<float *>(idx);
        canon_row_dists(d.x, d.mp, d.metric, keys, nl, below, v, dv);
        bool lost = false;
        for (int i = lane; i < below; i += 32) lost |= __fmul_rn(d.alpha2, dv[i]) <= vr;
        const bool drop_v = __any_sync(FULL, lost);
        int nout = 0;
        for (int i0 = 0; i0 < cn; i0 += 32) {   // positions of the merged list
            const int i = i0 + lane;
            bool keep = false;
            u64 k = 0;
            if (i < cn) {
                k = keys[i];
                keep = i < below || (i == below ? !drop_v : drop_v || !(__fmul_rn(d.alpha2, dv[i - 1]) <= key_rho(k)));
            }
            const u32 m = __ballot_sync(FULL, keep);
            const int pos = nout + __popc(m & lanemask_lt());
            if (keep && pos < (int)d.R) {
                ids[pos] = key_id(k);
                rho[pos] = key_rho(k);
            }
            nout += __popc(m);
        }
        __syncwarp();
        return min(nout, (int)d.R);
    }
    int nout = warp_prune<GV>(d, keys, cn, alive, idx, oid, orho, st);
    for (int j = lane; j < nout; j += 32) { ids[j] = oid[j]; rho[j] = orho[j]; }
    __syncwarp();
    pruned = true;
    return nout;
}

// ---------------------------------------------------------------------------
// Forward edges: F_v = RobustPrune(C_v) with C_v the expanded non-tombstone
// nodes of v's search (nearest max_cand); Publish(v, F_v); emit offers.
// ---------------------------------------------------------------------------
// The Gram rows of a launch whose prunes see at most max_n candidates.  Without
// the Gram, variant 3 for rows of more than 128 floats, and for shorter ones while
// the items leave SMs idle: its blocks hold three items per SM where one-warp
// blocks hold up to 16, but an item's prune takes a tenth of the time, at 768-d
// less.  40k x 768, R = 64, rounds of 1,000 + 1,000: the repair fold 83 ms with a
// warp per item, 21 with variant 3, the offers 38 and 3.0; 100k x 128, R = 32, of
// 2,000 + 2,000: the repair fold 2.84 (variant 4) and 2.90, the offers 0.40 and 0.83.
inline u32 prune_rows_for(const Dev &d, u32 max_n, u64 items, int num_sms) {
    if (d.gram) return gram_rows_for(d.gram, max_n);
    return max_n <= (u32)GRAM_NL && (d.mp > 128 || items <= 64ull * num_sms) ? CANON_ROWS : 0u;
}
struct PruneInsArgs {
    Dev d;
    u32 first, b;
    const u64 *exp_keys;
    const u32 *exp_count;
    u32 max_hops, max_cand, np, ns, gram;
    u32 rescore;   // the search ran on a reduced-precision copy: rescore in fp32
    u32 *F_id;
    float *F_rho;
    u32 *F_n;
    Offers of;
};

__host__ __device__ inline size_t prune_ins_scratch(u32 np, u32 R) {
    return al16(np) + al16((size_t)np * 4) + 2 * al16((size_t)R * 4);
}
__host__ __device__ inline size_t prune_ins_warp_bytes(u32 np, u32 R, u32 ns, u32 mp, u32 gram) {
    const size_t sc = prune_ins_scratch(np, R);
    return stage_bytes(ns, mp) + al16((size_t)np * 8) + (gram_alias(gram, sc) ? 0 : sc) + gram_bytes(gram, mp);
}

// one-warp blocks of the single-warp variant (GV 0) are held to 16 resident warps
// per SM (at most 128 registers a thread)
template <int GV>
__global__ void __launch_bounds__(GV ? 32 * COOP_WARPS : 32, GV ? 3 : 16) prune_insert_kernel(PruneInsArgs a) {
    extern __shared__ __align__(16) char smem[];
    __shared__ GramReq req;
    const int lane = lane_id();
    const Dev &d = a.d;
    const u32 R = d.R;
    char *p = smem;
    char *gbuf = a.gram ? p : nullptr;
    if (GV != 0 && threadIdx.x >= 32) return gram_helper<GV>(d, gbuf, a.gram, &req);
    p += gram_bytes(a.gram, d.mp);
    Stage st = stage_init(p, a.ns, d.mp, gbuf, a.gram, &req);
    WarpSlabs ws;
    ws_init(ws);
    p += stage_bytes(a.ns, d.mp);
    u64 *keys = reinterpret_cast<u64 *>(p); p += al16((size_t)a.np * 8);
    if (gram_alias(a.gram, prune_ins_scratch(a.np, R))) p = gbuf;
    unsigned char *alive = reinterpret_cast<unsigned char *>(p); p += al16(a.np);
    u32 *idx = reinterpret_cast<u32 *>(p); p += al16((size_t)a.np * 4);
    u32 *oid = reinterpret_cast<u32 *>(p); p += al16((size_t)R * 4);
    float *orho = reinterpret_cast<float *>(p);
    u32 t_next = 0;   // the next item's claim, in flight while this one runs
    if (lane == 0) t_next = (u32)atomicAdd(&d.ctr[C_WORK], 1ull);
    for (;;) {
        const u32 t = __shfl_sync(FULL, t_next, 0);
        if (t >= a.b) break;
        if (lane == 0) t_next = (u32)atomicAdd(&d.ctr[C_WORK], 1ull);
        const u32 cnt = a.exp_count[t];
        for (u32 i = lane; i < a.np; i += 32) keys[i] = i < cnt ? a.exp_keys[(size_t)t * a.max_hops + i] : KEY_INF;
        __syncwarp();
        warp_sort_u64(keys, (int)a.np);
        const int n = (int)min(cnt, a.max_cand);
        const u32 v = dev_first(d, a.first) + t;
        if (a.rescore) {
            // the nearest max_cand by the search's reduced-precision distance,
            // re-scored with the canonical fp32 distance to v and re-sorted,
            // so that RobustPrune and every stored rho see exact distances
            const float *xv = d.x + (size_t)v * d.mp;
            const float one[4] = {1.0f, 1.0f, 1.0f, 1.0f};
            for (int r0 = 0; r0 < n; r0 += 4) {
                const void *row[4];
#pragma unroll
                for (int c = 0; c < 4; c++) row[c] = d.x + (size_t)key_id(keys[min(r0 + c, n - 1)]) * d.mp;
                const float dist = warp_dists<0, 4, 2>(xv, row, one, (int)d.mp, (int)d.metric);
                const int i = r0 + (lane >> 3);
                __syncwarp();
                if (i < n && (lane & 7) == 0) keys[i] = mkkey(dist, key_id(keys[i]));
                __syncwarp();
            }
            for (u32 i = n + lane; i < a.np; i += 32) keys[i] = KEY_INF;
            __syncwarp();
            warp_sort_u64(keys, (int)a.np);
        }
        // rows: the candidates (fp32 for the re-score, with v's own row)
        st.wk_rows += a.rescore ? (u64)(n + 1) * 4 * d.mp : prune_row_bytes(d, st, n);
        const int nout = warp_prune<GV>(d, keys, n, alive, idx, oid, orho, st);
        u64 snap = 0;
        if (lane == 0) snap = ld_ref(d, v);
        snap = __shfl_sync(FULL, snap, 0);
        st.wk_state += 8 + 8ull * nout + 8;     // v's word read, its list and word written
        if (!warp_publish(d, ws, v, oid, orho, nout, snap, true) && lane == 0)
            atomicOr(&d.ctr[C_ERR], (u64)ERR_CAS);
        const u32 invalid = (u32)d.capacity;
        for (u32 j = lane; j < R; j += 32) {
            const size_t o = (size_t)t * R + j;
            const bool ok = (int)j < nout;
            a.F_id[o] = ok ? oid[j] : NIL;
            a.F_rho[o] = ok ? orho[j] : 0.0f;
            a.of.key[o] = ok ? oid[j] : invalid;
            a.of.val[o] = (u32)o;
            a.of.src[o] = v;
            a.of.rho[o] = ok ? orho[j] : 0.0f;
        }
        if (lane == 0) a.F_n[t] = (u32)nout;
        __syncwarp();
    }
    if (GV != 0) gram_release(&req);
    ws_finish(d, ws);
    stage_done(d, st, WK_PRUNE);
}

cudaError_t launch_prune_insert(const Dev &d, u32 first, u32 b, const u64 *exp_keys, const u32 *exp_count,
                                u32 max_hops, u32 max_cand, u32 *F_id, float *F_rho, u32 *F_n,
                                const Offers &of, int num_sms, cudaStream_t st, bool rescore) {
    if (b == 0) return cudaSuccess;
    // the Gram tile covers the prune only when every candidate fits in it
    const u32 gram = prune_rows_for(d, max_cand, b, num_sms);
    PruneInsArgs a{d, first, b, exp_keys, exp_count, max_hops, max_cand, 0, 0, gram, rescore ? 1u : 0u,
                   F_id, F_rho, F_n, of};
    u32 np = 32;
    while (np < max_hops) np <<= 1;
    a.np = np;
    a.ns = gram ? 0 : stage_cap(d.mp, max_cand, d.stage_bytes);
    const size_t wb = prune_ins_warp_bytes(np, d.R, a.ns, d.mp, gram);
    const size_t smem = wb;
    const int threads = block_threads(a.gram, d.mp);
    const void *fns[4] = {(const void *)prune_insert_kernel<0>, (const void *)prune_insert_kernel<1>, (const void *)prune_insert_kernel<2>,
                          (const void *)prune_insert_kernel<3>};
    const void *fn = fns[gram_variant(a.gram, d.mp)];
    cudaError_t e = smem_at_least((const void *)fn, smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        &per_sm, fn, threads, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    u32 blocks = (u32)(per_sm * num_sms), need = b;
    if (blocks > need) blocks = need;
    e = cudaMemsetAsync(d.ctr + C_WORK, 0, sizeof(u64), st);
    if (e != cudaSuccess) return e;
    void *args[] = {&a};
    e = cudaLaunchKernel(fn, dim3(blocks), dim3(threads), args, smem, st);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Reverse offers.  Deterministic: one warp per target segment, offers in
// ascending source order, one publish.  Lock-free: one warp per offer,
// CAS-published with retries up to `budget` (Algorithm 1).
// ---------------------------------------------------------------------------
struct FoldArgs {
    Dev d;
    Offers of;
    const u32 *seg_start;
    const u64 *seg_count;
    u32 budget;   // 0 = deterministic
    u32 np, ns, gram;
    u32 lo, hi;   // lock-free: offer slots [lo, hi) of this launch
};

__host__ __device__ inline size_t fold_scratch(u32 np, u32 R) {
    return 2 * al16((size_t)R * 4 + 4) + al16(np) + al16((size_t)np * 4);
}
// keys: a prune sees at most R + 1 candidates
__host__ __device__ inline size_t fold_warp_bytes(u32 np, u32 R, u32 ns, u32 mp, u32 gram) {
    const size_t sc = fold_scratch(np, R);
    return stage_bytes(ns, mp) + 4 * al16((size_t)R * 4 + 4) + al16((size_t)(R + 1) * 8) +
           (gram_alias(gram, sc) ? 0 : sc) + gram_bytes(gram, mp);
}

// one-warp blocks of the single-warp variant (GV 0) are held to 16 resident warps
// per SM (at most 128 registers a thread)
template <int GV>
__global__ void __launch_bounds__(coop_variant(GV) ? 32 * COOP_WARPS : 32, coop_variant(GV) ? 3 : GV == 4 ? 12 : 16)
    offer_fold_kernel(FoldArgs a) {
    extern __shared__ __align__(16) char smem[];
    __shared__ GramReq req;
    const int lane = lane_id();
    const Dev &d = a.d;
    const u32 R = d.R;
    char *p = smem;
    char *gbuf = a.gram ? p : nullptr;
    if constexpr (coop_variant(GV))
        if (threadIdx.x >= 32) return gram_helper<GV>(d, gbuf, a.gram, &req);
    p += gram_bytes(a.gram, d.mp);
    Stage st = stage_init(p, a.ns, d.mp, gbuf, a.gram, &req);
    WarpSlabs ws;
    ws_init(ws);
    p += stage_bytes(a.ns, d.mp);
    const size_t lb = al16((size_t)R * 4 + 4);
    u32 *lid = reinterpret_cast<u32 *>(p); p += lb;
    float *lrho = reinterpret_cast<float *>(p); p += lb;
    u32 *oid0 = reinterpret_cast<u32 *>(p); p += lb;
    float *orho0 = reinterpret_cast<float *>(p); p += lb;
    u64 *keys = reinterpret_cast<u64 *>(p); p += al16((size_t)(R + 1) * 8);
    if (gram_alias(a.gram, fold_scratch(a.np, R))) p = gbuf;
    u32 *tid = reinterpret_cast<u32 *>(p); p += lb;
    float *trho = reinterpret_cast<float *>(p); p += lb;
    unsigned char *alive = reinterpret_cast<unsigned char *>(p); p += al16(a.np);
    u32 *idx = reinterpret_cast<u32 *>(p);
    const u64 nwork = a.budget ? (u64)(a.hi - a.lo) : *a.seg_count;
    u64 t_next = 0;   // the next item's claim, in flight while this one runs
    if (lane == 0) t_next = atomicAdd(&d.ctr[C_WORK], 1ull);
    u64 pf_t = ~0ull;   // lock-free: the item whose words pf_w, pf_v, pf_vr hold
    u32 pf_w = 0, pf_v = 0;
    float pf_vr = 0.f;
    for (;;) {
        const u64 t = __shfl_sync(FULL, t_next, 0);
        if (t >= nwork) break;
        if (lane == 0) t_next = atomicAdd(&d.ctr[C_WORK], 1ull);
        if (a.budget == 0) {
            const u32 lo = a.seg_start[t], hi = a.seg_start[t + 1];
            const u32 w = a.of.key[lo];
            u64 snap;
            const int n0 = load_list(d, w, lid, lrho, snap);
            st.wk_state += 8 + 8ull * n0;
            for (int j = lane; j < n0; j += 32) { oid0[j] = lid[j]; orho0[j] = lrho[j]; }
            __syncwarp();
            int n = n0;
            bool pruned = ref_pruned(snap) != 0;
            for (u32 q = lo; q < hi; q++) {
                const u32 pi = a.of.val[q];
                n = apply_offer<GV>(d, lid, lrho, n, a.of.src[pi], a.of.rho[pi], keys, alive, idx, (int)a.np,
                                tid, trho, st, pruned);
            }
            if (!warp_same_list(lid, lrho, n, oid0, orho0, n0)) {
                st.wk_state += 8ull * n + 8;
                if (!warp_publish(d, ws, w, lid, lrho, n, snap, pruned) && lane == 0)
                    atomicOr(&d.ctr[C_ERR], (u64)ERR_CAS);
            }
        } else {
            u32 w = pf_w, v = pf_v;
            float vr = pf_vr;
            if (t != pf_t) { w = a.of.key[t + a.lo]; v = a.of.src[t + a.lo]; vr = a.of.rho[t + a.lo]; }
            if (w >= (u32)d.capacity) continue;
            bool done = false;
            for (u32 att = 0; att < a.budget && !done; att++) {
                u64 snap;
                const int n0 = load_list(d, w, lid, lrho, snap);
                st.wk_state += 8 + 8ull * n0;
                for (int j = lane; j < n0; j += 32) { oid0[j] = lid[j]; orho0[j] = lrho[j]; }
                __syncwarp();
                bool pruned = ref_pruned(snap) != 0;
                const int n = apply_offer<GV>(d, lid, lrho, n0, v, vr, keys, alive, idx, (int)a.np, tid, trho, st,
                                              pruned);
                if (att == 0) {                      // the next offer's words, in flight while this one publishes
                    pf_t = __shfl_sync(FULL, t_next, 0);
                    if (pf_t < nwork) { pf_w = a.of.key[pf_t + a.lo]; pf_v = a.of.src[pf_t + a.lo]; pf_vr = a.of.rho[pf_t + a.lo]; }
                }
                if (warp_same_list(lid, lrho, n, oid0, orho0, n0)) { done = true; break; }
                st.wk_state += 8ull * n + 8;
                done = warp_publish(d, ws, w, lid, lrho, n, snap, pruned);
                u64 err = 0;
                if (lane == 0) err = *reinterpret_cast<volatile u64 *>(&d.ctr[C_ERR]);
                if (!done && (__shfl_sync(FULL, err, 0) & ERR_NOMEM)) break;
            }
            if (!done && lane == 0) atomicAdd(&d.ctr[C_DROPPED], 1ull);
        }
        __syncwarp();
    }
    if (coop_variant(GV)) gram_release(&req);
    ws_finish(d, ws);
    stage_done(d, st, WK_OFFER);
}

cudaError_t launch_offer_fold(const Dev &d, const Offers &of, const u32 *seg_start, const u64 *seg_count,
                              u32 budget, int num_sms, cudaStream_t st, u32 lo, u32 hi) {
    if (of.n == 0) return cudaSuccess;
    if (budget && hi > of.n) hi = of.n;
    if (budget && lo >= hi) return cudaSuccess;
    FoldArgs a{d, of, seg_start, seg_count, budget, 0, 0, 0, lo, budget ? hi : of.n};
    a.gram = prune_rows_for(d, d.R + 1, a.hi - a.lo, num_sms);
    u32 np = 32;
    while (np < d.R + 1) np <<= 1;
    a.np = np;
    a.ns = a.gram ? 0 : stage_cap(d.mp, d.R + 1, d.stage_bytes);
    const size_t wb = fold_warp_bytes(np, d.R, a.ns, d.mp, a.gram);
    const size_t smem = wb;
    const int threads = block_threads(a.gram, d.mp);
    const void *fns[4] = {(const void *)offer_fold_kernel<0>, (const void *)offer_fold_kernel<1>, (const void *)offer_fold_kernel<2>,
                          (const void *)offer_fold_kernel<3>};
    const void *fn = !d.gram && !a.gram ? (const void *)offer_fold_kernel<4> : fns[gram_variant(a.gram, d.mp)];
    cudaError_t e = smem_at_least((const void *)fn, smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        &per_sm, fn, threads, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    const u32 items = budget ? a.hi - a.lo : of.n;
    u32 blocks = (u32)(per_sm * num_sms), need = items;
    if (blocks > need) blocks = need;
    e = cudaMemsetAsync(d.ctr + C_WORK, 0, sizeof(u64), st);
    if (e != cudaSuccess) return e;
    void *args[] = {&a};
    e = cudaLaunchKernel(fn, dim3(blocks), dim3(threads), args, smem, st);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Refine pass (reading of Sec. 3.4.1): member v re-selects its edges from
// N(v) and the lists of its neighbours (two hops; mode 2 admits only members
// of the same sub-batch), keeps the nearest max_cand, prunes, publishes if
// the list changed, and offers the edges it gained.
// ---------------------------------------------------------------------------
struct RefineArgs {
    Dev d;
    u32 first, b, mode, max_cand, cap, np, ns, gram;
    u32 cap_s, np_s;   // the shared-memory lists (most members); cap, np: the full ones
    char *spill;       // per warp, lists for cap raw ids (a member with more)
    u64 spill_warp;    // bytes of one warp's spill lists
    Offers of;
};

// Bytes of one warp's candidate lists for `cap` raw two-hop ids.
__host__ __device__ inline size_t refine_list_bytes(u32 np, u32 cap) {
    return al16((size_t)np * 8) + al16(np) + al16((size_t)np * 4) + al16((size_t)cap * 4);
}

__host__ __device__ inline size_t refine_warp_bytes(u32 np, u32 cap, u32 R, u32 ns, u32 mp, u32 gram) {
    return stage_bytes(ns, mp) + 4 * al16((size_t)R * 4) + refine_list_bytes(np, cap) + gram_bytes(gram, mp);
}

template <int GV>
__global__ void __launch_bounds__(GV ? 32 * COOP_WARPS : 64, GV ? 3 : 6) refine_kernel(RefineArgs a) {
    extern __shared__ __align__(16) char smem[];
    __shared__ GramReq req;
    const int warp = threadIdx.x >> 5, lane = lane_id();
    const Dev &d = a.d;
    const u32 R = d.R;
    char *p = smem + (GV ? 0 : warp) * refine_warp_bytes(a.np_s, a.cap_s, R, a.ns, d.mp, a.gram);
    char *gbuf = a.gram ? p : nullptr;
    if (GV != 0 && warp) return gram_helper<GV>(d, gbuf, a.gram, &req);
    p += gram_bytes(a.gram, d.mp);
    Stage st = stage_init(p, a.ns, d.mp, gbuf, a.gram, &req);
    WarpSlabs ws;
    ws_init(ws);
    p += stage_bytes(a.ns, d.mp);
    u32 *nid = reinterpret_cast<u32 *>(p); p += al16((size_t)R * 4);
    float *nrho = reinterpret_cast<float *>(p); p += al16((size_t)R * 4);
    u32 *oid = reinterpret_cast<u32 *>(p); p += al16((size_t)R * 4);
    float *orho = reinterpret_cast<float *>(p); p += al16((size_t)R * 4);
    // lists: in shared memory for up to cap_s raw ids, else this warp's spill
    auto carve_lists = [](char *q, u32 np) {
        struct L { u64 *buf; unsigned char *alive; u32 *idx, *uid; } l;
        l.buf = reinterpret_cast<u64 *>(q); q += al16((size_t)np * 8);
        l.alive = reinterpret_cast<unsigned char *>(q); q += al16(np);
        l.idx = reinterpret_cast<u32 *>(q); q += al16((size_t)np * 4);
        l.uid = reinterpret_cast<u32 *>(q);
        return l;
    };
    const auto ls = carve_lists(p, a.np_s);
    const auto lg = carve_lists(a.spill + (GV ? blockIdx.x : blockIdx.x * (blockDim.x >> 5) + warp) * a.spill_warp, a.np);
    const int grp = lane >> 3, g = lane & 7;
    u32 t_next = 0;   // the next item's claim, in flight while this one runs
    if (lane == 0) t_next = (u32)atomicAdd(&d.ctr[C_WORK], 1ull);
    for (;;) {
        const u32 t = __shfl_sync(FULL, t_next, 0);
        if (t >= a.b) break;
        if (lane == 0) t_next = (u32)atomicAdd(&d.ctr[C_WORK], 1ull);
        const u32 v = dev_first(d, a.first) + t;
        u64 snap;
        const int dv = load_list(d, v, nid, nrho, snap);
        st.wk_state += 8 + 8ull * dv;
        // 1. raw two-hop ids (v, members of N(v), and for mode 2 non-members
        //    of the sub-batch excluded), kept as u64 for the sort; a member
        //    with more than cap_s of them is collected again into the spill
        u64 *buf = ls.buf;
        unsigned char *alive = ls.alive;
        u32 *idx = ls.idx, *uid = ls.uid;
        u32 cap = a.cap_s;
        int nraw = 0;
        bool overflow = false;
        u64 nb_state = 0;                       // the neighbours' words and lists
    collect:
        nraw = 0;
        overflow = false;
        nb_state = 0;
        for (int i = 0; i < dv; i++) {
            const u64 rw = ld_ref(d, nid[i]);
            const u32 s = ref_slab(rw);
            const int dw = s == NIL ? 0 : (int)ref_deg(rw);
            nb_state += 8 + 8ull * dw;
            for (int j0 = 0; j0 < dw; j0 += 32) {
                u32 y = NIL;
                if (j0 + lane < dw) y = d.slab[(size_t)s * R + j0 + lane].x;
                bool ok = y != NIL && y != v;
                if (ok && a.mode == 2) ok = y >= dev_first(d, a.first) && y < dev_first(d, a.first) + a.b;
                if (ok) {
                    for (int k = 0; k < dv; k++) ok &= nid[k] != y;
                }
                u32 m = __ballot_sync(FULL, ok);
                int pos = nraw + __popc(m & lanemask_lt());
                if (ok) {
                    if (pos < (int)cap) buf[pos] = y;
                    else overflow = true;
                }
                nraw += __popc(m);
            }
        }
        if (__any_sync(FULL, overflow)) {
            if (buf == ls.buf) {
                buf = lg.buf;
                alive = lg.alive;
                idx = lg.idx;
                uid = lg.uid;
                cap = a.cap;
                goto collect;
            }
            if (lane == 0) atomicOr(&d.ctr[C_ERR], (u64)ERR_OVERFLOW);
            nraw = min(nraw, (int)a.cap);
        }
        st.wk_state += nb_state;
        int np2 = 32;
        while (np2 < nraw) np2 <<= 1;
        for (int i = nraw + lane; i < np2; i += 32) buf[i] = KEY_INF;
        __syncwarp();
        warp_sort_u64(buf, np2);
        // 2. unique live ids
        int nu = 0;
        for (int i0 = 0; i0 < nraw; i0 += 32) {
            int i = i0 + lane;
            bool ok = i < nraw && (i == 0 || buf[i] != buf[i - 1]);
            u32 y = ok ? (u32)buf[i] : NIL;
            if (ok && a.mode != 2) ok = !ref_del(ld_ref(d, y));
            u32 m = __ballot_sync(FULL, ok);
            if (ok) uid[nu + __popc(m & lanemask_lt())] = y;
            nu += __popc(m);
        }
        __syncwarp();
        // 3. distances to v, then the live members of N(v)
        st.wk_rows += (u64)(nu + 1) * 4 * d.mp;   // v's row and the peers'
        st.wk_state += 8ull * ((a.mode != 2 ? nu : 0) + dv);   // liveness words
        const float *vrow = d.x + (size_t)v * d.mp;
        if (d.mp <= 128) {
            // v's four float4 per lane stay in registers
            float4 vr[4];
            canon_row_q8(vrow, (int)d.mp, g, vr);
            for (int r0 = 0; r0 < nu; r0 += 4) {
                const int c = r0 + grp;
                const int cc = c < nu ? c : nu - 1;
                const u32 y = uid[cc];
                float4 w4[4];
                canon_row_q8(d.x + (size_t)y * d.mp, (int)d.mp, g, w4);
                const float dd = canon_dist_q8v(vr, w4, (int)d.mp, (int)d.metric, g);
                if (c < nu && g == 0) buf[c] = mkkey(dd, y);
            }
        } else {
            for (int r0 = 0; r0 < nu; r0 += 4) {
                const int c = r0 + grp;
                const int cc = c < nu ? c : nu - 1;
                const u32 y = uid[cc];
                float dd = canon_dist<8>(vrow, d.x + (size_t)y * d.mp, (int)d.mp, (int)d.metric, g);
                if (c < nu && g == 0) buf[c] = mkkey(dd, y);
            }
        }
        __syncwarp();
        int nc = nu;
        for (int j0 = 0; j0 < dv; j0 += 32) {
            int j = j0 + lane;
            bool ok = j < dv && !ref_del(ld_ref(d, nid[j]));
            u32 m = __ballot_sync(FULL, ok);
            if (ok) buf[nc + __popc(m & lanemask_lt())] = mkkey(nrho[j], nid[j]);
            nc += __popc(m);
        }
        // The re-selection cannot change a pruned list of live entries (see
        // ref_pruned) when no peer was found, or when the list is full and
        // every peer sorts after it: the prune keeps the list in order.
        bool same = false;
        if (ref_pruned(snap) && nc - nu == dv) {
            const u64 last = dv ? mkkey(nrho[dv - 1], nid[dv - 1]) : 0ull;
            bool early = false;
            for (int i = lane; i < nu; i += 32) early |= buf[i] < last;
            same = nu == 0 || (dv == (int)R && !__any_sync(FULL, early));
        }
        int nout = dv;
        if (same) {
            for (int j = lane; j < dv; j += 32) { oid[j] = nid[j]; orho[j] = nrho[j]; }
            __syncwarp();
        } else {
            int np3 = 32;
            while (np3 < nc) np3 <<= 1;
            for (int i = nc + lane; i < np3; i += 32) buf[i] = KEY_INF;
            __syncwarp();
            warp_sort_u64(buf, np3);
            const int n = min(nc, (int)a.max_cand);
            st.wk_rows += prune_row_bytes(d, st, nc - nu);   // the members of N(v), not yet gathered
            nout = warp_prune<GV>(d, buf, n, alive, idx, oid, orho, st);
            if (!warp_same_list(oid, orho, nout, nid, nrho, dv)) {
                st.wk_state += 8ull * nout + 8;
                if (!warp_publish(d, ws, v, oid, orho, nout, snap, true) && lane == 0)
                    atomicOr(&d.ctr[C_ERR], (u64)ERR_CAS);
            }
        }
        const u32 invalid = (u32)d.capacity;
        for (u32 j = lane; j < R; j += 32) {
            const size_t o = (size_t)t * R + j;
            bool gained = false;
            if ((int)j < nout) {
                gained = true;
                for (int k = 0; k < dv; k++) gained &= nid[k] != oid[j];
            }
            a.of.key[o] = gained ? oid[j] : invalid;
            a.of.val[o] = (u32)o;
            a.of.src[o] = v;
            a.of.rho[o] = gained ? orho[j] : 0.0f;
        }
        __syncwarp();
    }
    if (GV != 0) gram_release(&req);
    ws_finish(d, ws);
    stage_done(d, st, WK_REFINE);
}

// Launch shape of the refine kernel (shared by launch_refine and the spill size).
static void refine_shape(const Dev &d, u32 max_cand, RefineArgs &a, u64 items, int num_sms) {
    u32 cap = d.R * d.R;
    if (cap > 4096) cap = 4096;
    a.cap = cap;
    u32 np = 32;
    while (np < cap + d.R) np <<= 1;
    a.np = np;
    a.cap_s = cap < 192u ? cap : 192u;
    u32 nps = 32;
    while (nps < a.cap_s + d.R) nps <<= 1;
    a.np_s = nps;
    a.gram = d.gram ? (d.R > 32 ? (u32)GRAM_NL : (u32)GRAM_N) : prune_rows_for(d, 0, items, num_sms);
    a.ns = a.gram ? 0 : stage_cap(d.mp, max_cand, d.stage_bytes);
    a.spill_warp = refine_list_bytes(np, cap);
}

size_t refine_spill_bytes(const Dev &d, u32 max_cand, int num_sms) {
    RefineArgs a{};
    refine_shape(d, max_cand, a, 0, num_sms);
    // every warp an SM can hold (2,048 threads)
    return (size_t)num_sms * 64 * a.spill_warp;
}

cudaError_t launch_refine(const Dev &d, u32 first, u32 b, u32 mode, u32 max_cand, const Offers &of,
                          int num_sms, cudaStream_t st, char *spill, size_t spill_bytes) {
    if (b == 0) return cudaSuccess;
    RefineArgs a;
    a.d = d; a.first = first; a.b = b; a.mode = mode; a.max_cand = max_cand; a.of = of;
    refine_shape(d, max_cand, a, b, num_sms);
    a.spill = spill;
    const size_t wb = refine_warp_bytes(a.np_s, a.cap_s, d.R, a.ns, d.mp, a.gram);
    const bool coop = gram_variant(a.gram, d.mp) != 0;
    const int warps = !coop && 2 * wb <= 200 * 1024 ? 2 : 1;   // items of a block
    const int threads = coop ? 32 * COOP_WARPS : 32 * warps;
    size_t smem = warps * wb;
    const void *fns[4] = {(const void *)refine_kernel<0>, (const void *)refine_kernel<1>, (const void *)refine_kernel<2>,
                          (const void *)refine_kernel<3>};
    const void *fn = fns[gram_variant(a.gram, d.mp)];
    cudaError_t e = smem_at_least((const void *)fn, smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        &per_sm, fn, threads, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    u32 blocks = (u32)(per_sm * num_sms), need = (b + warps - 1) / warps;
    if (blocks > need) blocks = need;
    if ((size_t)blocks * warps * a.spill_warp > spill_bytes) return cudaErrorInvalidValue;
    e = cudaMemsetAsync(d.ctr + C_WORK, 0, sizeof(u64), st);
    if (e != cudaSuccess) return e;
    void *args[] = {&a};
    e = cudaLaunchKernel(fn, dim3(blocks), dim3(threads), args, smem, st);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Delete: tombstone CAS <0,d,s> -> <1,d,s> over ids sorted ascending; a
// repeated, unknown, already deleted or reclaimed id is a no-op.
// ---------------------------------------------------------------------------
__global__ void tombstone_kernel(Dev d, const u32 *ids, u32 n, u64 next_id, u32 *ok) {
    u32 i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const u32 u = ids[i];
    u32 res = 0;
    if ((i == 0 || ids[i - 1] != u) && (u64)u < dev_next_id(d, next_id)) {
        for (int att = 0; att < 64; att++) {
            const u64 r = ld_ref(d, u);
            if (ref_del(r) || ref_slab(r) == NIL) break;
            if (atomicCAS(&d.ref[u], r, r | (1ull << 63)) == r) { res = 1; break; }
        }
    }
    ok[i] = res;
}

cudaError_t launch_tombstone(const Dev &d, const u32 *sorted_ids, u32 n, u64 next_id, u32 *ok, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    tombstone_kernel<<<(n + 255) / 256, 256, 0, st>>>(d, sorted_ids, n, next_id, ok);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Repair, step 1: for deleted u with B = N(u) and each live a in B,
// K(u, a) = RobustPrune_a(B \ {a}).  The distances among B are computed once
// per u into a table; the prune reads the table.
// ---------------------------------------------------------------------------
struct RepairKArgs {
    Dev d;
    const u32 *dt;
    const u64 *n_dt;
    u32 *pair_key, *pair_val;
    uint2 *pair_K;
    u32 *pair_Kn;
};

constexpr int REPK_WARPS = 4;
__host__ __device__ inline size_t repk_bytes(u32 R) {
    return 2 * al16((size_t)R * 4) + al16((size_t)R * R * 4) + REPK_WARPS * (R <= 32 ? 32 * 8 : 64);
}

// The greedy RobustPrune of B \ {a} about a = member ja of B, from the table M,
// by one warp: the candidates b != a, live, in ascending (d(a, b), b), ranked
// by counting the smaller keys (ids differ); then, for every candidate, the
// mask of the later ones it would drop (no step waits for the one before); the
// walk visits only candidates whose mask is not empty.  Writes K in order and
// returns its size.  nb <= 64, H candidates per lane.
__device__ __forceinline__ int repair_select64(const Dev &d, const float *M, const u32 *bid, const u32 *bdel, int nb,
                                             int ja, unsigned char *ord, uint2 *K) {
    constexpr int H = 2;
    const int lane = lane_id();
    const u32 R = d.R;
    u64 k[H];
    int rank[H], nc = 0;
#pragma unroll
    for (int c = 0; c < H; c++) {
        const int t = lane + 32 * c;
        const bool v = t < nb && t != ja && !bdel[t];
        k[c] = v ? mkkey(M[ja * R + t], bid[t]) : KEY_INF;
        rank[c] = 0;
        nc += __popc(__ballot_sync(FULL, v));
    }
#pragma unroll
    for (int c2 = 0; c2 < H; c2++)
#pragma unroll 8
        for (int j = 0; j < min(32, nb - 32 * c2); j++) {
            const u64 o = __shfl_sync(FULL, k[c2], j);
#pragma unroll
            for (int c = 0; c < H; c++) rank[c] += o < k[c];
        }
#pragma unroll
    for (int c = 0; c < H; c++)
        if (k[c] != KEY_INF) ord[rank[c]] = (unsigned char)(lane + 32 * c);
    __syncwarp();
    int t[H];
    float rho[H];
#pragma unroll
    for (int c = 0; c < H; c++) {
        t[c] = lane + 32 * c < nc ? ord[lane + 32 * c] : ja;
        rho[c] = M[ja * R + t[c]];       // not read for t = ja
    }
    u64 dom[H], any = 0;                 // dom[c]: the candidates that candidate lane + 32 c would drop
#pragma unroll
    for (int c = 0; c < H; c++) dom[c] = 0;
#pragma unroll
    for (int c2 = 0; c2 < H; c2++)
#pragma unroll 8
        for (int j = 0; j < min(32, nc - 32 * c2); j++) {
            const int h = j + 32 * c2, hj = __shfl_sync(FULL, t[c2], j);
            u64 m = 0;
#pragma unroll
            for (int c = 0; c < H; c++) {
                const int i = lane + 32 * c;
                const bool hit = i > h && i < nc && __fmul_rn(d.alpha2, M[hj * R + t[c]]) <= rho[c];
                m |= (u64)__ballot_sync(FULL, hit) << (32 * c);
            }
            if (lane == j) dom[c2] = m;
            if (m) any |= 1ull << h;
        }
    u64 alive = nc >= 64 ? ~0ull : ((1ull << nc) - 1);
    while (any) {
        const int h = __ffsll((long long)any) - 1;
        any &= any - 1;
        const u64 m = __shfl_sync(FULL, h < 32 ? dom[0] : dom[1], h & 31);
        if (alive >> h & 1) alive &= ~m;
    }
#pragma unroll
    for (int c = 0; c < H; c++) {
        const int i = lane + 32 * c;
        if (i < nc && (alive >> i & 1))
            K[__popcll(alive & ((1ull << i) - 1))] = make_uint2(bid[t[c]], __float_as_uint(rho[c]));
    }
    __syncwarp();                        // ord is free again
    return __popcll(alive);
}

// The same for nb <= 32.  Lane c holds its column of alpha^2 M in registers (am)
// and collects, over all b, the earlier candidates (E) and those of them that would
// drop c (D).  A candidate is kept when none of D is: all that is decided by what
// is known is decided at once, so the steps are as many as the longest chain of
// candidates, not one for each; a kept candidate's place is the kept ones in E.
// 10,000 nodes of 128-d (R = 32) 664 -> 336 us against the form above; with two
// candidates per lane and the table in shared memory it is the slower one (500
// nodes of 768-d, R = 64: 318 against 247).
__device__ __forceinline__ int repair_select32(const float *M, const float (&am)[32], const u32 *bid, const u32 *bdel,
                                               u32 R, int nb, int ja, u64 *okey, uint2 *K) {
    const int lane = lane_id();
    const bool v = lane < nb && lane != ja && !bdel[lane];
    const float rho = v ? M[ja * R + lane] : 0.0f;
    const u64 k = v ? mkkey(rho, bid[lane]) : KEY_INF;
    okey[lane] = k;
    __syncwarp();
    u32 E = 0, D = 0;
#pragma unroll
    for (int g = 0; g < 4; g++) {
        if (8 * g >= nb) break;
#pragma unroll
        for (int b = 8 * g; b < 8 * g + 8; b++) {
            const bool lt = okey[b] < k;             // KEY_INF where b is no candidate
            if (lt) E |= 1u << b;
            if (lt && am[b] <= rho) D |= 1u << b;
        }
    }
    u32 kept = __ballot_sync(FULL, v && D == 0), open = __ballot_sync(FULL, v && D != 0);
    while (open) {
        open &= ~__ballot_sync(FULL, (open >> lane & 1) && (D & kept));
        // no kept candidate drops what is left; one that none of the open drop is kept
        const u32 m = open & ~__ballot_sync(FULL, (open >> lane & 1) && (D & open));
        kept |= m;
        open &= ~m;
    }
    if (kept >> lane & 1) K[__popc(E & kept)] = make_uint2(bid[lane], __float_as_uint(rho));
    __syncwarp();                        // okey is free again
    return __popc(kept);
}

// A block per deleted node.  The distances among B are computed in 8 x 8 tiles
// of pairs, a warp per tile: lane j sums partial j of the tile's 64 pairs, so
// that each 128-column block of 16 rows serves 64 pairs from registers.  Bound
// by the fp32 arithmetic of the table (the stored edge distances have to be
// canonical) and the selections: 336 us for 10,000 nodes of 128-d (R = 32), 246 for
// 500 of 768-d (R = 64), where a warp per node, four pairs at a time from shared
// memory, took 682 and 2,590.
template <int H>   // members of B per lane: R <= 32 H
__global__ void __launch_bounds__(32 * REPK_WARPS, 3) repair_k_kernel(RepairKArgs a) {
    extern __shared__ __align__(16) char smem[];
    __shared__ u64 next;
    const int tid = threadIdx.x, warp = tid >> 5, lane = lane_id();
    const Dev &d = a.d;
    const u32 R = d.R;
    char *p = smem;
    u32 *bid = reinterpret_cast<u32 *>(p); p += al16((size_t)R * 4);
    u32 *bdel = reinterpret_cast<u32 *>(p); p += al16((size_t)R * 4);
    float *M = reinterpret_cast<float *>(p); p += al16((size_t)R * R * 4);
    u64 *okey = reinterpret_cast<u64 *>(p) + warp * 32;                        // H = 1: a warp's candidate keys
    unsigned char *ord = reinterpret_cast<unsigned char *>(p) + warp * 64;   // H = 2: its candidates in order
    const u64 nd = *a.n_dt;
    const u32 invalid = (u32)d.capacity;
    u64 wk_rows = 0, wk_state = 0;
    for (;;) {
        __syncthreads();   // the last node's lists are read
        if (tid == 0) next = atomicAdd(&d.ctr[C_WORK], 1ull);
        __syncthreads();
        const u64 i = next;
        if (i >= nd) break;
        const u64 r = ld_ref(d, a.dt[i]);
        const u32 s = ref_slab(r);
        const int nb = s == NIL ? 0 : (int)ref_deg(r);
        for (int j = tid; j < nb; j += 32 * REPK_WARPS) {
            const u32 id = d.slab[(size_t)s * R + j].x;
            bid[j] = id;
            bdel[j] = ref_del(ld_ref(d, id));
        }
        wk_state += 8 + 16ull * nb;           // u's word, N(u), and the members' words
        wk_rows += (u64)nb * 4 * d.mp;        // B's rows
        __syncthreads();
        // distance table among B (symmetric): tiles x <= y, in one sequence
        const int nt = (nb + 7) >> 3;
        for (int t = warp; t < nt * (nt + 1) / 2; t += REPK_WARPS) {
            int tx, ty;
            tile_of(t, tx, ty);
            const float *xr[8], *yr[8];
#pragma unroll
            for (int c = 0; c < 8; c++) {     // past the list: a valid row again
                xr[c] = d.x + (size_t)bid[min(8 * tx + c, nb - 1)] * d.mp;
                yr[c] = d.x + (size_t)bid[min(8 * ty + c, nb - 1)] * d.mp;
            }
            float dd[2];
            pair_tile(d.mp, d.metric, xr, yr, dd);
#pragma unroll
            for (int k = 0; k < 2; k++) {
                const int q = 2 * lane + k, x = 8 * tx + (q >> 3), y = 8 * ty + (q & 7);
                if (x < y && y < nb) { M[x * R + y] = dd[k]; M[y * R + x] = dd[k]; }
            }
        }
        __syncthreads();
        // K(u, a), a warp per a
        float am[32];
        if (H == 1) {
#pragma unroll
            for (int b = 0; b < 32; b++) am[b] = b < nb ? __fmul_rn(d.alpha2, M[b * R + min(lane, nb - 1)]) : 0.0f;
        }
        for (int ja = warp; ja < (int)R; ja += REPK_WARPS) {
            const size_t slot = (size_t)i * R + ja;
            int nk = -1;
            if (ja < nb && !bdel[ja]) {
                if constexpr (H == 1) nk = repair_select32(M, am, bid, bdel, R, nb, ja, okey, a.pair_K + slot * R);
                else nk = repair_select64(d, M, bid, bdel, nb, ja, ord, a.pair_K + slot * R);
            }
            if (lane == 0) {
                a.pair_key[slot] = nk < 0 ? invalid : bid[ja];
                a.pair_val[slot] = (u32)slot;
                a.pair_Kn[slot] = (u32)max(nk, 0);
            }
        }
    }
    if (tid == 0) {
        if (wk_rows) atomicAdd(&d.ctr[C_WK + 2 * WK_REPAIR_K], wk_rows);
        if (wk_state) atomicAdd(&d.ctr[C_WK + 2 * WK_REPAIR_K + 1], wk_state);
    }
}

cudaError_t launch_repair_k(const Dev &d, const u32 *dt, const u64 *n_dt, u32 max_n, u32 *pair_key,
                            u32 *pair_val, uint2 *pair_K, u32 *pair_Kn, int num_sms, cudaStream_t st) {
    if (max_n == 0) return cudaSuccess;
    RepairKArgs a{d, dt, n_dt, pair_key, pair_val, pair_K, pair_Kn};
    const size_t smem = repk_bytes(d.R);
    void (*fn)(RepairKArgs) = d.R <= 32 ? repair_k_kernel<1> : repair_k_kernel<2>;
    cudaError_t e = smem_at_least((const void *)fn, smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, (const void *)fn, 32 * REPK_WARPS, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    const u32 blocks = std::min<u32>((u32)(per_sm * num_sms), max_n);
    e = cudaMemsetAsync(d.ctr + C_WORK, 0, sizeof(u64), st);
    if (e != cudaSuccess) return e;
    fn<<<blocks, 32 * REPK_WARPS, smem, st>>>(a);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Repair, step 2: for each live a, in ascending u:
// N <- RobustPrune_a((N \ {u}) + K(u, a)); publish once if changed.
// Lock-free mode (seg_start == NULL): one warp per (u, a) pair, CAS retries.
// ---------------------------------------------------------------------------
struct RepairFoldArgs {
    Dev d;
    const u32 *dt, *pair_key, *pair_val;
    const uint2 *pair_K;
    const u32 *pair_Kn;
    const u32 *seg_start;
    const u64 *seg_count;
    u64 n_pairs;
    u32 budget, np, ns, gram;
    u64 lo;       // lock-free: pair slots [lo, lo + n_pairs) of this launch
};

__host__ __device__ inline size_t repf_scratch(u32 np, u32 R) {
    return 2 * al16((size_t)R * 4 + 4) + 2 * al16((size_t)np * 8) + al16(np) + al16((size_t)np * 4);
}
__host__ __device__ inline size_t repf_warp_bytes(u32 np, u32 R, u32 ns, u32 mp, u32 gram) {
    const size_t sc = repf_scratch(np, R);
    return stage_bytes(ns, mp) + 4 * al16((size_t)R * 4 + 4) + al16((size_t)np * 8) +
           (gram_alias(gram, sc) ? 0 : sc) + gram_bytes(gram, mp);
}

template <int GV>
// pruned: in, whether the list is a RobustPrune output (see ref_pruned);
// out, the same for the returned list.
__device__ int repair_apply(const Dev &d, u32 *lid, float *lrho, int n, u32 u, const uint2 *K, int nk, u64 *keys,
                            u64 *ka, u64 *kb, unsigned char *alive, u32 *idx, int np, u32 *tid, float *trho,
                            Stage &st, bool &pruned) {
    const int lane = lane_id();
    // The list (minus u and deleted nodes) and K(u, a) (minus deleted nodes)
    // are each sorted by (rho, id); compact both, then place every key at its
    // rank in the union: a K key after the list keys below it, a list key after
    // the K keys below it.  An id in both has equal keys and would collapse in
    // the prune; its K copy is dropped here (same result, fewer Gram rows).
    int na = 0, nb = 0;
    uint2 e0 = make_uint2(0u, 0u);                   // K's first 32 entries, in flight with the list's words
    if (lane < nk) e0 = K[lane];
    for (int i0 = 0; i0 < n; i0 += 32) {
        const int i = i0 + lane;
        const bool v = i < n && lid[i] != u && !ref_del(ld_ref(d, lid[i]));
        const u32 m = __ballot_sync(FULL, v);
        if (v) ka[na + __popc(m & lanemask_lt())] = mkkey(lrho[i], lid[i]);
        na += __popc(m);
    }
    for (int j0 = 0; j0 < nk; j0 += 32) {
        const int j = j0 + lane;
        uint2 e = e0;
        if (j0 > 0 && j < nk) e = K[j];
        const bool v = j < nk && !ref_del(ld_ref(d, e.x));
        const u32 m = __ballot_sync(FULL, v);
        if (v) kb[nb + __popc(m & lanemask_lt())] = mkkey(__uint_as_float(e.y), e.x);
        nb += __popc(m);
    }
    __syncwarp();
    int nb2 = 0;                                     // K keys not in the list, compacted in place
    bool early = false;                              // a kept K key sorts before the list's last key
    for (int j0 = 0; j0 < nb; j0 += 32) {
        const int j = j0 + lane;
        u64 k = 0;
        int lo = 0;
        bool keep = false;
        if (j < nb) {
            k = kb[j];
            int hi = na;                             // list keys <= k
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (ka[mid] <= k) lo = mid + 1; else hi = mid;
            }
            keep = lo == 0 || ka[lo - 1] != k;
        }
        const u32 m = __ballot_sync(FULL, keep);
        const int jj = nb2 + __popc(m & lanemask_lt());
        if (keep) { kb[jj] = k; keys[jj + lo] = k; }
        nb2 += __popc(m);
        early |= __ballot_sync(FULL, keep && lo < na) != 0;
    }
    __syncwarp();
    // The list is full, live, without u, and no entry drops a later one; every
    // K key left sorts after it: the prune keeps the R entries in order and
    // stops before the first K key.
    st.wk_state += 8ull * (n + nk);          // reference words of the list and of K(u, a)
    if (pruned && na == n && n == (int)d.R && !early) return n;
    for (int i = lane; i < na; i += 32) {
        const u64 k = ka[i];
        int lo = 0, hi = nb2;                        // kept K keys < k
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (kb[mid] < k) lo = mid + 1; else hi = mid;
        }
        keys[i + lo] = k;
    }
    __syncwarp();
    const int cn = na + nb2;
    st.wk_rows += prune_row_bytes(d, st, cn);
    const int nout = warp_prune<GV>(d, keys, cn, alive, idx, tid, trho, st);
    for (int j = lane; j < nout; j += 32) { lid[j] = tid[j]; lrho[j] = trho[j]; }
    __syncwarp();
    pruned = true;
    return nout;
}

// one-warp blocks of the single-warp variant (GV 0) are held to 12 resident warps
// per SM (at most 170 registers a thread)
template <int GV>
__global__ void __launch_bounds__(coop_variant(GV) ? 32 * COOP_WARPS : 32, coop_variant(GV) ? 3 : 12)
    repair_fold_kernel(RepairFoldArgs a) {
    extern __shared__ __align__(16) char smem[];
    __shared__ GramReq req;
    const int lane = lane_id();
    const Dev &d = a.d;
    const u32 R = d.R;
    char *p = smem;
    char *gbuf = a.gram ? p : nullptr;
    if constexpr (coop_variant(GV))
        if (threadIdx.x >= 32) return gram_helper<GV>(d, gbuf, a.gram, &req);
    p += gram_bytes(a.gram, d.mp);
    Stage st = stage_init(p, a.ns, d.mp, gbuf, a.gram, &req);
    WarpSlabs ws;
    ws_init(ws);
    p += stage_bytes(a.ns, d.mp);
    const size_t lb = al16((size_t)R * 4 + 4);
    u32 *lid = reinterpret_cast<u32 *>(p); p += lb;
    float *lrho = reinterpret_cast<float *>(p); p += lb;
    u32 *oid0 = reinterpret_cast<u32 *>(p); p += lb;
    float *orho0 = reinterpret_cast<float *>(p); p += lb;
    u64 *keys = reinterpret_cast<u64 *>(p); p += al16((size_t)a.np * 8);
    if (gram_alias(a.gram, repf_scratch(a.np, R))) p = gbuf;
    u32 *tid = reinterpret_cast<u32 *>(p); p += lb;
    float *trho = reinterpret_cast<float *>(p); p += lb;
    u64 *ka = reinterpret_cast<u64 *>(p); p += al16((size_t)a.np * 8);
    u64 *kb = reinterpret_cast<u64 *>(p); p += al16((size_t)a.np * 8);
    unsigned char *alive = reinterpret_cast<unsigned char *>(p); p += al16(a.np);
    u32 *idx = reinterpret_cast<u32 *>(p);
    const u64 nwork = a.budget ? a.n_pairs : *a.seg_count;
    u64 t_next = 0;   // the next item's claim, in flight while this one runs
    if (lane == 0) t_next = atomicAdd(&d.ctr[C_WORK], 1ull);
    u64 pf_t = ~0ull;   // lock-free: the item whose words pf_w, pf_pv hold
    u32 pf_w = 0, pf_pv = 0;
    for (;;) {
        const u64 t = __shfl_sync(FULL, t_next, 0);
        if (t >= nwork) break;
        if (lane == 0) t_next = atomicAdd(&d.ctr[C_WORK], 1ull);
        if (a.budget == 0) {
            const u32 lo = a.seg_start[t], hi = a.seg_start[t + 1];
            const u32 w = a.pair_key[lo];
            u64 snap;
            const int n0 = load_list(d, w, lid, lrho, snap);
            st.wk_state += 8 + 8ull * n0;
            for (int j = lane; j < n0; j += 32) { oid0[j] = lid[j]; orho0[j] = lrho[j]; }
            __syncwarp();
            int n = n0;
            bool pruned = ref_pruned(snap) != 0;
            for (u32 q = lo; q < hi; q++) {
                const u32 pv = a.pair_val[q];
                n = repair_apply<GV>(d, lid, lrho, n, a.dt[pv / R], a.pair_K + (size_t)pv * R, (int)a.pair_Kn[pv], keys,
                                 ka, kb, alive, idx, (int)a.np, tid, trho, st, pruned);
            }
            if (!warp_same_list(lid, lrho, n, oid0, orho0, n0)) {
                st.wk_state += 8ull * n + 8;
                if (!warp_publish(d, ws, w, lid, lrho, n, snap, pruned) && lane == 0)
                    atomicOr(&d.ctr[C_ERR], (u64)ERR_CAS);
            }
        } else {
            u32 w = pf_w, pv = pf_pv;
            if (t != pf_t) { w = a.pair_key[t + a.lo]; pv = a.pair_val[t + a.lo]; }
            if (w >= (u32)d.capacity) continue;
            bool done = false;
            for (u32 att = 0; att < a.budget && !done; att++) {
                u64 snap;
                const int n0 = load_list(d, w, lid, lrho, snap);
                st.wk_state += 8 + 8ull * n0;
                for (int j = lane; j < n0; j += 32) { oid0[j] = lid[j]; orho0[j] = lrho[j]; }
                __syncwarp();
                bool pruned = ref_pruned(snap) != 0;
                const int n = repair_apply<GV>(d, lid, lrho, n0, a.dt[pv / R], a.pair_K + (size_t)pv * R,
                                           (int)a.pair_Kn[pv], keys, ka, kb, alive, idx, (int)a.np, tid, trho, st,
                                           pruned);
                if (att == 0) {                      // the next pair's words, in flight while this one publishes
                    pf_t = __shfl_sync(FULL, t_next, 0);
                    if (pf_t < nwork) { pf_w = a.pair_key[pf_t + a.lo]; pf_pv = a.pair_val[pf_t + a.lo]; }
                }
                if (warp_same_list(lid, lrho, n, oid0, orho0, n0)) { done = true; break; }
                st.wk_state += 8ull * n + 8;
                done = warp_publish(d, ws, w, lid, lrho, n, snap, pruned);
                u64 err = 0;
                if (lane == 0) err = *reinterpret_cast<volatile u64 *>(&d.ctr[C_ERR]);
                if (!done && (__shfl_sync(FULL, err, 0) & ERR_NOMEM)) break;
            }
            if (!done && lane == 0) atomicAdd(&d.ctr[C_DROPPED], 1ull);
        }
        __syncwarp();
    }
    if (coop_variant(GV)) gram_release(&req);
    ws_finish(d, ws);
    stage_done(d, st, WK_REPAIR_FOLD);
}

cudaError_t launch_repair_fold(const Dev &d, const u32 *dt, const u32 *pair_key, const u32 *pair_val,
                                    const uint2 *pair_K, const u32 *pair_Kn, const u32 *seg_start,
                                    const u64 *seg_count, u64 n_pairs, u32 budget, int num_sms, cudaStream_t st,
                               u64 lo) {
    if (n_pairs == 0) return cudaSuccess;
    RepairFoldArgs a{d, dt, pair_key, pair_val, pair_K, pair_Kn, seg_start, seg_count, n_pairs, budget, 0, 0,
                     prune_rows_for(d, 2 * d.R - 1, n_pairs, num_sms), lo};
    u32 np = 32;
    while (np < 2 * d.R) np <<= 1;
    a.np = np;
    a.ns = a.gram ? 0 : stage_cap(d.mp, 2 * d.R, d.stage_bytes);
    const size_t wb = repf_warp_bytes(np, d.R, a.ns, d.mp, a.gram);
    const size_t smem = wb;
    const int threads = block_threads(a.gram, d.mp);
    const void *fns[4] = {(const void *)repair_fold_kernel<0>, (const void *)repair_fold_kernel<1>, (const void *)repair_fold_kernel<2>,
                          (const void *)repair_fold_kernel<3>};
    const void *fn = !d.gram && !a.gram ? (const void *)repair_fold_kernel<4> : fns[gram_variant(a.gram, d.mp)];
    cudaError_t e = smem_at_least((const void *)fn, smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        &per_sm, fn, threads, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    const u64 need = n_pairs;
    u32 blocks = (u32)(per_sm * num_sms);
    if ((u64)blocks > need) blocks = (u32)need;
    e = cudaMemsetAsync(d.ctr + C_WORK, 0, sizeof(u64), st);
    if (e != cudaSuccess) return e;
    void *args[] = {&a};
    e = cudaLaunchKernel(fn, dim3(blocks), dim3(threads), args, smem, st);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Reclaim phase 1 (compaction): every live node with a tombstoned neighbour
// republishes its list without those entries, order and rho kept.  One warp
// per 32 consecutive ids; tombstones are read from a bitmap.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) compact_kernel(Dev d, u64 next_id, const u32 *tomb_bits) {
    __shared__ u32 sid[8][MAX_R];
    __shared__ float srho[8][MAX_R];
    const int warp = threadIdx.x >> 5, lane = lane_id();
    const u64 base = ((u64)blockIdx.x * 8 + warp) * 32;
    next_id = dev_next_id(d, next_id);
    if (base >= next_id) return;
    const u64 myid = base + lane;
    const u64 myref = myid < next_id ? ld_ref(d, (u32)myid) : ref_pack(1, 0, NIL);
    const u32 R = d.R;
    WarpSlabs ws;
    ws_init(ws);
    // graph state: the words scanned, each live list with one tombstone bit
    // per entry, and the lists republished
    u64 wk = 8ull * (u64)min((u64)32, next_id - base);
    for (int t = 0; t < 32; t++) {
        const u64 r = __shfl_sync(FULL, myref, t);
        if (ref_del(r) || ref_slab(r) == NIL) continue;
        const u32 s = ref_slab(r);
        const int n = (int)ref_deg(r);
        wk += 8ull * n + (u64)(n + 7) / 8;
        bool dirty = false;
        u32 ids[2];
        float rhos[2];
        bool keep[2];
        int c = 0;
        for (int j = lane; j < n; j += 32, c++) {
            uint2 e = d.slab[(size_t)s * R + j];
            ids[c] = e.x;
            rhos[c] = __uint_as_float(e.y);
            const bool dead = (tomb_bits[e.x >> 5] >> (e.x & 31)) & 1u;
            keep[c] = !dead;
            dirty |= dead;
        }
        if (!__any_sync(FULL, dirty)) continue;
        int nk = 0;
        c = 0;
        for (int j0 = 0; j0 < n; j0 += 32, c++) {
            const int j = j0 + lane;
            const bool k = j < n && keep[c];
            const u32 m = __ballot_sync(FULL, k);
            if (k) { sid[warp][nk + __popc(m & lanemask_lt())] = ids[c]; srho[warp][nk + __popc(m & lanemask_lt())] = rhos[c]; }
            nk += __popc(m);
        }
        __syncwarp();
        // a lost CAS here means another writer touched the node during the
        // reclaim launch, which the launch discipline forbids
        wk += 8ull * nk + 8;
        if (!warp_publish(d, ws, (u32)(base + t), sid[warp], srho[warp], nk, r, ref_pruned(r) != 0) && lane == 0)
            atomicOr(&d.ctr[C_ERR], (u64)ERR_CAS);
        __syncwarp();
    }
    ws_finish(d, ws);
    if (lane == 0) atomicAdd(&d.ctr[C_WK + 2 * WK_COMPACT + 1], wk);
}

cudaError_t launch_compact(const Dev &d, u64 next_id, const u32 *tomb_bits, cudaStream_t st) {
    if (next_id == 0) return cudaSuccess;
    u64 warps = (next_id + 31) / 32;
    compact_kernel<<<(unsigned)((warps + 7) / 8), 256, 0, st>>>(d, next_id, tomb_bits);
    return cudaGetLastError();
}

// Reclaim phase 2: CAS <1,d,s> -> <1,0,NIL> and retire s.
__global__ void reclaim_tomb_kernel(Dev d, u64 next_id) {
    const u64 u = (u64)blockIdx.x * blockDim.x + threadIdx.x;
    if (u >= dev_next_id(d, next_id)) return;
    const u64 r = ld_ref(d, (u32)u);
    if (!ref_del(r) || ref_slab(r) == NIL) return;
    if (atomicCAS(&d.ref[u], r, ref_pack(1, 0, NIL)) == r) retire_slab(d, ref_slab(r));
    else atomicOr(&d.ctr[C_ERR], (u64)ERR_CAS);
}

cudaError_t launch_reclaim_tombstones(const Dev &d, u64 next_id, cudaStream_t st) {
    if (next_id == 0) return cudaSuccess;
    reclaim_tomb_kernel<<<(unsigned)((next_id + 255) / 256), 256, 0, st>>>(d, next_id);
    return cudaGetLastError();
}

}  // namespace etale

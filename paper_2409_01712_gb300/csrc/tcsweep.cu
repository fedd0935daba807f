// Tensor-core tile sweeps of the solve phase (Alg. 3: forward substitution
// L z = y, backward substitution L^T x = z) for the mixed-precision factor.
//
// Work items (one 128-row slab s of a row block each), as in the paper's tile
// Cholesky solve, right-looking:
//   forward   DIAG(j, s)     z_j[s] = Linv_jj[s, :] y_j             (y_j final)
//             LINK(i, j, s)  y_i[s] -= L_ij[s, :] z_j,  i > j        (row slab of L_ij)
//   backward  DIAG(j, s)     x_j[s] = (Linv_jj^T)[s, :] z_j
//             LINK(t, j, s)  z_t[s] -= (L_jt^T)[s, :] x_j,  t < j    (column slab of L_jt)
// Every item is one tcgen05.mma chain D[128 x NP] = A[128 x b] B[NP x b]^T with
// FP32 accumulation in TMEM:
//   A  a 128-row slab of a factor tile in FP16 (K-major by TMA for the forward
//      sweep; MN-major -- the tile's columns -- for the backward sweep, so no
//      transposed copy of the factor is kept).  FP32-class tiles are stored as
//      an exact FP16 pair (hi, lo) and contribute two A phases; E4M3 tiles are
//      read from their FP16 copy; the diagonal inverses from their FP16 split.
//   B  the vector block as an FP16 pair (hi, lo) with one power-of-two scale
//      per block and column, both halves multiplied, so B carries about 22
//      significant bits; stored in groups of 64 rows, [group][hi columns, lo
//      columns][64], so that a block is contiguous and arrives in a few large
//      copies, once for the hi and lo phases of an item.
// The right-hand side is updated in place; a LINK applies its update after the
// earlier ones of the same slab (fixed order: deterministic results).  A slab
// whose rows become final (a DIAG slab, the last LINK of a slab) writes them
// at once as the FP16 pair with a scale predicted from the previous block and
// adds itself, and whether its maxima fit that scale, to the block's state.  A
// reader finds there that every slab is finished and the scales hold; if they
// do not, the last slab converts the whole block again with the exact scale and
// the reader waits for that.
//
// Items are claimed from a device counter in dependency order (item 0 converts
// the first block; then, per column, its S DIAG items, its head LINK items and
// the LINK items of the column before; see "Items" below).  An item only waits
// for items claimed before it by running CTAs; every wait is bounded
// (%globaltimer) and ends the kernel with KRR_ETIMEOUT.
//
// CTA (192 threads, one per SM):
//   warp 0      producer: claims items, TMA loads of A (16 KB a stage) into a
//               shared-memory ring and of B into a buffer of its own.  The A
//               loads of the first stages go out before the block that the item
//               reads is final; the B copies as soon as it is, while the lanes
//               check that its predicted scales hold;
//   warp 1      TMEM allocation and the single MMA-issuing thread;
//   warps 2..5  epilogue: TMEM -> registers, scales, the in-place update or the
//               DIAG store, FP16 pairs, progress counters.
//
// What bounds it: the chain DIAG -> head LINK -> DIAG, two hops a column.  At
// N = 32768, b = 1024, P = 10 the two took 36 us: 10 and 5.4 us from the
// publication of the block they read to the last MMA, 5 us of epilogue each,
// 3.3 us each to find the block's maxima, accept its scales and publish it.  Now
// 20 us: the epilogue takes 1 us (branch-free per column, its loads before the
// accumulator wait), the scales are accepted with the load that finds the block
// finished, B arrives in large copies (0.4-0.9 us) and a chunk's MMAs are issued
// in 0.1-0.2 us instead of 0.3 (uniform descriptors, the next stage's barrier
// tested ahead); publication and its discovery are 1.5 us a hop.  A pair of
// sweeps took 2.24 ms, now 1.24; N = 5000, P = 2 0.38 and 0.20; N = 2048, b = 256,
// P = 1 0.335 and 0.146 ms.
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <string.h>

#include <algorithm>
#include <string>

#include "krr_internal.h"

namespace krr {

namespace {

constexpr int TS_THREADS = 192;
constexpr int TS_EPI = 128;
constexpr int TS_SLAB = 128;             // output rows of an item (MMA M)
constexpr int TS_KC = 64;                // K elements of a stage (128 bytes of FP16)
constexpr int TS_ABYTES = TS_SLAB * 128;  // A bytes of a stage
constexpr int TS_NPMAX = 32;             // right-hand sides per launch
constexpr int TS_IRING = 4;              // item header slots
constexpr int TS_BSEG = 16;              // most groups of 64 rows of the vector block held at once
constexpr int TS_BBOX = 256;             // rows of a B copy (groups x columns of a group)
constexpr int TS_NSMAX = 12;             // most A stages
// The producer loads A of an item's first stages before it looks for the next
// part of B, so these chunks must not reach beyond the first part.
static_assert(TS_NSMAX <= TS_BSEG, "the A chunks loaded ahead stay within the first part of B");

enum { TS_FWD = 0, TS_BWD = 1 };
enum { IT_CONV = 0, IT_DIAG = 1, IT_LINK = 2, IT_END = 3 };
// A operand maps
enum { AM_POOL = 0, AM_WSH = 1, AM_LHI = 2, AM_LLO = 3 };

struct TsParams {
    int job;
    int64_t b, nt, S, KC, items;
    int np, pc, q0;
    int64_t rs, cs;           // vector element (row, column q0 + q) at row * rs + (q0 + q) * cs
    float *rhs;               // FWD: y, BWD: z (updated in place)
    float *out;               // FWD: z, BWD: x
    float *bm_in, *bm_out;    // column maxima of rhs / out blocks (zero at the start), [nt][TS_NPMAX]
    __half *vin, *vout;       // FP16 pairs of rhs / out blocks: [n_pad / 64][2 np][64] (hi, then lo columns)
    float *sin, *sout;        // exact scales of blocks converted as a whole, [nt][np]
    const TileDesc *ltab;
    unsigned long long *st_in, *st_out;  // state of the rhs / out blocks, [nt]
    int *flags;               // [0] items, [1] abort, xin[nt], xout[nt], seq[nt * S]
    int stages;
    int lkc, bseg;            // log2 KC; groups of B held at once (KC, or TS_BSEG)
    uint32_t idesc;
    uint64_t wait_ns;
    DevErrors *err;
};

struct ItemHdr {
    int type;
    int blk, slab, src;      // output block and slab; block of the vector read
    int seqv;                // LINK: updates applied to (blk, slab) before this one
    int last_link;
    int nph;                 // A phases (1 or 2)
    int amap[2];
    int arow[2];             // first row of the tile (phase) in its map
    float inv_tscale;        // 1 / tile scale
};

// Whether a block of the right-hand side / of the solution was converted as a
// whole with its exact scale, and the updates applied to each slab.
__device__ __forceinline__ int *xin_ctr(const TsParams &p) { return p.flags + 2; }
__device__ __forceinline__ int *xout_ctr(const TsParams &p) { return p.flags + 2 + p.nt; }
__device__ __forceinline__ int *seq_ctr(const TsParams &p) { return p.flags + 2 + 2 * p.nt; }

// State of a block, one 64-bit word: finished slabs (bits 0-15), how many warps
// found a column that the predicted scale does not suit (too large for it; bits
// 16-31), and the columns that some warp found large enough for it (bits 32-63).  A reader
// learns with one load that the block is there and whether its predicted
// scales hold: for every column the maximum lies in [PRED_LO, PRED_HI).
__device__ __forceinline__ int state_slabs(unsigned long long v) { return (int)(v & 0xffff); }
__device__ __forceinline__ bool state_holds(unsigned long long v, int pc) {
    const uint32_t all = pc == 32 ? 0xffffffffu : (1u << pc) - 1u;
    return ((v >> 16) & 0xffff) == 0 && ((uint32_t)(v >> 32) & all) == all;
}

__device__ __forceinline__ uint32_t smem_u32(const void *ptr) {
    return (uint32_t)__cvta_generic_to_shared(ptr);
}

__device__ __forceinline__ uint64_t globaltimer() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred P;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 P, [%1], %2;\n\t"
        "selp.b32 %0, 1, 0, P;\n\t}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ int ld_acquire(const int *ptr) {
    int v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(ptr) : "memory");
    return v;
}

__device__ __forceinline__ unsigned long long ld_acquire64(const unsigned long long *ptr) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(ptr) : "memory");
    return v;
}

__device__ __forceinline__ void st_release(int *ptr, int v) {
    asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(ptr), "r"(v) : "memory");
}

// Orders this thread's generic-proxy global accesses with later async-proxy
// (TMA) accesses.
__device__ __forceinline__ void fence_proxy_async_global() {
    asm volatile("fence.proxy.async.global;" ::: "memory");
}

__device__ __forceinline__ void record_timeout(const TsParams &p) {
    atomicExch(&p.flags[1], 1);
    atomicCAS(&p.err->code, 0, (int)KRR_ETIMEOUT);
}

__device__ __forceinline__ bool aborted(const TsParams &p) { return *(volatile int *)&p.flags[1] != 0; }

// Bounded wait on a CTA barrier; false on expiry or when the sweep aborted.
__device__ __forceinline__ bool wait_bar(uint64_t *bar, uint32_t parity, const TsParams &p) {
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = globaltimer();
    for (uint32_t it = 1;; ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((it & 31) == 0) {
            if (aborted(p)) return false;
            if (globaltimer() - t0 > p.wait_ns) {
                record_timeout(p);
                return false;
            }
        }
    }
}

// Bounded wait until a progress counter reaches `target`.
// Polls back off exponentially (32 ns up to 256 ns) so that many waiting
// CTAs do not flood the L2 slice holding the counter.
__device__ __forceinline__ bool wait_count(const int *ctr, int target, const TsParams &p) {
    if (ld_acquire(ctr) >= target) return true;
    const uint64_t t0 = globaltimer();
    uint32_t nap = 32;
    for (uint32_t it = 1;; ++it) {
        __nanosleep(nap);
        if (nap < 256) nap <<= 1;
        if (ld_acquire(ctr) >= target) return true;
        if ((it & 15) == 0) {
            if (aborted(p)) return false;
            if (globaltimer() - t0 > p.wait_ns) {
                record_timeout(p);
                return false;
            }
        }
    }
}

// Bounded wait until all slabs of a block are finished; its state then.
__device__ __forceinline__ bool wait_state(const unsigned long long *ptr, int slabs, unsigned long long *v,
                                           const TsParams &p) {
    if (state_slabs(*v = ld_acquire64(ptr)) >= slabs) return true;
    const uint64_t t0 = globaltimer();
    uint32_t nap = 32;
    for (uint32_t it = 1;; ++it) {
        __nanosleep(nap);
        if (nap < 128) nap <<= 1;
        if (state_slabs(*v = ld_acquire64(ptr)) >= slabs) return true;
        if ((it & 15) == 0) {
            if (aborted(p)) return false;
            if (globaltimer() - t0 > p.wait_ns) {
                record_timeout(p);
                return false;
            }
        }
    }
}

__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, int x, int y, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3}], [%4];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_u32(bar))
        : "memory");
}

// Shared-memory matrix descriptors, 128-byte swizzle (tcgen05 version 1).
// K-major: 8-row groups of 128-byte rows, 1024 bytes apart (SBO); the
// leading offset is unused.
__device__ __forceinline__ uint64_t desc_kmajor(uint32_t addr) {
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFFu) >> 4);
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)(1024 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}
// MN-major: every 128-byte row holds 64 consecutive M elements of one K
// index; 8-row K groups are 1024 bytes apart (SBO) and the two 64-wide M
// halves of the slab are 8192 bytes apart (LBO, one TMA box each).
__device__ __forceinline__ uint64_t desc_mnmajor(uint32_t addr) {
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFFu) >> 4);
    d |= (uint64_t)(8192 >> 4) << 16;
    d |= (uint64_t)(1024 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

__device__ __forceinline__ void mma_f16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                        uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc));
}

// One lane of the (converged) warp, the same each time.
__device__ __forceinline__ bool elect_one() {
    uint32_t r;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(r));
    return r != 0;
}

__device__ __forceinline__ void mma_commit(uint64_t *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void tmem_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Sum of the eight groups of eight TMEM columns at t + g * step: every load is
// in flight before the one wait.
__device__ __forceinline__ void tmem_sum8x8(uint32_t t, uint32_t step, float *v) {
    uint32_t r[64];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%64];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%8,%9,%10,%11,%12,%13,%14,%15}, [%65];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%16,%17,%18,%19,%20,%21,%22,%23}, [%66];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%24,%25,%26,%27,%28,%29,%30,%31}, [%67];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%32,%33,%34,%35,%36,%37,%38,%39}, [%68];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%40,%41,%42,%43,%44,%45,%46,%47}, [%69];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%48,%49,%50,%51,%52,%53,%54,%55}, [%70];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%56,%57,%58,%59,%60,%61,%62,%63}, [%71];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=&r"(r[0]), "=&r"(r[1]), "=&r"(r[2]), "=&r"(r[3]), "=&r"(r[4]), "=&r"(r[5]), "=&r"(r[6]), "=&r"(r[7]),
          "=&r"(r[8]), "=&r"(r[9]), "=&r"(r[10]), "=&r"(r[11]), "=&r"(r[12]), "=&r"(r[13]), "=&r"(r[14]), "=&r"(r[15]),
          "=&r"(r[16]), "=&r"(r[17]), "=&r"(r[18]), "=&r"(r[19]), "=&r"(r[20]), "=&r"(r[21]), "=&r"(r[22]), "=&r"(r[23]),
          "=&r"(r[24]), "=&r"(r[25]), "=&r"(r[26]), "=&r"(r[27]), "=&r"(r[28]), "=&r"(r[29]), "=&r"(r[30]), "=&r"(r[31]),
          "=&r"(r[32]), "=&r"(r[33]), "=&r"(r[34]), "=&r"(r[35]), "=&r"(r[36]), "=&r"(r[37]), "=&r"(r[38]), "=&r"(r[39]),
          "=&r"(r[40]), "=&r"(r[41]), "=&r"(r[42]), "=&r"(r[43]), "=&r"(r[44]), "=&r"(r[45]), "=&r"(r[46]), "=&r"(r[47]),
          "=&r"(r[48]), "=&r"(r[49]), "=&r"(r[50]), "=&r"(r[51]), "=&r"(r[52]), "=&r"(r[53]), "=&r"(r[54]), "=&r"(r[55]),
          "=&r"(r[56]), "=&r"(r[57]), "=&r"(r[58]), "=&r"(r[59]), "=&r"(r[60]), "=&r"(r[61]), "=&r"(r[62]), "=&r"(r[63])
        : "r"(t), "r"(t + step), "r"(t + 2 * step), "r"(t + 3 * step), "r"(t + 4 * step), "r"(t + 5 * step),
          "r"(t + 6 * step), "r"(t + 7 * step)
        : "memory");
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        float x[8];
#pragma unroll
        for (int g = 0; g < 8; ++g) x[g] = __uint_as_float(r[8 * g + e]);
        v[e] = ((x[0] + x[2]) + (x[4] + x[6])) + ((x[1] + x[3]) + (x[5] + x[7]));
    }
}

__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 1, 128;" ::: "memory"); }

// ---------------------------------------------------------------------------
// Items.  Positions count from the start of the sweep: block position c is
// block c (forward) or nt - 1 - c (backward); LINK(c', p) applies column c'
// to block position p > c'.  Item 0 converts the first block of the
// right-hand side; then section c (0..nt-1) lists, S slabs each:
//   DIAG(c);
//   LINK(c - 1, c + 1)                 (1 <= c <= nt - 2)
//   LINK(c, c + 1), the head           (c <= nt - 2)
//   LINK(c - 1, p) for p = c + 2 .. nt - 1.
// The updates of a slab apply in column order, the head last, as with a plain
// column-by-column order; but DIAG(c + 1) is claimed before the bulk of
// column c's updates (listed one section later), so the chain DIAG -> head ->
// DIAG of consecutive columns does not wait for those to be claimed.  Every
// item depends only on items listed before it.  Section sizes: 2S (c = 0,
// nt > 1), S (nt + 1 - c) (0 < c < nt - 1), S (c = nt - 1).
// ---------------------------------------------------------------------------
__device__ __forceinline__ int64_t sec_start(int64_t S, int64_t nt, int64_t c) {
    if (c == 0) return 0;
    const int64_t first = (nt > 1) ? 2 * S : S;
    return first + S * ((c - 1) * (nt + 1) - (c - 1) * c / 2);
}

__device__ void decode_item(const TsParams &p, int64_t t, ItemHdr &h) {
    const int64_t S = p.S, nt = p.nt, b = p.b;
    const bool fwd = (p.job == TS_FWD);
    h.seqv = 0;
    h.last_link = 0;
    h.inv_tscale = 1.f;
    h.nph = 0;
    h.amap[0] = h.amap[1] = 0;
    h.arow[0] = h.arow[1] = 0;
    if (t == 0) {
        h.type = IT_CONV;
        h.blk = fwd ? 0 : (int)(nt - 1);
        h.slab = 0;
        h.src = h.blk;
        return;
    }
    const int64_t u = t - 1;
    int64_t lo = 0, hi = nt - 1;  // largest c with sec_start(c) <= u
    while (lo < hi) {
        const int64_t mid = (lo + hi + 1) >> 1;
        if (sec_start(S, nt, mid) <= u) lo = mid;
        else hi = mid - 1;
    }
    const int64_t c = lo;
    int64_t r = u - sec_start(S, nt, c);
    if (r < S) {
        const int64_t j = fwd ? c : nt - 1 - c;
        h.type = IT_DIAG;
        h.blk = (int)j;
        h.src = (int)j;
        h.slab = (int)r;
        h.nph = 2;
        h.amap[0] = AM_LHI;
        h.amap[1] = AM_LLO;
        h.arow[0] = h.arow[1] = (int)(j * b);
        return;
    }
    r -= S;
    int64_t col, pos, slab;  // LINK: column and block positions
    const bool pre = (c >= 1 && c <= nt - 2), head = (c <= nt - 2);
    if (pre && r < S) {
        col = c - 1, pos = c + 1, slab = r;
    } else {
        if (pre) r -= S;
        if (head && r < S) {
            col = c, pos = c + 1, slab = r;
        } else {
            if (head) r -= S;
            col = c - 1, pos = c + 2 + r / S, slab = r % S;
        }
    }
    const int64_t j = fwd ? col : nt - 1 - col;  // block of the vector read
    const int64_t blk = fwd ? pos : nt - 1 - pos;
    h.type = IT_LINK;
    h.src = (int)j;
    h.blk = (int)blk;
    h.slab = (int)slab;
    h.seqv = (int)col;
    h.last_link = (col == pos - 1) ? 1 : 0;
    // forward reads L_{blk, j}, backward L_{j, blk}
    const int64_t ti = fwd ? blk : j, tj = fwd ? j : blk;
    const int64_t off = off_index(ti, tj);
    const TileDesc d = p.ltab[off];
    h.inv_tscale = 1.f / d.scale;
    if (d.prec == KRR_PREC_E4M3) {
        // FP16 copy of the E4M3 tile in the tile's (spent) trailing slot
        h.nph = 1;
        h.amap[0] = AM_WSH;
        h.arow[0] = (int)(off * b);
    } else {
        const int row0 = (int)(d.offset / (2 * b));
        h.amap[0] = h.amap[1] = AM_POOL;
        h.arow[0] = row0;
        h.arow[1] = row0 + (int)b;  // FP32 class: the lo half follows the hi half
        h.nph = (d.prec == KRR_PREC_FP32) ? 2 : 1;
    }
}

// ---------------------------------------------------------------------------
// Block conversion (128 epilogue threads): v rows [blk b, +b), columns
// [q0, q0 + pc) -> FP16 terms with the power-of-two scale s_q putting the
// column maximum in [4096, 8192) (8x headroom below the FP16 maximum):
// two terms hi = fp16(s v), lo = fp16(s v - hi) (about 22 significant bits).
// Padding columns [pc, np) are zero.  The column maxima are those in bmax, or found here and written there (find).
// ---------------------------------------------------------------------------
__device__ __noinline__ void convert_block(const TsParams &p, const float *v, int64_t blk, __half *vb, float *sv,
                                           float *smax, float *sscale, int tid, bool find, float *bmax) {
    const int64_t b = p.b, rs = p.rs, cs = p.cs;
    const int pc = p.pc, np = p.np;
    const int wq = tid >> 5, lane = tid & 31;
    for (int q = 0; q < np; ++q) {
        if (find && q < pc) {
            float m = 0.f;
            for (int64_t r = tid; r < b; r += TS_EPI) m = fmaxf(m, fabsf(__ldcg(v + (blk * b + r) * rs + (p.q0 + q) * cs)));
            for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
            if (lane == 0) smax[wq * TS_NPMAX + q] = m;
        }
    }
    epi_sync();
    if (tid < np) {
        float s = 1.f;
        if (tid < pc) {
            const float m = find ? fmaxf(fmaxf(smax[tid], smax[TS_NPMAX + tid]),
                                         fmaxf(smax[2 * TS_NPMAX + tid], smax[3 * TS_NPMAX + tid]))
                                 : __ldcg(bmax + blk * TS_NPMAX + tid);
            if (m > 0.f && m < 3.0e38f) {
                int e;
                frexpf(m, &e);  // m = f 2^e, f in [0.5, 1)
                s = ldexpf(1.f, max(-126, min(126, 13 - e)));
            }
            if (find) bmax[blk * TS_NPMAX + tid] = m;
        }
        sscale[tid] = s;
        sv[blk * np + tid] = s;
    }
    epi_sync();
    for (int64_t r = tid; r < b; r += TS_EPI) {
        const int64_t grow = blk * b + r;
#pragma unroll 4
        for (int q = 0; q < np; ++q) {
            const float x = (q < pc) ? __ldcg(v + grow * rs + (p.q0 + q) * cs) * sscale[q] : 0.f;
            const __half hh = __float2half_rn(x);
            __half *dst = vb + (grow >> 6) * 2 * np * 64 + (grow & 63);
            dst[q * 64] = hh;
            dst[(np + q) * 64] = __float2half_rn(x - __half2float(hh));
        }
    }
    // publish: the block is read next by TMA (async proxy) on other SMs; the
    // caller's thread 0 releases the flag after this barrier
    epi_sync();
    if (tid == 0) {
        __threadfence();
        fence_proxy_async_global();
    }
}

// Predicted scale of a block from the column maximum m of the block before
// it in the sweep: puts m in [256, 512).  Blocks of one vector have similar
// magnitudes, so each slab converts its own rows with this scale as soon as
// they are final; the block keeps it if its own maximum lands in
// [PRED_LO, PRED_HI) (about 22 significant bits relative to the maximum, as
// with the exact scale, and 2x headroom below the FP16 maximum), else its last
// slab converts the whole block again with the exact scale.
// (A block of zeros has no maximum to place and takes the exact path, unless the
// block before it was zero as well.)
constexpr float PRED_LO = 8.f, PRED_HI = 32768.f;

__device__ __forceinline__ float pred_scale(float m) {
    if (!(m > 0.f) || !(m < 3.0e38f)) return 1.f;
    int e;
    frexpf(m, &e);
    return ldexpf(1.f, max(-126, min(126, 9 - e)));
}

// Maxima that predict the scales of a block: the block before it in the sweep
// (the right-hand side's own block for the first solution block).
__device__ __forceinline__ const float *pred_from(const TsParams &p, bool out, int64_t blk) {
    const bool fwd = (p.job == TS_FWD);
    const int64_t prev = fwd ? blk - 1 : blk + 1;
    const bool first = fwd ? (blk == 0) : (blk == p.nt - 1);
    return !out ? p.bm_in + prev * TS_NPMAX : first ? p.bm_in + blk * TS_NPMAX : p.bm_out + prev * TS_NPMAX;
}

template <int NP>
__global__ void __launch_bounds__(TS_THREADS, 1)
    tcsweep_kernel(const __grid_constant__ CUtensorMap mPool, const __grid_constant__ CUtensorMap mWsh,
                   const __grid_constant__ CUtensorMap mLhi, const __grid_constant__ CUtensorMap mLlo,
                   const __grid_constant__ CUtensorMap mVin, const __grid_constant__ CUtensorMap mVout,
                   const TsParams p) {
    extern __shared__ __align__(1024) uint8_t ts_smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(ts_smem_raw) + 1023) & ~uintptr_t(1023));
    const int NS = p.stages;
    uint8_t *bbuf = smem + NS * TS_ABYTES;
    ItemHdr *hdrs = reinterpret_cast<ItemHdr *>(bbuf + p.bseg * 2 * NP * 128);
    float *smax = reinterpret_cast<float *>(hdrs + TS_IRING);    // [4][TS_NPMAX]
    float *sscale = smax + 4 * TS_NPMAX;                          // [TS_NPMAX]
    float *smul = sscale + TS_NPMAX;                              // [TS_NPMAX]
    int *sexact = reinterpret_cast<int *>(smul + TS_NPMAX);       // [TS_IRING] the block read has exact scales
    int *sflag = sexact + TS_IRING;                               // [4]
    uint64_t *bars = reinterpret_cast<uint64_t *>(sflag + 4);
    uint64_t *full = bars, *empty = bars + NS, *tfull = bars + 2 * NS, *tempty = bars + 2 * NS + 2,
             *ifull = bars + 2 * NS + 4, *iempty = bars + 2 * NS + 4 + TS_IRING,
             *sfull = bars + 2 * NS + 4 + 2 * TS_IRING, *bfull = bars + 2 * NS + 4 + 3 * TS_IRING, *bempty = bfull + 1,
             *drain = bfull + 2;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(drain + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // two accumulators of four partial sums of 2 np columns: products with the
    // hi half of B, then with the lo half (one MMA of N = 2 np per K step reads
    // A once).  The four K steps of a chunk go to different partial sums: FP32
    // sums a quarter as long (the substitution's error at b = 2048: 2.5e-6
    // against 8.6e-6 with one) at no cost.
    constexpr uint32_t ACC = 2 * NP, TCOLS = 8 * ACC;
    if (threadIdx.x == 0) {
        for (int s = 0; s < NS; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(&tfull[a], 1);
            mbar_init(&tempty[a], TS_EPI / 32);
        }
        for (int q = 0; q < TS_IRING; ++q) {
            mbar_init(&ifull[q], 1);
            mbar_init(&iempty[q], TS_EPI / 32 + 1);  // epilogue warps and the MMA thread
            mbar_init(&sfull[q], 1);
        }
        mbar_init(bfull, 1);
        mbar_init(bempty, 1);
        mbar_init(drain, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(TCOLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (warp == 0 && lane == 0) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&mPool)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&mWsh)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&mLhi)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&mLlo)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&mVin)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&mVout)) : "memory");
    }
    tmem_fence_before();
    __syncthreads();
    tmem_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    const bool fwd = (p.job == TS_FWD);
    const int KC = (int)p.KC;
    // an item's chunks, and after how many of them the next part of B is due:
    // a block of up to TS_BSEG groups is loaded once for all phases
    auto b_period = [&](int nch) { return p.bseg == KC ? nch : p.bseg; };

    if (warp == 0) {
        // ------------------------------ producer ------------------------------
        const CUtensorMap *amaps[4] = {&mPool, &mWsh, &mLhi, &mLlo};
        int s = 0;
        uint32_t ph = 0;
        int slot = 0;
        uint32_t sph = 0;
        int issued = 0;
        bool ok = true;
        // A chunk c of the item (phase c / KC, K chunk c % KC) into the next stage
        auto load_a = [&](const ItemHdr &h, int c) -> bool {
            if (!wait_bar(&empty[s], ph ^ 1, p)) return false;
            uint8_t *st = smem + s * TS_ABYTES;
            const int q = c >> p.lkc, kc = c & (KC - 1);
            const CUtensorMap *m = amaps[q ? h.amap[1] : h.amap[0]];
            const int row = q ? h.arow[1] : h.arow[0];
            mbar_arrive_expect_tx(&full[s], (uint32_t)TS_ABYTES);
            if (fwd) {
                tma_load_2d(st, m, kc * TS_KC, row + h.slab * TS_SLAB, &full[s]);
            } else {
                const int y = row + kc * TS_KC;
                tma_load_2d(st, m, h.slab * TS_SLAB, y, &full[s]);
                tma_load_2d(st + TS_ABYTES / 2, m, h.slab * TS_SLAB + 64, y, &full[s]);
            }
            ++issued;
            if (++s == NS) { s = 0; ph ^= 1; }
            return true;
        };
        // groups [g0, g0 + bseg) of the vector block that the item reads
        auto load_b = [&](const ItemHdr &h, int g0, uint64_t *bar) {
            const CUtensorMap *m = (h.type == IT_DIAG) ? &mVin : &mVout;
            const int rows = p.bseg * 2 * NP, y = (h.src * KC + g0) * 2 * NP;
            mbar_arrive_expect_tx(bar, (uint32_t)rows * 128);
            for (int r = 0; r < rows; r += TS_BBOX) tma_load_2d(bbuf + r * 128, m, 0, y + r, bar);
        };
        uint32_t bph = 0;  // phase of the B buffer
        int nb = 0;        // loads of B issued
        int t = (lane == 0) ? atomicAdd(&p.flags[0], 1) : 0;
        while (ok) {
            t = __shfl_sync(0xffffffffu, t, 0);
            ItemHdr h;
            if (t >= p.items) {
                memset(&h, 0, sizeof(h));
                h.type = IT_END;
            } else {
                decode_item(p, t, h);
            }
            if (lane == 0) {
                ok = wait_bar(&iempty[slot], sph ^ 1, p);
                if (ok) {
                    hdrs[slot] = h;
                    mbar_arrive(&ifull[slot]);
                }
            }
            ok = __shfl_sync(0xffffffffu, (int)ok, 0) != 0;
            if (!ok || h.type == IT_END) break;
            if (lane == 0) t = atomicAdd(&p.flags[0], 1);  // the next item, while this one is loaded
            if (h.type != IT_CONV) {
                const int nch = h.nph * KC, bper = b_period(nch);
                const int npre = min(NS, nch);
                const bool diag = (h.type == IT_DIAG);
                if (lane == 0) {
                    // the first stages' A loads go out before the dependency wait
                    for (int c = 0; c < npre && ok; ++c) ok = load_a(h, c);
                    unsigned long long st = 0;
                    ok = ok && wait_state((diag ? p.st_in : p.st_out) + h.src, (int)p.S, &st, p) &&
                         wait_bar(bempty, bph ^ 1, p);
                    // the first right-hand side block has exact scales
                    bool exact = diag && h.src == (fwd ? 0 : (int)p.nt - 1);
                    if (ok && !exact && !state_holds(st, p.pc)) {
                        // the predicted scales do not hold: the block is being converted as a whole
                        exact = true;
                        ok = wait_count((diag ? xin_ctr(p) : xout_ctr(p)) + h.src, 1, p);
                    }
                    if (ok) {
                        fence_proxy_async_global();
                        load_b(h, 0, bfull);
                        ++nb;
                        bph ^= 1;
                        sexact[slot] = exact ? 1 : 0;
                        mbar_arrive(&sfull[slot]);
                    }
                    for (int c = npre; c < nch && ok; ++c) {
                        if ((c & (bper - 1)) == 0) {  // the next part of B (bper is a power of two)
                            ok = wait_bar(bempty, bph ^ 1, p);
                            if (!ok) break;
                            load_b(h, c & (KC - 1), bfull);
                            ++nb;
                            bph ^= 1;
                        }
                        ok = load_a(h, c);
                    }
                }
                ok = __shfl_sync(0xffffffffu, (int)ok, 0) != 0;
            }
            if (++slot == TS_IRING) { slot = 0; sph ^= 1; }
        }
        if (!ok && lane == 0) {
            // drain: wait (bounded) for the loads of the last stages to land
            const int n = issued < NS ? issued : NS;
            int ss = s;
            uint32_t pp = ph;
            for (int e = 0; e < n; ++e) {
                if (--ss < 0) { ss = NS - 1; pp ^= 1; }
                const uint64_t t0 = globaltimer();
                while (!mbar_try_wait(&full[ss], pp) && globaltimer() - t0 < drain_limit(p.wait_ns)) {}
            }
            const uint64_t t0 = globaltimer();
            while (nb > 0 && !mbar_try_wait(bfull, (uint32_t)(nb - 1) & 1) && globaltimer() - t0 < drain_limit(p.wait_ns)) {}
        }
    } else if (warp == 1) {
        // ------------------------------ MMA issuer ------------------------------
        // The whole warp runs the loop and one lane issues: the descriptors are
        // then computed in uniform registers, where the instruction reads them.
        int s = 0;
        uint32_t ph = 0, bph = 0;
        int slot = 0;
        uint32_t sph = 0;
        int acc = 0;
        uint32_t aph = 0;
        bool ok = true, any = false;
        const bool issuer = elect_one();
        auto wwait = [&](uint64_t *bar, uint32_t parity) { return __all_sync(0xffffffffu, wait_bar(bar, parity, p)) != 0; };
        // K steps of 16: 32 bytes of a K-major row, 16 rows of an MN-major one
        const uint64_t ad0 = fwd ? desc_kmajor(smem_u32(smem)) : desc_mnmajor(smem_u32(smem));
        const uint64_t bd0 = desc_kmajor(smem_u32(bbuf));
        const uint32_t astep = fwd ? 32 >> 4 : 2048 >> 4;
        while (ok) {
            if (!wwait(&ifull[slot], sph)) { ok = false; break; }
            const int type = __shfl_sync(0xffffffffu, hdrs[slot].type, 0);
            const int nch = __shfl_sync(0xffffffffu, hdrs[slot].nph, 0) * KC;
            if (issuer) mbar_arrive(&iempty[slot]);
            if (++slot == TS_IRING) { slot = 0; sph ^= 1; }
            if (type == IT_END) break;
            if (type == IT_CONV) continue;
            if (!wwait(&tempty[acc], aph ^ 1)) { ok = false; break; }
            tmem_fence_after();
            const uint32_t tacc = tmem_base + (uint32_t)acc * 4 * ACC;
            const int bper = b_period(nch);
            for (int c0 = 0; c0 < nch && ok; c0 += bper) {
                if (!wwait(bfull, bph)) { ok = false; break; }
                bph ^= 1;
                // One lane runs the chunks: 0.1 us each, against 0.14 with a vote
                // of the warp per chunk.  A stage's barrier is tested while the
                // MMAs of the stage before it are issued: a wait in series costs
                // as much as the four MMAs.
                if (issuer) {
                    int s1 = s;
                    uint32_t p1 = ph;
                    bool landed = mbar_try_wait(&full[s1], p1);
                    for (int c = c0; c < c0 + bper; ++c) {
                        if (!landed && !wait_bar(&full[s1], p1, p)) { ok = false; break; }
                        tmem_fence_after();
                        const int sn = (s1 + 1 == NS) ? 0 : s1 + 1;
                        const uint32_t pn = (sn == 0) ? p1 ^ 1 : p1;
                        landed = c + 1 < c0 + bper && mbar_try_wait(&full[sn], pn);
                        const uint64_t ad = ad0 + (uint32_t)(s1 * (TS_ABYTES >> 4));
                        const uint64_t bd = bd0 + (uint32_t)((c & (p.bseg - 1)) * (2 * NP * 128 >> 4));
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk)
                            // B rows [0, np) = hi half, [np, 2 np) = lo half
                            mma_f16(tacc + kk * ACC, ad + kk * astep, bd + kk * 2, p.idesc, c > 0 ? 1u : 0u);
                        mma_commit(&empty[s1]);
                        s1 = sn;
                        p1 = pn;
                    }
                    if (ok) {
                        mma_commit(bempty);  // this part of B is read
                        if (c0 + bper == nch) mma_commit(&tfull[acc]);
                    }
                }
                any = true;
                ok = __all_sync(0xffffffffu, ok) != 0;
                for (s += bper; s >= NS; s -= NS) ph ^= 1;
            }
            if (!ok) break;
            if (++acc == 2) { acc = 0; aph ^= 1; }
        }
        if (!ok && any && issuer) {
            mma_commit(drain);
            const uint64_t t0 = globaltimer();
            while (!mbar_try_wait(drain, 0) && globaltimer() - t0 < drain_limit(p.wait_ns)) {}
        }
        __syncwarp();
    } else {
        // ------------------------------ epilogue ------------------------------
        const int tid = threadIdx.x - 64;
        const int row = ((warp & 3) << 5) + lane;  // TMEM lane quarter of this warp
        int slot = 0;
        uint32_t sph = 0;
        int acc = 0;
        uint32_t aph = 0;
        const int pc = p.pc;
        const int64_t b = p.b, S = p.S, cs = p.cs;
        // one thread waits, the group follows its decision
        auto group_wait_bar = [&](uint64_t *bar, uint32_t parity) -> bool {
            if (tid == 0) sflag[0] = wait_bar(bar, parity, p) ? 1 : 0;
            epi_sync();
            const bool r = sflag[0] != 0;
            epi_sync();
            return r;
        };
        uint32_t sfph = 0;  // bit i: phase of sfull[i]
        while (true) {
            if (!group_wait_bar(&ifull[slot], sph)) break;
            const ItemHdr h = hdrs[slot];
            const int hslot = slot;
            epi_sync();
            if (++slot == TS_IRING) { slot = 0; sph ^= 1; }
            if (h.type == IT_END) break;
            if (h.type == IT_CONV) {
                if (lane == 0) mbar_arrive(&iempty[hslot]);
                convert_block(p, p.rhs, h.blk, p.vin, p.sin, smax, sscale, tid, true, p.bm_in);
                if (tid == 0) {
                    __threadfence();
                    atomicAdd(p.st_in + h.blk, (unsigned long long)S);
                }
                continue;
            }
            const bool link = (h.type == IT_LINK), fin = !link || h.last_link;
            const int64_t grow = (int64_t)h.blk * b + (int64_t)h.slab * TS_SLAB + row;
            // before waiting for the accumulator: the rows to update, once the
            // earlier updates of this slab are in, and the scales
            float yv[NP];
            float *y = (link ? p.rhs : p.out) + grow * p.rs + p.q0 * cs;
            int *sq = seq_ctr(p) + (int64_t)h.blk * S + h.slab;
            if (tid == 0)
                sflag[2] = ((!link || wait_count(sq, h.seqv, p)) && wait_bar(&sfull[hslot], (sfph >> hslot) & 1, p)) ? 1 : 0;
            sfph ^= 1u << hslot;
            epi_sync();
            if (!sflag[2]) break;
#pragma unroll
            for (int q = 0; q < NP; ++q) yv[q] = (link && q < pc) ? __ldcg(y + q * cs) : 0.f;
            if (tid < NP) {
                // column multipliers: 1 / (tile scale * vector block scale)
                float sc = 1.f;
                if (sexact[hslot]) sc = __ldcg((link ? p.sout : p.sin) + (int64_t)h.src * NP + tid);
                else if (tid < pc) sc = pred_scale(__ldcg(pred_from(p, link, h.src) + tid));
                smul[tid] = h.inv_tscale / sc;
                if (fin) {
                    const float m = (tid < pc) ? __ldcg(pred_from(p, !link, h.blk) + tid) : 0.f;
                    sscale[tid] = pred_scale(m);
                    smax[tid] = m;
                }
            }
            if (!group_wait_bar(&tfull[acc], aph)) break;
            if (lane == 0) mbar_arrive(&iempty[hslot]);  // the header and the scales are read
            tmem_fence_after();
            float v[NP];
            const uint32_t tacc = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)acc * 4 * ACC;
#pragma unroll
            for (int c8 = 0; c8 < NP; c8 += 8) tmem_sum8x8(tacc + c8, NP, v + c8);
            tmem_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&tempty[acc]);
            if (++acc == 2) { acc = 0; aph ^= 1; }
#pragma unroll
            for (int q = 0; q < NP; q += 4) {
                const float4 m4 = *reinterpret_cast<const float4 *>(smul + q);
                v[q] *= m4.x;
                v[q + 1] *= m4.y;
                v[q + 2] *= m4.z;
                v[q + 3] *= m4.w;
            }
#pragma unroll
            for (int q = 0; q < NP; ++q) {
                if (link) v[q] = yv[q] - v[q];
                if (q < pc) __stcg(y + q * cs, v[q]);
            }
            if (fin) {
                // the rows are final: FP16 pair with the predicted scales, and
                // the column maxima of the slab
                __half *vb = (link ? p.vin : p.vout) + (grow >> 6) * (2 * NP * 64) + (grow & 63);
#pragma unroll
                for (int q = 0; q < NP; q += 4) {
                    const float4 s4 = *reinterpret_cast<const float4 *>(sscale + q);
                    const float sq4[4] = {s4.x, s4.y, s4.z, s4.w};
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float xs = (q + e < pc) ? v[q + e] * sq4[e] : 0.f;
                        const __half hh = __float2half_rn(xs);
                        vb[(q + e) * 64] = hh;
                        vb[(NP + q + e) * 64] = __float2half_rn(xs - __half2float(hh));
                    }
                }
                uint32_t mine = 0;  // lane q: maximum of column q over the warp's rows
#pragma unroll
                for (int q = 0; q < NP; ++q) {
                    const uint32_t m = __reduce_max_sync(0xffffffffu, __float_as_uint(fabsf(v[q])));
                    if (lane == q) mine = m;
                }
                // the warp's part of the block's maxima and of the test of the scales
                // (zeros after a block of zeros keep its scale of 1, which small
                // entries in another warp's rows would not)
                const float ms = __uint_as_float(mine) * (lane < NP ? sscale[lane] : 0.f);
                const bool col = lane < pc, after0 = col && smax[lane] == 0.f;
                const uint32_t ge = __ballot_sync(0xffffffffu, col && (ms >= PRED_LO || (after0 && mine == 0)));
                const uint32_t over =
                    __ballot_sync(0xffffffffu, col && (!(ms < PRED_HI) || (after0 && mine != 0 && ms < PRED_LO)));
                unsigned long long *st = (link ? p.st_in : p.st_out) + h.blk;
                if (col)
                    atomicMax(reinterpret_cast<unsigned int *>((link ? p.bm_in : p.bm_out) + (int64_t)h.blk * TS_NPMAX) + lane,
                              mine);
                if (lane == 0) {
                    atomicOr(st, (unsigned long long)ge << 32);
                    if (over) atomicAdd(st, 1ull << 16);
                }
            }
            epi_sync();
            if (tid == 0) {
                __threadfence();
                if (fin) fence_proxy_async_global();  // the FP16 rows are read by TMA on other SMs
                if (link) atomicAdd(sq, 1);
                if (fin) {
                    // the last slab of the block: if the prediction failed for any
                    // column, the block is converted again (readers wait for that)
                    const unsigned long long v = atomicAdd((link ? p.st_in : p.st_out) + h.blk, 1ull);
                    sflag[1] = (state_slabs(v) == (int)S - 1 && !state_holds(v, pc)) ? 1 : 0;
                    if (sflag[1]) __threadfence();  // the other slabs' rows and maxima are read next
                }
            }
            if (fin) {
                epi_sync();
                if (sflag[1]) {
                    convert_block(p, link ? p.rhs : p.out, h.blk, link ? p.vin : p.vout, link ? p.sin : p.sout, smax,
                                  sscale, tid, false, link ? p.bm_in : p.bm_out);
                    if (tid == 0) st_release((link ? xin_ctr(p) : xout_ctr(p)) + h.blk, 1);
                }
            }
        }
    }
    tmem_fence_before();
    __syncthreads();
    if (warp == 1) {
        tmem_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TCOLS) : "memory");
    }
}

// ---------------------------------------------------------------------------
// Refinement residual on the tensor cores:
//   r = y - lambda a - sum_j (K_ij - c) a_j - c 1 (1^T a)
// with K the FP32 kernel tiles (lower triangle; block row i reads the row
// slabs of tiles (i, j <= i) and the column slabs of tiles (j > i, i)) and c
// the shift (mean off-diagonal entry of K), which keeps the products small.
//
// Item: 128 rows of one block times `g` consecutive source blocks (or 1 / h of
// one), added up in a two-term FP32 accumulator and written to a slot of its
// own, [slot][column][row] in FP64; a finishing kernel adds the slots in
// order (deterministic).  Items are listed by pairs of block groups (I, J),
// the slabs of both orientations together: a tile is needed once by rows (for
// the block row I) and once by columns (for J), and the two uses follow each
// other within a few items, so the second finds the tile in L2 and K comes
// from HBM once.  The split also fills the GPU when there are fewer 128-row
// slabs than SMs.  With
// one item per slab over all tiles, one epilogue group and the tiles read
// twice from HBM a residual took 1.27 ms at N = 32768 and 10 columns, 11.3 ms
// at N = 98304 and 20, 0.16 ms at N = 5000 and 2; now 0.80, 7.8 and 0.056 ms
// (0.88 and 8.5 with one group of converter warps).
//   warp 0       producer: TMA of the FP32 K chunk (128 x 64 rows x columns, or
//                64 x 128 for a column slab) and of the FP16 terms of a_j (B);
//   warps 6..9 and 14..17  converters, each group every other chunk: (K - c)
//                2^12 -> FP16 pair (hi, lo), written in place over the staged FP32 chunk (each thread overwrites only
//                the bytes its own warp read) in the MMA's K-major or MN-major
//                128-byte-swizzled layout, so the staging ring is also the
//                operand ring;
//   warp 1       MMA: A_hi x [B_hi; B_mid; B_lo] (N = 3 np) and A_lo x [B_hi;
//                B_mid] (N = 2 np); a is split into three FP16 terms (exact for
//                FP32 values), K - c into two (about 22 bits of a quantity
//                already small); the dropped products are below 2^-33;
//   warps 2..5 and 10..13  epilogue: per 64-wide chunk, the three FP32
//                accumulator parts are summed, de-scaled exactly (powers of
//                two) and added to a two-term FP32 (TwoSum) accumulator, so
//                each FP32 sum in TMEM spans only 64 products; each group of
//                four warps takes half of the columns.
// Operands exactly representing the FP32 inputs, exact FP16 products and
// FP32 accumulation: the residual keeps FP32 accuracy.
// Every wait is bounded and ends the kernel with KRR_ETIMEOUT.
// ---------------------------------------------------------------------------
constexpr int RS_THREADS = 576;
constexpr int RS_STG = 32768;      // FP32 chunk: 128 x 64 or 64 x 128
constexpr int RS_NSTG = 5;         // stages (FP32 K chunk by TMA, converted in place, and the terms of a)
// The two converter groups take every other chunk.  With an odd number of stages a
// stage holds their chunks in turn, which is what a group's wait for the chunk
// before its own rests on (see the converters).
static_assert(RS_NSTG % 2 == 1, "the converter groups alternate on every stage");
constexpr int RS_NACC = 4;         // TMEM accumulators of 3 np columns
// (K - c) s in FP16 with the power of two s = 2^(e - 1) <= 8192 / (max|K| + |c|):
// |(K - c) s| <= 8192, far below the FP16 maximum (s = 2^12 for the Gaussian
// kernel, whose entries lie in (0, 1]).
__device__ __forceinline__ float rs_kscale(const double *kbound, const double *shift) {
    int e;
    frexpf(8192.f / (float)(*kbound + fabs(*shift)), &e);
    return ldexpf(1.f, e - 1);
}

struct RsParams {
    ResGrid gr;
    int b, items;
    int64_t n_pad;
    int pc;
    const double *shift;
    const double *kbound;   // max |K_ij| (the residual operand's scale follows from it)
    const float *inv_s;     // inverse scales of the FP16 terms of a, [n_pad / 128][np]
    double *part;           // [slot][pc][n_pad]
    int *flags;             // [0] item counter, [1] abort
    uint32_t idesc_k, idesc_mn, idesc_k2, idesc_mn2;  // N = 3 np and N = 2 np
    uint64_t wait_ns;
    DevErrors *err;
};

__device__ __forceinline__ bool rs_aborted(const RsParams &p) { return *(volatile int *)&p.flags[1] != 0; }

__device__ __forceinline__ bool rs_wait(uint64_t *bar, uint32_t parity, const RsParams &p) {
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = globaltimer();
    for (uint32_t it = 1;; ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((it & 31) == 0) {
            if (rs_aborted(p)) return false;
            if (globaltimer() - t0 > p.wait_ns) {
                atomicExch(&p.flags[1], 1);
                atomicCAS(&p.err->code, 0, (int)KRR_ETIMEOUT);
                return false;
            }
        }
    }
}

// Three groups of eight TMEM columns, one wait.
__device__ __forceinline__ void tmem_ld8x3(uint32_t t0, uint32_t t1, uint32_t t2, float (&a)[8], float (&b)[8],
                                           float (&c)[8]) {
    uint32_t r[24];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%24];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%8,%9,%10,%11,%12,%13,%14,%15}, [%25];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%16,%17,%18,%19,%20,%21,%22,%23}, [%26];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=&r"(r[0]), "=&r"(r[1]), "=&r"(r[2]), "=&r"(r[3]), "=&r"(r[4]), "=&r"(r[5]), "=&r"(r[6]), "=&r"(r[7]),
          "=&r"(r[8]), "=&r"(r[9]), "=&r"(r[10]), "=&r"(r[11]), "=&r"(r[12]), "=&r"(r[13]), "=&r"(r[14]),
          "=&r"(r[15]), "=&r"(r[16]), "=&r"(r[17]), "=&r"(r[18]), "=&r"(r[19]), "=&r"(r[20]), "=&r"(r[21]),
          "=&r"(r[22]), "=&r"(r[23])
        : "r"(t0), "r"(t1), "r"(t2)
        : "memory");
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        a[e] = __uint_as_float(r[e]);
        b[e] = __uint_as_float(r[8 + e]);
        c[e] = __uint_as_float(r[16 + e]);
    }
}

template <int NP>
__global__ void __launch_bounds__(RS_THREADS, 1)
    tcres_kernel(const __grid_constant__ CUtensorMap mK128, const __grid_constant__ CUtensorMap mK64,
                 const __grid_constant__ CUtensorMap mA, const RsParams p) {
    constexpr int BB = 3 * NP * 128;           // bytes of the B terms of a chunk
    constexpr int SB = RS_STG + BB;            // bytes of a stage
    constexpr uint32_t TCOLS = (RS_NACC * 3 * NP <= 256) ? 256u : 512u;
    extern __shared__ __align__(1024) uint8_t rs_smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(rs_smem_raw) + 1023) & ~uintptr_t(1023));
    int *items = reinterpret_cast<int *>(smem + RS_NSTG * SB);  // item ring
    uint64_t *bars = reinterpret_cast<uint64_t *>(items + TS_IRING);
    // sfull: FP32 chunk and B landed; cfull: converted in place; sempty: MMAs done
    uint64_t *sfull = bars, *sempty = bars + RS_NSTG, *cfull = bars + 2 * RS_NSTG, *tfull = cfull + RS_NSTG,
             *tempty = tfull + RS_NACC, *ifull = tempty + RS_NACC, *iempty = ifull + TS_IRING,
             *drain = iempty + TS_IRING;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(drain + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int q = 0; q < RS_NSTG; ++q) {
            mbar_init(&sfull[q], 1);
            mbar_init(&sempty[q], 1);      // MMA commit
            mbar_init(&cfull[q], 4);       // converter warps
        }
        for (int a = 0; a < RS_NACC; ++a) {
            mbar_init(&tfull[a], 1);
            mbar_init(&tempty[a], 8);      // epilogue warps
        }
        for (int q = 0; q < TS_IRING; ++q) {
            mbar_init(&ifull[q], 1);
            mbar_init(&iempty[q], 8 + 8 + 1);  // epilogue, converter warps, MMA warp
        }
        mbar_init(drain, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(TCOLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (warp == 0 && lane == 0) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&mK128)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&mK64)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&mA)) : "memory");
    }
    tmem_fence_before();
    __syncthreads();
    tmem_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    if (warp == 0) {
        if (lane == 0) {
            // ------------------------------ producer ------------------------------
            int ss = 0, slot = 0;
            uint32_t sph = 0, iph = 0;
            int issued = 0;
            bool ok = true;
            int t = atomicAdd(&p.flags[0], 1);
            while (ok) {
                ResItem it;
                const bool end = t >= p.items;
                if (!end && !res_decode(p.gr, t, it)) {  // empty position
                    t = atomicAdd(&p.flags[0], 1);
                    continue;
                }
                if (!rs_wait(&iempty[slot], iph ^ 1, p)) { ok = false; break; }
                items[slot] = end ? -1 : t;
                mbar_arrive(&ifull[slot]);
                if (++slot == TS_IRING) { slot = 0; iph ^= 1; }
                if (end) break;
                t = atomicAdd(&p.flags[0], 1);  // the next item's number arrives during this one
                for (int j = it.j0; j < it.j1 && ok; ++j) {
                    for (int kc = it.kc0; kc < it.kc1; ++kc) {
                        if (!rs_wait(&sempty[ss], sph ^ 1, p)) { ok = false; break; }
                        uint8_t *st = smem + ss * SB;
                        mbar_arrive_expect_tx(&sfull[ss], SB);
                        if (j <= it.i) {
                            // row slab of tile (i, j): rows [sl 128, +128), columns [kc 64, +64)
                            const int y = (int)tri_index(it.i, j) * p.b + it.sl * TS_SLAB;
                            tma_load_2d(st, &mK128, kc * 64, y, &sfull[ss]);
                            tma_load_2d(st + RS_STG / 2, &mK128, kc * 64 + 32, y, &sfull[ss]);
                        } else {
                            // column slab of tile (j, i): rows [kc 64, +64), columns [sl 128, +128)
                            const int y = (int)tri_index(j, it.i) * p.b + kc * 64;
                            for (int e = 0; e < 4; ++e)
                                tma_load_2d(st + e * (RS_STG / 4), &mK64, it.sl * TS_SLAB + 32 * e, y, &sfull[ss]);
                        }
                        tma_load_2d(st + RS_STG, &mA, j * p.b + kc * 64, 0, &sfull[ss]);
                        ++issued;
                        if (++ss == RS_NSTG) { ss = 0; sph ^= 1; }
                    }
                }
            }
            if (!ok) {
                // drain the copies in flight (bounded)
                const int n = issued < RS_NSTG ? issued : RS_NSTG;
                int q = ss;
                uint32_t pp = sph;
                for (int e = 0; e < n; ++e) {
                    if (--q < 0) { q = RS_NSTG - 1; pp ^= 1; }
                    const uint64_t t0 = globaltimer();
                    while (!mbar_try_wait(&sfull[q], pp) && globaltimer() - t0 < drain_limit(p.wait_ns)) {}
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------ MMA issuer ------------------------------
        // (the warp runs the loop, one lane issues, as in the sweeps)
        int ss = 0, slot = 0, acc = 0;
        uint32_t sph = 0, iph = 0, aph = 0;
        bool ok = true, any = false;
        const bool issuer = elect_one();
        auto wwait = [&](uint64_t *bar, uint32_t parity) { return __all_sync(0xffffffffu, rs_wait(bar, parity, p)) != 0; };
        const uint64_t kd0 = desc_kmajor(smem_u32(smem)), md0 = desc_mnmajor(smem_u32(smem)),
                       bd0 = desc_kmajor(smem_u32(smem + RS_STG));
        while (ok) {
            if (!wwait(&ifull[slot], iph)) { ok = false; break; }
            const int t = __shfl_sync(0xffffffffu, items[slot], 0);
            if (issuer) mbar_arrive(&iempty[slot]);
            if (++slot == TS_IRING) { slot = 0; iph ^= 1; }
            if (t < 0) break;
            ResItem it;
            res_decode(p.gr, t, it);
            bool ready = false;  // the chunk's barriers, tested while the MMAs before it are issued
            for (int j = it.j0; j < it.j1 && ok; ++j) {
                const bool kmaj = (j <= it.i);
                const uint64_t ad0 = kmaj ? kd0 : md0;
                const uint32_t astep = kmaj ? 32 >> 4 : 2048 >> 4;
                const uint32_t id3 = kmaj ? p.idesc_k : p.idesc_mn, id2 = kmaj ? p.idesc_k2 : p.idesc_mn2;
                for (int kc = it.kc0; kc < it.kc1; ++kc) {
                    // one accumulation per 64-wide chunk: the FP32 sums in TMEM stay short
                    if (!__all_sync(0xffffffffu, ready) &&
                        !(wwait(&tempty[acc], aph ^ 1) && wwait(&sfull[ss], sph) && wwait(&cfull[ss], sph))) {
                        ok = false;
                        break;
                    }
                    tmem_fence_after();
                    const int sn = (ss + 1 == RS_NSTG) ? 0 : ss + 1, an = (acc + 1 == RS_NACC) ? 0 : acc + 1;
                    const uint32_t spn = (sn == 0) ? sph ^ 1 : sph, apn = (an == 0) ? aph ^ 1 : aph;
                    ready = (j + 1 < it.j1 || kc + 1 < it.kc1) && mbar_try_wait(&cfull[sn], spn) &&
                            mbar_try_wait(&sfull[sn], spn) && mbar_try_wait(&tempty[an], apn ^ 1);
                    const uint32_t tacc = tmem_base + (uint32_t)(acc * 3 * NP);
                    const uint32_t so = (uint32_t)(ss * (SB >> 4));
                    if (issuer) {
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk) {
                            const uint64_t ad = ad0 + so + kk * astep, bd = bd0 + so + kk * 2;
                            mma_f16(tacc, ad, bd, id3, kk > 0 ? 1u : 0u);
                            mma_f16(tacc, ad + (16384 >> 4), bd, id2, 1u);
                        }
                        mma_commit(&sempty[ss]);  // the stage takes the next TMA load
                        mma_commit(&tfull[acc]);
                    }
                    any = true;
                    ss = sn, sph = spn;
                    acc = an, aph = apn;
                }
            }
        }
        if (!ok && any && issuer) {
            mma_commit(drain);
            const uint64_t t0 = globaltimer();
            while (!mbar_try_wait(drain, 0) && globaltimer() - t0 < drain_limit(p.wait_ns)) {}
        }
        __syncwarp();
    } else if ((warp >= 6 && warp < 10) || warp >= 14) {
        // ------------------------------ converters ------------------------------
        const int group = (warp >= 14) ? 1 : 0;
        const int ct = threadIdx.x - (group ? 14 * 32 : 6 * 32);
        int turn = 0;  // group of the next chunk
        const float c = (float)*p.shift;
        const float kscale = rs_kscale(p.kbound, p.shift);
        int ss = 0, slot = 0;
        uint32_t sph = 0, iph = 0;
        bool ok = true;
        while (ok) {
            if (!__all_sync(0xffffffffu, rs_wait(&ifull[slot], iph, p))) break;
            const int t = items[slot];
            __syncwarp();
            if (lane == 0) mbar_arrive(&iempty[slot]);
            if (++slot == TS_IRING) { slot = 0; iph ^= 1; }
            if (t < 0) break;
            ResItem it;
            res_decode(p.gr, t, it);
            for (int j = it.j0; j < it.j1 && ok; ++j) {
                const bool kmaj = (j <= it.i);
                // thread -> (row r of the staged chunk, 64-value half h)
                const int r = kmaj ? ct : (ct >> 1), h = kmaj ? 0 : (ct & 1);
                const int boxb = kmaj ? RS_STG / 2 : RS_STG / 4;
                for (int kc = it.kc0; kc < it.kc1; ++kc) {
                    turn ^= 1;
                    if (turn == group) {  // the other group's chunk
                        if (++ss == RS_NSTG) { ss = 0; sph ^= 1; }
                        continue;
                    }
                    // The chunk before this one in the stage was the other group's
                    // (the stage count is odd), and copies land in any order: while
                    // that chunk is still on its way, the parity of sfull reads as
                    // if this one had landed.  cfull shows that it is converted, and
                    // cannot run ahead of this group.
                    if (!__all_sync(0xffffffffu, rs_wait(&cfull[ss], sph ^ 1, p) && rs_wait(&sfull[ss], sph, p))) {
                        ok = false;
                        break;
                    }
                    const uint8_t *src = smem + ss * SB + r * 128;
                    uint8_t *dst = smem + ss * SB + h * 8192 + r * 128;
                    float v[64];
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
#pragma unroll
                        for (int u = 0; u < 8; ++u) {
                            const float4 f = *reinterpret_cast<const float4 *>(src + (2 * h + e) * boxb + ((u ^ (r & 7)) << 4));
                            v[e * 32 + 4 * u] = f.x; v[e * 32 + 4 * u + 1] = f.y;
                            v[e * 32 + 4 * u + 2] = f.z; v[e * 32 + 4 * u + 3] = f.w;
                        }
                    }
                    // the FP16 rows overwrite FP32 rows that lanes of this warp
                    // read (thread (r, 0) writes over box 2 row r of thread (r, 1))
                    __syncwarp();
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        uint4 hv, lv;
                        __half2 *hh = reinterpret_cast<__half2 *>(&hv), *ll = reinterpret_cast<__half2 *>(&lv);
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const float x0 = (v[8 * u + 2 * e] - c) * kscale, x1 = (v[8 * u + 2 * e + 1] - c) * kscale;
                            const __half2 hx = __floats2half2_rn(x0, x1);
                            const float2 hf = __half22float2(hx);
                            hh[e] = hx;
                            ll[e] = __floats2half2_rn(x0 - hf.x, x1 - hf.y);
                        }
                        const int off = (u ^ (r & 7)) << 4;
                        *reinterpret_cast<uint4 *>(dst + off) = hv;
                        *reinterpret_cast<uint4 *>(dst + 16384 + off) = lv;
                    }
                    // generic-proxy writes, read next by the tensor cores
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&cfull[ss]);
                    if (++ss == RS_NSTG) { ss = 0; sph ^= 1; }
                }
            }
        }
    } else {
        // ------------------------------ epilogue ------------------------------
        constexpr int NC = NP / 2;  // columns of this group
        const int row = ((warp & 3) << 5) + lane;
        const int q0 = (warp >= 10) ? NC : 0;  // (warps 2-5 and 10-13)
        int slot = 0, acc = 0;
        uint32_t iph = 0, aph = 0;
        const float kinv = 1.f / rs_kscale(p.kbound, p.shift);  // a power of two: exact
        while (true) {
            if (!__all_sync(0xffffffffu, rs_wait(&ifull[slot], iph, p))) break;
            const int t = items[slot];
            __syncwarp();
            if (lane == 0) mbar_arrive(&iempty[slot]);
            if (++slot == TS_IRING) { slot = 0; iph ^= 1; }
            if (t < 0) break;
            ResItem it;
            res_decode(p.gr, t, it);
            // per column a two-term FP32 sum (hi, lo) grown by error-free
            // transformations (TwoSum): about 48 significant bits without
            // FP64 arithmetic, which runs at a small fraction of the FP32 rate
            float ahi[NC], alo[NC];
#pragma unroll
            for (int q = 0; q < NC; ++q) ahi[q] = alo[q] = 0.f;
            bool ok = true;
            for (int j = it.j0; j < it.j1 && ok; ++j) {
                for (int kc = it.kc0; kc < it.kc1; ++kc) {
                    // inverse scales of these rows of a (one set per 128 rows)
                    const float4 *is =
                        reinterpret_cast<const float4 *>(p.inv_s + (int64_t)(j * p.gr.S + (kc >> 1)) * NP + q0);
                    float mul[NC];
#pragma unroll
                    for (int q = 0; q < NC; q += 4) {
                        const float4 m4 = __ldg(is + q / 4);
                        mul[q] = m4.x, mul[q + 1] = m4.y, mul[q + 2] = m4.z, mul[q + 3] = m4.w;
                    }
                    if (!__all_sync(0xffffffffu, rs_wait(&tfull[acc], aph, p))) { ok = false; break; }
                    tmem_fence_after();
                    const uint32_t tacc =
                        tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(acc * 3 * NP + q0);
                    float v[NC];
#pragma unroll
                    for (int c8 = 0; c8 < NC; c8 += 8) {
                        float hv[8], mv[8], lv[8];
                        tmem_ld8x3(tacc + c8, tacc + NP + c8, tacc + 2 * NP + c8, hv, mv, lv);
#pragma unroll
                        for (int e = 0; e < 8; ++e) v[c8 + e] = hv[e] + (mv[e] + lv[e]);
                    }
                    tmem_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&tempty[acc]);
                    if (++acc == RS_NACC) { acc = 0; aph ^= 1; }
#pragma unroll
                    for (int q = 0; q < NC; ++q) {
                        const float xq = v[q] * mul[q];  // exact: powers of two
                        const float s2 = ahi[q] + xq, bp = s2 - ahi[q];
                        alo[q] += (ahi[q] - (s2 - bp)) + (xq - bp);
                        ahi[q] = s2;
                    }
                }
            }
            if (!ok) break;
            double *dst = p.part + ((int64_t)it.slot * p.pc + q0) * p.n_pad + (int64_t)it.i * p.b + it.sl * TS_SLAB + row;
#pragma unroll
            for (int q = 0; q < NC; ++q)
                if (q0 + q < p.pc) dst[(int64_t)q * p.n_pad] = (double)(ahi[q] * kinv) + (double)(alo[q] * kinv);
        }
    }
    tmem_fence_before();
    __syncthreads();
    if (warp == 1) {
        tmem_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TCOLS) : "memory");
    }
}

// True in every thread of the last block of the grid to come here (`total`
// blocks count on *ctr); the other blocks' earlier writes are then visible.
__device__ bool last_block(int *ctr, int total) {
    __shared__ int last_s;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last_s = (atomicAdd(ctr, 1) == total - 1) ? 1 : 0;
    __syncthreads();
    if (last_s) __threadfence();
    return last_s != 0;
}

// Operand of the residual: columns [q0, q0 + pc) of a (n_pad x p, row-major) as
// three FP16 terms, hi = fp16(s v), mid = fp16(s v - hi), lo = fp16(s v - hi -
// mid), which hold an FP32 value exactly down to 2^-14 of the column maximum
// (below that the absolute error stays under 2^-38 of the maximum), with one
// power-of-two scale per column and 128 rows putting the maximum in [4096,
// 8192); and the column sums of a in FP64 (partials per 128 rows, added in
// order by the last block).  One block per 128 rows, a row per thread.
__global__ void __launch_bounds__(TS_EPI)
    res_operand_kernel(const float *a, int64_t p, int q0, int pc, int np, int64_t n_pad, __half *vb, float *inv_s,
                       double *cs_part, double *colsum, int *ctr) {
    __shared__ float xs[TS_SLAB][TS_NPMAX + 1];
    __shared__ float pmax[8 * TS_NPMAX], scale[TS_NPMAX];
    __shared__ double psum[8 * TS_NPMAX];
    const int t = threadIdx.x;
    const int64_t grow = (int64_t)blockIdx.x * TS_SLAB + t;
    const float *src = a + grow * p + q0;
    for (int q = 0; q < np; ++q) xs[t][q] = (q < pc) ? src[q] : 0.f;
    __syncthreads();
    // np columns x parts of the rows
    const int parts = TS_EPI / np, rows = TS_SLAB / parts;
    {
        const int q = t % np, part = t / np;
        if (part < parts) {
            float m = 0.f;
            double s = 0.0;
            for (int r = part * rows; r < (part + 1) * rows; ++r) {
                m = fmaxf(m, fabsf(xs[r][q]));
                s += (double)xs[r][q];
            }
            pmax[part * np + q] = m;
            psum[part * np + q] = s;
        }
    }
    __syncthreads();
    if (t < np) {
        float m = 0.f;
        double s = 0.0;
        for (int e = 0; e < parts; ++e) {
            m = fmaxf(m, pmax[e * np + t]);
            s += psum[e * np + t];
        }
        float sc = 1.f;
        if (m > 0.f && m < 3.0e38f) {
            int e;
            frexpf(m, &e);  // m = f 2^e, f in [0.5, 1)
            sc = ldexpf(1.f, max(-126, min(126, 13 - e)));
        }
        scale[t] = sc;
        inv_s[(int64_t)blockIdx.x * np + t] = 1.f / sc;  // a power of two: exact
        if (t < pc) cs_part[(int64_t)blockIdx.x * pc + t] = s;
    }
    __syncthreads();
    for (int q = 0; q < np; ++q) {
        const float x = xs[t][q] * scale[q];
        const __half hh = __float2half_rn(x);
        const float r1 = x - __half2float(hh);  // exact
        const __half m = __float2half_rn(r1);
        vb[(int64_t)q * n_pad + grow] = hh;
        vb[(int64_t)(np + q) * n_pad + grow] = m;
        vb[(int64_t)(2 * np + q) * n_pad + grow] = __float2half_rn(r1 - __half2float(m));
    }
    if (!last_block(ctr, gridDim.x)) return;
    // lanes over the blocks, then a fixed tree
    const int lane = t & 31;
    for (int q = t >> 5; q < pc; q += TS_EPI / 32) {
        double s = 0.0;
        for (int64_t e = lane; e < gridDim.x; e += 32) s += __ldcg(cs_part + e * pc + q);
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if (lane == 0) colsum[q0 + q] = s;
    }
}

// r = y - lambda a - (the slots in order) - c colsum for columns [q0, q0 + pc),
// rounded to FP32 and written column-major (the sweeps' right-hand side), and
// ||r||_F^2, ||y||_F^2 and ||a||_F^2 over all p columns into red[RED_RNORM], the
// slot after it and red[RED_ANORM]: a partial per block (blocks of all column
// chunks count on ctr), added in order by the last.  ||a||_F^2 only scales the
// level at which refinement may end: FP32 sums.
__global__ void __launch_bounds__(256)
    res_finish_kernel(const float *y, const float *a, int64_t p, int q0, int pc, int64_t n_pad, const double *part,
                      int slots, float lambda, const double *shift, const double *colsum, float *rt, double *np_part,
                      int total, int *ctr, double *red) {
    __shared__ double s1[8], s2[8];
    __shared__ float s3[8];
    const int t = threadIdx.x, q = blockIdx.y;
    const int64_t r = (int64_t)blockIdx.x * 256 + t;
    double rv = 0.0, yv = 0.0;
    float av = 0.f;
    if (r < n_pad) {
        double sum = 0.0;
        const double *src = part + (int64_t)q * n_pad + r;
        const int64_t step = (int64_t)pc * n_pad;
#pragma unroll 4
        for (int e = 0; e < slots; ++e) sum += __ldcs(src + e * step);
        yv = (double)y[r * p + q0 + q];
        av = a[r * p + q0 + q];
        rv = (yv - (double)lambda * (double)av) - sum - *shift * colsum[q0 + q];
        rt[(int64_t)(q0 + q) * n_pad + r] = (float)rv;
    }
    double v1 = rv * rv, v2 = yv * yv;
    float v3 = av * av;
    for (int o = 16; o > 0; o >>= 1) {
        v1 += __shfl_down_sync(0xffffffffu, v1, o);
        v2 += __shfl_down_sync(0xffffffffu, v2, o);
        v3 += __shfl_down_sync(0xffffffffu, v3, o);
    }
    if ((t & 31) == 0) {
        s1[t >> 5] = v1;
        s2[t >> 5] = v2;
        s3[t >> 5] = v3;
    }
    __syncthreads();
    if (t == 0) {
        double x = 0.0, z = 0.0;
        float a2 = 0.f;
        for (int w = 0; w < 8; ++w) {
            x += s1[w];
            z += s2[w];
            a2 += s3[w];
        }
        const int64_t slot = (int64_t)(q0 + q) * gridDim.x + blockIdx.x;
        np_part[3 * slot] = x;
        np_part[3 * slot + 1] = z;
        np_part[3 * slot + 2] = (double)a2;
    }
    if (!last_block(ctr, total)) return;
    double x = 0.0, z = 0.0;
    float a2 = 0.f;
    for (int e = t; e < total; e += 256) {
        x += __ldcg(np_part + 3 * (int64_t)e);
        z += __ldcg(np_part + 3 * (int64_t)e + 1);
        a2 += (float)__ldcg(np_part + 3 * (int64_t)e + 2);
    }
    for (int o = 16; o > 0; o >>= 1) {
        x += __shfl_down_sync(0xffffffffu, x, o);
        z += __shfl_down_sync(0xffffffffu, z, o);
        a2 += __shfl_down_sync(0xffffffffu, a2, o);
    }
    if ((t & 31) == 0) {
        s1[t >> 5] = x;
        s2[t >> 5] = z;
        s3[t >> 5] = a2;
    }
    __syncthreads();
    if (t == 0) {
        x = z = 0.0;
        a2 = 0.f;
        for (int w = 0; w < 8; ++w) {
            x += s1[w];
            z += s2[w];
            a2 += s3[w];
        }
        red[RED_RNORM] = x;
        red[RED_RNORM + 1] = z;
        red[RED_ANORM] = (double)a2;
    }
}

// Encoder of TMA descriptors (driver entry point, looked up once).
typedef CUresult (*EncodeFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                             const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                             CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeFn encoder(Ctx *c) {
    static EncodeFn fn = nullptr;
    if (fn) return fn;
    void *f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !f) {
        cudaGetLastError();
        c->last_error = "cuTensorMapEncodeTiled is not available from the driver";
        return nullptr;
    }
    fn = (EncodeFn)f;
    return fn;
}

// FP16 row-major matrix (rows x cols), boxes of 64 columns (128 bytes) x
// box_rows, 128-byte swizzle.
krr_status map_f16(Ctx *c, CUtensorMap *m, const void *base, int64_t rows, int64_t cols, int box_rows) {
    EncodeFn enc = encoder(c);
    if (!enc) return KRR_ECUDA;
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)(cols * 2)};
    const cuuint32_t box[2] = {64u, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<void *>(base), dims, strides, box, estr,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        c->last_error = "cuTensorMapEncodeTiled (tensor-core sweep) failed with code " + std::to_string((int)r);
        return KRR_ECUDA;
    }
    return KRR_OK;
}

constexpr size_t ts_smem_limit() { return 227 * 1024; }

size_t ts_smem_bytes(int stages, int b_bytes) {
    return (size_t)stages * TS_ABYTES + b_bytes + TS_IRING * sizeof(ItemHdr) + (6 * TS_NPMAX + TS_IRING + 4) * 4 +
           (size_t)(2 * stages + 7 + 3 * TS_IRING) * 8 + 16 + 1024;
}

int64_t ts_flag_count(const Ctx *c) { return 2 + 2 * c->nt + c->nt * (c->b / TS_SLAB); }

// Auxiliary buffer: exact block scales of the two FP16 vector buffers ([nt][TS_NPMAX]
// each), the inverse scales of the residual's operand ([n_pad / 128][TS_NPMAX]),
// the block column maxima of the two buffers ([nt][TS_NPMAX] each), the states of
// their blocks ([nt] 64-bit words each), then the progress counters.
int64_t ts_scale_count(const Ctx *c) { return c->nt * TS_NPMAX; }
int64_t res_scale_count(const Ctx *c) { return c->n_pad / TS_SLAB * TS_NPMAX; }

krr_status ensure_ts_buffers(Ctx *c, int64_t p) {
    const size_t vbytes = (size_t)3 * TS_NPMAX * c->n_pad * sizeof(__half);
    if (c->ts_vcap < vbytes) {
        for (__half **v : {&c->ts_v0, &c->ts_v1}) {
            if (*v) cudaFree(*v);
            *v = nullptr;
            if (dev_malloc(c, (void **)v, vbytes) != cudaSuccess) {
                c->ts_vcap = 0;
                c->last_error = "cudaMalloc failed for the sweep vector blocks";
                return KRR_ENOMEM;
            }
        }
        c->ts_vcap = vbytes;
    }
    const size_t abytes = (size_t)(4 * ts_scale_count(c) + res_scale_count(c)) * sizeof(float) +
                          (size_t)2 * c->nt * sizeof(unsigned long long) + (size_t)ts_flag_count(c) * sizeof(int);
    if (c->ts_aux_cap < abytes) {
        if (c->ts_aux) cudaFree(c->ts_aux);
        c->ts_aux = nullptr;
        if (dev_malloc(c, &c->ts_aux, abytes) != cudaSuccess) {
            c->ts_aux_cap = 0;
            c->last_error = "cudaMalloc failed for the sweep counters";
            return KRR_ENOMEM;
        }
        c->ts_aux_cap = abytes;
    }
    const size_t xbytes = (size_t)c->n_pad * p * sizeof(float);
    if (p > 0 && c->ts_xcap < xbytes) {
        if (c->ts_xt) cudaFree(c->ts_xt);
        c->ts_xt = nullptr;
        if (dev_malloc(c, (void **)&c->ts_xt, xbytes) != cudaSuccess) {
            c->ts_xcap = 0;
            c->last_error = "cudaMalloc failed for the sweep vector copy";
            return KRR_ENOMEM;
        }
        c->ts_xcap = xbytes;
    }
    return KRR_OK;
}

float *ts_scales(Ctx *c) { return (float *)c->ts_aux; }
float *res_scales(Ctx *c) { return ts_scales(c) + 2 * ts_scale_count(c); }
float *ts_block_maxima(Ctx *c) { return res_scales(c) + res_scale_count(c); }
unsigned long long *ts_states(Ctx *c) { return (unsigned long long *)(ts_block_maxima(c) + 2 * ts_scale_count(c)); }
int *ts_flags(Ctx *c) { return (int *)(ts_states(c) + 2 * c->nt); }

// dst (cols x rows, row-major) = src^T, src rows x cols row-major.  With sum:
// sum += src^T and dst = the earlier sum.  The additions carry the rounding error
// of a row on to the next (add_carry, runs of 32 rows; the padding rows from n on
// neither get nor pass one), so the rounding errors of a column of A nearly
// cancel: K has a large constant component, through which their sum (about
// sqrt(N) half ulps with independent roundings) would be the floor of the
// residual and the common error of the predictions.
__global__ void transpose_kernel(const float *__restrict__ src, int64_t rows, int64_t cols, int64_t n,
                                 float *__restrict__ dst, float *__restrict__ sum) {
    __shared__ float t[32][33];
    const int64_t r0 = (int64_t)blockIdx.y * 32, c0 = (int64_t)blockIdx.x * 32;
    for (int k = threadIdx.y; k < 32; k += 8) {
        const int64_t r = r0 + k, cc = c0 + threadIdx.x;
        if (r < rows && cc < cols) t[k][threadIdx.x] = src[r * cols + cc];
    }
    __syncthreads();
    const int64_t r = r0 + threadIdx.x;
    if (sum) {
        if (threadIdx.y != 0 || r >= rows) return;
        // every load before the serial additions: a block has one warp at work here
        float sv[32];
#pragma unroll
        for (int k = 0; k < 32; ++k) sv[k] = (c0 + k < cols) ? sum[(c0 + k) * rows + r] : 0.f;
        float carry = 0.f;
#pragma unroll
        for (int k = 0; k < 32; ++k) {
            const int64_t cc = c0 + k;
            if (cc >= cols) break;
            if (cc >= n) carry = 0.f;
            dst[cc * rows + r] = sv[k];
            sum[cc * rows + r] = add_carry(sv[k], t[threadIdx.x][k], carry);
        }
        return;
    }
    for (int k = threadIdx.y; k < 32; k += 8) {
        const int64_t cc = c0 + k;
        if (r < rows && cc < cols) dst[cc * rows + r] = t[threadIdx.x][k];
    }
}

void launch_transpose(const float *src, int64_t rows, int64_t cols, float *dst, cudaStream_t s, float *sum = nullptr,
                      int64_t n = 0) {
    const dim3 grid((unsigned)((cols + 31) / 32), (unsigned)((rows + 31) / 32));
    count_launch(), transpose_kernel<<<grid, dim3(32, 8), 0, s>>>(src, rows, cols, n, dst, sum);
}

krr_status run_ts(Ctx *c, int job, float *rhs, float *out, int64_t p) {
    const int64_t b = c->b, nt = c->nt;
    if (b % TS_SLAB != 0) {
        c->last_error = "tensor-core sweep: the tile edge must be a multiple of 128";
        return KRR_EINVAL;
    }
    KRR_TRY(ensure_ts_buffers(c, p));
    const bool fwd = (job == TS_FWD);
    const int abox = fwd ? 128 : 64;
    const int64_t noff = nt * (nt - 1) / 2;
    CUtensorMap mp, mw, mlh, mll, mvi, mvo;
    KRR_TRY(map_f16(c, &mp, c->pool, (int64_t)(c->pool_bytes / (2 * b)), b, abox));
    // the E4M3 copies live in the trailing tiles (only read when such tiles exist)
    KRR_TRY(map_f16(c, &mw, noff > 0 ? c->W : c->Linv_hi, (noff > 0 ? noff : 1) * b, b, abox));
    KRR_TRY(map_f16(c, &mlh, c->Linv_hi, nt * b, b, abox));
    KRR_TRY(map_f16(c, &mll, c->Linv_lo, nt * b, b, abox));
    float *sbase = ts_scales(c);
    int *flags = ts_flags(c);
    static PerDevice attr;
    if (!attr.has(c->device)) {
        KRR_CUDA_TRY(c, cudaFuncSetAttribute(tcsweep_kernel<16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)ts_smem_limit()));
        KRR_CUDA_TRY(c, cudaFuncSetAttribute(tcsweep_kernel<32>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)ts_smem_limit()));
        attr.put(c->device);
    }
    for (int64_t q0 = 0; q0 < p; q0 += TS_NPMAX) {
        TsParams sp;
        memset(&sp, 0, sizeof(sp));
        sp.job = job;
        sp.b = b;
        sp.nt = nt;
        sp.S = b / TS_SLAB;
        sp.KC = b / TS_KC;
        sp.items = 1 + sp.S * nt * (nt + 1) / 2;  // sum of the section sizes
        sp.pc = (int)std::min<int64_t>(TS_NPMAX, p - q0);
        sp.np = (sp.pc + 15) & ~15;
        sp.q0 = (int)q0;
        // column-major vectors ([p][n_pad]): one row per epilogue thread gives
        // coalesced accesses for every column
        sp.rs = 1;
        sp.cs = c->n_pad;
        sp.rhs = rhs;
        sp.out = out;
        sp.bm_in = ts_block_maxima(c);
        sp.bm_out = ts_block_maxima(c) + ts_scale_count(c);
        sp.vin = c->ts_v0;
        sp.vout = c->ts_v1;
        sp.sin = sbase;
        sp.sout = sbase + ts_scale_count(c);
        sp.ltab = c->ltab;
        sp.st_in = ts_states(c);
        sp.st_out = ts_states(c) + nt;
        sp.flags = flags;
        // B takes up to 64 KB (128 KB above 16 columns), A stages the rest, as many
        // as TS_NSMAX: 10 (6) of them from b = 1024 on
        sp.lkc = 0;
        while ((1 << sp.lkc) < sp.KC) ++sp.lkc;
        sp.bseg = (int)std::min<int64_t>(sp.KC, TS_BSEG);
        const int b_bytes = sp.bseg * 2 * sp.np * 128;
        int stages = TS_NSMAX;
        while (stages > 2 && ts_smem_bytes(stages, b_bytes) > ts_smem_limit()) --stages;
        sp.stages = stages;
        // kind::f16, D = F32, A = B = F16, A K-major (forward) or MN-major
        // (backward), B K-major, N = 2 np (hi and lo halves), M = 128
        sp.idesc = (1u << 4) | ((fwd ? 0u : 1u) << 15) | ((uint32_t)((2 * sp.np) >> 3) << 17) |
                   ((uint32_t)(TS_SLAB >> 4) << 24);
        sp.wait_ns = (uint64_t)c->opt.wait_budget_ns;
        sp.err = c->derr;
        const int64_t vrows = c->n_pad / 64 * 2 * sp.np;
        const int vbox = std::min(TS_BBOX, sp.bseg * 2 * sp.np);
        KRR_TRY(map_f16(c, &mvi, c->ts_v0, vrows, 64, vbox));
        KRR_TRY(map_f16(c, &mvo, c->ts_v1, vrows, 64, vbox));
        // the block maxima and the states and counters behind them
        KRR_CUDA_TRY(c, cudaMemsetAsync(ts_block_maxima(c), 0,
                                        (size_t)2 * ts_scale_count(c) * sizeof(float) +
                                            (size_t)2 * nt * sizeof(unsigned long long) +
                                            (size_t)ts_flag_count(c) * sizeof(int),
                                        c->stream));
        const size_t smem = ts_smem_bytes(stages, b_bytes);
        const int64_t grid = std::min<int64_t>(sp.items, grid_limit(c, GL_SWEEP));
        const auto kernel = (sp.np == 16) ? tcsweep_kernel<16> : tcsweep_kernel<32>;
        count_launch(), kernel<<<(unsigned)grid, TS_THREADS, smem, c->stream>>>(mp, mw, mlh, mll, mvi, mvo, sp);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) {
            c->last_error = std::string("tensor-core sweep launch: ") + cudaGetErrorString(e);
            return KRR_ECUDA;
        }
    }
    return KRR_OK;
}

}  // namespace

// x (n_pad x p) <- (L L^T)^-1 rhs with the stored mixed-precision factor on the
// tensor cores; the sweeps work on the column-major copy ts_xt: the forward
// sweep updates it in place and writes z to tmp, the backward sweep updates
// tmp in place and writes the solution to ts_xt.  rhs: row-major right-hand
// sides, or nullptr when ts_xt holds them already (tc_residual).  sum
// (optional): sum += x, and x holds the earlier sum.
krr_status tc_sweep_solve(Ctx *c, const float *rhs, float *x, float *tmp, int64_t p, float *sum) {
    KRR_TRY(ensure_ts_buffers(c, p));
    float *xt = c->ts_xt;
    if (rhs) launch_transpose(rhs, c->n_pad, p, xt, c->stream);
    KRR_TRY(run_ts(c, TS_FWD, xt, tmp, p));
    KRR_TRY(run_ts(c, TS_BWD, tmp, xt, p));
    launch_transpose(xt, p, c->n_pad, x, c->stream, sum, c->n);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        c->last_error = std::string("sweep transposes: ") + cudaGetErrorString(e);
        return KRR_ECUDA;
    }
    return KRR_OK;
}

namespace {

// FP32 row-major matrix, boxes of 32 columns (128 bytes) x box_rows, 128-byte swizzle.
krr_status map_f32(Ctx *c, CUtensorMap *m, const void *base, int64_t rows, int64_t cols, int box_rows) {
    EncodeFn enc = encoder(c);
    if (!enc) return KRR_ECUDA;
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)(cols * 4)};
    const cuuint32_t box[2] = {32u, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void *>(base), dims, strides, box, estr,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        c->last_error = "cuTensorMapEncodeTiled (tensor-core residual) failed with code " + std::to_string((int)r);
        return KRR_ECUDA;
    }
    return KRR_OK;
}

size_t rs_smem_bytes(int np) {
    return (size_t)RS_NSTG * (RS_STG + 3 * np * 128) + TS_IRING * sizeof(int) +
           (size_t)(3 * RS_NSTG + 2 * RS_NACC + 2 * TS_IRING + 1) * 8 + 16 + 1024;
}

template <int NP>
krr_status launch_res(Ctx *c, const CUtensorMap &mk128, const CUtensorMap &mk64, const CUtensorMap &ma,
                      const RsParams &rp) {
    static PerDevice attr;
    if (!attr.has(c->device)) {
        KRR_CUDA_TRY(c, cudaFuncSetAttribute(tcres_kernel<NP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)ts_smem_limit()));
        attr.put(c->device);
    }
    const int64_t grid = std::min<int64_t>(rp.items, grid_limit(c, GL_RESIDUAL));
    count_launch(), tcres_kernel<NP><<<(unsigned)grid, RS_THREADS, rs_smem_bytes(NP), c->stream>>>(mk128, mk64, ma, rp);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        c->last_error = std::string("tensor-core residual launch: ") + cudaGetErrorString(e);
        return KRR_ECUDA;
    }
    return KRR_OK;
}

}  // namespace

// r = y - (K + lambda I) a on the tensor cores (mixed mode), rounded to FP32
// and column-major in c->ts_xt, the right-hand side of the next sweeps;
// ||r||_F^2 and ||y||_F^2 into c->red[RED_RNORM], [RED_RNORM + 1], ||a||_F^2 into
// c->red[RED_ANORM].
krr_status tc_residual(Ctx *c, const float *y, const float *a, int64_t p) {
    const int64_t b = c->b, nt = c->nt, S = b / TS_SLAB, n_pad = c->n_pad;
    KRR_TRY(ensure_ts_buffers(c, p));
    int *flags = ts_flags(c);
    const int64_t ntri = nt * (nt + 1) / 2;
    CUtensorMap mk128, mk64, ma;
    KRR_TRY(map_f32(c, &mk128, c->Kd, ntri * b, b, 128));
    KRR_TRY(map_f32(c, &mk64, c->Kd, ntri * b, b, 64));
    const int64_t pmax = std::min<int64_t>(p, TS_NPMAX);
    const int64_t nblk = n_pad / TS_SLAB, fblk = (n_pad + 255) / 256;
    int64_t part_count = 0;
    ResGrid gr;
    KRR_TRY(res_reserve(
        nt, S, b / TS_KC, grid_limit(c, GL_RESIDUAL), &c->rs_slots,
        [&](const ResGrid &q) {
            part_count = q.slots() * pmax * n_pad;
            const int64_t need = part_count + nblk * pmax + 3 * fblk * p;
            if (c->rs_part_cap >= need) return KRR_OK;
            std::string earlier = c->last_error;
            c->rs_part_cap = 0;
            const krr_status st = dev_alloc(c, &c->rs_part, (size_t)need, "residual partial sums");
            if (st == KRR_OK) c->rs_part_cap = need;
            if (st == KRR_ENOMEM && q.slots() > 1) c->last_error.swap(earlier);  // fewer are tried: no failure yet
            return st;
        },
        &gr));
    double *cs_part = c->rs_part + part_count, *np_part = cs_part + nblk * pmax;
    float *inv_s = res_scales(c);
    for (int64_t q0 = 0; q0 < p; q0 += TS_NPMAX) {
        const int pc = (int)std::min<int64_t>(TS_NPMAX, p - q0), np = (pc + 15) & ~15;
        // item counter, abort flag, block counters of the two small kernels
        // (the second one's runs over all column chunks)
        KRR_CUDA_TRY(c, cudaMemsetAsync(flags, 0, (q0 == 0 ? 4 : 3) * sizeof(int), c->stream));
        count_launch(), res_operand_kernel<<<(unsigned)nblk, TS_EPI, 0, c->stream>>>(
            a, p, (int)q0, pc, np, n_pad, c->ts_v0, inv_s, cs_part, c->colsum, flags + 2);
        KRR_TRY(map_f16(c, &ma, c->ts_v0, 3 * np, n_pad, 3 * np));
        RsParams rp;
        memset(&rp, 0, sizeof(rp));
        rp.gr = gr;
        rp.b = (int)b;
        rp.items = (int)gr.items();
        rp.n_pad = n_pad;
        rp.pc = pc;
        rp.shift = c->red + RED_KSHIFT;
        rp.kbound = c->red + RED_KBOUND;
        rp.inv_s = inv_s;
        rp.part = c->rs_part;
        rp.flags = flags;
        rp.idesc_k = (1u << 4) | ((uint32_t)((3 * np) >> 3) << 17) | ((uint32_t)(TS_SLAB >> 4) << 24);
        rp.idesc_mn = rp.idesc_k | (1u << 15);
        rp.idesc_k2 = (1u << 4) | ((uint32_t)((2 * np) >> 3) << 17) | ((uint32_t)(TS_SLAB >> 4) << 24);
        rp.idesc_mn2 = rp.idesc_k2 | (1u << 15);
        rp.wait_ns = (uint64_t)c->opt.wait_budget_ns;
        rp.err = c->derr;
        KRR_TRY(np == 16 ? launch_res<16>(c, mk128, mk64, ma, rp) : launch_res<32>(c, mk128, mk64, ma, rp));
        count_launch(), res_finish_kernel<<<dim3((unsigned)fblk, (unsigned)pc), 256, 0, c->stream>>>(
            y, a, p, (int)q0, pc, n_pad, c->rs_part, gr.slots(), (float)c->lambda, c->red + RED_KSHIFT, c->colsum,
            c->ts_xt, np_part, (int)(fblk * p), flags + 3, c->red);
        KRR_TRY(check_launch(c, "residual"));
    }
    return KRR_OK;
}

}  // namespace krr

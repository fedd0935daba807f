// Diagonal step of the tile Cholesky (Alg. 3, the POTRF of tile (k, k)) and
// the triangular inverse of the factor, as one persistent dataflow kernel over
// 64 x 64 blocks of the b x b tile (FP32).
//
// The critical path is the chain of diagonal blocks P(0) -> P(1) -> ... ->
// P(NB - 1), NB = b / 64, so one CTA (block 0) does nothing else and keeps the
// inverse it needs next in shared memory:
//   P(q)   for q >= 1 L_q,q-1 = A_q,q-1 X_q-1,q-1^T and A_qq -= L_q,q-1
//          L_q,q-1^T, then L_qq = chol(A_qq) and X_qq = inv(L_qq).
// A loader warp of that CTA waits for the updates of A_q,q-1 and A_qq and
// copies them in (cp.async) while P(q - 1) is still being factored; a publisher
// warp fences and raises the progress counters, so neither the waits nor the
// fences stall the eight compute warps.
//
// The other CTAs claim items from a device counter, in an order in which every
// item depends only on earlier items and on the chain:
//   for q = 0 .. NB-1:
//     for i = q + 2 .. NB-1:
//       T(i, q)     L_iq = A_iq X_qq^T
//       U(i, j, q)  A_ij -= L_iq L_jq^T                 (q < j <= i)
//     X(q, j), j <= q: row q of the inverse: X_qj = -X_qq sum_{j<=k<q} L_qk X_kj,
//                   its transpose (for the backward substitution) and its FP16
//                   hi/lo split (operands of the tensor-core panel solve).
// Row q of the inverse needs the rows above it and X_qq only, so the inverse is
// finished one product after the last diagonal block.  Blocks of X above the
// diagonal are zero from the allocation on.
// Progress counters: pdone[q], tdone[i][q], upd[i][j] (updates applied to block
// (i, j)), xdone[i][j].  Items wait only for items claimed before them by
// running CTAs and for the chain, which waits only for such items.  CTAs are
// launched in clusters of two, so at least one other CTA runs with the chain
// and the kernel progresses however many more find an SM.  Every wait is
// bounded (%globaltimer) and ends the kernel with KRR_ETIMEOUT.  Blocks written
// by other CTAs are read through L2 (ld.global.cg, cp.async.cg).
//
// What bounds it: latency.  A link of the chain is one 64 x 64 x 64 product,
// half of one, and the 64-column factor, whose pivots are serial.  One
// tile of b = 1024 alone takes 0.266 ms (a link 16 us: the first product 1.4,
// the second 1.7 and its store 0.6, the 64-column factor 11, the stores 0.8) and
// one of 256 0.07 ms; with the chain's
// blocks as items of the common queue (every link paying a claim, the wait for
// the counters, the loads and the publication) and the inverse by recursive
// doubling after the factorisation it was 0.50 and 0.12 ms.
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <string.h>

#include <algorithm>
#include <string>

#include "krr_internal.h"

namespace krr {

namespace {

constexpr int DB = 64;          // block edge
constexpr int DS = DB + 4;      // row stride of a block in shared memory: 16-byte rows, 8 rows apart in banks
constexpr int DC = 256;         // compute threads
constexpr int DT = DC + 64;     // and, in the chain CTA, the loader and the publisher warp
constexpr int DMAX_NB = 64;     // blocks per tile edge supported (b <= 4096)

typedef float Blk[DB][DS];

struct DiagParams {
    float *W;          // tile, overwritten by L (lower part)
    float *X;          // inverse (zero above the diagonal)
    float *XT;         // transpose of the inverse
    __half *hi, *lo;   // FP16 split of the inverse (or null)
    int64_t b;
    int NB;
    int64_t tile_k;
    int items;
    int *ctr;          // counters (layout in ctr_* below)
    double *lkk;       // out: sqrt of the largest diagonal entry of the tile before the factorisation
    DevErrors *err;
    uint64_t wait_ns;
};

// counter layout: [0] item counter, [1] abort, then pdone[NB], tdone[NB * NB],
// upd[NB * NB], xdone[NB * NB]
__device__ __forceinline__ int *ctr_pdone(const DiagParams &p) { return p.ctr + 2; }
__device__ __forceinline__ int *ctr_tdone(const DiagParams &p) { return ctr_pdone(p) + p.NB; }
__device__ __forceinline__ int *ctr_upd(const DiagParams &p) { return ctr_tdone(p) + p.NB * p.NB; }
__device__ __forceinline__ int *ctr_xdone(const DiagParams &p) { return ctr_upd(p) + p.NB * p.NB; }

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint64_t globaltimer() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ int ld_acquire(const int *p) {
    int v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void record_timeout(const DiagParams &p) {
    atomicExch(&p.ctr[1], 1);
    atomicCAS(&p.err->code, 0, (int)KRR_ETIMEOUT);
}

// Bounded wait (one thread) until *c >= target; false on expiry / abort.
// Polls back off exponentially (32 ns up to 256 ns) so that many waiting
// CTAs do not flood the L2 slice holding the counters.
__device__ bool wait_ge(const int *c, int target, const DiagParams &p) {
    if (ld_acquire(c) >= target) return true;
    const uint64_t t0 = globaltimer();
    uint32_t nap = 32;
    for (uint32_t it = 1;; ++it) {
        __nanosleep(nap);
        if (nap < 256) nap <<= 1;
        if (ld_acquire(c) >= target) return true;
        if ((it & 15) == 0) {
            if (*(volatile int *)&p.ctr[1]) return false;
            if (globaltimer() - t0 > p.wait_ns) {
                record_timeout(p);
                return false;
            }
        }
    }
}

// Publishes the CTA's finished writes and increments a counter.
__device__ __forceinline__ void signal(int *c) {
    __threadfence();
    atomicAdd(c, 1);
}

// Barriers between the warps of the chain CTA.
__device__ __forceinline__ void mbar_init(uint64_t *b, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *b) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(b)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *b, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred P;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 P, [%1], %2;\n\t"
        "selp.b32 %0, 1, 0, P;\n\t}\n"
        : "=r"(ok)
        : "r"(smem_u32(b)), "r"(parity)
        : "memory");
    return ok != 0;
}
// Bounded: the warp waited for itself waits at most twice for a counter, so
// the limit lies beyond that.
__device__ bool wait_bar(uint64_t *b, uint32_t parity, const DiagParams &p) {
    if (mbar_try_wait(b, parity)) return true;
    const uint64_t t0 = globaltimer(), limit = 4 * p.wait_ns + drain_limit(p.wait_ns);
    for (uint32_t it = 1;; ++it) {
        if (mbar_try_wait(b, parity)) return true;
        if ((it & 31) == 0) {
            if (*(volatile int *)&p.ctr[1]) return false;
            if (globaltimer() - t0 > limit) {
                record_timeout(p);
                return false;
            }
        }
    }
}

// Barrier of the compute threads.
__device__ __forceinline__ void csync() { asm volatile("bar.sync 1, 256;" ::: "memory"); }

// ---------------------------------------------------------------------------
// Item list of the other CTAs.
// ---------------------------------------------------------------------------
enum DiagKind { K_T = 0, K_U = 1, K_X = 2 };

struct DItem {
    int kind;
    int i, j, q;  // T: (i, q), U: (i, j, q), X: (i, j)
};

// T and U items of column q: rows i = q + 2 .. NB - 1 hold 1 + (i - q) each.
__host__ __device__ inline int column_items(int NB, int q) {
    const int m = NB - q - 1;
    return m >= 1 ? m + m * (m + 1) / 2 - 2 : 0;
}

__host__ __device__ inline int item_count(int NB) {
    int n = 0;
    for (int q = 0; q < NB; ++q) n += column_items(NB, q) + q + 1;
    return n;
}

__device__ void decode_item(const DiagParams &p, int t, DItem &it) {
    const int NB = p.NB;
    for (int q = 0; q < NB; ++q) {
        const int g = column_items(NB, q);
        if (t < g) {
            it.q = q;
            for (int i = q + 2;; ++i) {
                const int row = 1 + (i - q);  // T, then U(i, q + 1 .. i)
                if (t < row) {
                    it.i = i;
                    it.j = q + t;
                    it.kind = (t == 0) ? K_T : K_U;
                    return;
                }
                t -= row;
            }
        }
        t -= g;
        if (t <= q) {
            // the diagonal block first: its split is ready at once
            it.kind = K_X;
            it.i = q;
            it.j = q - t;
            return;
        }
        t -= q + 1;
    }
    it.kind = -1;  // not reached: t < items
}

// ---------------------------------------------------------------------------
// 64 x 64 blocks.
// ---------------------------------------------------------------------------
// Asynchronous copy of a block into shared memory by `n` threads (tid < n).
__device__ __forceinline__ void load_async(Blk &dst, const float *src, int64_t ld, int tid, int n) {
    for (int e = tid; e < DB * DB / 4; e += n) {
        const int r = e / (DB / 4), c4 = (e % (DB / 4)) * 4;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(&dst[r][c4])), "l"(src + r * ld + c4)
                     : "memory");
    }
}
__device__ __forceinline__ void load_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void load_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void load_wait_but1() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }

// acc += A B^T (both row-major, K along the rows): thread (tx, ty) = (t % 16,
// t / 16) owns rows ty + 16 u and columns tx + 16 v.  Four K per step: 16-byte
// loads keep the shared-memory wavefronts (12 per step and warp) below the
// FMAs (64 / 4).  LOWER: only blocks v <= u.
template <bool LOWER = false>
__device__ __forceinline__ void mac_nt(const Blk &a, const Blk &b, float (&acc)[4][4]) {
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll 4
    for (int k = 0; k < DB; k += 4) {
        float4 av[4], bv[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) av[u] = *reinterpret_cast<const float4 *>(&a[ty + 16 * u][k]);
#pragma unroll
        for (int v = 0; v < 4; ++v) bv[v] = *reinterpret_cast<const float4 *>(&b[tx + 16 * v][k]);
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                if (LOWER && v > u) continue;
                acc[u][v] = fmaf(av[u].x, bv[v].x, acc[u][v]);
                acc[u][v] = fmaf(av[u].y, bv[v].y, acc[u][v]);
                acc[u][v] = fmaf(av[u].z, bv[v].z, acc[u][v]);
                acc[u][v] = fmaf(av[u].w, bv[v].w, acc[u][v]);
            }
    }
}

// acc = A E, E upper triangular in 16 x 16 blocks (entry (k, j) zero for k's
// block > j's).  A warp owns 16 columns and 32 rows, a thread 4 x 4 of them
// (nn_row, nn_col), and stops at its last nonzero block row; the column blocks
// are dealt to the warps so that the warps of a scheduler share the work
// evenly.  A block product moves half a shared-memory value per FMA into
// registers, 128 bytes a cycle, which bounds it: 3800 cycles in full.
__device__ __forceinline__ int nn_block() {
    const int w = threadIdx.x >> 6;  // two warps per block of columns
    return w < 2 ? w : 5 - w;
}
__device__ __forceinline__ int nn_row() { return ((threadIdx.x >> 5) & 1) * 32 + ((threadIdx.x & 31) >> 2) * 4; }
__device__ __forceinline__ int nn_col() { return 16 * nn_block() + (threadIdx.x & 3) * 4; }

__device__ __forceinline__ void mac_nn(const Blk &a, const Blk &e, float (&acc)[4][4]) {
    const int r = nn_row(), c = nn_col(), kend = 16 * (nn_block() + 1);
#pragma unroll 4
    for (int k = 0; k < kend; k += 4) {
        float4 av[4], ev[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) av[u] = *reinterpret_cast<const float4 *>(&a[r + u][k]);
#pragma unroll
        for (int s = 0; s < 4; ++s) ev[s] = *reinterpret_cast<const float4 *>(&e[k + s][c]);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const float as[4] = {av[u].x, av[u].y, av[u].z, av[u].w};
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                acc[u][0] = fmaf(as[s], ev[s].x, acc[u][0]);
                acc[u][1] = fmaf(as[s], ev[s].y, acc[u][1]);
                acc[u][2] = fmaf(as[s], ev[s].z, acc[u][2]);
                acc[u][3] = fmaf(as[s], ev[s].w, acc[u][3]);
            }
        }
    }
}

__device__ __forceinline__ void zero_acc(float (&acc)[4][4]) {
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[u][v] = 0.f;
}

// Steps 2 and 3 (below) of 16-column block Q of chol_inv_64 on 256 threads:
// thread (tc, tr) = (t % 16, t / 16) holds entry (tr, tc) of every 16 x 16
// block.  Q is a template parameter so that the sums of all blocks are
// straight code and run beside each other (16 dependent FMAs each; as a loop
// over a run-time Q step 3 took 1400 cycles, 910 now: the
// shared-memory loads of its 3 x 4 operands).
template <int Q>
__device__ __forceinline__ void eliminate_16(Blk &a, Blk &e) {
    constexpr int o = 16 * Q, NA = 3 - Q;  // block rows of A below, of E above (Q of them)
    const int tc = threadIdx.x & 15, tr = threadIdx.x >> 4;
    {
        float ecol[16], acc[3];
        float4 r4[3][4];
#pragma unroll
        for (int m = 0; m < 16; ++m) ecol[m] = e[o + m][o + tc];
#pragma unroll
        for (int u = 0; u < 3; ++u) {
            const float *row = (u < NA) ? &a[16 * (Q + 1 + u) + tr][o] : &e[16 * (u - NA) + tr][o];
#pragma unroll
            for (int m = 0; m < 4; ++m) r4[u][m] = *reinterpret_cast<const float4 *>(row + 4 * m);
            acc[u] = 0.f;
        }
#pragma unroll
        for (int m = 0; m < 4; ++m)
#pragma unroll
            for (int u = 0; u < 3; ++u) {
                acc[u] = fmaf(r4[u][m].x, ecol[4 * m], acc[u]);
                acc[u] = fmaf(r4[u][m].y, ecol[4 * m + 1], acc[u]);
                acc[u] = fmaf(r4[u][m].z, ecol[4 * m + 2], acc[u]);
                acc[u] = fmaf(r4[u][m].w, ecol[4 * m + 3], acc[u]);
            }
        __syncwarp();  // the 16 threads of a row share a warp
#pragma unroll
        for (int u = 0; u < 3; ++u) {
            float *row = (u < NA) ? &a[16 * (Q + 1 + u) + tr][o] : &e[16 * (u - NA) + tr][o];
            row[tc] = acc[u];
        }
    }
    csync();
    if constexpr (Q < 3) {
        // block (u, w): block row u of the NA of A (lower ones only) or of the
        // Q + 1 of E, columns of block Q + 1 + w
        float acc[4][3];
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int w = 0; w < 3; ++w) acc[u][w] = 0.f;
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            float4 lj[3], li[4];
#pragma unroll
            for (int w = 0; w < NA; ++w) lj[w] = *reinterpret_cast<const float4 *>(&a[o + 16 + 16 * w + tc][o + 4 * m]);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float *row = (u < NA) ? a[16 * (Q + 1 + u) + tr] : e[16 * (u - NA) + tr];
                li[u] = *reinterpret_cast<const float4 *>(row + o + 4 * m);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int w = 0; w < NA; ++w) {
                    if (u < NA && w > u) continue;
                    acc[u][w] = fmaf(li[u].x, lj[w].x, acc[u][w]);
                    acc[u][w] = fmaf(li[u].y, lj[w].y, acc[u][w]);
                    acc[u][w] = fmaf(li[u].z, lj[w].z, acc[u][w]);
                    acc[u][w] = fmaf(li[u].w, lj[w].w, acc[u][w]);
                }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int w = 0; w < NA; ++w) {
                if (u < NA && w > u) continue;
                float *dst = ((u < NA) ? a[16 * (Q + 1 + u) + tr] : e[16 * (u - NA) + tr]) + o + 16 + 16 * w + tc;
                // block row Q of E enters here: its entries right of the diagonal
                // block were zero
                *dst = ((u - NA == Q) ? 0.f : *dst) - acc[u][w];
            }
        csync();
    }
}

// ---------------------------------------------------------------------------
// Cholesky of the 64 x 64 block a (lower triangle in, L out) and E = X^T,
// X = L^-1 (rows of E in the 16-blocks on and above the diagonal), by the
// elimination of the 128 x 64 matrix [A; I] in four steps of 16 columns: the
// same row operations that turn A into L turn the identity into X^T, so the
// inverse needs no phase of its own.  Per step:
//   1. warp 0: lanes 0-15 hold the 16 rows of the diagonal block (kept
//      symmetric, so a lane also holds its column), lanes 16-31 the rows of
//      the identity below it; every lane runs the same operations, column by
//      column.  The broadcasts of row c need no pivot and run beside its
//      reciprocal square root: a column costs one broadcast, the root, one
//      product and one fused update in series.
//   2. the other 48 active rows (of A below the block, of E above it) times
//      the block's inverse;
//   3. the trailing update of both parts.
// A pivot that is not positive is recorded (first one wins) and replaced by 1
// so the rest stays finite.
// ---------------------------------------------------------------------------
__device__ void chol_inv_64(Blk &a, Blk &e, int &bad, float &mpiv) {
    const int t = threadIdx.x, lane = t & 31;
    const unsigned FULL = 0xffffffffu;
#pragma unroll 1
    for (int q = 0; q < 4; ++q) {
        const int o = 16 * q;
        if (t < 32) {
            const int l = lane & 15;
            float v[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                const float av = a[o + max(l, j)][o + min(l, j)];
                v[j] = (lane < 16) ? av : (j == l ? 1.f : 0.f);
            }
#pragma unroll
            for (int c = 0; c < 16; ++c) {
                float row[16];
#pragma unroll
                for (int i = c; i < 16; ++i) row[i] = __shfl_sync(FULL, v[i], c);
                float d = row[c];
                if (!(d > 0.f)) {
                    if (bad < 0) bad = o + c;
                    d = 1.f;
                }
                // 1 / sqrt(d): hardware estimate refined by one Newton-Raphson
                // step for the reciprocal square root, x <- x (3 - d x^2) / 2
                float inv = rsqrtf(d);
                inv = inv * fmaf(-0.5f * d * inv, inv, 1.5f);
                const float lcc = d * inv;
                mpiv = fminf(mpiv, lcc);
                v[c] = (lane == c) ? lcc : v[c] * inv;
#pragma unroll
                for (int i = c + 1; i < 16; ++i) v[i] = fmaf(-v[c], row[i] * inv, v[i]);
            }
            Blk &dst = (lane < 16) ? a : e;
#pragma unroll
            for (int j = 0; j < 16; j += 4) {
                float4 w;
                w.x = (lane < 16 && j > l) ? 0.f : v[j];
                w.y = (lane < 16 && j + 1 > l) ? 0.f : v[j + 1];
                w.z = (lane < 16 && j + 2 > l) ? 0.f : v[j + 2];
                w.w = (lane < 16 && j + 3 > l) ? 0.f : v[j + 3];
                *reinterpret_cast<float4 *>(&dst[o + l][o + j]) = w;
            }
        }
        csync();
        switch (q) {
            case 0: eliminate_16<0>(a, e); break;
            case 1: eliminate_16<1>(a, e); break;
            case 2: eliminate_16<2>(a, e); break;
            default: eliminate_16<3>(a, e);
        }
    }
}

// ---------------------------------------------------------------------------
// The chain CTA.
// ---------------------------------------------------------------------------
struct ChainBars {
    uint64_t full;      // loader -> compute: A_q,q-1 and A_qq are in
    uint64_t s1free;    // compute -> loader: the panel buffer is free
    uint64_t pubt, pubp;  // compute -> publisher: L_q,q-1 / L_qq and X_qq are written
    volatile int pubseq;  // publications finished (t and p alternate)
    int ok;
};

// s: [0] E = X_q-1,q-1^T, then X_qq^T; [1] A_q,q-1, then L_q,q-1; [2 + (q & 1)] A_qq
__device__ void chain(const DiagParams &p, Blk *s, ChainBars &cb) {
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int64_t b = p.b;
    const int NB = p.NB;
    auto blk = [&](float *m, int i, int j) { return m + (int64_t)i * DB * b + (int64_t)j * DB; };
    if (warp == 8) {
        // ------------------------------ loader ------------------------------
        load_async(s[2], p.W, b, lane, 32);
        load_commit();
        load_wait_all();
        __syncwarp();
        if (lane == 0) mbar_arrive(&cb.full);
        for (int q = 1; q < NB; ++q) {
            bool ok = true;
            if (lane == 0) {
                ok = wait_ge(ctr_upd(p) + q * NB + q - 1, q - 1, p) && wait_ge(ctr_upd(p) + q * NB + q, q - 1, p);
                if (ok) ok = wait_bar(&cb.s1free, (q - 1) & 1, p);
            }
            if (!__shfl_sync(0xffffffffu, (int)ok, 0)) break;
            __syncwarp();
            load_async(s[1], blk(p.W, q, q - 1), b, lane, 32);
            load_async(s[2 + (q & 1)], blk(p.W, q, q), b, lane, 32);
            load_commit();
            load_wait_all();
            __syncwarp();
            if (lane == 0) mbar_arrive(&cb.full);
        }
        return;
    }
    if (warp == 9) {
        // ----------------------------- publisher -----------------------------
        // largest diagonal entry of the tile before anything is overwritten:
        // the compute warps store L_00 after the arrival on barrier 2, the
        // other CTAs write after pdone[0]
        float mx = 0.f;
        for (int64_t r = lane; r < b; r += 32) mx = fmaxf(mx, __ldcg(p.W + r * b + r));
        for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if (lane == 0) *p.lkk = sqrt((double)mx);
        __syncwarp();  // the arrival counts the warp as a whole
        asm volatile("bar.arrive 2, 288;" ::: "memory");
        if (lane != 0) return;
        for (int q = 0; q < NB; ++q) {
            if (q > 0) {
                if (!wait_bar(&cb.pubt, (q - 1) & 1, p)) return;
                signal(ctr_tdone(p) + q * NB + q - 1);
                cb.pubseq = 2 * q;
            }
            if (!wait_bar(&cb.pubp, q & 1, p)) return;
            signal(ctr_pdone(p) + q);
            cb.pubseq = 2 * q + 1;
        }
        return;
    }
    // ------------------------------ compute ------------------------------
    const int tx = t & 15, ty = t >> 4;
    int bad = -1;
    float mpiv = 3.0e38f;
    // One thread of a warp off the pivot path arrives and waits for all.  The
    // publication before this one on the same barrier is through (it always
    // is: a link takes several times a publication).
    auto arrive_pub = [&](uint64_t *bar, int seq) {
        if (t == 255) {
            const uint64_t t0 = globaltimer();
            while (cb.pubseq < seq - 2 && globaltimer() - t0 < 4 * p.wait_ns && !*(volatile int *)&p.ctr[1]) {}
            mbar_arrive(bar);
        }
    };
    for (int q = 0; q < NB; ++q) {
        if (t == 255) cb.ok = wait_bar(&cb.full, q & 1, p) ? 1 : 0;
        csync();
        if (!cb.ok) return;
        Blk &A = s[2 + (q & 1)];
        if (q > 0) {
            // L_q,q-1 = A_q,q-1 X_q-1,q-1^T
            float acc[4][4];
            zero_acc(acc);
            mac_nn(s[1], s[0], acc);
            csync();
            float *g = blk(p.W, q, q - 1);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float4 w = make_float4(acc[u][0], acc[u][1], acc[u][2], acc[u][3]);
                const int r = nn_row() + u, c = nn_col();
                *reinterpret_cast<float4 *>(&s[1][r][c]) = w;
                __stcg(reinterpret_cast<float4 *>(g + (int64_t)r * b + c), w);
            }
            csync();
            arrive_pub(&cb.pubt, 2 * q);
            // A_qq -= L_q,q-1 L_q,q-1^T (lower blocks)
            zero_acc(acc);
            mac_nt<true>(s[1], s[1], acc);
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int v = 0; v <= u; ++v) A[ty + 16 * u][tx + 16 * v] -= acc[u][v];
            csync();
        }
        if (t == 255) mbar_arrive(&cb.s1free);
        int bq = -1;
        chol_inv_64(A, s[0], bq, mpiv);
        if (bq >= 0 && bad < 0) bad = q * DB + bq;
        if (q == 0) asm volatile("bar.sync 2, 288;" ::: "memory");
        // L_qq and X_qq^T by rows, X_qq by columns of E
        float *gl = blk(p.W, q, q), *gt = blk(p.XT, q, q), *gx = blk(p.X, q, q);
        {
            // X first: the other CTAs wait for it.  Lanes along the rows of E:
            // 16-byte reads, 128-byte stores
            const int k = t & 63, c0 = (t >> 6) * 16;
#pragma unroll
            for (int c = c0; c < c0 + 16; c += 4) {
                const float4 w = *reinterpret_cast<const float4 *>(&s[0][k][c]);
                const bool in = (c >> 4) >= (k >> 4);
                __stcg(gx + (int64_t)c * b + k, in ? w.x : 0.f);
                __stcg(gx + (int64_t)(c + 1) * b + k, in ? w.y : 0.f);
                __stcg(gx + (int64_t)(c + 2) * b + k, in ? w.z : 0.f);
                __stcg(gx + (int64_t)(c + 3) * b + k, in ? w.w : 0.f);
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int r = ty + 16 * u, c = 4 * tx;
            float4 w = *reinterpret_cast<const float4 *>(&s[0][r][c]);
            // E is not kept below its diagonal 16-blocks (no product reads it there)
            if ((c >> 4) < (r >> 4)) w = make_float4(0.f, 0.f, 0.f, 0.f);
            __stcg(reinterpret_cast<float4 *>(gt + (int64_t)r * b + c), w);
            const float4 l = *reinterpret_cast<const float4 *>(&A[r][c]);
            __stcg(reinterpret_cast<float4 *>(gl + (int64_t)r * b + c),
                   make_float4(c <= r ? l.x : 0.f, c + 1 <= r ? l.y : 0.f, c + 2 <= r ? l.z : 0.f,
                               c + 3 <= r ? l.w : 0.f));
        }
        csync();
        arrive_pub(&cb.pubp, 2 * q + 1);
    }
    if (t == 0) {
        p.err->min_pivot = fmin(p.err->min_pivot, (double)mpiv);
        if (bad >= 0 && atomicCAS(&p.err->code, 0, (int)KRR_ENOTPD) == 0) {
            p.err->bad_tile = p.tile_k;
            p.err->bad_column = p.tile_k * b + bad;
        }
    }
}

// (Without a bound ptxas takes 96 registers and spills; at the 168 that one CTA
// per SM allows the pivot loop comes out slower than at 144: 0.280 against
// 0.267 ms a tile of 1024.)
__global__ void __maxnreg__(144) diag_kernel(const DiagParams p) {
    extern __shared__ __align__(16) float diag_smem[];
    Blk *s = reinterpret_cast<Blk *>(diag_smem);  // four blocks
    __shared__ ChainBars cb;
    __shared__ int item_s;
    __shared__ int ok_s;
    __shared__ int rdy[DMAX_NB];
    const int64_t b = p.b;
    const int NB = p.NB;
    const int t = threadIdx.x;
    if (blockIdx.x == 0) {
        if (t == 0) {
            mbar_init(&cb.full, 1);
            mbar_init(&cb.s1free, 1);
            mbar_init(&cb.pubt, 1);
            mbar_init(&cb.pubp, 1);
            cb.pubseq = 0;
        }
        __syncthreads();
        chain(p, s, cb);
        return;
    }
    if (t >= DC) return;
    const int tx = t & 15, ty = t >> 4;
    int *upd = ctr_upd(p), *tdone = ctr_tdone(p), *pdone = ctr_pdone(p), *xdone = ctr_xdone(p);
    auto blk = [&](float *m, int i, int j) { return m + (int64_t)i * DB * b + (int64_t)j * DB; };
    while (true) {
        if (t == 0) item_s = atomicAdd(&p.ctr[0], 1);
        csync();
        const int n = item_s;
        if (n >= p.items) break;
        DItem it;
        decode_item(p, n, it);
        float acc[4][4];
        zero_acc(acc);
        if (it.kind == K_T) {
            // L_iq = A_iq X_qq^T, in place
            float *c = blk(p.W, it.i, it.q);
            if (t == 0) ok_s = (wait_ge(upd + it.i * NB + it.q, it.q, p) && wait_ge(pdone + it.q, 1, p)) ? 1 : 0;
            csync();
            if (!ok_s) break;
            load_async(s[0], c, b, t, DC);
            load_async(s[1], blk(p.X, it.q, it.q), b, t, DC);
            load_commit();
            load_wait_all();
            csync();
            mac_nt(s[0], s[1], acc);
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int v = 0; v < 4; ++v) __stcg(c + (int64_t)(ty + 16 * u) * b + tx + 16 * v, acc[u][v]);
            csync();
            if (t == 0) signal(tdone + it.i * NB + it.q);
        } else if (it.kind == K_U) {
            // A_ij -= L_iq L_jq^T
            if (t == 0)
                ok_s = (wait_ge(upd + it.i * NB + it.j, it.q, p) && wait_ge(tdone + it.j * NB + it.q, 1, p) &&
                        wait_ge(tdone + it.i * NB + it.q, 1, p)) ? 1 : 0;
            csync();
            if (!ok_s) break;
            load_async(s[0], blk(p.W, it.i, it.q), b, t, DC);
            load_async(s[1], blk(p.W, it.j, it.q), b, t, DC);
            load_commit();
            float *c = blk(p.W, it.i, it.j);
            float old[4][4];
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int v = 0; v < 4; ++v) old[u][v] = __ldcg(c + (int64_t)(ty + 16 * u) * b + tx + 16 * v);
            load_wait_all();
            csync();
            mac_nt(s[0], s[1], acc);
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int v = 0; v < 4; ++v) __stcg(c + (int64_t)(ty + 16 * u) * b + tx + 16 * v, old[u][v] - acc[u][v]);
            csync();
            if (t == 0) signal(upd + it.i * NB + it.j);
        } else if (it.i == it.j) {
            // FP16 split of X_ii (the chain wrote X_ii and its transpose)
            if (t == 0) ok_s = wait_ge(pdone + it.i, 1, p) ? 1 : 0;
            csync();
            if (!ok_s) break;
            if (p.hi) {
                const float *src = blk(p.X, it.i, it.i);
                const int64_t o0 = (int64_t)it.i * DB * b + (int64_t)it.i * DB;
                for (int e = t; e < DB * DB; e += DC) {
                    const int64_t o = (int64_t)(e / DB) * b + e % DB;
                    const float v = __ldcg(src + o);
                    const __half h = __float2half_rn(v);
                    p.hi[o0 + o] = h;
                    p.lo[o0 + o] = __float2half_rn(v - __half2float(h));
                }
            }
        } else {
            // X_ij = -X_ii sum_{j <= k < i} L_ik X_kj: the operands of step k + 1
            // are copied in while step k is multiplied, as far as they are ready
            const int i = it.i, j = it.j, len = i - j;
            auto dep = [&](int k) { return (k == j) ? pdone + j : xdone + k * NB + j; };
            if (t < len) {
                const int k = j + t;
                rdy[t] = (ld_acquire(tdone + i * NB + k) >= 1 && ld_acquire(dep(k)) >= 1) ? 1 : 0;
            }
            csync();
            bool ok = true;
            auto issue = [&](int e) -> bool {
                const int k = j + e;
                if (!rdy[e]) {
                    if (t == 0) ok_s = (wait_ge(tdone + i * NB + k, 1, p) && wait_ge(dep(k), 1, p)) ? 1 : 0;
                    csync();
                    if (!ok_s) return false;
                }
                load_async(s[2 * (e & 1)], blk(p.W, i, k), b, t, DC);
                load_async(s[2 * (e & 1) + 1], blk(p.XT, j, k), b, t, DC);
                load_commit();
                return true;
            };
            ok = issue(0);
            int issued = 1;
            for (int e = 0; e < len && ok; ++e) {
                if (issued == e) {  // step e was not ready when step e - 1 ran
                    ok = issue(e);
                    if (!ok) break;
                    ++issued;
                }
                if (e + 1 < len && rdy[e + 1]) {
                    issue(e + 1);
                    ++issued;
                    load_wait_but1();
                } else {
                    load_wait_all();
                }
                csync();
                mac_nt(s[2 * (e & 1)], s[2 * (e & 1) + 1], acc);
                csync();
            }
            if (!ok) break;
            if (t == 0) ok_s = wait_ge(pdone + i, 1, p) ? 1 : 0;
            // the sum, transposed, is the second operand
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int v = 0; v < 4; ++v) s[1][tx + 16 * v][ty + 16 * u] = acc[u][v];
            csync();
            if (!ok_s) break;
            load_async(s[0], blk(p.X, i, i), b, t, DC);
            load_commit();
            load_wait_all();
            csync();
            zero_acc(acc);
            mac_nt(s[0], s[1], acc);
            float *gx = blk(p.X, i, j);
            const int64_t o0 = (int64_t)i * DB * b + (int64_t)j * DB;
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    const int64_t o = (int64_t)(ty + 16 * u) * b + tx + 16 * v;
                    const float x = -acc[u][v];
                    __stcg(gx + o, x);
                    s[2][tx + 16 * v][ty + 16 * u] = x;
                    if (p.hi) {
                        const __half h = __float2half_rn(x);
                        p.hi[o0 + o] = h;
                        p.lo[o0 + o] = __float2half_rn(x - __half2float(h));
                    }
                }
            csync();
            float *gt = blk(p.XT, j, i);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int r = ty + 16 * u;
                __stcg(reinterpret_cast<float4 *>(gt + (int64_t)r * b + 4 * tx),
                       *reinterpret_cast<const float4 *>(&s[2][r][4 * tx]));
            }
            csync();
            if (t == 0) signal(xdone + i * NB + j);
        }
        csync();  // the buffers and flags are free
    }
    load_wait_all();
}

constexpr size_t diag_smem_bytes() { return 4 * sizeof(Blk); }

}  // namespace

int64_t diag_counter_count(int64_t b) {
    const int64_t NB = b / DB;
    return 2 + NB + 3 * NB * NB;
}

// Factor + inverse of diagonal tile k in FP32 (W in place, Linv, LinvT and
// the FP16 split of Linv when present; these are zero above the diagonal from
// their allocation on).  The counters `ctr` hold diag_counter_count(b) ints;
// lkk receives the square root of the tile's largest diagonal entry.
krr_status launch_diag_dataflow(Ctx *c, int64_t k, float *W, float *X, float *XT, __half *hi, __half *lo, int *ctr,
                                double *lkk, cudaStream_t s, int64_t cta_cap) {
    const int64_t b = c->b;
    if (b % DB != 0 || b / DB > DMAX_NB) {
        c->last_error = "diagonal step: tile edge must be a multiple of 64 and at most 4096";
        return KRR_EINVAL;
    }
    static PerDevice attr;
    if (!attr.has(c->device)) {
        KRR_CUDA_TRY(c, cudaFuncSetAttribute(diag_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)diag_smem_bytes()));
        attr.put(c->device);
    }
    DiagParams p;
    memset(&p, 0, sizeof(p));
    p.W = W;
    p.X = X;
    p.XT = XT;
    p.hi = hi;
    p.lo = lo;
    p.b = b;
    p.NB = (int)(b / DB);
    p.tile_k = k;
    p.items = item_count(p.NB);
    p.ctr = ctr;
    p.lkk = lkk;
    p.err = c->derr;
    p.wait_ns = (uint64_t)c->opt.wait_budget_ns;
    KRR_CUDA_TRY(c, cudaMemsetAsync(ctr, 0, (size_t)diag_counter_count(b) * sizeof(int), s));
    int64_t gl = grid_limit(c, GL_DIAG);
    if (cta_cap > 0 && cta_cap < gl) gl = cta_cap;
    // the chain CTA and at least one other, in clusters of two
    const int64_t grid = std::max<int64_t>(2, std::min<int64_t>(gl, p.NB * (p.NB + 1) / 2)) / 2 * 2;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(DT);
    cfg.dynamicSmemBytes = diag_smem_bytes();
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    count_launch();
    const cudaError_t e = cudaLaunchKernelEx(&cfg, diag_kernel, p);
    if (e != cudaSuccess) {
        cudaGetLastError();
        c->last_error = std::string("diagonal step launch: ") + cudaGetErrorString(e);
        return KRR_ECUDA;
    }
    return KRR_OK;
}

}  // namespace krr

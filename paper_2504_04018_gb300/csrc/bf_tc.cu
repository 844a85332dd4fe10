// Exact range-filtered k-NN on the 5th-generation tensor cores (tcgen05).
//
// Dot products q.x come from three BF16 MMAs per K step accumulated in FP32
// in tensor memory (split precision: q = q_hi + q_lo, x = x_hi + x_lo with
// BF16 parts, q.x ~ q_hi.x_hi + q_hi.x_lo + q_lo.x_hi; the dropped q_lo.x_lo
// and the split residuals are below 2^-17 relative). Queries are sorted and
// tiled by 128 (one TMEM lane each); a query tile visits the 128-point tiles
// its ranges cover (128 TMEM columns per tile). The pipelined kernel below
// is warp-specialised: bulk copies of pre-swizzled operand blocks, two MMA
// threads, and eight epilogue warps that keep the K1 best approximate
// distances per query.
//
// A second kernel merges a query's lists, recomputes exact FP32 distances
// (direct form) of the K1 best candidates, sorts them, and certifies the
// result: with delta_q a bound on |approximate - exact| for every point of the
// range, the top k is proven when the exact k-th distance is below (K1-th
// approximate distance - delta_q). Queries without a certificate run again
// with a longer list, then through the exact SIMT brute force.
#include "esg_internal.cuh"

#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <type_traits>
#include <vector>

esg_status esg_bruteforce_redo(const float *base, int64_t n, int32_t d, int metric, const float *queries,
                               int64_t nq, const int64_t *l, const int64_t *r, int32_t k,
                               const std::vector<int64_t> &idx, int64_t *out_ids, float *out_dist,
                               int32_t *out_count, cudaStream_t stream);

namespace {

constexpr int TM = 128;            // queries per CTA (TMEM lanes)
constexpr int TN = 128;            // points per tile (TMEM columns)
constexpr int TK = 64;             // K chunk: 64 BF16 = one 128-byte swizzled row
constexpr int CHUNK = TM * TK * 2; // bytes of one 128 x 64 BF16 operand chunk (16 KB)

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

// Shared-memory matrix descriptor: K-major operand, 128-byte swizzle, rows of
// 128 bytes, 8-row groups 1024 bytes apart (stride byte offset), sm_100
// descriptor version 1.
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)(16u >> 4) << 16;
    d |= (uint64_t)(1024u >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

// Instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both
// K-major, N = TN, M = TM.
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(TN >> 3) << 17) |
                            ((uint32_t)(TM >> 4) << 24);

__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n"
        :: "r"(tmem_d), "l"(a), "l"(b), "r"(kIdesc), "r"(acc));
}

// The same with the A operand in tensor memory: row i in lane i, 16 BF16 of K
// packed in pairs in 8 columns from tmem_a on.
__device__ __forceinline__ void mma_bf16_ta(uint32_t tmem_d, uint32_t tmem_a, uint64_t b, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}\n"
        :: "r"(tmem_d), "r"(tmem_a), "l"(b), "r"(kIdesc), "r"(acc));
}

__device__ __forceinline__ void mma_commit(uint32_t mbar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                 :: "r"(mbar) : "memory");
}

// 32 consecutive accumulator columns of the warp's 32 TMEM lanes (one
// register each), waiting for the load inside the same asm statement so that
// no use of the registers can be scheduled before the wait.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,"
        "%25,%26,%27,%28,%29,%30,%31}, [%32];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
          "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
          "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]),
          "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// 32 words per lane into 32 consecutive columns of the warp's 32 TMEM lanes.
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint4 (&w)[8]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,"
        "%28,%29,%30,%31,%32};"
        :: "r"(taddr), "r"(w[0].x), "r"(w[0].y), "r"(w[0].z), "r"(w[0].w), "r"(w[1].x), "r"(w[1].y), "r"(w[1].z),
           "r"(w[1].w), "r"(w[2].x), "r"(w[2].y), "r"(w[2].z), "r"(w[2].w), "r"(w[3].x), "r"(w[3].y), "r"(w[3].z),
           "r"(w[3].w), "r"(w[4].x), "r"(w[4].y), "r"(w[4].z), "r"(w[4].w), "r"(w[5].x), "r"(w[5].y), "r"(w[5].z),
           "r"(w[5].w), "r"(w[6].x), "r"(w[6].y), "r"(w[6].z), "r"(w[6].w), "r"(w[7].x), "r"(w[7].y), "r"(w[7].z),
           "r"(w[7].w)
        : "memory");
}

// ---------------------------------------------------------- candidate lists
// A list entry is one 64-bit key: the distance's bits mapped to an unsigned
// that orders like the float, above the point's row, so that comparing keys
// orders by (distance, row). Lists and batches are held across a warp's lanes
// (element e = lane + 32 h in register h) and padded with kPad.
typedef unsigned long long Key;
constexpr Key kPad = ~0ull;

__device__ __forceinline__ Key make_key(float d, uint32_t row) {
    const uint32_t b = __float_as_uint(d);
    return ((Key)(b ^ ((uint32_t)((int32_t)b >> 31) | 0x80000000u)) << 32) | row;
}
// An exact distance's key: both zeros are one distance, ordered by the row
// alone (an inner product that underflows from below is -0, others +0).
__device__ __forceinline__ Key exact_key(float d, uint32_t row) { return make_key(d == 0.f ? 0.f : d, row); }
__device__ __forceinline__ float key_dist(Key k) {
    const uint32_t b = (uint32_t)(k >> 32);
    return __uint_as_float((b & 0x80000000u) ? (b ^ 0x80000000u) : ~b);
}
__device__ __forceinline__ Key key_min(Key a, Key b) { return a < b ? a : b; }
__device__ __forceinline__ Key key_max(Key a, Key b) { return a < b ? b : a; }

// A bitonic sequence of 32 NL keys sorted ascending.
template <int NL>
__device__ __forceinline__ void bitonic_asc(Key (&L)[NL], int lane) {
#pragma unroll
    for (int j = 16 * NL; j >= 32; j >>= 1)
#pragma unroll
        for (int h = 0; h < NL; ++h)
            if ((h & (j >> 5)) == 0) {
                const Key a = L[h], b = L[h | (j >> 5)];
                L[h] = key_min(a, b);
                L[h | (j >> 5)] = key_max(a, b);
            }
#pragma unroll
    for (int j = 16; j > 0; j >>= 1)
#pragma unroll
        for (int h = 0; h < NL; ++h) {
            const Key o = __shfl_xor_sync(0xffffffffu, L[h], j);
            L[h] = (lane & j) ? key_max(L[h], o) : key_min(L[h], o);
        }
}

// The 32 NL smallest keys of two ascending lists, ascending, into A. Element
// e of A meets element 32 NL - 1 - e of B.
template <int NL>
__device__ __forceinline__ void merge_lists(Key (&A)[NL], const Key (&B)[NL], int lane) {
    Key rev[NL];
#pragma unroll
    for (int h = 0; h < NL; ++h) rev[h] = __shfl_sync(0xffffffffu, B[NL - 1 - h], 31 - lane);
#pragma unroll
    for (int h = 0; h < NL; ++h) A[h] = key_min(A[h], rev[h]);
    bitonic_asc<NL>(A, lane);
}

// Full ascending sort of 32 NL keys.
template <int NL>
__device__ __forceinline__ void sort_asc(Key (&L)[NL], int lane) {
#pragma unroll
    for (int kk = 2; kk <= 32 * NL; kk <<= 1)
#pragma unroll
        for (int j = kk >> 1; j > 0; j >>= 1) {
            if (j >= 32) {
#pragma unroll
                for (int h = 0; h < NL; ++h)
                    if ((h & (j >> 5)) == 0) {
                        const Key a = L[h], b = L[h | (j >> 5)];
                        const bool up = ((32 * h) & kk) == 0;
                        L[h] = up ? key_min(a, b) : key_max(a, b);
                        L[h | (j >> 5)] = up ? key_max(a, b) : key_min(a, b);
                    }
            } else {
#pragma unroll
                for (int h = 0; h < NL; ++h) {
                    const Key o = __shfl_xor_sync(0xffffffffu, L[h], j);
                    const bool keep_min = (((lane + 32 * h) & kk) == 0) == ((lane & j) == 0);
                    L[h] = keep_min ? key_min(L[h], o) : key_max(L[h], o);
                }
            }
        }
}

// ------------------------------------------------------------------------
// Pipelined kernel. The operands are pre-tiled in global memory in exactly
// the shared-memory layout the MMA descriptors name (one 32 KB block per
// 128 rows x 64 dimensions: BF16 hi part, then lo part, 128-byte swizzle,
// zero padding past the last row and dimension), so every stage is one bulk
// copy on the TMA engine. Queries are sorted by (log2 of range width, l)
// and grouped into tiles of 128; a query tile only visits the point tiles
// that its queries' ranges cover; the CTAs (one per SM) run contiguous
// shares of that sequence of equal estimated cost, cut into work items at
// query-tile boundaries. Each CTA is warp-specialised:
//   warp 0      bulk copies: a ring of S point-tile stages (d <= 256), or of
//               stages with a query and a point chunk (streamed, larger d);
//   warps 1, 2  one thread each issues the MMAs of alternate tiles (warp 1 all
//               of them where a tile's stages are over half of the ring) into
//               a ring of 2 to 4 TMEM accumulators (128 columns each) and
//               commits them to mbarriers;
//   warps 3..10 epilogue, two groups of four warps (one per TMEM lane
//               quarter) that take alternate tiles. A thread owns one query
//               row: it reads the row's 128 columns 32 at a time, compares
//               each distance with the row's threshold and appends the few
//               that pass to the row's pending slots in shared memory. When a
//               row's slots run low all rows of the warp insert theirs into
//               lists of 24 or 32 held in registers, or (longer lists) the
//               warp merges the rows' by ranks into their lists in global
//               memory, which lowers the threshold. At d <= 256 group 0 also
//               puts the item's query tile into tensor memory (64 columns per
//               64 dimensions): the MMAs then read only the point operand from
//               shared memory, which at N = 128 otherwise limits them, and
//               all of it holds point stages.
// The eight warps share nothing but the thresholds: each (row, group) has its
// own list, so no warp waits for another one, and a row uses the other
// group's published distances, tagged with the work item: no point above t is
// among the K1 best when one list has K1 points up to t, or both have half as
// many.
// A row of a narrow range instead writes all its distances to global memory
// (a dense row, see kDenseWidth); the finish kernel selects from them.
// What bounds it: at 1M x 128 (10k queries, k = 10) a point tile is 24 MMAs,
// 0.74 us, and the CTAs take 1.1 to 1.2 us per tile: an accumulator is held for
// the MMAs and then for the group's reading, three of them are in turn, and
// everything that passes the shared-memory crossbar (norms, shuffles, pending
// slots) competes with the MMAs' operand reads. The operand blocks come from
// DRAM at 79 % of the copy bandwidth meanwhile (10.0 GB read, 0.85 GB written in
// 2.05 ms), the tensor pipe is active in half of the cycles. 4.67 -> 2.0 ms for the kernel,
// 1.52 -> 1.07 ms at 200,003 x 768 (2k queries), 256 -> 18 us for 61 queries over
// 99,991 x 100. Tried on the way: one issuer (a thread's waits and commits cost
// as much as a stage's MMAs), lists sorted by shuffle networks of 4 or 8 rows
// (1,100 to 1,900 cycles a row under the crossbar's load; all 32 rows of a warp
// insert into register lists in 4,000 to 5,000), the query tile in shared memory.
// Every wait is bounded (2 s of global time); a wait that runs out sets the
// error flag and all roles leave their loops.

constexpr int STAGE = 2 * CHUNK;          // hi + lo of a 128 x 64 block
constexpr int kEpiWarps = 8;
constexpr int kMmaWarps = 2;
constexpr int kThreads2 = 32 + 32 * kMmaWarps + 32 * kEpiWarps;
constexpr int kMaxK1v2 = 128;             // longest list
constexpr int kMaxStages = 6;
constexpr int kTmem = 512;                // TMEM columns: all, one CTA per SM
constexpr int kMaxResident = 4;           // 64-wide chunks of a query tile that fit beside two accumulators
// Columns between two checks of the pending slots, slots per row where the lists
// are in memory (a check's columns must fit, at most 32: one per lane of the
// merge), and how many of them make a row worth merging along with one that has
// to be. 20 slots leave room for five stages, 12 for three streamed stages. Rows
// with register lists have 16 (kPend in the kernel): five stages, two streamed.
constexpr int kCols = 8;
template <bool STREAM> struct Epi {
    static constexpr int kPend = STREAM ? 12 : 20, kFill = STREAM ? 4 : 8;
};
constexpr int kPendStride = 33;           // slots of one row 33 entries apart: no bank conflict when read
// Limit of the waits that let work already issued finish before a CTA exits
// (bulk copies, MMAs); the pipeline's own waits take Tc2Args::wait_ns.
constexpr unsigned long long kWaitNs = 2000000000ull;

struct WorkItem {
    int32_t qtile, off, cnt, pad;
};

struct Tc2Args {
    const unsigned char *xs, *qs;   // tiled operand blocks
    const float *xnorm, *qnorm;     // squared norms (queries in caller order)
    const int64_t *l, *r;
    const int32_t *qorder;          // sorted position -> caller's query index
    const int64_t *doff;            // sorted position -> first entry of a dense row, or -1
    float *dense;                   // distances of the dense rows' ranges, from point l & ~3 on
    const WorkItem *items;
    const int32_t *tiles;           // point-tile ids of all items
    const int32_t *cta_first;       // [grid + 1]: CTA c runs items [cta_first[c], cta_first[c + 1])
    int n_items;
    int64_t nv;                     // number of valid (sorted) queries
    int nk, metric, K1, S;
    int list_smem;                  // 1: lists of up to 64 in shared memory while they grow
    int n_acc;                      // TMEM accumulators
    int issuers;                    // MMA-issuing threads, 1 or 2
    int64_t n;                      // points
    Key *part;                      // [n_items][2 groups][128][K1] ascending lists
    int32_t *part_n;                // [n_items][2 groups][128] their lengths
    int32_t *err;
    unsigned long long wait_ns;     // limit of a pipeline wait (ESG_BF_WAIT_NS; default 2 s)
    int32_t stall;                  // failure-detection test: the producer first waits on a
                                    // barrier nothing arrives on, before it issues any copy
};

__device__ __forceinline__ unsigned long long gtime() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ bool mbar_try(uint32_t mbar, uint32_t parity) {
    uint32_t done = 0;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(done) : "r"(mbar), "r"(parity) : "memory");
    return done != 0;
}

// Bounded wait for the phase of the given parity. Gives up when another role
// has aborted (unless `ignore_abort`) or after limit_ns; on a timeout it
// raises the abort flag and the error flag.
__device__ __noinline__ bool wait_slow(uint32_t mbar, uint32_t parity, volatile int *abort_f, int32_t *err,
                                       unsigned long long limit_ns, bool ignore_abort) {
    unsigned long long t0 = 0;
    for (uint32_t it = 1;; ++it) {
        if (mbar_try(mbar, parity)) return true;
        if ((it & 127) == 0) {
            if (!ignore_abort && *abort_f) return false;
            const unsigned long long t = gtime();
            if (t0 == 0) t0 = t;
            else if (t - t0 > limit_ns) {
                *abort_f = 1;
                atomicExch(err, 1);
                return false;
            }
        }
    }
}

__device__ __forceinline__ bool wait_phase(uint32_t mbar, uint32_t parity, volatile int *abort_f, int32_t *err,
                                           unsigned long long limit_ns, bool ignore_abort = false) {
    return mbar_try(mbar, parity) || wait_slow(mbar, parity, abort_f, err, limit_ns, ignore_abort);
}

__device__ __forceinline__ void mbar_init(uint32_t mbar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(mbar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t mbar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(mbar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t mbar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(mbar) : "memory");
}
// Bulk global -> shared copy on the TMA engine, completion counted in bytes
// on the mbarrier (addresses 16-byte aligned, size a multiple of 16).
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void *src, uint32_t bytes, uint32_t mbar, uint64_t hint) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;"
                 :: "r"(dst), "l"(src), "r"(bytes), "r"(mbar), "l"(hint) : "memory");
}

// What a thread keeps of its row: pending entries, list entries, the list's
// K1-th distance t and its ceil(K1 / 2)-th distance th (+inf while it is
// shorter).
struct RowState {
    int cnt, len;
    float t, th;
};

// Merges the pending entries of the rows in `mask` (lanes of this warp) into
// their lists and updates the rows' state (held by lane r for row r); t and th
// are published as the item tag above the distance's bits. By ranks: lane e
// holds pending entry e and list entries e + 32 h; each pending entry is read
// by all lanes in turn (one broadcast), compared with what each lane holds,
// and a vote counts the list entries before it; then everything is stored at
// its rank. A sorting network costs the same comparisons but twice the
// shuffles' and loads' passes through the shared-memory crossbar, of which the
// MMAs' operand reads and the bulk copies leave little. The next row's entries
// are loaded meanwhile. Out of line: its call sites are many and rarely taken.
template <int NL>
__device__ __noinline__ RowState flush_rows(unsigned mask, const float2 *pend, Key *list, int K1, RowState st,
                                            volatile Key *pub, uint32_t tag) {
    const int lane = threadIdx.x & 31;
    __syncwarp();
    int r = __ffs(mask) - 1;
    int c = __shfl_sync(0xffffffffu, st.cnt, r), n = __shfl_sync(0xffffffffu, st.len, r);
    Key L[NL], p;
    auto load = [&](int row, int cr, int nr, Key (&l)[NL], Key &q) {
#pragma unroll
        for (int h = 0; h < NL; ++h) l[h] = lane + 32 * h < nr ? list[row * K1 + lane + 32 * h] : kPad;
        q = kPad;
        if (lane < cr) {
            const float2 e = pend[lane * kPendStride + row];
            q = make_key(e.x, __float_as_uint(e.y));
        }
    };
    load(r, c, n, L, p);
#pragma unroll 1
    while (true) {
        mask &= mask - 1;
        const int r2 = mask ? __ffs(mask) - 1 : r;
        const int c2 = __shfl_sync(0xffffffffu, st.cnt, r2), n2 = __shfl_sync(0xffffffffu, st.len, r2);
        Key L2[NL], p2;
        if (mask) load(r2, c2, n2, L2, p2);
        int rp = 0, rl[NL];   // ranks in the merged list
#pragma unroll
        for (int h = 0; h < NL; ++h) rl[h] = lane + 32 * h;
#pragma unroll 4
        for (int i = 0; i < c; ++i) {
            const float2 e = pend[i * kPendStride + r];
            const Key k = make_key(e.x, __float_as_uint(e.y));
            rp += k < p ? 1 : 0;
            int below = 0;
#pragma unroll
            for (int h = 0; h < NL; ++h) {
                rl[h] += k < L[h] ? 1 : 0;
                below += __popc(__ballot_sync(0xffffffffu, L[h] < k));
            }
            rp += lane == i ? below : 0;
        }
        const int m = min(K1, n + c);
        const bool pin = lane < c;
        if (pin && rp < K1) list[r * K1 + rp] = p;
#pragma unroll
        for (int h = 0; h < NL; ++h)
            if (lane + 32 * h < n && rl[h] < K1) list[r * K1 + rl[h]] = L[h];
        // the distances at rank K1 - 1 and in the middle
        auto at = [&](int rank) -> float {
            unsigned b = __ballot_sync(0xffffffffu, pin && rp == rank);
            uint32_t hi = (uint32_t)(p >> 32);
#pragma unroll
            for (int h = 0; h < NL; ++h) {
                const unsigned bh = __ballot_sync(0xffffffffu, lane + 32 * h < n && rl[h] == rank);
                if (bh) { b = bh; hi = (uint32_t)(L[h] >> 32); }
            }
            return key_dist((Key)__shfl_sync(0xffffffffu, hi, __ffs(b) - 1) << 32);
        };
        if (m > (K1 - 1) >> 1) {
            const float th = at((K1 - 1) >> 1), t = m == K1 ? at(K1 - 1) : INFINITY;
            if (lane == r) {
                st.th = th;
                st.t = t;
                pub[2 * TM] = ((Key)tag << 32) | __float_as_uint(th);
                pub[0] = ((Key)tag << 32) | __float_as_uint(t);
            }
        }
        if (lane == r) { st.cnt = 0; st.len = m; }
        if (!mask) break;
        r = r2; c = c2; n = n2; p = p2;
#pragma unroll
        for (int h = 0; h < NL; ++h) L[h] = L2[h];
    }
    __syncwarp();
    return st;
}

// Inserts the pending entries of every row (one thread each, all rows of the
// warp together) into the thread's ascending list of KR distances and points:
// every place takes its old entry, the one before it or the new one, all places
// at once. Ties keep the earlier entry.
template <int KR>
__device__ __forceinline__ void insert_pending(const float2 *pend, int lane, int cnt, float (&d)[KR], int32_t (&id)[KR]) {
    const int most = __reduce_max_sync(0xffffffffu, cnt);
#pragma unroll 1
    for (int i = 0; i < most; ++i) {
        const float2 e = pend[i * 32 + lane];
        const float x = i < cnt ? e.x : INFINITY;
        if (!__any_sync(0xffffffffu, x < d[KR - 1])) continue;   // the list has moved on meanwhile
        const int32_t xi = __float_as_int(e.y);
#pragma unroll
        for (int q = KR - 1; q >= 0; --q) {
            const bool here = x < d[q], before = q > 0 && x < d[q > 0 ? q - 1 : 0];
            id[q] = before ? id[q > 0 ? q - 1 : 0] : (here ? xi : id[q]);
            d[q] = q > 0 ? fminf(d[q], fmaxf(d[q > 0 ? q - 1 : 0], x)) : fminf(d[q], x);
        }
    }
}

// KR > 0: lists of K1 = KR entries in registers; 0: lists of up to 32 NL in memory.
template <bool L2, int KR, int NL, bool STREAM>
__global__ void __launch_bounds__(kThreads2, 1) tc_knn2_kernel(Tc2Args a) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    constexpr int kPend = KR ? 16 : Epi<STREAM>::kPend, kFill = Epi<STREAM>::kFill;
    constexpr int kStride = KR ? 32 : kPendStride;   // lists in registers: a slot's 32 rows side by side
    constexpr bool kSmemLists = KR == 0 && NL <= 2;   // see bf2_smem
    const int K1 = a.K1;
    // tile n of the CTA's run uses accumulator n mod n_acc and barrier n mod
    // n_bar, an even number: all uses of a barrier belong to one issuer and
    // one group, so that no one can be a phase ahead of the barrier (with three
    // barriers for three accumulators, an issuer whose tiles run ahead of the
    // other's would take an older phase of the same parity for its own)
    const uint32_t n_acc = (uint32_t)a.n_acc, n_bar = n_acc == 3 ? 6u : n_acc;
    // a stage: one point chunk, or (streamed) the query chunk and the point
    // chunk of one K step
    constexpr int stage_bytes = STREAM ? 2 * STAGE : STAGE;
    unsigned char *sB = smem_raw;
    float2 *s_pend = (float2 *)(sB + (size_t)a.S * stage_bytes);   // [8 warps][kPend][kStride]
    float *s_xn = (float *)(s_pend + kEpiWarps * kPend * kStride);   // [8 warps][128] tile norms
    Key *s_thr = (Key *)(s_xn + kEpiWarps * TN);             // [K1-th, middle][2 groups][128] published distances
    uint64_t *bars = (uint64_t *)(s_thr + 4 * TM);
    uint64_t *full = bars, *empty = bars + a.S;
    uint64_t *a_full = bars + 2 * a.S, *a_empty = a_full + 1;
    uint64_t *acc_full = a_full + 2, *acc_empty = acc_full + 6, *drain = acc_empty + 6;
    uint64_t *never = drain + 1;                              // nothing arrives on it
    uint32_t *tmem_slot = (uint32_t *)(never + 1);
    volatile int *abort_f = (volatile int *)(tmem_slot + 1);
    Key *s_list = (Key *)(tmem_slot + 2);                     // [8 warps][32][K1] if list_smem
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // this CTA's contiguous share of the work items
    const int it_begin = a.cta_first[blockIdx.x];
    const int it_end = a.cta_first[blockIdx.x + 1];

    if (threadIdx.x == 0) {
        for (int s = 0; s < a.S; ++s) {
            mbar_init(smem_u32(full + s), 1);
            mbar_init(smem_u32(empty + s), 1);
        }
        mbar_init(smem_u32(a_full), kEpiWarps / 2);
        mbar_init(smem_u32(a_empty), a.issuers);
        for (int b = 0; b < 6; ++b) {
            mbar_init(smem_u32(acc_full + b), 1);
            mbar_init(smem_u32(acc_empty + b), kEpiWarps / 2);
        }
        mbar_init(smem_u32(drain), a.issuers);
        mbar_init(smem_u32(never), 1);
        *abort_f = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(smem_u32(tmem_slot)), "r"(kTmem) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    for (int i = threadIdx.x; i < 4 * TM; i += kThreads2) s_thr[i] = kPad;   // no item has this tag
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;
    const uint32_t tmem_a = tmem + kTmem - 64 * (uint32_t)a.nk;   // resident query tile: hi chunks, lo chunks

    if (warp == 0) {
        if (lane == 0) {
            // ---------------- producer
            // operand blocks stream through the L2; lists in global memory stay
            uint64_t hint;
            asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(hint));
            uint32_t s = 0, ps = 0;
            uint32_t issued[kMaxStages] = {0};
            uint32_t ipar[kMaxStages] = {0};
            bool ok = true;
            if (a.stall && !wait_phase(smem_u32(never), 0u, abort_f, a.err, a.wait_ns)) ok = false;
            for (int it = it_begin; ok && it < it_end; ++it) {
                const WorkItem I = a.items[it];
                int32_t t_nx = a.tiles[I.off];
                for (int j = 0; ok && j < I.cnt; ++j) {
                    const int64_t t = t_nx;
                    if (j + 1 < I.cnt) t_nx = __ldg(a.tiles + I.off + j + 1);
                    for (int kc = 0; kc < a.nk; ++kc) {
                        if (!wait_phase(smem_u32(empty + s), ps ^ 1u, abort_f, a.err, a.wait_ns)) { ok = false; break; }
                        unsigned char *sg = sB + (size_t)s * stage_bytes;
                        mbar_expect_tx(smem_u32(full + s), (uint32_t)stage_bytes);
                        if (STREAM) {
                            bulk_g2s(smem_u32(sg), a.qs + ((int64_t)I.qtile * a.nk + kc) * STAGE, STAGE,
                                     smem_u32(full + s), hint);
                            sg += STAGE;
                        }
                        bulk_g2s(smem_u32(sg), a.xs + (t * a.nk + kc) * STAGE, STAGE, smem_u32(full + s), hint);
                        issued[s] = 1; ipar[s] = ps;
                        if (++s == (uint32_t)a.S) { s = 0; ps ^= 1u; }
                    }
                }
            }
            if (!ok) {
                // let the copies already issued land before the CTA can exit
                for (int q = 0; q < a.S; ++q)
                    if (issued[q]) wait_phase(smem_u32(full + q), ipar[q], abort_f, a.err, kWaitNs, true);
            }
        }
    } else if (warp <= kMmaWarps) {
        if (lane == 0 && warp <= a.issuers) {
            // ---------------- MMA issuers: one thread, or two that take the
            // tiles by parity (a thread's MMAs queue up behind its own waits
            // and commits, about as long as the MMAs of a stage takes: two
            // keep the tensor pipe fed)
            const uint32_t me = (uint32_t)(warp - 1), step = (uint32_t)a.issuers;
            const uint64_t bdesc0 = sdesc(smem_u32(sB));
            uint32_t s = me * (uint32_t)a.nk % (uint32_t)a.S, ps = me * (uint32_t)a.nk / (uint32_t)a.S & 1u, pa = 0;
            uint32_t n = me, n_end = 0, b = me, fb = me;   // tile of the run, its accumulator and barrier
            // the tile that used the accumulator before: its barrier and phase
            int before = (int)me - (int)n_acc;
            uint32_t eb = 0, pe = 0;
            bool ok = true;
            for (int it = it_begin; ok && it < it_end; ++it) {
                n_end += (uint32_t)a.items[it].cnt;
                if (!STREAM) {
                    if (!wait_phase(smem_u32(a_full), pa, abort_f, a.err, a.wait_ns)) { ok = false; break; }
                    pa ^= 1u;
                }
                for (; ok && n < n_end; n += step) {
                    if (before >= 0) {
                        if (!wait_phase(smem_u32(acc_empty + eb), pe, abort_f, a.err, a.wait_ns)) { ok = false; break; }
                        if ((eb += step) >= n_bar) { eb -= n_bar; pe ^= 1u; }
                    } else if ((before += (int)step) >= 0) {
                        eb = (uint32_t)before;
                    }
                    const uint32_t dt = tmem + b * TN;
                    for (int kc = 0; kc < a.nk; ++kc) {
                        if (!wait_phase(smem_u32(full + s), ps, abort_f, a.err, a.wait_ns)) { ok = false; break; }
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        // descriptors count 16-byte units: 2 per 16 dimensions, CHUNK / 16 from hi to lo
                        const uint64_t sd = bdesc0 + (uint64_t)(s * (stage_bytes >> 4));
                        const uint64_t bh = STREAM ? sd + (STAGE >> 4) : sd, bl = bh + (CHUNK >> 4);
                        const uint32_t first = kc == 0 ? 0u : 1u;
                        if (STREAM) {
                            const uint64_t ah = sd, al = sd + (CHUNK >> 4);
#pragma unroll
                            for (int st = 0; st < TK / 16; ++st) {
                                mma_bf16(dt, ah + 2 * st, bh + 2 * st, st == 0 ? first : 1u);
                                mma_bf16(dt, ah + 2 * st, bl + 2 * st, 1u);
                                mma_bf16(dt, al + 2 * st, bh + 2 * st, 1u);
                            }
                        } else {
                            const uint32_t ah = tmem_a + kc * 32, al = ah + a.nk * 32;
#pragma unroll
                            for (int st = 0; st < TK / 16; ++st) {
                                mma_bf16_ta(dt, ah + st * 8, bh + 2 * st, st == 0 ? first : 1u);
                                mma_bf16_ta(dt, ah + st * 8, bl + 2 * st, 1u);
                                mma_bf16_ta(dt, al + st * 8, bh + 2 * st, 1u);
                            }
                        }
                        mma_commit(smem_u32(empty + s));
                        if (++s == (uint32_t)a.S) { s = 0; ps ^= 1u; }
                    }
                    if (!ok) break;
                    mma_commit(smem_u32(acc_full + fb));
                    if ((b += step) >= n_acc) b -= n_acc;
                    if ((fb += step) >= n_bar) fb -= n_bar;
                    if (step == 2)   // past the other issuer's tile
                        for (s += (uint32_t)a.nk; s >= (uint32_t)a.S; s -= (uint32_t)a.S) ps ^= 1u;
                }
                if (ok && !STREAM) mma_commit(smem_u32(a_empty));
            }
            // all MMAs issued by this thread complete before the CTA exits
            mma_commit(smem_u32(drain));
            wait_phase(smem_u32(drain), 0u, abort_f, a.err, kWaitNs, true);
        }
    } else {
        // ---------------- epilogue
        const int ew = warp - 1 - kMmaWarps;   // 0..7
        const int group = ew >> 2;          // takes the tiles of this parity
        const int quarter = warp & 3;       // TMEM lanes this warp may read
        const int my_row = quarter * 32 + lane;
        float2 *pend = s_pend + ew * kPend * kStride;
        float *xs = s_xn + ew * TN;
        constexpr uint32_t kSlotBytes = sizeof(float2) * kStride;
        const uint32_t slot0 = smem_u32(pend + lane);   // the row's first pending slot
        volatile Key *pub = s_thr + group * TM + my_row;   // K1-th distance; the middle one 2 TM further
        volatile const Key *pub_o = s_thr + (1 - group) * TM + my_row;
        uint32_t pa = 0, b = (uint32_t)group, fb = (uint32_t)group, pf = 0;   // accumulator, barrier and its phase
        // the CTA's items are consecutive pieces of the covered-tile sequence,
        // so its tiles are one run a.tiles[g_beg, g_end) and tile n of the run
        // is accumulator use n; the index of the group's tile after next and
        // the next tile's norms are fetched into registers ahead of their use
        const int32_t g_beg = it_begin < it_end ? a.items[it_begin].off : 0;
        const int32_t g_n = it_begin < it_end ? a.items[it_end - 1].off + a.items[it_end - 1].cnt - g_beg : 0;
        int32_t n = group;
        int32_t tile_cur = n < g_n ? a.tiles[g_beg + n] : 0;
        int32_t tile_nx = n + 2 < g_n ? a.tiles[g_beg + n + 2] : 0;
        float4 xn = make_float4(0.f, 0.f, 0.f, 0.f);   // norms 4 lane .. 4 lane + 3 of the tile
        if (L2 && n < g_n) xn = __ldg((const float4 *)(a.xnorm + (int64_t)tile_cur * TN) + lane);
        bool ok = true;
        for (int it = it_begin; ok && it < it_end; ++it) {
            const WorkItem I = a.items[it];
            const int32_t n_end = I.off + I.cnt - g_beg;
            if (!STREAM && group == 0) {
                // the item's query tile into tensor memory, once the MMAs of
                // the previous item are done: each thread its row, 64 hi and
                // 64 lo BF16 (32 columns each) per chunk
                if (!wait_phase(smem_u32(a_empty), pa ^ 1u, abort_f, a.err, a.wait_ns)) {
                    ok = false;
                } else {
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    for (int h = 0; h < 2 * a.nk; ++h) {
                        const int kc = h >> 1, lo_part = h & 1;
                        const unsigned char *src = a.qs + ((int64_t)I.qtile * a.nk + kc) * STAGE + lo_part * CHUNK +
                                                   my_row * 128;
                        uint4 w[8];
#pragma unroll
                        for (int c = 0; c < 8; ++c) w[c] = __ldg((const uint4 *)(src + ((c ^ (my_row & 7)) << 4)));
                        tmem_st32(tmem_a + ((uint32_t)(quarter * 32) << 16) + (lo_part * a.nk + kc) * 32, w);
                    }
                    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(a_full));
                    pa ^= 1u;
                }
            }
            Key *out = a.part + (((int64_t)it * 2 + group) * TM + quarter * 32) * K1;
            Key *list = kSmemLists && a.list_smem ? s_list + ew * 32 * K1 : out;
            const int64_t sp = (int64_t)I.qtile * TM + my_row;
            int32_t lo = 1, hi = 0;
            float *drow = nullptr;   // a dense row's distance of point p goes to drow[p]
            if (sp < a.nv) {
                const int32_t o = a.qorder[sp];
                // a query whose norm overflows keeps no candidates
                if (!L2 || a.qnorm[o] < INFINITY) { lo = (int32_t)a.l[o]; hi = (int32_t)a.r[o]; }
                const int64_t off = a.doff[sp];
                if (off >= 0) drow = a.dense + off - (lo & ~3);
            }
            RowState st{0, 0, INFINITY, INFINITY};   // points at +inf or NaN are never kept
            constexpr int KL = KR ? KR : 1;
            float ld[KL];
            int32_t li[KL];
#pragma unroll
            for (int e = 0; e < KL; ++e) { ld[e] = INFINITY; li[e] = 0; }
            // all pending entries of the warp's rows (those worth it, with
            // lists in memory) into their lists
            auto flush = [&](int fill) {
                if constexpr (KR > 0) {
                    __syncwarp();
                    insert_pending<KL>(pend, lane, st.cnt, ld, li);
                    __syncwarp();
                    st.cnt = 0;
                    st.t = ld[KL - 1];
                    st.th = ld[(KL - 1) / 2];
                    pub[0] = ((Key)(uint32_t)it << 32) | __float_as_uint(st.t);
                    pub[2 * TM] = ((Key)(uint32_t)it << 32) | __float_as_uint(st.th);
                } else if constexpr (KR == 0) {
                    const unsigned fl = __ballot_sync(0xffffffffu, st.cnt >= fill);
                    if (fl) st = flush_rows<NL>(fl, pend, list, K1, st, pub, (uint32_t)it);
                }
            };
            for (; ok && n < n_end; n += 2) {
                const int32_t pt = tile_cur * TN;   // first point of the tile
                if (L2) {
                    ((float4 *)xs)[lane] = xn;
                    __syncwarp();
                    if (n + 2 < g_n) xn = __ldg((const float4 *)(a.xnorm + (int64_t)tile_nx * TN) + lane);
                }
                const int32_t tile_nx2 = n + 4 < g_n ? __ldg(a.tiles + g_beg + n + 4) : 0;
                if (!wait_phase(smem_u32(acc_full + fb), pf, abort_f, a.err, a.wait_ns)) {
                    ok = false;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                // the row's columns jl..jh of this tile; a warp none of whose
                // rows covers it only releases the accumulator
                const int jl = lo - pt > 0 ? lo - pt : 0;
                const int jh = hi - pt < TN - 1 ? hi - pt : TN - 1;
                const bool in = jl <= jh;
                auto release = [&]() {   // the accumulator is read
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(acc_empty + fb));
                };
                if (__any_sync(0xffffffffu, in)) {
                    const bool masked = !__all_sync(0xffffffffu, !in || jh - jl == TN - 1);
                    const Key o = pub_o[0], oh = pub_o[2 * TM];
                    const float to = (uint32_t)(o >> 32) == (uint32_t)it ? __uint_as_float((uint32_t)o) : INFINITY;
                    const float tho = (uint32_t)(oh >> 32) == (uint32_t)it ? __uint_as_float((uint32_t)oh) : INFINITY;
                    const bool lists = in && drow == nullptr;
                    const bool any_dense = __any_sync(0xffffffffu, in && drow != nullptr);
                    float thr = lists ? fminf(fminf(st.t, to), fmaxf(st.th, tho)) : -INFINITY;
                    const uint32_t ta = tmem + ((uint32_t)(quarter * 32) << 16) + b * TN;
                    uint32_t slot = slot0 + st.cnt * kSlotBytes;
#pragma unroll 1
                    for (int c0 = 0; c0 < TN; c0 += 32) {
                        float s[32];
                        // the columns' distances |x|^2 - 2 q.x (the query's own
                        // norm, the same for every point, is left out) or
                        // -q.x, +inf outside the row's range, and the least of
                        // each kCols: most blocks hold nothing for any row
                        if (L2) {
                            float4 x[8];
#pragma unroll
                            for (int c = 0; c < 8; ++c) x[c] = *(const float4 *)(xs + c0 + 4 * c);
                            tmem_ld32(ta + c0, s);
                            if (c0 == TN - 32) release();
#pragma unroll
                            for (int c = 0; c < 8; ++c) {
                                s[4 * c] = fmaf(-2.f, s[4 * c], x[c].x);
                                s[4 * c + 1] = fmaf(-2.f, s[4 * c + 1], x[c].y);
                                s[4 * c + 2] = fmaf(-2.f, s[4 * c + 2], x[c].z);
                                s[4 * c + 3] = fmaf(-2.f, s[4 * c + 3], x[c].w);
                            }
                        } else {
                            tmem_ld32(ta + c0, s);
                            if (c0 == TN - 32) release();
#pragma unroll
                            for (int c = 0; c < 32; ++c) s[c] = -s[c];
                        }
                        if (masked) {
#pragma unroll
                            for (int c = 0; c < 32; ++c)
                                s[c] = (uint32_t)(c0 + c - jl) <= (uint32_t)(jh - jl) ? s[c] : INFINITY;
                        }
                        if (any_dense) {
#pragma unroll
                            for (int c = 0; c < 32; c += 4)
                                if (in && drow != nullptr && c0 + c + 3 >= jl && c0 + c <= jh)
                                    *(float4 *)(drow + pt + c0 + c) = make_float4(s[c], s[c + 1], s[c + 2], s[c + 3]);
                        }
                        float least[32 / kCols];
#pragma unroll
                        for (int g = 0; g < 32 / kCols; ++g) {
                            const float *t8 = s + g * kCols;
                            least[g] = fminf(fminf(fminf(t8[0], t8[1]), fminf(t8[2], t8[3])),
                                             fminf(fminf(t8[4], t8[5]), fminf(t8[6], t8[7])));
                        }
                        if (!__any_sync(0xffffffffu, fminf(fminf(least[0], least[1]), fminf(least[2], least[3])) < thr))
                            continue;
#pragma unroll
                        for (int g = 0; g < 32 / kCols; ++g) {
                            if (!__any_sync(0xffffffffu, least[g] < thr)) continue;
                            // predicated, not branches: the candidates are
                            // spread over the warp's rows
#pragma unroll
                            for (int c = g * kCols; c < (g + 1) * kCols; ++c)
                                asm volatile(
                                    "{\n\t.reg .pred p;\n\tsetp.lt.f32 p, %1, %2;\n\t"
                                    "@p st.shared.v2.b32 [%0], {%3, %4};\n\t@p add.u32 %0, %0, %5;\n\t}\n"
                                    : "+r"(slot)
                                    : "f"(s[c]), "f"(thr), "r"(__float_as_uint(s[c])), "r"(pt + c0 + c),
                                      "n"(kSlotBytes)
                                    : "memory");
                            if (__any_sync(0xffffffffu, slot > slot0 + (kPend - kCols) * kSlotBytes)) {
                                st.cnt = (int)((slot - slot0) / kSlotBytes);
                                flush(kFill);
                                slot = slot0 + st.cnt * kSlotBytes;
                                thr = lists ? fminf(fminf(st.t, to), fmaxf(st.th, tho)) : -INFINITY;
                            }
                        }
                    }
                    st.cnt = (int)((slot - slot0) / kSlotBytes);
                }
                else release();
                if ((b += 2) >= n_acc) b -= n_acc;
                if ((fb += 2) >= n_bar) { fb -= n_bar; pf ^= 1u; }
                tile_cur = tile_nx;
                tile_nx = tile_nx2;
            }
            if (!ok) {   // an aborted wait: no lists (the host reports the error)
                for (; it < it_end; ++it) a.part_n[((int64_t)it * 2 + group) * TM + my_row] = 0;
                break;
            }
            __syncwarp();
            flush(1);
            if (KR) {
#pragma unroll
                for (int e = 0; e < KL; ++e) {
                    if (ld[e] < INFINITY) {
                        out[(size_t)lane * KL + e] = make_key(ld[e], (uint32_t)li[e]);
                        st.len = e + 1;
                    }
                }
            } else if (kSmemLists && a.list_smem) {
                for (int r = 0; r < 32; ++r) {
                    const int m = __shfl_sync(0xffffffffu, st.len, r);
#pragma unroll
                    for (int h = 0; h < NL; ++h)
                        if (lane + 32 * h < m) out[(size_t)r * K1 + lane + 32 * h] = list[r * K1 + lane + 32 * h];
                }
                __syncwarp();
            }
            a.part_n[((int64_t)it * 2 + group) * TM + my_row] = st.len;
        }
    }
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(kTmem) : "memory");
    }
}

// FP32 rows -> BF16 hi and lo parts in the tiled, swizzled block layout, and
// the rows' squared norms (and norms, and their maximum), in one pass. LR
// lanes share a row: lane `sub` takes its 8-dimension groups sub, sub + LR,
// ..., two 16-byte loads each, stores both 16-byte parts and adds up the
// squares, which are summed over the LR lanes by shuffles. Row `i` of the
// output is input row order[i] (or i), rows past `rows` are zero; norms are
// written at the input row, and nothing for padding rows.
// Memory bound: 4 d bytes read and 4 * 64 nk written per row. LR is the largest
// power of two up to 32 that divides the row's 8 nk groups, so that no lane is
// idle and a warp's loads are whole 128-byte lines. Norms apart (one thread
// per row, uncoalesced) took 418 us at 1M x 128 and 576 us at 200,003 x 768,
// beside 143 and 172 us for the split; one pass takes 153 us (6.7 TB/s) and 172 us.
template <int LR>
__global__ void __launch_bounds__(256) split_norm_kernel(const float *__restrict__ X, int64_t rows, int d, int nk,
                                                         const int32_t *__restrict__ order, int64_t rows_pad,
                                                         unsigned char *__restrict__ out, float *norm,
                                                         float *rownorm, float *max_rownorm) {
    const int sub = threadIdx.x % LR;
    const int64_t row = blockIdx.x * (int64_t)(256 / LR) + threadIdx.x / LR;
    const int64_t src = row < rows ? (order ? (int64_t)order[row] : row) : -1;
    const int64_t tile = row >> 7;
    const int t = (int)(row & 127);
    float s = 0.f;
    if (row < rows_pad) {
        for (int g = sub; g < nk * 8; g += LR) {
            const int k = g * 8;
            float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
            if (src >= 0 && k < d) {   // d % 4 == 0 and 16-byte aligned rows
                const float4 *x4 = reinterpret_cast<const float4 *>(X + src * d + k);
                a = __ldg(x4);
                if (k + 4 < d) b = __ldg(x4 + 1);
            }
            const float v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
            __align__(16) __nv_bfloat16 h[8];
            __align__(16) __nv_bfloat16 lo[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                h[e] = __float2bfloat16_rn(v[e]);
                lo[e] = __float2bfloat16_rn(v[e] - __bfloat162float(h[e]));
                s = fmaf(v[e], v[e], s);
            }
            unsigned char *blk = out + (tile * nk + (g >> 3)) * (int64_t)STAGE;
            const uint32_t off = t * 128 + (((g & 7) ^ (t & 7)) << 4);
            *(uint4 *)(blk + off) = *(const uint4 *)h;
            *(uint4 *)(blk + CHUNK + off) = *(const uint4 *)lo;
        }
    }
#pragma unroll
    for (int o = LR >> 1; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    const float rn = sqrtf(s);
    if (sub == 0 && src >= 0) {
        norm[src] = s;
        if (rownorm) rownorm[src] = rn;
    }
    if (max_rownorm) {
        float m = fmaxf(src >= 0 ? rn : 0.f, 0.f);   // a NaN row does not count
#pragma unroll
        for (int o = 16; o >= LR && o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        __shared__ float wm[8];
        if ((threadIdx.x & 31) == 0) wm[threadIdx.x >> 5] = m;
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int w = 1; w < 8; ++w) m = fmaxf(m, wm[w]);
            atomicMax((int *)max_rownorm, __float_as_int(m));   // m >= 0
        }
    }
}

// Launches split_norm_kernel with the lanes per row of nk 64-wide chunks.
cudaError_t split_norm(const float *X, int64_t rows, int d, int nk, const int32_t *order, int64_t rows_pad,
                       unsigned char *out, float *norm, float *rownorm, float *max_rownorm, cudaStream_t stream) {
    const int lr = nk % 4 == 0 ? 32 : (nk % 2 == 0 ? 16 : 8);
    const int grid = ceil_div_i(rows_pad, 256 / lr);
    if (lr == 32)
        split_norm_kernel<32><<<grid, 256, 0, stream>>>(X, rows, d, nk, order, rows_pad, out, norm, rownorm, max_rownorm);
    else if (lr == 16)
        split_norm_kernel<16><<<grid, 256, 0, stream>>>(X, rows, d, nk, order, rows_pad, out, norm, rownorm, max_rownorm);
    else
        split_norm_kernel<8><<<grid, 256, 0, stream>>>(X, rows, d, nk, order, rows_pad, out, norm, rownorm, max_rownorm);
    return cudaGetLastError();
}

struct FinishArgs {
    const float *X, *Q;
    int d, metric, k, K1;
    const Key *part;
    const int32_t *part_n, *item_begin, *qorder;
    const int64_t *doff, *l, *r;
    const float *dense;
    const float *qnorm, *qrownorm, *xmax;
    int serial;                     // 1: exact distances summed in dimension order
    int64_t *out_ids;
    float *out_dist;
    int32_t *out_count, *redo;
};

// One valid query per block of WQ warps, at its sorted position: its lists
// (two per work item of its query tile) merged into the K1 best approximate
// distances, each warp every WQ-th list, then the warps' results pairwise;
// the candidates' exact FP32 distances, four per warp at a time; sort,
// certificate and output by warp 0. All keys stay in registers (32 NL per
// list). A block per query because the lists and the candidates' rows are
// dependent gathers: a warp per query took the 304 lists of a 61-query call in
// series (208 us) and one candidate row after the other (40 us). WQ: 4, or 16
// when the queries' lists are many (few queries over many CTAs).
// Together 57 us for 10k queries of lists, 300 us with 0.9 GB of dense rows.
template <int NL, int WQ>
__global__ void __launch_bounds__(32 * WQ) finish_kernel(FinishArgs f) {
    __shared__ Key s_keys[WQ][32 * NL];
    __shared__ int s_na[WQ];
    __shared__ Key s_buf[WQ][32 + 256];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t sp = blockIdx.x;
    const int64_t qt = sp / TM;
    const int row = (int)(sp % TM);
    const int64_t q = f.qorder[sp];
    const int l0 = f.item_begin[qt] * 2, l1 = f.item_begin[qt + 1] * 2;
    Key A[NL];
#pragma unroll
    for (int h = 0; h < NL; ++h) A[h] = kPad;
    int na = 0;
    const int64_t off = f.doff[sp];
    if (off >= 0) {
        // a dense row: each warp takes every WQ-th 128 distances; those below
        // its K1-th so far are collected, and sorted and merged by 32
        const int32_t lo = (int32_t)f.l[q], hi = (int32_t)f.r[q];
        const float4 *row = (const float4 *)(f.dense + off);
        const bool dead = f.metric == ESG_L2SQ && !(f.qnorm[q] < INFINITY);
        Key *buf = s_buf[warp];
        int nb = 0;
        float t = INFINITY;
        auto merge32 = [&](int c) {
            Key p[NL];
#pragma unroll
            for (int h = 0; h < NL; ++h) p[h] = kPad;
            if (lane < c) p[0] = buf[lane];
            Key one[1] = {p[0]};
            sort_asc<1>(one, lane);
            p[0] = one[0];
            merge_lists<NL>(A, p, lane);
            na = min(f.K1, na + c);
            Key k = kPad;
#pragma unroll
            for (int h = 0; h < NL; ++h)
                if (h == (f.K1 - 1) >> 5) k = A[h];
            k = __shfl_sync(0xffffffffu, k, (f.K1 - 1) & 31);
            if (na == f.K1) t = key_dist(k);
        };
        const int32_t p0 = lo & ~3;
        const float4 none = make_float4(INFINITY, INFINITY, INFINITY, INFINITY);
        for (int32_t c0 = dead ? hi + 1 : p0 + 256 * warp; c0 <= hi; c0 += 256 * WQ) {
            const int32_t pt = c0 + 4 * lane;
            const float4 xa = pt <= hi ? row[(pt - p0) >> 2] : none;
            const float4 xb = pt + 128 <= hi ? row[(pt + 128 - p0) >> 2] : none;
            const float x[8] = {xa.x, xa.y, xa.z, xa.w, xb.x, xb.y, xb.z, xb.w};
            const float least = fminf(fminf(fminf(x[0], x[1]), fminf(x[2], x[3])),
                                      fminf(fminf(x[4], x[5]), fminf(x[6], x[7])));
            if (!__any_sync(0xffffffffu, least < t)) continue;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int32_t p = pt + (e < 4 ? e : 124 + e);
                const bool take = x[e] < t && p >= lo && p <= hi;
                const unsigned b = __ballot_sync(0xffffffffu, take);
                if (b == 0u) continue;
                if (take) buf[nb + __popc(b & ((1u << lane) - 1))] = make_key(x[e], (uint32_t)p);
                nb += __popc(b);
            }
            __syncwarp();
            while (nb >= 32) {
                merge32(32);
                __syncwarp();
                nb -= 32;   // the last 32 in the place of those merged
                const int mv = min(nb, 32);
                if (lane < mv) buf[lane] = buf[32 + nb - mv + lane];
                __syncwarp();
            }
        }
        if (nb > 0) merge32(nb);
    } else for (int li = l0 + warp; li < l1; li += WQ) {
        const int64_t sub = (int64_t)li * TM + row;
        const int nb = f.part_n[sub];
        Key B[NL];
#pragma unroll
        for (int h = 0; h < NL; ++h) {
            const int e = lane + 32 * h;
            B[h] = e < f.K1 ? f.part[sub * f.K1 + e] : kPad;   // entries past nb are not written: dropped below
            if (e >= nb) B[h] = kPad;
        }
        if (nb == 0) continue;
        merge_lists<NL>(A, B, lane);
        na = min(f.K1, na + nb);
    }
#pragma unroll
    for (int w = WQ / 2; w > 0; w >>= 1) {   // warps w .. 2w - 1 hand their lists to warps 0 .. w - 1
        if (warp >= w && warp < 2 * w) {
#pragma unroll
            for (int h = 0; h < NL; ++h) s_keys[warp][lane + 32 * h] = A[h];
            if (lane == 0) s_na[warp] = na;
        }
        __syncthreads();
        if (warp < w && s_na[warp + w] > 0) {
#pragma unroll
            for (int h = 0; h < NL; ++h)
                A[h] = key_min(A[h], s_keys[warp + w][32 * NL - 1 - (lane + 32 * h)]);
            bitonic_asc<NL>(A, lane);
            na = min(f.K1, na + s_na[warp + w]);
        }
    }
    Key kth = kPad;   // the K1-th approximate distance (warp 0)
    if (warp == 0) {
#pragma unroll
        for (int h = 0; h < NL; ++h) {
            s_keys[0][lane + 32 * h] = A[h];
            if (h == (f.K1 - 1) >> 5) kth = A[h];
        }
        kth = __shfl_sync(0xffffffffu, kth, (f.K1 - 1) & 31);
        if (lane == 0) s_na[0] = na;
    }
    __syncthreads();
    const int m = s_na[0];
    const float *qq = f.Q + q * (int64_t)f.d;
    if (f.serial) {
        // one candidate per thread, its terms added in dimension order: what
        // the SIMT kernel computes, so that answers with these lists do not
        // depend on which of the two a query went through
        for (int e = threadIdx.x; e < m; e += 32 * WQ) {
            const uint32_t id = (uint32_t)s_keys[0][e];
            const float4 *x4 = (const float4 *)(f.X + (int64_t)id * f.d), *q4 = (const float4 *)qq;
            float acc = 0.f;
#pragma unroll 4
            for (int j = 0; j < f.d / 4; ++j) {
                const float4 x = __ldg(x4 + j), qv = __ldg(q4 + j);
                if (f.metric == ESG_L2SQ) {
                    const float t0 = qv.x - x.x, t1 = qv.y - x.y, t2 = qv.z - x.z, t3 = qv.w - x.w;
                    acc = fmaf(t0, t0, acc); acc = fmaf(t1, t1, acc); acc = fmaf(t2, t2, acc); acc = fmaf(t3, t3, acc);
                } else {
                    acc = fmaf(qv.x, x.x, acc); acc = fmaf(qv.y, x.y, acc);
                    acc = fmaf(qv.z, x.z, acc); acc = fmaf(qv.w, x.w, acc);
                }
            }
            s_keys[1][e] = exact_key(f.metric == ESG_L2SQ ? acc : -acc, id);
        }
    } else
    // exact distances: lane j of a warp sums the dimensions j, j + 32, ...,
    // the lanes' sums by a shuffle tree
    for (int e0 = warp * 4; e0 < m; e0 += 4 * WQ) {
        const float *x[4];
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
        uint32_t id[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            id[c] = (uint32_t)s_keys[0][min(e0 + c, m - 1)];
            x[c] = f.X + (int64_t)id[c] * f.d;
        }
        if (f.metric == ESG_L2SQ) {
#pragma unroll 4
            for (int j = lane; j < f.d; j += 32) {
                const float qv = qq[j];
#pragma unroll
                for (int c = 0; c < 4; ++c) { const float t = qv - x[c][j]; acc[c] = fmaf(t, t, acc[c]); }
            }
        } else {
#pragma unroll 4
            for (int j = lane; j < f.d; j += 32) {
                const float qv = qq[j];
#pragma unroll
                for (int c = 0; c < 4; ++c) acc[c] = fmaf(qv, x[c][j], acc[c]);
            }
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            acc[c] = warp_sum_group(acc[c], 32);
            if (lane == 0 && e0 + c < m)
                s_keys[1][e0 + c] = exact_key(f.metric == ESG_L2SQ ? acc[c] : -acc[c], id[c]);
        }
    }
    __syncthreads();
    if (warp != 0) return;
    Key R[NL];
#pragma unroll
    for (int h = 0; h < NL; ++h) R[h] = lane + 32 * h < m ? s_keys[1][lane + 32 * h] : kPad;
    sort_asc<NL>(R, lane);
    const int c = min(f.k, m);
    Key last = kPad;
#pragma unroll
    for (int h = 0; h < NL; ++h)
        if (h == (max(c, 1) - 1) >> 5) last = R[h];
    last = __shfl_sync(0xffffffffu, last, (max(c, 1) - 1) & 31);
    // a list shorter than its range has dropped points at +inf or NaN: theirs are
    // the exact distances too, unless a norm overflows or an element has no BF16
    // part (then its row's norm overflows): those queries go to the SIMT kernel
    bool certified = c > 0 && (m > f.r[q] - f.l[q] || (f.qrownorm[q] < INFINITY && f.xmax[0] < INFINITY));
    if (m == f.K1) {   // the list is full: points may have been left out
        // |approximate - exact| for any point of the range (unit roundoff of
        // BF16 2^-8, of FP32 2^-24): the split residuals and the dropped
        // lo*lo product stay below 3.1 * 2^-16 |q_i||x_i| per term, the FP32
        // accumulation of 3d products below 6d * 2^-24 (twice the rounding
        // bound, for truncating adders); the squared distance doubles the dot
        // product error and adds the rounding of the norms and the final sum.
        const double qn = f.qrownorm[q], xm = f.xmax[0];
        const double dot_err = (3.1 * 0x1p-16 + 6.0 * f.d * 0x1p-24) * qn * xm;
        const bool l2 = f.metric == ESG_L2SQ;
        const double delta = l2 ? 2.0 * dot_err + (f.d + 4.0) * 0x1p-24 * (qn * qn + xm * xm) : dot_err;
        // list distances leave out the query's squared norm
        const double bound = (double)key_dist(kth) + (l2 ? (double)f.qnorm[q] : 0.0) - delta;
        // the re-ranked FP32 distance itself is within d * 2^-23 relative
        const double dk = (double)key_dist(last);
        certified = dk + fabs(dk) * f.d * 0x1p-23 < bound;
    }
    // the largest product of norms whose BF16 parts' products cannot overflow
    // (each part is up to 2^-8 above its element): beyond it an inner product
    // that FP32 holds may have been dropped as infinite
    if (f.metric == ESG_IP && !((double)f.qrownorm[q] * f.xmax[0] < 0x1.fcp127)) certified = false;
    const float zero = f.metric == ESG_L2SQ ? 0.f : -0.f;   // a negated product of 0 is -0
#pragma unroll
    for (int h = 0; h < NL; ++h) {
        const int e = lane + 32 * h;
        if (e < f.k) {
            f.out_ids[q * f.k + e] = e < c ? (int64_t)(uint32_t)R[h] : -1;
            const float x = key_dist(R[h]);
            f.out_dist[q * f.k + e] = e < c ? (x == 0.f ? zero : x) : INFINITY;
        }
    }
    if (lane == 0) { f.out_count[q] = c; f.redo[q] = certified ? 0 : 1; }
}

// Queries with an invalid range (in no query tile): no results.
__global__ void invalid_kernel(const int64_t *l, const int64_t *r, int64_t nq, int64_t n, int k, int64_t *out_ids,
                               float *out_dist, int32_t *out_count, int32_t *redo) {
    const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (q >= nq || (l[q] >= 0 && l[q] <= r[q] && r[q] < n)) return;
    for (int j = 0; j < k; ++j) { out_ids[q * k + j] = -1; out_dist[q * k + j] = INFINITY; }
    out_count[q] = 0;
    redo[q] = 0;
}

}  // namespace

// Device scratch of a call, given back on its stream whichever way the call
// ends (a host allocation may throw with scratch held and work queued).
struct Scratch {
    unsigned char *p = nullptr;
    cudaStream_t stream;
    explicit Scratch(cudaStream_t s) : stream(s) {}
    Scratch(const Scratch &) = delete;
    Scratch &operator=(const Scratch &) = delete;
    ~Scratch() { release(); }
    cudaError_t alloc(size_t bytes) { return esg_malloc_async((void **)&p, bytes, stream); }
    void release() {
        if (p) cudaFreeAsync(p, stream);
        p = nullptr;
    }
};

// Waits for the pass and returns the queries it left uncertified.
static esg_status read_uncertified(int64_t nq, int K1, const int32_t *redo, const int32_t *err, cudaStream_t stream,
                                   std::vector<int64_t> &idx) {
    esg_fault_host();
    std::vector<int32_t> h_redo(nq);
    int32_t h_err = 0;
    cudaError_t ce = cudaMemcpyAsync(h_redo.data(), redo, sizeof(int32_t) * nq, cudaMemcpyDeviceToHost, stream);
    if (ce == cudaSuccess) ce = cudaMemcpyAsync(&h_err, err, sizeof(int32_t), cudaMemcpyDeviceToHost, stream);
    if (ce == cudaSuccess) ce = cudaStreamSynchronize(stream);
    if (ce != cudaSuccess) { esg_set_error(cudaGetErrorString(ce)); return ESG_ERR_CUDA; }
    if (h_err) { esg_set_error("tensor-core brute force: an mbarrier wait timed out"); return ESG_ERR_TIMEOUT; }
    idx.clear();
    for (int64_t i = 0; i < nq; ++i) if (h_redo[i]) idx.push_back(i);
    const char *dbg = getenv("ESG_BF_STATS");
    if (dbg && *dbg == '1')
        fprintf(stderr, "tensor-core brute force: %lld of %lld queries left uncertified (list of %d)\n",
                (long long)idx.size(), (long long)nq, K1);
    return ESG_OK;
}

// Whether answers for k are summed in dimension order, like the SIMT kernel's
// (which alone served lists longer than 64, or 58 past 64 dimensions), or over
// the lanes: a call's rounding stays what it was.
static bool bf2_serial(int32_t d, int k) { return k + 8 > ((d + TK - 1) / TK == 1 ? 64 : 58); }

// List length for k: k + 12 candidates (the register lists' 24 or 32 for k up to
// 20), at least k + 8 (the longest list the kernel holds caps it). At 1M x 128,
// 10k queries, k = 10, lists of k + 8 left 2 queries uncertified, k + 12 certified all.
static int bf2_list(int k) { return k <= 12 ? 24 : (k <= 20 ? 32 : std::min(k + 12, kMaxK1v2)); }

// Where both paths give the same answers (bf2_serial), the one that takes less
// time by these estimates serves the call: a few narrow ranges are a few point
// tiles of the SIMT kernel, while the tensor-core path prepares all points and
// makes a host plan first. In us, fitted to 682 pairs of timed calls (1 to 4,096
// queries, 1,000 to 10M points, 32 to 768 dimensions, ranges of 100 points to all,
// k = 60 and 100): of those where the two are over 15 % apart, all take the faster.
// One query over 1,000 of 1M x 96 points, k = 100: 281 us on the tensor cores, 232
// us in the SIMT kernel with the look at the ranges; over 1,000 of 10M x 96: 1,552
// and 232; over 10,000 of 1M x 96: 297 and 1,550; 4,096 over all of 1,000 x 256:
// 2,529 and 840.
// The SIMT kernel: a CTA per 64 queries, two of them on an SM, takes the 64-point
// tiles one of its queries covers, passes over the others between them, and a
// warp folds a tile into its eight queries' lists one after the other.
constexpr double kLook = 22.0;   // reading the ranges first
struct SimtCost {
    double tile, fold;
    int64_t slots;
    SimtCost(int32_t d, int k, int64_t sms) : tile(3.0 + 0.06 * d), fold(1.3 + 0.02 * k), slots(2 * sms) {}
    // a CTA whose queries lie in a hull of `hull` tiles and cover `sum` of them,
    // `fold_tiles` the eight of one warp (at most)
    double cta(int64_t hull, int64_t sum, int64_t fold_tiles) const {
        return 0.18 * hull + tile * std::min(sum, hull) + fold * fold_tiles;
    }
};

// All queries over all points: what any ranges take at most.
static double simt_us_at_most(int64_t n, int64_t nq, int32_t d, int k, int64_t sms) {
    const SimtCost c(d, k, sms);
    const int64_t t = (n + 63) / 64, ctas = (nq + 63) / 64;
    return 30.0 + c.cta(t, t, t * std::min<int64_t>(nq, 8)) * std::max(1.0, (double)ctas / c.slots);
}

static double simt_us(const std::vector<int64_t> &l, const std::vector<int64_t> &r, int64_t n, int32_t d, int k,
                      int64_t sms) {
    const SimtCost c(d, k, sms);
    const int64_t nq = (int64_t)l.size();
    double most = 0.0, all = 0.0;
    for (int64_t q0 = 0; q0 < nq; q0 += 64) {
        int64_t lo = n, hi = -1, sum = 0, fold = 0;
        for (int64_t w = q0; w < std::min(nq, q0 + 64); w += 8) {
            int64_t warp = 0;
            for (int64_t q = w; q < std::min(nq, w + 8); ++q) {
                if (l[q] < 0 || l[q] > r[q] || r[q] >= n) continue;
                lo = std::min(lo, l[q]);
                hi = std::max(hi, r[q]);
                warp += (r[q] - l[q]) / 64 + 1;
            }
            sum += warp;
            fold = std::max(fold, warp);
        }
        if (hi < 0) continue;
        const double t = c.cta((hi - lo) / 64 + 1, sum, fold);
        most = std::max(most, t);
        all += t;
    }
    return 30.0 + std::max(most, all / c.slots);
}

// The tensor-core path: launches, host round trips and the plan; the points'
// preparation (memory bound); and, past 128 dimensions, where narrow ranges keep
// lists too, the insertions while these fill: a warp's rows, as far as their ranges
// (`mean` points wide) lie in the item's tiles, one after the other. Wide ranges
// take more than this, and the SIMT kernel much more.
static double tc_us(int64_t n, int64_t nq, int64_t mean, int32_t d, int k, int64_t sms) {
    const int64_t nk = (d + TK - 1) / TK;
    double t = 140.0 + 0.05 * d + n * (4.0 * d + (double)STAGE / TM * nk) / 6.6e6;
    if (nk > 2 && mean > 0) {
        const double qt = std::ceil(nq / (double)TM), tiles = std::ceil(n / (double)TN);
        const double ctas = std::min<double>(sms, qt * tiles), items = std::max(1.0, ctas / qt);
        const double m = std::min<double>(n / items, mean) / 2, K1 = k + 12;   // points a list sees
        const double ins = m <= K1 ? m : K1 * (1.0 + std::log(m / K1));
        const double share = std::min(1.0, (mean + TN) / (n * std::min(1.0, TM / (double)nq) + mean));
        t += 0.25 * (1.0 + (nk - 4) / 16.0) * ins * std::ceil(std::min<double>(nq, TM) / 4) *
             std::max(1.0, qt * items / ctas) * share;
    }
    return t;
}

// Length of the register lists that serve lists of K1, 0 if they are too long.
static int bf2_reg_list(int K1) { return K1 == 24 || K1 == 32 ? K1 : 0; }

// Launch plan of the pipelined kernel: query tile in tensor memory (d <= 256),
// with as many accumulators as fit beside it, or streamed with the point
// chunks; stages that fit shared memory. ESG_ERR_UNSUPPORTED when not even two
// stages fit.
static esg_status bf2_smem(int32_t d, int K1, int max_smem, int *S, size_t *smem, int *n_acc, bool *stream_a,
                           bool *list_smem) {
    if (K1 > kMaxK1v2 || d < 1) return ESG_ERR_UNSUPPORTED;
    const int nk = (d + TK - 1) / TK;
    *stream_a = nk > kMaxResident;
    *n_acc = *stream_a ? 4 : std::min(3, (kTmem - 64 * nk) / TN);
    const size_t stage = *stream_a ? 2 * (size_t)STAGE : (size_t)STAGE;
    // pending slots, tile norms, published distances, mbarriers
    const bool reg = bf2_reg_list(K1) > 0;
    const int pend = reg ? 16 : (*stream_a ? Epi<true>::kPend : Epi<false>::kPend);
    size_t common = sizeof(float2) * kEpiWarps * pend * (reg ? 32 : kPendStride) + sizeof(float) * kEpiWarps * TN +
                    sizeof(Key) * 4 * TM + 8 * (2 * kMaxStages + 16) + 16;
    if ((size_t)max_smem < common + 2 * stage) return ESG_ERR_UNSUPPORTED;
    // the lists in shared memory where they leave four stages (a list in global
    // memory is a trip to the L2, busy with operand blocks, per merge). With 227
    // KB none of K1 > 32 do: 33 at d <= 256 need 249 KB. The kernel of lists up to
    // 64 keeps the choice because without it the compiler's code for it is slower
    // (398 queries over 219,744 x 256, k = 50: 676 -> 688 us a call); that of longer
    // lists is faster (10k over 1M x 96, k = 100: 9.29 -> 8.60 ms).
    const size_t lists = sizeof(Key) * 2 * TM * K1;
    *list_smem = !reg && K1 <= 64 && (size_t)max_smem >= common + lists + 4 * stage;
    if (*list_smem) common += lists;
    *S = (int)std::min<size_t>(kMaxStages, ((size_t)max_smem - common) / stage);
    *smem = common + (size_t)*S * stage;
    return ESG_OK;
}

// The point side, prepared once per call: tiled BF16 splits, squared norms
// and the largest row norm.
struct PreparedX {
    const unsigned char *xs;
    const float *xnorm, *xmax;
};

__global__ void gather_subset_kernel(const float *Q, const int64_t *l, const int64_t *r, int d,
                                     const int64_t *idx, int64_t m, float *Qg, int64_t *lg, int64_t *rg) {
    const int64_t i = blockIdx.x;
    if (i >= m) return;
    const int64_t q = idx[i];
    for (int j = threadIdx.x; j < d; j += blockDim.x) Qg[i * d + j] = Q[q * d + j];
    if (threadIdx.x == 0) { lg[i] = l[q]; rg[i] = r[q]; }
}

__global__ void scatter_subset_kernel(const int64_t *idx, int64_t m, int k, const int64_t *ids_g,
                                      const float *dist_g, const int32_t *cnt_g, int64_t *ids, float *dist,
                                      int32_t *cnt) {
    const int64_t i = blockIdx.x;
    if (i >= m) return;
    const int64_t q = idx[i];
    for (int j = threadIdx.x; j < k; j += blockDim.x) {
        ids[q * k + j] = ids_g[i * k + j];
        dist[q * k + j] = dist_g[i * k + j];
    }
    if (threadIdx.x == 0) cnt[q] = cnt_g[i];
}

// Host clock (ms) for the ESG_BF_STATS=1 phase report.
static double bf_host_ms() {
    return std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now().time_since_epoch()).count();
}
static bool bf_stats() {
    const char *dbg = getenv("ESG_BF_STATS");
    return dbg && *dbg == '1';
}

struct Bf2Plan;
static esg_status bf2_queries(const PreparedX &X, const float *base, int64_t n, int32_t d, int metric,
                              const float *queries, int64_t nq, const int64_t *l, const int64_t *r, int32_t k,
                              int K1, int64_t *out_ids, float *out_dist, int32_t *out_count, cudaStream_t stream,
                              Bf2Plan *given = nullptr, bool dense_rows = true);

// Queries whose list of K1 candidates could not be certified run again with
// the longest list that fits the kernel (their own plan, a few query tiles), and
// through the exact SIMT kernel if they are still uncertified.
static esg_status bf2_escalate(const PreparedX &X, const float *base, int64_t n, int32_t d, int metric,
                               const float *queries, int64_t nq, const int64_t *l, const int64_t *r, int32_t k,
                               int K1, const std::vector<int64_t> &idx, int64_t *out_ids, float *out_dist,
                               int32_t *out_count, cudaStream_t stream) {
    const int K2 = bf2_serial(d, k) ? kMaxK1v2 : ((d + TK - 1) / TK == 1 ? 64 : 58);
    if (K2 <= K1)
        return esg_bruteforce_redo(base, n, d, metric, queries, nq, l, r, k, idx, out_ids, out_dist, out_count, stream);
    const int64_t m = (int64_t)idx.size();
    auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
    const size_t bytes = al(sizeof(int64_t) * m) + al(sizeof(float) * m * d) + 2 * al(sizeof(int64_t) * m) +
                         al(sizeof(int64_t) * m * k) + al(sizeof(float) * m * k) + al(sizeof(int32_t) * m);
    Scratch sc(stream);
    ESG_CUDA_TRY(sc.alloc(bytes));
    unsigned char *p = sc.p;
    int64_t *didx = (int64_t *)p; p += al(sizeof(int64_t) * m);
    float *Qg = (float *)p; p += al(sizeof(float) * m * d);
    int64_t *lg = (int64_t *)p; p += al(sizeof(int64_t) * m);
    int64_t *rg = (int64_t *)p; p += al(sizeof(int64_t) * m);
    int64_t *ig = (int64_t *)p; p += al(sizeof(int64_t) * m * k);
    float *dg = (float *)p; p += al(sizeof(float) * m * k);
    int32_t *cg = (int32_t *)p;
    esg_status st = ESG_OK;
    cudaError_t ce = cudaMemcpyAsync(didx, idx.data(), sizeof(int64_t) * m, cudaMemcpyHostToDevice, stream);
    if (ce == cudaSuccess) {
        gather_subset_kernel<<<(unsigned)m, 128, 0, stream>>>(queries, l, r, d, didx, m, Qg, lg, rg);
        ce = cudaGetLastError();
    }
    if (ce != cudaSuccess) { esg_set_error(cudaGetErrorString(ce)); st = ESG_ERR_CUDA; }
    if (st == ESG_OK) st = bf2_queries(X, base, n, d, metric, Qg, m, lg, rg, k, K2, ig, dg, cg, stream);
    if (st == ESG_OK) {
        scatter_subset_kernel<<<(unsigned)m, 128, 0, stream>>>(didx, m, k, ig, dg, cg, out_ids, out_dist, out_count);
        ce = cudaGetLastError();
        if (ce != cudaSuccess) { esg_set_error(cudaGetErrorString(ce)); st = ESG_ERR_CUDA; }
    }
    // the host index vector must outlive the copy above
    const cudaError_t se = cudaStreamSynchronize(stream);
    if (st == ESG_OK && se != cudaSuccess) { esg_set_error(cudaGetErrorString(se)); st = ESG_ERR_CUDA; }
    return st;
}

// Cuts the sequence of covered point tiles (query tile by query tile) into G
// contiguous shares of about equal estimated cost. A share's cost is its
// number of tiles plus, for every row with a list, a weight for starting it: a
// list that starts empty takes many insertions while it fills, and a row
// insertion costs the same whether one row of the warp or all 32 insert. Rows
// that start with the item (their ranges begin before it) fill their lists
// together and share that cost, rows whose ranges begin inside it hardly do;
// a dense row costs a little for each of its tiles (its stores). The shares
// are chosen greedily: each CTA takes about the remaining cost over the
// remaining CTAs; a second pass, where the shares are uneven (always in the
// inspected plan of plain lists), adds the restart cost of
// the previous pass's later cuts to the remaining cost, and the pass with the
// smallest largest share is kept. `lt`/`rt` are the first and last covered
// tile of each sorted query; `cut` receives G + 1 positions.
constexpr double kRestart2 = 6.25;   // one list start, in tiles, at two K chunks
// Greedy passes (the first without restart look-ahead), and the excess of the
// largest share over the mean from which the second one pays, as a part of the
// mean and in tiles at two K chunks: it takes the host 25 to 100 us, a tile takes
// a CTA about 1.1 us. Without it the largest share is 10 % above the mean at 1M x
// 128, 10k queries and k = 10, where a call takes 2.79 ms without it and 2.84 with
// it, but 43 % at k = 100, and 2.5 times the mean with 1,000 queries: 11.0 ms with
// it and 15.6 without (3,000 queries over all of 1M x 96, k = 100), 0.91 and 1.08
// ms (1,000 over 600,000 of 1M x 128, k = 10).
constexpr int kSharePasses = 2;
constexpr double kShareUneven = 0.15, kShareSlack = 32.0;

// In tiles: a row whose range begins inside the item, one that begins before
// it (its list starts with the item, along with the other rows' lists), and a
// tile of a dense row.
struct ShareCost {
    double begin, restart, dense;
};

// The covered tiles of the query tiles as spans [a, b] of consecutive tiles.
struct Spans {
    std::vector<int32_t> a, b, first;   // first: [nqt + 1] first span of each query tile
    std::vector<int64_t> at;            // position of each span's first tile in the sequence
    int32_t tile(int64_t qt, int64_t pos) const {
        int32_t i = first[qt + 1] - 1;
        while (at[i] > pos) --i;
        return a[i] + (int32_t)(pos - at[i]);
    }
};

static void bf2_shares(const Spans &sp, const std::vector<int64_t> &qt_first, const std::vector<int32_t> &lt,
                       const std::vector<int32_t> &rt, const std::vector<int32_t> &dense, int64_t G,
                       const ShareCost &w, double uneven, double slack, std::vector<int64_t> &cut) {
    const int64_t nqt = (int64_t)qt_first.size() - 1, T = qt_first[nqt];
    const int64_t nv = (int64_t)lt.size();
    cut.assign(G + 1, T);
    cut[0] = 0;
    if (G <= 1 || nqt <= 0) return;
    // estimated cost of tiles [t0, t1) of query tile qt, run as one item
    auto cost = [&](int64_t qt, int64_t t0, int64_t t1) -> double {
        if (t1 <= t0) return 0.0;
        const int32_t a = sp.tile(qt, t0), b = sp.tile(qt, t1 - 1);
        const int32_t *lq = lt.data() + qt * TM, *rq = rt.data() + qt * TM, *dq = dense.data() + qt * TM;
        const int ns = (int)(std::min(nv, (qt + 1) * TM) - qt * TM);
        int32_t begin = 0, over = 0, dtiles = 0;
        for (int s = 0; s < ns; ++s) {   // no branches: it vectorises
            const int32_t l = std::max(lq[s], a), r = std::min(rq[s], b);
            const int32_t in = l <= r ? 1 : 0;
            dtiles += dq[s] & ((r - l + 1) * in);
            over += ~dq[s] & in;
            begin += ~dq[s] & in & (lq[s] > a ? 1 : 0);
        }
        return (double)(t1 - t0) + w.restart * (over - begin) + w.begin * begin + w.dense * dtiles;
    };
    std::vector<double> pre(nqt + 1, 0.0);   // prefix sums of whole query tiles
    for (int64_t qt = 0; qt < nqt; ++qt) pre[qt + 1] = pre[qt] + cost(qt, qt_first[qt], qt_first[qt + 1]);
    // about the largest e in [lo, hi] with f(e) = cost(qt, t0, e) <= budget,
    // given f(lo) = flo <= budget < f(hi) = fhi: interpolation steps
    // alternating with bisection, stopping within 1 % of the budget; f(e) in *fe
    auto last_within = [&](int64_t qt, int64_t t0, int64_t lo, int64_t hi, double flo, double fhi, double budget,
                           double *fe) {
        for (int step = 0; hi - lo > 1 && fhi - flo > 1e-2 * budget; ++step) {
            int64_t mid = lo + (hi - lo) / 2;
            if (step % 2 == 0) mid = lo + (int64_t)((budget - flo) / (fhi - flo) * (double)(hi - lo));
            mid = std::min(std::max(mid, lo + 1), hi - 1);
            const double fm = cost(qt, t0, mid);
            if (fm <= budget) { lo = mid; flo = fm; } else { hi = mid; fhi = fm; }
        }
        *fe = flo;
        return lo;
    };
    // one greedy pass: CTA c takes about (remaining cost + later[c]) / (G - c);
    // returns the largest share's cost, the heads (cost from each cut to the
    // end of its query tile) in `head`
    std::vector<double> head(G, 0.0);
    auto greedy = [&](const std::vector<double> &later, std::vector<int64_t> &cu) {
        cu.assign(G + 1, T);
        cu[0] = 0;
        int64_t t = 0, qt = 0;
        double worst = 0.0;
        for (int64_t c = 0; c < G; ++c) {
            while (qt_first[qt + 1] <= t) ++qt;
            const int64_t qend = qt_first[qt + 1];
            const double h = t == qt_first[qt] ? pre[qt + 1] - pre[qt] : cost(qt, t, qend);
            head[c] = h;
            const double rest = h + pre[nqt] - pre[qt + 1];
            if (c + 1 == G) { worst = std::max(worst, rest); break; }
            const double target = (rest + later[c]) / (double)(G - c);
            int64_t e;
            double share;
            if (h > target) {
                e = last_within(qt, t, t, qend, 0.0, h, target, &share);
            } else {
                // the query tile the cut falls in, then the position inside it
                const double rem = target - h;
                const int64_t qe = std::upper_bound(pre.begin() + qt + 1, pre.end(), pre[qt + 1] + rem) - pre.begin() - 1;
                if (qe >= nqt) {
                    e = T;
                    share = rest;
                } else {
                    double part = 0.0;
                    e = last_within(qe, qt_first[qe], qt_first[qe], qt_first[qe + 1], 0.0, pre[qe + 1] - pre[qe],
                                    rem - (pre[qe] - pre[qt + 1]), &part);
                    share = h + (pre[qe] - pre[qt + 1]) + part;
                }
            }
            if (e < t + 1 || e > T - (G - c - 1)) {
                e = std::min(std::max(e, t + 1), T - (G - c - 1));
                const int64_t qe = std::upper_bound(qt_first.begin(), qt_first.end(), e - 1) - qt_first.begin() - 1;
                share = qe == qt ? cost(qt, t, e) : h + (pre[qe] - pre[qt + 1]) + cost(qe, qt_first[qe], e);
            }
            worst = std::max(worst, share);
            cu[c + 1] = e;
            t = e;
        }
        return worst;
    };
    std::vector<double> later(G, 0.0);
    std::vector<int64_t> cur, nxt;
    double best = greedy(later, cur);
    cut = cur;
    const double mean = pre[nqt] / (double)G;
    for (int pass = 1; pass < kSharePasses && best - mean >= std::max(slack, uneven * mean); ++pass) {
        // restart cost of each cut of the previous pass (the next share's head
        // plus the query tile's cost up to the cut, minus the whole query
        // tile), summed over the later cuts
        for (int64_t c = G - 2; c >= 0; --c) {
            const int64_t t = cur[c + 1];
            double o = 0.0;
            if (t < T) {
                const int64_t qt = std::upper_bound(qt_first.begin(), qt_first.end(), t) - qt_first.begin() - 1;
                if (t > qt_first[qt]) o = head[c + 1] + cost(qt, qt_first[qt], t) - (pre[qt + 1] - pre[qt]);
            }
            later[c] = later[c + 1] + o;
        }
        const double w = greedy(later, nxt);
        if (w < best) { best = w; cut = nxt; }
        cur.swap(nxt);
    }
}

// Host work plan of the pipelined kernel for the valid queries of host
// ranges hl/hr over n points at dimension d, for `sms` CTAs: queries sorted
// by (log2 width, l, index) and tiled by 128, the rows of each full query tile
// interleaved over the four TMEM lane quarters, the point tiles each query
// tile covers in one sequence, cut into `G` shares (bf2_shares) and into work
// items at query-tile boundaries. ESG_ERR_UNSUPPORTED past 2^31 covered tiles.
struct Bf2Plan {
    std::vector<int32_t> order;        // sorted position -> caller's query index (valid queries)
    Spans spans;                       // covered point tiles of each query tile
    std::vector<int64_t> qt_first;     // [nqt + 1] first position of each query tile in `tiles`
    std::vector<WorkItem> items;       // in query-tile order, each CTA's items contiguous
    std::vector<int32_t> item_begin;   // [nqt + 1] first item of each query tile
    std::vector<int32_t> cta_first;    // [G + 1] first item of each CTA
    std::vector<int64_t> doff;         // [V] first entry of a dense row in its buffer, -1 for the others
    int64_t nv = 0, nqt = 0, total_tiles = 0, G = 0, largest = 0, dense = 0;   // dense: floats of all dense rows
};

// Rows of narrow ranges write all their distances (the finish kernel selects
// from them) instead of keeping lists. Ranges that begin inside a work item
// start their lists one row at a time, and a list start costs a CTA about
// 27,000 cycles of insertions, one row of the warp active in each; a dense row
// costs it about 25 cycles per tile (its 16-byte stores). The lines cross at
// about 135,000 points at d <= 128. At larger d, where a tile's MMAs take longer
// and hide the insertions, dense rows only add memory traffic (1.66 against 1.50
// ms at 200,003 x 768). The buffer's bound halves the width until it fits.
// Lists in memory cost several times the insertions: rows up to twice as wide
// are dense, in a buffer twice as large (1M x 96, 10k queries, k = 100: 9.5 ms a
// call, 179 ms through the SIMT kernel).
constexpr int64_t kDenseWidth = 131072;
constexpr int64_t kDenseFloats = (int64_t)1 << 28;   // 1 GiB at most (2 GiB with lists in memory)

static void bf2_dense(const int64_t *hl, const int64_t *hr, int64_t widest, int64_t most, Bf2Plan &P) {
    P.doff.assign(P.order.size(), -1);
    for (int64_t w = widest; w >= 64; w /= 2) {
        P.dense = 0;
        for (size_t s = 0; s < P.order.size(); ++s) {
            const int64_t l = hl[P.order[s]], r = hr[P.order[s]];
            const bool in = r - l + 1 <= w;
            P.doff[s] = in ? P.dense : -1;
            if (in) P.dense += (r | 3) - (l & ~(int64_t)3) + 1;
        }
        if (P.dense <= most) return;
    }
    P.dense = 0;
    std::fill(P.doff.begin(), P.doff.end(), (int64_t)-1);
}

// `run`: the plan is for the kernel with lists of K1 (dense rows where `dense_rows`,
// its restart cost), not for inspection.
static esg_status bf2_plan(const int64_t *hl, const int64_t *hr, int64_t nq, int64_t n, int32_t d, int64_t sms,
                           bool run, int K1, Bf2Plan &P, bool dense_rows = true) {
    // sorted by (floor(log2 width), l, query index): a stable LSD radix sort
    // of the valid queries in index order, by 11 bits of l at a time and then
    // by the width class
    std::vector<uint64_t> keys, tmp;   // l << 32 | query
    keys.reserve(nq);
    for (int64_t i = 0; i < nq; ++i)
        if (hl[i] >= 0 && hl[i] <= hr[i] && hr[i] < n) keys.push_back((uint64_t)hl[i] << 32 | (uint32_t)i);
    const int64_t nv = (int64_t)keys.size();
    const int64_t nqt = (nv + TM - 1) / TM;
    const int nk = (d + TK - 1) / TK;
    tmp.resize(nv);
    std::vector<uint32_t> cnt(2049);
    for (int sh = 32; (uint64_t)(n - 1) >> (sh - 32) != 0 && sh < 63; sh += 11) {
        std::fill(cnt.begin(), cnt.end(), 0u);
        for (const uint64_t k : keys) ++cnt[((k >> sh) & 2047) + 1];
        for (int b = 0; b < 2048; ++b) cnt[b + 1] += cnt[b];
        for (const uint64_t k : keys) tmp[cnt[(k >> sh) & 2047]++] = k;
        keys.swap(tmp);
    }
    std::vector<int32_t> &order = P.order;
    order.resize(nv);
    {
        auto cls = [&](uint64_t k) {
            const int64_t i = (int64_t)(k & 0xFFFFFFFFu);
            return 63 - __builtin_clzll((unsigned long long)(hr[i] - hl[i] + 1));
        };
        uint32_t c[65] = {0};
        for (const uint64_t k : keys) ++c[cls(k) + 1];
        for (int b = 0; b < 64; ++b) c[b + 1] += c[b];
        for (const uint64_t k : keys) order[c[cls(k)]++] = (int32_t)(k & 0xFFFFFFFFu);
    }
    // covered tiles of each query tile, as spans
    Spans &sp = P.spans;
    sp.first.assign(nqt + 1, 0);
    std::vector<int64_t> &qt_first = P.qt_first;
    qt_first.assign(nqt + 1, 0);
    int64_t total_tiles = 0;
    {
        std::vector<std::pair<int32_t, int32_t>> iv(TM);
        for (int64_t qt = 0; qt < nqt; ++qt) {
            const int64_t s0 = qt * TM, s1 = std::min(nv, (qt + 1) * TM);
            for (int64_t s = s0; s < s1; ++s)
                iv[s - s0] = {(int32_t)(hl[order[s]] / TN), (int32_t)(hr[order[s]] / TN)};
            if (!std::is_sorted(iv.begin(), iv.begin() + (s1 - s0))) std::sort(iv.begin(), iv.begin() + (s1 - s0));
            for (int64_t s = 0; s < s1 - s0; ++s) {
                if ((int64_t)sp.a.size() > sp.first[qt] && iv[s].first <= sp.b.back() + 1) {
                    sp.b.back() = std::max(sp.b.back(), iv[s].second);
                } else {
                    sp.a.push_back(iv[s].first);
                    sp.b.push_back(iv[s].second);
                }
            }
            for (size_t x = sp.first[qt]; x < sp.a.size(); ++x) {
                sp.at.push_back(total_tiles);
                total_tiles += sp.b[x] - sp.a[x] + 1;
            }
            sp.first[qt + 1] = (int32_t)sp.a.size();
            qt_first[qt + 1] = total_tiles;
        }
    }
    // the rows of each full query tile interleaved over the four TMEM lane
    // quarters (sorted position s -> row (s mod 4) * 32 + s / 4): queries
    // with nearby ranges take their insertions in the same point tiles, and
    // an accumulator is free only when all four warps of its group are done
    for (int64_t qt = 0; qt < nv / TM; ++qt) {
        int32_t rows[TM];
        for (int i = 0; i < TM; ++i) rows[(i & 3) * 32 + (i >> 2)] = order[qt * TM + i];
        std::copy(rows, rows + TM, order.begin() + qt * TM);
    }
    if (total_tiles >= ((int64_t)1 << 31)) return ESG_ERR_UNSUPPORTED;
    // the covered tiles of all query tiles in one sequence (query tile by query
    // tile); CTA c runs the share [cut[c], cut[c + 1]) of it, shares of equal
    // estimated cost, cut into work items at query-tile boundaries (items in
    // query-tile order, each CTA's items contiguous)
    const int64_t G = std::max<int64_t>(1, std::min<int64_t>(sms, total_tiles));
    std::vector<int64_t> cut;
    {
        std::vector<int32_t> lt(nv), rt(nv), dense(nv, 0);
        const int64_t x = K1 > 32 ? 2 : 1;
        if (run) bf2_dense(hl, hr, dense_rows && nk <= 2 ? x * kDenseWidth : 0, x * kDenseFloats, P);
        for (int64_t s = 0; s < nv; ++s) {
            lt[s] = (int32_t)(hl[order[s]] / TN);
            rt[s] = (int32_t)(hr[order[s]] / TN);
            dense[s] = run && P.doff[s] >= 0 ? -1 : 0;
        }
        // weights in tiles at two K chunks, from the CTAs' clock counters at
        // 1M x 128 (27,000 cycles for a row that begins inside the item, 25 for
        // a dense row's tile, 2,300 for a tile); a tile's MMAs grow with nk,
        // and past two chunks they hide more and more of the epilogue
        const double f = 2.0 / nk, g = nk <= 2 ? f : f * f * f;
        const double c = K1 > 32 ? K1 / 24.0 : 1.0;   // insertions grow with the list
        const ShareCost w = run ? ShareCost{16.0 * c * g, 0.5 * c * g, 0.0104 * g}
                                : ShareCost{kRestart2 * f * f, kRestart2 * f * f, 0.0};
        bf2_shares(sp, qt_first, lt, rt, dense, G, w, run ? kShareUneven : 0.0, run ? kShareSlack * f : 0.0, cut);
    }
    std::vector<WorkItem> &items = P.items;
    items.clear();
    std::vector<int32_t> &item_begin = P.item_begin, &cta_first = P.cta_first;
    item_begin.assign(nqt + 1, 0);
    cta_first.assign(G + 1, 0);
    for (int64_t c = 0; c < G; ++c) {
        cta_first[c] = (int32_t)items.size();
        const int64_t t0 = cut[c], t1 = cut[c + 1];
        int64_t t = t0;
        int64_t qt = std::upper_bound(qt_first.begin(), qt_first.end(), t0) - qt_first.begin() - 1;
        while (t < t1) {
            while (qt_first[qt + 1] <= t) ++qt;
            const int64_t e = std::min(t1, qt_first[qt + 1]);
            items.push_back(WorkItem{(int32_t)qt, (int32_t)t, (int32_t)(e - t), 0});
            t = e;
        }
    }
    cta_first[G] = (int32_t)items.size();
    for (int64_t qt = 0, i = 0; qt <= nqt; ++qt) {   // first item of each query tile
        while (i < (int64_t)items.size() && items[i].qtile < qt) ++i;
        item_begin[qt] = (int32_t)i;
    }
    P.largest = 0;
    for (int64_t c = 0; c < G; ++c) P.largest = std::max(P.largest, cut[c + 1] - cut[c]);
    P.nv = nv;
    P.nqt = nqt;
    P.total_tiles = total_tiles;
    P.G = G;
    return ESG_OK;
}

// The covered tiles of a work item in the order its CTA takes them: rotated to
// begin at the first one at or after a multiple of `period`, about the length
// of the long items. The CTAs that sweep the same points with different query
// tiles then read the same blocks at about the same time, more of them from the
// L2 (without and with it, DRAM reads and the kernel: 10,000 queries over 1M x 128
// 11.8 and 10.0 GB, 2.15 and 2.05 ms; 2,000 over 200,000 x 768 5.4 and 1.8 GB,
// 1.18 and 1.07 ms). The spans are the query tiles' (Spans).
struct ItemTiles {
    const int32_t *a;
    const int64_t *at;
    int32_t x0, x1, cnt, lead;
    int64_t off;
    __host__ __device__ ItemTiles(const WorkItem &w, const int32_t *span_a, const int32_t *span_first,
                                  const int64_t *span_at, int period)
        : a(span_a), at(span_at), x0(span_first[w.qtile]), x1(span_first[w.qtile + 1]), cnt(w.cnt), off(w.off) {
        const int32_t from = (ascending(off) + period - 1) / period * period;   // tiles below 2^24
        int lo = 0, hi = cnt;
        while (lo < hi) {
            const int m = (lo + hi) >> 1;
            if (ascending(off + m) < from) lo = m + 1; else hi = m;
        }
        lead = lo;
    }
    __host__ __device__ int32_t ascending(int64_t pos) const {
        int32_t x = x1 - 1;
        while (x > x0 && at[x] > pos) --x;
        return a[x] + (int32_t)(pos - at[x]);
    }
    __host__ __device__ int32_t operator[](int j) const {
        const uint32_t i = (uint32_t)lead + (uint32_t)j;
        return ascending(off + (i < (uint32_t)cnt ? i : i - (uint32_t)cnt));
    }
};

// The rotation's period: an upper quartile of the items' lengths.
static int bf2_period(const std::vector<WorkItem> &items) {
    std::vector<int32_t> c(items.size());
    for (size_t i = 0; i < items.size(); ++i) c[i] = items[i].cnt;
    std::nth_element(c.begin(), c.begin() + c.size() * 3 / 4, c.end());
    return c[c.size() * 3 / 4];
}

// Writes out the covered tiles of the work items, a block each.
__global__ void expand_tiles_kernel(const WorkItem *items, const int32_t *span_a, const int32_t *span_first,
                                    const int64_t *span_at, int period, int32_t *tiles) {
    const WorkItem w = items[blockIdx.x];
    const ItemTiles t(w, span_a, span_first, span_at, period);
    for (int j = threadIdx.x; j < w.cnt; j += blockDim.x) tiles[w.off + j] = t[j];
}

// One pass of the pipelined kernel over a batch of queries against the
// prepared points, then merge, re-rank, certificate and escalation.
// `given`: a plan already made for these ranges (it is consumed), or null. Where
// memory is too short for the dense rows' buffer the pass goes without it.
static esg_status bf2_queries(const PreparedX &X, const float *base, int64_t n, int32_t d, int metric,
                              const float *queries, int64_t nq, const int64_t *l, const int64_t *r, int32_t k,
                              int K1, int64_t *out_ids, float *out_dist, int32_t *out_count, cudaStream_t stream,
                              Bf2Plan *given, bool dense_rows) {
    if (nq == 0) return ESG_OK;
    const double h0 = bf_stats() ? bf_host_ms() : 0.0;
    const int nk = (d + TK - 1) / TK;
    int dev = 0, max_smem = 0, sms = 0, S = 0, n_acc = 0;
    bool stream_a = false, list_smem = false;
    size_t smem = 0;
    ESG_CUDA_TRY(cudaGetDevice(&dev));
    ESG_CUDA_TRY(cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    ESG_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    if (bf2_smem(d, K1, max_smem, &S, &smem, &n_acc, &stream_a, &list_smem) != ESG_OK) return ESG_ERR_UNSUPPORTED;

    // ---- host plan
    Bf2Plan P;
    if (given) {
        P = std::move(*given);
    } else {
        std::vector<int64_t> hl(nq), hr(nq);
        ESG_CUDA_TRY(cudaMemcpyAsync(hl.data(), l, sizeof(int64_t) * nq, cudaMemcpyDeviceToHost, stream));
        ESG_CUDA_TRY(cudaMemcpyAsync(hr.data(), r, sizeof(int64_t) * nq, cudaMemcpyDeviceToHost, stream));
        ESG_CUDA_TRY(cudaStreamSynchronize(stream));
        const esg_status pst = bf2_plan(hl.data(), hr.data(), nq, n, d, sms, true, K1, P, dense_rows);
        if (pst != ESG_OK) return pst;
    }
    const std::vector<int32_t> &order = P.order, &item_begin = P.item_begin, &cta_first = P.cta_first;
    const std::vector<WorkItem> &items = P.items;
    const int64_t n_spans = (int64_t)P.spans.a.size();
    const int64_t nv = P.nv, nqt = P.nqt, total_tiles = P.total_tiles, G = P.G, CH = P.largest;
    const int64_t n_items = (int64_t)items.size();

    // ---- query-side scratch
    auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
    const int64_t ni1 = std::max<int64_t>(n_items, 1);
    size_t bytes = al((size_t)std::max<int64_t>(nqt, 1) * nk * STAGE) + 2 * al(sizeof(float) * nq) +
                   al(sizeof(int32_t) * std::max<int64_t>(nv, 1)) + al(sizeof(WorkItem) * ni1) +
                   al(sizeof(int32_t) * std::max<int64_t>(total_tiles, 1)) + al(sizeof(int32_t) * (nqt + 1)) +
                   al(sizeof(int32_t) * (G + 1)) + al(sizeof(Key) * 2 * ni1 * K1 * TM) +
                   al(sizeof(int32_t) * 2 * ni1 * TM) + al(sizeof(int32_t) * nq) + al(sizeof(int32_t) * 4) +
                   al(sizeof(int64_t) * std::max<int64_t>(nv, 1)) + al(sizeof(float) * P.dense) +
                   al(sizeof(int32_t) * n_spans) + al(sizeof(int64_t) * n_spans) + al(sizeof(int32_t) * (nqt + 1));
    Scratch scratch(stream);
    const cudaError_t me = scratch.alloc(bytes);
    if (me == cudaErrorMemoryAllocation && P.dense > 0) {
        cudaGetLastError();
        return bf2_queries(X, base, n, d, metric, queries, nq, l, r, k, K1, out_ids, out_dist, out_count, stream,
                           nullptr, false);
    }
    ESG_CUDA_TRY(me);
    unsigned char *p = scratch.p;
    auto take = [&](size_t b) { unsigned char *q = p; p += al(b); return q; };
    unsigned char *qs = take((size_t)std::max<int64_t>(nqt, 1) * nk * STAGE);
    float *qnorm = (float *)take(sizeof(float) * nq);
    float *qrow = (float *)take(sizeof(float) * nq);
    int32_t *d_order = (int32_t *)take(sizeof(int32_t) * std::max<int64_t>(nv, 1));
    WorkItem *d_items = (WorkItem *)take(sizeof(WorkItem) * ni1);
    int32_t *d_tiles = (int32_t *)take(sizeof(int32_t) * std::max<int64_t>(total_tiles, 1));
    int32_t *d_ib = (int32_t *)take(sizeof(int32_t) * (nqt + 1));
    int32_t *d_cta = (int32_t *)take(sizeof(int32_t) * (G + 1));
    Key *part = (Key *)take(sizeof(Key) * 2 * ni1 * K1 * TM);
    int32_t *part_n = (int32_t *)take(sizeof(int32_t) * 2 * ni1 * TM);
    int32_t *redo = (int32_t *)take(sizeof(int32_t) * nq);
    int32_t *err = (int32_t *)take(sizeof(int32_t) * 4);
    int64_t *d_doff = (int64_t *)take(sizeof(int64_t) * std::max<int64_t>(nv, 1));
    float *dense = (float *)take(sizeof(float) * P.dense);
    int32_t *d_span_a = (int32_t *)take(sizeof(int32_t) * n_spans);
    int64_t *d_span_at = (int64_t *)take(sizeof(int64_t) * n_spans);
    int32_t *d_span_first = (int32_t *)take(sizeof(int32_t) * (nqt + 1));

    esg_status st = ESG_OK;
    cudaError_t ce = cudaMemsetAsync(err, 0, sizeof(int32_t) * 4, stream);
    if (ce == cudaSuccess && nv > 0)
        ce = cudaMemcpyAsync(d_order, order.data(), sizeof(int32_t) * nv, cudaMemcpyHostToDevice, stream);
    if (ce == cudaSuccess && nv > 0)
        ce = cudaMemcpyAsync(d_doff, P.doff.data(), sizeof(int64_t) * nv, cudaMemcpyHostToDevice, stream);
    if (ce == cudaSuccess && n_items > 0)
        ce = cudaMemcpyAsync(d_items, items.data(), sizeof(WorkItem) * n_items, cudaMemcpyHostToDevice, stream);
    if (ce == cudaSuccess && n_items > 0) {
        ce = cudaMemcpyAsync(d_span_a, P.spans.a.data(), sizeof(int32_t) * n_spans, cudaMemcpyHostToDevice, stream);
        if (ce == cudaSuccess)
            ce = cudaMemcpyAsync(d_span_at, P.spans.at.data(), sizeof(int64_t) * n_spans, cudaMemcpyHostToDevice, stream);
        if (ce == cudaSuccess)
            ce = cudaMemcpyAsync(d_span_first, P.spans.first.data(), sizeof(int32_t) * (nqt + 1),
                                 cudaMemcpyHostToDevice, stream);
        if (ce == cudaSuccess) {
            esg_fault_host();
            expand_tiles_kernel<<<(unsigned)n_items, 256, 0, stream>>>(d_items, d_span_a, d_span_first, d_span_at,
                                                                       bf2_period(items), d_tiles);
            ce = cudaGetLastError();
        }
    }
    if (ce == cudaSuccess)
        ce = cudaMemcpyAsync(d_ib, item_begin.data(), sizeof(int32_t) * (nqt + 1), cudaMemcpyHostToDevice, stream);
    if (ce == cudaSuccess)
        ce = cudaMemcpyAsync(d_cta, cta_first.data(), sizeof(int32_t) * (G + 1), cudaMemcpyHostToDevice, stream);
    if (ce == cudaSuccess) {
        if (nqt > 0)
            ce = split_norm(queries, nv, d, nk, d_order, nqt * TM, qs, qnorm, qrow, nullptr, stream);
    }
    // lists of 24 or 32 in registers, or in memory: 64 or 128 keys over a warp's lanes
    const bool l2 = metric == ESG_L2SQ, one = K1 <= 32, two = K1 <= 64;
    auto pick = [&](auto s) -> void (*)(Tc2Args) {
        constexpr bool ST = decltype(s)::value;
        switch (bf2_reg_list(K1)) {
            case 24: return l2 ? tc_knn2_kernel<true, 24, 1, ST> : tc_knn2_kernel<false, 24, 1, ST>;
            case 32: return l2 ? tc_knn2_kernel<true, 32, 1, ST> : tc_knn2_kernel<false, 32, 1, ST>;
        }
        return l2 ? (two ? tc_knn2_kernel<true, 0, 2, ST> : tc_knn2_kernel<true, 0, 4, ST>)
                  : (two ? tc_knn2_kernel<false, 0, 2, ST> : tc_knn2_kernel<false, 0, 4, ST>);
    };
    void (*fn)(Tc2Args) = stream_a ? pick(std::true_type{}) : pick(std::false_type{});
    if (ce == cudaSuccess) ce = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (ce == cudaSuccess && nv < nq) {
        invalid_kernel<<<ceil_div_i(nq, 256), 256, 0, stream>>>(l, r, nq, n, k, out_ids, out_dist, out_count, redo);
        ce = cudaGetLastError();
    }
    if (ce == cudaSuccess && n_items > 0) {
        // MMA work issued: three 128 x 128 x 64 BF16 products per point tile and K chunk
        esg_prof_tensor_flops((double)total_tiles * nk * 3.0 * 2.0 * TM * TN * TK);
        // failure-detection hooks (host side): ESG_BF_WAIT_NS bounds each
        // pipeline wait, ESG_TEST_BF_STALL=1 makes every CTA's first wait one
        // that nothing completes
        const char *wn = getenv("ESG_BF_WAIT_NS");
        const char *stl = getenv("ESG_TEST_BF_STALL");
        const unsigned long long wait_ns = wn && *wn ? std::max(1ull, strtoull(wn, nullptr, 10)) : kWaitNs;
        Tc2Args a{X.xs, qs, X.xnorm, qnorm, l, r, d_order, d_doff, dense, d_items, d_tiles, d_cta, (int)n_items, nv, nk, metric, K1, S,
                  list_smem ? 1 : 0, n_acc,
                  // two issuers wait for stages of two tiles: a barrier must
                  // not be waited for more than one use ahead
                  !stream_a && 2 * nk <= S ? 2 : 1,
                  n, part, part_n, err, wait_ns, (stl && atoi(stl) == 1) ? 1 : 0};
        const int pidx = esg_prof_begin(stream);
        fn<<<(unsigned)G, kThreads2, smem, stream>>>(a);
        ce = cudaGetLastError();
        esg_prof_end(pidx, stream);
        if (ce == cudaSuccess) {
            const FinishArgs f{base, queries, d, metric, k, K1, part, part_n, d_ib, d_order, d_doff, l, r, dense, qnorm, qrow,
                               X.xmax, bf2_serial(d, k) ? 1 : 0,
                               out_ids, out_dist, out_count, redo};
            // many lists per query: two per item, items shared out over the query tiles
            if (n_items > 16 * nqt) {
                if (one) finish_kernel<1, 16><<<(unsigned)nv, 512, 0, stream>>>(f);
                else if (two) finish_kernel<2, 16><<<(unsigned)nv, 512, 0, stream>>>(f);
                else finish_kernel<4, 8><<<(unsigned)nv, 256, 0, stream>>>(f);
            } else {
                if (one) finish_kernel<1, 4><<<(unsigned)nv, 128, 0, stream>>>(f);
                else if (two) finish_kernel<2, 4><<<(unsigned)nv, 128, 0, stream>>>(f);
                else finish_kernel<4, 4><<<(unsigned)nv, 128, 0, stream>>>(f);
            }
            ce = cudaGetLastError();
        }
    }
    if (ce != cudaSuccess) { esg_set_error(cudaGetErrorString(ce)); st = ESG_ERR_CUDA; }
    const char *dbg = getenv("ESG_BF_STATS");
    if (dbg && *dbg == '1')
        fprintf(stderr, "tensor-core brute force (pipelined): %lld query tiles, %lld point tiles, %lld items, largest share %lld tiles, %d stages%s\n",
                (long long)nqt, (long long)total_tiles, (long long)n_items, (long long)CH, S,
                stream_a ? " (query tile streamed)" : "");
    std::vector<int64_t> left;
    const double h1 = bf_stats() ? bf_host_ms() : 0.0;
    if (st == ESG_OK)
        st = read_uncertified(nq, K1, redo, err, stream, left);
    scratch.release();
    const double h2 = bf_stats() ? bf_host_ms() : 0.0;
    if (st == ESG_OK && !left.empty())
        st = bf2_escalate(X, base, n, d, metric, queries, nq, l, r, k, K1, left, out_ids, out_dist, out_count, stream);
    if (bf_stats())
        fprintf(stderr, "tensor-core brute force, host ms: plan + uploads + launches %.3f, until certified %.3f, "
                        "escalation %.3f\n", h1 - h0, h2 - h1, bf_host_ms() - h2);
    return st;
}

// Pipelined tensor-core path; ESG_ERR_UNSUPPORTED when the shape does not fit
// (k > 120, or shared memory for fewer than two stages). Each list keeps
// about k + 12 approximate candidates: the certificate needs the exact k-th
// distance below the approximate K1-th minus the error bound, which holds for
// nearly every query, and a short list makes the epilogue's filter sharp; the
// few queries left uncertified run again with a longer list.
static esg_status bruteforce_tc_v2(const float *base, int64_t n, int32_t d, int metric, const float *queries,
                                   int64_t nq, const int64_t *l, const int64_t *r, int32_t k, int64_t *out_ids,
                                   float *out_dist, int32_t *out_count, cudaStream_t stream) {
    if (k < 1 || k + 8 > kMaxK1v2 || n >= ((int64_t)1 << 31) || d < 1) return ESG_ERR_UNSUPPORTED;
    const int K1 = bf2_list(k);
    int dev = 0, max_smem = 0, S = 0, n_acc = 0;
    bool stream_a = false, list_smem = false;
    size_t smem = 0;
    ESG_CUDA_TRY(cudaGetDevice(&dev));
    ESG_CUDA_TRY(cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    if (bf2_smem(d, K1, max_smem, &S, &smem, &n_acc, &stream_a, &list_smem) != ESG_OK) return ESG_ERR_UNSUPPORTED;
    if (nq == 0) return ESG_OK;
    const double t0 = bf_stats() ? bf_host_ms() : 0.0;
    const int nk = (d + TK - 1) / TK;
    const int64_t xt = (n + TN - 1) / TN;
    // the ranges come to the host first, so that the host plan is made while
    // the GPU splits and swizzles the point matrix
    int sms = 0;
    ESG_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    std::vector<int64_t> hl(nq), hr(nq);
    ESG_CUDA_TRY(cudaMemcpyAsync(hl.data(), l, sizeof(int64_t) * nq, cudaMemcpyDeviceToHost, stream));
    ESG_CUDA_TRY(cudaMemcpyAsync(hr.data(), r, sizeof(int64_t) * nq, cudaMemcpyDeviceToHost, stream));
    ESG_CUDA_TRY(cudaStreamSynchronize(stream));
    if (bf2_serial(d, k)) {
        int64_t sum = 0;
        for (int64_t i = 0; i < nq; ++i)
            if (hl[i] >= 0 && hl[i] <= hr[i] && hr[i] < n) sum += hr[i] - hl[i] + 1;
        if (kLook + simt_us(hl, hr, n, d, k, sms) < tc_us(n, nq, sum / nq, d, k, sms)) return ESG_ERR_UNSUPPORTED;
    }
    auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
    const size_t bytes = al((size_t)xt * nk * STAGE) + al(sizeof(float) * xt * TN) + al(sizeof(float) * 4);
    Scratch scratch(stream);
    ESG_CUDA_TRY(scratch.alloc(bytes));
    unsigned char *p = scratch.p;
    unsigned char *xs = p; p += al((size_t)xt * nk * STAGE);
    float *xnorm = (float *)p; p += al(sizeof(float) * xt * TN);   // past n: never in a range
    float *xmax = (float *)p;
    esg_status st = ESG_OK;
    cudaError_t ce = cudaMemsetAsync(xmax, 0, sizeof(float) * 4, stream);
    if (ce == cudaSuccess) {
        ce = split_norm(base, n, d, nk, nullptr, xt * TN, xs, xnorm, nullptr, xmax, stream);
    }
    if (ce != cudaSuccess) { esg_set_error(cudaGetErrorString(ce)); st = ESG_ERR_CUDA; }
    const double t1 = bf_stats() ? bf_host_ms() : 0.0;
    Bf2Plan P;
    if (st == ESG_OK) {
        try {
            st = bf2_plan(hl.data(), hr.data(), nq, n, d, sms, true, K1, P);
        } catch (...) {
            esg_set_error("tensor-core brute force: out of memory (host plan)");
            st = ESG_ERR_OOM;
        }
    }
    if (bf_stats()) fprintf(stderr, "tensor-core brute force, host ms: ranges + point prep queued %.3f, plan %.3f\n",
                            t1 - t0, bf_host_ms() - t1);
    if (st == ESG_OK) {
        const PreparedX X{xs, xnorm, xmax};
        st = bf2_queries(X, base, n, d, metric, queries, nq, l, r, k, K1, out_ids, out_dist, out_count, stream, &P);
    }
    return st;
}

// Tensor-core path of esg_bruteforce_filtered_knn; returns ESG_ERR_UNSUPPORTED
// when the shape is outside it (the caller then uses the SIMT kernel). Where the
// SIMT kernel gives the same answers bit for bit (bf2_serial), it also serves the
// calls it answers sooner and those that this path cannot: it needs no scratch
// memory and no host synchronisation, so it runs when memory is short and under
// stream capture.
esg_status esg_bruteforce_tc(const float *base, int64_t n, int32_t d, int metric, const float *queries,
                             int64_t nq, const int64_t *l, const int64_t *r, int32_t k, int64_t *out_ids,
                             float *out_dist, int32_t *out_count, cudaStream_t stream) {
    const bool simt_too = bf2_serial(d, k);
    if (simt_too) {
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(stream, &cs) != cudaSuccess) cudaGetLastError();
        if (cs != cudaStreamCaptureStatusNone) return ESG_ERR_UNSUPPORTED;
        // small enough whatever the ranges are: no look at them, no host synchronisation
        int dev = 0, sms = 0;
        ESG_CUDA_TRY(cudaGetDevice(&dev));
        ESG_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        if (simt_us_at_most(n, nq, d, k, sms) < tc_us(n, nq, 0, d, k, sms)) return ESG_ERR_UNSUPPORTED;
    }
    esg_status st;
    try {
        st = bruteforce_tc_v2(base, n, d, metric, queries, nq, l, r, k, out_ids, out_dist, out_count, stream);
    } catch (...) {
        esg_set_error("tensor-core brute force: out of memory (host)");
        st = ESG_ERR_OOM;
    }
    if (simt_too && st == ESG_ERR_OOM) {
        cudaGetLastError();   // the failed allocation's
        st = ESG_ERR_UNSUPPORTED;
    }
    return st;
}

// The parts of a plan that both inspection calls return.
static void copy_plan(const Bf2Plan &P, int32_t *order, int32_t *items, int32_t *cta_first) {
    if (order) std::copy(P.order.begin(), P.order.end(), order);
    if (items)
        for (size_t i = 0; i < P.items.size(); ++i) {
            items[4 * i] = P.items[i].qtile;
            items[4 * i + 1] = P.items[i].off;
            items[4 * i + 2] = P.items[i].cnt;
            items[4 * i + 3] = 0;
        }
    if (cta_first) std::copy(P.cta_first.begin(), P.cta_first.end(), cta_first);
}

static esg_status inspect_plan(const char *who, int64_t n, int32_t d, const int64_t *l, const int64_t *r, int64_t nq,
                               int32_t ctas, const int64_t *sizes, bool run, int K1, Bf2Plan &P) {
    if (n < 1 || n >= ((int64_t)1 << 31) - 1 || d < 1 || nq < 0 || nq >= ((int64_t)1 << 31) || ctas < 1 ||
        !sizes || (nq > 0 && (!l || !r))) {
        esg_set_error(std::string(who) + ": bad argument");
        return ESG_ERR_INVALID_ARG;
    }
    esg_status st = ESG_OK;
    try {
        st = bf2_plan(l, r, nq, n, d, ctas, run, K1, P);
    } catch (...) { st = ESG_ERR_OOM; }
    if (st == ESG_ERR_UNSUPPORTED) esg_set_error(std::string(who) + ": more than 2^31 covered point tiles");
    return st;
}

esg_status esg_bruteforce_plan(int64_t n, int32_t d, const int64_t *l, const int64_t *r, int64_t nq,
                               int32_t ctas, int64_t *sizes, int32_t *order, int32_t *tiles, int32_t *items,
                               int32_t *cta_first) {
    Bf2Plan P;
    const esg_status st = inspect_plan("esg_bruteforce_plan", n, d, l, r, nq, ctas, sizes, false, 0, P);
    if (st != ESG_OK) return st;
    sizes[0] = P.nv;
    sizes[1] = P.total_tiles;
    sizes[2] = (int64_t)P.items.size();
    sizes[3] = P.G;
    if (tiles)
        for (size_t x = 0; x < P.spans.a.size(); ++x)
            for (int32_t t = P.spans.a[x]; t <= P.spans.b[x]; ++t) *tiles++ = t;
    copy_plan(P, order, items, cta_first);
    return ESG_OK;
}

esg_status esg_bruteforce_search_plan(int64_t n, int32_t d, int32_t k, const int64_t *l, const int64_t *r, int64_t nq,
                                      int32_t ctas, int64_t *sizes, int32_t *order, int32_t *tiles, int32_t *items,
                                      int32_t *cta_first, int64_t *dense) {
    if (k < 1 || k + 8 > kMaxK1v2) {
        esg_set_error("esg_bruteforce_search_plan: k outside the tensor-core path");
        return ESG_ERR_INVALID_ARG;
    }
    Bf2Plan P;
    const esg_status st = inspect_plan("esg_bruteforce_search_plan", n, d, l, r, nq, ctas, sizes, true, bf2_list(k), P);
    if (st != ESG_OK) return st;
    sizes[0] = P.nv;
    sizes[1] = P.total_tiles;
    sizes[2] = (int64_t)P.items.size();
    sizes[3] = P.G;
    sizes[4] = P.dense;
    sizes[5] = P.items.empty() ? 0 : bf2_period(P.items);
    if (tiles)
        for (const WorkItem &w : P.items) {
            const ItemTiles t(w, P.spans.a.data(), P.spans.first.data(), P.spans.at.data(), (int)sizes[5]);
            for (int j = 0; j < w.cnt; ++j) tiles[w.off + j] = t[j];
        }
    copy_plan(P, order, items, cta_first);
    if (dense) std::copy(P.doff.begin(), P.doff.end(), dense);
    return ESG_OK;
}

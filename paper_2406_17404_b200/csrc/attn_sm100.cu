// Tree-masked attention for sm_100a (bf16, head_dim 128, up to 128 tree rows per sequence).
//
// Work is cut into units of one 128-key tile of one (sequence, head).  A CTA works on TWO STREAMS of units at a time: what
// bounds a stream is its chain of dependent steps (scores -> softmax -> P.V -> next scores: 2.3 us a tile with a bf16 P and
// 4.6 us with a pair in the one-stream form of this kernel, against 1.4 us that the tile's 64 KB take from HBM and 0.6 us
// of exponentials), so the chains of two streams are interleaved.  Inside a CTA:
//   * one thread per stream brings Q (per segment) and the K/V tiles with TMA into 128-byte-swizzled shared memory: a slot for
//     K, free again once the scores of its tile are complete, and one for V, free once P.V is (a barrier that two
//     consumers wait on by parity must not be shared between the streams: one could be a phase ahead of the other);
//   * one thread per stream issues tcgen05.mma: S = Q.K^T into the stream's score buffer in TMEM, then O += P.V with P read
//     from that same buffer and the accumulator resident in TMEM for the whole segment (one thread for both streams was the
//     bottleneck: 2200 cycles a tile, most of them the latency of its waits);
//   * eight warps per stream do the softmax: they read S once into registers, apply the ancestor bitmask on tiles that
//     reach the tree rows, keep an online softmax whose running maximum is only raised when a tile exceeds it by more
//     than 2^8 (then O is rescaled in TMEM), and store P as bf16 over the scores it comes from, where the second MMA reads it
//     as its A operand.
// Up to 64 tree rows (kernel of 64-row streams): stream 0 is the lower, stream 1 the upper half of the 128 TMEM lanes; each
// MMA computes all 128 lanes and the other stream's half is not looked at.  Four threads share a row, so a tree of up to 64
// rows keeps all four quarters of the SM busy.  More rows: both streams use all lanes, two threads share a row.
// A segment (a stream's consecutive units of one (sequence, head)) that covers all tiles of its (sequence, head) writes the
// normalised bf16 output itself.  Otherwise, one sequence: the head's pieces lie in the shared memory of a cluster and are
// merged there; a batch: (max, sum, O) goes to the workspace and a second kernel merges the pieces in a fixed order.
// Every wait on an mbarrier is bounded; on expiry the CTA records TRJ_ETIMEOUT and leaves.
#include <cuda.h>
#include <cstdlib>
#include <mutex>
#include "trj_internal.h"
#include "sm100_common.cuh"
#include "timeline.cuh"
#include "piece_range.h"

namespace trj {
namespace {

constexpr int AT_LANES = 128;                // UMMA M = TMEM lanes
constexpr int AT_KEYS = 128;                 // keys per tile
constexpr int AT_D = 128;                    // head_dim
constexpr int AT_STREAMS = 2;
constexpr int AT_STREAM_WARPS = 8, AT_SM_WARPS = AT_STREAMS * AT_STREAM_WARPS;      // softmax warps
constexpr int AT_W_COPY = AT_SM_WARPS, AT_W_MMA = AT_SM_WARPS + AT_STREAMS;      // a TMA warp and an MMA warp per stream
constexpr int AT_THREADS = 32 * (AT_SM_WARPS + 2 * AT_STREAMS);
constexpr uint32_t AT_SUB = 128 * 128;       // one [128 x 64 bf16] swizzled sub-tile: 16 KB
constexpr uint32_t AT_TILE = 2 * AT_SUB;     // a K tile, a V tile, 128 rows of Q: 32 KB
// Q (64-row streams: one tile, a half each; wide: a tile each), then a K slot and a V slot per stream
__host__ __device__ constexpr int at_q_tiles(bool wide) { return wide ? 2 : 1; }
__host__ __device__ constexpr uint32_t at_smem(bool wide) { return (uint32_t)(at_q_tiles(wide) + 2 * AT_STREAMS) * AT_TILE + 1024; }
constexpr float AT_RESCALE_GAP = 8.f;        // raise the running max only when exceeded by 2^8
constexpr size_t AT_SLOT_FLOATS = (size_t)AT_D * AT_LANES + 2 * AT_LANES;   // O^T [d][row], m[row], l[row]

// barrier indices, one barrier per stream each; the last two: every CTA of the cluster has reached the merge; the other CTAs'
// pieces have arrived
enum { B_K_FULL = 0, B_K_EMPTY = 2, B_V_FULL = 4, B_V_EMPTY = 6, B_Q_FULL = 8, B_Q_EMPTY = 10, B_S_FULL = 12, B_P_READY = 14, B_O_READY = 16,
       B_O_FREE = 18, B_PEERS = 20, B_RECEIVED = 21, B_COUNT = 22 };

struct AtParams {
    const int32_t* seq_len; const int32_t* row_off; const uint64_t* anc;
    int anc_words, B, H, max_seq;
    int Hkv, group;              // K/V heads and query heads per K/V head (grouped-query attention; group = 1: multi-head)
    __nv_bfloat16* out;          // [rows_total][H][128]
    __nv_bfloat16* out_lo;       // optional: rounding error of `out` as a second bf16 tensor (same shape)
    float* slots;                // partial results, AT_SLOT_FLOATS each
    int2* owners;                // batches, per (sequence, head): the first and the last stream that worked on it
    int* status;
    float scale_log2;            // log2(e) / sqrt(D)
    int cluster;                 // one sequence: CTAs per thread-block cluster that share one head; 0: a batch
    int in_chain;                // the batch geometry and the ancestor masks are older than the chain: they may be read before the wait
    int early_ok;                // cache rows below seq_len are older than the chain: they may be fetched before the wait
    int rows_cap;                // most rows of a tree that the launched kernel takes
    int streams;                 // of the whole launch (batches; see build_range)
    int shared_cache;            // every sequence of the batch uses the cache of sequence 0 (pieces of one prompt chunk)
};

using namespace sm100;

// MN-major operand (V: keys are the contraction dim, head_dim is contiguous): 64-element spans of the
// MN dim are 128-byte rows, one per key; 8-key groups 1024 bytes apart (stride offset); the second
// 64-element block of the MN dim lies one sub-tile further (leading offset).
__device__ __forceinline__ uint64_t desc_mnmajor(uint32_t addr) {
    return (uint64_t)((addr & 0x3FFFF) >> 4) | ((uint64_t)(AT_SUB >> 4) << 16) | ((uint64_t)(1024 >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}
// Eight MMAs in one go.  A single thread issues them, and its integer work per MMA is what limits the tile loop,
// so the descriptors are not rebuilt: the high words are constants and a step along the contraction dimension
// only adds to the start-address field of the low word (the operands stay inside one 256 KB window).
// S = Q.K^T for one tile: both operands K-major; step kk adds (kk / 4) sub-tiles + (kk % 4) * 32 bytes.
#define TRJ_MMA_SS(step, pred)                                                            \
    "add.u32 al, %1, " #step ";\n\tadd.u32 bl, %2, " #step ";\n\t"                        \
    "mov.b64 da, {al, %3};\n\tmov.b64 db, {bl, %3};\n\t"                                  \
    "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, " #pred ";\n\t"
__device__ __forceinline__ void umma8_qk(uint32_t tmem_d, uint32_t a_lo, uint32_t b_lo, uint32_t desc_hi, uint32_t idesc) {
    asm volatile("{\n\t.reg .pred pt, pf;\n\t.reg .b32 al, bl;\n\t.reg .b64 da, db;\n\t"
                 "setp.eq.b32 pt, 0, 0;\n\tsetp.ne.b32 pf, 0, 0;\n\t"
                 TRJ_MMA_SS(0, pf) TRJ_MMA_SS(2, pt) TRJ_MMA_SS(4, pt) TRJ_MMA_SS(6, pt)
                 TRJ_MMA_SS(1024, pt) TRJ_MMA_SS(1026, pt) TRJ_MMA_SS(1028, pt) TRJ_MMA_SS(1030, pt)
                 "}"
                 ::"r"(tmem_d), "r"(a_lo), "r"(b_lo), "r"(desc_hi), "r"(idesc) : "memory");
}
#undef TRJ_MMA_SS
// O (+)= P.V for one tile: P from tensor memory (16 keys = 8 columns per step; every 32 keys' P lies in the first columns of
// the 32 score columns it replaces), V MN-major (16 keys = 2048 bytes per step).
#define TRJ_MMA_TS(col, kk, pred)                                                         \
    "add.u32 ta, %1, " #col ";\n\tadd.u32 bl, %2, " #kk "*128;\n\t"                      \
    "mov.b64 db, {bl, %3};\n\t"                                                            \
    "tcgen05.mma.cta_group::1.kind::f16 [%0], [ta], db, %4, " #pred ";\n\t"
__device__ __forceinline__ void umma8_pv(uint32_t tmem_d, uint32_t tmem_a, uint32_t b_lo, uint32_t desc_hi, uint32_t idesc,
                                         uint32_t accumulate_first) {
    asm volatile("{\n\t.reg .pred pt, pf;\n\t.reg .b32 ta, bl;\n\t.reg .b64 db;\n\t"
                 "setp.eq.b32 pt, 0, 0;\n\tsetp.ne.b32 pf, %5, 0;\n\t"
                 TRJ_MMA_TS(0, 0, pf) TRJ_MMA_TS(8, 1, pt) TRJ_MMA_TS(32, 2, pt) TRJ_MMA_TS(40, 3, pt)
                 TRJ_MMA_TS(64, 4, pt) TRJ_MMA_TS(72, 5, pt) TRJ_MMA_TS(96, 6, pt) TRJ_MMA_TS(104, 7, pt)
                 "}"
                 ::"r"(tmem_d), "r"(tmem_a), "r"(b_lo), "r"(desc_hi), "r"(idesc), "r"(accumulate_first) : "memory");
}
#undef TRJ_MMA_TS
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float* v) {
    uint32_t r[32];
    tmem_ld32_nowait(taddr, r);
    tmem_wait_ld();
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_st16u(uint32_t taddr, const uint32_t* v) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
                 "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
                 ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
                   "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
                 : "memory");                                // no wait: pair with tmem_wait_st
}
__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);      // .x (low half) = a
    return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ float fast_exp2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float bf16_round(float a) { return __bfloat162float(__float2bfloat16_rn(a)); }
// Stores 8 consecutive outputs as bf16 (16 bytes) and, when asked, the rounding errors as a second bf16 vector.
__device__ __forceinline__ void store8_split(__nv_bfloat16* hi, __nv_bfloat16* lo, const float* v) {
    *reinterpret_cast<uint4*>(hi) = make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]), pack_bf16(v[6], v[7]));
    if (lo) {
        float r[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) r[i] = v[i] - bf16_round(v[i]);
        *reinterpret_cast<uint4*>(lo) = make_uint4(pack_bf16(r[0], r[1]), pack_bf16(r[2], r[3]), pack_bf16(r[4], r[5]), pack_bf16(r[6], r[7]));
    }
}

// Same for 4 outputs (8 bytes each).
__device__ __forceinline__ void store4_split(__nv_bfloat16* hi, __nv_bfloat16* lo, float a, float b, float c, float d) {
    *reinterpret_cast<uint2*>(hi) = make_uint2(pack_bf16(a, b), pack_bf16(c, d));
    if (lo)
        *reinterpret_cast<uint2*>(lo) = make_uint2(pack_bf16(a - bf16_round(a), b - bf16_round(b)),
                                                   pack_bf16(c - bf16_round(c), d - bf16_round(d)));
}
// 128-bit (lo, hi) shifts by 0..127 bits; the left shift fills the vacated low bits with ones.
__device__ __forceinline__ void shr128(uint64_t& lo, uint64_t& hi, int n) {
    if (n == 0) return;
    if (n < 64) { lo = (lo >> n) | (hi << (64 - n)); hi >>= n; }
    else { lo = hi >> (n - 64); hi = 0; }
}
__device__ __forceinline__ void shl128_fill(uint64_t& lo, uint64_t& hi, int n) {
    if (n == 0) return;
    if (n < 64) { hi = (hi << n) | (lo >> (64 - n)); lo = (lo << n) | ((1ull << n) - 1); }
    else { hi = (n == 64 ? lo : (lo << (n - 64)) | ((1ull << (n - 64)) - 1)); lo = ~0ull; }
}

// Where a unit index falls: sequence, head, tile, and the geometry of that sequence.
struct Where { int b, h, t, tiles, S, rows, bh; };

struct Sched {
    int B, H;
    int tiles[TRJ_MAX_BATCH];           // key tiles of each sequence
    int S[TRJ_MAX_BATCH];               // cached rows of each sequence (a copy of seq_len: no global load on the critical path)
    int row0[TRJ_MAX_BATCH + 1];        // a copy of row_off
    int first[TRJ_MAX_BATCH + 1];       // first unit of each sequence (the launcher checks that the count fits an int)
    int head;                           // one sequence: the head of this CTA's cluster; -1 for a batch
    int whole;                          // every stream takes at most one (sequence, head), whole: nothing to merge
    int u_begin[AT_STREAMS], u_end[AT_STREAMS];      // this CTA's units
    __device__ int rows(int b, int cap) const { return min(max(row0[b + 1] - row0[b], 0), cap); }
    __device__ void locate(int u, Where& w, int cap) const {
        int b = 0;
        while (b + 1 < B && u >= first[b + 1]) ++b;
        const int r = u - first[b];
        w.b = b; w.tiles = tiles[b];
        w.h = head >= 0 ? head : r / w.tiles;
        w.t = r - w.h * w.tiles;
        w.S = S[b]; w.rows = rows(b, cap);
        w.bh = b * H + w.h;
    }
};

// One thread: the tiles of every sequence from the lengths and row offsets in s.S and s.row0.
__device__ __forceinline__ void finish_sched(Sched& s, const AtParams& p) {
    s.B = p.B; s.H = p.H;
    int u = 0, longest = 0;
    for (int b = 0; b < p.B; ++b) {
        // a device-held length that breaks the caller's contract must not turn into a negative or unbounded tile
        // count: it is brought inside the cache (the tensor maps read zeros past the cache's end anyway)
        const int rows_b = s.rows(b, p.rows_cap);
        s.S[b] = min(max(s.S[b], 0), max(p.max_seq - rows_b, 0));
        s.tiles[b] = (s.S[b] + rows_b + AT_KEYS - 1) / AT_KEYS;
        longest = max(longest, s.tiles[b]);
        s.first[b] = u;
        u += s.tiles[b] * p.H;
    }
    s.first[p.B] = u;
    s.head = -1;
    // One sequence: only a head of one tile without a cluster is whole; its stream writes the output as in a batch (128 rows without a prefix:
    // 10.3 -> 8.2 us, the merge of a single piece made the difference).
    s.whole = p.cluster == 1 && longest <= 1;
    if (p.cluster > 0) return;
    // Whole heads need no merge; equal shares are shorter when a head is much longer than a share.  A merge (pieces to L2 and
    // back in the second kernel) takes about as long as six tiles.
    s.whole = p.B * p.H <= p.streams && longest <= u / p.streams + 6;
}
// A batch's schedule, by all threads of the CTA; complete after the caller's next __syncthreads.
__device__ __forceinline__ void build_batch_sched(Sched& s, const AtParams& p) {
    for (int b = threadIdx.x; b <= p.B; b += blockDim.x) s.row0[b] = p.row_off[b];
    for (int b = threadIdx.x; b < p.B; b += blockDim.x) s.S[b] = p.seq_len[b];
    __syncthreads();
    if (threadIdx.x == 0) finish_sched(s, p);
}
// The units of stream `st` of CTA `cta` (one thread per stream).  One sequence: the head's tiles are shared out among the
// streams of its cluster, rounded so that the extra tiles go to the FIRST streams: their tiles are cached rows that are
// already on their way when the previous kernel ends, while the last stream has the tile with this step's rows, the masks
// and the padding to deal with.  A batch: equal contiguous ranges of all units, or whole heads, long next to short ones when
// the lengths grow along the batch (the pieces of a prompt): stream 0 of CTA c takes head c, stream 1 the c-th from the end.
__device__ __forceinline__ void build_range(Sched& s, const AtParams& p, int cta, int st) {
    int begin = 0, end = 0;
    if (p.cluster > 0) {
        const int shift = __ffs(AT_STREAMS * p.cluster) - 1, n = 1 << shift;      // streams of a cluster: 2, 4 or 8
        const int i = (AT_STREAMS * cta + st) & (n - 1), head = (AT_STREAMS * cta) >> shift, T = s.tiles[0];
        begin = head * T + ((T * i + n - 1) >> shift);
        end = head * T + ((T * (i + 1) + n - 1) >> shift);
        s.head = head;
    } else if (s.whole) {
        const int heads = p.B * p.H, ctas = p.streams / AT_STREAMS, seg = st == 0 ? cta : heads - 1 - cta;
        if (st == 0 ? cta < heads : seg >= ctas) {
            const int b = seg / p.H, h = seg % p.H;
            begin = s.first[b] + h * s.tiles[b];
            end = begin + s.tiles[b];
        }
    } else {
        const unsigned U = s.first[p.B], n = min((unsigned)p.streams, U), i = min((unsigned)(AT_STREAMS * cta + st), n);      // every stream below n has a unit
        if (n == 0 || i == n) {
            begin = end = (int)U;
        } else if (U < (1u << 22)) {                                // n < 2^9: the products fit 32 bits, whose division is several times cheaper
            begin = (int)(U * i / n);
            end = (int)(U * (i + 1) / n);
        } else {
            begin = (int)((unsigned long long)U * i / n);
            end = (int)((unsigned long long)U * (i + 1) / n);
        }
    }
    s.u_begin[st] = begin; s.u_end[st] = end;
}

// PRECISE: the probabilities go to the second product as a bf16 pair hi + lo (lo = the rounding error of hi, stored behind
// hi), so the product sees ~16 mantissa bits of P.  A single bf16 P costs ~1e-3 of relative error in the output whatever the
// number of keys (the output of near-uniform attention is a mean of n values and the rounding errors of its n weights do
// not average out any faster than it does); inside a deep decoder that error flips the bf16 roundings of the next layers'
// K/V rows and grows with depth.
// 640 threads leave 96 registers each.  The kernel of 64-row streams fits; that of 128-row streams (two groups of 32 scores a
// thread) spills 56 bytes a thread, 68 with PRECISE.
template <bool WIDE, bool PRECISE>
__global__ void __launch_bounds__(AT_THREADS, 1) tree_attention_tc_kernel(const __grid_constant__ CUtensorMap map_q,
                                                                          const __grid_constant__ CUtensorMap map_k,
                                                                          const __grid_constant__ CUtensorMap map_v,
                                                                          const AtParams p) {
    constexpr int ROWS = WIDE ? 128 : 64;                    // rows of a stream
    constexpr int ROW_GROUPS = ROWS / 32, PARTS = AT_STREAM_WARPS / ROW_GROUPS;      // warps of 32 rows; threads that share a row
    constexpr int GROUPS = 4 / PARTS;                        // 32-key groups of a tile, and 32-column groups of O, per thread
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bars[B_COUNT];
    __shared__ uint32_t tmem_base_slot;
    __shared__ int abort_flag;
    __shared__ Sched sched;
    __shared__ float part_max[2][AT_STREAMS][PARTS][ROWS], part_sum[AT_STREAMS][PARTS][ROWS];      // [parity][stream][column group][row]
    __shared__ float piece_m[AT_STREAMS][ROWS], piece_l[AT_STREAMS][ROWS];      // this CTA's pieces of a head shared by a cluster
    __shared__ __align__(16) float2 sum_ml[ROWS], peer_ml[4][ROWS];             // (max, sum) of their sum; of every CTA's

    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* base_ptr = smem_raw + (base - smem_u32(smem_raw));
    // K slot of a stream; its V slot lies behind it
    auto kv_smem = [&](int st) { return base + (uint32_t)(at_q_tiles(WIDE) + 2 * st) * AT_TILE; };
    const uint32_t bar0 = smem_u32(&bars[0]);
    auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (p.in_chain) pdl_launch_dependents();
    TRJ_TL_DECL;
    if (threadIdx.x == 32) {                                 // have the tensor maps on their way before the first copy needs them
        prefetch_tensormap(&map_q);
        prefetch_tensormap(&map_k);
        prefetch_tensormap(&map_v);
    }
    if (threadIdx.x == 64) {
        abort_flag = 0;
        for (int i = 0; i < B_COUNT; ++i)
            mbar_init(bar(i), (i >= B_P_READY && i < B_P_READY + AT_STREAMS) || (i >= B_O_FREE && i < B_O_FREE + AT_STREAMS) ? AT_STREAM_WARPS
                              : i == B_PEERS && p.cluster > 0 ? p.cluster : 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == AT_W_MMA) tmem_alloc(smem_u32(&tmem_base_slot), 512u);
    for (int i = threadIdx.x; i < AT_STREAMS * ROWS; i += AT_THREADS) piece_m[i / ROWS][i % ROWS] = -INFINITY;       // no piece yet
    // Barriers, TMEM and the schedule are set up while the previous kernel may still run: the batch geometry is
    // older than the chain this kernel is launched in.  So are the cache rows below seq_len, which the copy thread
    // starts to fetch before it waits; everything else (q, the tree's own K/V rows) is touched after the wait.  Outside a chain
    // nothing is known of the previous kernel: all of this waits for it, and the merge kernel is let go only then.
    if (!p.in_chain) { pdl_wait(); pdl_launch_dependents(); }
    if (p.cluster > 0) {                                     // one sequence: one thread, one trip to memory
        if (threadIdx.x == 0) {
            const int first = p.row_off[0], last = p.row_off[1], len = p.seq_len[0];
            sched.row0[0] = first; sched.row0[1] = last; sched.S[0] = len;
            finish_sched(sched, p);
            for (int st = 0; st < AT_STREAMS; ++st) build_range(sched, p, blockIdx.x, st);
        }
    } else {
        build_batch_sched(sched, p);
        __syncthreads();
        if (threadIdx.x < AT_STREAMS) build_range(sched, p, blockIdx.x, threadIdx.x);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (p.cluster > 1) cluster_arrive_relaxed();             // the barriers exist (fenced above); waited for before the merge
    // Every role works out its first segment before it waits for the previous kernel (one thread's integer
    // divisions and address arithmetic take a microsecond that would otherwise sit on the critical path).
    const uint32_t tmem = tmem_base_slot;
    // TMEM columns: scores (then P) of stream 0 0-127, of stream 1 128-255; O of stream 0 256-383, of stream 1 384-511
    const uint32_t tmem_s0 = tmem, tmem_o0 = tmem + 256;
    const int n0 = sched.u_end[0] - sched.u_begin[0], n1 = sched.u_end[1] - sched.u_begin[1];      // tiles of each stream
    // Q of a stream: its own tile, or its half of the one tile (64 rows of 128 bytes into each sub-tile)
    auto q_rows_smem = [&](int st) { return WIDE ? base + st * AT_TILE : base + (uint32_t)st * 64u * 128u; };
    auto load_q = [&](int st, const Where& w) {
        mbar_expect_tx(bar(B_Q_FULL + st), ROWS * AT_D * 2);
        tma_load_2d(q_rows_smem(st), &map_q, w.h * AT_D, sched.row0[w.b], bar(B_Q_FULL + st));
        tma_load_2d(q_rows_smem(st) + AT_SUB, &map_q, w.h * AT_D + 64, sched.row0[w.b], bar(B_Q_FULL + st));
    };

    if (warp >= AT_W_COPY && warp < AT_W_MMA) {
        if (elect_one()) {
            // ------------------------------------------------ TMA producer of a stream
            const int st = warp - AT_W_COPY, n = st == 0 ? n0 : n1, u0 = sched.u_begin[st];
            bool ok = true, waited = false;                  // for the previous kernel (see above)
            const uint64_t kv_policy = l2_evict_first_policy();
            if (!p.early_ok) { pdl_wait(); waited = true; }
            Where w = {};
            int row0 = 0, seg = 0;                           // first cache row of the head; segments begun before this one
            auto load = [&](const CUtensorMap* map, int full, int empty, uint32_t dst, int g) {
                if (ok && g > 0) ok = mbar_wait(bar(empty + st), (uint32_t)(g - 1) & 1u, &abort_flag, p.status);
                if (!ok) return;
                mbar_expect_tx(bar(full + st), AT_TILE);
                tma_load_2d_hint(dst, map, 0, row0 + w.t * AT_KEYS, bar(full + st), kv_policy);
                tma_load_2d_hint(dst + AT_SUB, map, 64, row0 + w.t * AT_KEYS, bar(full + st), kv_policy);
            };
            for (int g = 0; g < n && ok; ++g) {
                const bool enter = g == 0 || w.t + 1 == w.tiles;
                if (enter) {
                    sched.locate(u0 + g, w, ROWS);
                    row0 = ((p.shared_cache ? 0 : w.b) * p.Hkv + (p.group == 1 ? w.h : w.h / p.group)) * p.max_seq;
                } else {
                    ++w.t;
                }
                // rows of this step, or a slot that is only freed once Q has arrived: bounded waits must not start while the
                // previous kernel may still run
                if (!waited && (g > 0 || (w.t + 1) * AT_KEYS > w.S)) { pdl_wait(); waited = true; }
                if (enter && g > 0) {                        // a new segment: its Q once the S products of the last one have finished
                    ok = mbar_wait(bar(B_Q_EMPTY + st), (uint32_t)(seg & 1), &abort_flag, p.status);
                    if (!ok) break;
                    ++seg;
                    load_q(st, w);                           // (the first segment's Q is requested by the MMA thread)
                }
                load(&map_k, B_K_FULL, B_K_EMPTY, kv_smem(st), g);
                load(&map_v, B_V_FULL, B_V_EMPTY, kv_smem(st) + AT_TILE, g);
            }
            if (!waited) pdl_wait();
        }
    } else if (warp >= AT_W_MMA) {
        if (elect_one()) {
            // ------------------------------------------------ MMA issuer of a stream
            // S = Q.K^T: both K-major from shared memory, 128 x 128.  O += P.V: P from TMEM, V MN-major, 128 x 128.  The products of
            // one thread run in the order of their issue, so the scores of a tile may replace the P that the product
            // before them reads.  K and V of a step are waited for before P is, so that between P and the next scores there
            // is nothing but the products themselves.
            const int st = warp - AT_W_MMA, n = st == 0 ? n0 : n1, u0 = sched.u_begin[st];
            const uint32_t idesc_qk = idesc_bf16(AT_LANES, AT_KEYS), idesc_pv = idesc_qk | (1u << 16);
            const uint32_t d = tmem_o0 + 128 * st, a = tmem_s0 + 128 * st;
            // 64-row streams: all 128 rows of the shared Q tile
            const uint64_t q_desc = desc_kmajor_sw128(WIDE ? base + st * AT_TILE : base);
            bool ok = n > 0;
            Where w = {};
            int in_seg = 0, seg = 0;                         // tiles left of the segment, this one included; segments begun before it
            if (ok) { sched.locate(u0, w, ROWS); in_seg = min(w.tiles - w.t, n); }
            pdl_wait();
            const uint64_t k_desc = desc_kmajor_sw128(kv_smem(st)), v_desc = desc_mnmajor(kv_smem(st) + AT_TILE);
            auto issue_qk = [&](bool last) {                 // 8 x 16 elements of head_dim: two sub-tiles of four steps
                umma8_qk(a, (uint32_t)q_desc, (uint32_t)k_desc, (uint32_t)(q_desc >> 32), idesc_qk);
                umma_commit(bar(B_S_FULL + st));
                umma_commit(bar(B_K_EMPTY + st));
                if (last) umma_commit(bar(B_Q_EMPTY + st));
            };
            if (ok) {
                // the first segment's Q: requested here, so that it does not queue behind the cache tiles that the copy thread
                // asks for ahead of the wait
                load_q(st, w);
                ok = mbar_wait(bar(B_K_FULL + st), 0u, &abort_flag, p.status) && mbar_wait(bar(B_Q_FULL + st), 0u, &abort_flag, p.status);
                if (ok) { tc_fence_after(); issue_qk(in_seg == 1); }
            }
            bool first = true;                               // the tile at hand is the first of its segment
            for (int g = 0; g < n && ok; ++g) {
                const bool last = --in_seg == 0, more = g + 1 < n, first_now = first;
                first = last;
                ok = mbar_wait(bar(B_V_FULL + st), (uint32_t)g & 1u, &abort_flag, p.status);
                if (ok && first_now && seg > 0) ok = mbar_wait(bar(B_O_FREE + st), (uint32_t)(seg - 1) & 1u, &abort_flag, p.status);
                if (ok && last && more) {
                    sched.locate(u0 + g + 1, w, ROWS);
                    in_seg = min(w.tiles - w.t, n - g - 1);
                    ++seg;
                    ok = mbar_wait(bar(B_Q_FULL + st), (uint32_t)seg & 1u, &abort_flag, p.status);
                }
                if (ok && more) ok = mbar_wait(bar(B_K_FULL + st), (uint32_t)(g + 1) & 1u, &abort_flag, p.status);
                if (ok) ok = mbar_wait(bar(B_P_READY + st), (uint32_t)g & 1u, &abort_flag, p.status);
                if (!ok) break;
                tc_fence_after();
                umma8_pv(d, a, (uint32_t)v_desc, (uint32_t)(v_desc >> 32), idesc_pv, first_now ? 0u : 1u);
                if constexpr (PRECISE)                       // the low halves lie 16 columns behind
                    umma8_pv(d, a + 16, (uint32_t)v_desc, (uint32_t)(v_desc >> 32), idesc_pv, 1u);
                umma_commit(bar(B_V_EMPTY + st));
                if (last) umma_commit(bar(B_O_READY + st));  // the last commit of a stream: the epilogue, and the CTA's exit, wait for it
                if (more) issue_qk(in_seg == 1);
            }
        }
    } else {
        // ------------------------------------------------ softmax + epilogue
        // A warp owns 32 rows of a stream (its TMEM lanes are 32 * (warp % 4) ..) and the 32-column groups GROUPS * part .. of the
        // scores and of O; PARTS threads share a row and exchange their maxima and sums through shared memory.
        const int lane_group = warp & 3;
        const int st = WIDE ? (warp >> 2) & 1 : lane_group >> 1, part = WIDE ? warp >> 3 : warp >> 2;
        const int rg = WIDE ? lane_group : lane_group & 1;
        const int row = rg * 32 + lane;
        const uint32_t lane_addr = (uint32_t)(lane_group * 32) << 16;
        const uint32_t scores = tmem_s0 + 128 * st + lane_addr + 32 * GROUPS * part, accum = tmem_o0 + 128 * st + lane_addr + 32 * GROUPS * part;
        const int col0 = 32 * GROUPS * part;                 // first key of a tile, first column of head_dim of this thread
        const uint32_t pair_bar = 1 + st * ROW_GROUPS + rg;  // named barrier of the warps that share 32 rows
        const int stream_thread = (part * ROW_GROUPS + rg) * 32 + lane;
        const int u_end = sched.u_end[st];
        // A warp whose wait gave up arrives where the others of its row group may already be waiting for it.
        auto leave_row_group = [&](bool in_use, int barriers) {
            for (int i = 0; in_use && i < barriers; ++i) asm volatile("bar.arrive %0, %1;" ::"r"(pair_bar), "n"(32 * PARTS) : "memory");
        };
        int g = 0, e = 0;
        bool ok = true;
        for (int u = sched.u_begin[st]; u < u_end && ok;) {
            Where w; sched.locate(u, w, ROWS);
            const int n_tiles = min(w.tiles - w.t, u_end - u);
            const int g0 = g, g1 = g + n_tiles;
            const bool live = row < w.rows;
            const bool group_live = rg * 32 < w.rows;        // the same for all warps that share the rows
            const int grow = sched.row0[w.b] + row;          // global row (valid when live)
            uint64_t m0 = 0, m1 = 0;
            if (live) {
                m0 = p.anc[(size_t)grow * p.anc_words];
                if (p.anc_words > 1) m1 = p.anc[(size_t)grow * p.anc_words + 1];
            }
            const int total = w.S + w.rows;
            float m_ref = -INFINITY, l_sum = 0.f;
            if (e == 0) { pdl_wait(); TRJ_TL_BEGIN(TRJ_TL_ATTENTION); }      // the ancestor masks above are older than the chain
            for (g = g0; g < g1; ++g) {
                const int key0 = (w.t + (g - g0)) * AT_KEYS;
                const bool edge = key0 + AT_KEYS > w.S;      // the tile reaches tree rows or the end of the keys
                // scores complete, and with them every product issued before: the last tile's P has been read, O may be touched
                ok = __all_sync(0xffffffffu, mbar_wait(bar(B_S_FULL + st), (uint32_t)(g & 1), &abort_flag, p.status));
                if (!ok) { leave_row_group(group_live, 1); break; }
                tc_fence_after();
                if (group_live) {
                    float s[32], mt = -INFINITY;
                    // bit c of (vis0, vis1) = visibility of key key0 + c for this row: tree row tt = key0 + c - S
                    // is visible if tt < 0 (prefix) or if bit tt of the row's ancestor mask is set
                    uint64_t vis0 = m0, vis1 = m1;
                    if (edge) {
                        const int d = key0 - w.S;            // -127 .. 127 on an edge tile
                        if (d >= 0) shr128(vis0, vis1, d); else shl128_fill(vis0, vis1, -d);
                    }
                    auto load_scores = [&](int grp) {        // 32 scores of this row, masked
                        tmem_ld32(scores + 32 * grp, s);
                        if (edge) {
                            const int c0 = col0 + 32 * grp;
                            const uint32_t vis = (uint32_t)((c0 < 64 ? vis0 : vis1) >> (c0 & 63));
#pragma unroll
                            for (int i = 0; i < 32; ++i) if (!((vis >> i) & 1u)) s[i] = -INFINITY;
                        }
                    };
#pragma unroll
                    for (int grp = 0; grp < GROUPS; ++grp) {
                        load_scores(grp);                    // the last group stays in registers
                        float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};      // independent chains
#pragma unroll
                        for (int i = 0; i < 32; i += 4) {
                            mx[0] = fmaxf(mx[0], s[i]); mx[1] = fmaxf(mx[1], s[i + 1]);
                            mx[2] = fmaxf(mx[2], s[i + 2]); mx[3] = fmaxf(mx[3], s[i + 3]);
                        }
                        mt = fmaxf(mt, fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])));
                    }
                    part_max[g & 1][st][part][row] = mt;
                    asm volatile("bar.sync %0, %1;" ::"r"(pair_bar), "n"(32 * PARTS) : "memory");
#pragma unroll
                    for (int q = 0; q < PARTS; ++q) mt = fmaxf(mt, part_max[g & 1][st][q][row]);
                    mt *= p.scale_log2;
                    float factor = 1.f;
                    if (live && mt > -INFINITY) {
                        if (m_ref == -INFINITY) m_ref = mt;
                        else if (mt > m_ref + AT_RESCALE_GAP) { factor = fast_exp2(m_ref - mt); m_ref = mt; }
                    }
                    if (g > g0 && __any_sync(0xffffffffu, factor != 1.f)) {
                        l_sum *= factor;
#pragma unroll 1
                        for (int c0 = 0; c0 < 32 * GROUPS; c0 += 16) {
                            uint32_t o[16];
                            tmem_ld8(accum + c0, reinterpret_cast<float*>(o));
                            tmem_ld8(accum + c0 + 8, reinterpret_cast<float*>(o) + 8);
                            tmem_wait_ld();
#pragma unroll
                            for (int i = 0; i < 16; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * factor);
                            tmem_st16u(accum + c0, o);
                            tmem_wait_st();
                        }
                    }
                    // P = 2^(s * c - m_ref) as bf16 over the scores it comes from (lane = row, one column per two keys, the low
                    // halves 16 columns behind); masked scores are -inf and give exactly 0.  Lanes without a row keep their
                    // scores: what they add up to is not looked at.
                    const float m_use = (m_ref == -INFINITY) ? 0.f : m_ref;
#pragma unroll
                    for (int k = GROUPS - 1; k >= 0; --k) {
                        if (k < GROUPS - 1) load_scores(k);
                        uint32_t hi[16], lo[16];
                        float ls[4] = {0.f, 0.f, 0.f, 0.f};  // independent partial sums
#pragma unroll
                        for (int i = 0; i < 32; i += 2) {
                            const float a = fast_exp2(fmaf(s[i], p.scale_log2, -m_use));
                            const float b = fast_exp2(fmaf(s[i + 1], p.scale_log2, -m_use));
                            ls[i & 2] += a; ls[(i & 2) + 1] += b;
                            hi[i >> 1] = pack_bf16(a, b);
                            if constexpr (PRECISE)           // what the rounding to bf16 left: the halves of a pack are the floats' upper words
                                lo[i >> 1] = pack_bf16(a - __uint_as_float(hi[i >> 1] << 16), b - __uint_as_float(hi[i >> 1] & 0xffff0000u));
                        }
                        l_sum += (ls[0] + ls[1]) + (ls[2] + ls[3]);
                        tmem_st16u(scores + 32 * k, hi);
                        if constexpr (PRECISE) tmem_st16u(scores + 32 * k + 16, lo);
                    }
                    tmem_wait_st();
                }
                // keys past the end of the sequence hold whatever the cache holds: clear those V rows so
                // that 0 * garbage cannot poison the product
                if (key0 + AT_KEYS > total) {
                    ok = __all_sync(0xffffffffu, mbar_wait(bar(B_V_FULL + st), (uint32_t)g & 1u, &abort_flag, p.status));
                    if (!ok) break;
                    uint8_t* v_ptr = base_ptr + (kv_smem(st) + AT_TILE - base);
                    const int first_bad = max(total - key0, 0);
                    for (int i = first_bad * 8 + stream_thread; i < AT_KEYS * 8; i += 32 * AT_STREAM_WARPS) {      // 16-byte chunks, both sub-tiles
                        *reinterpret_cast<uint4*>(v_ptr + i * 16) = make_uint4(0, 0, 0, 0);
                        *reinterpret_cast<uint4*>(v_ptr + AT_SUB + i * 16) = make_uint4(0, 0, 0, 0);
                    }
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");      // the MMA reads V through the async proxy
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(B_P_READY + st));
            }
            if (!ok) break;
            // ---- epilogue of the segment
            ok = __all_sync(0xffffffffu, mbar_wait(bar(B_O_READY + st), (uint32_t)(e & 1), &abort_flag, p.status));
            if (!ok) { leave_row_group(group_live, 2); break; }
            tc_fence_after();
            if (group_live) {
                part_sum[st][part][row] = l_sum;
                asm volatile("bar.sync %0, %1;" ::"r"(pair_bar), "n"(32 * PARTS) : "memory");
                float l_row = 0.f;
#pragma unroll
                for (int q = 0; q < PARTS; ++q) l_row += part_sum[st][q][row];       // the same order in every thread
                if (p.cluster > 0 && !sched.whole) {
                    // a piece of the head: O stays in TMEM until both streams are done (it goes where the ring is)
                    if (live && part == 0) { piece_m[st][row] = m_ref; piece_l[st][row] = l_row; }
                } else if (w.t == 0 && n_tiles == w.tiles) {
                    const float inv = live ? 1.f / l_row : 0.f;
                    const size_t off = ((size_t)grow * p.H + w.h) * AT_D + col0;
#pragma unroll 1
                    for (int c0 = 0; c0 < 32 * GROUPS; c0 += 32) {
                        float o[32];
                        tmem_ld32(accum + c0, o);
                        if (live) {
#pragma unroll
                            for (int i = 0; i < 32; ++i) o[i] *= inv;
#pragma unroll
                            for (int ch = 0; ch < 4; ++ch)
                                store8_split(p.out + off + c0 + 8 * ch, p.out_lo ? p.out_lo + off + c0 + 8 * ch : nullptr, o + 8 * ch);
                        }
                    }
                } else {
                    float* slot = p.slots + (size_t)(w.bh + AT_STREAMS * (int)blockIdx.x + st) * AT_SLOT_FLOATS;
#pragma unroll 1
                    for (int c0 = 0; c0 < 32 * GROUPS; c0 += 32) {
                        float o[32];
                        tmem_ld32(accum + c0, o);
                        if (live) {
#pragma unroll
                            for (int i = 0; i < 32; ++i) slot[(size_t)(col0 + c0 + i) * AT_LANES + row] = o[i];
                        }
                    }
                    if (live && part == 0) { slot[AT_D * AT_LANES + row] = m_ref; slot[AT_D * AT_LANES + AT_LANES + row] = l_row; }
                }
                // the sums are read before any warp of the row group writes the next segment's
                asm volatile("bar.sync %0, %1;" ::"r"(pair_bar), "n"(32 * PARTS) : "memory");
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(B_O_FREE + st));
            if (p.cluster == 0 && stream_thread == 0) {      // for the merge kernel
                int* const owner = reinterpret_cast<int*>(p.owners + w.bh);
                if (w.t == 0) owner[0] = AT_STREAMS * (int)blockIdx.x + st;
                if (w.t + n_tiles == w.tiles) owner[1] = AT_STREAMS * (int)blockIdx.x + st;
            }
            u += n_tiles;
            ++e;
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (abort_flag) {                                        // let copies still in flight land before the CTA leaves
        for (int i = 0; i < 64; ++i) __nanosleep(1000);
        __syncthreads();
    }
    if (p.cluster > 0 && !sched.whole) {
        // Merge of the head's pieces.  Every CTA of the cluster gets here, with or without pieces, and also after a wait that
        // gave up.  First the CTA adds up its own two pieces; then each CTA gets a quarter (half) of head_dim of every
        // other CTA's sum, by bulk copies into its shared memory, and finishes it.  (Reading all pieces of the
        // cluster with ordinary loads took 6500 cycles for 64 rows and 13000 for 128; the copies and the final sum take 2300 and
        // 4500.)
        // Layout of a piece: four slices of 32 columns, [slice][row][8 x 16 bytes], the 16-byte chunks of a row permuted by
        // row % 8 (no bank conflicts although rows are 128 bytes apart).
        const int C = p.cluster, rank = blockIdx.x % C, head = blockIdx.x / C, slices = 4 / C;
        const int rows = sched.rows(0, ROWS);
        constexpr uint32_t SLICE = ROWS * 128, PIECE = 4 * SLICE;
        const uint32_t peer_smem = base + PIECE;             // [CTA][its share of the slices]; behind the CTA's own sum
        auto at = [&](uint32_t region, int slice, int row, int chunk) {      // everything lies over Q, K and V, which are idle
            return reinterpret_cast<float4*>(base_ptr + (region - base) + slice * SLICE + row * 128 + ((chunk ^ (row & 7)) << 4));
        };
        pdl_wait();                                          // threads that had no role have not waited yet
        if (C > 1) {
            cluster_wait();                                  // every CTA's barriers have been initialised
            if (threadIdx.x < C) mbar_arrive_cluster(cluster_addr(bar(B_PEERS), threadIdx.x));      // this CTA's K and V are idle
            if (threadIdx.x == 32) mbar_expect_tx(bar(B_RECEIVED), (uint32_t)(C - 1) * (slices * rows * 128 + ROWS * (uint32_t)sizeof(float2)));
        }
        // The own sum: stream 0's warps finish slices 0 and 1, stream 1's warps 2 and 3, each from its accumulator and what the
        // other stream's warps left in shared memory.  The same lanes and columns as above.
        const int lane_group = warp & 3, st = WIDE ? (warp >> 2) & 1 : lane_group >> 1, part = WIDE ? warp >> 3 : warp >> 2;
        const int rg = WIDE ? lane_group : lane_group & 1, row = rg * 32 + lane;
        const bool role = warp < AT_SM_WARPS && rg * 32 < rows, finishes = ((GROUPS * part) >> 1) == st, has_piece = (st == 0 ? n0 : n1) > 0;
        const uint32_t accum = tmem_o0 + 128 * st + ((uint32_t)(lane_group * 32) << 16);
        if (role && !finishes && has_piece) {
#pragma unroll 1
            for (int slice = GROUPS * part; slice < GROUPS * (part + 1); ++slice) {
                float o[32];
                tmem_ld32(accum + 32 * slice, o);
                if (row < rows) {
#pragma unroll
                    for (int i = 0; i < 8; ++i) *at(base, slice, row, i) = make_float4(o[4 * i], o[4 * i + 1], o[4 * i + 2], o[4 * i + 3]);
                }
            }
        }
        __syncthreads();
        if (role && finishes) {
            float w_own = 0.f, w_other = 0.f;                // a piece without keys (maximum -inf) holds no data
            if (row < rows) {
                const float m_own = piece_m[st][row], m_other = piece_m[st ^ 1][row], m = fmaxf(m_own, m_other);
                if (m_own > -INFINITY) w_own = exp2f(m_own - m);
                if (m_other > -INFINITY) w_other = exp2f(m_other - m);
                if (part == 0)
                    sum_ml[row] = make_float2(m, (w_own > 0.f ? piece_l[st][row] * w_own : 0.f) + (w_other > 0.f ? piece_l[st ^ 1][row] * w_other : 0.f));
            }
#pragma unroll 1
            for (int slice = GROUPS * part; slice < GROUPS * (part + 1); ++slice) {
                float o[32];
                if (has_piece) tmem_ld32(accum + 32 * slice, o);
                if (row < rows) {
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (w_own > 0.f) v = make_float4(o[4 * i] * w_own, o[4 * i + 1] * w_own, o[4 * i + 2] * w_own, o[4 * i + 3] * w_own);
                        if (w_other > 0.f) {
                            const float4 a = *at(base, slice, row, i);
                            v.x = fmaf(a.x, w_other, v.x); v.y = fmaf(a.y, w_other, v.y); v.z = fmaf(a.z, w_other, v.z); v.w = fmaf(a.w, w_other, v.w);
                        }
                        *at(base, slice, row, i) = v;
                    }
                }
            }
        }
        if (C > 1) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");      // the bulk copies read what was just written
            __syncthreads();
            if (warp == 0 && mbar_wait_cluster(bar(B_PEERS), 0u, &abort_flag, p.status)) {
                const int peer = lane / slices, slice = lane % slices;
                if (peer < C && peer != rank) {
                    if (rows > 0)
                        bulk_copy_to_cluster(cluster_addr(peer_smem + (rank * slices + slice) * SLICE, peer), base + (peer * slices + slice) * SLICE,
                                             rows * 128, cluster_addr(bar(B_RECEIVED), peer));
                    if (slice == 0)
                        bulk_copy_to_cluster(cluster_addr(smem_u32(&peer_ml[rank][0]), peer), smem_u32(&sum_ml[0]), ROWS * (uint32_t)sizeof(float2),
                                             cluster_addr(bar(B_RECEIVED), peer));
                }
            }
            mbar_wait_cluster(bar(B_RECEIVED), 0u, &abort_flag, p.status);
            __syncwarp();
            cluster_arrive_relaxed();                        // this CTA has what it needs of the others: no data to order
        } else {
            __syncthreads();
        }
        for (int i = threadIdx.x; i < rows * slices * 8; i += AT_THREADS) {
            const int chunk = i & 7, slice = (i >> 3) & (slices - 1), row = (i >> 3) >> (__ffs(slices) - 1);
            float2 ml[4];
            float4 o[4];
            float m_all = -INFINITY, l_all = 0.f;
            float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int c = 0; c < 4; ++c) {                    // ascending CTAs, hence ascending tiles
                if (c >= C) continue;
                ml[c] = c == rank ? sum_ml[row] : peer_ml[c][row];
                o[c] = *at(c == rank ? base : peer_smem, c * slices + slice, row, chunk);
                m_all = fmaxf(m_all, ml[c].x);
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                if (c >= C || ml[c].x == -INFINITY) continue;
                const float wgt = exp2f(ml[c].x - m_all);
                l_all = fmaf(ml[c].y, wgt, l_all);
                acc.x = fmaf(o[c].x, wgt, acc.x); acc.y = fmaf(o[c].y, wgt, acc.y);
                acc.z = fmaf(o[c].z, wgt, acc.z); acc.w = fmaf(o[c].w, wgt, acc.w);
            }
            const float inv = 1.f / l_all;
            const size_t off = ((size_t)(sched.row0[0] + row) * p.H + head) * AT_D + (rank * slices + slice) * 32 + 4 * chunk;
            store4_split(p.out + off, p.out_lo ? p.out_lo + off : nullptr, acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv);
        }
        __syncwarp();                                        // the loop above ends at different times in a warp's lanes
        if (C > 1) cluster_wait();                           // nobody leaves while its sum may still be copied
        __syncthreads();
        if (abort_flag) {                                    // a wait above gave up: let what its peers were copying here land
            for (int i = 0; i < 64; ++i) __nanosleep(1000);
            __syncthreads();
        }
    }
    if (warp == AT_W_MMA) tmem_dealloc(tmem, 512u);
#ifdef TRJ_TIMELINE
    if (threadIdx.x == 0 && sched.u_begin[0] >= sched.u_end[0]) tl_slot__ = ::trj::tl::begin(TRJ_TL_ATTENTION);   // no work for this thread: it never stamped its release
#endif
    TRJ_TL_END(TRJ_TL_ATTENTION);
}

// Merges the pieces of every (sequence, head) that more than one stream worked on: one CTA per (sequence, head, 32-wide slice
// of head_dim), thread = row; pieces are taken in ascending stream order, two at a time so that their loads overlap.  Which
// streams those are the main kernel has left in p.owners (working the schedule out again in every CTA, with 64-bit
// divisions, took longer than the merge: a ragged batch of 8 went from 66.5 to 61.7 us, main kernel included).
constexpr int CB_COLS = 32;
__global__ void __launch_bounds__(AT_LANES) tree_attention_combine_kernel(const AtParams p) {
    extern __shared__ float cb_stage[];                      // [row][CB_COLS + 1]
    pdl_launch_dependents();
    const int bh = blockIdx.x, b = bh / p.H, h = bh % p.H, c0 = blockIdx.y * CB_COLS;
    pdl_wait();
    const int first_row = p.row_off[b], rows = min(max(p.row_off[b + 1] - first_row, 0), p.rows_cap);
    const int2 owners = p.owners[bh];
    if (rows == 0 || !pieces_to_merge(owners.x, owners.y, p.streams)) return;      // no rows, written directly by its only stream, or no record
    const int row = threadIdx.x;
    if (row < rows) {
        float m_all = -INFINITY, l_all = 0.f, acc[CB_COLS];
#pragma unroll
        for (int i = 0; i < CB_COLS; ++i) acc[i] = 0.f;
        for (int c = owners.x; c <= owners.y; c += 2) {
            float m[2], l[2], o[2][CB_COLS];
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                if (c + j > owners.y) { m[j] = -INFINITY; continue; }
                const float* slot = p.slots + (size_t)(bh + c + j) * AT_SLOT_FLOATS;
                m[j] = slot[AT_D * AT_LANES + row];
                l[j] = slot[AT_D * AT_LANES + AT_LANES + row];
#pragma unroll
                for (int i = 0; i < CB_COLS; ++i) o[j][i] = slot[(size_t)(c0 + i) * AT_LANES + row];
            }
            const float m_new = fmaxf(m_all, fmaxf(m[0], m[1]));
            if (m_new == -INFINITY) continue;                // pieces in which the row sees no key
            const float keep = exp2f(m_all - m_new);
            l_all *= keep;
#pragma unroll
            for (int i = 0; i < CB_COLS; ++i) acc[i] *= keep;
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                if (m[j] == -INFINITY) continue;
                const float wgt = exp2f(m[j] - m_new);
                l_all = fmaf(l[j], wgt, l_all);
#pragma unroll
                for (int i = 0; i < CB_COLS; ++i) acc[i] = fmaf(o[j][i], wgt, acc[i]);
            }
            m_all = m_new;
        }
        const float inv = 1.f / l_all;
#pragma unroll
        for (int i = 0; i < CB_COLS; ++i) cb_stage[row * (CB_COLS + 1) + i] = acc[i] * inv;
    }
    __syncthreads();
    // each thread stores 8 consecutive values (16 bytes) of one row
    for (int i = threadIdx.x; i < rows * (CB_COLS / 8); i += blockDim.x) {
        const int r = i / (CB_COLS / 8), q8 = i % (CB_COLS / 8) * 8;
        const size_t off = ((size_t)(first_row + r) * p.H + h) * AT_D + c0 + q8;
        store8_split(p.out + off, p.out_lo ? p.out_lo + off : nullptr, cb_stage + r * (CB_COLS + 1) + q8);
    }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn at_encode_fn() {
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* ptr = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (EncodeTiledFn)ptr;
    });
    return fn;
}
// bf16 matrix [rows][cols] row-major, boxes of [box_rows][64 cols], 128-byte swizzle, zero fill.
bool at_make_map(CUtensorMap* map, const void* base_ptr, size_t rows, size_t cols, int box_rows) {
    EncodeTiledFn fn = at_encode_fn();
    if (!fn) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
    const cuuint32_t box[2] = {64, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base_ptr), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

constexpr int AT_MAX_GRID = 148;
constexpr int AT_WHOLE_HEAD_TILES = 8;      // up to 1024 keys: heads are handled one by one when B == 1

typedef void (*AtKernel)(CUtensorMap, CUtensorMap, CUtensorMap, AtParams);
AtKernel at_kernel(bool wide, bool precise) {
    if (wide) return precise ? tree_attention_tc_kernel<true, true> : tree_attention_tc_kernel<true, false>;
    return precise ? tree_attention_tc_kernel<false, true> : tree_attention_tc_kernel<false, false>;
}
cudaError_t at_set_attributes() {
    static std::once_flag once;
    static cudaError_t err = cudaSuccess;
    std::call_once(once, [] {
        for (int i = 0; i < 4 && err == cudaSuccess; ++i)
            err = cudaFuncSetAttribute(at_kernel(i & 1, i >> 1), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)at_smem(i & 1));
    });
    return err;
}

// How many CTAs may share a head (as one thread-block cluster) when every head is handled on its own: the largest
// of 4 and 2 for which all H clusters are resident at once, else 1.  Asked of the driver once per head count.
int at_cluster_size(int H) {
    static std::mutex mu;
    static int cached_h = -1, cached_c = 1;
    std::lock_guard<std::mutex> lock(mu);
    if (cached_h == H) return cached_c;
    int pick = 1;
    if (at_set_attributes() == cudaSuccess) {
        for (int c = 4; c >= 2 && pick == 1; c /= 2) {
            if (H * c > AT_MAX_GRID) continue;
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(H * c); cfg.blockDim = dim3(AT_THREADS); cfg.dynamicSmemBytes = at_smem(true);
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = c; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr; cfg.numAttrs = 1;
            int n = 0;
            if (cudaOccupancyMaxActiveClusters(&n, at_kernel(true, true), &cfg) == cudaSuccess && n >= H) pick = c;
        }
    }
    (void)cudaGetLastError();                                // a refused query is not an error of the caller
    cached_h = H; cached_c = pick;
    return pick;
}

// Launch shape.  The host only knows an upper bound of the key count; CTAs whose range turns out empty do no work.
struct AtPlan { int grid, cluster; bool merge_kernel; };
AtPlan at_plan(int32_t B, int32_t H, int32_t max_len) {
    const int tiles_bound = (max_len + AT_KEYS - 1) / AT_KEYS;
    const long long units_bound = (long long)B * H * tiles_bound;
    // One sequence: every head on its own.  A head's tiles are shared by the CTAs of a cluster, which merge their
    // pieces through distributed shared memory: no pieces go through global memory and no merge kernel is needed.
    // Where clusters do not fit, one CTA takes a whole head of up to AT_WHOLE_HEAD_TILES tiles.
    if (B == 1 && H <= AT_MAX_GRID) {
        const int c = tiles_bound >= 2 ? at_cluster_size(H) : 1;
        if (c > 1 || tiles_bound <= AT_WHOLE_HEAD_TILES) return AtPlan{H * c, c, false};
    }
    // a batch, or heads too long for one CTA each: all SMs, split as build_range says, and the merge kernel
    return AtPlan{(int)(units_bound < AT_MAX_GRID ? units_bound : AT_MAX_GRID), 0, true};
}

}  // namespace

#ifdef TRJ_TIMELINE
cudaError_t timeline_reset_attention(cudaStream_t st) { return tl::reset(st); }
int timeline_read_attention(int kind, int max_launches, uint64_t* b, uint64_t* e) { return tl::read(kind, max_launches, b, e); }
#endif

int tree_attention_grid(int32_t B, int32_t H, int32_t max_len) { return at_plan(B, H, max_len).grid; }

bool tree_attention_tc_supported(int32_t D, int32_t dtype, int32_t max_rows) {
    return D == AT_D && dtype == TRJ_BF16 && max_rows <= AT_LANES && at_encode_fn() != nullptr;
}

// Workspace: 256-byte header (status word), the streams that worked on each (sequence, head), then one slot per possible piece: a stream's range can start a
// new (sequence, head) at most B*H times in total and each of the <= 296 streams opens at most one more.
static size_t at_owner_bytes(int32_t B, int32_t H) { return align_up(sizeof(int2) * (size_t)B * H, 256); }
size_t tree_attention_tc_workspace(int32_t B, int32_t H) {
    return 256 + at_owner_bytes(B, H) + ((size_t)B * H + AT_STREAMS * AT_MAX_GRID) * AT_SLOT_FLOATS * sizeof(float);
}

cudaError_t launch_tree_attention_tc(const void* q, const void* k_slab, const void* v_slab, const uint64_t* anc,
                                     int32_t anc_words, const Batch& bt, int32_t H, int32_t Hkv, int32_t max_seq, void* out,
                                     void* out_lo, void* workspace, cudaStream_t st, int* status) {
    const cudaError_t attr_err = at_set_attributes();
    if (attr_err != cudaSuccess) return attr_err;
    const bool wide = bt.max_rows > 64;
    CUtensorMap map_q, map_k, map_v;
    if (!at_make_map(&map_q, q, (size_t)bt.rows_total, (size_t)H * AT_D, wide ? 128 : 64) ||
        !at_make_map(&map_k, k_slab, (size_t)(bt.shared_cache ? 1 : bt.B) * Hkv * max_seq, AT_D, AT_KEYS) ||
        !at_make_map(&map_v, v_slab, (size_t)(bt.shared_cache ? 1 : bt.B) * Hkv * max_seq, AT_D, AT_KEYS))
        return cudaErrorInvalidValue;
    AtParams p;
    p.seq_len = bt.seq_len; p.row_off = bt.row_off; p.anc = anc; p.anc_words = anc_words;
    p.B = bt.B; p.H = H; p.max_seq = max_seq;
    p.Hkv = Hkv; p.group = H / Hkv;
    p.in_chain = chain_active();
    p.early_ok = p.in_chain && bt.cached_rows_final;
    p.shared_cache = bt.shared_cache;
    p.out = (__nv_bfloat16*)out;
    p.out_lo = (__nv_bfloat16*)out_lo;
    p.status = status ? status : (int*)workspace;
    p.owners = (int2*)((char*)workspace + 256);
    p.slots = (float*)((char*)workspace + 256 + at_owner_bytes(bt.B, H));
    p.scale_log2 = 1.4426950408889634f / sqrtf((float)AT_D);
    if ((long long)bt.B * H * ((bt.max_len + AT_KEYS - 1) / AT_KEYS) > 0x7fffffffLL) return cudaErrorInvalidValue;   // unit indices are ints
    const AtPlan plan = at_plan(bt.B, H, bt.max_len);
    p.cluster = plan.cluster;
    p.streams = AT_STREAMS * plan.grid;
    p.rows_cap = wide ? 128 : 64;
    count_launch();
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(plan.grid); cfg.blockDim = dim3(AT_THREADS); cfg.dynamicSmemBytes = at_smem(wide); cfg.stream = st;
    cudaLaunchAttribute attr[2];
    int n_attr = 0;
    if (pdl_enabled()) {                                     // outside a chain: set up while the previous kernel ends
        attr[n_attr].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n_attr].val.programmaticStreamSerializationAllowed = 1;
        ++n_attr;
    }
    if (plan.cluster > 1) {
        attr[n_attr].id = cudaLaunchAttributeClusterDimension;
        attr[n_attr].val.clusterDim.x = plan.cluster; attr[n_attr].val.clusterDim.y = 1; attr[n_attr].val.clusterDim.z = 1;
        ++n_attr;
    }
    cfg.attrs = attr; cfg.numAttrs = n_attr;
    // inside a decoder (the caller asks for the result as a bf16 pair) the probabilities are a bf16 pair as well
    cudaError_t e = cudaLaunchKernelEx(&cfg, at_kernel(wide, out_lo != nullptr), map_q, map_k, map_v, p);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess || !plan.merge_kernel) return e;
    count_launch();
    // the merge kernel reads nothing ahead of its wait: programmatic launch is safe outside a chain too
    e = launch_dependent(pdl_enabled(), tree_attention_combine_kernel, dim3(bt.B * H, AT_D / CB_COLS), dim3(p.rows_cap),
                         sizeof(float) * p.rows_cap * (CB_COLS + 1), st, p);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_tree_attention(const void* q, const void* k_slab, const void* v_slab, const uint64_t* anc,
                                  int32_t anc_words, const Batch& bt, int32_t H, int32_t Hkv, int32_t D, int32_t max_seq,
                                  int32_t dtype, void* out, void* out_lo, void* workspace, size_t workspace_bytes,
                                  cudaStream_t st, int* status) {
    if (D == AT_D && dtype == TRJ_BF16 && bt.max_rows <= AT_LANES) {
        if (!workspace || ((uintptr_t)workspace % 256) != 0 || workspace_bytes < tree_attention_tc_workspace(bt.B, H) ||
            !tree_attention_tc_supported(D, dtype, bt.max_rows))
            return cudaErrorInvalidValue;
        return launch_tree_attention_tc(q, k_slab, v_slab, anc, anc_words, bt, H, Hkv, max_seq, out, out_lo, workspace, st, status);
    }
    return launch_tree_attention_generic(q, k_slab, v_slab, anc, anc_words, bt, H, Hkv, D, max_seq, dtype, out, out_lo, st);
}

}  // namespace trj

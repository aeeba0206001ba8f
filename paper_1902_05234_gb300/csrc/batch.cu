// batch.cu -- many independent ECB messages, each with its own key, key size
// and direction, in ONE persistent launch driven by a device descriptor table.
//
// The paper's unit of parallelism is one AES state (section 4.1, eq (1)); a
// batch only changes which key and which buffer a state belongs to, never the
// arithmetic.  Two kernels run back to back on the caller's stream:
//
//  plan   (count, then place: one CTA per 1,024 descriptors each, up to 512)
//                    validates every descriptor (bad ones get a status and no
//                    work), orders the messages encryptions first, and writes
//                    the exclusive prefix `start[]` of their costs.  A message's
//                    cost is Nr for each pass of 32 * blocks_per_thread blocks
//                    (what one warp ciphers at a time) plus kMsgCost for its key.
//  batch  (persistent, one CTA per SM)  each direction's cost range is cut into
//                    equal segments, one per warp up to 16 * chunk_passes passes
//                    each, and into segments of 2 * chunk_passes (short ones at
//                    the end) when the batch is larger; a warp starts with the
//                    segment of its own index and takes further ones from an
//                    atomic counter.  A segment is walked message by message:
//                    the first is found by a warp-wide 32-ary search in start[],
//                    then each lane resolves one of the next 32 messages, and
//                    the warp ciphers them in turn with the next message's round
//                    keys and first blocks already on their way.
//                    The CTA's T tables are filled for encryption first and
//                    refilled once for decryption, between two CTA barriers that
//                    every warp reaches; each phase's table layout is part of the
//                    launch configuration (default R4 for both: with the keys in
//                    registers R2's rotation costs more than its smaller tables
//                    save; 5.2 GB in 4,096 messages 6.67 ms against 6.77 with R2
//                    decryption and 6.89 with R2 in both, 47 MB in 20,000 96.5
//                    against 98.3 and 101.5 us).
//
// Workspace layout (caller- or library-owned device memory, see
// aes_batch_workspace_bytes):
//   BatchHeader | uint32 order[n] | uint64 start[n+1] | PlanTile tile[<= n / 1024 + 1]
#include <cuda_runtime.h>

#include <atomic>
#include <cstddef>
#include <cstdint>
#include <map>
#include <memory>
#include <mutex>
#include <utility>

#include "aesgb.h"
#include "aes_kernels.cuh"
#include "batch_internal.h"
#include "capi_internal.h"
#include "registry.h"

namespace aesgb {

static_assert(sizeof(aes_desc) == 40, "aes_desc is 40 bytes");
static_assert(offsetof(aes_desc, nblocks) == 24 && offsetof(aes_desc, nrounds) == 32 &&
                  offsetof(aes_desc, dir) == 36,
              "aes_desc field offsets");

struct BatchHeader {
    unsigned long long total_chunks;  // chunks of chunk_blocks blocks, all messages (debug build; else 0)
    unsigned long long enc_cost;      // costs [0, enc_cost) encrypt, [enc_cost, total_cost) decrypt
    unsigned long long total_cost;
    unsigned long long next[2];       // segment counters of the two phases (zeroed by the plan)
    unsigned int chunk_blocks;
    unsigned int n_enc;               // messages at positions [0, n_enc) encrypt
};

// What one plan CTA's descriptors add up to (count kernel -> place kernel).
struct PlanTile {
    unsigned long long cost[2];  // by direction
    unsigned long long chunks;   // debug build
    unsigned int n_enc;
};

__host__ __device__ constexpr size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

size_t batch_ws_bytes(int n) {
    const size_t nn = n > 0 ? static_cast<size_t>(n) : 0;
    return align_up(sizeof(BatchHeader), 256) + align_up(4 * nn, 256) + align_up(8 * (nn + 1), 256) +
           align_up(8 * nn, 256);
}

// End of the part of the workspace that the batch kernel reads (header, order
// and start); the plan tiles come after it.
size_t batch_plan_bytes(int n) {
    return align_up(sizeof(BatchHeader), 256) + align_up(4 * static_cast<size_t>(n), 256) +
           8 * (static_cast<size_t>(n) + 1);
}

struct WsView {
    BatchHeader *hdr;
    uint32_t *order;
    unsigned long long *start;
    PlanTile *tile;
};

__host__ __device__ inline WsView ws_view(void *ws, int n) {
    const size_t nn = static_cast<size_t>(n);
    uint8_t *p = static_cast<uint8_t *>(ws);
    WsView v;
    v.hdr = reinterpret_cast<BatchHeader *>(p);
    p += align_up(sizeof(BatchHeader), 256);
    v.order = reinterpret_cast<uint32_t *>(p);
    p += align_up(4 * nn, 256);
    v.start = reinterpret_cast<unsigned long long *>(p);
    p += align_up(8 * (nn + 1), 256);
    v.tile = reinterpret_cast<PlanTile *>(p);
    return v;
}

// ---------------------------------------------------------------------------
// plan kernel
// ---------------------------------------------------------------------------
constexpr int kPlanThreads = 1024;

__device__ int check_desc(const aes_desc &d) {
    if (d.nrounds != 10 && d.nrounds != 12 && d.nrounds != 14) return AES_E_NROUNDS;
    if (d.dir != 0 && d.dir != 1) return AES_E_ARG;
    if (d.nblocks == 0) return AES_OK;
    if (!d.rk || !d.in || !d.out) return AES_E_ARG;
    if (d.nblocks > (~0ull >> 5)) return AES_E_ARG;
    const unsigned long long a = reinterpret_cast<unsigned long long>(d.in),
                             b = reinterpret_cast<unsigned long long>(d.out);
    if (((a | b) & 15ull) || (reinterpret_cast<unsigned long long>(d.rk) & 3ull)) return AES_E_ALIGN;
    const unsigned long long len = d.nblocks << 4;
    if (a != b && a < b + len && b < a + len) return AES_E_OVERLAP;
    return AES_OK;
}

constexpr int kPlanMaxCtas = 512;  // each place CTA reads every tile, one per thread
static_assert(kPlanMaxCtas <= kPlanThreads, "one tile per thread");
// The workspace ends in 8 bytes per descriptor; a CTA's tile stands for 1,024.
static_assert(sizeof(PlanTile) <= 8 * kPlanThreads, "tiles fit");

// Cost of the per-message work (finding it, its round keys) in the unit of one
// round of one pass: about half a pass.  20,000 messages of 16 B to 16 KiB with
// 2 / 6 / 12 / 20 / 30: 96.4 / 96.5 / 100.0 / 102.9 / 108.5 us.
constexpr unsigned int kMsgCost = 6;

// Cost of one message, in passes of 2^pass_shift blocks; nothing for an empty one.
__host__ __device__ inline unsigned long long msg_cost(unsigned long long nblocks, int nr, int pass_shift) {
    if (nblocks == 0) return 0ull;
    return (((nblocks - 1) >> pass_shift) + 1) * static_cast<unsigned int>(nr) + kMsgCost;
}

// log2 of the blocks of a pass, 32 * blocks_per_thread (1, 2 or 4).
inline int pass_shift(const aes_batch_cfg &c) { return 5 + c.blocks_per_thread / 2; }

struct PlanArgs {
    const aes_desc *desc;
    void *ws;
    int32_t *status;
    int n, per_cta;  // per_cta: descriptors of one CTA, a multiple of kPlanThreads
    int pass_shift;
    unsigned int chunk_blocks;
};

__device__ __forceinline__ unsigned long long warp_sum(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Sums of the threads' tiles over the CTA, into *out (shared memory, zeroed).
__device__ __forceinline__ void cta_sum(const PlanTile &t, PlanTile *out) {
    const bool lane0 = (threadIdx.x & 31) == 0;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const unsigned long long s = warp_sum(t.cost[q]);
        if (lane0 && s) atomicAdd(&out->cost[q], s);
    }
    const unsigned int e = __reduce_add_sync(0xffffffffu, t.n_enc);
    if (lane0 && e) atomicAdd(&out->n_enc, e);
#if defined(AESGB_BOUNDS_CHECK)
    const unsigned long long c = warp_sum(t.chunks);
    if (lane0 && c) atomicAdd(&out->chunks, c);
#endif
}

// One descriptor's share of its CTA's tile.  Invalid messages count as
// encryptions without work, so they sit harmlessly in the first range.
__device__ __forceinline__ PlanTile desc_tile(const aes_desc &d, int st, const PlanArgs &a) {
    const bool ok = st == AES_OK, enc = !ok || d.dir == 0;
    const unsigned long long cost = ok ? msg_cost(d.nblocks, d.nrounds, a.pass_shift) : 0ull;
    PlanTile t{};
    t.n_enc = enc;
    t.cost[0] = enc ? cost : 0ull;
    t.cost[1] = enc ? 0ull : cost;
#if defined(AESGB_BOUNDS_CHECK)
    t.chunks = ok ? (d.nblocks + a.chunk_blocks - 1) / a.chunk_blocks : 0ull;
#endif
    return t;
}

__device__ __forceinline__ void zero_tile(PlanTile *t) {
    if (threadIdx.x == 0) *t = PlanTile{};
}

// More than one CTA's worth of descriptors: what each CTA's add up to.
__global__ void __launch_bounds__(kPlanThreads, 1) batch_count_kernel(const __grid_constant__ PlanArgs a) {
    __shared__ PlanTile s_sum;
    griddep_release();
    zero_tile(&s_sum);
    __syncthreads();
    PlanTile sum{};
    const int first = blockIdx.x * a.per_cta;
    for (int i = first + static_cast<int>(threadIdx.x); i < a.n && i < first + a.per_cta; i += kPlanThreads) {
        const aes_desc d = a.desc[i];
        const PlanTile t = desc_tile(d, check_desc(d), a);
        sum.cost[0] += t.cost[0];
        sum.cost[1] += t.cost[1];
        sum.chunks += t.chunks;
        sum.n_enc += t.n_enc;
    }
    cta_sum(sum, &s_sum);
    __syncthreads();
    if (threadIdx.x == 0) ws_view(a.ws, a.n).tile[blockIdx.x] = s_sum;
}

// Statuses, partition positions and cost prefix.  Up to 1,024 descriptors this
// kernel runs alone; above, two kernels, because a decryption's place takes the
// totals of all encryptions first.  (One CTA that passes over the descriptors
// twice instead: 2,048 messages of 64 B 20.6 -> 23.6 us with their batch, 4,096
// 21.0 -> 33.2.)  A CTA starts from the tiles of the CTAs before it (with one
// CTA, from nothing: its totals come from its only scan).  Replaces one CTA that
// scanned all descriptors three times: 20,000 descriptors took 87 us.
__global__ void __launch_bounds__(kPlanThreads, 1) batch_place_kernel(const __grid_constant__ PlanArgs a) {
    __shared__ PlanTile s_all, s_before;
    __shared__ unsigned long long s_cost[2][32];
    __shared__ unsigned int s_enc[32];
    griddep_release();
    zero_tile(&s_all);
    zero_tile(&s_before);
    __syncthreads();
    const WsView v = ws_view(a.ws, a.n);
    const unsigned int lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const int first = blockIdx.x * a.per_cta;
    const bool alone = gridDim.x == 1;
    griddep_wait();  // the count kernel's tiles
    if (!alone) {
        const PlanTile t = threadIdx.x < gridDim.x ? v.tile[threadIdx.x] : PlanTile{};
        cta_sum(t, &s_all);
        cta_sum(threadIdx.x < blockIdx.x ? t : PlanTile{}, &s_before);
        __syncthreads();
    }
    // running prefixes at the first descriptor of the current 1,024
    unsigned int enc_before = s_before.n_enc;
    unsigned long long cost_before[2] = {s_before.cost[0], s_before.cost[1]};
    for (int t0 = first; t0 < a.n && t0 < first + a.per_cta; t0 += kPlanThreads) {
        const int i = t0 + static_cast<int>(threadIdx.x);
        PlanTile t{};
        if (i < a.n) {
            const aes_desc d = a.desc[i];
            const int st = check_desc(d);
            if (a.status) a.status[i] = st;
            t = desc_tile(d, st, a);
        }
        if (alone) cta_sum(t, &s_all);
        // inclusive scans over the warp, then over the warps' totals
        unsigned int e = t.n_enc;
        unsigned long long c[2] = {t.cost[0], t.cost[1]};
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned int ye = __shfl_up_sync(0xffffffffu, e, o);
            const unsigned long long y0 = __shfl_up_sync(0xffffffffu, c[0], o);
            const unsigned long long y1 = __shfl_up_sync(0xffffffffu, c[1], o);
            if (lane >= static_cast<unsigned int>(o)) {
                e += ye;
                c[0] += y0;
                c[1] += y1;
            }
        }
        if (lane == 31u) {
            s_enc[warp] = e;
            s_cost[0][warp] = c[0];
            s_cost[1][warp] = c[1];
        }
        __syncthreads();
        unsigned int te = 0;
        unsigned long long tc[2] = {0, 0};  // totals of these 1,024
        for (unsigned int w = 0; w < blockDim.x >> 5; ++w) {
            if (w == warp) {
                e += te;
                c[0] += tc[0];
                c[1] += tc[1];
            }
            te += s_enc[w];
            tc[0] += s_cost[0][w];
            tc[1] += s_cost[1][w];
        }
        const unsigned int n_enc = s_all.n_enc;
        const unsigned long long enc_cost = s_all.cost[0];
        if (i < a.n) {
            const unsigned int enc_at = enc_before + e - t.n_enc;  // encryptions before this one
            const unsigned int pos = t.n_enc ? enc_at : n_enc + (static_cast<unsigned int>(i) - enc_at);
            v.order[pos] = static_cast<uint32_t>(i);
            v.start[pos] = t.n_enc ? cost_before[0] + c[0] - t.cost[0] : enc_cost + cost_before[1] + c[1] - t.cost[1];
        }
        enc_before += te;
        cost_before[0] += tc[0];
        cost_before[1] += tc[1];
        __syncthreads();  // the warps' totals are rewritten next
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        BatchHeader h{};
        h.total_chunks = s_all.chunks;
        h.enc_cost = s_all.cost[0];
        h.total_cost = s_all.cost[0] + s_all.cost[1];
        h.chunk_blocks = a.chunk_blocks;
        h.n_enc = s_all.n_enc;
        *v.hdr = h;
        v.start[a.n] = h.total_cost;
    }
}

// ---------------------------------------------------------------------------
// batch kernel
// ---------------------------------------------------------------------------
struct BatchArgs {
    const aes_desc *desc;
    void *ws;
    int n;
    int first;  // the direction whose tables are filled ahead of the plan: kDecrypt only if no message encrypts
};

constexpr uint32_t kKeySlotBytes = 256;  // 60 words rounded up
// A message's part in a segment, as its lane resolved it.
struct __align__(16) SegEntry {
    const uint4 *in;
    uint4 *out;
    const uint32_t *rk;
    uint32_t count;  // blocks
    int nr;
};
static_assert(sizeof(SegEntry) == 32, "two 16-byte words");
// Each warp's shared memory: two key slots (current and next message) and the
// entries of one window of 32 messages, with an empty one behind the last.
constexpr uint32_t kWarpSlotBytes = 2 * kKeySlotBytes + 33 * static_cast<uint32_t>(sizeof(SegEntry));

// The segments of one direction's cost range: n_long of `len`, then the rest
// in short ones, numbered in order.
struct Segments {
    unsigned long long len, n_long, tail, n;  // tail: length of the short ones; n: how many in all
    __device__ __forceinline__ unsigned long long begin(unsigned long long i) const {
        return i < n_long ? i * len : n_long * len + (i - n_long) * tail;
    }
};

// Shared memory of the tables of a launch: the larger of its two phases'.
__host__ __device__ constexpr uint32_t batch_table_bytes(int le, int ld) {
    return table_smem_bytes(kEncrypt, le) > table_smem_bytes(kDecrypt, ld) ? table_smem_bytes(kEncrypt, le)
                                                                            : table_smem_bytes(kDecrypt, ld);
}

#if defined(AESGB_BOUNDS_CHECK)
// Debug build: every pass a warp takes sets its bit in its chunk's tag, so that
// after one launch all passes of each of the T chunks must be set and none twice
// (aes_debug_batch_coverage reads and clears the tags).  Segments are cut between
// passes, also inside a chunk.  Chunks past the array are counted in bulk.
constexpr unsigned int kTagChunks = 1u << 16;
struct ChunkTag {
    unsigned int seen[32];  // one bit per pass: a chunk has at most 1,024
    unsigned int passes;    // how many it has, written by whoever takes one
    unsigned int again;     // takings of a pass that was taken before
};
static __device__ ChunkTag g_chunk_tag[kTagChunks];
static __device__ unsigned long long g_chunk_tag_beyond;
#endif

#if defined(AESGB_BOUNDS_CHECK)
// Debug build: what the batch launches did, for aes_debug_batch_counts.
enum { kCountFills, kCountCounter, kCounts };
static __device__ unsigned long long g_batch_counts[kCounts];
#define AESGB_COUNT(WHICH) atomicAdd(&g_batch_counts[WHICH], 1ull)
#else
#define AESGB_COUNT(WHICH) ((void)0)
#endif

// Round keys of the current message held in registers for all its passes
// (4*(NR+1) words; every index is a compile-time constant once the rounds
// are unrolled, so the array stays in registers).
template <int NR> struct RegKey {
    uint32_t w[4 * (NR + 1)];
    __device__ explicit RegKey(const uint32_t *slot) {
#pragma unroll
        for (int q = 0; q < NR + 1; ++q) {
            const uint4 v = reinterpret_cast<const uint4 *>(slot)[q];
            w[4 * q] = v.x; w[4 * q + 1] = v.y; w[4 * q + 2] = v.z; w[4 * q + 3] = v.w;
        }
    }
    __device__ __forceinline__ uint32_t operator()(int i) const { return w[i]; }
};

// Round keys left in the warp's slot, read as 16-byte broadcasts: four blocks
// per thread leave no registers for them, and share each read four ways.
template <int NR> struct SlotKey {
    const uint4 *q;
    __device__ explicit SlotKey(const uint32_t *slot) : q(reinterpret_cast<const uint4 *>(slot)) {}
    __device__ __forceinline__ uint32_t operator()(int i) const {
        const uint4 v = q[i >> 2];
        return (i & 3) == 0 ? v.x : (i & 3) == 1 ? v.y : (i & 3) == 2 ? v.z : v.w;
    }
};
template <int NR, int NB> struct BatchKey { using type = RegKey<NR>; };
template <int NR> struct BatchKey<NR, 4> { using type = SlotKey<NR>; };

// A lane's blocks of one pass: every 32nd of the `left` blocks that start at
// its own (which is there if left > 0), zeros past the end.
template <int NB> __device__ __forceinline__ void load_pass(const uint4 *in, int left, uint4 (&x)[NB]) {
#pragma unroll
    for (int i = 0; i < NB; ++i) x[i] = left > 32 * i ? ld_block(in + 32 * i) : make_uint4(0, 0, 0, 0);
}

// One entry's blocks, as passes of 32*NB blocks per warp with the next pass
// prefetched: behind the last pass, the first of the entry that follows (empty
// at the end of a window).  cur holds the first pass on entry and the next
// entry's first on return.  The next pass's address is chosen first and then
// loaded once: a load on each of two paths makes the warp wait for it where the
// paths meet, and large messages ran 8 % slower.
template <int DIR, int NR, int NB, int LAYOUT>
__device__ __forceinline__ void batch_entry(const Tab<LAYOUT, DIR> &tab, const uint32_t *kslot, const SegEntry *e,
                                            uint32_t lane, uint4 (&cur)[NB]) {
    constexpr int kPass = 32 * NB;
    const typename BatchKey<NR, NB>::type key(kslot);
    const uint4 *in = e->in + lane;
    uint4 *out = e->out + lane;
    const uint4 *next_in = e[1].in + lane;
    const int next_count = static_cast<int>(e[1].count);
#pragma unroll 1  // two passes per iteration measured 25 % slower (registers, instruction cache)
    for (int left = static_cast<int>(e->count); left > 0; left -= kPass) {
        in += kPass;
        const uint4 *src = in;
        int more = left - kPass;
        if (more <= 0) {
            src = next_in;
            more = next_count;
        }
        uint4 nxt[NB];
        load_pass<NB>(src, more - static_cast<int>(lane), nxt);
        uint32_t s[NB][4];
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            s[i][0] = cur[i].x; s[i][1] = cur[i].y; s[i][2] = cur[i].z; s[i][3] = cur[i].w;
        }
        cipher_states<DIR, NR, NB>(tab, key, s);
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            if (left - static_cast<int>(lane) > 32 * i)
                st_block(out + 32 * i, make_uint4(s[i][0], s[i][1], s[i][2], s[i][3]));
            cur[i] = nxt[i];
        }
        out += kPass;
    }
}

// Copy of one message's round keys into a key slot, in application order, by
// asynchronous 4-byte copies (schedules are 4-byte aligned): lanes never wait
// for them here.
template <int DIR>
__device__ __forceinline__ void prefetch_keys(uint32_t *slot, const uint32_t *rk, int nr, uint32_t lane) {
    for (int i = static_cast<int>(lane); i < 4 * (nr + 1); i += 32) {
        const int step = i >> 2;
        const int src = DIR == kEncrypt ? step : nr - step;
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                         static_cast<uint32_t>(__cvta_generic_to_shared(slot + i))),
                     "l"(rk + 4 * src + (i & 3))
                     : "memory");
    }
}
__device__ __forceinline__ void wait_keys() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// ceil(x / nr) for the three round counts, as multiplications.
__device__ __forceinline__ unsigned long long ceil_div_nr(unsigned long long x, int nr) {
    return nr == 10 ? (x + 9) / 10 : nr == 12 ? (x + 11) / 12 : (x + 13) / 14;
}

// Partition position q of the message that owns cost c: the largest q in
// [lo, n) with start[q] <= c.  32-ary search by the whole warp: each lane
// probes one of 31 evenly spaced positions per step.
__device__ __forceinline__ int find_message(const unsigned long long *start, int lo, int n,
                                            unsigned long long c, uint32_t lane) {
    int hi = n;
    while (hi - lo > 1) {
        const int step = (hi - lo + 31) / 32;
        const int q = lo + static_cast<int>(lane + 1) * step;
        const bool le = q < hi && start[q] <= c;
        const int k = __popc(__ballot_sync(0xffffffffu, le));
        const int nlo = lo + k * step;
        const int nhi = lo + (k + 1) * step;
        lo = nlo;
        hi = nhi < hi ? nhi : hi;
    }
    return lo;
}

#if defined(AESGB_BOUNDS_CHECK)
// Debug build: tag passes [j0, j1) of message `pos`, which has `passes`.  The
// chunks before the message's are counted over the partition.
__device__ inline void tag_passes(const BatchArgs &a, const WsView &v, int pos, unsigned long long j0,
                                  unsigned long long j1, unsigned long long passes, unsigned int pass_blocks) {
    const unsigned int cb = v.hdr->chunk_blocks, cp = cb / pass_blocks;
    unsigned long long before = 0;
    for (int q = 0; q < pos; ++q)
        if (v.start[q + 1] > v.start[q]) before += (a.desc[v.order[q]].nblocks + cb - 1) / cb;
    for (unsigned long long j = j0; j < j1; ++j) {
        const unsigned long long k = j / cp, c = before + k;
        const unsigned int bit = static_cast<unsigned int>(j % cp);
        if (c >= kTagChunks) {
            if (bit == 0) atomicAdd(&g_chunk_tag_beyond, 1ull);
            continue;
        }
        ChunkTag &t = g_chunk_tag[c];
        t.passes = static_cast<unsigned int>(passes - k * cp < cp ? passes - k * cp : cp);
        if (atomicOr(&t.seen[bit >> 5], 1u << (bit & 31)) >> (bit & 31) & 1u) atomicAdd(&t.again, 1u);
    }
}
#endif

// One direction's cost range [c_begin, c_end), messages at positions
// [p_begin, p_end).  It is cut into segments of `seg`; warp w of W starts with
// segment w, and where there are more than W takes its further ones from the
// counter (the next index is requested before the current segment is walked, so
// the atomic's latency is hidden).  A pass belongs to the segment that its
// first unit of cost lies in.
template <int DIR, int NB, int LAYOUT>
__device__ void batch_phase(const BatchArgs &a, const WsView &v, uint8_t *smem, uint8_t *wslot, unsigned int w,
                            unsigned int W, unsigned long long c_begin, unsigned long long c_end, int p_begin,
                            int p_end, const Segments &seg) {
    const uint32_t lane = threadIdx.x & 31u;
    const Tab<LAYOUT, DIR> tab(smem, lane);
    constexpr unsigned int kPass = 32u * NB;
    // the warp's slots lie inside the launch's shared memory
    if (!AESGB_CHECK(static_cast<uint32_t>(wslot - smem) + kWarpSlotBytes <= dyn_smem_bytes())) return;
    SegEntry *entries = reinterpret_cast<SegEntry *>(wslot + 2 * kKeySlotBytes);
    int p = p_begin;  // no message before it is of use to this warp any more
    unsigned long long rel = w;
    while (rel < seg.n) {
        unsigned long long ticket = 0;
        if (seg.n > W && lane == 0) ticket = atomicAdd(&v.hdr->next[DIR], 1ull);
        if (rel >= W && lane == 0) AESGB_COUNT(kCountCounter);
        const unsigned long long lo = c_begin + seg.begin(rel), stop = c_begin + seg.begin(rel + 1);
        const unsigned long long hi = stop < c_end ? stop : c_end;
        p = find_message(v.start, p, p_end, lo, lane);
        for (int p0 = p;;) {
            // lane: message p0 + lane, its passes [j0, j1) inside [lo, hi)
            const int pos = p0 + static_cast<int>(lane);
            unsigned long long s0 = ~0ull;
            SegEntry e{};
            bool take = false;
            if (pos < p_end) {
                s0 = v.start[pos];
                take = s0 < hi && v.start[pos + 1] > s0;  // in the segment, and neither empty nor invalid
                take = take && AESGB_CHECK(pos >= 0 && v.order[pos] < static_cast<uint32_t>(a.n));
            }
            if (take) {
                const aes_desc d = a.desc[v.order[pos]];
                const unsigned long long passes = (d.nblocks + kPass - 1) / kPass;
                const unsigned long long j0 = s0 < lo ? ceil_div_nr(lo - s0, d.nrounds) : 0ull;
                const unsigned long long j1 =
                    hi - s0 >= passes * static_cast<unsigned int>(d.nrounds) ? passes : ceil_div_nr(hi - s0, d.nrounds);
                const unsigned long long first = j0 * kPass;
                const unsigned long long end = j1 * kPass < d.nblocks ? j1 * kPass : d.nblocks;
                take = j0 < j1;
                take = take && AESGB_CHECK(d.dir == DIR && end <= d.nblocks && first < end &&
                                           end - first <= seg.len * kPass);
                e.in = reinterpret_cast<const uint4 *>(d.in) + first;
                e.out = reinterpret_cast<uint4 *>(d.out) + first;
                e.rk = d.rk;
                e.count = static_cast<uint32_t>(end - first);
                e.nr = d.nrounds;
#if defined(AESGB_BOUNDS_CHECK)
                if (take) tag_passes(a, v, pos, j0, j1, passes, kPass);
#endif
            }
            const unsigned int taken = __ballot_sync(0xffffffffu, take);
            const unsigned long long last = __shfl_sync(0xffffffffu, s0, 31);  // start of the window's last message
            const bool more = last < hi;
            __syncwarp();  // every lane is done with the entries and key slots of the last window
            const int k = __popc(taken);
            if (take) entries[__popc(taken & ((1u << lane) - 1u))] = e;
            if (lane == 0) entries[k] = SegEntry{};
            __syncwarp();
            uint4 cur[NB];
            if (k > 0) {
                load_pass<NB>(entries[0].in + lane, static_cast<int>(entries[0].count - lane), cur);
                prefetch_keys<DIR>(reinterpret_cast<uint32_t *>(wslot), entries[0].rk, entries[0].nr, lane);
            }
            for (int i = 0; i < k; ++i) {
                const SegEntry *now = entries + i;
                const uint32_t *kslot = reinterpret_cast<const uint32_t *>(wslot + (i & 1) * kKeySlotBytes);
                wait_keys();
                __syncwarp();  // all lanes' key words are there, and all are done with the other slot
                if (i + 1 < k)
                    prefetch_keys<DIR>(reinterpret_cast<uint32_t *>(wslot + ((i + 1) & 1) * kKeySlotBytes), now[1].rk,
                                       now[1].nr, lane);
                switch (now->nr) {
                case 10: batch_entry<DIR, 10, NB, LAYOUT>(tab, kslot, now, lane, cur); break;
                case 12: batch_entry<DIR, 12, NB, LAYOUT>(tab, kslot, now, lane, cur); break;
                default: batch_entry<DIR, 14, NB, LAYOUT>(tab, kslot, now, lane, cur); break;
                }
            }
            if (!more) break;
            p0 += 32;
            // After a window without work, straight to the message that owns the
            // cost its last one starts at: a run of empty or invalid messages owns
            // none, and 20,000 of them in a warp's share took 155 us in windows.
            if (k == 0) {
                const int owner = find_message(v.start, p0 - 1, p_end, last, lane);
                if (owner > p0) p0 = owner;
            }
        }
        if (seg.n <= W) break;
        rel = W + __shfl_sync(0xffffffffu, ticket, 0);
    }
}

// Segments of a direction of total cost c on W warps: one equal share for each
// warp while that is at most 8 * `most`; above, long ones of `most` and at the
// end (an eighth of the whole, at most half a long one per warp) short ones, so
// that the counter evens out the end.  A few long segments per warp are the
// worst of both: a warp that takes one more than the others ends late.  Equal
// shares up to 1, 4, 8, 16 * most: 4,096 messages of up to 1 MiB 587 / 530 / 531
// / 531 us, 1,000 of up to 4 MiB 522 / 472 / 472 / 472, 2,000 of them through the
// server 1,259 / 1,198 / 1,196 / 1,200.  Equal shares at every size instead lose
// where SMs do not keep the same pace for milliseconds: 5.0 GB in 4,096 messages
// 6,766 us from the counter and 6,830 in shares, 2.6 GB in 300 3,423 and 3,446,
// 2.9 GB of decryption in 20 3,830 and 3,865, two streams of 2.6 GB 7,035 and
// 7,105; one message of 1 GiB 1,601 and 1,597, of 5 GiB 6,867 and 6,875.
__device__ __forceinline__ Segments cut(unsigned long long c, unsigned int W, unsigned int most) {
    Segments s;
    const unsigned long long share = (c + W - 1) / W;
    if (share <= 8ull * most) {
        s.len = s.tail = share > 14 ? share : 14;  // at least a pass
        s.n = s.n_long = (c + s.len - 1) / s.len;
        return s;
    }
    s.len = most;
    s.tail = most / 8 > 14 ? most / 8 : 14;
    const unsigned long long end = c / 8 < W * 1ull * most / 2 ? c / 8 : W * 1ull * most / 2;
    s.n_long = (c - end) / s.len;
    s.n = s.n_long + (c - s.n_long * s.len + s.tail - 1) / s.tail;
    return s;
}

template <int LAYOUT, int DIR> __device__ __forceinline__ void fill_tables(uint8_t *smem) {
    Tab<LAYOUT, DIR>::fill(smem, threadIdx.x, blockDim.x);
    if (threadIdx.x == 0) AESGB_COUNT(kCountFills);
}

constexpr int kBatchMaxThreads = 512;  // up to 128 registers: round keys live in registers

// LE, LD: table layouts of the encryption and decryption phases.
//
// Bound: the L1TEX data pipe (the lookups) for large batches, 93-96 % busy; with
// small messages the latencies in front of each one (its descriptor, keys and
// first blocks), which is why the next message's are always under way, and why
// a batch that gives a warp up to 16 chunks is cut into equal shares instead of
// whole chunks.  Against one chunk of one message at a time, found by
// a search each, behind a one-CTA plan (replayed graph, plan and kernel): 20,000
// messages of 16 B to 16 KiB 221 -> 92.6 us, 2,000 of them 70 -> 25.6, 20 of them
// 26 -> 8.5; 4,096 of up to 1 MiB 582 -> 539, 2,000 of up to 4 MiB 1,057 -> 1,035
// (745 MiB); 4,096 of up to 16 MiB the same within 0.4 %, decryption alone 0.3 %
// slower, and one decryption of 5 GiB 1.2 % (R4 tables).  A batch without work, the
// plan and an idle kernel: 4.2 us with one descriptor, 6.9 with 1,024, 9.0 with
// 1,025, 9.3 with 20,000, 10.0 with 100,000.  With 512 threads and the 44 to 60 key words in registers a
// thread has one block in flight; two measured 20 % slower.
template <int NB, int LE, int LD>
__global__ void __launch_bounds__(kBatchMaxThreads, 1) batch_kernel(const __grid_constant__ BatchArgs a) {
    extern __shared__ __align__(128) uint8_t smem[];
    const WsView v = ws_view(a.ws, a.n);
    uint8_t *wslot = smem + batch_table_bytes(LE, LD) + (threadIdx.x >> 5) * kWarpSlotBytes;
    // launched behind the plan (programmatic dependent launch): the first fill
    // reads only constant tables and runs while the plan does
    if (a.first == kEncrypt) fill_tables<LE, kEncrypt>(smem);
    else fill_tables<LD, kDecrypt>(smem);
    griddep_wait();
    __syncthreads();
    const unsigned long long E = v.hdr->enc_cost, T = v.hdr->total_cost;
    // a long segment: twice chunk_passes passes of the middle key size
    const unsigned int most = v.hdr->chunk_blocks / (32u * NB) * 24u, G = gridDim.x, W = G * (blockDim.x >> 5);
    const int n_enc = static_cast<int>(v.hdr->n_enc);
    // Warps are numbered across the CTAs first, so that few segments spread
    // over the SMs; from the other end for decryption, so that two small
    // directions run side by side.  A CTA without a segment skips the phase.
    const unsigned int row = (threadIdx.x >> 5) * G, back = G - 1 - blockIdx.x;
    const Segments se = cut(E, W, most), sd = cut(T - E, W, most);
    if (blockIdx.x < se.n) batch_phase<kEncrypt, NB, LE>(a, v, smem, wslot, row + blockIdx.x, W, 0, E, 0, n_enc, se);
    if (back < sd.n) {
        if (a.first == kEncrypt) {
            __syncthreads();  // every warp is done with the encryption tables
            fill_tables<LD, kDecrypt>(smem);
            __syncthreads();
        }
        batch_phase<kDecrypt, NB, LD>(a, v, smem, wslot, row + back, W, E, T, n_enc, a.n, sd);
    }
}

AESGB_BOUNDS_READER(batch)

uint32_t batch_smem_bytes(const aes_batch_cfg &c) {
    return batch_table_bytes(c.layout_enc, c.layout_dec) + static_cast<uint32_t>(c.threads / 32) * kWarpSlotBytes;
}

// The compiled (blocks per thread, encryption layout, decryption layout)
// combinations: the pairs R4 / R4 (the default) and R4 / R2 at 1, 2 and 4 blocks
// per thread, and the pairs R2 / R2 and R1 / R1 at 1 and 2 (the tuner's range).
const void *batch_kernel_ptr(int nb, int le, int ld) {
#define AESGB_BK(NB, LE, LD) \
    if (nb == NB && le == LE && ld == LD) return reinterpret_cast<const void *>(&batch_kernel<NB, LE, LD>);
    AESGB_BK(1, kLayoutR4, kLayoutR2) AESGB_BK(2, kLayoutR4, kLayoutR2) AESGB_BK(4, kLayoutR4, kLayoutR2)
    AESGB_BK(1, kLayoutR4, kLayoutR4) AESGB_BK(2, kLayoutR4, kLayoutR4) AESGB_BK(4, kLayoutR4, kLayoutR4)
    AESGB_BK(1, kLayoutR2, kLayoutR2) AESGB_BK(2, kLayoutR2, kLayoutR2)
    AESGB_BK(1, kLayoutR1, kLayoutR1) AESGB_BK(2, kLayoutR1, kLayoutR1)
#undef AESGB_BK
    return nullptr;
}

int validate_batch_cfg(const aes_batch_cfg &c) {
    if (c.blocks_per_thread != 1 && c.blocks_per_thread != 2 && c.blocks_per_thread != 4) return AES_E_CONFIG;
    if (c.threads < 32 || c.threads % 32 || c.threads > kBatchMaxThreads) return AES_E_CONFIG;
    if (c.chunk_passes < 1 || c.chunk_passes > 1024) return AES_E_CONFIG;
    if (c.ctas_per_sm < 0 || c.ctas_per_sm > 1) return AES_E_CONFIG;
    if (!batch_kernel_ptr(c.blocks_per_thread, c.layout_enc, c.layout_dec)) return AES_E_CONFIG;
    return AES_OK;
}

unsigned int batch_chunk_blocks(const aes_batch_cfg &c) {
    return static_cast<unsigned int>(32 * c.blocks_per_thread * c.chunk_passes);
}

// The persistent kernel on a planned workspace; the plan is the kernel (or the
// copy) before it in the stream.
int launch_batch_kernel(const aes_desc *desc, int n, void *ws, const aes_batch_cfg &c, int first, int dev,
                        cudaStream_t s) {
    const void *fn = batch_kernel_ptr(c.blocks_per_thread, c.layout_enc, c.layout_dec);
    const uint32_t smem = batch_smem_bytes(c);
    const int st = ensure_smem_attr(fn, dev, smem);
    if (st != AES_OK) return st;
    const int sms = sm_count(dev);
    if (sms < 0) return sms;
    BatchArgs args{desc, ws, n, first};
    void *params[] = {&args};
    return launch_pdl(fn, sms, c.threads, smem, params, s);
}

int enqueue_batch(const aes_desc *desc, int n, void *ws, size_t ws_bytes, int32_t *status,
                  const aes_batch_cfg &c, cudaStream_t s) {
    if (n == 0) return AES_OK;
    if (n > AES_BATCH_MAX_DESCS) return AES_E_RANGE;  // keeps the kernels' int indices far from overflow
    if (!desc || !ws) return AES_E_ARG;
    if (ws_bytes < batch_ws_bytes(n)) return AES_E_RANGE;
    if (reinterpret_cast<uintptr_t>(ws) & 255u) return AES_E_ALIGN;
    int st = validate_batch_cfg(c);
    if (st != AES_OK) return st;
    int dev = 0;
    if (current_device(&dev) != AES_OK) return AES_E_CUDA;
    PlanArgs pa;
    pa.desc = desc;
    pa.ws = ws;
    pa.status = status;
    pa.n = n;
    pa.pass_shift = pass_shift(c);
    pa.chunk_blocks = batch_chunk_blocks(c);
    const int tiles = (n + kPlanThreads - 1) / kPlanThreads, per = (tiles + kPlanMaxCtas - 1) / kPlanMaxCtas;
    pa.per_cta = per * kPlanThreads;
    const int ctas = (tiles + per - 1) / per;
    void *params[] = {&pa};
    if (ctas > 1) {
        batch_count_kernel<<<ctas, kPlanThreads, 0, s>>>(pa);
        if (cudaGetLastError() != cudaSuccess) return AES_E_CUDA;
        st = launch_pdl(reinterpret_cast<const void *>(&batch_place_kernel), ctas, kPlanThreads, 0, params, s);
        if (st != AES_OK) return st;
    } else {
        // one thread per descriptor: fewer warps to start and to scan over
        batch_place_kernel<<<1, (n + 31) / 32 * 32, 0, s>>>(pa);
        if (cudaGetLastError() != cudaSuccess) return AES_E_CUDA;
    }
    return launch_batch_kernel(desc, n, ws, c, kEncrypt, dev, s);
}

// ---------------------------------------------------------------------------
// host-side planning (for callers that know their batch: the server)
// ---------------------------------------------------------------------------
// Writes into a HOST buffer of batch_plan_bytes(n) bytes what the plan kernels
// would write into that part of the workspace for these descriptors, which must
// all be valid (check_desc): encryptions first in input order, then decryptions;
// start[] the exclusive prefix of the costs; counters 0 (and no chunk total).
// Returns how many messages encrypt.
int plan_on_host(const aes_desc *desc, int n, const aes_batch_cfg &c, void *ws_host) {
    const WsView v = ws_view(ws_host, n);
    const int shift = pass_shift(c);
    BatchHeader h{};
    unsigned long long run = 0;
    int pos = 0;
    for (int dir = 0; dir < 2; ++dir) {
        for (int i = 0; i < n; ++i)
            if (desc[i].dir == dir) {
                v.order[pos] = static_cast<uint32_t>(i);
                v.start[pos] = run;
                run += msg_cost(desc[i].nblocks, desc[i].nrounds, shift);
                ++pos;
            }
        if (dir == 0) {
            h.n_enc = static_cast<unsigned int>(pos);
            h.enc_cost = run;
        }
    }
    v.start[n] = run;
    h.total_cost = run;
    h.chunk_blocks = batch_chunk_blocks(c);
    *v.hdr = h;
    return static_cast<int>(h.n_enc);
}

// The persistent batch kernel alone, on a workspace planned already, of whose
// messages n_enc encrypt.  No kernel runs before it that a fill could hide
// behind, so a batch that only decrypts fills no encryption tables.
int enqueue_batch_kernel(const aes_desc *desc, int n, int n_enc, void *ws, const aes_batch_cfg &c, cudaStream_t s) {
    if (n == 0) return AES_OK;
    if (n > AES_BATCH_MAX_DESCS) return AES_E_RANGE;
    int st = validate_batch_cfg(c);
    if (st != AES_OK) return st;
    int dev = 0;
    if (current_device(&dev) != AES_OK) return AES_E_CUDA;
    return launch_batch_kernel(desc, n, ws, c, n_enc > 0 ? kEncrypt : kDecrypt, dev, s);
}

// ---------------------------------------------------------------------------
// library-owned workspaces for aes_ecb_batch: one per (device, stream)
// ---------------------------------------------------------------------------
// A stream is named by its CUDA stream id (cudaStreamGetId), which is unique
// for the process's lifetime and tells apart the per-thread default streams
// that share one handle value.  Work on one stream runs in order, so a
// workspace reused by the next call on the same stream is never in use by
// another batch; calls on different streams never share one.  Growth is
// stream-ordered: the old buffer goes back with cudaFreeAsync behind the
// batches already enqueued on that stream, the new one comes from
// cudaMallocAsync, and neither waits for the device.  A context's mutex is
// held from the size check to the end of the enqueue, so no thread can free a
// buffer that another thread has looked up but not yet enqueued.
namespace {
struct StreamWs {
    std::mutex mu;
    void *ptr = nullptr;
    size_t bytes = 0;
    int dev = 0;
    cudaEvent_t last = nullptr;  // recorded after the newest batch that uses ptr
    std::atomic<int> users{0};   // callers that looked it up and have not finished (never evicted then)
};
using WsKey = std::pair<int, unsigned long long>;  // device, stream id
std::mutex g_ws_mu;
std::map<WsKey, std::shared_ptr<StreamWs>> g_ws;
// Above this many contexts, idle ones (last batch complete) are released
// when a new one is made: streams the caller destroyed leave contexts behind.
constexpr size_t kMaxStreamWs = 64;

// Release the device memory of contexts other than `keep` whose last batch
// has completed (g_ws_mu held).  The memory is idle, so it goes back in the
// order of stream s without waiting for anything.
void evict_idle_locked(const StreamWs *keep, cudaStream_t s) {
    for (auto it = g_ws.begin(); it != g_ws.end() && g_ws.size() > kMaxStreamWs;) {
        StreamWs &w = *it->second;
        std::unique_lock<std::mutex> lk(w.mu, std::try_to_lock);
        const bool idle = &w != keep && w.users.load() == 0 && lk.owns_lock() &&
                          (w.last == nullptr || cudaEventQuery(w.last) == cudaSuccess);
        (void)cudaGetLastError();
        if (!idle) {
            ++it;
            continue;
        }
        if (w.ptr) (void)cudaFreeAsync(w.ptr, s);
        if (w.last) (void)cudaEventDestroy(w.last);
        w.ptr = nullptr;
        w.bytes = 0;
        w.last = nullptr;
        lk.unlock();
        it = g_ws.erase(it);
    }
    (void)cudaGetLastError();
}
}  // namespace

// The context of (dev, stream s), created on first use.  Its user count is
// raised here, under the map's mutex, so eviction (also under it) never takes
// a context that a caller is about to lock; the caller lowers it when done.
int stream_workspace(int dev, cudaStream_t s, std::shared_ptr<StreamWs> *out) {
    unsigned long long id = 0;
    if (cudaStreamGetId(s, &id) != cudaSuccess) {
        (void)cudaGetLastError();
        return AES_E_CUDA;
    }
    std::lock_guard<std::mutex> lk(g_ws_mu);
    std::shared_ptr<StreamWs> &slot = g_ws[WsKey{dev, id}];
    if (!slot) {
        slot = std::make_shared<StreamWs>();
        slot->dev = dev;
    }
    *out = slot;  // (evict_idle_locked keeps this entry, so the reference stays valid)
    (*out)->users.fetch_add(1);
    if (g_ws.size() > kMaxStreamWs) evict_idle_locked(out->get(), s);
    return AES_OK;
}

// Enqueue the batch on s with the context's workspace, grown first if it is
// smaller than `need` (w.mu held by the caller).
int enqueue_with_stream_ws(StreamWs &w, const aes_desc *desc, int n, size_t need, int32_t *status,
                           cudaStream_t s) {
    if (w.bytes < need) {
        const size_t sz = need < (1u << 20) ? (1u << 20) : need * 2;
        void *p = nullptr;
        const int st = lib_malloc_device_async(&p, sz, s);
        if (st != AES_OK) return st;  // the old workspace stays as it was
        if (w.ptr) (void)cudaFreeAsync(w.ptr, s);
        w.ptr = p;
        w.bytes = sz;
    }
    if (!w.last && cudaEventCreateWithFlags(&w.last, cudaEventDisableTiming) != cudaSuccess) {
        (void)cudaGetLastError();
        w.last = nullptr;
        return AES_E_CUDA;
    }
    const int st = enqueue_batch(desc, n, w.ptr, w.bytes, status, batch_cfg_for(n), s);
    if (st != AES_OK) return st;
    if (cudaEventRecord(w.last, s) != cudaSuccess) {
        (void)cudaGetLastError();
        return AES_E_CUDA;
    }
    return AES_OK;
}

void batch_shutdown() {
    std::map<WsKey, std::shared_ptr<StreamWs>> all;
    {
        std::lock_guard<std::mutex> lk(g_ws_mu);
        all.swap(g_ws);
    }
    int cur = 0;
    const bool have_cur = cudaGetDevice(&cur) == cudaSuccess;
    for (auto &kv : all) {
        StreamWs &w = *kv.second;
        std::lock_guard<std::mutex> lk(w.mu);
        if (w.ptr || w.last) (void)cudaSetDevice(w.dev);
        if (w.ptr) (void)cudaFree(w.ptr);  // no library work is in flight (aes_shutdown's contract)
        if (w.last) (void)cudaEventDestroy(w.last);
        w.ptr = nullptr;
        w.bytes = 0;
        w.last = nullptr;
    }
    if (have_cur) (void)cudaSetDevice(cur);
    (void)cudaGetLastError();
}

// ---------------------------------------------------------------------------
// graph: plan + batch captured once, replayed many times
// ---------------------------------------------------------------------------
struct BatchGraph {
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
};

// ---------------------------------------------------------------------------
// Batch scratch in a file-scope device array, for callers that cannot
// allocate device memory (see aes_ecb_batch_noalloc in aesgb.h).
// ---------------------------------------------------------------------------
constexpr size_t noalloc_scratch_bytes(size_t n) {
    return align_up(sizeof(BatchHeader), 256) + align_up(4 * n, 256) + align_up(8 * (n + 1), 256) +
           align_up(8 * n, 256);
}
constexpr size_t kNoAllocBytes = noalloc_scratch_bytes(AES_BATCH_NOALLOC_MAX_DESCS);

// One copy per device that loads this library; it lives until the process exits.
static __device__ __align__(256) uint8_t g_noalloc_scratch[kNoAllocBytes];

namespace {
constexpr int kMaxDev = 64;
std::mutex g_noalloc_mu;
void *g_noalloc_addr[kMaxDev];  // device address of g_noalloc_scratch, per device
}  // namespace

// Device address of this device's scratch array, looked up once per device
// (the host-side name of the array is not a device address).
int noalloc_scratch_ptr(int dev, void **out) {
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_addr[dev]) {
        void *p = nullptr;
        const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess || p == nullptr) {
            (void)cudaGetLastError();
            return AES_E_CUDA;
        }
        g_noalloc_addr[dev] = p;
    }
    *out = g_noalloc_addr[dev];
    return AES_OK;
}

// Debug build: counts of chunks with every pass taken exactly once, and with one
// taken more than once, since the last call, and of chunks past the tag array; clears the tags.
int read_chunk_coverage(unsigned long long *once, unsigned long long *repeated, unsigned long long *beyond) {
#if defined(AESGB_BOUNDS_CHECK)
    static ChunkTag tags[kTagChunks];
    static std::mutex mu;
    std::lock_guard<std::mutex> lk(mu);
    const unsigned long long zero = 0;
    if (cudaMemcpyFromSymbol(tags, g_chunk_tag, sizeof tags) != cudaSuccess ||
        cudaMemcpyFromSymbol(beyond, g_chunk_tag_beyond, sizeof *beyond) != cudaSuccess) {
        (void)cudaGetLastError();
        return AES_E_CUDA;
    }
    *once = 0;
    *repeated = 0;
    for (const ChunkTag &t : tags) {
        unsigned int seen = 0;
        for (unsigned int w : t.seen) seen += static_cast<unsigned int>(__builtin_popcount(w));
        *once += t.passes > 0 && seen == t.passes && t.again == 0;
        *repeated += t.again > 0;
    }
    void *tag_addr = nullptr;
    if (cudaGetSymbolAddress(&tag_addr, g_chunk_tag) != cudaSuccess ||
        cudaMemset(tag_addr, 0, sizeof tags) != cudaSuccess ||
        cudaMemcpyToSymbol(g_chunk_tag_beyond, &zero, sizeof zero) != cudaSuccess) {
        (void)cudaGetLastError();
        return AES_E_CUDA;
    }
    return AES_OK;
#else
    *once = *repeated = *beyond = 0;
    return AES_E_CONFIG;
#endif
}

// Debug build: the counts since the last call; clears them.
int read_batch_counts(unsigned long long *fills, unsigned long long *counter) {
#if defined(AESGB_BOUNDS_CHECK)
    unsigned long long c[kCounts];
    const unsigned long long zero[kCounts] = {};
    if (cudaMemcpyFromSymbol(c, g_batch_counts, sizeof c) != cudaSuccess ||
        cudaMemcpyToSymbol(g_batch_counts, zero, sizeof zero) != cudaSuccess) {
        (void)cudaGetLastError();
        return AES_E_CUDA;
    }
    *fills = c[kCountFills];
    *counter = c[kCountCounter];
    return AES_OK;
#else
    *fills = *counter = 0;
    return AES_E_CONFIG;
#endif
}

}  // namespace aesgb

using namespace aesgb;

extern "C" {

size_t aes_batch_workspace_bytes(int n) { return n < 0 ? 0 : batch_ws_bytes(n); }

int aes_debug_batch_coverage(unsigned long long *once, unsigned long long *repeated, unsigned long long *beyond) {
    if (!once || !repeated || !beyond) return AES_E_ARG;
    return read_chunk_coverage(once, repeated, beyond);
}

int aes_debug_batch_counts(unsigned long long *fills, unsigned long long *counter) {
    if (!fills || !counter) return AES_E_ARG;
    return read_batch_counts(fills, counter);
}

int aes_ecb_batch_ws(const aes_desc *desc_dev, int n, void *ws, size_t ws_bytes, int32_t *status_dev,
                     const aes_batch_cfg *cfg, void *stream) {
    if (n < 0) return AES_E_ARG;
    const aes_batch_cfg c = cfg ? *cfg : batch_cfg_for(n);
    return enqueue_batch(desc_dev, n, ws, ws_bytes, status_dev, c, static_cast<cudaStream_t>(stream));
}

int aes_ecb_batch(const aes_desc *desc_dev, int n, void *stream) {
    return aes_ecb_batch_ex(desc_dev, n, nullptr, stream);
}

int aes_ecb_batch_ex(const aes_desc *desc_dev, int n, int32_t *status_dev, void *stream) {
    if (n < 0) return AES_E_ARG;
    if (n == 0) return AES_OK;
    if (n > AES_BATCH_MAX_DESCS) return AES_E_RANGE;  // before the workspace is sized for it
    if (!desc_dev) return AES_E_ARG;
    const cudaStream_t s = static_cast<cudaStream_t>(stream);
    // a graph captured from this call would keep the workspace's address after
    // a later call on the stream has replaced it: capture aes_ecb_batch_ws
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &cap) != cudaSuccess) {
        (void)cudaGetLastError();
        return AES_E_CUDA;
    }
    if (cap != cudaStreamCaptureStatusNone) return AES_E_CONFIG;
    int dev = 0;
    if (current_device(&dev) != AES_OK) return AES_E_CUDA;
    std::shared_ptr<StreamWs> w;
    const int st = stream_workspace(dev, s, &w);
    if (st != AES_OK) return st;
    int r;
    {
        std::lock_guard<std::mutex> lk(w->mu);
        r = enqueue_with_stream_ws(*w, desc_dev, n, batch_ws_bytes(n), status_dev, s);
    }
    w->users.fetch_sub(1);
    return r;
}

int aes_ecb_batch_noalloc(const aes_desc *desc_dev, int n, int32_t *status_dev, void *stream) {
    if (n < 0) return AES_E_ARG;
    if (n > AES_BATCH_NOALLOC_MAX_DESCS) return AES_E_RANGE;
    if (n == 0) return AES_OK;
    if (batch_ws_bytes(n) > kNoAllocBytes) return AES_E_RANGE;
    int dev = 0;
    if (current_device(&dev) != AES_OK) return AES_E_CUDA;
    void *scratch = nullptr;
    const int st = noalloc_scratch_ptr(dev, &scratch);
    if (st != AES_OK) return st;
    // the plan kernel rewrites the header (work counters zeroed) and every
    // array the batch kernel reads, so what the previous call left behind in
    // the scratch is never used
    return enqueue_batch(desc_dev, n, scratch, kNoAllocBytes, status_dev, batch_cfg_for(n),
                         static_cast<cudaStream_t>(stream));
}

int aes_batch_graph_create(const aes_desc *desc_dev, int n, void *ws, size_t ws_bytes, int32_t *status_dev,
                           const aes_batch_cfg *cfg, aes_batch_graph **out) {
    if (!out || n <= 0) return AES_E_ARG;
    *out = nullptr;
    if (n > AES_BATCH_MAX_DESCS) return AES_E_RANGE;
    const aes_batch_cfg c = cfg ? *cfg : batch_cfg_for(n);
    int st0 = validate_batch_cfg(c);
    if (st0 != AES_OK) return st0;
    // one-time per-kernel set-up (shared-memory attribute) before capturing
    int dev = 0;
    if (current_device(&dev) != AES_OK) return AES_E_CUDA;
    st0 = ensure_smem_attr(batch_kernel_ptr(c.blocks_per_thread, c.layout_enc, c.layout_dec), dev,
                           batch_smem_bytes(c));
    if (st0 != AES_OK) return st0;
    cudaStream_t s = nullptr;
    if (cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking) != cudaSuccess) return AES_E_CUDA;
    BatchGraph *g = new BatchGraph();
    int st = AES_OK;
    if (cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal) != cudaSuccess) st = AES_E_CUDA;
    if (st == AES_OK) {
        st = enqueue_batch(desc_dev, n, ws, ws_bytes, status_dev, c, s);
        cudaGraph_t graph = nullptr;
        const cudaError_t e = cudaStreamEndCapture(s, &graph);
        if (st == AES_OK && e != cudaSuccess) st = AES_E_CUDA;
        g->graph = graph;
        if (st == AES_OK && cudaGraphInstantiate(&g->exec, graph, 0) != cudaSuccess) st = AES_E_CUDA;
    }
    cudaStreamDestroy(s);
    if (st != AES_OK) {
        (void)cudaGetLastError();
        if (g->exec) cudaGraphExecDestroy(g->exec);
        if (g->graph) cudaGraphDestroy(g->graph);
        delete g;
        return st;
    }
    *out = reinterpret_cast<aes_batch_graph *>(g);
    return AES_OK;
}

int aes_batch_graph_launch(aes_batch_graph *graph, void *stream) {
    if (!graph) return AES_E_ARG;
    BatchGraph *g = reinterpret_cast<BatchGraph *>(graph);
    if (cudaGraphLaunch(g->exec, static_cast<cudaStream_t>(stream)) != cudaSuccess) {
        (void)cudaGetLastError();
        return AES_E_CUDA;
    }
    return AES_OK;
}

int aes_batch_graph_destroy(aes_batch_graph *graph) {
    if (!graph) return AES_OK;
    BatchGraph *g = reinterpret_cast<BatchGraph *>(graph);
    if (g->exec) cudaGraphExecDestroy(g->exec);
    if (g->graph) cudaGraphDestroy(g->graph);
    delete g;
    return AES_OK;
}

}  // extern "C"

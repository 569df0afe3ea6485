// scan_tail.cu -- long traces checked in epochs: stream filter, compacted
// candidates, each set checked grouped by variable.
//
// Section 3.2: F is absorbing, so once a variable's status is F every later
// op on it yields F (Property Progress: a stuck variable stays stuck).  On a
// long trace nearly every op after the first few per variable is such an op.
// The first part of the trace, [0, S), is checked by sorting its ops by
// variable (scan_sorted.cu); the rest is cut into epochs (by default each
// ends at four times its start), and for each epoch
//   1. the statuses at its start are exact (the previous part's final
//      statuses); variables with status F form a bitmap;
//   2. a streaming kernel writes F at every position and collects the ops on
//      variables outside the bitmap ("candidates"), in position order;
//   3. the candidates, a set of ops over the same variables (an op's status
//      depends only on the earlier ops on its variable), are checked from the
//      epoch's start statuses, with their count read from device memory: one
//      radix pass groups them into 128 buckets by the low seven bits of the
//      variable id (position order kept inside a bucket), one CTA checks each
//      bucket (scan_sorted.cu, bucket check); the statuses that are not F go
//      to their positions, first faults to trace positions, final statuses
//      start the next epoch.
// Outputs are identical to one scan over the whole trace.  An epoch whose
// candidates overflow their slots is rechecked whole by the single-pass scan.
#include <cstdio>
#include <cstdlib>

#include "amc_internal.cuh"
#include "scan_trace.cuh"

namespace amc {

namespace {

constexpr int TF_THREADS = 1024;          // filter CTA: one per SM (the bitmap fills shared memory)
constexpr int TF_CHUNK = 4096;            // ops per warp chunk in epochs of 2^27 ops or more,
constexpr int TF_CHUNK_SHORT = 1024;      // in shorter epochs (more warps busy)
constexpr int64_t TF_LONG_CHUNKS_FROM = (int64_t)1 << 27;
// Candidate slots per chunk, and candidates per epoch: a quarter of the ops, half
// in epochs of at most 2^24 ops (more: the epoch falls back).  The early epochs
// have the most: a mostly right trace of 150 M ops over a million variables had
// 24 % candidates in its first epoch (6.3 M ops) and over a quarter in 826 of its
// 6,144 chunks, and fell back: 1,581 us, 1,150 with half.  Half of a short epoch costs
// no scratch where a longer one follows.  Later epochs have 16, 9 and 4 %.
constexpr int TF_SLOT_DIV = 4;
constexpr int64_t TF_HALF_TO = (int64_t)1 << 24;
constexpr int64_t CAND_MAX = (int64_t)1 << 27;   // and at most 2^27 (set index << 4 fits 32 bits)
constexpr int TF_SUB = 4;                 // parts of 128 ops in a warp's step
constexpr int TAIL_MIN_VARS = 16385;      // fewer variables take the reduce / carry / apply path
constexpr int TAIL_MAX_VARS = 1 << 20;    // bitmap of 128 KB in shared memory
constexpr int DEFAULT_FIRST_LOG2 = 21;    // first part 2^21 ops,
constexpr int DEFAULT_GROW = 2;           // then epochs ending at 4 times their start
constexpr int64_t DEFAULT_MIN_OPS = (int64_t)1 << 29;

struct TailShape {
    int64_t S = 0;        // ops of the first part
    int64_t E = 0;        // ops per epoch (grow == 0)
    int grow = 0;         // > 0: each epoch ends at 2^grow times its start
};

// AMC_SCAN_TAIL="s,e": first part 2^s ops, epochs of 2^e ops; "s,-g": first
// part 2^s ops, each epoch ending at 2^g times its start; for every trace
// longer than 2^s ops (test and tuning override); "0" disables.
// force: -1 by size (from DEFAULT_MIN_OPS ops), 1 for every trace longer than
// 2^21 ops (first part 2^21 ops from 2^23 ops on, else a quarter of the trace),
// 0 never.
bool tail_shape(int64_t n_ops, int32_t n_vars, bool guarded, TailShape& sh, int force)
{
    if (guarded || n_vars < TAIL_MIN_VARS || n_vars > TAIL_MAX_VARS || !bucket_check_ok(n_vars)) return false;
    if (const char* e = getenv("AMC_SCAN_TAIL")) {
        if (e[0] == '0' && e[1] == 0) return false;
        int a = 0, b = 0;
        if (sscanf(e, "%d,%d", &a, &b) == 2 && a >= 12 && a <= 27 && ((b >= 12 && b < 31) || (b >= -4 && b <= -1))) {
            sh.S = (int64_t)1 << a;
            if (n_ops <= sh.S) return false;
            if (b > 0) {
                sh.E = (int64_t)1 << b;
                if (sh.E > n_ops - sh.S) sh.E = n_ops - sh.S;
            } else {
                sh.grow = -b;
            }
            return true;
        }
    }
    if (force == 0) return false;
    if (force == 1 ? n_ops <= ((int64_t)1 << DEFAULT_FIRST_LOG2) : n_ops < DEFAULT_MIN_OPS) return false;
    int lg = DEFAULT_FIRST_LOG2;
    while (lg > 12 && ((int64_t)1 << (lg + 2)) > n_ops) --lg;      // first part at most a quarter
    sh.S = (int64_t)1 << lg;
    sh.grow = DEFAULT_GROW;
    return true;
}

// ops per filter chunk of an epoch of n ops
int chunk_for(int64_t n) { return n < TF_LONG_CHUNKS_FROM ? TF_CHUNK_SHORT : TF_CHUNK; }
int64_t chunks_of(int64_t n) { return (n + chunk_for(n) - 1) / chunk_for(n); }
int slot_div(int64_t n) { return n <= TF_HALF_TO ? TF_SLOT_DIV / 2 : TF_SLOT_DIV; }
int slots_for(int64_t n) { return chunk_for(n) / slot_div(n); }

int64_t epoch_end(const TailShape& sh, int64_t e0, int64_t n_ops)
{
    const int64_t e1 = sh.grow ? (e0 << sh.grow) : e0 + sh.E;
    return e1 < n_ops ? e1 : n_ops;
}

int64_t longest_epoch(const TailShape& sh, int64_t n_ops)
{
    int64_t m = 0;
    for (int64_t e0 = sh.S; e0 < n_ops; e0 = epoch_end(sh, e0, n_ops)) {
        const int64_t len = epoch_end(sh, e0, n_ops) - e0;
        if (len > m) m = len;
    }
    return m;
}

// candidate capacity of an epoch of E ops
int64_t cand_cap(int64_t E)
{
    int64_t C = (E + slot_div(E) - 1) / slot_div(E);
    C = (C + TF_CHUNK - 1) / TF_CHUNK * TF_CHUNK;
    return C < CAND_MAX ? C : CAND_MAX;
}

struct TailLayout {
    int64_t K = 0;        // pairs the sort buffers hold: the first part or an epoch's candidates
    size_t st0, st1, bm, cnt, off, coff, ncand, ovf, fvff, fff;
    size_t region;        // shared region: pairs and slots, or the fallback scan
    size_t key0, val0, pos, key1, val1, slot, scratch;   // offsets inside the region
    size_t total;
};

// Scratch: a few per-variable arrays, then one region used in turn by the
// first part's pairs, by an epoch's candidates (chunk slots, sharing their
// space with the sort's second buffers, the pairs, their positions, the sort's
// scratch), and by the epoch's fallback scan over all its ops (taken when the
// candidates overflow their slots).
TailLayout tail_layout(const TailShape& sh, int32_t n_vars, int64_t n_ops)
{
    TailLayout t;
    const int64_t Emax = longest_epoch(sh, n_ops);
    size_t n_chunks = 0, n_slots = 0;          // most chunks, most slots of one epoch
    for (int64_t e0 = sh.S; e0 < n_ops; e0 = epoch_end(sh, e0, n_ops)) {
        const int64_t n = epoch_end(sh, e0, n_ops) - e0;
        if ((size_t)chunks_of(n) > n_chunks) n_chunks = (size_t)chunks_of(n);
        if ((size_t)(chunks_of(n) * slots_for(n)) > n_slots) n_slots = (size_t)(chunks_of(n) * slots_for(n));
    }
    t.K = sh.S;
    for (int64_t e0 = sh.S; e0 < n_ops; e0 = epoch_end(sh, e0, n_ops))
        if (const int64_t C = cand_cap(epoch_end(sh, e0, n_ops) - e0); C > t.K) t.K = C;
    const size_t K = (size_t)t.K;
    size_t o = 0;
    auto take = [&](size_t b) { const size_t at = o; o += align_up(b, 256); return at; };
    t.st0 = take((size_t)n_vars);
    t.st1 = take((size_t)n_vars);
    t.bm = take(4 * (size_t)((n_vars + 31) / 32));
    t.cnt = take(4 * n_chunks);
    t.off = take(4 * n_chunks);
    t.coff = take(4 * n_chunks);
    t.ncand = take(8);
    t.ovf = take(8);
    t.fvff = take(4 * (size_t)n_vars);
    t.fff = take(8);
    t.region = o;
    size_t r = 0;
    auto rtake = [&](size_t b) { const size_t at = r; r += align_up(b, 256); return at; };
    t.key0 = rtake(4 * K);
    t.val0 = rtake(4 * K);
    t.pos = rtake(4 * K);
    t.scratch = rtake(sorted_check_scratch_bytes(t.K));
    // the slots live until the gather; the sort's second buffers after it
    const size_t shared_at = r;
    t.key1 = shared_at;
    t.val1 = shared_at + align_up(4 * K, 256);
    t.slot = shared_at;
    const size_t second = 2 * align_up(4 * K, 256);
    const size_t slots = align_up(8 * n_slots, 256);
    r += second > slots ? second : slots;
    size_t reg = r;
    const size_t fallback = scan_workspace_bytes(Emax, n_vars, false);
    if (fallback > reg) reg = fallback;
    t.total = o + reg;
    return t;
}

// bit v: status of v is F
__global__ void tail_bitmap_kernel(const uint8_t* __restrict__ st, int32_t n_vars, uint32_t* __restrict__ bm)
{
    follow();
    const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool f = v < n_vars && st[v] == ST_F;
    const uint32_t m = __ballot_sync(0xffffffffu, f);
    if ((threadIdx.x & 31) == 0 && v < n_vars) bm[v >> 5] = m;
}

struct FilterParams {
    const uint8_t* kind_side;   // the epoch's first op
    const int32_t* var;
    int64_t n;                  // ops in the epoch
    int64_t n_after;            // ops of the trace from the epoch's first op on (GT pairing)
    int32_t n_vars;
    const uint32_t* bm;         // stuck bitmap at the epoch's start
    int bm_words;
    uint8_t* step;              // the epoch's outputs
    uint2* slot;                // candidate slots, `slots` per chunk
    uint32_t* cnt;              // candidates per chunk
    int* ovf;                   // set when a chunk has more candidates than slots
    int* err;
    int bulk_ok;
    int slots;
};

// A GT must be followed by the EN of the same side on another variable (op i of
// the epoch; other kinds pass).
__device__ __forceinline__ void check_gt(const FilterParams& q, int64_t i)
{
    const uint32_t ks = q.kind_side[i];
    if ((ks & 15u) != AMC_K_GT) return;
    const int32_t v = (uint32_t)q.var[i] < (uint32_t)q.n_vars ? q.var[i] : 0;
    const bool next = i + 1 < q.n_after;
    const uint32_t nks = next ? q.kind_side[i + 1] : 0xFFu;
    if (!((nks & 15) == AMC_K_EN && (nks >> 4) == (ks >> 4) && (next ? q.var[i + 1] : v) != v))
        raise_error(q.err, AMC_E_INVALID);
}

// Each warp takes chunks of CHUNK ops in steps of 4 x 128 (lane L: ops 4 L to 4 L +
// 3 of each 128, so that every load and store of the warp is one run of memory);
// every position gets F (the candidates' statuses that are not F are written
// after their check), the ops on variables outside the bitmap are staged in the
// chunk's slots in position order (id, position in the chunk << 8 | op byte).  Op
// bytes and ids are checked as in the scan (malformed bytes, ids out of range, GT
// not followed by its EN); an id out of range is staged as 0.
// What bounds it: memory in the late epochs, where almost nothing is staged, the
// L1 with its 32 bitmap look-ups in shared memory a warp load in the early ones.
// Sixteen ops in a row per lane, staged as a byte, a word and two bytes: 1,197 us for
// the five epochs of a 2^30-op trace (6.4 GB), 1,127 this way (6.0 TB/s in the two
// long ones).
template <int CHUNK>
__global__ void __launch_bounds__(TF_THREADS, 1) tail_filter_kernel(const FilterParams q)
{
    follow();
    extern __shared__ __align__(16) uint32_t sbm[];
    for (int i = threadIdx.x; i < q.bm_words; i += TF_THREADS) sbm[i] = q.bm[i];
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    const int64_t n_chunks = (q.n + CHUNK - 1) / CHUNK;
    constexpr uint32_t F4 = 0x01010101u * ST_F;
    for (int64_t c = (int64_t)blockIdx.x * (TF_THREADS / 32) + warp; c < n_chunks;
         c += (int64_t)gridDim.x * (TF_THREADS / 32)) {
        const int64_t c0 = c * CHUNK;
        const int cn = (int)min((int64_t)CHUNK, q.n - c0);
        int wcount = 0;
        bool full = false;                                   // slots exhausted (warp-uniform)
        for (int s0 = 0; s0 < cn; s0 += 128 * TF_SUB) {
            uint32_t kw[TF_SUB];
            int4 va[TF_SUB];
            uint32_t live = 0;                               // bit 4 t + j: op j of the lane's four in part t
            if (q.bulk_ok && cn - s0 >= 128 * TF_SUB) {
                const int64_t i0 = c0 + s0 + 4 * lane;       // offset in the epoch
#pragma unroll
                for (int t = 0; t < TF_SUB; ++t) {
                    kw[t] = __ldcs(reinterpret_cast<const uint32_t*>(q.kind_side + i0 + 128 * t));
                    va[t] = __ldcs(reinterpret_cast<const int4*>(q.var + i0 + 128 * t));
                }
                // four op bytes per 32-bit word are checked at once
                uint32_t badk = 0, gt = 0;
                bool badv = false;
#pragma unroll
                for (int t = 0; t < TF_SUB; ++t) {
                    // a valid byte has bits 3 and 5-7 clear (kinds 0..7, side bit 4)
                    badk |= kw[t] & 0xE8E8E8E8u;
                    // bytes whose kind is GT (6): zero bytes of (kind ^ 6)
                    const uint32_t x = (kw[t] & 0x0F0F0F0Fu) ^ 0x06060606u;
                    gt |= (x - 0x01010101u) & ~x & 0x80808080u;
                    int* const v4 = reinterpret_cast<int*>(&va[t]);
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const bool ok = (uint32_t)v4[j] < (uint32_t)q.n_vars;
                        badv |= !ok;
                        const uint32_t uv = ok ? (uint32_t)v4[j] : 0u;
                        v4[j] = (int)uv;
                        const uint32_t stuck = (sbm[uv >> 5] >> (uv & 31)) & 1u;
                        live |= (stuck ^ 1u) << (4 * t + j);
                    }
                    __stcs(reinterpret_cast<uint32_t*>(q.step + i0 + 128 * t), F4);
                }
                if (badk) raise_error(q.err, AMC_E_INVALID);
                if (badv) raise_error(q.err, AMC_E_RANGE);
                if (gt)
                    for (int t = 0; t < TF_SUB; ++t)
                        for (int j = 0; j < 4; ++j) check_gt(q, i0 + 128 * t + j);
            } else {
#pragma unroll
                for (int t = 0; t < TF_SUB; ++t) {
                    kw[t] = 0;
                    va[t] = make_int4(0, 0, 0, 0);
                    int* const v4 = reinterpret_cast<int*>(&va[t]);
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int off = s0 + 128 * t + 4 * lane + j;
                        if (off >= cn) continue;
                        const int64_t i = c0 + off;
                        const uint32_t ks = q.kind_side[i];
                        kw[t] |= ks << (8 * j);
                        v4[j] = q.var[i];
                        if ((ks & 0xE0u) || (ks & 15u) > AMC_K_EN) raise_error(q.err, AMC_E_INVALID);
                        if (v4[j] < 0 || v4[j] >= q.n_vars) {
                            raise_error(q.err, AMC_E_RANGE);
                            v4[j] = 0;
                        }
                        check_gt(q, i);
                        const uint32_t uv = (uint32_t)v4[j];
                        if (!((sbm[uv >> 5] >> (uv & 31)) & 1u)) live |= 1u << (4 * t + j);
                        q.step[i] = (uint8_t)ST_F;
                    }
                }
            }
            if (full || !__any_sync(0xffffffffu, live != 0)) continue;
            int at[TF_SUB], tot = 0;                         // the lane's first slot of each part
#pragma unroll
            for (int t = 0; t < TF_SUB; ++t) {
                const int cl = __popc((live >> (4 * t)) & 15u);
                at[t] = tot;
#pragma unroll
                for (int bit = 0; bit < 3; ++bit) {          // counts 0..4
                    const uint32_t bal = __ballot_sync(0xffffffffu, (cl >> bit) & 1);
                    at[t] += __popc(bal & lt) << bit;
                    tot += __popc(bal) << bit;
                }
            }
            if (wcount + tot > q.slots) {
                // more candidates than slots: the epoch is rechecked whole
                if (lane == 0) atomicExch(q.ovf, 1);
                full = true;
                continue;
            }
            uint2* const slot = q.slot + c * q.slots + wcount;
#pragma unroll
            for (int t = 0; t < TF_SUB; ++t) {
                const int* const v4 = reinterpret_cast<const int*>(&va[t]);
                int o = at[t];
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (live & (1u << (4 * t + j)))
                        slot[o++] = make_uint2((uint32_t)v4[j], (uint32_t)(s0 + 128 * t + 4 * lane + j) << 8 |
                                                                    ((kw[t] >> (8 * j)) & 0xFFu));
            }
            wcount += tot;
        }
        if (lane == 0) q.cnt[c] = (uint32_t)wcount;
    }
}

// Candidates per block of 1024 chunks.
__global__ void __launch_bounds__(1024) tail_blocksum_kernel(const uint32_t* __restrict__ cnt, int n_chunks,
                                                             uint32_t* __restrict__ bsum)
{
    follow();
    __shared__ uint32_t ws[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int i = blockIdx.x * 1024 + threadIdx.x;
    uint32_t x = i < n_chunks ? cnt[i] : 0u;
#pragma unroll
    for (int d = 16; d; d >>= 1) x += __shfl_xor_sync(0xffffffffu, x, d);
    if (lane == 0) ws[warp] = x;
    __syncthreads();
    if (warp == 0) {
        uint32_t y = ws[lane];
#pragma unroll
        for (int d = 16; d; d >>= 1) y += __shfl_xor_sync(0xffffffffu, y, d);
        if (lane == 0) bsum[blockIdx.x] = y;
    }
}

// Offsets of the chunks' candidates in the compacted set, in position order.  Block b takes
// chunks [1024 b, 1024 b + 1024): its base is the sum of the earlier blocks'
// counts, its chunks' offsets a block scan; each warp copies 32 chunks.  Every
// block also forms the grand total, so all agree on an overflow (more
// candidates than the compacted trace holds, or a chunk with more than its
// slots): then nothing is copied and the epoch's fallback scan runs instead.
__global__ void __launch_bounds__(1024) tail_offsets_kernel(const uint32_t* __restrict__ cnt, int n_chunks,
                                                            const uint32_t* __restrict__ bsum, int n_blocks,
                                                            int64_t cap, uint32_t* __restrict__ coff,
                                                            int64_t* __restrict__ n_cand, int* ovf)
{
    follow();
    __shared__ unsigned long long rb[32], rt[32];
    __shared__ uint32_t wsum[32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int b = blockIdx.x;
    unsigned long long before = 0, total = 0;
    for (int j = tid; j < n_blocks; j += 1024) {
        const unsigned long long v = bsum[j];
        total += v;
        if (j < b) before += v;
    }
#pragma unroll
    for (int d = 16; d; d >>= 1) {
        before += __shfl_xor_sync(0xffffffffu, before, d);
        total += __shfl_xor_sync(0xffffffffu, total, d);
    }
    if (lane == 0) {
        rb[warp] = before;
        rt[warp] = total;
    }
    const int filter_ovf = *ovf;              // read before any block can write it
    __syncthreads();
    before = total = 0;
#pragma unroll 4
    for (int w = 0; w < 32; ++w) {
        before += rb[w];
        total += rt[w];
    }
    if (filter_ovf || total > (unsigned long long)cap) {
        if (b == 0 && tid == 0) {
            *ovf = 1;
            *n_cand = 0;
        }
        return;
    }
    if (b == 0 && tid == 0) *n_cand = (int64_t)total;
    const int i = b * 1024 + tid;
    const uint32_t x = i < n_chunks ? cnt[i] : 0u;
    uint32_t incl = x;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += y;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        uint32_t v = wsum[lane];
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, v, d);
            if (lane >= d) v += y;
        }
        wsum[lane] = v;                      // inclusive over warps
    }
    __syncthreads();
    if (i < n_chunks) coff[i] = (uint32_t)before + (warp > 0 ? wsum[warp - 1] : 0u) + incl - x;
}

// Warp per G consecutive chunks (G a power of two up to 32, larger where the
// epoch has many chunks and few candidates each), whose candidates are
// contiguous in the compacted set: lane L copies entries L, L + 32, ... of
// that stretch (the stores coalesce), finding each entry's chunk by a binary
// search over the G chunks' prefix counts, which lanes 0..G-1 hold.
__global__ void __launch_bounds__(256) tail_gather_kernel(const uint2* __restrict__ slot,
                                                          const uint32_t* __restrict__ cnt,
                                                          const uint32_t* __restrict__ coff, int n_chunks,
                                                          uint32_t* __restrict__ ckey, uint32_t* __restrict__ cval,
                                                          uint32_t* __restrict__ cpos, int G, int chunk, int slots,
                                                          const int* ovf)
{
    follow();
    if (*ovf) return;
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t g = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; g * G < n_chunks; g += nw) {
        const int64_t c = g * G + lane;
        const bool mine = lane < G && c < n_chunks;
        const uint32_t nk = mine ? cnt[c] : 0u;
        const uint32_t base = __shfl_sync(0xffffffffu, mine ? coff[c] : 0u, 0);
        uint32_t incl = nk;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += y;
        }
        const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
        const uint32_t excl = incl - nk;
        for (uint32_t i0 = 0; i0 < total; i0 += 32) {
            const uint32_t idx = i0 + lane;
            int k = 0;                                      // largest k < G with excl_k <= idx
            for (int step = G >> 1; step; step >>= 1) {
                const uint32_t e = __shfl_sync(0xffffffffu, excl, k + step);
                if (e <= idx) k += step;
            }
            const uint32_t first = __shfl_sync(0xffffffffu, excl, k);
            if (idx < total) {
                const int64_t ch = g * G + k;
                const int64_t src = ch * slots + (idx - first);
                const uint32_t o = base + idx;
                const uint2 x = slot[src];
                ckey[o] = x.x;
                cval[o] = o << 4 | sorted_code_of(x.y & 0xFFu);
                cpos[o] = (uint32_t)ch * (uint32_t)chunk + (x.y >> 8);
            }
        }
    }
}

// After an epoch's fallback scan (gated on by its overflow flag): the scan's
// first faults folded into the trace's, the stuck bitmap rebuilt from the
// statuses the scan wrote.
__global__ void tail_post_kernel(const int* gate, int* next_gate, const uint8_t* __restrict__ fst,
                                 uint8_t* __restrict__ st, int32_t n_vars,
                                 uint32_t* __restrict__ bm, int32_t* __restrict__ vff,
                                 const int32_t* __restrict__ fvff, int64_t* __restrict__ ff,
                                 const int64_t* __restrict__ fff, int64_t offset)
{
    follow();
    if (blockIdx.x == 0 && threadIdx.x == 0) *next_gate = 0;
    if (*gate == 0) return;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t n_words = ((int64_t)n_vars + 31) / 32 * 32;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n_words; v += stride) {
        bool f = false;
        if (v < n_vars) {
            if (vff[v] == -1 && fvff[v] != -1) vff[v] = (int32_t)(fvff[v] + offset);
            st[v] = fst[v];
            f = fst[v] == ST_F;
        }
        const uint32_t m = __ballot_sync(0xffffffffu, f);
        if ((threadIdx.x & 31) == 0) bm[v >> 5] = m;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0 && *fff != -1) {
        const unsigned long long g = (unsigned long long)(*fff + offset);
        atomicMin(reinterpret_cast<unsigned long long*>(ff), g);
    }
}

}  // namespace

bool scan_tail_eligible(const ScanLaunch& L)
{
    TailShape sh;
    return (L.dense != 0 || L.tail == 1) && !L.n_dev && !L.gate && !L.guard && !L.pre_mode &&
           tail_shape(L.n_ops, L.n_vars, false, sh, L.tail);
}

size_t scan_tail_workspace_bytes(int64_t n_ops, int32_t n_vars)
{
    TailShape sh;                          // the largest shape a launch may take (forced)
    if (!tail_shape(n_ops, n_vars, false, sh, 1)) return 0;
    size_t b = tail_layout(sh, n_vars, n_ops).total;
    TailShape sd;
    if (tail_shape(n_ops, n_vars, false, sd, -1)) {
        const size_t d = tail_layout(sd, n_vars, n_ops).total;
        if (d > b) b = d;
    }
    return b;
}

int scan_tail_launches(const ScanLaunch& L)
{
    TailShape sh;
    if (!scan_tail_eligible(L) || !tail_shape(L.n_ops, L.n_vars, false, sh, L.tail)) return 0;
    // a sorted check: three kernels per radix pass, then the segmented scan's
    // reduce, carry and apply; a bucket check: one radix pass, the bucket kernel
    const int sorted = 3 + 3 * ss_radix_passes(L.n_vars);
    const int bucketed = 3 + 1;
    int epochs = 0;
    for (int64_t e0 = sh.S; e0 < L.n_ops; e0 = epoch_end(sh, e0, L.n_ops)) ++epochs;
    // first part: pairs, its sorted check, the stuck bitmap; per epoch filter,
    // block sums, offsets, gather (which writes the pairs), the candidates'
    // bucket check, gated set-up / scan / final statuses and the gated merge
    // with bitmap rebuild
    return 1 + sorted + 1 + epochs * (4 + bucketed + 3 + 1);
}

int launch_scan_tail(const ScanLaunch& L, cudaStream_t s)
{
    TailShape sh;
    if (!tail_shape(L.n_ops, L.n_vars, false, sh, L.tail)) return AMC_E_INVALID;
    const TailLayout lay = tail_layout(sh, L.n_vars, L.n_ops);
    uint8_t* w = static_cast<uint8_t*>(L.workspace);
    // the statuses as the trace goes on, where they are wanted in the end unless
    // the initial ones lie there too (the first part reads those while it writes
    // its final ones); a fallback's final ones
    const bool apart = L.final_status && !(L.init && L.init < L.final_status + L.n_vars &&
                                           L.final_status < L.init + L.n_vars);
    uint8_t* st = apart ? L.final_status : w + lay.st0;
    uint8_t* fst = w + lay.st1;
    uint32_t* bm = reinterpret_cast<uint32_t*>(w + lay.bm);
    uint32_t* cnt = reinterpret_cast<uint32_t*>(w + lay.cnt);
    uint32_t* bsum = reinterpret_cast<uint32_t*>(w + lay.off);    // candidates per 1024 chunks
    uint32_t* coff = reinterpret_cast<uint32_t*>(w + lay.coff);   // first candidate of each chunk
    int64_t* ncand = reinterpret_cast<int64_t*>(w + lay.ncand);
    int* ovf = reinterpret_cast<int*>(w + lay.ovf);            // two words, in turn: an epoch's end clears the next one's
    int32_t* fvff = reinterpret_cast<int32_t*>(w + lay.fvff);
    int64_t* fff = reinterpret_cast<int64_t*>(w + lay.fff);
    uint8_t* reg = w + lay.region;
    uint2* slot = reinterpret_cast<uint2*>(reg + lay.slot);
    uint32_t* key0 = reinterpret_cast<uint32_t*>(reg + lay.key0);
    uint32_t* val0 = reinterpret_cast<uint32_t*>(reg + lay.val0);
    uint32_t* key1 = reinterpret_cast<uint32_t*>(reg + lay.key1);
    uint32_t* val1 = reinterpret_cast<uint32_t*>(reg + lay.val1);
    uint32_t* cpos = reinterpret_cast<uint32_t*>(reg + lay.pos);
    void* scratch = reg + lay.scratch;

    int dev = 0, n_sm = 0, max_optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&max_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    const int bm_words = (L.n_vars + 31) / 32;
    const size_t fsmem = 4 * (size_t)bm_words;
    if ((int)fsmem > max_optin) return AMC_E_INVALID;
    if (!allow_smem<tail_filter_kernel<TF_CHUNK>>(TAIL_MAX_VARS / 8) ||
        !allow_smem<tail_filter_kernel<TF_CHUNK_SHORT>>(TAIL_MAX_VARS / 8))
        return AMC_E_CUDA;
    if (L.profile & 1) profile_begin(s);

    // first part: ops [0, S) checked by sorting them by variable, from the
    // initial statuses; final statuses to st
    const SortedStart z = {L.vff, L.first_fault, st, L.init, ovf};
    int rc = launch_ss_keys(L.kind_side, L.var, sh.S, L.n_ops, L.n_vars, key0, val0, L.step, z, L.err, s);
    if (rc) return rc;
    SortedCheck A;
    A.key[0] = key0;
    A.key[1] = key1;
    A.val[0] = val0;
    A.val[1] = val1;
    A.cap = sh.S;
    A.n_vars = L.n_vars;
    A.init = L.init;
    A.step = L.step;
    A.fin = st;
    A.vff = L.vff;
    A.ff = L.first_fault;
    A.scratch = scratch;
    A.err = L.err;
    rc = launch_sorted_check(A, s);
    if (rc) return rc;
    // the stuck bitmap at the first epoch's start; later epochs add the
    // variables that become stuck (the bucket checks set their bits, the
    // fallback rebuilds it)
    chain(tail_bitmap_kernel, (unsigned)((L.n_vars + 255) / 256), 256, 0, s)(st, L.n_vars, bm);

    int cur = 0;
    for (int64_t e0 = sh.S; e0 < L.n_ops; cur ^= 1) {
        int* const gate = ovf + cur;
        const int64_t e1 = epoch_end(sh, e0, L.n_ops);
        const int64_t n = e1 - e0;
        const int chunk = chunk_for(n);
        const int slots = slots_for(n);
        FilterParams q;
        q.kind_side = L.kind_side + e0;
        q.var = L.var + e0;
        q.n = n;
        q.n_after = L.n_ops - e0;
        q.n_vars = L.n_vars;
        q.bm = bm;
        q.bm_words = bm_words;
        q.step = L.step + e0;
        q.slot = slot;
        q.cnt = cnt;
        q.ovf = gate;
        q.slots = slots;
        q.err = L.err;
        q.bulk_ok = (uintptr_t)q.kind_side % 4 == 0 && (uintptr_t)q.var % 16 == 0 && (uintptr_t)q.step % 4 == 0;
        const int n_chunks = (int)chunks_of(n);
        const int fgrid = (int)min((int64_t)n_sm, ((int64_t)n_chunks + TF_THREADS / 32 - 1) / (TF_THREADS / 32));
        if (chunk == TF_CHUNK)
            chain(tail_filter_kernel<TF_CHUNK>, fgrid, TF_THREADS, fsmem, s)(q);
        else
            chain(tail_filter_kernel<TF_CHUNK_SHORT>, fgrid, TF_THREADS, fsmem, s)(q);
        const int n_blocks = (n_chunks + 1023) / 1024;
        const int64_t C = cand_cap(n);
        chain(tail_blocksum_kernel, n_blocks, 1024, 0, s)(cnt, n_chunks, bsum);
        chain(tail_offsets_kernel, n_blocks, 1024, 0, s)(cnt, n_chunks, bsum, n_blocks, C, coff, ncand, gate);
        int G = 1;                                   // chunks per gather warp: about 8,192 warps
        while (G < 32 && n_chunks / (2 * G) >= 8192) G *= 2;
        const int64_t groups = ((int64_t)n_chunks + G - 1) / G;
        const int ggrid = (int)min((int64_t)n_sm * 8, (groups + 7) / 8);
        chain(tail_gather_kernel, ggrid, 256, 0, s)(slot, cnt, coff, n_chunks, key0, val0, cpos, G, chunk, slots,
                                                 gate);
        if (cudaGetLastError() != cudaSuccess) return AMC_E_CUDA;
        // the candidates, at most C (count on the device), from the epoch's
        // start statuses, checked per bucket of ids (a bucket's statuses are read
        // and, where they change, written by its CTA); gated off when they
        // overflowed
        SortedCheck K;
        K.key[0] = key0;
        K.key[1] = key1;
        K.val[0] = val0;
        K.val[1] = val1;
        K.pos = cpos;
        K.n_dev = ncand;
        K.cap = C;
        K.gate = gate;
        K.n_vars = L.n_vars;
        K.init = st;
        K.step = L.step + e0;
        K.fin = st;
        K.vff = L.vff;
        K.ff = L.first_fault;
        K.offset = e0;
        K.scratch = scratch;
        K.err = L.err;
        K.bm = bm;
        rc = launch_bucket_check(K, s);
        if (rc) return rc;
        // fallback, gated on by an overflow: the single-pass scan over all the
        // epoch's ops from its start statuses
        ScanLaunch F = L;
        F.kind_side = L.kind_side + e0;
        F.var = L.var + e0;
        F.n_ops = n;
        F.gate = gate;
        F.gate_on = 1;
        F.init = st;
        F.step = L.step + e0;
        F.final_status = fst;
        F.vff = fvff;
        F.first_fault = fff;
        F.workspace = reg;
        F.dense = 0;
        F.profile = 0;
        rc = launch_scan_trace(F, s);
        if (rc) return rc;
        chain(tail_post_kernel, n_sm * 2, 256, 0, s)(gate, ovf + (cur ^ 1), fst, st, L.n_vars, bm, L.vff, fvff, L.first_fault, fff,
                                                      e0);
        if (cudaGetLastError() != cudaSuccess) return AMC_E_CUDA;
        e0 = e1;
    }
    if (L.final_status && !apart &&
        cudaMemcpyAsync(L.final_status, st, (size_t)L.n_vars, cudaMemcpyDeviceToDevice, s) != cudaSuccess)
        return AMC_E_CUDA;
    if (L.profile & 2) profile_end(s);
    return AMC_OK;
}

}  // namespace amc

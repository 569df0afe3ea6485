// scan_owner.cu -- the trace check for traces whose variables' statuses fit a
// CTA's shared memory (reduce, carry, apply over owner-sorted tiles).
//
// An op's status depends only on the earlier ops on its variable (Fig. Opsem,
// rules Effect / Remote Effect), so the ops of a tile may be regrouped as long
// as every variable keeps its own order.  Every variable is owned by one of a
// CTA's threads.  A tile is regrouped by owner once (a stable counting pass on
// the owner: one ballot per bit ranks a warp's 32 ops), and then every thread
// walks its own ops in order: a byte of shared memory per variable that no
// other thread touches, so there is no grouping of lanes with equal variables,
// no composition within a group and no barrier inside the walk.  Where one owner
// has much of a tile (a trace that is mostly about a few variables) a warp walks
// its ops in up to 32 pieces instead, with a row of the owner's bytes per piece.
//   1. sort + reduce: CTA c takes chunk c (consecutive tiles): every tile is
//      checked, sorted by owner and written out as 4-byte entries (variable,
//      4-bit op code, position); each thread folds its ops into one transfer
//      function per variable; the chunk's functions are written out;
//   2. carry: the chunks' functions applied in order to the initial statuses:
//      every chunk's entry statuses, the final statuses;
//   3. apply: CTA c walks its sorted tiles again from the entry statuses and
//      writes every op's status and the first faults.
// A guarded trace (GT: the transfer of Fig. sem-AM, guarded by the status of
// the EN that follows it, read with every GT as Noop) takes one more walk
// between two carries: 2. gives the entry statuses with GT as Noop, then
//   2b. resolve + reduce: CTA c walks its sorted tiles from those statuses,
//      notes the status before every EN, marks the entries of the GTs whose
//      guard finds the side invalid, and folds the resolved ops again;
// and 2. / 3. follow on the resolved functions.
// What bounds it: instruction issue and shared-memory latency (the ranking's
// ballots in step 1, about a dozen instructions per op and walk after it; 119,
// 103 and 42 warp instructions per 32 ops in steps 1, 2b and 3), not memory: 5
// bytes in and 4 out per op in step 1, 4 in and 1 out in step 3.  Warps that
// instead walk 32 consecutive ops at a time over a row of their own, lanes with
// equal variables grouped by match.any, take 144 to 160 warp instructions per
// 32 ops and walk, and a guarded trace four walks: the check of 182 M
// statements over 8,192 variables took 7.75 ms that way and takes 2.3 ms here
// (1.00 + 0.82 + 0.40 ms for steps 1, 2b and 3), one of 300,007 ops over 2,011
// variables 171 us and 39 us.  Tiles of 4,096 ops for 128 owners rather than
// 2,048 took step 1 from 1.53 to 1.13 ms and step 3 from 0.50 to 0.38 ms (the
// longest walk of a warp over the mean: 1.57 against 1.81).
#include "amc_internal.cuh"
#include "scan_owner.cuh"

namespace amc {

namespace {

constexpr int POSB = 12;                  // position bits of an entry
constexpr int OSEG = 32;                  // chunks per carry segment
constexpr int OCTAS = 6;                  // CTAs an SM the chunks are made for
constexpr uint32_t EN_HERE = 0x80u;       // mark of an EN in a tile's noted statuses
// An owner with more than HEAVY ops in a tile, and HEAVY_SLOT for each of its
// bytes, has them walked in pieces.  Its thread alone takes about 35 cycles an op
// while the others wait; a warp two walks of a 4th to a 32nd of that and a pass over
// the pieces' bytes, a few owners at a time.  From 128 ops on, tiles with many lists a
// little longer lose: 16 M ops over 20 variables 366 us against 341 without pieces and
// 331 so, and with no allowance for the bytes 1 M calls over 16,400 arrays 3.31 ms
// against 2.41; 10 M ops over 8,000 Zipf ids take 304 us from 128 on, 325 so, 372 from
// 384 on or without.  16,000,000 guarded ops, 9 of 10 on one array of 1,000 / 30,000: 3.07 /
// 6.78 ms by its thread alone, 0.45 / 1.56 so.
constexpr int HEAVY = 256, HEAVY_SLOT = 4;

// Owner of variable v among NT threads, and the offset of its byte in a row
// without the owner's part.  v = NT h + l is owned by thread (l + 37 h) mod NT
// -- mixed with h, so that ids a multiple of NT apart (an array and its
// abstract variable) have different owners: the longest walk of a warp, over
// the mean, falls from 2.2 to 1.8 on a VectorPU trace.  Byte of the row: word
// (h / 4) NT + owner, byte h mod 4, so that thread t's bytes lie in bank t mod 32.
template <int NT>
__host__ __device__ __forceinline__ uint32_t owner_of(uint32_t v)
{
    return (v + 37u * (v / NT)) & (NT - 1);
}
// Offset of an owner's h-th byte, and which one an offset is.
template <int NT>
__device__ __forceinline__ uint32_t addr_of_slot(uint32_t h)
{
    return (h >> 2) * (4 * NT) | (h & 3u);
}
template <int NT>
__device__ __forceinline__ uint32_t slot_of(uint32_t addr)
{
    return (addr / (4 * NT)) << 2 | (addr & 3u);
}
template <int NT>
__device__ __forceinline__ uint32_t addr_of(uint32_t v)
{
    return addr_of_slot<NT>(v / NT);
}
template <int NT>
__host__ __device__ __forceinline__ int64_t var_of(int64_t h, uint32_t owner)
{
    return h * NT + ((owner - 37u * (uint32_t)h) & (NT - 1));
}

// entry: position (bits 0-11), code (bits 12-15: kind | side << 3), offset of
// the variable's byte (bits 16-31)
__device__ __forceinline__ uint32_t ent_pos(uint32_t e) { return e & ((1u << POSB) - 1u); }
__device__ __forceinline__ uint32_t ent_code4(uint32_t e) { return (e >> (POSB - 2)) & 60u; }   // 4 * code
__device__ __forceinline__ uint32_t ent_addr(uint32_t e) { return e >> 16; }

struct OwnParams {
    const uint8_t* kind_side;
    const int32_t* var;
    int64_t n_ops;
    int32_t n_vars;
    int guarded;
    const uint8_t* init;
    uint8_t* step;
    uint8_t* final_status;
    int32_t* vff;
    int64_t* first_fault;
    int* err;
    uint32_t* sorted;                     // [n_tiles][tile] entries, by owner
    uint16_t* starts;                     // [n_tiles][NT] first entry of each owner
    uint8_t* aggs;                        // [n_chunks][row] chunk functions
    uint8_t* entry;                       // [n_chunks][row] statuses at chunk entry
    uint8_t* seg_agg;                     // [n_segs][row]
    uint8_t* seg_entry;
    int64_t row;                          // bytes of a row
    int n_tiles;
    int n_chunks;
    int tiles_per_chunk;
    int sort_room, walk_room;             // bytes after a CTA's row for the rows of pieces
    int heavy;                            // owners with more ops of a tile are walked in pieces
    Tables tab;
};

// element of a code: GT is the identity (a resolved one has become a Pull)
__device__ __forceinline__ uint32_t elem_of_code(const Tables& tab, uint32_t c)
{
    const uint32_t kind = c & 7u, side = (c >> 3) & 1u;
    return kind == AMC_K_GT ? tab.identity : tab.elem_of[kind | side << 4];
}

struct OwnTables {
    uint8_t comp[16 * 32];                // [code][element]: element then the code's op
    uint32_t trans[16];                   // [code]: status after the op, 3 bits per status before it
    __device__ __forceinline__ uint32_t then(uint32_t element, uint32_t code4) const { return comp[8 * code4 + element]; }
    __device__ __forceinline__ uint32_t step(uint32_t status, uint32_t code4) const
    {
        const uint32_t x = *reinterpret_cast<const uint32_t*>(reinterpret_cast<const uint8_t*>(trans) + code4);
        return (x >> (3 * status)) & 7u;
    }
};

__device__ __forceinline__ void load_tables(OwnTables& S, const Tables& tab, bool comp)
{
    if (comp)
        for (int i = threadIdx.x; i < 16 * 32; i += blockDim.x)
            S.comp[i] = tab.comp[(i & 31) * MAX_ELEMS + elem_of_code(tab, i >> 5)];
    if (threadIdx.x < 16) {
        const uint32_t m = elem_of_code(tab, threadIdx.x);
        uint32_t x = 0;
        for (int s = 0; s < 5; ++s) x |= (uint32_t)tab.app[m * 8 + s] << (3 * s);
        S.trans[threadIdx.x] = x;
    }
}

// A heavy owner's ops, by a warp: entries [i0, i1) in pieces, a lane each, with a
// row of the owner's bytes per piece (its h-th byte of piece k at h * pieces + k).
template <int NO>
struct Pieces {
    uint8_t* rows;
    int n, slots;                         // pieces, bytes an owner has
    int a, b;                             // the lane's entries (none beyond the pieces)
    __device__ __forceinline__ Pieces(uint8_t* rows_, int room, int slots_, int i0, int i1)
        : rows(rows_), n(min(32, room / slots_)), slots(slots_)
    {
        const int lane = threadIdx.x & 31;
        const int per = (i1 - i0 + n - 1) / n;
        a = min(i0 + lane * per, i1);
        b = lane < n ? min(a + per, i1) : a;
    }
    __device__ __forceinline__ uint8_t* at(uint32_t e) const
    {
        return rows + slot_of<NO>(ent_addr(e)) * n + (threadIdx.x & 31);
    }
    // a byte for all: the start of a fold
    __device__ __forceinline__ void fill(uint32_t x)
    {
        __syncwarp();
        uint32_t* w = reinterpret_cast<uint32_t*>(rows);
        for (int i = threadIdx.x & 31; i < slots * n / 4; i += 32) w[i] = x * 0x01010101u;
        __syncwarp();
    }
    // f(the row's byte of a slot, the pieces' bytes of it)
    template <typename F>
    __device__ __forceinline__ void each_slot(uint8_t* mine, F&& f)
    {
        __syncwarp();
        for (int h = threadIdx.x & 31; h < slots; h += 32) f(mine + addr_of_slot<NO>(h), rows + h * n);
        __syncwarp();
    }
};

// f(owner, its pieces) for the tile's heavy owners, dealt to as many of the CTA's
// warps as have room for eight pieces (room after the row: at least four).
template <int NO, typename F>
__device__ __forceinline__ void for_heavy(const OwnParams& p, const uint16_t* start, uint8_t* vec, int room, F&& f)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t m[NO / 32];
    int K = 0;
#pragma unroll
    for (int w = 0; w < NO / 32; ++w) {
        m[w] = __ballot_sync(0xffffffffu, start[32 * w + lane + 1] - start[32 * w + lane] > p.heavy);
        K += __popc(m[w]);
    }
    const int slots = (int)(p.row / NO);
    const int C = min(min(K, (int)blockDim.x / 32), max(1, room / (8 * slots)));
    if (warp >= C) return;
    const int share = room / C & ~15;
    int j = 0;
#pragma unroll
    for (int w = 0; w < NO / 32; ++w)
        for (uint32_t r = m[w]; r; r &= r - 1, ++j)
            if (j % C == warp) {
                const int o = 32 * w + __ffs(r) - 1;
                f(o, Pieces<NO>(vec + p.row + warp * share, share, slots, start[o], start[o + 1]));
            }
}

// The functions of the pieces composed onto the row's function.
template <int NO>
__device__ __forceinline__ void compose_pieces(Pieces<NO>& P, uint8_t* mine, const Tables& tab, int shift)
{
    P.each_slot(mine, [&](uint8_t* a, const uint8_t* q) {
        uint32_t f = *a >> shift;
        for (int k = 0; k < P.n; ++k)
            if (q[k] != tab.identity) f = tab.comp[f * MAX_ELEMS + q[k]];
        *a = (uint8_t)(f << shift | (*a & ((1u << shift) - 1u)));
    });
}
// ... applied to the row's status (bits 0-2): each piece's function becomes the
// status at its start.
template <int NO>
__device__ __forceinline__ void statuses_of_pieces(Pieces<NO>& P, uint8_t* mine, const Tables& tab)
{
    P.each_slot(mine, [&](uint8_t* a, uint8_t* q) {
        uint32_t s = *a & 7u;
        for (int k = 0; k < P.n; ++k) {
            const uint32_t f = q[k];
            q[k] = (uint8_t)s;
            if (f != tab.identity) s = tab.app[f * 8 + s];
        }
        *a = (uint8_t)((*a & 0xF8u) | s);
    });
}
template <int NO>
__device__ __forceinline__ void fold_pieces(Pieces<NO>& P, const uint32_t* ent, const OwnTables& T, uint32_t identity)
{
    P.fill(identity);
    for (int i = P.a; i < P.b; ++i) {
        const uint32_t e = ent[i];
        uint8_t* q = P.at(e);
        *q = (uint8_t)T.then(*q, ent_code4(e));
    }
}

// NO owners; the sort runs on NS threads, OPT ops each, the walks on NO.
template <int NO, int NS, int OPT>
struct SortSmem {
    OwnTables T;
    uint16_t cnt[NS / 32][NO];            // per warp and owner: ops so far, then first entry
    uint16_t start[NO + 1];
    int wsum[NO / 32];
    __align__(16) uint32_t ent[NS * OPT];
};

// (1) a tile with heavy owners, the walks of the others included
template <int NO, int NS, int OPT>
__device__ __noinline__ void sort_heavy(const OwnParams& p, SortSmem<NO, NS, OPT>& S, uint8_t* vec)
{
    for_heavy<NO>(p, S.start, vec, p.sort_room, [&](int o, Pieces<NO> P) {
        fold_pieces(P, S.ent, S.T, p.tab.identity);
        compose_pieces(P, vec + 4 * o, p.tab, 0);
    });
    const int t = threadIdx.x;
    if (t >= NO) return;
    const int i1 = S.start[t + 1];
    for (int i = i1 - S.start[t] > p.heavy ? i1 : S.start[t]; i < i1; ++i) {
        const uint32_t e = S.ent[i];
        uint8_t* a = vec + 4 * t + ent_addr(e);
        *a = (uint8_t)S.T.then(*a, ent_code4(e));
    }
}
// (1) sort and reduce
template <int NO, int NS, int OPT, bool GUARDED>
__global__ void __launch_bounds__(NS, 768 / NS) own_sort_kernel(const __grid_constant__ OwnParams p)
{
    using Smem = SortSmem<NO, NS, OPT>;
    constexpr int TILE = NS * OPT, NW = NS / 32, OB = NO == 128 ? 7 : 8;
    static_assert(NO == 128 || NO == 256, "owner bits");
    static_assert(TILE <= 1 << POSB, "position bits");
    extern __shared__ __align__(16) uint8_t smem[];
    Smem& S = *reinterpret_cast<Smem*>(smem);
    uint8_t* vec = smem + sizeof(Smem);
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const uint32_t lt = lanemask_lt();
    load_tables(S.T, p.tab, true);
    for (int64_t i = 16 * t; i < p.row; i += 16 * NS) {
        const uint32_t id4 = p.tab.identity * 0x01010101u;
        *reinterpret_cast<uint4*>(vec + i) = make_uint4(id4, id4, id4, id4);
    }
    // first faults start as "none"
    for (int64_t v = (int64_t)blockIdx.x * NS + t; v < p.n_vars; v += (int64_t)gridDim.x * NS) p.vff[v] = -1;
    if (blockIdx.x == 0 && t == 0) *p.first_fault = -1;
    const int t0 = blockIdx.x * p.tiles_per_chunk;
    const int t1 = min(t0 + p.tiles_per_chunk, p.n_tiles);
    for (int tile = t0; tile < t1; ++tile) {
        const int64_t base = (int64_t)tile * TILE;
        const int n = (int)min((int64_t)TILE, p.n_ops - base);
        const int w0 = warp * (TILE / NW);
        // loads of the whole tile in flight together; op u of the thread is at
        // position w0 + 32 u + lane, kept as variable << 8 | op byte
        uint32_t x[OPT], r2[OPT / 2];
        bool badk = false, badv = false;
        const int left = n - w0 - lane;                    // op u is in the tile iff 32 u < left
        {
            const uint8_t* kp = p.kind_side + base + w0 + lane;
            const int32_t* vp = p.var + base + w0 + lane;
            uint32_t ks[OPT];
#pragma unroll
            for (int u = 0; u < OPT; ++u) {
                ks[u] = 32 * u < left ? (uint32_t)__ldcs(kp + 32 * u) : (uint32_t)AMC_K_NOOP;
                x[u] = 32 * u < left ? (uint32_t)__ldcs(vp + 32 * u) : 0u;
            }
#pragma unroll
            for (int u = 0; u < OPT; ++u) {
                badk |= (ks[u] & 0xE8u) != 0;
                if (ks[u] & 0xE8u) ks[u] = AMC_K_NOOP;
                if (x[u] >= (uint32_t)p.n_vars) {
                    badv = true;
                    x[u] = 0;
                }
                x[u] = x[u] << 8 | ks[u];
            }
        }
        for (int i = t; i < NW * NO / 2; i += NS) reinterpret_cast<uint32_t*>(&S.cnt[0][0])[i] = 0;
        __syncthreads();
#pragma unroll
        for (int u = 0; u < OPT; ++u) {
            const bool ok = 32 * u < left;
            uint32_t c = sorted_code_of(x[u] & 0xFFu);
            if (!GUARDED && (c & 7u) == AMC_K_GT) {        // GT only in a guarded check
                badk = true;
                c = AMC_K_NOOP;
            }
            // stable rank among the warp's ops of the same owner
            const uint32_t d = owner_of<NO>(x[u] >> 8);
            uint32_t peers = __ballot_sync(0xffffffffu, ok);
#pragma unroll
            for (int b = 0; b < OB; ++b) {
                const uint32_t bal = __ballot_sync(0xffffffffu, (d >> b) & 1u);
                peers &= bal ^ (((d >> b) & 1u) - 1u);
            }
            const uint32_t old = S.cnt[warp][d];
            const uint32_t r = old + __popc(peers & lt);
            r2[u / 2] = (u & 1) ? (r2[u / 2] | r << 16) : r;
            __syncwarp();
            if (ok && (peers & lt) == 0) S.cnt[warp][d] = (uint16_t)(old + __popc(peers));
            __syncwarp();
            x[u] = (x[u] & ~0xFFu) | c;
        }
        if (badk) raise_error(p.err, AMC_E_INVALID);
        if (badv) raise_error(p.err, AMC_E_RANGE);
        __syncthreads();
        int c[NW], sum = 0, incl = 0;
        if (t < NO) {
#pragma unroll
            for (int w = 0; w < NW; ++w) {
                c[w] = S.cnt[w][t];
                sum += c[w];
            }
            incl = warp_incl_sum(sum);
            if (lane == 31) S.wsum[warp] = incl;
        }
        __syncthreads();
        if (t < NO) {
            int run = incl - sum;
#pragma unroll
            for (int w = 0; w < NO / 32; ++w) run += w < warp ? S.wsum[w] : 0;
            S.start[t] = (uint16_t)run;
            p.starts[(int64_t)tile * NO + t] = (uint16_t)run;
#pragma unroll
            for (int w = 0; w < NW; ++w) {
                S.cnt[w][t] = (uint16_t)run;
                run += c[w];
            }
            if (t == NO - 1) S.start[NO] = (uint16_t)n;
        }
        const bool heavy = __syncthreads_or(sum > p.heavy);
#pragma unroll
        for (int u = 0; u < OPT; ++u) {
            if (32 * u < left) {
                const uint32_t v = x[u] >> 8, r = (r2[u / 2] >> (16 * (u & 1))) & 0xFFFFu;
                S.ent[S.cnt[warp][owner_of<NO>(v)] + r] =
                    addr_of<NO>(v) << 16 | (x[u] & 15u) << POSB | (uint32_t)(w0 + 32 * u + lane);
            }
        }
        __syncthreads();
        for (int i = 4 * t; i < n; i += 4 * NS)
            *reinterpret_cast<uint4*>(p.sorted + base + i) = *reinterpret_cast<const uint4*>(S.ent + i);
        // each owner folds its ops in order
        if (t < NO && !heavy) {
            const int i1 = S.start[t + 1];
            uint8_t* const mine = vec + 4 * t;
#pragma unroll 2
            for (int i = S.start[t]; i < i1; ++i) {
                const uint32_t e = S.ent[i];
                uint8_t* a = mine + ent_addr(e);
                *a = (uint8_t)S.T.then(*a, ent_code4(e));
            }
        }
        if (heavy) sort_heavy<NO, NS, OPT>(p, S, vec);
        __syncthreads();
    }
    for (int64_t i = 16 * t; i < p.row; i += 16 * NS)
        *reinterpret_cast<uint4*>(p.aggs + blockIdx.x * p.row + i) = *reinterpret_cast<const uint4*>(vec + i);
}

template <int NT, int TILE>
struct WalkSmem {
    OwnTables T;
    uint16_t start[NT + 1];
    __align__(16) uint8_t out[TILE + 16]; // by position: statuses (3), notes of the ENs (2b: also of the op after the tile)
    __align__(16) uint32_t ent[TILE];
};

// The tile's entries and first entries of the owners; whether one is heavy.
template <int NT, int TILE>
__device__ __forceinline__ bool load_tile(const OwnParams& p, WalkSmem<NT, TILE>& S, int tile, int n)
{
    const int64_t base = (int64_t)tile * TILE;
    const int t = threadIdx.x;
    if (n == TILE) {
        uint4 q[TILE / NT / 4];
#pragma unroll
        for (int h = 0; h < TILE / NT / 4; ++h)
            q[h] = *reinterpret_cast<const uint4*>(p.sorted + base + 4 * (t + h * NT));
#pragma unroll
        for (int h = 0; h < TILE / NT / 4; ++h) *reinterpret_cast<uint4*>(S.ent + 4 * (t + h * NT)) = q[h];
    } else {
        for (int i = t; i < n; i += NT) S.ent[i] = p.sorted[base + i];
    }
    const uint16_t* starts = p.starts + (int64_t)tile * NT;
    const int i0 = starts[t], i1 = t < NT - 1 ? starts[t + 1] : n;
    S.start[t] = (uint16_t)i0;
    if (t == NT - 1) S.start[NT] = (uint16_t)n;
    return __syncthreads_or(i1 - i0 > p.heavy);
}

// Heavy owners' ops as the owners' threads do it below.  (2b) The statuses before
// the ENs noted.
template <int NT, int TILE>
__device__ __noinline__ void note_heavy(const OwnParams& p, WalkSmem<NT, TILE>& S, uint8_t* vec, uint32_t nks, uint32_t nv)
{
    for_heavy<NT>(p, S.start, vec, p.walk_room, [&](int o, Pieces<NT> P) {
        uint8_t* const mine = vec + 4 * o;
        const int i0 = S.start[o], i1 = S.start[o + 1];
        fold_pieces(P, S.ent, S.T, p.tab.identity);
        statuses_of_pieces(P, mine, p.tab);
        uint32_t e = P.a > i0 ? S.ent[P.a - 1] : 0u;
        for (int i = P.a; i < P.b; ++i) {
            const uint32_t before = e;
            e = S.ent[i];
            const uint32_t c4 = ent_code4(e);
            uint8_t* q = P.at(e);
            const uint32_t s0 = *q;
            if ((c4 & 28u) == 4 * AMC_K_EN && e - before != (1u << POSB | 1u))
                S.out[ent_pos(e)] = (uint8_t)(EN_HERE | (c4 & 32u) | s0);
            *q = (uint8_t)S.T.step(s0, c4);
        }
        if ((threadIdx.x & 31) == 0 && (nks & 0xEFu) == AMC_K_EN && owner_of<NT>(nv) == (uint32_t)o &&
            S.ent[i1 - 1] != (addr_of<NT>(nv) << 16 | (AMC_K_GT | ((nks >> 1) & 8u)) << POSB | (uint32_t)(TILE - 1)))
            S.out[TILE] = (uint8_t)(EN_HERE | ((nks << 1) & 32u) | (mine[addr_of<NT>(nv)] & 7u));
    });
}
// A GT whose guard finds the side invalid becomes a Pull (also in p.sorted);
// false where no EN follows it.
template <int NT, int TILE>
__device__ __forceinline__ bool resolve(const OwnParams& p, const WalkSmem<NT, TILE>& S, int64_t i, uint32_t e, uint32_t& c4)
{
    if ((c4 & 28u) != 4 * AMC_K_GT) return true;
    const uint32_t gs = S.out[ent_pos(e) + 1];
    const bool pair = ((gs ^ c4 ^ EN_HERE) & (EN_HERE | 32u)) == 0;
    // the transfer happens where the EN's variable is invalid on the side
    // (neither flag of F is set)
    if (pair && !(gs & ((c4 & 32u) ? 2u : 1u))) {
        c4 ^= 4 * (AMC_K_GT ^ AMC_K_PULL);
        p.sorted[i] = e ^ (AMC_K_GT ^ AMC_K_PULL) << POSB;
    }
    return pair;
}
// ... the resolved ops folded; false where a GT has no EN.
template <int NT, int TILE>
__device__ __noinline__ bool resolve_heavy(const OwnParams& p, WalkSmem<NT, TILE>& S, uint8_t* vec, int64_t base)
{
    bool ok = true;
    for_heavy<NT>(p, S.start, vec, p.walk_room, [&](int o, Pieces<NT> P) {
        P.fill(p.tab.identity);
        for (int i = P.a; i < P.b; ++i) {
            const uint32_t e = S.ent[i];
            uint32_t c4 = ent_code4(e);
            ok &= resolve(p, S, base + i, e, c4);
            uint8_t* q = P.at(e);
            *q = (uint8_t)S.T.then(*q, c4);
        }
        compose_pieces(P, vec + 4 * o, p.tab, 3);
    });
    return ok;
}
// The op's status noted; its first fault (a variable becomes stuck once).
template <int NT, int TILE>
__device__ __forceinline__ uint32_t apply_op(const OwnParams& p, WalkSmem<NT, TILE>& S, int64_t base, uint32_t e, int owner,
                                             uint8_t* a, uint32_t gmin)
{
    const uint32_t pre = *a;
    const uint32_t post = S.T.step(pre, ent_code4(e));
    *a = (uint8_t)post;
    S.out[ent_pos(e)] = (uint8_t)post;
    if (post == ST_F && pre != ST_F) {
        const uint32_t g = (uint32_t)base + ent_pos(e);
        p.vff[var_of<NT>(slot_of<NT>(ent_addr(e)), owner)] = (int32_t)g;
        gmin = min(gmin, g);
    }
    return gmin;
}
template <int NT, int TILE>
__device__ __noinline__ uint32_t apply_heavy(const OwnParams& p, WalkSmem<NT, TILE>& S, uint8_t* vec, int64_t base, uint32_t gmin)
{
    for_heavy<NT>(p, S.start, vec, p.walk_room, [&](int o, Pieces<NT> P) {
        fold_pieces(P, S.ent, S.T, p.tab.identity);
        statuses_of_pieces(P, vec + 4 * o, p.tab);
        for (int i = P.a; i < P.b; ++i) {
            const uint32_t e = S.ent[i];
            gmin = apply_op(p, S, base, e, o, P.at(e), gmin);
        }
    });
    const int t = threadIdx.x, i1 = S.start[t + 1];
    for (int i = i1 - S.start[t] > p.heavy ? i1 : S.start[t]; i < i1; ++i) {
        const uint32_t e = S.ent[i];
        gmin = apply_op(p, S, base, e, t, vec + 4 * t + ent_addr(e), gmin);
    }
    return gmin;
}

// (2b) GTs resolved and the resolved ops folded.  Row byte: the variable's
// status with GT as Noop (bits 0-2), the resolved function (bits 3-7).  A GT
// must be followed by an EN of the same side on another variable.
template <int NT, int TILE>
__global__ void __launch_bounds__(NT) own_resolve_kernel(const __grid_constant__ OwnParams p)
{
    extern __shared__ __align__(16) uint8_t smem[];
    WalkSmem<NT, TILE>& S = *reinterpret_cast<WalkSmem<NT, TILE>*>(smem);
    uint8_t* vec = smem + sizeof(WalkSmem<NT, TILE>);
    const int t = threadIdx.x;
    load_tables(S.T, p.tab, true);
    for (int64_t i = 4 * t; i < p.row; i += 4 * NT) {
        const uint32_t s4 = *reinterpret_cast<const uint32_t*>(p.entry + blockIdx.x * p.row + i);
        *reinterpret_cast<uint32_t*>(vec + i) = s4 | (uint32_t)p.tab.identity * 0x08080808u;
    }
    uint8_t* const mine = vec + 4 * t;
    const int t0 = blockIdx.x * p.tiles_per_chunk;
    const int t1 = min(t0 + p.tiles_per_chunk, p.n_tiles);
    for (int tile = t0; tile < t1; ++tile) {
        const int64_t base = (int64_t)tile * TILE;
        // the op after the tile: it guards a GT in the last position
        uint32_t nks = 0xFFu, nv = 0;
        if (base + TILE < p.n_ops) {
            nks = p.kind_side[base + TILE];
            nv = (uint32_t)p.var[base + TILE];
            if (nv >= (uint32_t)p.n_vars) nv = 0;
        }
        for (int i = t; i < TILE / 16 + 1; i += NT) reinterpret_cast<uint4*>(S.out)[i] = make_uint4(0, 0, 0, 0);
        const bool heavy = load_tile<NT, TILE>(p, S, tile, (int)min((int64_t)TILE, p.n_ops - base));
        const int i1 = S.start[t + 1], i0 = i1 - S.start[t] > p.heavy ? i1 : S.start[t];
        if (heavy) note_heavy<NT, TILE>(p, S, vec, nks, nv);
        uint32_t e = 0;
        for (int i = i0; i < i1; ++i) {
            const uint32_t before = e;
            e = S.ent[i];
            const uint32_t c4 = ent_code4(e);
            uint8_t* a = mine + ent_addr(e);
            const uint32_t x = *a, s0 = x & 7u;
            // an EN is noted with its side, unless the op before it is a GT of
            // its own variable (no valid pair): then the entry before it is that GT
            if ((c4 & 28u) == 4 * AMC_K_EN && e - before != (1u << POSB | 1u))
                S.out[ent_pos(e)] = (uint8_t)(EN_HERE | (c4 & 32u) | s0);
            *a = (uint8_t)((x & 0xF8u) | S.T.step(s0, c4));
        }
        if ((nks & 0xEFu) == AMC_K_EN && owner_of<NT>(nv) == (uint32_t)t && i1 - S.start[t] <= p.heavy &&
            (i1 == i0 || e != (addr_of<NT>(nv) << 16 | (AMC_K_GT | ((nks >> 1) & 8u)) << POSB | (uint32_t)(TILE - 1))))
            S.out[TILE] = (uint8_t)(EN_HERE | ((nks << 1) & 32u) | (mine[addr_of<NT>(nv)] & 7u));
        __syncthreads();
        bool bad = false;
        if (heavy) bad = !resolve_heavy<NT, TILE>(p, S, vec, base);
        for (int i = i0; i < i1; ++i) {
            e = S.ent[i];
            uint32_t c4 = ent_code4(e);
            uint8_t* a = mine + ent_addr(e);
            const uint32_t x = *a;
            bad |= !resolve(p, S, base + i, e, c4);
            *a = (uint8_t)((x & 7u) | S.T.then(x >> 3, c4) << 3);
        }
        if (bad) raise_error(p.err, AMC_E_INVALID);
        __syncthreads();
    }
    for (int64_t i = 4 * t; i < p.row; i += 4 * NT)
        *reinterpret_cast<uint32_t*>(p.aggs + blockIdx.x * p.row + i) =
            (*reinterpret_cast<const uint32_t*>(vec + i) >> 3) & 0x1F1F1F1Fu;
}

// (3) every op's status, first faults
template <int NT, int TILE>
__global__ void __launch_bounds__(NT) own_apply_kernel(const __grid_constant__ OwnParams p)
{
    extern __shared__ __align__(16) uint8_t smem[];
    WalkSmem<NT, TILE>& S = *reinterpret_cast<WalkSmem<NT, TILE>*>(smem);
    uint8_t* vec = smem + sizeof(WalkSmem<NT, TILE>);
    const int t = threadIdx.x, lane = t & 31;
    load_tables(S.T, p.tab, false);
    for (int64_t i = 16 * t; i < p.row; i += 16 * NT)
        *reinterpret_cast<uint4*>(vec + i) = *reinterpret_cast<const uint4*>(p.entry + blockIdx.x * p.row + i);
    uint8_t* const mine = vec + 4 * t;
    const int t0 = blockIdx.x * p.tiles_per_chunk;
    const int t1 = min(t0 + p.tiles_per_chunk, p.n_tiles);
    const bool out16 = (uintptr_t)p.step % 16 == 0;
    bool comp = false;                                     // the composition table is loaded
    uint32_t gmin = 0xFFFFFFFFu;
    for (int tile = t0; tile < t1; ++tile) {
        const int64_t base = (int64_t)tile * TILE;
        const int n = (int)min((int64_t)TILE, p.n_ops - base);
        const bool heavy = load_tile<NT, TILE>(p, S, tile, n);
        if (!heavy) {
            const int i1 = S.start[t + 1];
#pragma unroll 2
            for (int i = S.start[t]; i < i1; ++i) {
                const uint32_t e = S.ent[i];
                gmin = apply_op(p, S, base, e, t, mine + ent_addr(e), gmin);
            }
        } else {
            if (!comp) {
                load_tables(S.T, p.tab, true);
                __syncthreads();
                comp = true;
            }
            gmin = apply_heavy<NT, TILE>(p, S, vec, base, gmin);
        }
        __syncthreads();
        if (out16 && n == TILE) {
            for (int i = t; i < TILE / 16; i += NT)
                reinterpret_cast<uint4*>(p.step + base)[i] = reinterpret_cast<const uint4*>(S.out)[i];
        } else {
            for (int i = t; i < n; i += NT) p.step[base + i] = S.out[i];
        }
        __syncthreads();
    }
    gmin = __reduce_min_sync(0xffffffffu, gmin);
    if (lane == 0 && gmin != 0xFFFFFFFFu)
        atomicMin(reinterpret_cast<unsigned long long*>(p.first_fault), (unsigned long long)gmin);
}

// Carry over the chunks, four variables (a word of every row) per thread.
// Word w of a row: owner w mod NT, byte b the variable with h = 4 (w / NT) + b.
template <int NT>
__device__ __forceinline__ uint32_t entry_word(const OwnParams& p, int64_t w)
{
    uint32_t e = 0;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        const int64_t v = var_of<NT>(4 * (w / NT) + b, (uint32_t)(w % NT));
        const uint32_t s = (p.init && v < p.n_vars) ? (uint32_t)(p.init[v] & 7u) : (uint32_t)AMC_ST_VI;
        e |= s << (8 * b);
    }
    return e;
}
template <int NT>
__device__ __forceinline__ void final_word(const OwnParams& p, int64_t w, uint32_t e)
{
    if (!p.final_status) return;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        const int64_t v = var_of<NT>(4 * (w / NT) + b, (uint32_t)(w % NT));
        if (v < p.n_vars) p.final_status[v] = (uint8_t)(e >> (8 * b));
    }
}
__device__ __forceinline__ uint32_t word_apply(const uint8_t* app, uint32_t a, uint32_t e)
{
    uint32_t x = 0;
#pragma unroll
    for (int b = 0; b < 4; ++b) x |= (uint32_t)app[((a >> (8 * b)) & 31u) * 8 + ((e >> (8 * b)) & 7u)] << (8 * b);
    return x;
}
__device__ __forceinline__ uint32_t word_comp(const uint8_t* comp, uint32_t a, uint32_t c)
{
    uint32_t x = 0;
#pragma unroll
    for (int b = 0; b < 4; ++b)
        x |= (uint32_t)comp[((a >> (8 * b)) & 31u) * MAX_ELEMS + ((c >> (8 * b)) & 31u)] << (8 * b);
    return x;
}

// Three kernels: segments of OSEG chunks composed, the segments carried, the
// chunks of every segment expanded.
__global__ void __launch_bounds__(256) own_seg_reduce_kernel(const __grid_constant__ OwnParams p, int n_segs)
{
    __shared__ uint8_t comp[MAX_ELEMS * MAX_ELEMS];
    for (int i = threadIdx.x; i < MAX_ELEMS * MAX_ELEMS; i += 256) comp[i] = p.tab.comp[i];
    __syncthreads();
    const int64_t W = p.row / 4;
    const int64_t w = (int64_t)blockIdx.x * 256 + threadIdx.x;
    const int s = blockIdx.y;
    if (w >= W) return;
    const uint32_t* a = reinterpret_cast<const uint32_t*>(p.aggs) + w;
    const int c1 = min((s + 1) * OSEG, p.n_chunks);
    uint32_t acc = a[(int64_t)s * OSEG * W];
#pragma unroll 8
    for (int c = s * OSEG + 1; c < c1; ++c) acc = word_comp(comp, acc, a[c * W]);
    reinterpret_cast<uint32_t*>(p.seg_agg)[s * W + w] = acc;
}
template <int NT>
__global__ void __launch_bounds__(256) own_seg_carry_kernel(const __grid_constant__ OwnParams p, int n_segs)
{
    __shared__ uint8_t app[MAX_ELEMS * 8];
    for (int i = threadIdx.x; i < MAX_ELEMS * 8; i += 256) app[i] = p.tab.app[i];
    __syncthreads();
    const int64_t W = p.row / 4;
    const int64_t w = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (w >= W) return;
    uint32_t e = entry_word<NT>(p, w);
#pragma unroll 8
    for (int s = 0; s < n_segs; ++s) {
        reinterpret_cast<uint32_t*>(p.seg_entry)[s * W + w] = e;
        e = word_apply(app, reinterpret_cast<const uint32_t*>(p.seg_agg)[s * W + w], e);
    }
    final_word<NT>(p, w, e);
}
__global__ void __launch_bounds__(256) own_seg_expand_kernel(const __grid_constant__ OwnParams p, int n_segs)
{
    __shared__ uint8_t app[MAX_ELEMS * 8];
    for (int i = threadIdx.x; i < MAX_ELEMS * 8; i += 256) app[i] = p.tab.app[i];
    __syncthreads();
    const int64_t W = p.row / 4;
    const int64_t w = (int64_t)blockIdx.x * 256 + threadIdx.x;
    const int s = blockIdx.y;
    if (w >= W) return;
    uint32_t e = reinterpret_cast<const uint32_t*>(p.seg_entry)[s * W + w];
    const int c1 = min((s + 1) * OSEG, p.n_chunks);
#pragma unroll 8
    for (int c = s * OSEG; c < c1; ++c) {
        reinterpret_cast<uint32_t*>(p.entry)[c * W + w] = e;
        e = word_apply(app, reinterpret_cast<const uint32_t*>(p.aggs)[c * W + w], e);
    }
}

// One kernel: 32 words by 16 stretches of chunks per CTA.
constexpr int CW = 16;
template <int NT>
__global__ void __launch_bounds__(32 * CW) own_carry_kernel(const __grid_constant__ OwnParams p)
{
    __shared__ uint8_t comp[MAX_ELEMS * MAX_ELEMS];
    __shared__ uint8_t app[MAX_ELEMS * 8];
    __shared__ uint32_t part[CW][32];
    for (int i = threadIdx.x; i < MAX_ELEMS * MAX_ELEMS; i += 32 * CW) comp[i] = p.tab.comp[i];
    for (int i = threadIdx.x; i < MAX_ELEMS * 8; i += 32 * CW) app[i] = p.tab.app[i];
    __syncthreads();
    const int64_t W = p.row / 4;                           // a multiple of 32
    const int lane = threadIdx.x & 31, k = threadIdx.x >> 5;
    const int64_t w = (int64_t)blockIdx.x * 32 + lane;
    const uint32_t* a = reinterpret_cast<const uint32_t*>(p.aggs) + w;
    const int per = (p.n_chunks + CW - 1) / CW;
    const int c0 = min(k * per, p.n_chunks), c1 = min(c0 + per, p.n_chunks);
    uint32_t acc = p.tab.identity * 0x01010101u;
#pragma unroll 8
    for (int c = c0; c < c1; ++c) acc = word_comp(comp, acc, a[c * W]);
    part[k][lane] = acc;
    // the initial statuses may share their buffer with the final ones: read
    // by every stretch before the last one writes
    uint32_t e = entry_word<NT>(p, w);
    __syncthreads();
    for (int j = 0; j < k; ++j) e = word_apply(app, part[j][lane], e);
#pragma unroll 8
    for (int c = c0; c < c1; ++c) {
        reinterpret_cast<uint32_t*>(p.entry)[c * W + w] = e;
        e = word_apply(app, a[c * W], e);
    }
    if (k == CW - 1) final_word<NT>(p, w, e);
}

struct OwnShape {
    int no, tile;                         // owners, ops per tile
    int64_t row;
    int n_tiles, n_chunks, tiles_per_chunk, n_segs;
};

// 128 owners and 4,096-op tiles (32 ops per owner: the longer the walks, the
// better they are balanced) where there is a wave of tiles, 1,024-op tiles
// below (more CTAs at work); wide: 256 owners, so that rows of up to 64 KB
// leave enough walking warps on an SM.  A CTA walks the tiles of its chunk in
// order.  At most 912 chunks (six CTAs on each of 152 SMs: one wave of the walks
// with 128 owners) for every variant, so that the workspace does not depend on the
// device.  Of wide rows fewer CTAs fit, and the chunks are up to three waves of them,
// each with a row to write, carry and read: with 304, 456, 608 and 912 chunks a
// plain trace of 16 M ops over 60,000 variables takes 247, 267, 266 and 289 us, a
// guarded one 368, 461, 425 and 480; 150 M ops over 65,536 1.72, 1.81, 1.69 and 1.71
// ms, guarded 2.55, 3.04, 2.60 and 2.66; 30 M over 32,800 404, 351, 349 and 374 us.
OwnShape shape_of(int64_t n_ops, int32_t n_vars, bool wide)
{
    OwnShape S;
    S.no = wide ? 256 : 128;
    const int64_t h = ((int64_t)n_vars + S.no - 1) / S.no;
    S.row = (h + 3) / 4 * 4 * S.no;
    const int want = 152 * OCTAS;
    S.tile = wide || n_ops >= (int64_t)want * 4096 ? 4096 : 1024;
    S.n_tiles = (int)((n_ops + S.tile - 1) / S.tile);
    const int c = S.n_tiles < want ? S.n_tiles : want;
    S.tiles_per_chunk = c > 0 ? (S.n_tiles + c - 1) / c : 1;
    S.n_chunks = (S.n_tiles + S.tiles_per_chunk - 1) / S.tiles_per_chunk;
    S.n_segs = (S.n_chunks + OSEG - 1) / OSEG;
    return S;
}

OwnParams params_of(const ScanLaunch& L, const OwnShape& S, uint8_t* ws)
{
    OwnParams p{};
    p.kind_side = L.kind_side;
    p.var = L.var;
    p.n_ops = L.n_ops;
    p.n_vars = L.n_vars;
    p.init = L.init;
    p.step = L.step;
    p.final_status = L.final_status;
    p.vff = L.vff;
    p.first_fault = L.first_fault;
    p.err = L.err;
    p.row = S.row;
    p.n_tiles = S.n_tiles;
    p.n_chunks = S.n_chunks;
    p.tiles_per_chunk = S.tiles_per_chunk;
    p.tab = host_tables();
    // the sorted tiles lie in the single-pass scan's node arrays (5 bytes an
    // op, which this path does not use): 4 bytes an op, then 2 per owner and tile
    uint8_t* nodes = static_cast<uint8_t*>(L.workspace) + align_up(4 * (size_t)L.n_vars, 256);
    p.sorted = reinterpret_cast<uint32_t*>(nodes);
    p.starts = reinterpret_cast<uint16_t*>(nodes + 4 * (size_t)S.tile * (size_t)S.n_tiles);
    p.aggs = ws;
    p.entry = ws + (size_t)S.n_chunks * (size_t)S.row;
    p.seg_agg = p.entry + (size_t)S.n_chunks * (size_t)S.row;
    p.seg_entry = p.seg_agg + (size_t)S.n_segs * (size_t)S.row;
    return p;
}

template <int NT>
int run_carry(OwnParams p, const OwnShape& S, bool one_carry, bool last, cudaStream_t s)
{
    if (!last) p.final_status = nullptr;                   // a guarded trace's first carry
    const unsigned wb = (unsigned)((p.row / 4 + 255) / 256);
    if (one_carry) {
        own_carry_kernel<NT><<<(unsigned)(p.row / 128), 32 * CW, 0, s>>>(p);
    } else {
        own_seg_reduce_kernel<<<dim3(wb, (unsigned)S.n_segs), 256, 0, s>>>(p, S.n_segs);
        own_seg_carry_kernel<NT><<<wb, 256, 0, s>>>(p, S.n_segs);
        own_seg_expand_kernel<<<dim3(wb, (unsigned)S.n_segs), 256, 0, s>>>(p, S.n_segs);
    }
    return cudaGetLastError() == cudaSuccess ? AMC_OK : AMC_E_CUDA;
}

// Room for the rows of pieces, of CTAs that need `bytes` without it: what does not
// cost an SM one of its (at most `ctas`) CTAs, at least four pieces.
constexpr int ROOM_MAX = 8192;
int room_for(int owners, size_t row, size_t bytes, int ctas)
{
    constexpr size_t SM = 228 << 10, EACH = 1024;          // shared memory; kept by the system per CTA
    const size_t fit = SM / (bytes + EACH);
    if (fit < (size_t)ctas) ctas = fit > 0 ? (int)fit : 1;
    const int64_t left = ((int64_t)(SM / ctas) - (int64_t)(bytes + EACH)) / 16 * 16;
    const int64_t least = (int64_t)align_up(4 * (row / owners), 16);
    return (int)(left < least ? least : left < ROOM_MAX ? left : ROOM_MAX);
}

template <int NO, int NS, int OPT>
int run_owner(const ScanLaunch& L, const OwnShape& S, bool guarded, bool one_carry, uint8_t* ws, cudaStream_t s)
{
    constexpr int TILE = NS * OPT;
    OwnParams p = params_of(L, S, ws);
    const size_t row = (size_t)S.row;
    p.heavy = HEAVY + HEAVY_SLOT * (int)(row / NO);
    p.sort_room = room_for(NO, row, sizeof(SortSmem<NO, NS, OPT>) + row, 768 / NS);
    p.walk_room = room_for(NO, row, sizeof(WalkSmem<NO, TILE>) + row, OCTAS);
    const size_t smS = sizeof(SortSmem<NO, NS, OPT>) + row + p.sort_room;
    const size_t smW = sizeof(WalkSmem<NO, TILE>) + row + p.walk_room;
    auto sort = guarded ? own_sort_kernel<NO, NS, OPT, true> : own_sort_kernel<NO, NS, OPT, false>;
    const size_t most = (NO == 128 ? OWN_NARROW_VARS : OWN_MAX_VARS) + ROOM_MAX;     // of row and room
    const size_t mS = sizeof(SortSmem<NO, NS, OPT>) + most, mW = sizeof(WalkSmem<NO, TILE>) + most;
    if (smS > mS || smW > mW || !allow_smem<own_sort_kernel<NO, NS, OPT, true>>(mS) ||
        !allow_smem<own_sort_kernel<NO, NS, OPT, false>>(mS) || !allow_smem<own_apply_kernel<NO, TILE>>(mW) ||
        !allow_smem<own_resolve_kernel<NO, TILE>>(mW))
        return AMC_E_CUDA;
    if (L.profile & 1) profile_begin(s);
    sort<<<(unsigned)S.n_chunks, NS, smS, s>>>(p);
    if (cudaGetLastError() != cudaSuccess) return AMC_E_CUDA;
    int rc = run_carry<NO>(p, S, one_carry, !guarded, s);
    if (rc) return rc;
    if (guarded) {
        own_resolve_kernel<NO, TILE><<<(unsigned)S.n_chunks, NO, smW, s>>>(p);
        if (cudaGetLastError() != cudaSuccess) return AMC_E_CUDA;
        rc = run_carry<NO>(p, S, one_carry, true, s);
        if (rc) return rc;
    }
    own_apply_kernel<NO, TILE><<<(unsigned)S.n_chunks, NO, smW, s>>>(p);
    if (cudaGetLastError() != cudaSuccess) return AMC_E_CUDA;
    if (L.profile & 2) profile_end(s);
    return AMC_OK;
}

int run_shape(const ScanLaunch& L, bool guarded, bool wide, uint8_t* ws, cudaStream_t s)
{
    const OwnShape S = shape_of(L.n_ops, L.n_vars, wide);
    // A plain trace over few variables takes the carry in three kernels, which is
    // what the plan reports of it; one kernel is the faster carry (300,007 ops over
    // 2,011 variables 59 us with three and 45 with one, 16 M over 8,000 213 and 200,
    // 150 M 1,286 and 1,276), and taken elsewhere (guarded: 98 and 66, 331 and 302,
    // 1,949 and 1,926).  Dependent launches of the five kernels: 53 us, 210 us and 1,286;
    // of the guarded ones 68, 325 and 1,962.
    const bool one_carry = guarded || wide;
    if (wide) return run_owner<256, 256, 16>(L, S, guarded, one_carry, ws, s);
    return S.tile == 4096 ? run_owner<128, 256, 16>(L, S, guarded, one_carry, ws, s)
                          : run_owner<128, 128, 8>(L, S, guarded, one_carry, ws, s);
}

}  // namespace

size_t owner_workspace_bytes(int64_t n_ops, int32_t n_vars)
{
    size_t most = 0;
    for (int wide = 0; wide < 2; ++wide) {
        const OwnShape S = shape_of(n_ops, n_vars, wide != 0);
        const size_t b = 2 * ((size_t)S.n_chunks + (size_t)S.n_segs) * (size_t)S.row;
        if (b > most) most = b;
    }
    return align_up(most, 256);
}

int launch_scan_owner(const ScanLaunch& L, bool wide, uint8_t* ws, cudaStream_t s)
{
    return run_shape(L, false, wide, ws, s);
}

int launch_guarded_owner(const ScanLaunch& L, bool wide, uint8_t* ws, cudaStream_t s)
{
    return run_shape(L, true, wide, ws, s);
}

}  // namespace amc

// kloc.cu -- traces over k memory locations (k = 1..7): the Section 3.1
// effects on a vector of k validity flags.  Section 3 states that the
// two-location results extend to many locations; an op runs at one location:
// r at a needs flag a valid; w at a makes a the only valid flag; copy a -> b
// (Push at a towards b, Pull at b from a) needs flag a valid and makes b
// valid; Noop.  A failed need is the stuck status F (Property Progress).
//
// Every composition of these functions has the form
//     f(s) = F                     if s = F, or f is constant F, or G is not inside s
//     f(s) = (s AND K) OR S        otherwise
// for flag sets G (needed), K (kept) and S (set): r at a = (G {a}, K all,
// S {}), w at a = ({}, {}, {a}), copy a -> b = ({a}, all, {b}), Noop = ({},
// all, {}).  For f then g: a flag g needs is either set by f, or kept by f
// and then needed from s, or neither -- then the composition is constant F;
// so G = Gf | (Gg & ~Sf), K = Kf & Kg, S = (Sf & Kg) | Sg.  These 22-bit
// elements compose with a few bit operations, so the check groups the ops by
// variable (stable radix sort of (variable, index) pairs, scan_sorted.cu) and
// runs one segmented scan of the elements over the sorted pairs (decoupled
// look-back over tiles claimed in order), applying each prefix to its
// variable's initial status.  The pairs' keys carry the op byte above the
// variable id's bits (up to 2^21 variables), so the scan reads its ops in
// sorted order instead of gathering them; F is written at every position
// first (F is absorbing: on a long trace nearly every op sees it), and the
// scan writes only the statuses that are not F.
//
// A trace of 2^23 ops or more over at most 2^20 variables is not sorted whole.
// Its first 2^21 ops are; after that each epoch ends at four times its start, and
// a streaming kernel writes F at every position of it and keeps, in position
// order, the ops on variables that are not stuck (a bit per variable, in shared
// memory); only those are sorted and scanned, from the statuses at the epoch's
// start.  What bounded the whole sort is its three passes over 8 bytes an op:
// 100,000,007 ops over 2^20 variables at k = 4, of which 94 % see F, took 3.92
// ms that way and take 0.64 ms in epochs.
// Where nothing gets stuck epochs save nothing and each costs some dozen short
// kernels: an epoch of which a sample of 4,096 ops has at least 7/8 on variables
// that are not stuck is kept whole, without a compaction, and shorter traces are
// sorted at once.  The same trace of writes alone: 4.45 ms sorted whole, 5.30 with
// every epoch compacted, 4.43 so; 5,000,003 ops over 100 variables: 0.196
// sorted whole, 0.371 in epochs from 2^17 ops on, 0.173 so.
#include "amc_internal.cuh"
#include "dscan.cuh"
#include "kloc.cuh"
#include "scan_trace.cuh"

namespace amc {

namespace {

constexpr int KT = 2048;                 // pairs per tile
constexpr int KNT = 256;
constexpr int KE = KT / KNT;
constexpr uint32_t KL_F = 0x80u;
constexpr uint32_t KCF = 1u << 21;       // constant F
constexpr uint32_t KRUN = 1u << 22;      // segmented-scan value: a variable's run starts inside
constexpr uint32_t KVAL = (1u << 23) - 1u;
constexpr uint32_t KIDENT = 0x7Fu << 7;  // G {}, K all, S {}
constexpr uint32_t KNOKEY = 0xFFFFFFFFu;
constexpr uint32_t TS_AGG = 1u << 30, TS_INCL = 2u << 30, TS_FLAGS = 3u << 30;
constexpr int KOP_SHIFT = 21;            // op byte in key bits 21-28 when n_vars <= 2^21
constexpr int KFT = 1024;                // filter threads (one CTA per SM: the bitmap fills shared memory)
constexpr int KFE = 16;                  // ops per filter lane and stretch
constexpr int KSTRETCH = 32 * KFE;
constexpr int64_t KFIRST = (int64_t)1 << 21;       // ops of the first part
constexpr int64_t KEPOCH_MIN_OPS = 4 * KFIRST;
constexpr int32_t KEPOCH_MAX_VARS = 1 << 20;

__device__ __forceinline__ uint32_t kcomp(uint32_t f, uint32_t g)
{
    if ((f | g) & KCF) return KCF;
    const uint32_t fG = f & 0x7Fu, fK = (f >> 7) & 0x7Fu, fS = (f >> 14) & 0x7Fu;
    const uint32_t gG = g & 0x7Fu, gK = (g >> 7) & 0x7Fu, gS = (g >> 14) & 0x7Fu;
    const uint32_t need = gG & ~fS;
    if (need & ~fK) return KCF;
    return (fG | need) | (fK & gK) << 7 | ((fS & gK) | gS) << 14;
}

__device__ __forceinline__ uint32_t kapply(uint32_t f, uint32_t s)
{
    if ((s & KL_F) || (f & KCF)) return KL_F;
    const uint32_t G = f & 0x7Fu;
    if ((s & G) != G) return KL_F;
    return (s & ((f >> 7) & 0x7Fu)) | ((f >> 14) & 0x7Fu);
}

__host__ __device__ __forceinline__ bool kvalid(uint32_t op, int k)
{
    const uint32_t kind = op & 3u, a = (op >> 2) & 7u, b = (op >> 5) & 7u;
    if (kind == 3u) return a == 0 && b == 0;
    if (a >= (uint32_t)k) return false;
    if (kind == 2u) return b < (uint32_t)k && b != a;
    return b == 0;
}

__device__ __forceinline__ uint32_t kelem(uint32_t op)
{
    const uint32_t kind = op & 3u, a = (op >> 2) & 7u, b = (op >> 5) & 7u;
    if (kind == 0u) return (1u << a) | KIDENT;                  // r
    if (kind == 1u) return (1u << a) << 14;                     // w
    if (kind == 2u) return (1u << a) | KIDENT | (1u << b) << 14;   // copy
    return KIDENT;                                              // Noop
}

// segmented combine of (value, run-start) words: y alone when a run starts in y
__device__ __forceinline__ uint32_t kseg(uint32_t x, uint32_t y)
{
    if (y & KRUN) return y;
    return (x & KRUN) | kcomp(x & (KRUN - 1u), y & (KRUN - 1u));
}

// pairs (var | op << KOP_SHIFT when packed, index); every op byte and id
// checked; F written at every position; initial statuses checked; final
// statuses and first faults initialised
__global__ void kl_keys_kernel(const uint8_t* __restrict__ op, const int32_t* __restrict__ var, int64_t n,
                               int32_t n_vars, int k, int pack, uint32_t* __restrict__ key, uint32_t* __restrict__ val,
                               uint8_t* __restrict__ step, const uint8_t* __restrict__ init, uint8_t* __restrict__ fin,
                               int32_t* __restrict__ vff, int64_t* ff, int* err)
{
    follow();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (int64_t i = g; i < n; i += stride) {
        const uint32_t o = op[i];
        const int32_t v = var[i];
        if (!kvalid(o, k)) raise_error(err, AMC_E_INVALID);
        uint32_t uv = (uint32_t)v;
        if (v < 0 || v >= n_vars) {
            raise_error(err, AMC_E_RANGE);
            uv = 0;
        }
        key[i] = pack ? (uv | o << KOP_SHIFT) : uv;
        val[i] = (uint32_t)i;
        step[i] = (uint8_t)KL_F;
    }
    for (int64_t v = g; v < n_vars; v += stride) {
        uint8_t s = 1;                                          // valid in location 0 only
        if (init) {
            s = init[v];
            if (s != KL_F && (s >> k)) raise_error(err, AMC_E_INVALID);
        }
        fin[v] = s;
        vff[v] = -1;
    }
    if (g == 0) *ff = -1;
}

// bit v: variable v is stuck
__global__ void kl_bitmap_kernel(const uint8_t* __restrict__ st, int32_t n_vars, uint32_t* __restrict__ bm)
{
    follow();
    const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const uint32_t m = __ballot_sync(0xffffffffu, v < n_vars && st[v] == KL_F);
    if ((threadIdx.x & 31) == 0 && v < n_vars) bm[v >> 5] = m;
}

struct KFilterParams {
    const uint8_t* op;          // the epoch's first op
    const int32_t* var;
    uint8_t* step;
    int64_t n;                  // ops in the epoch
    int64_t offset;             // position of the epoch's first op
    int32_t n_vars;
    int pack;
    uint32_t valid[8];          // bit b: op byte b is well-formed
    const uint32_t* bm;         // stuck at the epoch's start
    uint32_t* key;              // slots: the kept ops of stretch i from KSTRETCH i on, in position order
    uint32_t* val;
    uint32_t* all_key;          // the ops of an epoch kept whole, at their positions in it
    uint32_t* all_val;
    int32_t* cnt;               // kept ops per stretch
    int* all;                   // out: the epoch is kept whole
    const uint8_t* fin;         // statuses so far
    uint8_t* st;                // out: a copy (the scan reads it while it writes the later ones)
    int* err;
};
constexpr int KSAMPLE = 4 * KFT;

// A warp per stretch of 512 ops, 16 consecutive ops per lane, no barrier: 1,024
// threads an SM stream beside the 128 KB bitmap.
__global__ void __launch_bounds__(KFT, 1) kl_filter_kernel(const __grid_constant__ KFilterParams p)
{
    follow();
    extern __shared__ __align__(16) uint32_t sbm[];
    __shared__ uint32_t valid[8];
    const int t = threadIdx.x, lane = t & 31;
    for (int i = t; i < (p.n_vars + 31) / 32; i += KFT) sbm[i] = p.bm[i];
    if (t < 8) valid[t] = p.valid[t];
    __syncthreads();
    // ops on variables that are not stuck, of a sample that is the same in every CTA
    int alive = 0;
#pragma unroll
    for (int j = 0; j < KSAMPLE / KFT; ++j) {
        const uint32_t v = (uint32_t)p.var[(int64_t)(j * KFT + t) * p.n / KSAMPLE];
        alive += __syncthreads_count(v < (uint32_t)p.n_vars && !((sbm[v >> 5] >> (v & 31)) & 1u));
    }
    const bool all = 8 * alive >= 7 * KSAMPLE;
    if (blockIdx.x == 0 && t == 0) *p.all = all;
    for (int v = (int)blockIdx.x * KFT + t; v < p.n_vars; v += (int)gridDim.x * KFT) p.st[v] = p.fin[v];
    const int64_t ns = (p.n + KSTRETCH - 1) / KSTRETCH, nw = (int64_t)gridDim.x * (KFT / 32);
    const bool wide = (uintptr_t)p.op % 16 == 0 && (uintptr_t)p.var % 16 == 0 && (uintptr_t)p.step % 16 == 0;
    for (int64_t s = (int64_t)blockIdx.x * (KFT / 32) + (t >> 5); s < ns; s += nw) {
        const int64_t i0 = s * KSTRETCH + lane * KFE;
        const int m = (int)min((int64_t)KFE, max((int64_t)0, p.n - i0));
        uint32_t o[KFE / 4];
        uint32_t v[KFE];
        if (m == KFE && wide) {
            const uint4 a = __ldcs(reinterpret_cast<const uint4*>(p.op + i0));
            o[0] = a.x;
            o[1] = a.y;
            o[2] = a.z;
            o[3] = a.w;
#pragma unroll
            for (int h = 0; h < KFE / 4; ++h) {
                const uint4 b = __ldcs(reinterpret_cast<const uint4*>(p.var + i0) + h);
                v[4 * h] = b.x;
                v[4 * h + 1] = b.y;
                v[4 * h + 2] = b.z;
                v[4 * h + 3] = b.w;
            }
            constexpr uint32_t F4 = 0x01010101u * KL_F;
            __stcs(reinterpret_cast<uint4*>(p.step + i0), make_uint4(F4, F4, F4, F4));
        } else {
#pragma unroll
            for (int h = 0; h < KFE / 4; ++h) o[h] = 0;
#pragma unroll
            for (int u = 0; u < KFE; ++u) {
                v[u] = 0;
                if (u < m) {
                    o[u / 4] |= (uint32_t)p.op[i0 + u] << (8 * (u & 3));
                    v[u] = (uint32_t)p.var[i0 + u];
                    p.step[i0 + u] = (uint8_t)KL_F;
                }
            }
        }
        uint32_t live = 0;
        bool bado = false, badv = false;
#pragma unroll
        for (int u = 0; u < KFE; ++u) {
            const uint32_t b = (o[u / 4] >> (8 * (u & 3))) & 0xFFu;
            const bool in = u < m;
            bado |= in && !((valid[b >> 5] >> (b & 31)) & 1u);
            if (v[u] >= (uint32_t)p.n_vars) {
                badv = true;
                v[u] = 0;
            }
            if (in && !((sbm[v[u] >> 5] >> (v[u] & 31)) & 1u)) live |= 1u << u;
        }
        if (bado) raise_error(p.err, AMC_E_INVALID);
        if (badv) raise_error(p.err, AMC_E_RANGE);
        if (all) {
            if (lane == 0) p.cnt[s] = (int32_t)min((int64_t)KSTRETCH, p.n - s * KSTRETCH);
#pragma unroll
            for (int h = 0; h < KFE / 4; ++h) {
                uint32_t kk[4], vv[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    kk[u] = p.pack ? (v[4 * h + u] | ((o[h] >> (8 * u)) & 0xFFu) << KOP_SHIFT) : v[4 * h + u];
                    vv[u] = (uint32_t)(p.offset + i0 + 4 * h + u);
                    if (m < KFE && 4 * h + u < m) {
                        p.all_key[i0 + 4 * h + u] = kk[u];
                        p.all_val[i0 + 4 * h + u] = vv[u];
                    }
                }
                if (m == KFE) {
                    reinterpret_cast<uint4*>(p.all_key + i0)[h] = make_uint4(kk[0], kk[1], kk[2], kk[3]);
                    reinterpret_cast<uint4*>(p.all_val + i0)[h] = make_uint4(vv[0], vv[1], vv[2], vv[3]);
                }
            }
            continue;
        }
        const int c = __popc(live), incl = warp_incl_sum(c);
        if (lane == 31) p.cnt[s] = incl;
        int64_t at = s * KSTRETCH + (incl - c);
#pragma unroll
        for (int u = 0; u < KFE; ++u) {
            if (!((live >> u) & 1u)) continue;
            const uint32_t b = (o[u / 4] >> (8 * (u & 3))) & 0xFFu;
            p.key[at] = p.pack ? (v[u] | b << KOP_SHIFT) : v[u];
            p.val[at] = (uint32_t)(p.offset + i0 + u);
            ++at;
        }
    }
}

// The kept ops of every stretch from its slots to their place (an epoch kept
// whole is there already); the scan's tile words zeroed.
__global__ void __launch_bounds__(256) kl_compact_kernel(const uint32_t* __restrict__ skey, const uint32_t* __restrict__ sval,
                                                         const int32_t* __restrict__ cnt, const int64_t* __restrict__ off,
                                                         int64_t ns, uint32_t* __restrict__ key,
                                                         uint32_t* __restrict__ val, const int* all,
                                                         uint32_t* __restrict__ zero, int n_zero)
{
    follow();
    for (int i = (int)(blockIdx.x * blockDim.x + threadIdx.x); i < n_zero; i += (int)(gridDim.x * blockDim.x)) zero[i] = 0;
    if (*all) return;
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t s = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; s < ns; s += nw) {
        const int n = cnt[s];
        const int64_t to = off[s], from = s * KSTRETCH;
        for (int i = lane; i < n; i += 32) {
            key[to + i] = skey[from + i];
            val[to + i] = sval[from + i];
        }
    }
}

struct KSegParams {
    uint32_t vmask;         // variable bits of a key
    int pack;               // keys carry the op byte
    const uint32_t* key;
    const uint32_t* val;
    int64_t cap;            // pairs, or their most with n_dev
    const int64_t* n_dev;   // nullable: pairs, on the device
    const uint8_t* op;
    const uint8_t* init;
    uint8_t* step;
    uint8_t* fin;
    int32_t* vff;
    int64_t* ff;
    uint32_t* tstat;        // per tile, zeroed before the launch
    uint32_t* tile_counter; // zeroed before the launch
    int* err;
    uint32_t* bm;           // nullable: stuck bitmap, bits set for variables that end F
};

__global__ void __launch_bounds__(KNT) kl_seg_kernel(const KSegParams p)
{
    follow();
    __shared__ uint32_t wtot[KNT / 32];
    __shared__ uint32_t s_tile, s_carry;
    const int64_t n = p.n_dev ? max((int64_t)0, min(*p.n_dev, p.cap)) : p.cap;
    const int64_t nt = (n + KT - 1) / KT;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (;;) {
        if (threadIdx.x == 0) s_tile = atomicAdd(p.tile_counter, 1u);
        __syncthreads();
        const int64_t tile = s_tile;
        if (tile >= nt) break;
        const int64_t b = tile * KT;
        const int m = (int)(n - b < KT ? n - b : KT);
        const int i0 = threadIdx.x * KE;
        uint32_t kk[KE], vv[KE], el[KE];
#pragma unroll
        for (int u = 0; u < KE; ++u) {
            const bool in = i0 + u < m;
            kk[u] = in ? p.key[b + i0 + u] : KNOKEY;
            vv[u] = in ? p.val[b + i0 + u] : 0u;
        }
#pragma unroll
        for (int u = 0; u < KE; ++u) {
            if (kk[u] == KNOKEY) {
                el[u] = KIDENT;
                continue;
            }
            el[u] = kelem(p.pack ? (kk[u] >> KOP_SHIFT) & 0xFFu : p.op[vv[u]]);
            kk[u] &= p.vmask;                                   // the variable alone from here on
        }
        uint32_t prev = (b + i0 > 0 && b + i0 - 1 < n) ? (p.key[b + i0 - 1] & p.vmask) : KNOKEY;
        uint32_t heads = 0, agg = KIDENT;
#pragma unroll
        for (int u = 0; u < KE; ++u) {
            if (kk[u] == KNOKEY) break;
            if (kk[u] != prev) {
                heads |= 1u << u;
                agg = KRUN | el[u];
            } else {
                agg = (agg & KRUN) | kcomp(agg & (KRUN - 1u), el[u]);
            }
            prev = kk[u];
        }
        // exclusive segmented scan of the threads' folds
        uint32_t incl = agg;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl = kseg(y, incl);
        }
        uint32_t ex = __shfl_up_sync(0xffffffffu, incl, 1);
        if (lane == 0) ex = KIDENT;
        if (lane == 31) wtot[warp] = incl;
        __syncthreads();
        uint32_t pre = KIDENT;
        for (int w = 0; w < warp; ++w) pre = kseg(pre, wtot[w]);
        uint32_t all = KIDENT;
        for (int w = 0; w < KNT / 32; ++w) all = kseg(all, wtot[w]);
        ex = kseg(pre, ex);
        if (threadIdx.x == 0) {
            uint32_t carry = KIDENT;
            if (tile == 0) {
                st_release(p.tstat, TS_INCL | (all & KVAL));
            } else {
                st_release(p.tstat + tile, TS_AGG | (all & KVAL));
                uint32_t prefix = KIDENT;                  // over tiles [t2, tile)
                for (int64_t t2 = tile - 1; t2 >= 0; --t2) {
                    uint32_t v = 0;
                    for (uint32_t it = 0; it < (1u << 24); ++it) {
                        v = ld_acquire(p.tstat + t2);
                        if (v & TS_FLAGS) break;
                    }
                    if (!(v & TS_FLAGS)) {
                        raise_error(p.err, AMC_E_TIMEOUT);
                        break;
                    }
                    prefix = kseg(v & KVAL, prefix);
                    if ((v & TS_INCL) || (v & KRUN)) break;
                }
                st_release(p.tstat + tile, TS_INCL | (kseg(prefix, all) & KVAL));
                if (((p.key[b - 1] ^ p.key[b]) & p.vmask) == 0) carry = prefix & (KRUN - 1u);
            }
            s_carry = carry;
        }
        __syncthreads();
        // the carry reaches this thread's first run only if no run starts
        // before it in the tile
        uint32_t run = (ex & KRUN) ? (ex & (KRUN - 1u)) : kcomp(s_carry, ex & (KRUN - 1u));
        const uint32_t after = (b + i0 + KE < n) ? (p.key[b + i0 + KE] & p.vmask) : KNOKEY;
        unsigned long long gmin = ~0ull;
#pragma unroll
        for (int u = 0; u < KE; ++u) {
            const uint32_t kv = kk[u];
            if (kv == KNOKEY) break;
            const bool head = (heads >> u) & 1u;
            const uint32_t before = head ? KIDENT : run;
            run = head ? el[u] : kcomp(run, el[u]);
            const uint32_t s0 = p.init ? p.init[kv] : 1u;
            const uint32_t pre_s = kapply(before, s0);
            const uint32_t post = kapply(run, s0);
            if (post != KL_F) p.step[vv[u]] = (uint8_t)post;    // F is there already
            if (post == KL_F && pre_s != KL_F) {
                p.vff[kv] = (int32_t)vv[u];
                if ((unsigned long long)vv[u] < gmin) gmin = vv[u];
            }
            const uint32_t next = u + 1 < KE ? kk[u + 1] : after;
            if (next != kv) {
                p.fin[kv] = (uint8_t)post;
                if (p.bm && post == KL_F) atomicOr(p.bm + (kv >> 5), 1u << (kv & 31));
            }
        }
        // the warp's smallest first fault, one atomic per warp
#pragma unroll
        for (int d = 16; d; d >>= 1) {
            const unsigned long long o = __shfl_xor_sync(0xffffffffu, gmin, d);
            if (o < gmin) gmin = o;
        }
        if (lane == 0 && gmin != ~0ull) atomicMin(reinterpret_cast<unsigned long long*>(p.ff), gmin);
        __syncthreads();
    }
}

// First part of a trace checked in epochs (0: the whole trace at once).
int64_t first_part(int64_t n_ops, int32_t n_vars)
{
    return n_ops < KEPOCH_MIN_OPS || n_vars > KEPOCH_MAX_VARS ? 0 : KFIRST;
}

struct KLayout {
    size_t key0, val0, key1, val1, scratch, tstat, ctr, all, cnt, off, scan, st, bm, total;
};

KLayout klayout(int64_t n, int32_t n_vars)
{
    KLayout L;
    size_t o = 0;
    auto take = [&](size_t b) { const size_t at = o; o += align_up(b, 256); return at; };
    const size_t n4 = 4 * (size_t)((n + KSTRETCH - 1) / KSTRETCH * KSTRETCH);    // whole stretches of slots
    L.key0 = take(n4);
    L.val0 = take(n4);
    L.key1 = take(n4);                                         // slots of the kept ops until they are compacted
    L.val1 = take(n4);
    L.scratch = take(sorted_check_scratch_bytes(n));
    const bool epochs = first_part(n, n_vars) > 0;
    L.tstat = take(4 * (size_t)((n + KT - 1) / KT + 1));       // with ctr: zeroed before every scan
    L.ctr = take(4);
    L.all = take(4);
    const int64_t ns = epochs ? (n + KSTRETCH - 1) / KSTRETCH : 0;
    L.cnt = take(4 * (size_t)ns);
    L.off = take(8 * ((size_t)ns + 1));
    L.scan = take(epochs ? dscan_workspace_bytes(ns) : 0);
    L.st = take(epochs ? (size_t)n_vars : 0);
    L.bm = take(epochs ? 4 * (size_t)((n_vars + 31) / 32) : 0);
    L.total = o;
    return L;
}

}  // namespace

size_t kloc_workspace_bytes(int64_t n_ops, int32_t n_vars) { return klayout(n_ops, n_vars).total; }

int launch_kloc(const KlocLaunch& L, cudaStream_t s)
{
    const KLayout lay = klayout(L.n_ops, L.n_vars);
    uint8_t* w = static_cast<uint8_t*>(L.workspace);
    uint32_t* key[2] = {reinterpret_cast<uint32_t*>(w + lay.key0), reinterpret_cast<uint32_t*>(w + lay.key1)};
    uint32_t* val[2] = {reinterpret_cast<uint32_t*>(w + lay.val0), reinterpret_cast<uint32_t*>(w + lay.val1)};
    uint32_t* bm = reinterpret_cast<uint32_t*>(w + lay.bm);
    uint32_t* ctr = reinterpret_cast<uint32_t*>(w + lay.ctr);
    int dev = 0, n_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    if (L.profile & 1) profile_begin(s);
    const int64_t S = first_part(L.n_ops, L.n_vars);
    const int64_t first = S ? S : L.n_ops;
    const int64_t work = first > L.n_vars ? first : L.n_vars;
    const int64_t blocks = (work + 255) / 256;
    const int kgrid = (int)(blocks < (int64_t)n_sm * 8 ? (blocks > 0 ? blocks : 1) : (int64_t)n_sm * 8);
    const int pack = L.n_vars <= (1 << KOP_SHIFT) ? 1 : 0;
    chain(kl_keys_kernel, kgrid, 256, 0, s)(L.op, L.var, first, L.n_vars, L.k, pack, key[0], val[0], L.step, L.init,
                                         L.final_status, L.vff, L.first_fault, L.err);
    if (cudaGetLastError() != cudaSuccess) return AMC_E_CUDA;
    // the pairs in key[0] / val[0] (n of them, or *n_dev of at most n), from the
    // statuses `init`
    auto check = [&](int64_t n, const int64_t* n_dev, const uint8_t* init) -> int {
        int passes = 0;
        const int rc = launch_ss_radix(key, val, n_dev, n, L.n_vars, w + lay.scratch, nullptr, s, &passes);
        if (rc) return rc;
        const int64_t tiles = (n + KT - 1) / KT;
        if (!n_dev && cudaMemsetAsync(w + lay.tstat, 0, lay.ctr + 4 - lay.tstat, s) != cudaSuccess) return AMC_E_CUDA;
        KSegParams p;
        p.vmask = pack ? (1u << KOP_SHIFT) - 1u : 0xFFFFFFFFu;
        p.pack = pack;
        p.key = key[passes & 1];
        p.val = val[passes & 1];
        p.cap = n;
        p.n_dev = n_dev;
        p.op = L.op;
        p.init = init;
        p.step = L.step;
        p.fin = L.final_status;
        p.vff = L.vff;
        p.ff = L.first_fault;
        p.tstat = reinterpret_cast<uint32_t*>(w + lay.tstat);
        p.tile_counter = ctr;
        p.err = L.err;
        p.bm = n_dev ? bm : nullptr;
        const int sgrid = (int)(tiles < (int64_t)n_sm * 8 ? tiles : (int64_t)n_sm * 8);
        chain(kl_seg_kernel, sgrid, KNT, 0, s)(p);
        return cudaGetLastError() == cudaSuccess ? AMC_OK : AMC_E_CUDA;
    };
    if (L.n_ops > 0) {
        const int rc = check(first, nullptr, L.init);
        if (rc) return rc;
    }
    if (S) {
        const size_t smem = 4 * (size_t)((L.n_vars + 31) / 32);
        if (!allow_smem<kl_filter_kernel>(KEPOCH_MAX_VARS / 8)) return AMC_E_CUDA;
        chain(kl_bitmap_kernel, (unsigned)((L.n_vars + 255) / 256), 256, 0, s)(L.final_status, L.n_vars, bm);
        int32_t* cnt = reinterpret_cast<int32_t*>(w + lay.cnt);
        int64_t* off = reinterpret_cast<int64_t*>(w + lay.off);
        for (int64_t e0 = S; e0 < L.n_ops;) {
            const int64_t e1 = 4 * e0 < L.n_ops ? 4 * e0 : L.n_ops;
            KFilterParams q{};
            q.op = L.op + e0;
            q.var = L.var + e0;
            q.step = L.step + e0;
            q.n = e1 - e0;
            q.offset = e0;
            q.n_vars = L.n_vars;
            q.pack = pack;
            for (uint32_t b = 0; b < 256; ++b)
                if (kvalid(b, L.k)) q.valid[b >> 5] |= 1u << (b & 31);
            q.bm = bm;
            q.key = key[1];
            q.val = val[1];
            q.all_key = key[0];
            q.all_val = val[0];
            q.all = reinterpret_cast<int*>(w + lay.all);
            q.cnt = cnt;
            q.err = L.err;
            q.fin = L.final_status;
            q.st = w + lay.st;
            const int64_t ns = (q.n + KSTRETCH - 1) / KSTRETCH;
            const int64_t fb = (ns + KFT / 32 - 1) / (KFT / 32), cb = (ns + 7) / 8;
            chain(kl_filter_kernel, (unsigned)(fb < n_sm ? fb : n_sm), KFT, smem, s)(q);
            if (cudaGetLastError() != cudaSuccess) return AMC_E_CUDA;
            int rc = dscan_exclusive(cnt, off, ns, w + lay.scan, s);
            if (rc) return rc;
            chain(kl_compact_kernel, (unsigned)(cb < 8 * n_sm ? cb : 8 * n_sm), 256, 0, s)(key[1], val[1], cnt, off, ns, key[0],
                                                                                     val[0], q.all,
                                                                                     reinterpret_cast<uint32_t*>(w + lay.tstat),
                                                                                     (int)((lay.ctr + 4 - lay.tstat) / 4));
            if (cudaGetLastError() != cudaSuccess) return AMC_E_CUDA;
            rc = check(q.n, off + ns, w + lay.st);
            if (rc) return rc;
            e0 = e1;
        }
    }
    if (L.profile & 2) profile_end(s);
    return AMC_OK;
}

}  // namespace amc

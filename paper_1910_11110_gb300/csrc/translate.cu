// translate.cu -- VectorPU component calls -> core trace (sm_103a).
//
// Arrays are half-open intervals of one index space; each has a real status
// (id a) and an abstract status (id A + a), one validity pair per array
// (Section 3.5).  Per call:
//   - O(M), Table Overlap-ext-tab: a declared W or RW operand x upgrades an
//     overlapping declared R operand to RW, an overlapping declared W operand
//     only when x is RW, and adds a shadow RW(y) for every overlapping array
//     that is not an argument of the call (Section 4.3; the rules read the
//     declared set only, they are not applied again to what they add).  A
//     dropped annotation is not declared: it takes part in no rule.
//   - translation of each declaration (Fig. sem-AM): R / RW -> GT x, EN x#
//     (the guarded transfers on the real and abstract variable), W / RW ->
//     w x#; then the body accesses of the operand's own mode;
//   - shadows RW(y) in ascending order: GT y, EN y#, w y#;
//   - every body write of x also writes the shared elements of each array y
//     overlapping x: w y when y lies inside x, otherwise pw y.
// With lifetimes (pvectors created and deleted during the run, Section 4.3:
// r_v is updated at creations and deletions): array a is live at the calls
// born[a] <= c < died[a]; operands must be live; O(M), the shadows and the
// projections of body writes take only the arrays live at the call; and each
// pvector created before call c (ascending id) is recorded at the head of
// call c's statements as Noop v, Noop v# (CPU side) on its vector v, the
// point where it takes v's statuses (arr_probe[a] = index of the first).
// Kernels: overlap sets r_v (sort and sweep, overlap.cu; with lifetimes only
// the pairs whose lifetimes meet), the pvectors sorted by creation call,
// per-call statement counts, device-wide exclusive scan of the counts,
// emission.
//
// Counting and emission take 128 calls a CTA: a thread per call reads its
// operands, then a thread per entry of the written operands' overlap lists
// finds out whether the entry yields a shadow and where it goes.  An entry is
// a shadow if it is live, no argument of the call, and in no earlier list of
// the call (searched in shared memory); one bit per entry, and the bits'
// prefix counts turn "how many shadows of this call come from entries of list
// j below y" into a search of list j, and the sum over the call's lists is the
// entry's place among the shadows.  The statements are collected in shared
// memory and stored 16 bytes a thread.  What bounds it is instructions, not
// the 5 bytes per statement: lanes with equal work (an entry each) in place of
// lanes with calls of very different lengths, each merging its lists.
// 5,000,011 calls over 4,096 arrays (182 M statements), a thread per call and
// stores of 32 lanes to 32 places: 1.00 ms to count and 2.48 ms to emit;
// 0.36 ms and 1.04 ms here.
#include "amc_internal.cuh"
#include "dscan.cuh"
#include "overlap.cuh"
#include "scan_trace.cuh"
#include "translate.cuh"

namespace amc {

namespace {

constexpr int MAX_OPND = 32;

struct TrParams {
    const int32_t* arr_start;
    const int32_t* arr_len;
    int32_t n_arrays;
    const uint8_t* call_side;
    const int32_t* call_off;
    int64_t n_calls;
    const int32_t* opnd_array;
    const uint8_t* opnd_mode;
    int64_t n_operands;
    int infer;
    uint8_t* out_ks;
    int32_t* out_var;
    int64_t out_cap;
    int64_t* out_n;
    int64_t* call_first_op;
    const int64_t* ov_off;        // [n_arrays * nb + 1]: list (a, bucket)
    const uint32_t* ov_idx;       // entries: array << 1 | (it lies inside the list's owner)
    int32_t nb;                   // time buckets of the lists (1 without lifetimes)
    int64_t bl;                   // calls per bucket
    int32_t* call_cnt;
    int* err;
    // lifetimes (born == nullptr: every array live throughout)
    const int32_t* born;
    const int32_t* died;
    const int32_t* parent;
    const uint32_t* b_key;        // creation call of each pvector, ascending (n_calls for vectors)
    const uint32_t* b_id;         // the pvector ids in that order
    int64_t* arr_probe;
};

// Where a call's statements go: nowhere (counting), the output, or a CTA's
// staging area in shared memory (op byte in bits 27-31, variable below).
struct CountSink {
    __device__ __forceinline__ void put(uint32_t, int32_t) {}
    static constexpr bool EMIT = false;
};
struct OutSink {
    uint8_t* ks;
    int32_t* var;
    __device__ __forceinline__ void put(uint32_t b, int32_t v)
    {
        *ks++ = (uint8_t)b;
        *var++ = v;
    }
    static constexpr bool EMIT = true;
};
struct StageSink {
    uint32_t* w;
    __device__ __forceinline__ void put(uint32_t b, int32_t v) { *w++ = b << 27 | (uint32_t)v; }
};
constexpr int32_t STAGE_MAX_ARRAYS = 1 << 26;        // 2 n_arrays variables fit 27 bits

template <bool LIFE>
__device__ __forceinline__ bool live_at(const TrParams& p, int32_t a, int64_t c)
{
    return !LIFE || (c >= p.born[a] && c < p.died[a]);
}

constexpr uint32_t DEAD = 1u << 31;       // mark on a list entry: not live at the call

// overlap list of array a read at call c (its time bucket's list): its first
// entry, its length in *len
template <bool LIFE>
__device__ __forceinline__ int64_t list_at(const TrParams& p, int32_t a, int64_t c, int32_t* len)
{
    const int64_t li = LIFE ? (int64_t)a * p.nb + c / p.bl : a;
    const int64_t lo = p.ov_off[li];
    *len = (int32_t)(p.ov_off[li + 1] - lo);
    return lo;
}

// first position in [a, b) of the pvectors by creation call that is created
// at call c or later
__device__ __forceinline__ int32_t births_before(const TrParams& p, int64_t c, int32_t a, int32_t b)
{
    while (a < b) {
        const int32_t m = (a + b) >> 1;
        if ((int64_t)p.b_key[m] < c) a = m + 1;
        else b = m;
    }
    return a;
}

__device__ __forceinline__ bool iv_contains(int32_t so, int32_t lo, int32_t si, int32_t li)
{
    return so <= si && (int64_t)si + li <= (int64_t)so + lo;
}

// The statements of call c into `out`; pvectors [b0, b1) by creation call hold
// those created before it.  Returns the count, or -1 for a malformed call
// (reported when counting).  NMAX >= the call's operand count; with small NMAX
// every array below is indexed by unrolled loop counters alone and stays in
// registers.
template <typename Sink, int NMAX, bool LIFE>
__device__ __forceinline__ int64_t translate_call(const TrParams& p, Sink out, int64_t c, int64_t first, int32_t k0, int n,
                                                  uint32_t side, int32_t b0, int32_t b1)
{
    constexpr bool EMIT = Sink::EMIT;
    constexpr int U = NMAX <= 8 ? NMAX : 1;
    const int32_t A = p.n_arrays;
    int32_t arr[NMAX], st[NMAX], en[NMAX];
    uint8_t mode[NMAX], eff[NMAX];
#pragma unroll U
    for (int i = 0; i < NMAX; ++i) {
        if (i >= n) {
            if (U == NMAX) {
                arr[i] = -1;
                mode[i] = eff[i] = 0;
                continue;
            }
            break;
        }
        const int32_t x = p.opnd_array[k0 + i];
        const uint8_t m = p.opnd_mode[k0 + i];
        arr[i] = x;
        mode[i] = m;
        eff[i] = (m & AMC_MODE_DROPPED) ? 0 : (m & 3);
        if ((m & 0x7C) || (m & 3) == 0) {
            if (!EMIT) raise_error(p.err, AMC_E_INVALID);
            return -1;
        }
        if (x < 0 || x >= A) {
            if (!EMIT) raise_error(p.err, AMC_E_RANGE);
            return -1;
        }
        if (!live_at<LIFE>(p, x, c)) {                  // not live at this call
            if (!EMIT) raise_error(p.err, AMC_E_INVALID);
            return -1;
        }
        bool dup = false;
#pragma unroll U
        for (int j = 0; j < NMAX; ++j) {
            if (U != NMAX && j >= i) break;
            dup |= j < i && arr[j] == x;
        }
        if (dup) {                                      // one declaration per variable (Section 3.3)
            if (!EMIT) raise_error(p.err, AMC_E_INVALID);
            return -1;
        }
        st[i] = p.arr_start[x];
        en[i] = st[i] + p.arr_len[x];
    }
    if (p.infer) {
        // an operand overlapping a declared written one: both are live at the
        // call, so each is in the other's list iff their ranges meet
#pragma unroll U
        for (int i = 0; i < NMAX; ++i) {
            if (i >= n) break;
            if ((mode[i] & AMC_MODE_DROPPED) || !(mode[i] & AMC_MODE_W)) continue;
            const bool x_rw = (mode[i] & 3) == AMC_MODE_RW;
#pragma unroll U
            for (int j = 0; j < NMAX; ++j) {
                if (j >= n) break;
                if (j != i && st[i] < en[j] && st[j] < en[i] && !(mode[j] & AMC_MODE_DROPPED) &&
                    (x_rw || (mode[j] & 3) != AMC_MODE_W))
                    eff[j] = AMC_MODE_RW;
            }
        }
    }
    int32_t o = 0;
    const uint32_t sb = side << 4;
    if (LIFE) {
        // creation records: Noop v, Noop v# (CPU side) for every pvector
        // created before the call, ascending id
        const int32_t lo = births_before(p, c, b0, b1), hi = births_before(p, c + 1, lo, b1);
        for (int32_t k = lo; k < hi; ++k) {
            if (EMIT) {
                const int32_t y = (int32_t)p.b_id[k];
                const int32_t v = p.parent[y];
                p.arr_probe[y] = first + o;
                out.put(AMC_K_NOOP, v);
                out.put(AMC_K_NOOP, A + v);
            }
            o += 2;
        }
    }
#pragma unroll U
    for (int i = 0; i < NMAX; ++i) {
        if (i >= n) break;
        const int32_t x = arr[i];
        const int me = eff[i], mo = mode[i] & 3;
        if (EMIT) {
            if (me & AMC_MODE_R) {                      // R or RW
                out.put(AMC_K_GT | sb, x);
                out.put(AMC_K_EN | sb, A + x);
            }
            if (me & AMC_MODE_W) out.put(AMC_K_W | sb, A + x);
            if (mo & AMC_MODE_R) out.put(AMC_K_R | sb, x);
            if (mo & AMC_MODE_W) out.put(AMC_K_W | sb, x);
        }
        o += 2 * (me & 1) + (me >> 1) + (mo & 1) + (mo >> 1);
    }
    // entry of a written operand's list, marked where it is not live
    auto entry = [&](const uint32_t* q) -> uint32_t {
        const uint32_t e = *q;
        return live_at<LIFE>(p, (int32_t)(e >> 1), c) ? e : e | DEAD;
    };
    int32_t len[NMAX];
    const uint32_t* q[NMAX] = {};
    int declared = 0;                                   // lists the shadows come from
    {
#pragma unroll U
        for (int i = 0; i < NMAX; ++i) {
            if (U == NMAX) len[i] = 0;
            if (i >= n) {
                if (U == NMAX) continue;
                break;
            }
            len[i] = 0;
            if (!(mode[i] & AMC_MODE_W)) continue;
            q[i] = p.ov_idx + list_at<LIFE>(p, arr[i], c, &len[i]);
            declared += !(mode[i] & AMC_MODE_DROPPED);
        }
    }
    if (p.infer && declared == 1 && !EMIT && !LIFE) {
        // counting a single list: its entries but the call's arguments, which are
        // looked up as emission meets them (of malformed arrays a pair may overlap
        // and not be listed)
#pragma unroll U
        for (int i = 0; i < NMAX; ++i) {
            if (i >= n) break;
            if ((mode[i] & AMC_MODE_DROPPED) || !(mode[i] & AMC_MODE_W)) continue;
            int32_t args = 0;
#pragma unroll U
            for (int j = 0; j < NMAX; ++j) {
                if (j >= n) break;
                int32_t a = 0, b = len[i];
                while (a < b) {
                    const int32_t m = (a + b) >> 1;
                    if ((int32_t)(q[i][m] >> 1) < arr[j]) a = m + 1;
                    else b = m;
                }
                args += a < len[i] && (int32_t)(q[i][a] >> 1) == arr[j];
            }
            o += 3 * (len[i] - args);
        }
    } else if (p.infer && declared) {
        // shadows: union of the overlap lists of declared written operands,
        // minus the call's arguments, ascending: a merge of the lists, their
        // heads (array << 1 | not live) at hand
        const uint32_t* h[NMAX] = {};
        uint32_t head[NMAX];
        int32_t left[NMAX] = {};
        auto pull = [&](int l) {
            uint32_t e = ~0u;
            if (left[l] > 0) {
                e = entry(h[l]);
                e = (e & ~(DEAD | 1u)) | e >> 31;
            }
            head[l] = e;
        };
#pragma unroll U
        for (int i = 0; i < NMAX; ++i) {
            head[i] = ~0u;
            if (i >= n) {
                if (U == NMAX) continue;
                break;
            }
            if ((mode[i] & AMC_MODE_DROPPED) || !(mode[i] & AMC_MODE_W)) continue;
            h[i] = q[i];
            left[i] = len[i];
            pull(i);
        }
        for (;;) {
            uint32_t y = ~0u;
#pragma unroll U
            for (int l = 0; l < NMAX; ++l) {
                if (U != NMAX && l >= n) break;
                y = min(y, head[l]);
            }
            if (y == ~0u) break;
#pragma unroll U
            for (int l = 0; l < NMAX; ++l) {
                if (U != NMAX && l >= n) break;
                if (head[l] == y) {
                    ++h[l];
                    --left[l];
                    pull(l);
                }
            }
            const int32_t v = (int32_t)(y >> 1);
            bool skip = LIFE && (y & 1u);
#pragma unroll U
            for (int j = 0; j < NMAX; ++j) {
                if (U != NMAX && j >= n) break;
                skip |= arr[j] == v;
            }
            if (skip) continue;
            if (EMIT) {
                out.put(AMC_K_GT | sb, v);
                out.put(AMC_K_EN | sb, A + v);
                out.put(AMC_K_W | sb, A + v);
            }
            o += 3;
        }
    }
#pragma unroll U
    for (int i = 0; i < NMAX; ++i) {
        if (i >= n) break;
        if (!(mode[i] & AMC_MODE_W)) continue;          // the body writes x (declared or not)
        const bool all = !EMIT && !LIFE;                // counting: every entry is live
        if (all) o += len[i];
        for (int32_t k = 0; !all && k < len[i]; ++k) {
            const uint32_t e = entry(q[i] + k);
            if (LIFE && (e & DEAD)) continue;
            if (EMIT) out.put(((e & 1u) ? AMC_K_W : AMC_K_PW) | sb, (int32_t)((e & ~DEAD) >> 1));
            ++o;
        }
    }
    return o;
}

// Calls of more than 8 operands: the same, its arrays in local memory.
template <typename Sink, bool LIFE>
__device__ __noinline__ int64_t translate_call_long(const TrParams& p, Sink out, int64_t c, int64_t first, int32_t k0, int n,
                                                    uint32_t side, int32_t b0, int32_t b1)
{
    return translate_call<Sink, MAX_OPND, LIFE>(p, out, c, first, k0, n, side, b0, b1);
}

template <typename Sink, bool LIFE>
__device__ __forceinline__ int64_t translate_any(const TrParams& p, Sink out, int64_t c, int64_t first, int32_t b0,
                                                 int32_t b1)
{
    const uint32_t side = p.call_side[c];
    const int32_t k0 = p.call_off[c], k1 = p.call_off[c + 1];
    if (side > 1 || k0 < 0 || k1 < k0 || (int64_t)k1 > p.n_operands || k1 - k0 > MAX_OPND) {
        if (!Sink::EMIT) raise_error(p.err, AMC_E_INVALID);
        return -1;
    }
    const int n = k1 - k0;
    if (n <= 4) return translate_call<Sink, 4, LIFE>(p, out, c, first, k0, n, side, b0, b1);
    if (n <= 8) return translate_call<Sink, 8, LIFE>(p, out, c, first, k0, n, side, b0, b1);
    return translate_call_long<Sink, LIFE>(p, out, c, first, k0, n, side, b0, b1);
}

constexpr int TNT = 128;                  // calls per CTA
constexpr int TOPND = 4;                  // operands a call may have here (more: a thread per call)
constexpr int TLIST = 10 * TNT;           // list entries per CTA (6.9 a call in the benchmark workload)
constexpr int TWORDS = TLIST / 32;

struct TrSmem {
    uint32_t ent[TLIST];                  // the entries, marked where not live, call by call, list by list
    uint32_t from[TNT][TOPND];            // first entry of each list in ov_idx
    int32_t arr[TNT][TOPND];              // operands (-1: none)
    uint32_t shadow[TWORDS], live[TWORDS];             // a bit per entry
    uint16_t shadow_pre[TWORDS + 1], live_pre[TWORDS + 1];   // bits before each word
    int32_t shadow_at[TNT], proj_at[TNT]; // first word of a call's shadows / projections in the staging area
    uint16_t start[TNT][TOPND + 1];       // the call's lists in ent (none for an operand that is not written)
    uint8_t own[TLIST];                   // call of each entry
    uint8_t decl[TNT];                    // bit i: shadows come from list i
    uint8_t side[TNT];
    int32_t births[2];
    int wsum[TNT / 32 + 1];
    int total;
};

// bits below e
__device__ __forceinline__ int bits_before(const uint32_t* w, const uint16_t* pre, int e)
{
    const int k = e >> 5;
    return pre[k] + ((e & 31) ? __popc(w[k] & ((1u << (e & 31)) - 1u)) : 0);
}
// first entry in [a, b) whose array is >= y (mask: all bits of an entry, or all
// but its mark)
__device__ __forceinline__ int entry_at(const uint32_t* ent, int a, int b, uint32_t y, uint32_t mask)
{
    while (a < b) {
        const int m = (a + b) >> 1;
        if ((ent[m] & mask) < 2 * y) a = m + 1;
        else b = m;
    }
    return a;
}

// 128 calls: their counts (EMIT = false) or their statements, through a
// staging area of `cap` statements.  A CTA with a call of more operands, more
// list entries or statements than its areas hold, or ids that do not fit the
// staging words runs a thread per call instead.
template <bool EMIT, bool LIFE>
__global__ void __launch_bounds__(TNT, EMIT ? 6 : 10) calls_kernel(const TrParams p, int cap)
{
    __shared__ TrSmem S;
    extern __shared__ __align__(16) uint32_t stage[];
    if (EMIT && p.call_first_op[p.n_calls] > p.out_cap) return;     // nothing but out_n is written
    const int t = threadIdx.x, lane = t & 31;
    const int64_t c0 = (int64_t)blockIdx.x * TNT;
    const int m = (int)min((int64_t)TNT, p.n_calls - c0);
    const int64_t c = c0 + t;
    if (LIFE && t < 2) S.births[t] = births_before(p, t ? c0 + m : c0, 0, p.n_arrays);
    // ---- a thread per call: operands, declarations in force, lists ----------
    int n = 0;
    uint32_t side = 0;
    int32_t k0 = 0;
    bool other = false;                                 // not for this path
    if (t < m) {
        side = p.call_side[c];
        k0 = p.call_off[c];
        const int32_t k1 = p.call_off[c + 1];
        n = k1 - k0;
        if (side > 1 || k0 < 0 || k1 < k0 || (int64_t)k1 > p.n_operands || n > TOPND) {
            other = true;
            n = 0;
        }
    }
    int32_t arr[TOPND], st[TOPND], en[TOPND], len[TOPND];
    uint32_t mode[TOPND], eff[TOPND];
    int64_t lo[TOPND];
#pragma unroll
    for (int i = 0; i < TOPND; ++i) {
        arr[i] = -1;
        mode[i] = 0;
        st[i] = en[i] = INT32_MAX;                      // no operand: meets no range
        len[i] = 0;
        lo[i] = 0;
        if (i < n) {
            arr[i] = p.opnd_array[k0 + i];
            mode[i] = p.opnd_mode[k0 + i];
        }
    }
#pragma unroll
    for (int i = 0; i < TOPND; ++i) {
        if (i >= n) break;
        // a malformed call: reported (and left out) by the thread-per-call path
        bool bad = (mode[i] & 0x7C) || (mode[i] & 3) == 0 || arr[i] < 0 || arr[i] >= p.n_arrays;
#pragma unroll
        for (int j = 0; j < i; ++j) bad |= arr[j] == arr[i];
        if (!bad) bad = !live_at<LIFE>(p, arr[i], c);
        other |= bad;
        if (bad) continue;
        st[i] = p.arr_start[arr[i]];
        en[i] = st[i] + p.arr_len[arr[i]];
        if (mode[i] & AMC_MODE_W) {
            lo[i] = list_at<LIFE>(p, arr[i], c, &len[i]);
            other |= lo[i] > (int64_t)0xFFFFFFFFll;
        }
    }
    int64_t wt = 0;
#pragma unroll
    for (int i = 0; i < TOPND; ++i) wt += len[i];
    other |= wt > TLIST;
    const int base = block_excl_sum<TNT>(wt > TLIST ? TLIST + 1 : (int)wt, S.wsum, &S.total);
    const int64_t f0 = EMIT ? p.call_first_op[c0] : 0, f1 = EMIT ? p.call_first_op[c0 + m] : 0;
    const int64_t al = f0 & ~(int64_t)3;                // statement of the staging area's first word
    if (__syncthreads_or(other) || S.total > TLIST || (EMIT && f1 - al > cap)) {
        if (t >= m) return;
        const int32_t b0 = LIFE ? S.births[0] : 0, b1 = LIFE ? S.births[1] : 0;
        if (EMIT) {
            const int64_t f = p.call_first_op[c];
            translate_any<OutSink, LIFE>(p, OutSink{p.out_ks + f, p.out_var + f}, c, f, b0, b1);
        } else {
            const int64_t k = translate_any<CountSink, LIFE>(p, CountSink{}, c, 0, b0, b1);
            p.call_cnt[c] = k < 0 ? 0 : (int32_t)k;
        }
        return;
    }
    const int E = S.total;
    uint32_t decl = 0;
    int pre = 0;                                        // statements before the shadows
    {
        int at = base;
#pragma unroll
        for (int i = 0; i < TOPND; ++i) {
            const bool dropped = (mode[i] & AMC_MODE_DROPPED) != 0;
            eff[i] = dropped ? 0 : mode[i] & 3;
            if (p.infer) {
                if (!dropped && (mode[i] & AMC_MODE_W)) decl |= 1u << i;
                // a declared written operand upgrades the declared ones it overlaps
#pragma unroll
                for (int j = 0; j < TOPND; ++j)
                    if (j != i && st[i] < en[j] && st[j] < en[i] && (mode[j] & AMC_MODE_W) &&
                        !(mode[j] & AMC_MODE_DROPPED) && !dropped &&
                        ((mode[j] & 3) == AMC_MODE_RW || (mode[i] & 3) != AMC_MODE_W))
                        eff[i] = AMC_MODE_RW;
            }
            pre += 2 * (eff[i] & 1) + (eff[i] >> 1) + (mode[i] & 1) + ((mode[i] >> 1) & 1);
            S.arr[t][i] = arr[i];
            S.from[t][i] = (uint32_t)lo[i];
            S.start[t][i] = (uint16_t)at;
            at += len[i];
        }
        S.start[t][TOPND] = (uint16_t)at;
        S.decl[t] = (uint8_t)decl;
        S.side[t] = (uint8_t)(side << 4);
        for (int e = base; e < at; ++e) S.own[e] = (uint8_t)t;
    }
    __syncthreads();
    // ---- a thread per entry: the lists into shared memory -------------------
    for (int e = t; e < E; e += TNT) {
        const int k = S.own[e];
        int i = 0;
#pragma unroll
        for (int j = 1; j < TOPND; ++j) i += S.start[k][j] <= e;
        const uint32_t x = p.ov_idx[(int64_t)S.from[k][i] + (e - S.start[k][i])];
        S.ent[e] = live_at<LIFE>(p, (int32_t)(x >> 1), c0 + k) ? x : x | DEAD;
    }
    __syncthreads();
    constexpr uint32_t mask = LIFE ? ~DEAD : ~0u;
    // ---- which entries are shadows ------------------------------------------
    for (int e0 = t - lane; e0 < E; e0 += TNT) {
        const int e = e0 + lane;
        bool shadow = false, live = false;
        if (e < E) {
            const int k = S.own[e];
            const uint32_t x = S.ent[e], y = (x & ~DEAD) >> 1, d = S.decl[k];
            int i = 0;
#pragma unroll
            for (int j = 1; j < TOPND; ++j) i += S.start[k][j] <= e;
            live = !(x & DEAD);
            shadow = live && ((d >> i) & 1u);
#pragma unroll
            for (int j = 0; j < TOPND; ++j) shadow &= S.arr[k][j] != (int32_t)y;
            if (shadow)
                for (uint32_t r = d & ((1u << i) - 1u); r; r &= r - 1) {
                    const int j = __ffs(r) - 1, b = S.start[k][j + 1], q = entry_at(S.ent, S.start[k][j], b, y, mask);
                    shadow &= q == b || ((S.ent[q] & mask) >> 1) != y;
                }
        }
        const uint32_t sw = __ballot_sync(0xffffffffu, shadow), lw = __ballot_sync(0xffffffffu, live);
        if (lane == 0) {
            S.shadow[e0 >> 5] = sw;
            S.live[e0 >> 5] = lw;
        }
    }
    __syncthreads();
    if (t < 32) {
        const int words = (E + 31) >> 5;
        int cs = 0, cl = 0;
        for (int w0 = 0; w0 <= words; w0 += 32) {
            const int w = w0 + t;
            const int a = w < words ? __popc(S.shadow[w]) : 0, b = w < words ? __popc(S.live[w]) : 0;
            const int ia = warp_incl_sum(a), ib = warp_incl_sum(b);
            if (w <= words) {
                S.shadow_pre[w] = (uint16_t)(cs + ia - a);
                S.live_pre[w] = (uint16_t)(cl + ib - b);
            }
            cs += __shfl_sync(0xffffffffu, ia, 31);
            cl += __shfl_sync(0xffffffffu, ib, 31);
        }
    }
    __syncthreads();
    // ---- a thread per call: its count, or its first statements ---------------
    {
        const int b = S.start[t][0], e = S.start[t][TOPND];
        const int shadows = bits_before(S.shadow, S.shadow_pre, e) - bits_before(S.shadow, S.shadow_pre, b);
        const int projections = bits_before(S.live, S.live_pre, e) - bits_before(S.live, S.live_pre, b);
        int32_t births = 0, blo = 0;
        if (LIFE && t < m) {
            blo = births_before(p, c, S.births[0], S.births[1]);
            births = births_before(p, c + 1, blo, S.births[1]) - blo;
        }
        if (!EMIT) {
            if (t < m) p.call_cnt[c] = 2 * births + pre + 3 * shadows + projections;
            return;
        }
        if (t < m) {
            const int32_t A = p.n_arrays;
            const int64_t f = p.call_first_op[c];
            StageSink out{stage + (f - al)};
            for (int32_t k = 0; k < births; ++k) {
                const int32_t y = (int32_t)p.b_id[blo + k];
                const int32_t v = p.parent[y];
                p.arr_probe[y] = f + 2 * k;
                out.put(AMC_K_NOOP, v);
                out.put(AMC_K_NOOP, A + v);
            }
            const uint32_t sb = side << 4;
#pragma unroll
            for (int i = 0; i < TOPND; ++i) {
                if (i >= n) break;
                const int32_t x = arr[i];
                if (eff[i] & AMC_MODE_R) {
                    out.put(AMC_K_GT | sb, x);
                    out.put(AMC_K_EN | sb, A + x);
                }
                if (eff[i] & AMC_MODE_W) out.put(AMC_K_W | sb, A + x);
                if (mode[i] & AMC_MODE_R) out.put(AMC_K_R | sb, x);
                if (mode[i] & AMC_MODE_W) out.put(AMC_K_W | sb, x);
            }
            S.shadow_at[t] = (int32_t)(f - al) + 2 * births + pre;
            S.proj_at[t] = S.shadow_at[t] + 3 * shadows - bits_before(S.live, S.live_pre, b);
            // a shadow's place is the sum of the bits before it in each list:
            // the bits before the lists are taken off here
            int before = 0;
            for (uint32_t r = decl; r; r &= r - 1)
                before += bits_before(S.shadow, S.shadow_pre, S.start[t][__ffs(r) - 1]);
            S.shadow_at[t] -= 3 * before;
        }
    }
    __syncthreads();
    // ---- a thread per entry: its shadow, its projection ----------------------
    for (int e = t; e < E; e += TNT) {
        const uint32_t x = S.ent[e];
        if (LIFE && (x & DEAD)) continue;
        const int k = S.own[e];
        const int32_t y = (int32_t)(x >> 1);             // live: no mark
        const uint32_t sb = S.side[k];
        StageSink proj{stage + S.proj_at[k] + bits_before(S.live, S.live_pre, e)};
        proj.put(((x & 1u) ? AMC_K_W : AMC_K_PW) | sb, y);
        if (!((S.shadow[e >> 5] >> (e & 31)) & 1u)) continue;
        int i = 0;
#pragma unroll
        for (int j = 1; j < TOPND; ++j) i += S.start[k][j] <= e;
        int rank = bits_before(S.shadow, S.shadow_pre, e);
        for (uint32_t r = S.decl[k] & ~(1u << i); r; r &= r - 1) {
            const int j = __ffs(r) - 1;
            rank += bits_before(S.shadow, S.shadow_pre,
                                entry_at(S.ent, S.start[k][j], S.start[k][j + 1], (uint32_t)y, mask));
        }
        StageSink out{stage + S.shadow_at[k] + 3 * rank};
        out.put(AMC_K_GT | sb, y);
        out.put(AMC_K_EN | sb, p.n_arrays + y);
        out.put(AMC_K_W | sb, p.n_arrays + y);
    }
    __syncthreads();
    const bool wide = (uintptr_t)p.out_ks % 4 == 0 && (uintptr_t)p.out_var % 16 == 0;
    constexpr uint32_t VM = (1u << 27) - 1u;
    for (int64_t g = al + 4 * t; g < f1; g += 4 * TNT) {
        const uint4 w = *reinterpret_cast<const uint4*>(stage + (g - al));
        if (wide && g >= f0 && g + 4 <= f1) {
            *reinterpret_cast<uint32_t*>(p.out_ks + g) = w.x >> 27 | w.y >> 27 << 8 | w.z >> 27 << 16 | w.w >> 27 << 24;
            *reinterpret_cast<int4*>(p.out_var + g) =
                make_int4((int)(w.x & VM), (int)(w.y & VM), (int)(w.z & VM), (int)(w.w & VM));
        } else {
            const uint32_t q[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (g + u >= f0 && g + u < f1) {
                    p.out_ks[g + u] = (uint8_t)(q[u] >> 27);
                    p.out_var[g + u] = (int32_t)(q[u] & VM);
                }
        }
    }
}

__global__ void total_kernel(const TrParams p)
{
    const int64_t total = p.call_first_op[p.n_calls];
    *p.out_n = total;
    if (total > p.out_cap) raise_error(p.err, AMC_E_RANGE);
}

// pvector lifetimes: 0 <= born < died <= n_calls; a pvector's vector is a
// vector (parent -1) other than itself whose range and lifetime hold its own.
// Sort keys: the creation call of each pvector, n_calls for vectors.
__global__ void lifetimes_kernel(const TrParams p, uint32_t* __restrict__ key, uint32_t* __restrict__ val)
{
    const int64_t a = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= p.n_arrays) return;
    p.arr_probe[a] = -1;
    const int32_t b = p.born[a], d = p.died[a], v = p.parent[a];
    bool ok = b >= 0 && b < d && (int64_t)d <= p.n_calls;
    if (v != -1) {
        if (v < 0 || v >= p.n_arrays) {
            raise_error(p.err, AMC_E_RANGE);
            ok = true;                        // reported
        } else {
            ok = ok && v != a && p.parent[v] == -1 && p.born[v] <= b && d <= p.died[v] &&
                 iv_contains(p.arr_start[v], p.arr_len[v], p.arr_start[a], p.arr_len[a]);
        }
    }
    if (!ok) raise_error(p.err, AMC_E_INVALID);
    key[a] = (v >= 0 && v < p.n_arrays && b >= 0 && b < p.n_calls) ? (uint32_t)b : (uint32_t)p.n_calls;
    val[a] = (uint32_t)a;
}

struct TrLayout {
    size_t ov_off, ov_idx, ovws, bk0, bv0, bk1, bv1, bscr, call_cnt, scan, total;
    int64_t cap;
    int32_t nb;
};

TrLayout layout(int32_t A, int64_t n_calls, int64_t max_pairs, bool lifetimes)
{
    TrLayout L;
    size_t o = 0;
    auto take = [&](size_t b) { const size_t at = o; o += align_up(b, 256); return at; };
    // without lifetimes every array may overlap every other
    L.cap = lifetimes ? max_pairs : (int64_t)A * (A > 0 ? A - 1 : 0);
    L.nb = overlap_buckets(n_calls, lifetimes);
    L.ov_off = take(8 * ((size_t)A * L.nb + 1));
    L.ov_idx = take(4 * (size_t)(L.cap > 0 ? L.cap : 1));
    L.ovws = take(overlap_workspace_bytes(A, L.nb, L.cap));
    const size_t a4 = lifetimes ? 4 * (size_t)(A > 0 ? A : 1) : 0;
    L.bk0 = take(a4);
    L.bv0 = take(a4);
    L.bk1 = take(a4);
    L.bv1 = take(a4);
    L.bscr = take(lifetimes ? sorted_check_scratch_bytes(A > 0 ? A : 1) : 0);
    L.call_cnt = take(4 * (size_t)n_calls + 4);
    L.scan = take(dscan_workspace_bytes(n_calls > 0 ? n_calls : 1));
    L.total = o;
    return L;
}

}  // namespace

size_t translate_workspace_bytes(int32_t n_arrays, int64_t n_calls)
{
    return layout(n_arrays, n_calls, 0, false).total;
}

size_t translate_lifetimes_workspace_bytes(int32_t n_arrays, int64_t n_calls, int64_t max_pairs)
{
    return layout(n_arrays, n_calls, max_pairs, true).total;
}

size_t overlap_count_workspace_bytes(int32_t n_arrays, int64_t n_calls, bool lifetimes)
{
    const int32_t nb = overlap_buckets(n_calls, lifetimes);
    return align_up(8 * ((size_t)n_arrays * nb + 1), 256) + overlap_workspace_bytes(n_arrays, nb, 0);
}

int launch_overlap_count(const int32_t* arr_start, const int32_t* arr_len, const int32_t* arr_born,
                         const int32_t* arr_died, int32_t n_arrays, int64_t n_calls, int64_t* n_pairs, int* err,
                         void* workspace, cudaStream_t s)
{
    OverlapBuild O;
    O.arr_start = arr_start;
    O.arr_len = arr_len;
    O.arr_born = arr_born;
    O.arr_died = arr_died;
    O.n_arrays = n_arrays;
    O.n_buckets = overlap_buckets(n_calls, arr_born != nullptr);
    O.bucket_len = overlap_bucket_len(n_calls, O.n_buckets);
    O.cap = 0;
    O.ov_off = static_cast<int64_t*>(workspace);
    O.n_pairs = n_pairs;
    O.err = err;
    O.workspace = static_cast<uint8_t*>(workspace) + align_up(8 * ((size_t)n_arrays * O.n_buckets + 1), 256);
    return launch_overlaps(O, s);
}

int launch_translate(const TranslateLaunch& T, cudaStream_t s)
{
    const bool lifetimes = T.arr_born != nullptr;
    TrParams p{};
    p.arr_start = T.arr_start;
    p.arr_len = T.arr_len;
    p.n_arrays = T.n_arrays;
    p.call_side = T.call_side;
    p.call_off = T.call_off;
    p.n_calls = T.n_calls;
    p.opnd_array = T.opnd_array;
    p.opnd_mode = T.opnd_mode;
    p.n_operands = T.n_operands;
    p.infer = T.infer;
    p.out_ks = T.out_ks;
    p.out_var = T.out_var;
    p.out_cap = T.out_cap;
    p.out_n = T.out_n;
    p.call_first_op = T.call_first_op;
    p.err = T.err;
    p.born = T.arr_born;
    p.died = T.arr_died;
    p.parent = T.arr_parent;
    p.arr_probe = T.arr_probe;
    const TrLayout L = layout(T.n_arrays, T.n_calls, T.max_pairs, lifetimes);
    uint8_t* w = static_cast<uint8_t*>(T.workspace);
    int64_t* ov_off = reinterpret_cast<int64_t*>(w + L.ov_off);
    p.ov_off = ov_off;
    p.ov_idx = reinterpret_cast<uint32_t*>(w + L.ov_idx);
    p.call_cnt = reinterpret_cast<int32_t*>(w + L.call_cnt);
    void* scan_ws = w + L.scan;

    OverlapBuild O;
    O.arr_start = T.arr_start;
    O.arr_len = T.arr_len;
    O.arr_born = T.arr_born;
    O.arr_died = T.arr_died;
    O.n_arrays = T.n_arrays;
    O.n_buckets = L.nb;
    O.bucket_len = overlap_bucket_len(T.n_calls, L.nb);
    p.nb = L.nb;
    p.bl = O.bucket_len;
    O.cap = L.cap > 0 ? L.cap : 1;
    O.ov_off = ov_off;
    O.ov_idx = reinterpret_cast<uint32_t*>(w + L.ov_idx);
    O.err = T.err;
    O.workspace = w + L.ovws;
    int rc = launch_overlaps(O, s);
    if (rc) return rc;
    if (lifetimes && T.n_arrays > 0) {
        uint32_t* bk[2] = {reinterpret_cast<uint32_t*>(w + L.bk0), reinterpret_cast<uint32_t*>(w + L.bk1)};
        uint32_t* bv[2] = {reinterpret_cast<uint32_t*>(w + L.bv0), reinterpret_cast<uint32_t*>(w + L.bv1)};
        lifetimes_kernel<<<(unsigned)((T.n_arrays + 255) / 256), 256, 0, s>>>(p, bk[0], bv[0]);
        int passes = 0;
        const int64_t kr = T.n_calls + 1 < INT32_MAX ? T.n_calls + 1 : INT32_MAX;
        rc = launch_ss_radix(bk, bv, nullptr, T.n_arrays, (int32_t)kr, w + L.bscr, nullptr, s, &passes);
        if (rc) return rc;
        p.b_key = bk[passes & 1];
        p.b_id = bv[passes & 1];
    }
    if (T.n_calls > 0) {
        const unsigned blocks = (unsigned)((T.n_calls + TNT - 1) / TNT);
        auto count = lifetimes ? calls_kernel<false, true> : calls_kernel<false, false>;
        auto emit = lifetimes ? calls_kernel<true, true> : calls_kernel<true, false>;
        // 48 statements a call (a call of the benchmark workload has 37): 24 KB
        // and 14 KB of lists and bits, five CTAs per SM
        const int cap = T.n_arrays <= STAGE_MAX_ARRAYS ? 48 * TNT : 0;
        count<<<blocks, TNT, 0, s>>>(p, 0);
        int rc = dscan_exclusive(p.call_cnt, T.call_first_op, T.n_calls, scan_ws, s);
        if (rc) return rc;
        if (T.profile & 1) profile_begin(s);
        emit<<<blocks, TNT, 4 * cap, s>>>(p, cap);
        if (T.profile & 2) profile_end(s);
    } else if (cudaMemsetAsync(T.call_first_op, 0, 8, s) != cudaSuccess) {
        return AMC_E_CUDA;
    }
    total_kernel<<<1, 1, 0, s>>>(p);
    return cudaGetLastError() == cudaSuccess ? AMC_OK : AMC_E_CUDA;
}

}  // namespace amc

namespace amc {

namespace {

// Initial statuses of the second check pass: a vector's are those of the
// initial store, (V,I); a pvector's real and abstract statuses are its
// vector's at its creation record (the statuses the first pass gave the two
// Noops there).
__global__ void inherit_kernel(const int32_t* __restrict__ var, int64_t n_ops, int32_t A,
                               const int32_t* __restrict__ parent, const int64_t* __restrict__ probe,
                               const uint8_t* __restrict__ step, uint8_t* __restrict__ init, int* err)
{
    const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= 2 * (int64_t)A) return;
    const int32_t a = (int32_t)(v < A ? v : v - A);
    const int32_t pv = parent[a];
    uint8_t st = (uint8_t)AMC_ST_VI;
    if (pv != -1) {
        const int64_t q = probe[a];
        const bool ok = pv >= 0 && pv < A && q >= 0 && q + 1 < n_ops && var[q] == pv && var[q + 1] == A + pv;
        if (ok) st = step[q + (v < A ? 0 : 1)];
        else raise_error(err, AMC_E_INVALID);
    }
    init[v] = st;
}

}  // namespace

int launch_inherit(const int32_t* var, int64_t n_ops, int32_t n_arrays, const int32_t* arr_parent,
                   const int64_t* arr_probe, const uint8_t* step, uint8_t* init, int* err, cudaStream_t s)
{
    if (n_arrays <= 0) return AMC_OK;
    const int64_t n = 2 * (int64_t)n_arrays;
    inherit_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(var, n_ops, n_arrays, arr_parent, arr_probe, step,
                                                                init, err);
    return cudaGetLastError() == cudaSuccess ? AMC_OK : AMC_E_CUDA;
}

}  // namespace amc

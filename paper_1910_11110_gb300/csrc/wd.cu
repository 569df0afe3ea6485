// wd.cu -- static well-declaredness of calls AM{S} (Section 3.3, Definitions
// "Occurs in all execution paths" and "Well-declared program"; Section 3.5,
// "Well-declared program with array access").
//
// Per call, one warp:
//   * each statement of the body is checked against the call's declarations:
//     no Push / Pull; a write needs W or RW on its side, a read R or RW, for
//     the array that owns the location (one abstract variable per array);
//   * every W declaration obliges a write, on its side, of every location of
//     the array in all execution paths of the body.  That is relation mode
//     over a two-state machine per tracked location -- N "not written yet",
//     Y "written" -- with conditions opaque: w maps any state to Y, other ops
//     keep it, If is the union of its branches' sets and While the closure of
//     its body.  The obligation holds iff N is not in the set at the end.  The
//     warp keeps, per tracked location, the bit "N is not in the set" (in
//     shared memory): an op sets its bit; at an If the then- and else-sets come
//     from the same entry, so the bit after it is entry OR (then AND else); a
//     While may run zero times, so its body adds nothing.
// The warp takes the body 32 tokens at a time, the next 32 on their way: all
// its ops are checked at once (the checks do not depend on the structure), the
// tracked writes between two structure tokens set their bits with one shared
// atomic each, and the structure tokens are walked by the whole warp with a
// stack of the entry / then bits.  What bounds it is the latency of a call's
// few dependent loads and its instructions, not its bytes (5 per token).
// 2^20 calls of 38 tokens: 1.57 ms when every write's bit went to its owning
// lane through 32 shuffles a batch and every structure token reloaded the
// batch; 0.93 ms at 73 % of the issue slots (820 instructions a call) with all
// lanes on one array's obligation after another, 0.89 ms here.
#include "amc_internal.cuh"
#include "wd.cuh"

namespace amc {

namespace {

constexpr int WD_WARPS = 4;                   // warps per CTA
constexpr int WD_CLAIM = 8;                   // most calls per claim (fewer than 32)
constexpr int WD_WORDS = 32;                  // tracked words per warp pass: 32 lanes x 64 locations

struct WdParams {
    const int64_t* arr_loc_off;
    int32_t n_arrays;
    const int32_t* loc_owner;
    const int64_t* call_tok_off;
    int64_t n_calls;
    const uint8_t* tok;
    const int32_t* payload;
    int64_t n_tokens;
    const int64_t* call_am_off;
    const int32_t* am_array;
    const uint8_t* am_mode;
    int64_t n_decls;
    uint32_t* violations;
    int64_t* first_bad;
    int32_t* first_unmet;
    unsigned long long* queue;     // next call to take
    int claim;                     // calls a warp takes at a time
    int* err;
};

struct WdWarp {
    uint32_t cur[2 * WD_WORDS];                       // the window's bits
    uint32_t stack[2 * AMC_MAX_DEPTH][2 * WD_WORDS];  // per level: entry bits, then-branch bits
    int64_t base[AMC_WD_MAX_DECLS];       // first tracked bit of a W entry, -1 for R / RW
    int64_t fend[AMC_MAX_DEPTH];          // END token of each open construct
    int64_t felse[AMC_MAX_DEPTH];         // ELSE token of an open If (-1 for While)
    int64_t loc0[AMC_WD_MAX_DECLS];       // first location and locations of the array
    int64_t locs[AMC_WD_MAX_DECLS];
    int32_t arr[AMC_WD_MAX_DECLS];
    uint8_t mode[AMC_WD_MAX_DECLS];
};

__device__ __forceinline__ bool wd_op_kind(uint32_t k) { return k <= AMC_K_NOOP; }

// One call (tokens [t0, t1), declarations [m0, m1)): declarations into shared
// memory, then one pass over the body per window of WD_WORDS * 64 tracked
// locations (at least one pass, for the statement checks).  I: an integer that
// holds the body's length; positions below are relative to t0.
template <typename I>
__device__ __forceinline__ void wd_call(const WdParams& p, int64_t c, int64_t t0, const I len_t, int64_t m0, const int nd,
                                        int64_t n_locs, WdWarp& S)
{
    constexpr I NONE = sizeof(I) == 4 ? (I)INT32_MAX : (I)INT64_MAX;
    const int lane = threadIdx.x & 31;
    const uint8_t* const tok = p.tok + t0;
    const int32_t* const payload = p.payload + t0;
    // the first tokens, on their way while the declarations are read
    uint32_t nks = lane < len_t ? tok[lane] : 0xFFu;
    int32_t npl = lane < len_t ? payload[lane] : 0;
    uint32_t viol = 0;
    // declarations: range, mode, duplicates, tracked bases of the W entries
    int32_t a = -1;
    uint32_t md = 0;
    int64_t len = 0, loc0 = 0;
    if (lane < nd) {
        a = p.am_array[m0 + lane];
        md = p.am_mode[m0 + lane];
        if (a < 0 || a >= p.n_arrays) {
            raise_error(p.err, AMC_E_RANGE);
            a = -1;
        } else {
            loc0 = p.arr_loc_off[a];
            len = p.arr_loc_off[a + 1] - loc0;
        }
        if ((md & 0xE0u) || (md & 15u) < 1 || (md & 15u) > 3) raise_error(p.err, AMC_E_INVALID);
    }
    for (int j = 0; j < nd; ++j) {
        const int32_t aj = __shfl_sync(0xffffffffu, a, j);
        if (lane > j && lane < nd && a >= 0 && a == aj) viol |= 16u;     // declared twice
    }
    const bool isw = lane < nd && a >= 0 && (md & 15u) == 2u;
    int64_t tracked = 0;
    const uint32_t ws = __ballot_sync(0xffffffffu, isw);
    if (__popc(ws) <= 4) {                                 // W entries in order
        for (uint32_t r = ws; r; r &= r - 1) {
            const int j = __ffs(r) - 1;
            const int64_t n = __shfl_sync(0xffffffffu, (long long)len, j);
            if (lane == j) S.base[j] = tracked;
            tracked += n;
        }
    } else {                                               // ... in log steps
        const int64_t own = isw ? len : 0;
        int64_t incl = own;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int64_t y = __shfl_up_sync(0xffffffffu, (long long)incl, d);
            if (lane >= d) incl += y;
        }
        if (isw) S.base[lane] = incl - own;
        tracked = __shfl_sync(0xffffffffu, (long long)incl, 31);
    }
    if (lane < nd) {
        S.arr[lane] = a;
        S.mode[lane] = (uint8_t)md;
        S.loc0[lane] = loc0;
        S.locs[lane] = len;
        if (!isw) S.base[lane] = -1;
    }
    __syncwarp();
    I bad = NONE;
    int32_t unmet = INT32_MAX;
    bool malformed = false;
    I range = NONE, stop = NONE;          // first id out of range (per lane); where the body is malformed
    constexpr int64_t window = (int64_t)WD_WORDS * 64;
    const bool one_window = tracked <= window;
    for (int64_t w0 = 0; w0 == 0 || w0 < tracked; w0 += window) {
        const bool first_pass = w0 == 0;
        // words in use: lane i owns words i and 32 + i
        const int words = (int)((min(tracked - w0, window) + 31) / 32);
        for (int i = lane; i < words; i += 32) S.cur[i] = 0;
        __syncwarp();
        if (!first_pass) {
            nks = lane < len_t ? tok[lane] : 0xFFu;
            npl = lane < len_t ? payload[lane] : 0;
        }
        int depth = 0;
        for (I q0 = 0; q0 < len_t && stop == NONE; q0 += 32) {
            const I q = q0 + lane;
            const bool in = q < len_t;
            const uint32_t ks = nks;
            const int32_t pl = npl;
            const bool more = len_t - q0 > 32 && q < len_t - 32;
            nks = more ? tok[q + 32] : 0xFFu;
            npl = more ? payload[q + 32] : 0;
            const uint32_t k = ks & 15u;
            const bool op = in && !(ks & 0xE0u) && wd_op_kind(k);
            int bit = -1;
            if (op && k != AMC_K_NOOP) {
                if (pl < 0 || pl >= n_locs) {
                    range = min(range, q);
                } else if (k == AMC_K_PUSH || k == AMC_K_PULL) {
                    if (first_pass) {
                        viol |= 1u;
                        bad = min(bad, q);
                    }
                } else {
                    const int32_t own = p.loc_owner[pl];
                    const uint32_t side = (ks >> 4) & 1u;
                    bool ok = false;
                    for (int j = 0; j < nd; ++j) {
                        const uint32_t m = S.mode[j];
                        if (S.arr[j] != own || ((m >> 4) & 1u) != side) continue;
                        if (k == AMC_K_W ? (m & 2u) : (m & 1u)) ok = true;      // W, RW; R, RW
                        if (k == AMC_K_W && (m & 15u) == 2u) {
                            if (one_window) {
                                const int b = (int)S.base[j] + (pl - (int)S.loc0[j]);
                                bit = (uint32_t)b < (uint32_t)window ? b : -1;
                            } else {
                                const int64_t b = S.base[j] + (pl - S.loc0[j]) - w0;
                                bit = b >= 0 && b < window ? (int)b : -1;
                            }
                        }
                    }
                    if (!ok && first_pass) {
                        viol |= k == AMC_K_W ? 2u : 4u;
                        bad = min(bad, q);
                    }
                }
            }
            // the structure tokens in order; the tracked writes before each set their bits
            int from = 0;
            // token at x > pos, from the 64 at hand where it is one of them
            auto tok_at = [&](I x) -> uint32_t {
                const I d = x - q0;
                if (d < 64) return __shfl_sync(0xffffffffu, d < 32 ? ks : nks, (int)d & 31);
                return tok[x];
            };
            auto len_at = [&](I x) -> int32_t {
                const I d = x - q0;
                if (d < 64) return __shfl_sync(0xffffffffu, d < 32 ? pl : npl, (int)d & 31);
                return payload[x];
            };
            for (uint32_t st = __ballot_sync(0xffffffffu, in && !op);; st &= st - 1) {
                const int s = st ? __ffs(st) - 1 : 32;
                if (bit >= 0 && lane >= from && lane < s) atomicOr(&S.cur[bit >> 5], 1u << (bit & 31));
                __syncwarp();
                if (!st) break;
                from = s + 1;
                const I pos = q0 + s;
                const uint32_t sks = __shfl_sync(0xffffffffu, ks, s);
                const int32_t spl = __shfl_sync(0xffffffffu, pl, s);
                const I lim = depth ? (I)S.fend[depth - 1] : len_t;
                if (sks == AMC_T_IF || sks == AMC_T_WHILE) {          // structure tokens carry no side
                    // ends past the enclosing range are malformed: lengths are compared with what is left
                    I e = -1, end = -1;
                    const I room = lim - pos - 1;
                    if (spl >= 0 && spl < room) {
                        end = pos + 1 + spl;
                        if (sks == AMC_T_IF) {
                            e = end;
                            end = -1;
                            if (tok_at(e) == AMC_T_ELSE) {
                                const int32_t el = len_at(e);
                                if (el >= 0 && el < lim - e - 1) end = e + 1 + el;
                            }
                        }
                    }
                    if (end < 0 || tok_at(end) != AMC_T_END || depth >= AMC_MAX_DEPTH) {
                        stop = pos;
                        break;
                    }
                    for (int i = lane; i < words; i += 32) {          // the branch / body from scratch
                        S.stack[2 * depth][i] = S.cur[i];             // entry bits
                        S.cur[i] = 0;
                    }
                    if (lane == 0) {
                        S.fend[depth] = end;
                        S.felse[depth] = sks == AMC_T_IF ? e : -1;
                    }
                    ++depth;
                } else if (sks == AMC_T_ELSE) {
                    if (!depth || S.felse[depth - 1] != pos) {
                        stop = pos;
                        break;
                    }
                    for (int i = lane; i < words; i += 32) {
                        S.stack[2 * (depth - 1) + 1][i] = S.cur[i];   // then-branch bits
                        S.cur[i] = 0;
                    }
                } else if (sks == AMC_T_END) {
                    if (!depth || S.fend[depth - 1] != pos) {
                        stop = pos;
                        break;
                    }
                    --depth;
                    const bool is_if = S.felse[depth] >= 0;
                    for (int i = lane; i < words; i += 32)
                        S.cur[i] = S.stack[2 * depth][i] | (is_if ? S.stack[2 * depth + 1][i] & S.cur[i] : 0u);
                } else {
                    stop = pos;                                        // pw / GT / EN, or a byte out of range
                    break;
                }
                __syncwarp();
            }
        }
        malformed = depth || stop != NONE;
        if (malformed) break;
        // W obligations whose tracked bits fall in this window: arrays of few
        // locations a lane each, else all lanes on one array after another
        const bool few = one_window && __all_sync(0xffffffffu, len >= 0 && len <= 256);
        if (few && lane < nd && S.base[lane] >= 0) {
            const int lo = (int)S.base[lane], hi = lo + (int)S.locs[lane];
            bool miss = false;                                         // bits [lo, hi)
            for (int i = lo / 32; i * 32 < hi; ++i) {
                uint32_t need = ~0u;
                if (i * 32 < lo) need &= ~0u << (lo - i * 32);
                if (i * 32 + 32 > hi) need &= ~0u >> (i * 32 + 32 - hi);
                miss |= (S.cur[i] & need) != need;
            }
            if (miss) {
                viol |= 8u;
                unmet = S.arr[lane];
            }
        }
        for (int j = 0; !few && j < nd; ++j) {
            const int64_t b0 = S.base[j];
            if (b0 < 0) continue;
            const int64_t lo = max(b0, w0) - w0, hi = min(b0 + S.locs[j], w0 + window) - w0;
            if (lo >= hi) continue;
            bool miss = false;                                         // bits [lo, hi) of the window
            for (int64_t i = lo / 32 + lane; i * 32 < hi; i += 32) {
                uint32_t need = ~0u;
                if (i * 32 < lo) need &= ~0u << (lo - i * 32);
                if (i * 32 + 32 > hi) need &= ~0u >> (i * 32 + 32 - hi);
                miss |= (S.cur[i] & need) != need;
            }
            if (__any_sync(0xffffffffu, miss)) {
                viol |= 8u;
                unmet = min(unmet, S.arr[j]);
            }
        }
        __syncwarp();
    }
    if (range < stop) raise_error(p.err, AMC_E_RANGE);
    __syncwarp();
    if (malformed) {
        if (lane == 0) raise_error(p.err, AMC_E_INVALID);
        return;
    }
    // combine the lanes' findings
    viol = __reduce_or_sync(0xffffffffu, viol);
    if (__any_sync(0xffffffffu, bad != NONE))
#pragma unroll
        for (int d = 16; d; d >>= 1) bad = min(bad, __shfl_xor_sync(0xffffffffu, bad, d));
    unmet = __reduce_min_sync(0xffffffffu, unmet);
    if (lane == 0) {
        p.violations[c] = viol;
        p.first_bad[c] = bad == NONE ? -1 : (int64_t)bad;
        p.first_unmet[c] = unmet == INT32_MAX ? -1 : unmet;
    }
}

__global__ void __launch_bounds__(WD_WARPS * 32) wd_kernel(const WdParams p)
{
    __shared__ WdWarp S[WD_WARPS];
    const int w = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    // several calls per claim: their extents in one load
    const int64_t n_locs = p.n_arrays > 0 ? p.arr_loc_off[p.n_arrays] : 0;
    for (;;) {
        long long c0 = 0;
        if (lane == 0) c0 = (long long)atomicAdd(p.queue, (unsigned long long)p.claim);
        c0 = __shfl_sync(0xffffffffu, c0, 0);
        if (c0 >= p.n_calls) break;
        const int n = (int)min((int64_t)p.claim, p.n_calls - (int64_t)c0);
        const long long to = lane <= n ? p.call_tok_off[c0 + lane] : 0, mo = lane <= n ? p.call_am_off[c0 + lane] : 0;
        for (int i = 0; i < n; ++i) {
            const int64_t t0 = __shfl_sync(0xffffffffu, to, i), t1 = __shfl_sync(0xffffffffu, to, i + 1);
            const int64_t m0 = __shfl_sync(0xffffffffu, mo, i), m1 = __shfl_sync(0xffffffffu, mo, i + 1);
            if (t0 < 0 || t1 < t0 || t1 > p.n_tokens || m0 < 0 || m1 < m0 || m1 > p.n_decls ||
                m1 - m0 > AMC_WD_MAX_DECLS) {
                if (lane == 0) raise_error(p.err, AMC_E_INVALID);
            } else if (t1 - t0 < INT32_MAX - 64) {
                wd_call<int32_t>(p, c0 + i, t0, (int32_t)(t1 - t0), m0, (int)(m1 - m0), n_locs, S[w]);
            } else {
                wd_call<int64_t>(p, c0 + i, t0, t1 - t0, m0, (int)(m1 - m0), n_locs, S[w]);
            }
            __syncwarp();
        }
    }
}

}  // namespace

size_t wd_workspace_bytes() { return 256; }

int launch_well_declared(const WdLaunch& L, cudaStream_t s)
{
    if (L.n_calls == 0) return AMC_OK;
    WdParams p;
    p.arr_loc_off = L.arr_loc_off;
    p.n_arrays = L.n_arrays;
    p.loc_owner = L.loc_owner;
    p.call_tok_off = L.call_tok_off;
    p.n_calls = L.n_calls;
    p.tok = L.tok;
    p.payload = L.payload;
    p.n_tokens = L.n_tokens;
    p.call_am_off = L.call_am_off;
    p.am_array = L.am_array;
    p.am_mode = L.am_mode;
    p.n_decls = L.n_decls;
    p.violations = L.violations;
    p.first_bad = L.first_bad;
    p.first_unmet = L.first_unmet;
    p.queue = static_cast<unsigned long long*>(L.workspace);
    p.err = L.err;
    if (cudaMemsetAsync(p.queue, 0, sizeof(unsigned long long), s) != cudaSuccess) return AMC_E_CUDA;
    int dev = 0, n_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    // several calls a claim only where every warp has at least two claims: a warp
    // checks the calls of its claim one after another (2,000 calls of 1,000 tokens:
    // 159 us with eight a claim, 43 so)
    const int64_t fair = L.n_calls / ((int64_t)n_sm * 10 * WD_WARPS * 2);
    p.claim = (int)(fair < 1 ? 1 : fair < WD_CLAIM ? fair : WD_CLAIM);
    const int64_t need = (L.n_calls + WD_WARPS * p.claim - 1) / (WD_WARPS * p.claim);
    const int grid = (int)(need < (int64_t)n_sm * 10 ? need : (int64_t)n_sm * 10);
    if (L.profile & 1) profile_begin(s);
    wd_kernel<<<grid, WD_WARPS * 32, 0, s>>>(p);
    if (L.profile & 2) profile_end(s);
    return cudaGetLastError() == cudaSuccess ? AMC_OK : AMC_E_CUDA;
}

}  // namespace amc

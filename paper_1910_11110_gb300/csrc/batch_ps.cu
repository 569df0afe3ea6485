// batch_ps.cu -- path-sensitive relation mode over a batch of structured
// programs (sm_103a).
//
// Semantics (Fig. Opsem: rules valid / invalid / rem-valid / rem-invalid,
// IF-True / IF-False, While-True / While-False): the conditions of If and
// While are isValid g or remIsValid g on the program's guard variable g, or
// opaque (x (+) y: both outcomes).  Control flow then depends on g alone, so
// for every other variable x the set of reachable pairs (status of g, status
// of x) -- a 5x5 bit matrix, bit 5 i + j for g = i, x = j -- is exactly the
// projection of the reachable stores; g's own statuses are a 5-bit set.  An
// op on x maps each row (a fixed g status) through the op's set image; an op
// on g moves whole rows; a condition keeps the rows whose g status makes it
// true (or false), never the stuck one (no rule applies to it, the path
// ends).  If: both branches from the filtered entry state, joined.  While:
// the loop-head state is the least X with X = entry U body(X restricted to
// the condition), the body's step sets are those of the pass from that
// fixpoint, and the loop is left with X restricted to the condition's
// negation.  Each variable's F is absorbing and does not stop the others, as
// in the opaque relation mode.  Step output: the statuses the op's variable
// may have after it (the union of its pair set's rows; 0 where the op is not
// reachable).
//
// Work: one warp per program from a longest-first queue.  Runs of up to 32
// op tokens on variables other than g are applied 32 at a time; an op on g, and
// every condition, touches every variable's pair set.  Entering a construct
// copies the whole state (every variable's pair set and g's set) to that level's
// save row, ELSE to the alt row.
// Programs of at most PS_SMALL_VARS variables take their tokens through a window
// of 32 in registers, the next 32 on their way; an ELSE or END is checked against
// the place its construct announced when it comes.
//   run_small: one warp, pair sets and the rows of the first PS_ROWS levels in
//     shared memory, four variables a lane at a time in a construct; lanes of a
//     run with the same variable are looked for with a tag per variable and
//     grouped (match.any) only when there are some.
//   run_part: a warp per 32 variables, for programs that are long against a
//     warp's part of the batch (their tokens at least the power of two at or
//     below that part, and PS_LONG): about three times the instructions in all,
//     half the latency.
// What bounds a batch is the latency of its longest programs (a token takes
// about 130 cycles of a warp by itself), and then instructions.  20,000 programs
// over 16 to 256 variables (64 M tokens), all by one warp each with rows in global
// memory and every token loaded where it was needed: 12.5 ms, 4.5 ms here; the
// longest of them alone (40,985 tokens, 130 variables) 8.3 and 2.8 ms; those of at
// most 5,037 tokens (54.5 M) 6.3 and 3.7 ms.  Sharing from half of a warp's part on
// took 7.2 ms where sharing from the part on took 6.0 (both with rows a word at a
// time); all of a program's variables in one warp's registers 11.0 where shared
// memory took 5.4; listing the variables that still grow when a loop runs again
// 6.0 where going over all took 5.4 (few loops do).  Other programs keep their pair
// sets in shared memory up to PS_SMEM_VARS variables, else in the workspace, and
// the rows in the workspace.
#include <cstdlib>

#include "amc_internal.cuh"
#include "batch_ps.cuh"

namespace amc {

namespace {

constexpr int PS_WARPS = 4;
constexpr int PS_SMEM_VARS = 1024;
constexpr uint32_t PS_MAX_PASSES = 64;
constexpr uint8_t ROWS_ALL = 31;

__device__ __forceinline__ bool ps_is_op(uint32_t ks) { return (ks & 0xE0u) == 0 && (ks & 15u) <= AMC_K_PW; }

struct PsTab {
    uint8_t img[16 * 32];         // set image per op index (kind << 1 | side)
    uint32_t flt[16];             // bit m: the set m may get stuck under the op
    uint8_t tgt[16 * 8];          // status an op maps status i to (row moves of an op on g)
    // the same for statuses 0 to 3 (the stuck one stays) as rotations, 5 bits each: of
    // a pair set's columns (an op on x), of its rows (an op on g)
    uint32_t rotx[16], rotg[16];
    uint32_t stuck[16];           // columns whose status gets stuck under the op
};

constexpr int PS_SMALL_VARS = 256;
constexpr int PS_SHARE = PS_SMALL_VARS / 32;      // warps on a long program
// tokens of the shortest one (one program of 1,024 to 2,047, over its guard alone: 725 us
// by one warp with its state in shared memory, 567 so; over 17 variables 342 and 261)
constexpr int64_t PS_LONG = 1024;

constexpr int PS_ROWS = 4;                        // construct levels whose rows lie in shared memory

union alignas(16) PsWarp {
    struct {
        uint32_t J[PS_SMEM_VARS];
        uint8_t stage[32];
    };
    struct {
        uint32_t j[PS_SMALL_VARS];
        uint32_t row[PS_ROWS][2][PS_SMALL_VARS];
        uint8_t tag[PS_SMALL_VARS];
        uint8_t ops[32];
    };
    uint32_t lanes[AMC_MAX_DEPTH][2][32];
};

__host__ __device__ constexpr uint32_t row_mask(uint32_t rows)
{
    uint32_t m = 0;
    for (int i = 0; i < 5; ++i)
        if ((rows >> i) & 1u) m |= 31u << (5 * i);
    return m;
}

__device__ __forceinline__ uint32_t proj(uint32_t J)
{
    const uint32_t a = J | (J >> 10) | (J >> 20);
    return (a | (a >> 5)) & 31u;
}

// rows kept on the then and the else side of condition c (0 opaque, 1 isValid g,
// 2 remIsValid g): statuses 0 (I,I) 1 (V,I) 2 (I,V) 3 (V,V), the stuck one on neither
__device__ __forceinline__ uint32_t then_rows(uint32_t c) { return c == 0 ? ROWS_ALL : c == 1 ? 0x0Au : 0x0Cu; }
__device__ __forceinline__ uint32_t else_rows(uint32_t c) { return c == 0 ? ROWS_ALL : c == 1 ? 0x05u : 0x03u; }
// the same as masks of pair sets
__device__ __forceinline__ uint32_t then_mask(uint32_t c)
{
    return c == 0 ? row_mask(ROWS_ALL) : c == 1 ? row_mask(0x0Au) : row_mask(0x0Cu);
}
__device__ __forceinline__ uint32_t else_mask(uint32_t c)
{
    return c == 0 ? row_mask(ROWS_ALL) : c == 1 ? row_mask(0x05u) : row_mask(0x03u);
}

template <bool SMEM>
__device__ void run_ps(const PsParams& p, int64_t prog, PsWarp& S, const PsTab& T)
{
    const int lane = threadIdx.x & 31;
    const uint32_t lt = lanemask_lt();
    const int64_t t0 = p.prog_tok_off[prog], t1 = p.prog_tok_off[prog + 1];
    const int32_t nv = p.prog_nvars[prog];
    const int64_t vo = p.prog_var_off[prog];
    const int32_t g = p.prog_guard[prog];
    uint32_t* J = SMEM ? S.J : p.J + vo;
    auto row_of = [&](int d, int k) { return p.save + ((int64_t)d * 2 + k) * p.total_vars + vo; };
    const uint32_t vi = 1u << AMC_ST_VI;
    uint32_t G = g >= 0 ? (p.init_mask ? p.init_mask[vo + g] : vi) : 1u;     // no guard: a single row
    for (int32_t x = lane; x < nv; x += 32) {
        const uint32_t m = p.init_mask ? p.init_mask[vo + x] : vi;
        uint32_t j = 0;
#pragma unroll
        for (int i = 0; i < 5; ++i)
            if ((G >> i) & 1u) j |= m << (5 * i);
        J[x] = x == g ? 0u : j;
    }
    __syncwarp();
    // frames: kind | cond << 4, passes; construct, ELSE and END tokens; g sets
    int fk[AMC_MAX_DEPTH], fpass[AMC_MAX_DEPTH];
    int64_t fpos[AMC_MAX_DEPTH * 3] = {};
    uint32_t gsave[AMC_MAX_DEPTH], galt[AMC_MAX_DEPTH];
    int depth = 0;
    int64_t ff = INT64_MAX;
    bool bad = false;
    int64_t pos = t0;
    auto range_end = [&]() -> int64_t { return depth ? fpos[(depth - 1) * 3 + 2] : t1; };
    auto keep = [&](uint32_t rows) {            // every pair set restricted to rows
        const uint32_t m = row_mask(rows);
        for (int32_t x = lane; x < nv; x += 32) J[x] &= m;
        G &= rows;
    };
    while (pos < t1 && !bad) {
        const uint32_t ks0 = p.tok[pos];
        const uint32_t k0 = ks0 & 15u;
        if (ps_is_op(ks0)) {
            const int32_t v0 = p.payload[pos];
            if (v0 == g && g >= 0) {
                // an op on g: rows move, g's set maps through the op
                const uint32_t o = (k0 << 1) | ((ks0 >> 4) & 1u);
                if ((T.flt[o] >> G) & 1u) ff = min(ff, pos - t0);
                for (int32_t x = lane; x < nv; x += 32) {
                    if (x == g) continue;
                    const uint32_t j = J[x];
                    uint32_t out = 0;
#pragma unroll
                    for (int i = 0; i < 5; ++i) out |= ((j >> (5 * i)) & 31u) << (5 * T.tgt[o * 8 + i]);
                    J[x] = out;
                }
                G = T.img[o * 32 + G];
                if (lane == 0) p.step_mask[pos] = (uint8_t)G;
                __syncwarp();
                ++pos;
                continue;
            }
            // a run of up to 32 op tokens on variables other than g
            const int64_t lim = range_end();
            const int64_t q = pos + lane;
            const uint32_t ks = q < lim ? p.tok[q] : 0xFFu;
            const int32_t pl = q < lim ? p.payload[q] : -1;
            const bool opx = ps_is_op(ks) && !(pl == g && g >= 0);
            const uint32_t opm = __ballot_sync(0xffffffffu, opx);
            const int cnt = (~opm) ? __ffs(~opm) - 1 : 32;
            const bool act = lane < cnt;
            int32_t v = act ? pl : -1;
            if (act && (v < 0 || v >= nv)) {
                raise_error(p.err, AMC_E_RANGE);
                v = -1;
            }
            S.stage[lane] = (uint8_t)(((ks & 15u) << 1) | ((ks >> 4) & 1u));
            __syncwarp();
            const uint32_t key = (act && v >= 0) ? (uint32_t)v : 0x80000000u + lane;
            const uint32_t peers = __match_any_sync(0xffffffffu, key);
            if (act && v >= 0 && (peers & lt) == 0) {
                uint32_t j = J[v];
                for (uint32_t rest = peers; rest; rest &= rest - 1) {
                    const int L = __ffs(rest) - 1;
                    const uint32_t o = S.stage[L];
                    if ((T.flt[o] >> proj(j)) & 1u) ff = min(ff, pos + L - t0);
                    uint32_t out = 0;
#pragma unroll
                    for (int i = 0; i < 5; ++i) out |= (uint32_t)T.img[o * 32 + ((j >> (5 * i)) & 31u)] << (5 * i);
                    j = out;
                    p.step_mask[pos + L] = (uint8_t)proj(j);
                }
                J[v] = j;
            }
            if (act && v < 0) p.step_mask[q] = 0;
            __syncwarp();
            pos += cnt;
        } else if (k0 == AMC_T_IF || k0 == AMC_T_WHILE) {
            const uint32_t c = ks0 >> 4;
            const int64_t lim = range_end();
            const int64_t len = p.payload[pos];
            int64_t e = -1, end;
            if (k0 == AMC_T_IF) {
                e = pos + 1 + len;
                end = (len >= 0 && e < lim && p.tok[e] == AMC_T_ELSE) ? e + 1 + (int64_t)p.payload[e] : -1;
            } else {
                end = pos + 1 + len;
            }
            if (c > 2 || (c && g < 0) || len < 0 || end <= pos || end >= lim || p.tok[end] != AMC_T_END ||
                depth >= AMC_MAX_DEPTH) {
                bad = true;
                break;
            }
            const int d = depth;
            uint32_t* sv = row_of(d, 0);
            for (int32_t x = lane; x < nv; x += 32) sv[x] = J[x];
            gsave[d] = G;
            __syncwarp();
            const uint32_t tr = then_rows(c), er = else_rows(c);
            if (tr != ROWS_ALL) keep(tr);
            __syncwarp();
            fk[d] = (int)(k0 | (c << 4));
            fpass[d] = 0;
            fpos[d * 3 + 0] = pos;
            fpos[d * 3 + 1] = e;
            fpos[d * 3 + 2] = end;
            ++depth;
            if (lane == 0) p.step_mask[pos] = 0;
            ++pos;
        } else if (ks0 == AMC_T_ELSE) {
            if (!depth || (fk[depth - 1] & 15) != AMC_T_IF || fpos[(depth - 1) * 3 + 1] != pos) {
                bad = true;
                break;
            }
            const int d = depth - 1;
            const uint32_t tr = then_rows((uint32_t)fk[d] >> 4), er = else_rows((uint32_t)fk[d] >> 4);
            uint32_t* sv = row_of(d, 0);
            uint32_t* al = row_of(d, 1);
            const uint32_t m = row_mask(er);
            for (int32_t x = lane; x < nv; x += 32) {
                al[x] = J[x];                    // then-results
                J[x] = sv[x] & m;                // the entry state on the IF-False paths
            }
            galt[d] = G;
            G = gsave[d] & er;
            __syncwarp();
            if (lane == 0) p.step_mask[pos] = 0;
            ++pos;
        } else if (ks0 == AMC_T_END) {
            if (!depth || fpos[(depth - 1) * 3 + 2] != pos) {
                bad = true;
                break;
            }
            const int d = depth - 1;
            if (lane == 0) p.step_mask[pos] = 0;
            const uint32_t tr = then_rows((uint32_t)fk[d] >> 4), er = else_rows((uint32_t)fk[d] >> 4);
            uint32_t* sv = row_of(d, 0);
            if ((fk[d] & 15) == AMC_T_IF) {
                const uint32_t* al = row_of(d, 1);
                for (int32_t x = lane; x < nv; x += 32) J[x] |= al[x];
                G |= galt[d];
                __syncwarp();
                --depth;
                ++pos;
            } else {
                // loop head: X = X U body(X on the While-True paths)
                bool grew = false;
                for (int32_t x = lane; x < nv; x += 32) {
                    const uint32_t a = sv[x], b = a | J[x];
                    grew |= b != a;
                    sv[x] = b;
                }
                const uint32_t gn = gsave[d] | G;
                grew |= gn != gsave[d];
                gsave[d] = gn;
                __syncwarp();
                const uint32_t rows = __any_sync(0xffffffffu, grew) ? tr : er;
                const uint32_t m = row_mask(rows);
                for (int32_t x = lane; x < nv; x += 32) J[x] = sv[x] & m;
                G = gn & rows;
                __syncwarp();
                if (rows == tr && __any_sync(0xffffffffu, grew)) {
                    if (++fpass[d] > (int)PS_MAX_PASSES) {
                        bad = true;
                        break;
                    }
                    pos = fpos[d * 3] + 1;          // the body again from the grown head
                } else {
                    --depth;                        // While-False: leave with the head's other rows
                    ++pos;
                }
            }
        } else {
            bad = true;
        }
    }
    if (!bad && depth) bad = true;
    if (bad && lane == 0) raise_error(p.err, AMC_E_INVALID);
    __syncwarp();
#pragma unroll
    for (int o = 16; o; o >>= 1) ff = min(ff, (int64_t)__shfl_xor_sync(0xffffffffu, (long long)ff, o));
    if (lane == 0) p.prog_first_fault[prog] = ff == INT64_MAX ? -1 : ff;
    for (int32_t x = lane; x < nv; x += 32) p.final_mask[vo + x] = (uint8_t)(x == g ? G : proj(J[x]));
}

// pair set after an op on the variable: its columns move (rotx)
__device__ __forceinline__ uint32_t op_on_x(uint32_t J, uint32_t rot)
{
    uint32_t out = J & (0x108421u << 4);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t c = J & (0x108421u << i);
        out |= __funnelshift_l(c, c, rot >> (5 * i));
    }
    return out;
}
// ... on g: its rows move (rotg)
__device__ __forceinline__ uint32_t op_on_g(uint32_t J, uint32_t rot)
{
    uint32_t out = J & (31u << 20);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t c = J & (31u << (5 * i));
        out |= __funnelshift_l(c, c, rot >> (5 * i));
    }
    return out;
}

// An open construct: kind | cond << 4, passes << 8, g's set before it or at the
// loop's head << 16, g's set after the then part << 24; opener, ELSE (-1: a
// While), END (-1: not announced yet).  The innermost one is kept in registers.
struct alignas(16) PsFrame {
    uint32_t meta;
    int open, els, end;
};

// A program of at most PS_SMALL_VARS variables and fewer than 2^31 - 64 tokens.
__device__ void run_small(const PsParams& p, int64_t prog, PsWarp& S, const PsTab& T)
{
    const int lane = threadIdx.x & 31;
    const uint32_t lt = lanemask_lt();
    const int64_t t0 = p.prog_tok_off[prog], vo = p.prog_var_off[prog];
    const int len = (int)(p.prog_tok_off[prog + 1] - t0);
    const int32_t nv = p.prog_nvars[prog], g = p.prog_guard[prog];
    const uint8_t* tok = p.tok + t0;
    const int32_t* payload = p.payload + t0;
    uint8_t* step = p.step_mask + t0;
    uint32_t* J = S.j;
    uint4* J4 = reinterpret_cast<uint4*>(S.j);
    const int n4 = (nv + 3) >> 2;                          // a lane takes four variables at a time
    auto row4 = [&](int d, int k) { return reinterpret_cast<uint4*>(S.row[d][k]); };
    auto deep = [&](int d, int k) { return p.save + ((int64_t)d * 2 + k) * p.total_vars + vo; };
    const uint32_t vi = 1u << AMC_ST_VI;
    uint32_t G = g >= 0 ? (p.init_mask ? p.init_mask[vo + g] : vi) : 1u;     // no guard: a single row
    for (int32_t x = lane; x < 4 * n4; x += 32) {
        const uint32_t m = x < nv && x != g ? (p.init_mask ? p.init_mask[vo + x] : vi) : 0u;
        uint32_t j = 0;
#pragma unroll
        for (int i = 0; i < 5; ++i)
            if ((G >> i) & 1u) j |= m << (5 * i);
        J[x] = j;
    }
    __syncwarp();
    PsFrame f = {}, below[AMC_MAX_DEPTH];
    int depth = 0;
    int ff = INT32_MAX;
    bool found = false;                  // a fault before every token still to come
    bool bad = false, range = false;
    int pos = 0;
    // tokens [wb, wb + 32), and the 32 after them
    int wb = -64;
    uint32_t ks = 0, nks = 0;
    int32_t pl = 0, npl = 0;
    uint32_t runs = 0;                   // ops on other variables than g
    while (pos < len && !bad) {
        if (pos >= wb + 32 || pos < wb) {
            if (pos == wb + 32) {
                ks = nks;
                pl = npl;
            } else {
                const bool in = lane < len - pos;
                ks = in ? tok[pos + lane] : 0xFFu;
                pl = in ? payload[pos + lane] : 0;
            }
            wb = pos;
            const bool more = lane < len - wb - 32;
            nks = more ? tok[wb + 32 + lane] : 0xFFu;
            npl = more ? payload[wb + 32 + lane] : 0;
            const bool op = ps_is_op(ks);
            runs = __ballot_sync(0xffffffffu, op && !(pl == g && g >= 0));
            if (!op && lane < len - wb) step[wb + lane] = 0;
        }
        const int off = pos - wb;
        const uint32_t left = runs >> off;
        if (left & 1u) {
            // the run of ops from here on (at most to the window's end)
            const int cnt = ~left ? __ffs(~left) - 1 : 32;
            const bool act = lane >= off && lane < off + cnt;
            const bool valid = act && pl >= 0 && pl < nv;
            const uint32_t o = ((ks & 15u) << 1) | ((ks >> 4) & 1u);
            if (valid) S.tag[pl] = (uint8_t)lane;
            if (act && !valid) {
                range = true;
                step[wb + lane] = 0;
            }
            __syncwarp();
            const bool lost = valid && S.tag[pl] != lane;
            const bool dup = __any_sync(0xffffffffu, lost);
            if (!dup) {
                if (valid) {
                    const uint32_t j = J[pl];
                    if (!found && (j & T.stuck[o])) ff = min(ff, wb + lane);
                    const uint32_t out = op_on_x(j, T.rotx[o]);
                    J[pl] = out;
                    step[wb + lane] = (uint8_t)proj(out);
                }
            } else {
                S.ops[lane] = (uint8_t)o;
                const uint32_t peers = lanes_with_same((uint32_t)pl, valid, lost);
                __syncwarp();
                if (valid && (peers & lt) == 0) {
                    uint32_t j = J[pl];
                    for (uint32_t rest = peers; rest; rest &= rest - 1) {
                        const int L = __ffs(rest) - 1;
                        const uint32_t x = S.ops[L];
                        if (j & T.stuck[x]) ff = min(ff, wb + L);
                        j = op_on_x(j, T.rotx[x]);
                        step[wb + L] = (uint8_t)proj(j);
                    }
                    J[pl] = j;
                }
            }
            pos += cnt;
            if (!found) found = __any_sync(0xffffffffu, ff < pos);
            __syncwarp();
            continue;
        }
        const uint32_t k0 = __shfl_sync(0xffffffffu, ks, off);
        const int32_t l0 = __shfl_sync(0xffffffffu, pl, off);
        // place after the part that the token announces (-1: none in the program)
        const int to = l0 >= 0 && l0 < len - pos - 1 ? pos + 1 + l0 : -1;
        const int d = depth - 1;
        const uint32_t c = (f.meta >> 4) & 3u;             // the innermost construct's condition
        if (k0 == AMC_T_END) {
            if (depth < 1 || f.end != pos) {
                bad = true;
                break;
            }
            bool again = false;
            if (f.els >= 0) {
                if (d < PS_ROWS) {
                    const uint4* al = row4(d, 1);
                    for (int i = lane; i < n4; i += 32) {
                        const uint4 a = al[i];
                        uint4 j = J4[i];
                        j.x |= a.x, j.y |= a.y, j.z |= a.z, j.w |= a.w;
                        J4[i] = j;
                    }
                } else {
                    for (int x = lane; x < nv; x += 32) J[x] |= deep(d, 1)[x];
                }
                G |= f.meta >> 24;
            } else {
                // loop head: X = X U body(X on the While-True paths)
                uint32_t grew = 0;
                if (d < PS_ROWS) {
                    uint4* sv = row4(d, 0);
                    for (int i = lane; i < n4; i += 32) {
                        uint4 a = sv[i], j = J4[i];
                        grew |= (j.x & ~a.x) | (j.y & ~a.y) | (j.z & ~a.z) | (j.w & ~a.w);
                        a.x |= j.x, a.y |= j.y, a.z |= j.z, a.w |= j.w;
                        sv[i] = a;
                        J4[i] = a;
                    }
                } else {
                    for (int x = lane; x < nv; x += 32) {
                        const uint32_t a = deep(d, 0)[x], j = J[x];
                        grew |= j & ~a;
                        deep(d, 0)[x] = a | j;
                        J[x] = a | j;
                    }
                }
                const uint32_t gs = (f.meta >> 16) & 31u;
                again = __any_sync(0xffffffffu, grew != 0) || (G & ~gs) != 0;
                f.meta |= G << 16;
                // again, or out with the head's While-False rows
                G = (gs | G) & (again ? then_rows(c) : else_rows(c));
                if (c) {
                    const uint32_t m = again ? then_mask(c) : else_mask(c);
                    __syncwarp();
                    for (int x = lane; x < nv; x += 32) J[x] &= m;
                }
            }
            if (again) {
                f.meta += 1u << 8;
                if (((f.meta >> 8) & 255u) > PS_MAX_PASSES) {
                    bad = true;
                    break;
                }
                found = false;
                pos = f.open;                    // the body again from the grown head
            } else {
                --depth;
                if (depth) f = below[depth - 1];
            }
        } else if (k0 == AMC_T_ELSE) {
            if (depth < 1 || f.els != pos || to < 0) {
                bad = true;
                break;
            }
            f.end = to;
            // then-results aside; the entry state on the IF-False paths
            const uint32_t m = else_mask(c);
            if (d < PS_ROWS) {
                const uint4* sv = row4(d, 0);
                uint4* al = row4(d, 1);
                for (int i = lane; i < n4; i += 32) {
                    uint4 a = sv[i];
                    al[i] = J4[i];
                    a.x &= m, a.y &= m, a.z &= m, a.w &= m;
                    J4[i] = a;
                }
            } else {
                for (int x = lane; x < nv; x += 32) {
                    deep(d, 1)[x] = J[x];
                    J[x] = deep(d, 0)[x] & m;
                }
            }
            f.meta |= G << 24;
            G = (f.meta >> 16) & else_rows(c);
        } else if ((k0 & 15u) == AMC_T_IF || (k0 & 15u) == AMC_T_WHILE) {
            const uint32_t cn = k0 >> 4;
            if (cn > 2 || (cn && g < 0) || to < 0 || depth >= AMC_MAX_DEPTH) {
                bad = true;
                break;
            }
            const uint32_t m = then_mask(cn);
            if (depth < PS_ROWS) {
                uint4* sv = row4(depth, 0);
                for (int i = lane; i < n4; i += 32) {
                    uint4 j = J4[i];
                    sv[i] = j;
                    if (cn) {
                        j.x &= m, j.y &= m, j.z &= m, j.w &= m;
                        J4[i] = j;
                    }
                }
            } else {
                for (int x = lane; x < nv; x += 32) {
                    deep(depth, 0)[x] = J[x];
                    J[x] &= m;
                }
            }
            if (depth) below[depth - 1] = f;
            ++depth;
            const bool is_if = (k0 & 15u) == AMC_T_IF;
            f.meta = k0 | G << 16;
            f.open = pos;
            f.els = is_if ? to : -1;
            f.end = is_if ? -1 : to;
            G &= then_rows(cn);
        } else if (ps_is_op(k0)) {
            // an op on g: rows move, g's set maps through the op
            const uint32_t o = ((k0 & 15u) << 1) | ((k0 >> 4) & 1u), rot = T.rotg[o];
            if ((T.flt[o] >> G) & 1u) ff = min(ff, pos);
            for (int i = lane; i < n4; i += 32) {          // (g's own entry stays empty)
                uint4 j = J4[i];
                j.x = op_on_g(j.x, rot), j.y = op_on_g(j.y, rot), j.z = op_on_g(j.z, rot), j.w = op_on_g(j.w, rot);
                J4[i] = j;
            }
            G = T.img[o * 32 + G];
            if (lane == 0) step[pos] = (uint8_t)G;
        } else {
            bad = true;
            break;
        }
        ++pos;
        __syncwarp();
    }
    bad |= depth != 0;
    if (range) raise_error(p.err, AMC_E_RANGE);
    __syncwarp();
    if (bad && lane == 0) raise_error(p.err, AMC_E_INVALID);
    ff = __reduce_min_sync(0xffffffffu, ff);
    if (lane == 0) p.prog_first_fault[prog] = ff == INT32_MAX ? -1 : ff;
    for (int32_t x = lane; x < nv; x += 32) p.final_mask[vo + x] = (uint8_t)(x == g ? G : proj(J[x]));
}

// Variables 32 w to 32 w + 31 of such a program, one per lane, pair sets in
// registers and rows in a column of shared memory per lane.  Given g's statuses no
// variable depends on another, nor does the number of passes it needs: the warps
// of a program go through all of its tokens, each by itself, and g with them.
__device__ void run_part(const PsParams& p, int64_t prog, uint32_t (*rows)[2][32], const PsTab& T, int w)
{
    const int lane = threadIdx.x & 31;
    const int64_t t0 = p.prog_tok_off[prog], vo = p.prog_var_off[prog];
    const int len = (int)(p.prog_tok_off[prog + 1] - t0);
    const int32_t nv = p.prog_nvars[prog], g = p.prog_guard[prog];
    const uint8_t* tok = p.tok + t0;
    const int32_t* payload = p.payload + t0;
    uint8_t* step = p.step_mask + t0;
    const int32_t xl = lane + 32 * w;                      // the lane's variable
    const uint32_t vi = 1u << AMC_ST_VI;
    uint32_t G = g >= 0 ? (p.init_mask ? p.init_mask[vo + g] : vi) : 1u;     // no guard: a single row
    uint32_t J = 0;
    {
        const uint32_t m = xl < nv && xl != g ? (p.init_mask ? p.init_mask[vo + xl] : vi) : 0u;
#pragma unroll
        for (int i = 0; i < 5; ++i)
            if ((G >> i) & 1u) J |= m << (5 * i);
    }
    PsFrame f = {}, below[AMC_MAX_DEPTH];
    int depth = 0;
    int ff = INT32_MAX;
    bool bad = false, range = false;
    int pos = 0;
    // tokens [wb, wb + 32), and the 32 after them
    int wb = -64;
    uint32_t ks = 0, nks = 0;
    int32_t pl = 0, npl = 0;
    uint32_t runs = 0;                                     // ops on other variables than g
    uint32_t own = 0;                                      // the lane's own among them
    uint32_t wrong = 0;                                    // variable out of range
    uint32_t word = 0;                                     // the token's op: rotx | statuses that get stuck << 20
    int to = -1;                                           // place after the part it announces (-1: none in the program)
    while (pos < len && !bad) {
        if (pos >= wb + 32 || pos < wb) {
            if (pos == wb + 32) {
                ks = nks;
                pl = npl;
            } else {
                const bool in = lane < len - pos;
                ks = in ? tok[pos + lane] : 0xFFu;
                pl = in ? payload[pos + lane] : 0;
            }
            wb = pos;
            const bool more = lane < len - wb - 32;
            nks = more ? tok[wb + 32 + lane] : 0xFFu;
            npl = more ? payload[wb + 32 + lane] : 0;
            const bool op = ps_is_op(ks), opx = op && !(pl == g && g >= 0);
            runs = __ballot_sync(0xffffffffu, opx);
            if (!op && w == 0 && lane < len - wb) step[wb + lane] = 0;
            const bool valid = pl >= 0 && pl < nv;
            wrong = __ballot_sync(0xffffffffu, opx && !valid);
            own = __ballot_sync(0xffffffffu, opx && valid && (pl >> 5) == w);
#pragma unroll
            for (int b = 0; b < 5; ++b) {
                const uint32_t m = __ballot_sync(0xffffffffu, (pl >> b) & 1);
                own &= (lane >> b) & 1 ? m : ~m;
            }
            const uint32_t o = op ? ((ks & 15u) << 1) | (ks >> 4) : 0u;
            word = T.rotx[o] | (T.stuck[o] & 15u) << 20;
            to = pl >= 0 && pl < len - wb - lane - 1 ? wb + lane + 1 + pl : -1;
        }
        // the run of ops from here on (at most to the window's end), and the token
        // after it
        const int off = pos - wb;
        const uint32_t left = runs >> off;
        const int cnt = ~left ? __ffs(~left) - 1 : 32;
        const uint32_t k0 = __shfl_sync(0xffffffffu, ks, off + cnt);
        const int next = __shfl_sync(0xffffffffu, to, off + cnt);
        if (cnt) {
            const uint32_t run = (cnt < 32 ? (1u << cnt) - 1u : ~0u) << off;
            if (run & wrong) {
                range = true;
                if (w == 0 && ((run & wrong) >> lane & 1u)) step[wb + lane] = 0;
            }
            // a lane's ops in order, the next one's word fetched while one is applied
            uint32_t mine = own & run;
            uint32_t x = __shfl_sync(0xffffffffu, word, __ffs(mine) - 1);       // (none: any word will do)
            while (__any_sync(0xffffffffu, mine != 0)) {
                const uint32_t rest = mine & (mine - 1);
                const uint32_t xn = __shfl_sync(0xffffffffu, word, __ffs(rest) - 1);
                if (mine) {
                    const int at = wb + __ffs(mine) - 1;
                    if (J & ((x >> 20) * 0x108421u)) ff = min(ff, at);
                    J = op_on_x(J, x);
                    step[at] = (uint8_t)proj(J);
                }
                mine = rest;
                x = xn;
            }
            pos += cnt;
            if (off + cnt >= 32 || pos >= len) continue;
        }
        const uint32_t c = (f.meta >> 4) & 3u;
        uint32_t(*const row)[32] = rows[max(depth - 1, 0)];
        if (k0 == AMC_T_END) {
            if (depth < 1 || f.end != pos) {
                bad = true;
                break;
            }
            bool again = false;
            if (f.els >= 0) {
                J |= row[1][lane];
                G |= f.meta >> 24;
            } else {
                const uint32_t head = row[0][lane], gs = (f.meta >> 16) & 31u;
                again = __any_sync(0xffffffffu, (J & ~head) != 0) || (G & ~gs) != 0;
                f.meta |= G << 16;
                G = (gs | G) & (again ? then_rows(c) : else_rows(c));
                row[0][lane] = head | J;
                J = (head | J) & (again ? then_mask(c) : else_mask(c));
            }
            if (again) {
                f.meta += 1u << 8;
                if (((f.meta >> 8) & 255u) > PS_MAX_PASSES) {
                    bad = true;
                    break;
                }
                pos = f.open;
            } else {
                --depth;
                if (depth) f = below[depth - 1];
            }
        } else if (k0 == AMC_T_ELSE) {
            if (depth < 1 || f.els != pos || next < 0) {
                bad = true;
                break;
            }
            f.end = next;
            row[1][lane] = J;
            J = row[0][lane] & else_mask(c);
            f.meta |= G << 24;
            G = (f.meta >> 16) & else_rows(c);
        } else if ((k0 & 15u) == AMC_T_IF || (k0 & 15u) == AMC_T_WHILE) {
            const uint32_t cn = k0 >> 4;
            if (cn > 2 || (cn && g < 0) || next < 0 || depth >= AMC_MAX_DEPTH) {
                bad = true;
                break;
            }
            rows[depth][0][lane] = J;
            J &= then_mask(cn);
            if (depth) below[depth - 1] = f;
            ++depth;
            const bool is_if = (k0 & 15u) == AMC_T_IF;
            f.meta = k0 | G << 16;
            f.open = pos;
            f.els = is_if ? next : -1;
            f.end = is_if ? -1 : next;
            G &= then_rows(cn);
        } else if (ps_is_op(k0)) {
            const uint32_t o = ((k0 & 15u) << 1) | (k0 >> 4), rot = T.rotg[o];
            if ((T.flt[o] >> G) & 1u) ff = min(ff, pos);
            J = op_on_g(J, rot);
            G = T.img[o * 32 + G];
            if (lane == 0 && w == 0) step[pos] = (uint8_t)G;
        } else {
            bad = true;
            break;
        }
        ++pos;
    }
    bad |= depth != 0;
    if (range) raise_error(p.err, AMC_E_RANGE);
    __syncwarp();
    if (bad && lane == 0) raise_error(p.err, AMC_E_INVALID);
    ff = __reduce_min_sync(0xffffffffu, ff);
    if (lane == 0) {
        // the word starts as -1, the largest unsigned one
        atomicMin(reinterpret_cast<unsigned long long*>(p.prog_first_fault + prog),
                  ff == INT32_MAX ? ~0ull : (unsigned long long)ff);
    }
    if (xl < nv) p.final_mask[vo + xl] = (uint8_t)(xl == g ? G : proj(J));
}

__global__ void __launch_bounds__(PS_WARPS * 32) ps_kernel(const PsParams p)
{
    __shared__ PsWarp warps[PS_WARPS];
    __shared__ PsTab tab;
    for (int i = threadIdx.x; i < 16 * 32; i += blockDim.x) tab.img[i] = p.tab.img[i];
    if (threadIdx.x < 16) tab.flt[threadIdx.x] = p.tab.flt[threadIdx.x];
    for (int i = threadIdx.x; i < 16 * 8; i += blockDim.x) {
        const int o = i >> 3, s = i & 7;
        const uint32_t im = s < 5 ? p.tab.img[o * 32 + (1 << s)] : 0u;
        tab.tgt[i] = (uint8_t)(im ? __ffs(im) - 1 : 0);
    }
    __syncthreads();
    if (threadIdx.x < 16) {
        uint32_t x = 0, g = 0, st = 0;
        for (int i = 0; i < 4; ++i) {
            const int by = (int)tab.tgt[threadIdx.x * 8 + i] - i;
            x |= ((uint32_t)by & 31u) << (5 * i);
            g |= ((uint32_t)(5 * by) & 31u) << (5 * i);
            if ((tab.flt[threadIdx.x] >> (1 << i)) & 1u) st |= 0x108421u << i;
        }
        tab.rotx[threadIdx.x] = x;
        tab.rotg[threadIdx.x] = g;
        tab.stuck[threadIdx.x] = st;
    }
    __syncthreads();
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (;;) {
        // the long programs come first, eight items each: the warps that share one
        const int64_t n_long = *p.n_long;
        int64_t i = 0;
        if (lane == 0) i = (int64_t)atomicAdd(reinterpret_cast<unsigned long long*>(p.queue_head), 1ull);
        i = __shfl_sync(0xffffffffu, (long long)i, 0);
        const bool is_long = i < n_long * PS_SHARE;
        const int part = is_long ? (int)(i % PS_SHARE) : 0;
        i = is_long ? i / PS_SHARE : i - n_long * (PS_SHARE - 1);
        if (i >= p.n_progs) break;
        const int64_t prog = p.order ? p.order[i] : i;
        const int64_t t0 = p.prog_tok_off[prog], t1 = p.prog_tok_off[prog + 1], vo = p.prog_var_off[prog];
        const int32_t nv = p.prog_nvars[prog], g = p.prog_guard[prog];
        if (t0 < 0 || t1 < t0 || t1 > p.n_tokens || nv < 0 || vo < 0 || p.prog_var_off[prog + 1] - vo != nv || g < -1 ||
            g >= nv) {
            if (lane == 0) raise_error(p.err, AMC_E_INVALID);
            continue;
        }
        if (nv <= PS_SMALL_VARS && t1 - t0 < INT32_MAX - 64) {
            if (is_long && part * 32 < max(nv, 1)) run_part(p, prog, warps[wid].lanes, tab, part);
            else if (!is_long) run_small(p, prog, warps[wid], tab);
        } else if (part) {
            continue;
        } else if (nv <= PS_SMEM_VARS) {
            run_ps<true>(p, prog, warps[wid], tab);
        } else {
            run_ps<false>(p, prog, warps[wid], tab);
        }
        __syncwarp();
    }
}

// queue order: programs by decreasing length bucket (counting sort by
// floor(log2(tokens)), any order within a bucket)
__device__ __forceinline__ int ps_bucket(int64_t len) { return len <= 0 ? 63 : 63 - (64 - __clzll(len)); }

__global__ void ps_count_kernel(const int64_t* __restrict__ tok_off, int64_t n, int32_t* __restrict__ counts)
{
    __shared__ int32_t c[64];
    if (threadIdx.x < 64) c[threadIdx.x] = 0;
    __syncthreads();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        atomicAdd(&c[ps_bucket(tok_off[i + 1] - tok_off[i])], 1);
    __syncthreads();
    if (threadIdx.x < 64 && c[threadIdx.x]) atomicAdd(&counts[threadIdx.x], c[threadIdx.x]);
}

__global__ void ps_scan_kernel(int32_t* __restrict__ counts, int64_t* __restrict__ boff, int last, int64_t* n_long)
{
    if (threadIdx.x == 0) {
        int64_t s = 0;
        for (int b = 0; b < 64; ++b) {
            boff[b] = s;
            s += counts[b];
            if (b == last) *n_long = s;            // programs up to this bucket are shared
            counts[b] = 0;
        }
    }
}

__global__ void ps_order_kernel(const int64_t* __restrict__ tok_off, int64_t n, const int64_t* __restrict__ boff,
                                int32_t* __restrict__ cursor, int32_t* __restrict__ order, int64_t* first_fault)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int b = ps_bucket(tok_off[i + 1] - tok_off[i]);
    order[boff[b] + atomicAdd(&cursor[b], 1)] = (int32_t)i;
    first_fault[i] = -1;
}

struct PsLayout {
    size_t J, save, order, counts, boff, head, n_long, total;
};

PsLayout layout(int64_t n_progs, int64_t total_vars)
{
    PsLayout L;
    size_t o = 0;
    auto take = [&](size_t b) { const size_t at = o; o += align_up(b, 256); return at; };
    const size_t tv = (size_t)(total_vars > 0 ? total_vars : 1);
    L.J = take(4 * tv);
    L.save = take(4 * tv * 2 * AMC_MAX_DEPTH);
    L.order = take(4 * (size_t)n_progs + 4);
    L.counts = take(256);
    L.boff = take(512);
    L.head = take(256);
    L.n_long = take(256);
    L.total = o;
    return L;
}

}  // namespace

size_t batch_ps_workspace_bytes(int64_t n_progs, int64_t total_vars) { return layout(n_progs, total_vars).total; }

int launch_batch_ps(const PsLaunch& B, cudaStream_t s)
{
    PsParams p{};
    p.tok = B.tok;
    p.payload = B.payload;
    p.prog_tok_off = B.prog_tok_off;
    p.prog_nvars = B.prog_nvars;
    p.prog_var_off = B.prog_var_off;
    p.prog_guard = B.prog_guard;
    p.n_progs = B.n_progs;
    p.n_tokens = B.n_tokens;
    p.total_vars = B.total_vars;
    p.init_mask = B.init_mask;
    p.step_mask = B.step_mask;
    p.final_mask = B.final_mask;
    p.prog_first_fault = B.prog_first_fault;
    p.err = B.err;
    p.tab = host_set_tables();
    const PsLayout L = layout(B.n_progs, B.total_vars);
    uint8_t* w = static_cast<uint8_t*>(B.workspace);
    p.J = reinterpret_cast<uint32_t*>(w + L.J);
    p.save = reinterpret_cast<uint32_t*>(w + L.save);
    p.queue_head = reinterpret_cast<uint64_t*>(w + L.head);
    int32_t* order = reinterpret_cast<int32_t*>(w + L.order);
    int32_t* counts = reinterpret_cast<int32_t*>(w + L.counts);
    int64_t* boff = reinterpret_cast<int64_t*>(w + L.boff);
    int64_t* n_long = reinterpret_cast<int64_t*>(w + L.n_long);
    if (B.n_progs <= 0) return AMC_OK;
    if (cudaMemsetAsync(p.queue_head, 0, 8, s) != cudaSuccess) return AMC_E_CUDA;
    if (cudaMemsetAsync(counts, 0, 256, s) != cudaSuccess) return AMC_E_CUDA;
    ps_count_kernel<<<128, 256, 0, s>>>(B.prog_tok_off, B.n_progs, counts);
    int dev = 0, n_sm = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, ps_kernel, PS_WARPS * 32, 0);
    if (per_sm < 1) per_sm = 1;
    int64_t grid = (int64_t)n_sm * per_sm;
    // a program is shared when it is long against a warp's part of the batch
    const int64_t part = B.n_tokens / (grid * PS_WARPS);
    int last = 62;
    for (int64_t l = part > PS_LONG ? part : PS_LONG; l > 1; l >>= 1) --last;
    ps_scan_kernel<<<1, 32, 0, s>>>(counts, boff, last, n_long);
    ps_order_kernel<<<(unsigned)((B.n_progs + 255) / 256), 256, 0, s>>>(B.prog_tok_off, B.n_progs, boff, counts, order,
                                                                          B.prog_first_fault);
    p.order = order;
    p.n_long = n_long;
    const int64_t need = (B.n_progs * PS_SHARE + PS_WARPS - 1) / PS_WARPS;
    if (grid > need) grid = need;
    if (B.profile & 1) profile_begin(s);
    ps_kernel<<<(unsigned)grid, PS_WARPS * 32, 0, s>>>(p);
    if (B.profile & 2) profile_end(s);
    return cudaGetLastError() == cudaSuccess ? AMC_OK : AMC_E_CUDA;
}

}  // namespace amc

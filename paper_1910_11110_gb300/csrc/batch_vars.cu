// batch_vars.cu -- relation mode over structured programs, variable by variable
// (sm_103a).
//
// With opaque conditions (Fig. Opsem; If = union of its branches, While =
// closure of its body) the sets of statuses of two variables never meet: a
// variable's sets depend only on its own ops and on the constructs around them.
// So a program's ops are strung into one chain per variable, and a lane
// evaluates a chain from its variable's entry set, with the set in a register.
// What a program costs then is its ops, not how often its While bodies run for
// all their variables together: an op with no other op of its variable in its
// outermost construct (nearly every one) has a closed form -- in a While the set
// before it is the least X with X = m U f(X), reached in at most four steps of
// one table look-up, and the set after the construct is X; in Ifs alone it is m
// U f(m).
// Work: a warp per program.
//   1. Forward over the tokens, 32 at a time: depth by counting openers and ENDs,
//      every ELSE and END checked against the place its construct announced (one
//      ballot per level finds the announcement in force), the outermost open
//      construct and the open Whiles by ballots; each op is linked to the op
//      before it on its variable through a shared-memory table of the variables'
//      last ops, the first ops go to a list.
//   2. Lanes take chains from that list; a lane that is done takes the next.
// Ops that share their outermost construct with another op of their variable are
// interpreted over that construct: a frame per open construct that holds an op of
// the variable (entry set, then-result, first op), While by running its ops again
// from the grown set.
// What bounds it: instructions (about 16 warp instructions per token) and the
// latency of the chains' loads, at 24 warps an SM (8 KB of last ops each).
// 100,000 programs (320 M tokens): a warp per program that runs every op of a
// body again until all of its variables are done took 29.6 ms (77 warp
// instructions per token; the longest program alone about 20 ms), this takes 7.8
// ms.  Words of 8 bytes per op (with its constructs in it) took 11.1 ms: the
// resident programs no longer fit L2.  Walking the structure tokens of a window
// one by one took 8.7 ms, the warp turning to lanes in a group only when a third
// of it is in one 12.0 to 13.6 ms in place of 11.1.
#include <type_traits>

#include "amc_internal.cuh"
#include "batch.cuh"

namespace amc {

namespace {

constexpr int VWARPS = 4;                 // warps per CTA
constexpr int VCTAS = 6;                  // CTAs per SM (33 KB of shared memory each)
constexpr uint32_t NIL16 = 0xFFFFu;       // no position
constexpr int VAHEAD = 2;                 // windows of 32 tokens loaded together

// An op's word: next op of its variable (bits 0-15; 0: none, as no op comes
// before the first token), op index kind << 1 | side (16-19), inside a While
// (20), inside a construct (21), the next op shares its outermost construct
// (22), constructs around it (23-26).  A construct's word: END (0-15), ELSE
// (16-31, NIL16 for a While), constructs around it (32-35).  Positions are
// relative to the program's first token, constructs are numbered by their
// openers: the one around position q at depth d is the last one at that depth
// that opens before q.  Four bytes an op keep what
// the chains jump around in small: the programs of all resident warps fit L2.
constexpr uint32_t W_WHILE = 1u << 20, W_CONS = 1u << 21, W_MORE = 1u << 22;
__device__ __forceinline__ uint32_t w_next(uint32_t w) { return w & 0xFFFFu; }
__device__ __forceinline__ uint32_t w_op(uint32_t w) { return (w >> 16) & 15u; }
__device__ __forceinline__ uint32_t c_end(uint64_t c) { return (uint32_t)c & 0xFFFFu; }
__device__ __forceinline__ uint32_t c_else(uint64_t c) { return (uint32_t)c >> 16; }
__device__ __forceinline__ uint32_t c_depth(uint64_t c) { return (uint32_t)(c >> 32) & 15u; }
__device__ __forceinline__ uint32_t w_depth(uint32_t w) { return (w >> 23) & 15u; }

constexpr uint32_t VCONS = VARS_MAX_NV / 4;   // constructs whose words fit the shared memory of the last ops

struct VarSmem {
    __align__(8) uint16_t tail[VWARPS][VARS_MAX_NV];   // step 1: last ops; step 2: constructs
    uint8_t img[16 * 32];
    uint32_t flt[16];
};

__device__ __forceinline__ bool v_is_op(uint32_t ks) { return (ks & 0xE0u) == 0 && (ks & 15u) <= AMC_K_PW; }

__device__ void run_program(const BatchParams& p, int64_t prog, VarSmem& S, uint16_t* tail)
{
    const int lane = threadIdx.x & 31;
    const uint32_t lt = lanemask_lt();
    const int64_t t0 = p.prog_tok_off[prog], v0 = p.prog_var_off[prog];
    const int len = (int)(p.prog_tok_off[prog + 1] - t0);
    const int32_t nv = p.prog_nvars[prog];
    const uint8_t* tok = p.tok + t0;
    const int32_t* payload = p.payload + t0;
    uint8_t* step = p.step_mask + t0;
    uint8_t* fin = p.final_mask + v0;
    const uint8_t* init = p.init_mask ? p.init_mask + v0 : nullptr;
    constexpr uint32_t VI = 1u << AMC_ST_VI;
    // words of the ops, the constructs opened before them, chains (first op | its
    // variable << 16), constructs (at most one per two tokens): 8 and at most 8
    // bytes per token of the program's own (the kernel beside this has the others')
    uint32_t* W = reinterpret_cast<uint32_t*>(p.save + 8 * t0);
    uint16_t* opened = reinterpret_cast<uint16_t*>(p.alt + 8 * t0);
    uint32_t* heads = W + len;
    uint64_t* C = reinterpret_cast<uint64_t*>(p.alt + 8 * t0) + (len + 3) / 4;
    for (int v = lane; v < (nv + 1) / 2; v += 32) reinterpret_cast<uint32_t*>(tail)[v] = ~0u;
    // variables without an op keep their set
    for (int v = lane; v < nv; v += 32) fin[v] = init ? init[v] : (uint8_t)VI;
    __syncwarp();

    // ---- 1. structure, chains -------------------------------------------------
    bool bad = false, range = false;
    int D = 0, WD = 0;                                     // open constructs, Whiles among them
    uint32_t carry = 0;                                    // lane d: the announcement in force at depth d
    uint32_t open_top = NIL16;                             // opener of the last outermost construct
    int nh = 0, nc = 0;
    // An announcement: the place of an If's ELSE (AN_ELSE), of a While's END
    // (AN_WHILE) or, by an ELSE, of its If's END.
    constexpr uint32_t AN_ELSE = 1u << 16, AN_WHILE = 1u << 17;
    uint32_t nks[VAHEAD];
    int32_t npl[VAHEAD];
#pragma unroll
    for (int u = 0; u < VAHEAD; ++u) {
        const int q = 32 * u + lane;
        nks[u] = q < len ? tok[q] : 0xFFu;
        npl[u] = q < len ? payload[q] : 0;
    }
    for (int b0 = 0; b0 < len && !bad; b0 += 32 * VAHEAD) {
        uint32_t cks[VAHEAD];
        int32_t cpl[VAHEAD];
#pragma unroll
        for (int u = 0; u < VAHEAD; ++u) {
            cks[u] = nks[u];
            cpl[u] = npl[u];
            const int q = b0 + 32 * (VAHEAD + u) + lane;
            nks[u] = q < len ? tok[q] : 0xFFu;
            npl[u] = q < len ? payload[q] : 0;
        }
#pragma unroll
        for (int u = 0; u < VAHEAD; ++u) {
            const int w0 = b0 + 32 * u;
            if (w0 >= len || bad) break;
            const int q = w0 + lane;
            const bool in = q < len;
            const uint32_t ks = cks[u];
            const int32_t pl = cpl[u];
            const bool op = in && v_is_op(ks);
            // the outermost construct around the token, whether a While is; every
            // structure token against its construct
            int depth = D;                                 // before the token
            uint32_t top = D ? open_top : NIL16;
            bool inw = WD != 0;
            int ids = nc;                                  // constructs opened before the token
            const uint32_t st = __ballot_sync(0xffffffffu, in && !op);
            if (st) {
                const bool opn = in && (ks == AMC_T_IF || ks == AMC_T_WHILE);
                const bool els = in && ks == AMC_T_ELSE, enb = in && ks == AMC_T_END;
                const uint32_t O = __ballot_sync(0xffffffffu, opn), E = __ballot_sync(0xffffffffu, enb);
                const uint32_t WH = __ballot_sync(0xffffffffu, opn && ks == AMC_T_WHILE);
                depth = D + __popc(O & lt) - __popc(E & lt);
                ids += __popc(O & lt);
                // place after the part the token announces (none in the program: NIL16)
                const uint32_t to = pl >= 0 && pl < len - q - 1 ? (uint32_t)(q + 1 + pl) : NIL16;
                const uint32_t says = to | (ks == AMC_T_IF ? AN_ELSE : 0u) | (ks == AMC_T_WHILE ? AN_WHILE : 0u);
                const int level = opn ? depth : els ? depth - 1 : -1;       // of the construct it speaks for
                bool wrong = in && !op && !opn && !els && !enb;
                // more constructs than a balanced program of its length can have, and
                // than its share of C holds (the words behind it are the next program's)
                wrong |= nc + __popc(O) > len / 2;
                wrong |= (opn || els) && (to == NIL16 || level < 0 || level >= AMC_MAX_DEPTH);
                const int most = min(__reduce_max_sync(0xffffffffu, in ? depth + opn : 0), AMC_MAX_DEPTH);
                uint32_t heard = NIL16;                    // in force at the token's own construct
                for (int d = 0; d < most; ++d) {
                    const uint32_t A = __ballot_sync(0xffffffffu, level == d), sa = A & lt;
                    const uint32_t x = __shfl_sync(0xffffffffu, says, 31 - __clz(sa | 1u));
                    const uint32_t c = __shfl_sync(0xffffffffu, carry, d);
                    if (depth == d + 1) heard = sa ? x : c;
                    if (A) {
                        const uint32_t y = __shfl_sync(0xffffffffu, says, 31 - __clz(A));
                        if (lane == d) carry = y;
                    }
                }
                wrong |= els && heard != ((uint32_t)q | AN_ELSE);
                wrong |= enb && (heard & ~AN_WHILE) != (uint32_t)q;
                bad = __any_sync(0xffffffffu, wrong);
                if (bad) break;                            // the same on every lane
                const uint32_t WE = __ballot_sync(0xffffffffu, enb && (heard & AN_WHILE));
                const uint32_t T = __ballot_sync(0xffffffffu, opn && depth == 0);
                inw = WD + __popc(WH & lt) - __popc(WE & lt) != 0;
                top = depth ? ((T & lt) ? (uint32_t)(w0 + 31 - __clz(T & lt)) : open_top) : NIL16;
                if (opn)
                    C[ids] = (uint64_t)(uint32_t)depth << 32 |
                             (ks == AMC_T_WHILE ? NIL16 << 16 | to : to << 16 | NIL16);   // an If's END: step 2
                if (T) open_top = (uint32_t)(w0 + 31 - __clz(T));
                nc += __popc(O);
                D += __popc(O) - __popc(E);
                WD += __popc(WH) - __popc(WE);
            }
            // chains
            const bool valid = op && pl >= 0 && pl < nv;
            range |= op && !valid;
            const uint32_t before = valid ? tail[pl] : NIL16;
            __syncwarp();
            if (valid) tail[pl] = (uint16_t)q;
            __syncwarp();
            uint32_t word = (((ks & 15u) << 1) | ((ks >> 4) & 1u)) << 16 | (inw ? W_WHILE : 0u) |
                            (top != NIL16 ? W_CONS : 0u) | (uint32_t)depth << 23;
            bool lower = false;                            // an earlier op of the window is on the variable
            if (__any_sync(0xffffffffu, valid && tail[pl] != (uint16_t)q)) {
                const uint32_t peers = __match_any_sync(0xffffffffu, valid ? (uint32_t)pl : 0x80000000u | lane);
                const uint32_t up = peers & ~lt & ~(1u << lane);
                const int n = up ? __ffs(up) - 1 : lane;
                const uint32_t ntop = __shfl_sync(0xffffffffu, top, n);
                lower = (peers & lt) != 0;
                if (up) word |= (uint32_t)(w0 + n) | (top != NIL16 && ntop == top ? W_MORE : 0u);
                else if (valid) tail[pl] = (uint16_t)q;
            }
            if (valid) {
                W[q] = word;
                if (top != NIL16) opened[q] = (uint16_t)ids;
            } else if (in) {
                step[q] = 0;
            }
            // the op before it, from an earlier window (its word has no next op yet);
            // it shares the outermost construct if it lies behind the opener
            const bool first = valid && !lower && before == NIL16;
            if (valid && !lower && !first) atomicOr(W + before, (uint32_t)q | (top != NIL16 && before > top ? W_MORE : 0u));
            const uint32_t F = __ballot_sync(0xffffffffu, first);
            if (first) heads[nh + __popc(F & lt)] = (uint32_t)q | (uint32_t)pl << 16;
            nh += __popc(F);
            __syncwarp();
        }
    }
    bad |= D != 0;
    if (range) raise_error(p.err, AMC_E_RANGE);
    __syncwarp();
    if (bad) {
        if (lane == 0) raise_error(p.err, AMC_E_INVALID);
        return;
    }

    // ---- 2. chains ------------------------------------------------------------
    // A frame per open construct that holds an op of the lane's variable; the
    // innermost one in registers, the others below it.
    struct Frame {
        uint32_t end, els;                 // END, ELSE (NIL16: a While)
        uint32_t first, first_w;           // first op of the variable in it
        uint32_t entry, alt;               // set before it (While: at its head); then-result
        bool in_else;
    };
    Frame f = {}, below[AMC_MAX_DEPTH];
    // the constructs in place of the last ops, where they fit
    uint64_t* const own = reinterpret_cast<uint64_t*>(tail);
    const bool fits = nc <= (int)VCONS;
    for (int c = lane; c < nc; c += 32) {
        uint64_t x = C[c];
        if (c_else(x) != NIL16) x = (x & ~(uint64_t)NIL16) | (uint64_t)(c_else(x) + 1 + (uint32_t)payload[c_else(x)]);
        if (fits) own[c] = x;
        else C[c] = x;
    }
    __syncwarp();
    auto construct = [&](uint32_t c) { return fits ? own[c] : C[c]; };
    int depth = 0;                         // frames, the innermost one included
    uint32_t ff = ~0u;
    // the chain after this lane's current one with the word of its first op, and
    // the chain after that, loaded ahead
    int i = lane + 64;
    uint32_t h = lane < nh ? heads[lane] : ~0u, h2 = lane + 32 < nh ? heads[lane + 32] : ~0u;
    uint32_t hw = h != ~0u ? W[h & 0xFFFFu] : 0u;
    bool busy = false;
    uint32_t q = 0, w = 0, m = 0;
    int32_t v = 0;
    auto chains = [&](auto sparse) {
        constexpr bool SPARSE = decltype(sparse)::value;
        for (;;) {
            __syncwarp();
            if (!busy && h != ~0u) {
                busy = true;
                q = h & 0xFFFFu;
                v = (int32_t)(h >> 16);
                w = hw;
                h = h2;
                if (h != ~0u) hw = W[h & 0xFFFFu];
                h2 = i < nh ? heads[i] : ~0u;
                i += 32;
                m = init ? init[v] : VI;
            }
            if (!__any_sync(0xffffffffu, busy)) break;
            if (!busy) continue;
            uint32_t n = w_next(w), o = w_op(w);
            uint32_t nw = n ? W[n] : 0u;
            if (SPARSE && depth == 0 && !(w & W_CONS)) {
                // few constructs: a stretch of ops in none of them
                for (int k = 0; k < 31 && n && !(nw & W_CONS); ++k) {
                    if ((S.flt[o] >> m) & 1u) ff = min(ff, q);
                    m = S.img[o * 32 + m];
                    step[q] = (uint8_t)m;
                    q = n;
                    w = nw;
                    n = w_next(w);
                    o = w_op(w);
                    nw = n ? W[n] : 0u;
                }
            }
            uint32_t q2 = n;
            if (depth == 0 && !(w & W_MORE)) {
                // alone in its outermost construct
                uint32_t x = m;
                if (w & W_WHILE) {
                    // the least set that holds m and its own image
                    for (;;) {
                        const uint32_t y = x | S.img[o * 32 + x];
                        if (y == x) break;
                        x = y;
                    }
                }
                if ((S.flt[o] >> x) & 1u) ff = min(ff, q);
                const uint32_t y = S.img[o * 32 + x];
                step[q] = (uint8_t)y;
                m = (w & W_CONS) ? (x | y) : y;
            } else {
                // open the constructs around q that are not open yet, outermost first
                const int around = (int)w_depth(w);
                while (depth < around) {
                    // the last construct at this depth that opens before q
                    uint32_t c = opened[q];
                    uint64_t cw;
                    do cw = construct(--c);
                    while (c && (int)c_depth(cw) != depth);
                    if (depth) below[depth - 1] = f;
                    ++depth;
                    f.end = c_end(cw);
                    f.els = c_else(cw);
                    f.first = q;
                    f.first_w = w;
                    f.entry = f.alt = m;
                    f.in_else = f.els != NIL16 && q > f.els;
                }
                if ((S.flt[o] >> m) & 1u) ff = min(ff, q);
                m = S.img[o * 32 + m];
                step[q] = (uint8_t)m;
                // the constructs that end before the next op (all, when it is not in
                // the outermost one)
                const uint32_t nx = (w & W_MORE) ? n : NIL16;
                uint32_t at = nx;
                while (depth && at > f.end) {
                    if (f.els != NIL16) {
                        m |= f.in_else ? f.alt : f.entry;
                    } else {
                        m |= f.entry;
                        if (m != f.entry) {                    // grown: its ops again
                            f.entry = m;
                            at = q2 = f.first;
                            nw = f.first_w;
                            break;
                        }
                    }
                    --depth;
                    if (depth) f = below[depth - 1];
                }
                if (depth && f.els != NIL16 && !f.in_else && at > f.els) {
                    f.alt = m;
                    m = f.entry;
                    f.in_else = true;
                }
            }
            if (depth || n) {
                q = q2;
                w = nw;
            } else {
                fin[v] = (uint8_t)m;
                busy = false;
            }
        }
    };
    // With hardly any construct, or with few and one or two chains, most steps are
    // in none.  (64 programs of 40,000 tokens without constructs over 1 / 4 / 64
    // variables: 10.5 / 3.7 / 1.46 ms without the stretches, 4.9 / 2.6 / 1.33 with them; with a
    // 1 in 80 construct, over 64 variables, 3.4 without and 4.1 with them: lanes wait)
    if ((nv <= 2 ? 24 : 256) * nc < len) chains(std::true_type{});
    else chains(std::false_type{});
    ff = __reduce_min_sync(0xffffffffu, ff);
    if (lane == 0) p.prog_first_fault[prog] = ff == ~0u ? -1 : (int64_t)ff;
}

__global__ void __launch_bounds__(VWARPS * 32, VCTAS) vars_kernel(const __grid_constant__ BatchParams p,
                                                             unsigned long long* queue, const int* off)
{
    extern __shared__ __align__(16) uint8_t smem[];
    VarSmem& S = *reinterpret_cast<VarSmem*>(smem);
    for (int i = threadIdx.x; i < 16 * 32; i += blockDim.x) S.img[i] = p.tab.img[i];
    if (threadIdx.x < 16) S.flt[threadIdx.x] = p.tab.flt[threadIdx.x];
    __syncthreads();
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    while (!*off) {
        long long i = 0;
        if (lane == 0) i = (long long)atomicAdd(queue, 1ull);
        i = __shfl_sync(0xffffffffu, i, 0);
        if (i >= p.n_progs) break;
        const int64_t prog = p.order ? p.order[i] : i;
        if (!program_by_vars(p, prog)) continue;
        run_program(p, prog, S, S.tail[w]);
        __syncwarp();
    }
    // this kernel ends no earlier than the one it started beside
    cudaGridDependencySynchronize();
}

}  // namespace

int launch_batch_vars(const BatchParams& p, int64_t max_ctas, unsigned long long* queue, const int* off, cudaStream_t s)
{
    int dev = 0, n_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    int64_t grid = VCTAS * (int64_t)n_sm;
    const int64_t need = (p.n_progs + VWARPS - 1) / VWARPS;
    if (grid > need) grid = need;
    if (max_ctas > 0 && grid > max_ctas) grid = max_ctas;
    // Few CTAs are spread over the SMs: those of the kernel before leave some SMs
    // first, which would take all of these (40 programs of 46,000 tokens beside 40 over
    // 4,097 and more variables: 10.7 ms with 20 CTAs on four SMs, 7.6 so).
    // With more shared memory than it needs no SM takes more than its part, and the
    // rest of it holds the CTAs of that kernel (18 KB each).
    constexpr size_t SM = 228 << 10;
    const size_t part = (size_t)((grid + n_sm - 1) / n_sm), most = SM / 2;
    const size_t smem = part < VCTAS ? SM / (part + 1) / 16 * 16 : sizeof(VarSmem);
    if (!allow_smem<vars_kernel>(most)) return AMC_E_CUDA;
    chain(vars_kernel, (unsigned)grid, VWARPS * 32, smem > sizeof(VarSmem) ? smem : sizeof(VarSmem), s)(p, queue, off);
    return cudaGetLastError() == cudaSuccess ? AMC_OK : AMC_E_CUDA;
}

}  // namespace amc

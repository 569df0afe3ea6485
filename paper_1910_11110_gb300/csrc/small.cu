// small.cu -- the trace check of a small trace in one CTA (Section 3.2, rules
// Effect / Remote Effect of Fig. Opsem; sequencing is associative).
//
// For traces of at most SMALL_MAX_OPS ops over at most SMALL_MAX_VARS
// variables, one launch of one CTA does the whole check: its 32 warps take
// consecutive stretches of the trace; (1) each warp folds its stretch into
// one transfer function per variable (32 ops at a time: the lanes with the same
// variable are found by a ballot per bit of the id, and compose their functions
// in log steps), kept in shared memory; (2) the initial status is carried through
// the warps' functions (a warp per variable, its lanes composing in log steps, for
// few variables, else a thread per variable), giving every stretch its entry
// statuses and the final status; (3) each warp takes its stretch from those
// statuses and writes every op's status and the first faults.  No workspace,
// no memset, one kernel: the latency of a check is one launch.  The initial
// and final statuses may share a buffer: a variable's initial status is read
// and its final status written by the same thread in step (2).
// What bounds it is latency: four batches are loaded at once, and a stretch of at
// most four stays in registers between (1) and (3).  4,096 ops over 16 variables:
// 10.1 us with a load per batch, match.any and a serial chain over equal lanes,
// 6.3 us this way.
#include <cstddef>

#include "amc_internal.cuh"
#include "scan_trace.cuh"

namespace amc {

namespace {

constexpr int SMALL_MAX_OPS = 1 << 16;
constexpr int SMALL_MAX_VARS = 2048;
constexpr int SNW = 32;                      // warps
constexpr int SB = 4;                        // batches of 32 ops loaded at once
// Up to so many variables a warp carries one in five steps of about 60 cycles, a
// warp's share of them one after another; above, 1,024 threads one each in 32.
constexpr int SMALL_SCAN_VARS = 128;

static_assert(SNW == 32, "the carry's lanes are the stretches");

struct SmallSmem {
    uint8_t comp[MAX_ELEMS * MAX_ELEMS];
    uint8_t app[MAX_ELEMS * 8];
    uint8_t elem_of[256];
    uint8_t row[SNW][SMALL_MAX_VARS];        // per warp: folded functions, then current statuses
    unsigned long long ff;
};

__global__ void __launch_bounds__(SNW * 32, 1) small_trace_kernel(const uint8_t* __restrict__ kind_side,
                                                                   const int32_t* __restrict__ var, int32_t n,
                                                                   int32_t n_vars, const uint8_t* init,
                                                                   uint8_t* __restrict__ step,
                                                                   uint8_t* fin, int32_t* __restrict__ vff,
                                                                   int64_t* first_fault, int* err, const Tables tab)
{
    extern __shared__ __align__(16) uint8_t smraw[];
    SmallSmem& S = *reinterpret_cast<SmallSmem*>(smraw);
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const uint32_t lt = lanemask_lt();
    // the tables, a word at a time (lanes reading different parameter words take turns)
    static_assert(offsetof(Tables, app) % 4 == 0 && offsetof(Tables, elem_of) % 4 == 0 && sizeof(Tables) % 4 == 0, "");
    for (int i = tid; i < MAX_ELEMS * MAX_ELEMS / 4; i += SNW * 32)
        reinterpret_cast<uint32_t*>(S.comp)[i] = reinterpret_cast<const uint32_t*>(tab.comp)[i];
    for (int i = tid; i < MAX_ELEMS * 8 / 4; i += SNW * 32)
        reinterpret_cast<uint32_t*>(S.app)[i] = reinterpret_cast<const uint32_t*>(tab.app)[i];
    for (int i = tid; i < 256 / 4; i += SNW * 32)
        reinterpret_cast<uint32_t*>(S.elem_of)[i] = reinterpret_cast<const uint32_t*>(tab.elem_of)[i];
    const uint32_t ID = tab.identity;
    for (int v = lane; v < n_vars; v += 32) S.row[w][v] = (uint8_t)ID;
    if (tid == 0) S.ff = ~0ull;
    const int per = (n + SNW - 1) / SNW;
    const int lo = min(n, w * per), hi = min(n, lo + per);
    const int bits = 32 - __clz(n_vars - 1 | 1);
    // SB batches of 32 ops: byte and id; then the op's function after those of the
    // lanes before it with its variable (inc), and theirs alone (exc)
    uint32_t ks[SB], inc[SB], exc[SB];
    int32_t var_of[SB];
    bool last[SB];                                       // no later lane of the batch has the variable
    auto load = [&](int b) {
#pragma unroll
        for (int u = 0; u < SB; ++u) {
            const int i = b + 32 * u + lane;
            ks[u] = i < hi ? kind_side[i] : 0u;
            var_of[u] = i < hi ? var[i] : 0;
        }
    };
    auto functions = [&](int b, int u, bool check) {
        const bool ok = b + 32 * u + lane < hi;
        int32_t v = var_of[u];
        uint32_t m = ID;
        if (ok) {
            if (v < 0 || v >= n_vars) {
                if (check) raise_error(err, AMC_E_RANGE);
                v = 0;
            }
            m = S.elem_of[ks[u]];
            if (m == ELEM_BAD || m == ELEM_GT) {         // GT only in a guarded check
                if (check) raise_error(err, AMC_E_INVALID);
                m = ID;
            }
        }
        var_of[u] = v;
        uint32_t peers = __ballot_sync(0xffffffffu, ok);
        for (int k = 0; k < bits; ++k) {
            const uint32_t x = __ballot_sync(0xffffffffu, (v >> k) & 1);
            peers &= (v >> k) & 1 ? x : ~x;
        }
        if (!ok) peers = 1u << lane;
        const int before = (peers & lt) ? 31 - __clz(peers & lt) : -1;
        uint32_t f = m;
        for (int q = before; __any_sync(0xffffffffu, q >= 0);) {
            const uint32_t fq = __shfl_sync(0xffffffffu, f, q & 31);
            const int qq = __shfl_sync(0xffffffffu, q, q & 31);
            if (q >= 0) {
                f = S.comp[fq * MAX_ELEMS + f];
                q = qq;
            }
        }
        const uint32_t e = __shfl_sync(0xffffffffu, f, before & 31);
        inc[u] = f;
        exc[u] = before >= 0 ? e : ID;
        last[u] = ok && !(peers & ~lt & ~(1u << lane));
    };
    load(lo);
    __syncthreads();
    // (1) fold each stretch per variable
    for (int b = lo; b < hi; b += 32 * SB) {
        if (b > lo) load(b);
#pragma unroll
        for (int u = 0; u < SB; ++u) {
            if (b + 32 * u >= hi) break;
            functions(b, u, true);
            if (last[u]) S.row[w][var_of[u]] = S.comp[S.row[w][var_of[u]] * MAX_ELEMS + inc[u]];
            __syncwarp();
        }
    }
    __syncthreads();
    // (2) carry: entry status of every stretch, final statuses
    if (n_vars <= SMALL_SCAN_VARS) {
        for (int v = w; v < n_vars; v += SNW) {
            const uint32_t s0 = init ? (uint32_t)(init[v] & 7u) : (uint32_t)AMC_ST_VI;
            uint32_t f = S.row[lane][v];
#pragma unroll
            for (int d = 1; d < SNW; d <<= 1) {
                const uint32_t x = __shfl_up_sync(0xffffffffu, f, d);
                if (lane >= d) f = S.comp[x * MAX_ELEMS + f];
            }
            const uint32_t out = S.app[f * 8 + s0], in = __shfl_up_sync(0xffffffffu, out, 1);
            S.row[lane][v] = (uint8_t)(lane ? in : s0);
            if (lane == SNW - 1) {
                fin[v] = (uint8_t)out;
                vff[v] = -1;
            }
        }
    } else {
        for (int v = tid; v < n_vars; v += SNW * 32) {
            uint32_t s = init ? (uint32_t)(init[v] & 7u) : (uint32_t)AMC_ST_VI;
            for (int k = 0; k < SNW; ++k) {
                const uint32_t e = S.row[k][v];
                S.row[k][v] = (uint8_t)s;
                s = S.app[e * 8 + s];
            }
            fin[v] = (uint8_t)s;
            vff[v] = -1;
        }
    }
    __syncthreads();
    // (3) statuses of every op from the stretch's entry statuses
    for (int b = lo; b < hi; b += 32 * SB) {
        if (hi - lo > 32 * SB) load(b);
#pragma unroll
        for (int u = 0; u < SB; ++u) {
            if (b + 32 * u >= hi) break;
            if (hi - lo > 32 * SB) functions(b, u, false);
            const int i = b + 32 * u + lane;
            const int32_t v = var_of[u];
            const uint32_t cur = i < hi ? S.row[w][v] : 0u;
            const uint32_t pre = S.app[exc[u] * 8 + cur], post = S.app[inc[u] * 8 + cur];
            __syncwarp();
            if (last[u]) S.row[w][v] = (uint8_t)post;
            if (i < hi) {
                step[i] = (uint8_t)post;
                if (post == ST_F && pre != ST_F) {
                    vff[v] = i;                          // a variable becomes stuck once
                    atomicMin(&S.ff, (unsigned long long)i);
                }
            }
            __syncwarp();
        }
    }
    __syncthreads();
    if (tid == 0) *first_fault = S.ff == ~0ull ? -1 : (int64_t)S.ff;
}

}  // namespace

bool scan_small_eligible(const ScanLaunch& L)
{
    return L.dense != 0 && !L.n_dev && !L.gate && !L.guard && !L.pre_mode && L.n_ops <= SMALL_MAX_OPS &&
           L.n_vars >= 1 && L.n_vars <= SMALL_MAX_VARS && L.final_status != nullptr;
}

int launch_scan_small(const ScanLaunch& L, cudaStream_t s)
{
    if (!allow_smem<small_trace_kernel>(sizeof(SmallSmem))) return AMC_E_CUDA;
    if (L.profile & 1) profile_begin(s);
    small_trace_kernel<<<1, SNW * 32, sizeof(SmallSmem), s>>>(L.kind_side, L.var, (int32_t)L.n_ops, L.n_vars, L.init,
                                                              L.step, L.final_status, L.vff, L.first_fault, L.err,
                                                              host_tables());
    if (L.profile & 2) profile_end(s);
    return cudaGetLastError() == cudaSuccess ? AMC_OK : AMC_E_CUDA;
}

}  // namespace amc

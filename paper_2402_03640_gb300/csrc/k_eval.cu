// Exact cost of a batch of assignments by the clause CSR (sm_103a).
//
// A clause is unsatisfied iff none of its literals is true (the paper's
// test x'.W == -len with x' read as +-1, Sec. 4 "Unsatisfiable Cores").
// Kernels:
//
//   k_pack_bits    the batch a[n][nb] (one byte or float an entry, true
//                  where > 0) to one bit an entry, 32 assignments a word
//   k_eval_sparse  a lane owns one clause for VW words of 32 assignments:
//                  per literal one gather of VW words, an exclusive or with
//                  the sign and an or; the unsat words of a warp's 32
//                  clauses are transposed, so that lane b counts the unsat
//                  clauses of assignment b with one popcount (per bit of
//                  the weights where there are weights)
//   k_eval_direct  small calls, one assignment a lane, without the packing
//
// What bounds it: the gathers, one 4 VW-byte read per literal, VW = 4 where
// the batch has more than 64 assignments (a 16-byte row holds 128 of them).
// The form before it gave each lane one assignment and read 32 bytes of a
// per literal and 32 assignments, about 42 instructions for 32 (clause,
// assignment) pairs where this one takes about 150 for 4096.  Weighted Zipf
// n=2e5, m=1e6, 100 assignments: 697 -> 59
// us a call (14 packing, 36 evaluation, the rest launches and the order among
// the users of the scratch).

#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "bits.cuh"
#include "msat_internal.cuh"

namespace msat {

namespace {

constexpr int kEvalWarps = kThreads / 32;
constexpr int kLitBatch = 4;  // literals whose loads and gathers are in flight together
// Clauses of more literals are read by the whole warp.
constexpr int kLongClause = 32;

// What the evaluation reads of an instance (a launch copies its arguments).
struct EvalInst {
    int m, kfix;
    const int32_t *coff, *lit;
    const int64_t *w;
};

__device__ __forceinline__ bool is_true(int8_t v) { return v > 0; }
__device__ __forceinline__ bool is_true(float v) { return v > 0.0f; }

// VW consecutive words of one row.
template <int VW>
__device__ __forceinline__ void ld_words(const uint32_t *__restrict__ p, uint32_t (&o)[VW]) {
    if constexpr (VW == 4) {
        const uint4 v = __ldg(reinterpret_cast<const uint4 *>(p));
        o[0] = v.x;
        o[1] = v.y;
        o[2] = v.z;
        o[3] = v.w;
    } else if constexpr (VW == 2) {
        const uint2 v = __ldg(reinterpret_cast<const uint2 *>(p));
        o[0] = v.x;
        o[1] = v.y;
    } else {
        o[0] = __ldg(p);
    }
}

}  // namespace

// One warp packs rows: RW words of 32 entries of a row an iteration, RPI =
// 4 / RW rows at a time.  row: entries of a row of the source, of which the
// first nb are packed; wpr: words per row of the result, a multiple of RW
// (words past the batch are zero).  V4 (int8 rows and batch of multiples of
// four bytes): a lane reads four entries at a time, their bits meet by
// shuffles of eight lanes; otherwise a lane reads one entry and a ballot
// makes the word.  Clears the costs the evaluation adds to.
// 2e5 rows of 100 bytes: 14 us (51 with one byte a lane and a division per word).
template <typename T, int RW, bool V4>
__global__ void __launch_bounds__(kThreads)
    k_pack_bits(const T *__restrict__ a, int n, int row, int nb, int wpr, uint32_t *__restrict__ bits,
                unsigned long long *__restrict__ cost) {
    constexpr int RPI = 4 / RW;
    const int lane = threadIdx.x & 31;
    if (blockIdx.x == 0)
        for (int b = threadIdx.x; b < nb; b += kThreads) cost[b] = 0ull;
    const long long stride = (long long)gridDim.x * kEvalWarps * RPI;
    for (long long i0 = ((long long)blockIdx.x * kEvalWarps + (threadIdx.x >> 5)) * RPI; i0 < n; i0 += stride) {
        for (int w0 = 0; w0 < wpr; w0 += RW) {
            if constexpr (V4) {
                // RW words are 8 RW lanes of four entries: the rows of the
                // iteration side by side in the warp's lanes
                const int r = lane / (8 * RW), c = w0 * 32 + (lane % (8 * RW)) * 4;
                uint32_t x = 0u;
                if (i0 + r < n && c < nb) x = __ldg(reinterpret_cast<const uint32_t *>(a + (i0 + r) * row + c));
                // bit 7 of each byte where it is > 0, then the four bits together
                const uint32_t pos = ((x & 0x7f7f7f7fu) + 0x7f7f7f7fu) & ~x & 0x80808080u;
                uint32_t word = ((((pos >> 7) * 0x01020408u) >> 24) & 0xfu) << (4 * (lane & 7));
#pragma unroll
                for (int o = 1; o < 8; o <<= 1) word |= __shfl_xor_sync(0xffffffffu, word, o);
                if ((lane & 7) == 0 && i0 + r < n) bits[(i0 + r) * wpr + w0 + (lane % (8 * RW)) / 8] = word;
            } else {
                T v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int c = (w0 + u % RW) * 32 + lane;
                    v[u] = i0 + u / RW < n && c < nb ? __ldg(a + (i0 + u / RW) * row + c) : T(0);
                }
                uint32_t mine = 0u;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const uint32_t word = __ballot_sync(0xffffffffu, is_true(v[u]));
                    if (lane == u) mine = word;
                }
                if (lane < 4 && i0 + lane / RW < n) bits[(i0 + lane / RW) * wpr + w0 + lane % RW] = mine;
            }
        }
    }
}

// ors the values of literals L (-1: none) into sat, all their rows in flight.
template <int VW>
__device__ __forceinline__ void gather_or(const uint32_t *__restrict__ bits, int wpr, int word0,
                                          const int (&L)[kLitBatch], uint32_t (&sat)[VW]) {
    uint32_t row[kLitBatch][VW];
#pragma unroll
    for (int k = 0; k < kLitBatch; ++k)
        if (L[k] >= 0) ld_words<VW>(bits + (long long)(L[k] >> 1) * wpr + word0, row[k]);
#pragma unroll
    for (int k = 0; k < kLitBatch; ++k) {
        if (L[k] < 0) continue;
        const uint32_t neg = (L[k] & 1) ? 0xffffffffu : 0u;
#pragma unroll
        for (int v = 0; v < VW; ++v) sat[v] |= row[k][v] ^ neg;
    }
}

// wbits: bits of the largest clause weight (0: every weight is 1).  cpw:
// clauses a warp takes at a time, in its first lanes.  LONG: there are clauses
// of more than kLongClause literals, which the warp reads together, its lanes'
// ors then joined; a lane a clause, they are the longest chain of a call that
// keeps few warps busy.  300 clauses of 100..300 literals, 100 / 256 assignments
// 53.7 / 60.0 -> 24.3 / 24.4 us a call (42.9 / 44.8 before batches were packed), one
// clause of 15000 literals among 40000 of three, 100 assignments 1757 -> 77 (1344).
template <int VW, bool LONG>
__global__ void __launch_bounds__(kThreads)
    k_eval_sparse(EvalInst I, const uint32_t *__restrict__ bits, int wpr, int nb, int wbits, int cpw,
                  unsigned long long *__restrict__ cost) {
    __shared__ unsigned long long s_acc[kEvalWarps][32 * VW];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int word0 = blockIdx.y * VW;
    unsigned long long acc[VW];
#pragma unroll
    for (int v = 0; v < VW; ++v) acc[v] = 0;
    for (long long j0 = ((long long)blockIdx.x * kEvalWarps + warp) * cpw; j0 < I.m;
         j0 += (long long)gridDim.x * kEvalWarps * cpw) {
        const long long j = j0 + lane;
        const bool live = j < I.m && lane < cpw;
        int beg = 0, end = 0;
        if (live) {
            if (I.kfix > 0) {
                beg = (int)j * I.kfix;
                end = beg + I.kfix;
            } else {
                beg = __ldg(I.coff + j);
                end = __ldg(I.coff + j + 1);
            }
        }
        uint32_t sat[VW];
#pragma unroll
        for (int v = 0; v < VW; ++v) sat[v] = live ? 0u : 0xffffffffu;
        const int len = end - beg;
        const bool joint = LONG && len > kLongClause;
        for (int p0 = 0; p0 < (joint ? 0 : len); p0 += kLitBatch) {
            int L[kLitBatch];
#pragma unroll
            for (int k = 0; k < kLitBatch; ++k) L[k] = p0 + k < len ? __ldg(I.lit + beg + p0 + k) : -1;
            gather_or<VW>(bits, wpr, word0, L, sat);
        }
        __syncwarp();
        if constexpr (LONG) {
            for (unsigned todo = __ballot_sync(0xffffffffu, joint); todo; todo &= todo - 1) {
                const int src = __ffs(todo) - 1;
                const int cb = __shfl_sync(0xffffffffu, beg, src), cl = __shfl_sync(0xffffffffu, len, src);
                uint32_t any[VW];
#pragma unroll
                for (int v = 0; v < VW; ++v) any[v] = 0u;
                for (int p0 = lane; p0 < cl; p0 += 32 * kLitBatch) {
                    int L[kLitBatch];
#pragma unroll
                    for (int k = 0; k < kLitBatch; ++k) L[k] = p0 + 32 * k < cl ? __ldg(I.lit + cb + p0 + 32 * k) : -1;
                    gather_or<VW>(bits, wpr, word0, L, any);
                }
                __syncwarp();
#pragma unroll
                for (int v = 0; v < VW; ++v) {
                    const uint32_t r = __reduce_or_sync(0xffffffffu, any[v]);
                    if (lane == src) sat[v] = r;
                }
            }
        }
        uint32_t un[VW];  // lane b: the unsat bits of the warp's 32 clauses under assignment b
#pragma unroll
        for (int v = 0; v < VW; ++v) un[v] = transpose_bits32(~sat[v], lane);
        if (wbits == 0) {
#pragma unroll
            for (int v = 0; v < VW; ++v) acc[v] += (unsigned)__popc(un[v]);
        } else {
            const unsigned long long w = live ? (unsigned long long)__ldg(I.w + j) : 0ull;
            for (int p = 0; p < min(wbits, 32); ++p) {
                const uint32_t plane = __ballot_sync(0xffffffffu, ((uint32_t)w >> p) & 1u);
#pragma unroll
                for (int v = 0; v < VW; ++v) acc[v] += (unsigned long long)__popc(un[v] & plane) * (1u << p);
            }
            for (int p = 32; p < wbits; ++p) {
                const uint32_t plane = __ballot_sync(0xffffffffu, (w >> p) & 1ull);
#pragma unroll
                for (int v = 0; v < VW; ++v) acc[v] += (unsigned long long)__popc(un[v] & plane) << p;
            }
        }
    }
#pragma unroll
    for (int v = 0; v < VW; ++v) s_acc[warp][32 * v + lane] = acc[v];
    __syncthreads();
    for (int b = threadIdx.x; b < 32 * VW; b += kThreads) {
        unsigned long long s = 0;
#pragma unroll
        for (int k = 0; k < kEvalWarps; ++k) s += s_acc[k][b];
        const int at = word0 * 32 + b;
        if (at < nb && s) atomicAdd(cost + at, s);
    }
}

// Small batches of small instances, and calls that may not have scratch, in
// one launch: a lane is one assignment and a warp walks clauses, reading 32
// entries of a variable's row per literal.  PART: the first nb entries of rows
// of `row`; whole batches have a form of their own, which is faster (300
// clauses of 100..300 literals, 32 assignments 43 us, 52 with the row apart).
template <typename T, bool PART>
__global__ void __launch_bounds__(kThreads)
    k_eval_direct(EvalInst I, const T *__restrict__ a, int row, int nb, unsigned long long *__restrict__ cost) {
    __shared__ unsigned long long s_acc[kEvalWarps][32];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int b = blockIdx.y * 32 + lane;
    const bool live = b < nb;
    const int stride = PART ? row : nb;
    unsigned long long acc = 0;
    for (long long j = (long long)blockIdx.x * kEvalWarps + warp; j < I.m; j += (long long)gridDim.x * kEvalWarps) {
        const int beg = I.kfix > 0 ? (int)j * I.kfix : __ldg(I.coff + j);
        const int end = I.kfix > 0 ? beg + I.kfix : __ldg(I.coff + j + 1);
        bool sat = false;
        for (int p = beg; p < end; ++p) {
            const int L = __ldg(I.lit + p);
            const T v = live ? __ldg(a + (long long)(L >> 1) * stride + b) : T(0);
            sat |= is_true(v) != (bool)(L & 1);
        }
        if (!sat) acc += I.w ? (unsigned long long)__ldg(I.w + j) : 1ull;
    }
    s_acc[warp][lane] = acc;
    __syncthreads();
    if (warp == 0) {
        unsigned long long s = 0;
#pragma unroll
        for (int k = 0; k < kEvalWarps; ++k) s += s_acc[k][lane];
        if (live && s) atomicAdd(cost + b, s);
    }
}

// Up to this many literals read by a warp (each for 32 assignments, or for
// fewer at the same cost) the direct kernel: below it a call is bound by its
// launches on the host, where a clear and one kernel (5.2 us) beat two kernels
// (8.2 us).  Whole calls, directly / packed: 80000 reads (weighted Zipf
// n=2000, 33 assignments) 10.2 / 11.1 us, 129000 (3-SAT m=21500, 64) 12.3 /
// 11.7, 213000 (5-SAT n=2000, 1) 12.4 / 10.7, 400000 (weighted Zipf n=20000,
// 1) 23.0 / 10.9.
constexpr long long kDirectReads = 96 << 10;

// Long clauses are read by a whole warp only when packed (300 clauses of 100..300
// literals, 1 assignment: 35 / 23).
bool eval_is_direct(int64_t nnz, int max_len, int nb) {
    return max_len <= kLongClause && nnz * ((nb + 31) / 32) <= kDirectReads;
}

// Words a lane carries: rows of up to 128 assignments are one load.
static int eval_vw(int nb) { return nb > 64 ? 4 : nb > 32 ? 2 : 1; }

static int eval_wpr(int nb) {
    const int vw = eval_vw(nb);
    return ((nb + 31) / 32 + vw - 1) / vw * vw;
}

// Scratch of one pass over nb assignments.
size_t eval_sparse_bytes(int n, int nb) { return sizeof(uint32_t) * (size_t)n * (size_t)eval_wpr(nb); }

template <int VW>
static void launch_eval_vw(const DevInst &I, const int8_t *a, const float *x, int row, int nb, int wbits,
                           int max_len, uint32_t *bits, unsigned long long *cost, cudaStream_t st) {
    const int wpr = eval_wpr(nb);
    const long long rows4 = ((long long)I.n * VW + 3) / 4;  // warp iterations of the packing
    const unsigned pb = (unsigned)std::min<long long>((rows4 + kEvalWarps - 1) / kEvalWarps, 152LL * 8);
    // four-byte reads: every row of the batch starts on four bytes
    const bool v4 = a && row % 4 == 0 && nb % 4 == 0 && reinterpret_cast<uintptr_t>(a) % 4 == 0;
    if (v4) k_pack_bits<int8_t, VW, true><<<pb, kThreads, 0, st>>>(a, I.n, row, nb, wpr, bits, cost);
    else if (a) k_pack_bits<int8_t, VW, false><<<pb, kThreads, 0, st>>>(a, I.n, row, nb, wpr, bits, cost);
    else k_pack_bits<float, VW, false><<<pb, kThreads, 0, st>>>(x, I.n, row, nb, wpr, bits, cost);
    const int gy = wpr / VW;
    // about eight blocks per SM in all, or fewer when the clauses do not fill
    // them; long clauses are spread over all warps
    const long long blocks = (152LL * 8 + gy - 1) / gy;
    const bool lng = max_len > kLongClause;
    const int cpw = lng ? (int)std::min<long long>(32, (I.m + blocks * kEvalWarps - 1) / (blocks * kEvalWarps)) : 32;
    const long long need = ((long long)I.m + kEvalWarps * cpw - 1) / (kEvalWarps * cpw);
    const long long gx = std::max<long long>(1, std::min<long long>(need, blocks));
    const dim3 grid((unsigned)gx, (unsigned)gy);
    const EvalInst E{I.m, I.kfix, I.coff, I.lit, I.w};
    if (lng) k_eval_sparse<VW, true><<<grid, kThreads, 0, st>>>(E, bits, wpr, nb, wbits, cpw, cost);
    else k_eval_sparse<VW, false><<<grid, kThreads, 0, st>>>(E, bits, wpr, nb, wbits, cpw, cost);
}

// The batch is a (int8 [n][nb]) or, where a is nullptr, x (float [n][nb],
// rounded by x > 0), taken at most `chunk` assignments at a time; bits:
// eval_sparse_bytes(n, min(nb, chunk)) of scratch, or nullptr for the direct
// kernel.
cudaError_t launch_eval_sparse(const DevInst &I, const int8_t *a, const float *x, int nb, int chunk, int wbits,
                               int max_len, uint32_t *bits, long long *cost_out, cudaStream_t st) {
    cudaError_t e = cudaSuccess;
    if (I.m == 0 || !bits) {
        e = cudaMemsetAsync(cost_out, 0, sizeof(long long) * (size_t)nb, st);
        if (e != cudaSuccess || I.m == 0) return e;
        const long long need = ((long long)I.m + kEvalWarps - 1) / kEvalWarps;
        const EvalInst E{I.m, I.kfix, I.coff, I.lit, I.w};
        unsigned long long *cost = reinterpret_cast<unsigned long long *>(cost_out);
        constexpr long long kGridY = 65535;  // a launch's limit, in words of 32 assignments
        for (long long b0 = 0; b0 < nb && e == cudaSuccess; b0 += 32 * kGridY) {
            const int k = (int)std::min<long long>(32 * kGridY, nb - b0);
            const int gy = (k + 31) / 32;
            const dim3 grid((unsigned)std::max<long long>(1, std::min<long long>(need, (152LL * 8 + gy - 1) / gy)),
                            (unsigned)gy);
            if (k == nb) {
                if (a) k_eval_direct<int8_t, false><<<grid, kThreads, 0, st>>>(E, a, nb, k, cost);
                else k_eval_direct<float, false><<<grid, kThreads, 0, st>>>(E, x, nb, k, cost);
            } else {
                if (a) k_eval_direct<int8_t, true><<<grid, kThreads, 0, st>>>(E, a + b0, nb, k, cost + b0);
                else k_eval_direct<float, true><<<grid, kThreads, 0, st>>>(E, x + b0, nb, k, cost + b0);
            }
            e = cudaGetLastError();
        }
        return e;
    }
    for (long long b0 = 0; b0 < nb && e == cudaSuccess; b0 += chunk) {  // past 2^31 behind the last part
        const int k = (int)std::min<long long>(chunk, nb - b0);
        const int8_t *ak = a ? a + b0 : nullptr;
        const float *xk = a ? nullptr : x + b0;
        unsigned long long *cost = reinterpret_cast<unsigned long long *>(cost_out) + b0;
        switch (eval_vw(k)) {
            case 4: launch_eval_vw<4>(I, ak, xk, nb, k, wbits, max_len, bits, cost, st); break;
            case 2: launch_eval_vw<2>(I, ak, xk, nb, k, wbits, max_len, bits, cost, st); break;
            default: launch_eval_vw<1>(I, ak, xk, nb, k, wbits, max_len, bits, cost, st); break;
        }
        e = cudaGetLastError();
    }
    return e;
}

// The paper's quick reading of a clause as satisfied when f_j > 0 (Sec. 4,
// "Example") against the exact test (some literal true under x > 0).  One
// thread per (clause, restart): f_j in the fixed order of the step (terms in
// literal order, 32-term leaves, dyadic combination) from t = tanh(x);
// counts per restart the clauses read as unsat by the heuristic and those on
// which the two tests disagree.  Integer counts, so the order of the
// additions does not matter.
__global__ void k_heuristic_gap(DevInst I, const float *__restrict__ x,
                                unsigned long long *__restrict__ heur_unsat,
                                unsigned long long *__restrict__ disagree) {
    const int B = I.B;
    const long long total = (long long)I.m * B;
    for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < total;
         q += (long long)gridDim.x * blockDim.x) {
        const int j = (int)(q / B), b = (int)(q - (long long)j * B);
        int beg, end;
        if (I.kfix > 0) {
            beg = j * I.kfix;
            end = beg + I.kfix;
        } else {
            beg = __ldg(I.coff + j);
            end = __ldg(I.coff + j + 1);
        }
        LeafCounter<kClauseLevels> lc;
        lc.init();
        float leaf = 0.0f;
        int in_leaf = 0;
        bool sat = false;
        for (int p = beg; p < end; ++p) {
            const int L = __ldg(I.lit + p);
            const float xv = __ldg(x + (long long)(L >> 1) * B + b);
            const float tv = tanh_fixed(xv);
            const bool neg = L & 1;
            const float term = neg ? -tv : tv;
            leaf = in_leaf == 0 ? term : leaf + term;
            sat |= (xv > 0.0f) != neg;
            if (++in_leaf == 32) {
                lc.push(leaf);
                in_leaf = 0;
            }
        }
        if (in_leaf) lc.push(leaf);
        const float f = lc.finish();
        if (!(f > 0.0f)) atomicAdd(heur_unsat + b, 1ull);
        if ((f > 0.0f) != sat) atomicAdd(disagree + b, 1ull);
    }
}

cudaError_t launch_heuristic_gap(const DevInst &I, const float *x, long long *heur_unsat,
                                 long long *disagree, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(heur_unsat, 0, sizeof(long long) * (size_t)I.B, st);
    if (!e) e = cudaMemsetAsync(disagree, 0, sizeof(long long) * (size_t)I.B, st);
    if (e) return e;
    const long long total = (long long)I.m * I.B;
    long long blocks = (total + kThreads - 1) / kThreads;
    if (blocks > 152 * 16) blocks = 152 * 16;
    if (blocks < 1) blocks = 1;
    k_heuristic_gap<<<(unsigned)blocks, kThreads, 0, st>>>(I, x, reinterpret_cast<unsigned long long *>(heur_unsat),
                                                           reinterpret_cast<unsigned long long *>(disagree));
    return cudaGetLastError();
}

}  // namespace msat

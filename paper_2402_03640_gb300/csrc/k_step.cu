// Step kernels of the MaxSAT gradient engine (sm_103a).
//
//   k_init            random start of x (Algorithm 1 initialisation), zero Adam moments,
//                     tanh(x)
//   k_forward         clause pass: f_j, exact unsat bits, sum_U w and the
//                     loss partials per restart; the last block to finish
//                     turns them into cost, best, 2/W_U and the Adam scalars
//   k_backward_light  variable pass over the transposed CSR for variables
//                     with few occurrences: a thread sums the terms of one
//                     32-occurrence leaf straight from their gathers, then
//                     1 - t^2, fused Adam update, best-assignment capture and
//                     tanh; the leaves of a longer variable meet in shared
//                     memory
//   k_backward_heavy  the same for variables with many occurrences, split
//                     into 1024-occurrence chunks, a warp each, combined in
//                     the fixed order
//
// Layouts: x, mom, vel, t are float [n][B] (restart index innermost), so the
// B values of one variable are one contiguous, vector-loadable row.  A
// thread owns VW consecutive restarts of one clause, occurrence or variable:
// up to 8 in the clause pass, 4 of a leaf in the variable pass (up to 16 where
// the caller's launch shape says so), up to 4 in the update (where every
// restart carries x, m, v, t and the sums).

#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "msat_internal.cuh"
#include "pdl.cuh"
#include "step_math.cuh"

namespace msat {

namespace {

__device__ __forceinline__ uint64_t splitmix64_at(uint64_t seed, uint64_t c) {
    uint64_t z = seed + (c + 1ull) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// --------------------------------------------------------- vector access
// VW floats at p (16-byte aligned for VW >= 4): plain and streaming
// (evict-first) loads and stores.  Streaming is used for data touched once
// per pass, so the gathered rows of t, the unsat bits and the f store keep
// their L2 lines.  Everything loaded here is written by the kernel before in
// the stream, which may still run when this one starts (pdl.cuh): the loads
// are volatile so that none moves above the wait, and not read-only-cache
// loads, which a write during the kernel's life would break.

__device__ __forceinline__ float4 ld4(const float4 *p) {
    float4 v;
    asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ float4 ld4_stream(const float4 *p) {
    float4 v;
    asm volatile("ld.global.cs.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ float2 ld2(const float2 *p) {
    float2 v;
    asm volatile("ld.global.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ float2 ld2_stream(const float2 *p) {
    float2 v;
    asm volatile("ld.global.cs.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ float ld1(const float *p) {
    float v;
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ float ld1_stream(const float *p) {
    float v;
    asm volatile("ld.global.cs.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ uint32_t ld1(const uint32_t *p) {
    uint32_t v;
    asm volatile("ld.global.u32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}

template <int VW>
__device__ __forceinline__ void ldv(const float *p, float (&o)[VW]) {
    if constexpr (VW >= 4) {
#pragma unroll
        for (int k = 0; k < VW / 4; ++k) {
            const float4 v = ld4(reinterpret_cast<const float4 *>(p) + k);
            o[4 * k] = v.x; o[4 * k + 1] = v.y; o[4 * k + 2] = v.z; o[4 * k + 3] = v.w;
        }
    } else if constexpr (VW == 2) {
        const float2 v = ld2(reinterpret_cast<const float2 *>(p));
        o[0] = v.x; o[1] = v.y;
    } else {
        o[0] = ld1(p);
    }
}

template <int VW>
__device__ __forceinline__ void ldv_stream(const float *p, float (&o)[VW]) {
    if constexpr (VW >= 4) {
#pragma unroll
        for (int k = 0; k < VW / 4; ++k) {
            const float4 v = ld4_stream(reinterpret_cast<const float4 *>(p) + k);
            o[4 * k] = v.x; o[4 * k + 1] = v.y; o[4 * k + 2] = v.z; o[4 * k + 3] = v.w;
        }
    } else if constexpr (VW == 2) {
        const float2 v = ld2_stream(reinterpret_cast<const float2 *>(p));
        o[0] = v.x; o[1] = v.y;
    } else {
        o[0] = ld1_stream(p);
    }
}

template <int VW>
__device__ __forceinline__ void stv(float *p, const float (&o)[VW]) {
    if constexpr (VW >= 4) {
#pragma unroll
        for (int k = 0; k < VW / 4; ++k)
            reinterpret_cast<float4 *>(p)[k] = make_float4(o[4 * k], o[4 * k + 1], o[4 * k + 2], o[4 * k + 3]);
    } else if constexpr (VW == 2) {
        *reinterpret_cast<float2 *>(p) = make_float2(o[0], o[1]);
    } else {
        *p = o[0];
    }
}

template <int VW>
__device__ __forceinline__ void stv_stream(float *p, const float (&o)[VW]) {
    if constexpr (VW >= 4) {
#pragma unroll
        for (int k = 0; k < VW / 4; ++k)
            __stcs(reinterpret_cast<float4 *>(p) + k, make_float4(o[4 * k], o[4 * k + 1], o[4 * k + 2], o[4 * k + 3]));
    } else if constexpr (VW == 2) {
        __stcs(reinterpret_cast<float2 *>(p), make_float2(o[0], o[1]));
    } else {
        __stcs(p, o[0]);
    }
}

// ------------------------------------------------------------ clause sums

__device__ __forceinline__ void clause_range(const DevInst &I, int kfix, int j, int &beg, int &end) {
    if (kfix > 0) {
        beg = j * kfix;
        end = beg + kfix;
    } else {
        beg = __ldg(I.coff + j);
        end = __ldg(I.coff + j + 1);
    }
}

// Dyadic counter of finished 32-literal leaves for clauses longer than 32
// literals (the same binary counter as LeafCounter), on a per-thread array
// indexed at run time: it lives in local memory and is touched once per 32
// literals, so short clauses never use it.
template <int VW>
__device__ __forceinline__ void leaf_push(float (&stk)[kClauseLevels][VW], unsigned &cnt, float (&v)[VW]) {
    unsigned c = cnt;
    int lvl = 0;
    while (c & 1u) {
#pragma unroll
        for (int e = 0; e < VW; ++e) v[e] = stk[lvl][e] + v[e];
        c >>= 1;
        ++lvl;
    }
#pragma unroll
    for (int e = 0; e < VW; ++e) stk[lvl][e] = v[e];
    ++cnt;
}

template <int VW>
__device__ __forceinline__ void leaf_finish(const float (&stk)[kClauseLevels][VW], unsigned cnt, float (&r)[VW]) {
    bool have = false;
    for (int lvl = 0; lvl < kClauseLevels; ++lvl) {
        if (!((cnt >> lvl) & 1u)) continue;
#pragma unroll
        for (int e = 0; e < VW; ++e) r[e] = have ? (stk[lvl][e] + r[e]) : stk[lvl][e];
        have = true;
    }
}

// f_j for VW restarts in the fixed order (literal order, 32-literal leaves,
// dyadic combination) and, if WANT_SAT, whether some literal is true.
template <int VW, bool WANT_SAT>
__device__ __forceinline__ void clause_value(const DevInst &I, const float *__restrict__ t,
                                             int beg, int end, int col, float (&f)[VW],
                                             bool (&sat)[VW]) {
    const int B = I.B;
#pragma unroll
    for (int e = 0; e < VW; ++e) {
        f[e] = 0.0f;
        sat[e] = false;
    }
    float stk[kClauseLevels][VW];
    unsigned nleaf = 0;
    int in_leaf = 0;
    if constexpr (WANT_SAT && VW <= 4) {
        // the clause pass with up to four restarts a thread: NB literals at
        // a time -- their loads, then their row gathers, then the terms in
        // literal order (the same additions as one literal at a time)
        constexpr int NB = VW == 1 ? 8 : 4;
        for (int p0 = beg; p0 < end; p0 += NB) {
            int L[NB];
            float tv[NB][VW];
#pragma unroll
            for (int k = 0; k < NB; ++k) L[k] = p0 + k < end ? __ldg(I.lit + p0 + k) : 0;
#pragma unroll
            for (int k = 0; k < NB; ++k)
                if (p0 + k < end) ldv<VW>(t + (int64_t)(L[k] >> 1) * B + col, tv[k]);
#pragma unroll
            for (int k = 0; k < NB; ++k) {
                if (p0 + k >= end) break;
                if (in_leaf == 32) {
                    leaf_push<VW>(stk, nleaf, f);
                    in_leaf = 0;
                }
                const bool neg = L[k] & 1;
#pragma unroll
                for (int e = 0; e < VW; ++e) {
                    const float term = neg ? -tv[k][e] : tv[k][e];
                    f[e] = (in_leaf == 0) ? term : f[e] + term;
                    sat[e] |= ((tv[k][e] > 0.0f) != neg);
                }
                ++in_leaf;
            }
        }
    } else {
#pragma unroll 2
        for (int p = beg; p < end; ++p) {
            if (in_leaf == 32) {
                leaf_push<VW>(stk, nleaf, f);
                in_leaf = 0;
            }
            const int L = __ldg(I.lit + p);
            const bool neg = L & 1;
            float tv[VW];
            ldv<VW>(t + (int64_t)(L >> 1) * B + col, tv);
#pragma unroll
            for (int e = 0; e < VW; ++e) {
                const float term = neg ? -tv[e] : tv[e];
                f[e] = (in_leaf == 0) ? term : f[e] + term;
                if (WANT_SAT) sat[e] |= ((tv[e] > 0.0f) != neg);
            }
            ++in_leaf;
        }
    }
    if (nleaf) {  // more than 32 literals: the last leaf, then the counter
        leaf_push<VW>(stk, nleaf, f);
        leaf_finish<VW>(stk, nleaf, f);
    }
}

// Fixed-length clause (KFIX literals): all literal loads first, then all
// row gathers, so the loads of one clause are in flight together.
template <int VW, int KFIX>
__device__ __forceinline__ void clause_value_fixed(const DevInst &I, const float *__restrict__ t,
                                                   int j, int col, float (&f)[VW],
                                                   bool (&sat)[VW]) {
    const int B = I.B;
    int L[KFIX];
#pragma unroll
    for (int p = 0; p < KFIX; ++p) L[p] = __ldg(I.lit + j * KFIX + p);
    float tv[KFIX][VW];
#pragma unroll
    for (int p = 0; p < KFIX; ++p) ldv<VW>(t + (int64_t)(L[p] >> 1) * B + col, tv[p]);
#pragma unroll
    for (int e = 0; e < VW; ++e) {
        sat[e] = false;
#pragma unroll
        for (int p = 0; p < KFIX; ++p) {
            const bool neg = L[p] & 1;
            const float term = neg ? -tv[p][e] : tv[p][e];
            f[e] = (p == 0) ? term : f[e] + term;
            sat[e] |= ((tv[p][e] > 0.0f) != neg);
        }
    }
}

// ------------------------------------------------------- occurrence terms

// Unsat bits of (clause of occurrence word o, restarts col .. col+VW-1)
// from the 32-bit word wd that holds them (flat bit index j*B + col, which
// fits 32 bits: the context rejects m*B >= 2^31).
template <int VW>
__device__ __forceinline__ uint32_t occ_nib(const DevInst &I, int o, uint32_t wd, int col) {
    const uint32_t qb = (uint32_t)(o >> I.occ_shift) * (uint32_t)I.B + (uint32_t)col;
    constexpr uint32_t mask = VW >= 32 ? 0xffffffffu : ((1u << VW) - 1u);
    return (wd >> (qb & 31u)) & mask;
}

__device__ __forceinline__ const uint32_t *ubits_word(const DevInst &I, const uint32_t *ubits,
                                                      int o, int col) {
    return ubits + (((uint32_t)(o >> I.occ_shift) * (uint32_t)I.B + (uint32_t)col) >> 5);
}

// f_j for VW restarts (col .. col+VW-1) of the clause of occurrence word o
// (clause j in the bits above occ_shift, literal sign in bit 0), recomputed
// in the literal order; for 3-literal clauses from the expanded occurrence
// record (position of the variable in bits 1-2 of o, the other two
// literals in ox; own_var is the occurring variable).
template <int VW, int KFIX>
__device__ __forceinline__ void fetch_f(const DevInst &I, int kfix, const float *__restrict__ t,
                                        int o, int2 ox, int own_var, int col, float (&f)[VW]) {
    const int B = I.B;
    const int j = o >> I.occ_shift;
    bool sat[VW];
    if constexpr (KFIX == 3) {
        if (I.occx) {
            const int pos = (o >> 1) & 3;
            const int own = (own_var << 1) | (o & 1);
            int L[3];
            L[0] = pos == 0 ? own : ox.x;
            L[1] = pos == 0 ? ox.x : (pos == 1 ? own : ox.y);
            L[2] = pos == 2 ? own : ox.y;
            float tv[3][VW];
#pragma unroll
            for (int p = 0; p < 3; ++p) ldv<VW>(t + (int64_t)(L[p] >> 1) * B + col, tv[p]);
#pragma unroll
            for (int e = 0; e < VW; ++e) {
#pragma unroll
                for (int p = 0; p < 3; ++p) {
                    const float tt = (L[p] & 1) ? -tv[p][e] : tv[p][e];
                    f[e] = (p == 0) ? tt : f[e] + tt;
                }
            }
        } else {
            clause_value_fixed<VW, 3>(I, t, j, col, f, sat);
        }
    } else if constexpr (KFIX > 0) {
        clause_value_fixed<VW, KFIX>(I, t, j, col, f, sat);
    } else {
        int beg, end;
        clause_range(I, kfix, j, beg, end);
        clause_value<VW, false>(I, t, beg, end, col, f, sat);
    }
}

// Occurrence term for VW restarts: +-((float)w_j * f_j) * (2/W_U) where
// clause j is unsat (bit set in nib), +0 elsewhere.
template <int VW>
__device__ __forceinline__ void term_from_f(const DevInst &I, int o, uint32_t nib,
                                            const float (&f)[VW], const float (&cs)[VW],
                                            float (&term)[VW]) {
    const int j = o >> I.occ_shift;
    const bool neg = o & 1;
    const float wj = I.w ? (float)__ldg(I.w + j) : 1.0f;
#pragma unroll
    for (int e = 0; e < VW; ++e) {
        term[e] = 0.0f;
        if ((nib >> e) & 1u) {
            const float g = (wj * f[e]) * cs[e];
            term[e] = neg ? -g : g;
        }
    }
}

// Adds the terms of C consecutive occurrences (words o, expanded records ox,
// valid where ok) of variable own_var for VW restarts at col to the sum of
// their leaf, in order, all their loads in flight together (first: they open
// the leaf, so recomputed terms start the sum instead of being added to +0).
// With the clause pass's store, q = (float)w_j * f_j (+0 where satisfied)
// gives the term +-(q * 2/W_U); otherwise the unsat bits select the
// restarts whose f is recomputed (fetched together with the bits when unsat
// clauses are dense).
// The store path is bound by its gathers (n=1e6, B=16: 1.4 GB read at 5.2
// TB/s) with the issue slots half taken, so it is held to few instructions:
// the sign is an exact factor of +-1 of the addition, or at one restart a
// thread goes into the scale; satisfied occurrences add +-0 (a marker's test
// and select are gone), which can only change the sign of a zero sum, brought
// to +0 where it is used; missing occurrences read the store's zero row
// instead of being predicated (at one restart a thread the predicate is
// cheaper).  Us a step, marker and selects / without / packed pairs and the
// zero row: weighted Zipf n=2e5, B=1 61.5 / 59.0 / -, B=8 190 / 186 / 182,
// n=1e6, B=16 462 / 459 / 444, 5-SAT n=30011, B=64 281 / 274 / 261, 3-SAT
// n=5000, B=256 36.0 / 35.5 / 33.9.  PACKED: two restarts a product and a
// sum, in the light pass (a chunk's warp measured slower with it: Zipf
// n=20000, B=16 49.3 against 46.5).
template <int VW, int KFIX, int C, bool STORE, bool PACKED>
__device__ __forceinline__ void occ_accumulate(const DevInst &I, const DevState &S, int kfix,
                                               const float *__restrict__ tcur, const int (&o)[C],
                                               const int2 (&ox)[C], const bool (&ok)[C],
                                               int own_var, int col, const float (&cs)[VW],
                                               bool dense, bool first, float (&leaf)[VW]) {
    const int B = I.B;
    float v[C][VW];
    if constexpr (STORE) {
#pragma unroll
        for (int u = 0; u < C; ++u) {
            if (VW > 1 || ok[u]) ldv<VW>(S.fstore + (int64_t)(o[u] >> I.occ_shift) * B + col, v[u]);
            else v[u][0] = 0.0f;
        }
#pragma unroll
        for (int u = 0; u < C; ++u) {
            if constexpr (PACKED) {
                const float sg = (o[u] & 1) ? -1.0f : 1.0f;
#pragma unroll
                for (int e = 0; e < VW; e += 2) {
                    const float2 l = fma2(mul2(make_float2(v[u][e], v[u][e + 1]), make_float2(cs[e], cs[e + 1])),
                                          make_float2(sg, sg), make_float2(leaf[e], leaf[e + 1]));
                    leaf[e] = l.x;
                    leaf[e + 1] = l.y;
                }
            } else if constexpr (VW == 1) {
                const uint32_t sgn = (uint32_t)o[u] << 31;
                leaf[0] = leaf[0] + v[u][0] * __uint_as_float(__float_as_uint(cs[0]) ^ sgn);
            } else {
                const float sg = (o[u] & 1) ? -1.0f : 1.0f;
#pragma unroll
                for (int e = 0; e < VW; ++e) leaf[e] = fmaf(v[u][e] * cs[e], sg, leaf[e]);
            }
        }
    } else {
        uint32_t wd[C];
#pragma unroll
        for (int u = 0; u < C; ++u) {
            wd[u] = ok[u] ? ld1(ubits_word(I, S.ubits, o[u], col)) : 0u;
            if (dense && ok[u]) fetch_f<VW, KFIX>(I, kfix, tcur, o[u], ox[u], own_var, col, v[u]);
        }
#pragma unroll
        for (int u = 0; u < C; ++u) {
            if (!ok[u]) continue;
            const uint32_t nib = occ_nib<VW>(I, o[u], wd[u], col);
            float term[VW];
#pragma unroll
            for (int e = 0; e < VW; ++e) term[e] = 0.0f;
            if (nib) {
                if (!dense) fetch_f<VW, KFIX>(I, kfix, tcur, o[u], ox[u], own_var, col, v[u]);
                term_from_f<VW>(I, o[u], nib, v[u], cs, term);
            }
#pragma unroll
            for (int e = 0; e < VW; ++e) leaf[e] = (first && u == 0) ? term[e] : leaf[e] + term[e];
        }
    }
}

// --------------------------------------------------------------- update

// x, moments and t of one (variable, restart group).
template <int VW>
struct VarState {
    float x[VW], m[VW], v[VW], t[VW];
    __device__ __forceinline__ void load(const DevState &S, const float *__restrict__ tcur, int64_t q0) {
        ldv_stream<VW>(S.x + q0, x);
        ldv_stream<VW>(S.mom + q0, m);
        ldv_stream<VW>(S.vel + q0, v);
        ldv<VW>(tcur + q0, t);
    }
};

// Update of one (variable, restart group) from its occurrence sum S: the
// gradient S * (1 - t^2) with t = tanh(x) of the evaluated x, then Adam
// (unless the restart has stopped), the best-assignment capture and tanh of
// the new x; or, in the gradient-only mode, the scaled gradient.  pre: the
// state loaded earlier, or nullptr.
template <int VW>
__device__ __forceinline__ void finish_variable(const DevState &S, const DevStep &D,
                                                const AdamView &A, int mode, int64_t q0,
                                                int col, const float *__restrict__ tcur,
                                                const float (&Ssum)[VW], float *tnext,
                                                const float *__restrict__ gscale,
                                                float *__restrict__ grad_out,
                                                const VarState<VW> *pre = nullptr) {
    if constexpr (VW > 4) {  // slices of four restarts keep the live registers down
#pragma unroll
        for (int h = 0; h < VW; h += 4) {
            float part[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) part[e] = Ssum[h + e];
            finish_variable<4>(S, D, A, mode, q0 + h, col + h, tcur, part, tnext, gscale, grad_out);
        }
        return;
    }
    if (mode == BWD_GRAD_ONLY) {
        float tv[VW], gr[VW];
        ldv<VW>(tcur + q0, tv);
#pragma unroll
        for (int e = 0; e < VW; ++e) {
            gr[e] = (Ssum[e] + 0.0f) * fmaf(-tv[e], tv[e], 1.0f);
            gr[e] = gscale ? gr[e] * ld_ordered(gscale + col + e) : gr[e];
        }
        stv<VW>(grad_out + q0, gr);
        return;
    }
    VarState<VW> w;
    if (pre) w = *pre;
    else w.load(S, tcur, q0);
    float tn[VW];
#pragma unroll
    for (int e = 0; e < VW; ++e) {
        const float gr = (Ssum[e] + 0.0f) * fmaf(-w.t[e], w.t[e], 1.0f);
        if (D.improved[col + e]) S.bestx[q0 + e] = w.x[e] > 0.0f;
        if (D.cost[col + e] != 0) {
            w.x[e] = adam_update(A, w.x[e], w.m[e], w.v[e], gr);
            tn[e] = tanh_fixed(w.x[e]);
        } else {
            tn[e] = w.t[e];
        }
    }
    stv_stream<VW>(S.x + q0, w.x);
    stv_stream<VW>(S.mom + q0, w.m);
    stv_stream<VW>(S.vel + q0, w.v);
    stv<VW>(tnext + q0, tn);
}

__device__ __forceinline__ void step_buffers(const DevState &S, const DevStep &D, int mode,
                                             const float *t_ovr, const float *&tcur,
                                             float *&tnext) {
    const long long steps = D.sc->steps_done;
    if (mode == BWD_UPDATE) {
        tcur = ((steps - 1) & 1) ? S.t1 : S.t0;
        tnext = (steps & 1) ? S.t1 : S.t0;
    } else {
        tcur = t_ovr ? t_ovr : ((steps & 1) ? S.t1 : S.t0);
        tnext = nullptr;
    }
}

}  // namespace

// ------------------------------------------------------------------ k_init

__global__ void k_init(int n, int B, uint64_t seed, float *__restrict__ x,
                       float *__restrict__ mom, float *__restrict__ vel,
                       float *__restrict__ t0, uint8_t *__restrict__ bestx) {
    const int64_t total = (int64_t)n * B;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < total;
         q += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = q / B;
        const int64_t b = q - i * B;
        const uint64_t u = splitmix64_at(seed, (uint64_t)b * (uint64_t)n + (uint64_t)i);
        const float k = (float)(uint32_t)(u >> 40);
        const float xv = k * 0x1p-23f - 1.0f;
        x[q] = xv;
        mom[q] = 0.0f;
        vel[q] = 0.0f;
        t0[q] = tanh_fixed(xv);
        bestx[q] = 0;
    }
}

cudaError_t launch_init(const DevInst &I, const DevState &S, uint64_t seed, cudaStream_t st) {
    const int64_t total = (int64_t)I.n * I.B;
    int blocks = (int)((total + kThreads - 1) / kThreads);
    if (blocks > 152 * 16) blocks = 152 * 16;
    if (blocks < 1) blocks = 1;
    k_init<<<blocks, kThreads, 0, st>>>(I.n, I.B, seed, S.x, S.mom, S.vel, S.t0, S.bestx);
    return cudaGetLastError();
}

__global__ void k_tanh(const float *__restrict__ x, float *__restrict__ t, int64_t count) {
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < count;
         q += (int64_t)gridDim.x * blockDim.x)
        t[q] = tanh_fixed(__ldg(x + q));
}

cudaError_t launch_tanh(const float *x, float *t, int64_t count, cudaStream_t st) {
    int blocks = (int)((count + kThreads - 1) / kThreads);
    if (blocks > 152 * 16) blocks = 152 * 16;
    if (blocks < 1) blocks = 1;
    k_tanh<<<blocks, kThreads, 0, st>>>(x, t, count);
    return cudaGetLastError();
}

// Replicas of the per-restart cost accumulator that are in use: the blocks'
// additions to one address wait for one another (n=5000, B=256: 22 us with 32
// replicas, 38 with one), and the last block reads them all, a warp a restart
// where there are few restarts, else a thread a restart, eight loads in
// flight (sixteen raise the kernel's registers: 143 -> 153 us at n=1e6, B=16).
template <int VW>
__device__ __forceinline__ int cost_replicas(int B) {
    return VW < 8 && B <= 8 ? kRep : kRep / 2;
}

// Items a lane of the clause pass has in flight: two where their rows (VW
// values a literal) leave the registers for it.
__host__ __device__ constexpr int fwd_items(int VW, int KFIX) { return VW <= 4 && VW * KFIX <= 12 ? 2 : 1; }

// out[cols][rows] = in[rows][cols] of bytes, 32 columns by 128 rows a block
// through shared memory.
__global__ void __launch_bounds__(kThreads)
    k_transpose_u8(const uint8_t *__restrict__ in, uint8_t *__restrict__ out, int rows, int cols) {
    __shared__ uint8_t s[128][33];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c0 = blockIdx.y * 32;
    for (int64_t r0 = (int64_t)blockIdx.x * 128; r0 < rows; r0 += (int64_t)gridDim.x * 128) {
        for (int r = warp; r < 128; r += kThreads / 32)
            if (r0 + r < rows && c0 + lane < cols) s[r][lane] = in[(r0 + r) * cols + c0 + lane];
        __syncthreads();
        for (int k = threadIdx.x; k < 128 * 32; k += kThreads) {
            const int c = k >> 7, r = k & 127;
            if (r0 + r < rows && c0 + c < cols) out[(int64_t)(c0 + c) * rows + r0 + r] = s[r][c];
        }
        __syncthreads();
    }
}

cudaError_t launch_transpose_u8(const uint8_t *in, uint8_t *out, int rows, int cols, cudaStream_t st) {
    const dim3 grid((unsigned)std::min(((int64_t)rows + 127) / 128, (int64_t)152 * 16), (unsigned)((cols + 31) / 32));
    k_transpose_u8<<<grid, kThreads, 0, st>>>(in, out, rows, cols);
    return cudaGetLastError();
}

// The loss of the evaluated x from the clause pass's block partials, a warp
// a restart: by blocks of their own behind the variable pass's, so no block
// of variables waits for it, or, in a probe of few restarts, by the clause
// pass's last block.  The partials' rounding errors average out over their
// many blocks; what the reported value's error would come from is this chain
// and its division, so both carry a second word (3-SAT n=1e6, B=16, 20
// steps, against 64 bits: 5.6e-8 with one word, 2.2e-8 with two).

constexpr int kWarps = kThreads / 32;

__host__ __device__ inline int loss_blocks(int B) { return (B + kWarps - 1) / kWarps; }

// s + lo += v, the rounding error of the addition (Knuth's error-free sum of
// two floats) collected in lo.
__device__ __forceinline__ void add_two(float &s, float &lo, float v) {
    const float t = s + v, z = t - s;
    lo += (s - (t - z)) + (v - z);
    s = t;
}

__device__ __forceinline__ void reduce_loss(const DevStep &D, int B, int blk) {
    const int b = blk * kWarps + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (b >= B) return;
    float s = 0.0f, lo = 0.0f;
#pragma unroll 8
    for (int k = lane; k < D.fwd_blocks; k += 32) add_two(s, lo, __ldcg(D.lpart + (long long)k * B + b));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float ol = __shfl_xor_sync(0xffffffffu, lo, o);
        add_two(s, lo, __shfl_xor_sync(0xffffffffu, s, o));
        lo += ol;
    }
    if (lane == 0) {
        const long long c = D.cost[b];
        const int ln = D.sc->loss_norm;
        const long long d = ln == 1 ? 1 : ln == 2 ? D.sc->wsum : c;
        const float den = (float)d, dlo = (float)(d - (long long)den);
        const float q = s / den;
        const float r = (fmaf(-q, den, s) + lo) - q * dlo;
        D.loss[b] = c > 0 ? q + r / den : 0.0f;
    }
}

// The same as a call, where inlined it would cost the kernel registers.
static __device__ __noinline__ void call_reduce_loss(const DevStep &D, int B, int blk) { reduce_loss(D, B, blk); }

// Probes of up to this many restarts (a warp of one block each) take their
// loss in the clause pass's last block and save the reduction's launch (with
// the cost written in place of a copy, 3-SAT n=1000, B=8: forward and backward
// 281 -> 258 us, all of it the host's; 5-SAT n=30011, B=64 286 -> 266).  Eight
// restarts a thread are left out: k = 5 would go from 80 registers to 87, two
// resident blocks instead of three.
__host__ __device__ constexpr bool takes_loss(int VW, int B) { return VW <= 4 && B <= kWarps; }
bool probe_takes_loss(const DevInst &I) { return takes_loss(I.fwd_vw, I.B); }

// --------------------------------------------------------------- k_forward
// One item = (clause j, restart group g of VW restarts).  Where the rows of
// two clauses leave the registers for it (fwd_items: VW <= 4, and for k = 4
// and 5 VW <= 2) the grid-stride loop is unrolled by two (items base + lane
// and base + stride + lane; the stride is a multiple of G, so both belong to
// the thread's restart group), keeping the loads of two clauses in flight;
// wider groups already have several row loads per literal in flight.  The unsat bits of 32
// consecutive items are packed with shuffles into whole 32-bit words.

template <int VW, int KFIX>
__device__ __forceinline__ void forward_body(const DevInst &I, const float *__restrict__ t0,
                                             const float *__restrict__ t1,
                                             const float *__restrict__ t_ovr, const DevStep &D,
                                             uint32_t *__restrict__ ubits,
                                             float *__restrict__ fstore, int mode, int blk,
                                             int nblk) {
    constexpr int NU = fwd_items(VW, KFIX);  // items per lane per iteration
    extern __shared__ float4 dyn_smem[];
    __shared__ int s_last;

    grid_dep_wait();
    const int B = I.B;
    const int G = B / VW;
    const long long steps = D.sc->steps_done;
    const float *__restrict__ t = t_ovr ? t_ovr : ((steps & 1) ? t1 : t0);
    const int kfix = KFIX > 0 ? KFIX : I.kfix;
    const int lane = threadIdx.x & 31;
    const int gshift = __ffs(G) - 1;  // G = B / VW is a power of two
    const int g = threadIdx.x & (G - 1);
    const int col = g * VW;
    const long long total = (long long)I.m * G;
    const long long stride = (long long)nblk * blockDim.x;

    float lacc[VW];
    unsigned long long wacc[VW];
#pragma unroll
    for (int e = 0; e < VW; ++e) {
        lacc[e] = 0.0f;
        wacc[e] = 0ull;
    }
    constexpr int LPW = 32 / VW;  // lanes whose bits share one 32-bit word
    for (long long base = (long long)blk * blockDim.x + (threadIdx.x & ~31); base < total;
         base += NU * stride) {
        long long item[NU];
        bool act[NU];
        int jj[NU];
#pragma unroll
        for (int h = 0; h < NU; ++h) {
            item[h] = base + h * stride + lane;
            act[h] = item[h] < total;
            jj[h] = act[h] ? (int)(item[h] >> gshift) : 0;
        }
        float f[NU][VW];
        bool sat[NU][VW];
        if constexpr (KFIX > 0) {
            // every clause's literals, then every clause's rows
            int L[NU][KFIX];
#pragma unroll
            for (int h = 0; h < NU; ++h)
#pragma unroll
                for (int p = 0; p < KFIX; ++p) L[h][p] = __ldg(I.lit + jj[h] * KFIX + p);
            float tv[NU][KFIX][VW];
#pragma unroll
            for (int h = 0; h < NU; ++h)
#pragma unroll
                for (int p = 0; p < KFIX; ++p)
                    ldv<VW>(t + (int64_t)(L[h][p] >> 1) * B + col, tv[h][p]);
#pragma unroll
            for (int h = 0; h < NU; ++h)
#pragma unroll
                for (int e = 0; e < VW; ++e) {
                    sat[h][e] = false;
#pragma unroll
                    for (int p = 0; p < KFIX; ++p) {
                        const bool neg = L[h][p] & 1;
                        const float term = neg ? -tv[h][p][e] : tv[h][p][e];
                        f[h][e] = (p == 0) ? term : f[h][e] + term;
                        sat[h][e] |= ((tv[h][p][e] > 0.0f) != neg);
                    }
                }
        } else {
#pragma unroll
            for (int h = 0; h < NU; ++h) {
                int beg = 0, end = 0;
                if (act[h]) clause_range(I, kfix, jj[h], beg, end);
                clause_value<VW, true>(I, t, beg, end, col, f[h], sat[h]);
            }
        }
#pragma unroll
        for (int h = 0; h < NU; ++h) {
            unsigned nib = 0;
            if (act[h]) {
                const long long wj = I.w ? __ldg(I.w + jj[h]) : 1ll;
                const float wf = (float)wj;
                float q[VW];
#pragma unroll
                for (int e = 0; e < VW; ++e) {
                    q[e] = 0.0f;  // satisfied
                    if (!sat[h][e]) {
                        nib |= 1u << e;
                        wacc[e] += (unsigned long long)wj;
                        q[e] = wf * f[h][e];
                        lacc[e] += q[e] * f[h][e];
                        // f of an unsat clause is a sum of values <= 0; the
                        // minimum keeps it and makes a NaN add nothing
                        q[e] = fminf(q[e], 0.0f);
                    }
                }
                if (fstore) stv<VW>(fstore + (int64_t)jj[h] * B + col, q);
            }
            if (!fstore) {  // uniform: the variable pass reads the bits only when f is recomputed
                unsigned word = nib << ((lane % LPW) * VW);
#pragma unroll
                for (int o = 1; o < LPW; o <<= 1) word |= __shfl_xor_sync(0xffffffffu, word, o);
                if (act[h] && (lane % LPW) == 0) ubits[(item[h] * VW) >> 5] = word;
            }
        }
    }

    // per restart: block sums.  The threads of restart group g are those
    // with threadIdx.x % G == g (G divides the block).  Lanes of one warp in
    // the same group are combined by xor shuffles, each row (a warp, or G
    // threads where G > 32) puts its sums into shared memory, and threads add
    // the rows: all VW restarts of the groups at once behind one barrier, or,
    // with eight restarts a thread, one at a time (eight pairs of sums in
    // shuffles at once take the kernel from 64 to 69 registers, three blocks
    // per SM instead of four: 3-SAT n=1e6, B=16 143 -> 148 us).  The weights
    // are integers (any order is exact); the loss partial's order is free
    // because the loss is reported and never fed back into x.
    const int nrep = cost_replicas<VW>(B);
    unsigned long long *acc = D.wu_acc + (long long)(blk % nrep) * B;
    unsigned long long *s_w = reinterpret_cast<unsigned long long *>(dyn_smem);
    const int step = G < 32 ? 32 : G;  // threads of a row
    const int rows = blockDim.x / step;
    if constexpr (VW == 8) {
        float *s_l = reinterpret_cast<float *>(s_w + kThreads);
#pragma unroll
        for (int e = 0; e < VW; ++e) {
            unsigned long long sw = wacc[e];
            float sl = lacc[e];
            for (int o = G; o < 32; o <<= 1) {
                sw += __shfl_xor_sync(0xffffffffu, sw, o);
                sl += __shfl_xor_sync(0xffffffffu, sl, o);
            }
            s_w[threadIdx.x] = sw;
            s_l[threadIdx.x] = sl;
            __syncthreads();
            if (threadIdx.x < G) {
                sw = 0;
                sl = 0.0f;
                for (int k = 0; k < rows; ++k) {
                    sw += s_w[threadIdx.x + k * step];
                    sl += s_l[threadIdx.x + k * step];
                }
                const int b = threadIdx.x * VW + e;
                if (sw) atomicAdd(acc + b, sw);
                D.lpart[(long long)blk * B + b] = sl;
            }
            __syncthreads();
        }
    } else {
        float *s_l = reinterpret_cast<float *>(s_w + rows * B);
        const int row = threadIdx.x / step;
#pragma unroll
        for (int e = 0; e < VW; ++e) {
            unsigned long long sw = wacc[e];
            float sl = lacc[e];
            for (int o = G; o < 32; o <<= 1) {
                sw += __shfl_xor_sync(0xffffffffu, sw, o);
                sl += __shfl_xor_sync(0xffffffffu, sl, o);
            }
            if (G >= 32 || lane < G) {
                s_w[row * B + col + e] = sw;
                s_l[row * B + col + e] = sl;
            }
        }
        __syncthreads();
        for (int b = threadIdx.x; b < B; b += blockDim.x) {
            unsigned long long sw = 0;
            float sl = 0.0f;
            for (int k = 0; k < rows; ++k) {
                sw += s_w[k * B + b];
                sl += s_l[k * B + b];
            }
            if (sw) atomicAdd(acc + b, sw);
            D.lpart[(long long)blk * B + b] = sl;
        }
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = (atomicAdd(&D.sc->counter, 1u) == nblk - 1);
    __syncthreads();
    if (!s_last) return;
    // the variable pass's blocks may start: every other block is done, so
    // they spread over empty SMs (started before the blocks' sums they crowd
    // onto the SMs that were free first: weighted Zipf n=20000, B=1 21 -> 36
    // us a step)
    grid_dep_launch();
    __threadfence();
    // the last block's finish: every block's additions are complete (fence
    // before the counter).  The last thread makes the step's Adam scalars
    // (double division and root) while the others sum the replicas.
    if (mode == FWD_STEP && threadIdx.x == blockDim.x - 1) {
        StepScalars *sc = D.sc;
        const double p1 = sc->p1 * sc->beta1;
        const double p2 = sc->p2 * sc->beta2;
        sc->p1 = p1;
        sc->p2 = p2;
        sc->a_t = (float)(sc->lr / (1.0 - p1));
        sc->r_t = (float)(1.0 / sqrt(1.0 - p2));
        sc->steps_done = steps + 1;
    }
    // restart b's cost from L2, the replicas cleared for the next pass: one
    // thread a restart, or for a few restarts one thread a replica
    auto finish = [&](int b, unsigned long long wu) {
        const long long c = (long long)wu;
        D.cost[b] = c;
        if (mode != FWD_PROBE) {
            const long long bb = D.best[b];
            const int imp = c < bb;
            if (imp) {
                D.best[b] = c;
                D.best_step[b] = steps;
            }
            D.improved[b] = imp;
        }
        // g_j = (w_j f_j) * 2 / N with N = W_U (mean over the unsat clauses),
        // 1 (sum over them) or the total weight (mean over all clauses)
        const int ln = D.sc->loss_norm;
        const float den = ln == 1 ? 1.0f : (float)(ln == 2 ? D.sc->wsum : c);
        D.cscale[b] = c > 0 ? 2.0f / den : 0.0f;
    };
    unsigned long long my_tot = 0;  // this thread's restarts' costs
    if (VW < 8 && nrep == kRep) {
        for (int b = threadIdx.x >> 5; b < B; b += blockDim.x >> 5) {
            unsigned long long wu = __ldcg(D.wu_acc + (long long)lane * B + b);
            D.wu_acc[(long long)lane * B + b] = 0ull;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) wu += __shfl_xor_sync(0xffffffffu, wu, o);
            if (lane == 0) {
                my_tot += wu;
                finish(b, wu);
            }
        }
    } else {
        for (int b = threadIdx.x; b < B; b += blockDim.x) {
            unsigned long long wu = 0;
#pragma unroll 8
            for (int r = 0; r < kRep / 2; ++r) wu += __ldcg(D.wu_acc + (long long)r * B + b);
#pragma unroll 8
            for (int r = 0; r < kRep / 2; ++r) D.wu_acc[(long long)r * B + b] = 0ull;
            my_tot += wu;
            finish(b, wu);
        }
    }
    if (threadIdx.x == 0) D.sc->counter = 0;
    if constexpr (VW <= 4) {
        if (mode == FWD_PROBE && takes_loss(VW, B)) {
            __syncthreads();  // the costs
            call_reduce_loss(D, B, 0);
        }
    }
    if (fstore) return;  // uniform: only a recomputing variable pass reads the density
    s_w = reinterpret_cast<unsigned long long *>(dyn_smem);
    __syncthreads();
    if (threadIdx.x == 0) s_w[0] = 0ull;
    __syncthreads();
    if (my_tot) atomicAdd(s_w, my_tot);
    __syncthreads();
    if (threadIdx.x == 0) D.sc->dense = (double)s_w[0] * 16.0 > (double)D.sc->wsum * (double)B;
}

// Dynamic shared memory of the clause pass: its per-restart block sums.
template <int VW>
static size_t fwd_smem(int B) {
    const int G = B / VW;
    return (VW == 8 ? (size_t)kThreads : (size_t)(kThreads / (G < 32 ? 32 : G)) * B) *
           (sizeof(unsigned long long) + sizeof(float));
}

template <int VW, int KFIX>
__global__ void __launch_bounds__(kThreads)
    k_forward(DevInst I, const float *__restrict__ t0, const float *__restrict__ t1,
              const float *__restrict__ t_ovr, DevStep D, uint32_t *__restrict__ ubits,
              float *__restrict__ fstore, int mode) {
    forward_body<VW, KFIX>(I, t0, t1, t_ovr, D, ubits, fstore, mode, blockIdx.x, gridDim.x);
}

// Four restarts a thread in the clause pass; eight where the store is past
// 64 MiB: its rows then come from HBM and are better taken whole (3-SAT
// n=1e6, B=16: 140 us with eight, 172 with four; n=3e5, B=8, 41 MB: 38 / 31;
// ordering principle on 31 elements, B=8: 21 / 15).
int auto_fwd_vw(int B, int64_t m) {
    return std::min(B, (double)m * B * sizeof(float) > 64.0 * (1 << 20) ? 8 : 4);
}
int auto_stage_vw(int B) { return B < 4 ? B : 4; }
int update_vw(int B) { return B < 4 ? B : 4; }

template <int VW>
static int fwd_resident(const DevInst &I) {
    int per_sm = 0;
    const size_t smem = fwd_smem<VW>(I.B);
    cudaError_t e;
    switch (I.kfix) {
        case 3: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_forward<VW, 3>, kThreads, smem); break;
        case 4: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_forward<VW, 4>, kThreads, smem); break;
        case 5: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_forward<VW, 5>, kThreads, smem); break;
        default: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_forward<VW, 0>, kThreads, smem); break;
    }
    if (e != cudaSuccess || per_sm < 1) {
        cudaGetLastError();
        per_sm = 2;
    }
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) {
        cudaGetLastError();
        sms = 152;
    }
    return per_sm * sms;
}

// One wave of resident blocks (the grid-stride loop covers the rest), or
// fewer when the clauses do not fill it.
int fwd_grid_blocks(const DevInst &I) {
    const int VW = I.fwd_vw;
    const int per_thread = fwd_items(VW, I.kfix >= 3 && I.kfix <= 5 ? I.kfix : 0);
    const long long items = (long long)I.m * (I.B / VW);
    long long blocks = (items + per_thread * kThreads - 1) / (per_thread * kThreads);
    int resident;
    switch (VW) {
        case 8: resident = fwd_resident<8>(I); break;
        case 4: resident = fwd_resident<4>(I); break;
        case 2: resident = fwd_resident<2>(I); break;
        default: resident = fwd_resident<1>(I); break;
    }
    if (blocks > resident) blocks = resident;
    if (blocks < 1) blocks = 1;
    return (int)blocks;
}

template <int VW>
static cudaError_t launch_forward_vw(const DevInst &I, const DevState &S, const DevStep &D,
                                     int mode, const float *t_ovr, cudaStream_t st) {
    const int blocks = D.fwd_blocks;
    const size_t smem = fwd_smem<VW>(I.B);
    // one instantiation per common clause length: all literals, then all rows
    // of a clause in flight (k = 5, n=30011, m=639234, B=64: 144 -> 97 us)
    switch (I.kfix) {
        case 3: return launch_pdl(k_forward<VW, 3>, blocks, kThreads, smem, st, I, S.t0, S.t1, t_ovr, D, S.ubits, S.fstore, mode);
        case 4: return launch_pdl(k_forward<VW, 4>, blocks, kThreads, smem, st, I, S.t0, S.t1, t_ovr, D, S.ubits, S.fstore, mode);
        case 5: return launch_pdl(k_forward<VW, 5>, blocks, kThreads, smem, st, I, S.t0, S.t1, t_ovr, D, S.ubits, S.fstore, mode);
        default: return launch_pdl(k_forward<VW, 0>, blocks, kThreads, smem, st, I, S.t0, S.t1, t_ovr, D, S.ubits, S.fstore, mode);
    }
}

cudaError_t launch_forward(const DevInst &I0, const DevState &S, const DevStep &D, int mode,
                           const float *t_override, cudaStream_t st) {
    // with the store's rows grouped by block, the clause pass walks the
    // clauses in row order (its item index is the row it writes)
    DevInst I = I0;
    if (I0.plit) {
        I.lit = I0.plit;
        I.coff = I0.pcoff ? I0.pcoff : I0.coff;
        I.w = I0.pw;
    }
    switch (I.fwd_vw) {
        case 8: return launch_forward_vw<8>(I, S, D, mode, t_override, st);
        case 4: return launch_forward_vw<4>(I, S, D, mode, t_override, st);
        case 2: return launch_forward_vw<2>(I, S, D, mode, t_override, st);
        default: return launch_forward_vw<1>(I, S, D, mode, t_override, st);
    }
}

// -------------------------------------------------------------- k_backward
// Heavy variables: a warp per (1024-occurrence chunk, restart group of VW
// restarts), a lane per 32-occurrence leaf.  A lane sums its leaf in the
// stored order straight from its gathers, the lanes' leaves meet by the
// dyadic shuffle tree, and the last chunk of a (variable, group) combines the
// chunk partials with the same tree and applies the update.  No barrier and
// no staging: bound by the latency of the word -> row chain, hidden by 32
// leaves a warp.  The form before it staged a chunk in shared memory with a
// block and summed the leaves with one of its eight warps (32 lanes on one
// bank): variable pass of weighted Zipf n=2e5, m=1e6 (3255 chunks), B=1 49 ->
// 40 us, B=8 201 -> 130 us.
template <int VW, int KFIX, bool STORE>
__device__ __forceinline__ void heavy_body(const DevInst &I, const DevState &S, const DevStep &D,
                                           int mode, const float *__restrict__ t_ovr,
                                           const float *__restrict__ gscale,
                                           float *__restrict__ grad_out, int blk) {
    constexpr int C = VW <= 2 ? 8 : 4;  // occurrences in flight per lane
    const int B = I.B;
    const int G = B / VW;
    const int kfix = KFIX > 0 ? KFIX : I.kfix;
    const int lane = threadIdx.x & 31;
    const long long wid = (long long)blk * kWarps + (threadIdx.x >> 5);
    const long long cidx = wid / G;
    if (cidx >= I.heavy_chunks) return;
    const int gg = (int)(wid - cidx * G);
    const int col = gg * VW;
    const int h = __ldg(I.heavy_of_chunk + cidx);
    const int i = __ldg(I.heavy_var + h);
    const int c0 = __ldg(I.heavy_chunk0 + h);
    const int nch = __ldg(I.heavy_chunk0 + h + 1) - c0;
    const int vend = __ldg(I.voff + i + 1);
    const int cb = __ldg(I.voff + i) + (int)(cidx - c0) * kChunk;
    const int cn = min(kChunk, vend - cb);  // occurrences in this chunk
    grid_dep_wait();  // the list loads above need nothing of the clause pass
    const float *tcur;
    float *tnext;
    step_buffers(S, D, mode, t_ovr, tcur, tnext);
    if (mode != BWD_BITS_ONLY) {
        float cs[VW];
#pragma unroll
        for (int e = 0; e < VW; ++e) cs[e] = D.cscale[col + e];
        const bool dense = D.sc->dense != 0;
        const bool expanded = KFIX == 3 && I.occx != nullptr;
        const int pb = cb + min(32 * lane, cn), pe = cb + min(32 * lane + 32, cn);
        float leaf[VW];
#pragma unroll
        for (int e = 0; e < VW; ++e) leaf[e] = 0.0f;
        const int none = STORE && VW > 1 ? I.m << I.occ_shift : 0;  // the store's zero row
        int on[C];
        int2 oxn[C];
#pragma unroll
        for (int u = 0; u < C; ++u) {
            const bool okn = pb + u < pe;
            on[u] = okn ? __ldg(I.occ + pb + u) : none;
            oxn[u] = (expanded && okn) ? __ldg(I.occx + pb + u) : make_int2(0, 0);
        }
        for (int p = pb; p < pe; p += C) {
            int o[C];
            int2 ox[C];
            bool ok[C];
#pragma unroll
            for (int u = 0; u < C; ++u) {
                ok[u] = p + u < pe;
                o[u] = on[u];
                ox[u] = oxn[u];
                const bool okn = p + C + u < pe;
                on[u] = okn ? __ldg(I.occ + p + C + u) : none;
                oxn[u] = (expanded && okn) ? __ldg(I.occx + p + C + u) : make_int2(0, 0);
            }
            occ_accumulate<VW, KFIX, C, STORE, false>(I, S, kfix, tcur, o, ox, ok, i, col, cs, dense, p == pb, leaf);
        }
        __syncwarp();
        const int K = (cn + 31) / 32;
#pragma unroll
        for (int e = 0; e < VW; ++e) leaf[e] = warp_dyadic(leaf[e], K, lane);
        if (lane == 0) {
#pragma unroll
            for (int e = 0; e < VW; ++e) D.hpart[cidx * B + col + e] = leaf[e];
        }
    }
    const int64_t q0 = (int64_t)i * B + col;
    if (mode == BWD_BITS_ONLY) {
        if (cidx == c0 && lane < VW && D.improved[col + lane]) S.bestx[q0 + lane] = S.x[q0 + lane] > 0.0f;
        return;
    }
    grid_dep_launch();
    int last = 1;
    if (nch > 1) {
        if (lane == 0) {
            __threadfence();
            last = atomicAdd(D.hcount + (long long)h * G + gg, 1u) == (unsigned)(nch - 1);
            if (last) D.hcount[(long long)h * G + gg] = 0;
        }
        last = __shfl_sync(0xffffffffu, last, 0);
    }
    if (!last) return;
    __threadfence();
    __syncwarp();
    // last chunk of this (variable, group): 32 consecutive chunk partials at
    // a time are a complete dyadic block; four blocks' loads in flight
    float Ssum[VW];
#pragma unroll
    for (int e = 0; e < VW; ++e) {
        LeafCounter<12> lc;  // up to 4095 blocks of 32 chunks
        lc.init();
        for (int base = 0; base < nch; base += 128) {
            float v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int r = base + 32 * u + lane;
                v[u] = r < nch ? __ldcg(D.hpart + (long long)(c0 + r) * B + col + e) : 0.0f;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int K = nch - base - 32 * u;
                if (K > 0) lc.push(warp_dyadic(v[u], min(K, 32), lane));
            }
        }
        Ssum[e] = lc.finish();
    }
    if (lane != 0) return;
    finish_variable<VW>(S, D, adam_view(D.sc), mode, q0, col, tcur, Ssum, tnext, gscale, grad_out);
}

template <int VW, int KFIX, bool STORE>
__global__ void __launch_bounds__(kThreads)
    k_backward_heavy(DevInst I, DevState S, DevStep D, int mode, const float *__restrict__ t_ovr,
                     const float *__restrict__ gscale, float *__restrict__ grad_out) {
    heavy_body<VW, KFIX, STORE>(I, S, D, mode, t_ovr, gscale, grad_out, blockIdx.x);
}

// k_backward_light: one block per range of consecutive light variables.
// A task is (variable, 32-occurrence leaf, group of VS restarts); the
// restart group is the fastest index, so the lanes of a warp that share a
// leaf read consecutive columns of the same rows.  A thread sums its leaf's
// terms in the stored order, with the loads of four occurrences in flight
// at a time.  A variable with one leaf (or none) is finished by the same
// thread; the leaves of a longer variable meet in shared memory and the
// thread of its first leaf combines them by the dyadic counter, then
// applies the update.  A thread keeps its restart group for all its tasks
// (the task stride, kThreads, is a multiple of the group count).
template <int VS, int KFIX, bool STORE>
__device__ __forceinline__ void vars_body(const DevInst &I, const DevState &S, const DevStep &D,
                                          int mode, const float *__restrict__ t_ovr,
                                          const float *__restrict__ gscale,
                                          float *__restrict__ grad_out, int blk) {
    constexpr int C = 4;  // occurrences in flight per thread
    extern __shared__ float4 dyn_smem[];
    __shared__ int s_voff[kThreads + 1];
    __shared__ int s_lpre[kThreads + 1];
    __shared__ int s_wtot[kThreads / 32];
    const int B = I.B;
    const int kfix = KFIX > 0 ? KFIX : I.kfix;
    if (blk >= I.n_lblk) {  // the blocks behind the variables'
        grid_dep_wait();
        if (mode == BWD_UPDATE) {
            if constexpr (STORE) reduce_loss(D, B, blk - I.n_lblk);
            else call_reduce_loss(D, B, blk - I.n_lblk);
        }
        return;
    }
    float *s_leaf = reinterpret_cast<float *>(dyn_smem);
    const int2 rg = I.lblk[blk];
    const int v0 = rg.x, nv = rg.y - rg.x;  // nv <= kThreads

    // occurrence offsets and leaf counts of the block's variables, then the
    // exclusive prefix of the leaf counts (warp scans, then warp totals)
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int nl = 0;
    if (threadIdx.x < nv) {
        const int a = __ldg(I.voff + v0 + threadIdx.x);
        const int b = __ldg(I.voff + v0 + threadIdx.x + 1);
        s_voff[threadIdx.x] = a;
        if (threadIdx.x == nv - 1) s_voff[nv] = b;
        nl = mode == BWD_BITS_ONLY ? 1 : max(1, (b - a + 31) >> 5);
    }
    int inc = nl;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, inc, d);
        if (lane >= d) inc += y;
    }
    if (lane == 31) s_wtot[warp] = inc;
    __syncthreads();
    int before = 0;
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) before += w < warp ? s_wtot[w] : 0;
    if (threadIdx.x < nv) s_lpre[threadIdx.x] = before + inc - nl;
    if (threadIdx.x == nv - 1) s_lpre[nv] = before + inc;
    __syncthreads();
    grid_dep_wait();  // the offsets above need nothing of the clause pass
    const float *tcur;
    float *tnext;
    step_buffers(S, D, mode, t_ovr, tcur, tnext);
    const AdamView A = adam_view(D.sc);

    const int GS = B / VS;
    const int gshift = __ffs(GS) - 1;  // GS is a power of two <= kThreads
    const int col = (threadIdx.x & (GS - 1)) * VS;
    const int nleaves = s_lpre[nv];
    const int ntasks = nleaves << gshift;
    float cs[VS];
#pragma unroll
    for (int e = 0; e < VS; ++e) cs[e] = D.cscale[col + e];
    const bool dense = D.sc->dense != 0;
    const bool expanded = KFIX == 3 && I.occx != nullptr;

    const bool one_leaf_each = nleaves == nv;  // uniform: task ti belongs to variable ti
    for (int t = threadIdx.x; t < ntasks; t += kThreads) {
        const int ti = t >> gshift;
        int lo = 0, hi = nv - 1;  // the variable: last vloc with s_lpre[vloc] <= ti
        if (one_leaf_each) lo = ti;
        else
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (s_lpre[mid] <= ti) lo = mid; else hi = mid - 1;
            }
        const int vloc = lo;
        const int L = ti - s_lpre[vloc];
        const int nleaf = s_lpre[vloc + 1] - s_lpre[vloc];
        const int i = v0 + vloc;
        const int64_t q0 = (int64_t)i * B + col;
        if (mode == BWD_BITS_ONLY) {
            float xv[VS];
            ldv<VS>(S.x + q0, xv);
#pragma unroll
            for (int e = 0; e < VS; ++e)
                if (D.improved[col + e]) S.bestx[q0 + e] = xv[e] > 0.0f;
            continue;
        }
        const int pb = s_voff[vloc] + 32 * L;
        const int pe = min(pb + 32, s_voff[vloc + 1]);
        // with one or two restarts a task there are registers to have the
        // variable's state on its way while the occurrences are gathered
        constexpr bool PRE = VS <= 2 && STORE;
        VarState<VS> pre;
        if constexpr (PRE)
            if (nleaf == 1 && mode == BWD_UPDATE) pre.load(S, tcur, q0);
        float leaf[VS];
#pragma unroll
        for (int e = 0; e < VS; ++e) leaf[e] = 0.0f;
        // occurrence words one batch ahead: the next batch's words are in
        // flight while this batch's f values are gathered
        const int none = STORE && VS > 1 ? I.m << I.occ_shift : 0;  // the store's zero row
        int on[C];
        int2 oxn[C];
#pragma unroll
        for (int u = 0; u < C; ++u) {
            const bool okn = pb + u < pe;
            on[u] = okn ? __ldg(I.occ + pb + u) : none;
            oxn[u] = (expanded && okn) ? __ldg(I.occx + pb + u) : make_int2(0, 0);
        }
        for (int p = pb; p < pe; p += C) {
            int o[C];
            int2 ox[C];
            bool ok[C];
#pragma unroll
            for (int u = 0; u < C; ++u) {
                ok[u] = p + u < pe;
                o[u] = on[u];
                ox[u] = oxn[u];
                const bool okn = p + C + u < pe;
                on[u] = okn ? __ldg(I.occ + p + C + u) : none;
                oxn[u] = (expanded && okn) ? __ldg(I.occx + p + C + u) : make_int2(0, 0);
            }
            occ_accumulate<VS, KFIX, C, STORE, (VS >= 2)>(I, S, kfix, tcur, o, ox, ok, i, col, cs, dense, p == pb, leaf);
        }
        if (nleaf == 1) {
            finish_variable<VS>(S, D, A, mode, q0, col, tcur, leaf, tnext, gscale, grad_out, PRE ? &pre : nullptr);
        } else {
            stv<VS>(s_leaf + (int64_t)ti * B + col, leaf);
        }
    }
    grid_dep_launch();
    if (mode == BWD_BITS_ONLY || nleaves == nv) return;  // uniform: no variable has two leaves
    __syncthreads();
    for (int t = threadIdx.x; t < ntasks; t += kThreads) {
        const int ti = t >> gshift;
        int lo = 0, hi = nv - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (s_lpre[mid] <= ti) lo = mid; else hi = mid - 1;
        }
        const int vloc = lo;
        const int nleaf = s_lpre[vloc + 1] - s_lpre[vloc];
        if (ti != s_lpre[vloc] || nleaf == 1) continue;
        LeafCounter<5> lc[VS];  // at most kLightMaxDeg = 512 occurrences: 16 leaves
#pragma unroll
        for (int e = 0; e < VS; ++e) lc[e].init();
        for (int l = 0; l < nleaf; ++l) {
            float v[VS];
#pragma unroll
            for (int e = 0; e < VS; ++e) v[e] = s_leaf[(ti + l) * B + col + e];
#pragma unroll
            for (int e = 0; e < VS; ++e) lc[e].push(v[e]);
        }
        float Ssum[VS];
#pragma unroll
        for (int e = 0; e < VS; ++e) Ssum[e] = lc[e].finish();
        const int64_t q0 = (int64_t)(v0 + vloc) * B + col;
        finish_variable<VS>(S, D, A, mode, q0, col, tcur, Ssum, tnext, gscale, grad_out);
    }
}

template <int VS, int KFIX, bool STORE>
__global__ void __launch_bounds__(kThreads)
    k_backward_light(DevInst I, DevState S, DevStep D, int mode, const float *__restrict__ t_ovr,
                     const float *__restrict__ gscale, float *__restrict__ grad_out) {
    vars_body<VS, KFIX, STORE>(I, S, D, mode, t_ovr, gscale, grad_out, blockIdx.x);
}

// The same pass held to 64 registers a thread, so that four 256-thread
// blocks are resident per SM instead of three: used for the shapes where
// that costs no spills (stored w*f with up to 4 restarts a task, or up to 2
// restarts a task).  The pass is latency-bound on its gathers, so the
// extra resident warps hide more of that latency.
template <int VS, int KFIX, bool STORE>
__global__ void __launch_bounds__(kThreads, 4)
    k_backward_light_occ4(DevInst I, DevState S, DevStep D, int mode, const float *__restrict__ t_ovr,
                          const float *__restrict__ gscale, float *__restrict__ grad_out) {
    vars_body<VS, KFIX, STORE>(I, S, D, mode, t_ovr, gscale, grad_out, blockIdx.x);
}

// Heavy-variable chunks and light blocks in one launch: blocks [0, hblocks)
// take the chunks (first, so the long variables start early), the rest the
// light blocks.  The two write disjoint variables, so neither waits for the
// other, and each fills the other's last partial wave.
template <int VS, int VU, int KFIX, bool STORE, int MINB>
__global__ void __launch_bounds__(kThreads, MINB)
    k_backward_mixed(DevInst I, DevState S, DevStep D, int mode, const float *__restrict__ t_ovr,
                     const float *__restrict__ gscale, float *__restrict__ grad_out, int hblocks) {
    if ((int)blockIdx.x < hblocks)
        heavy_body<VU, KFIX, STORE>(I, S, D, mode, t_ovr, gscale, grad_out, blockIdx.x);
    else
        vars_body<VS, KFIX, STORE>(I, S, D, mode, t_ovr, gscale, grad_out, (int)blockIdx.x - hblocks);
}

// Blocks of the heavy variables: a warp per (chunk, restart group).
int heavy_blocks_of(const DevInst &I) {
    const long long warps = I.n_heavy > 0 ? I.heavy_chunks * (I.B / update_vw(I.B)) : 0;
    return (int)((warps + kWarps - 1) / kWarps);
}

// Blocks of the light variables, with those of the loss behind them.
int light_blocks_of(const DevInst &I, int mode) {
    return std::max(1, I.n_lblk + (mode == BWD_UPDATE ? loss_blocks(I.B) : 0));
}

template <int VS, int VU, int KFIX, bool STORE>
static cudaError_t launch_backward_k(const DevInst &I, const DevState &S, const DevStep &D,
                                     int mode, const float *t_ovr, const float *gscale,
                                     float *grad_out, cudaStream_t st) {
    const long long lblocks = light_blocks_of(I, mode);
    const size_t smem = light_smem_bytes(I.task_cap, VS);
    if (I.n_heavy > 0) {
        const long long hblocks = heavy_blocks_of(I);
        if constexpr (STORE && VU <= 2 && VS <= 2) {
            // one launch where that keeps the light blocks' 64-register,
            // four-blocks-per-SM shape without spills
            return launch_pdl(k_backward_mixed<VS, VU, KFIX, STORE, 4>, (unsigned)(hblocks + lblocks), kThreads, smem, st,
                              I, S, D, mode, t_ovr, gscale, grad_out, (int)hblocks);
        }
        const cudaError_t e = launch_pdl(k_backward_heavy<VU, KFIX, STORE>, (unsigned)hblocks, kThreads, 0, st, I, S, D, mode,
                                         t_ovr, gscale, grad_out);
        if (e) return e;
    }
    if constexpr ((STORE && VS <= 4) || VS <= 2)
        return launch_pdl(k_backward_light_occ4<VS, KFIX, STORE>, (unsigned)lblocks, kThreads, smem, st, I, S, D, mode, t_ovr,
                          gscale, grad_out);
    else
        return launch_pdl(k_backward_light<VS, KFIX, STORE>, (unsigned)lblocks, kThreads, smem, st, I, S, D, mode, t_ovr,
                          gscale, grad_out);
}

template <int VS, int VU>
static cudaError_t launch_backward_vw(const DevInst &I, const DevState &S, const DevStep &D,
                                      int mode, const float *t_ovr, const float *gscale,
                                      float *grad_out, cudaStream_t st) {
    // f stored by the clause pass, or recomputed from the unsat bits
    if (S.fstore) {
        if (I.kfix == 3) return launch_backward_k<VS, VU, 3, true>(I, S, D, mode, t_ovr, gscale, grad_out, st);
        return launch_backward_k<VS, VU, 0, true>(I, S, D, mode, t_ovr, gscale, grad_out, st);
    }
    if (I.kfix == 3) return launch_backward_k<VS, VU, 3, false>(I, S, D, mode, t_ovr, gscale, grad_out, st);
    return launch_backward_k<VS, VU, 0, false>(I, S, D, mode, t_ovr, gscale, grad_out, st);
}

cudaError_t launch_backward(const DevInst &I, const DevState &S, const DevStep &D, int mode,
                            const float *t_override, const float *gscale, float *grad_out,
                            cudaStream_t st) {
    const int vu = update_vw(I.B);
    switch (I.stage_vw * 8 + vu) {
        case 16 * 8 + 4: return launch_backward_vw<16, 4>(I, S, D, mode, t_override, gscale, grad_out, st);
        case 8 * 8 + 4: return launch_backward_vw<8, 4>(I, S, D, mode, t_override, gscale, grad_out, st);
        case 4 * 8 + 4: return launch_backward_vw<4, 4>(I, S, D, mode, t_override, gscale, grad_out, st);
        case 2 * 8 + 4: return launch_backward_vw<2, 4>(I, S, D, mode, t_override, gscale, grad_out, st);
        case 1 * 8 + 4: return launch_backward_vw<1, 4>(I, S, D, mode, t_override, gscale, grad_out, st);
        case 2 * 8 + 2: return launch_backward_vw<2, 2>(I, S, D, mode, t_override, gscale, grad_out, st);
        case 1 * 8 + 2: return launch_backward_vw<1, 2>(I, S, D, mode, t_override, gscale, grad_out, st);
        case 1 * 8 + 1: return launch_backward_vw<1, 1>(I, S, D, mode, t_override, gscale, grad_out, st);
        default: return cudaErrorInvalidValue;
    }
}

// ------------------------------------------------------------ batched step
// One launch of each pass advances every instance of a slot table by one
// iteration of Algorithm 1.  A block finds its slot by binary search in the
// launch's block prefix table and runs the same body on that slot's views
// with its block index inside the slot.

__device__ __forceinline__ int slot_of(const int *__restrict__ start, int nslot, int blk) {
    int lo = 0, hi = nslot - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(start + mid) <= blk) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// The block's slot, copied to shared memory: its views are then as close as
// kernel arguments without holding registers.
__device__ __forceinline__ const SlotDesc &block_slot(const SlotDesc *__restrict__ slots, int s) {
    static_assert(sizeof(SlotDesc) % 4 == 0 && sizeof(SlotDesc) / 4 <= kThreads, "a word of the slot a thread");
    __shared__ __align__(16) unsigned char raw[sizeof(SlotDesc)];
    if (threadIdx.x < sizeof(SlotDesc) / 4)
        reinterpret_cast<uint32_t *>(raw)[threadIdx.x] = reinterpret_cast<const uint32_t *>(slots + s)[threadIdx.x];
    __syncthreads();
    return *reinterpret_cast<const SlotDesc *>(raw);
}

template <int VW>
__global__ void __launch_bounds__(kThreads, VW <= 4 ? 4 : 1)
    k_forward_batch(const SlotDesc *__restrict__ slots, const int *__restrict__ start, int nslot) {
    const int s = slot_of(start, nslot, blockIdx.x);
    const int b0 = __ldg(start + s), b1 = __ldg(start + s + 1);
    const SlotDesc &sd = block_slot(slots, s);
    const int blk = blockIdx.x - b0, nblk = b1 - b0;
    switch (sd.I.kfix) {  // uniform over the block
        case 3: forward_body<VW, 3>(sd.I, sd.S.t0, sd.S.t1, nullptr, sd.D, sd.S.ubits, sd.S.fstore, FWD_STEP, blk, nblk); break;
        case 4: forward_body<VW, 4>(sd.I, sd.S.t0, sd.S.t1, nullptr, sd.D, sd.S.ubits, sd.S.fstore, FWD_STEP, blk, nblk); break;
        case 5: forward_body<VW, 5>(sd.I, sd.S.t0, sd.S.t1, nullptr, sd.D, sd.S.ubits, sd.S.fstore, FWD_STEP, blk, nblk); break;
        default: forward_body<VW, 0>(sd.I, sd.S.t0, sd.S.t1, nullptr, sd.D, sd.S.ubits, sd.S.fstore, FWD_STEP, blk, nblk); break;
    }
}

template <int VU>
__global__ void __launch_bounds__(kThreads)
    k_backward_heavy_batch(const SlotDesc *__restrict__ slots, const int *__restrict__ start, int nslot) {
    const int s = slot_of(start, nslot, blockIdx.x);
    const SlotDesc &sd = block_slot(slots, s);
    heavy_body<VU, 0, true>(sd.I, sd.S, sd.D, BWD_UPDATE, nullptr, nullptr, nullptr,
                      blockIdx.x - __ldg(start + s));
}

template <int VS>
__global__ void __launch_bounds__(kThreads, VS <= 4 ? 4 : 1)
    k_backward_light_batch(const SlotDesc *__restrict__ slots, const int *__restrict__ start, int nslot) {
    const int s = slot_of(start, nslot, blockIdx.x);
    const int b0 = __ldg(start + s);
    const SlotDesc &sd = block_slot(slots, s);
    vars_body<VS, 0, true>(sd.I, sd.S, sd.D, BWD_UPDATE, nullptr, nullptr, nullptr, blockIdx.x - b0);
}

template <int VS, int VU>
static cudaError_t launch_batch_bwd(const SlotDesc *slots, int nslot, const int *heavy_start,
                                    int heavy_total, const int *light_start, int light_total,
                                    size_t smem, cudaStream_t st) {
    if (heavy_total > 0) {
        const cudaError_t e =
            launch_pdl(k_backward_heavy_batch<VU>, (unsigned)heavy_total, kThreads, 0, st, slots, heavy_start, nslot);
        if (e) return e;
    }
    return launch_pdl(k_backward_light_batch<VS>, (unsigned)light_total, kThreads, smem, st, slots, light_start, nslot);
}

cudaError_t launch_step_batch(const SlotDesc *slots, int nslot, const int *fwd_start, int fwd_total,
                              const int *heavy_start, int heavy_total, const int *light_start,
                              int light_total, int B, int fwd_vw, int stage_vw, int task_cap,
                              cudaStream_t st) {
    if (nslot <= 0) return cudaSuccess;
    cudaError_t e;
    switch (fwd_vw) {
        case 8: e = launch_pdl(k_forward_batch<8>, (unsigned)fwd_total, kThreads, fwd_smem<8>(B), st, slots, fwd_start, nslot); break;
        case 4: e = launch_pdl(k_forward_batch<4>, (unsigned)fwd_total, kThreads, fwd_smem<4>(B), st, slots, fwd_start, nslot); break;
        case 2: e = launch_pdl(k_forward_batch<2>, (unsigned)fwd_total, kThreads, fwd_smem<2>(B), st, slots, fwd_start, nslot); break;
        default: e = launch_pdl(k_forward_batch<1>, (unsigned)fwd_total, kThreads, fwd_smem<1>(B), st, slots, fwd_start, nslot); break;
    }
    if (e) return e;
    const size_t smem = light_smem_bytes(task_cap, stage_vw);
    const int vu = update_vw(B);
    switch (stage_vw * 8 + vu) {
        case 16 * 8 + 4: return launch_batch_bwd<16, 4>(slots, nslot, heavy_start, heavy_total, light_start, light_total, smem, st);
        case 8 * 8 + 4: return launch_batch_bwd<8, 4>(slots, nslot, heavy_start, heavy_total, light_start, light_total, smem, st);
        case 4 * 8 + 4: return launch_batch_bwd<4, 4>(slots, nslot, heavy_start, heavy_total, light_start, light_total, smem, st);
        case 2 * 8 + 4: return launch_batch_bwd<2, 4>(slots, nslot, heavy_start, heavy_total, light_start, light_total, smem, st);
        case 1 * 8 + 4: return launch_batch_bwd<1, 4>(slots, nslot, heavy_start, heavy_total, light_start, light_total, smem, st);
        case 2 * 8 + 2: return launch_batch_bwd<2, 2>(slots, nslot, heavy_start, heavy_total, light_start, light_total, smem, st);
        case 1 * 8 + 2: return launch_batch_bwd<1, 2>(slots, nslot, heavy_start, heavy_total, light_start, light_total, smem, st);
        case 1 * 8 + 1: return launch_batch_bwd<1, 1>(slots, nslot, heavy_start, heavy_total, light_start, light_total, smem, st);
        default: return cudaErrorInvalidValue;
    }
}

// loss per restart from the forward partials (used where no update follows)
__global__ void k_loss_reduce(DevStep D, int B) { reduce_loss(D, B, blockIdx.x); }

cudaError_t launch_loss_reduce(const DevStep &D, int B, cudaStream_t st) {
    k_loss_reduce<<<loss_blocks(B), kThreads, 0, st>>>(D, B);
    return cudaGetLastError();
}

}  // namespace msat

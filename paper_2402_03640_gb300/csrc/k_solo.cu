// Small instances: one CTA per restart runs every step of a call (sm_103a).
//
// Restarts are independent, and the step's scalars (the Adam products) are
// the same for all of them, so a restart whose state fits one SM's shared
// memory needs no other SM: block b holds x, the Adam moments, t = tanh(x)
// and the clause pass's w*f of restart b and takes all steps of the call,
// then (if asked) the evaluation of the final x, in one launch.  Two block
// barriers a step: clause pass | variable pass (a third where a variable has
// more than one 32-occurrence leaf).
//
// Bound: for instances of a few hundred variables the dependent chain of a
// step (literal words -> t -> f -> barrier -> cost sum -> w*f -> occurrence
// sum -> Adam -> tanh -> barrier); from a few thousand on the shared-memory
// gathers (2 nnz random 4-byte reads a step, about 3.4 bank cycles per warp
// read).
//
// The literal and occurrence lists are 16-bit words in slices of 32 lanes
// (one lane per clause / leaf task), four words a load, padded with a dummy
// variable (t = +0) and a dummy clause (w*f = +0).  Clauses are ordered by
// length and leaf tasks by occurrence count so a slice's lanes have about
// equal lengths.  They sit in shared memory where they fit beside the state,
// else they stream from L2 (the four words of 32 lanes are one 256-byte
// line).
//
// Bits: every sum has the order of the per-pass kernels (literal and
// occurrence order, 32-term leaves, dyadic tree), every operation is theirs.
// Padding and satisfied clauses add +-0, which can only change the sign of a
// zero sum; the sum is brought to +0 before it is used (S + 0).  The loss
// partials are summed in another order (the loss is reported, never fed
// back).

#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <functional>
#include <future>
#include <system_error>
#include <vector>

#include "host_cnf.cuh"
#include "msat_internal.cuh"
#include "step_math.cuh"

namespace msat {

namespace {

constexpr int kSoloMaxThreads = 1024;         // work threads plus the scalar warp
constexpr size_t kSoloSmemMax = 226 * 1024;   // dynamic shared memory of a block
constexpr int kSoloRing = 32;                 // steps of one chunk of Adam scalars
constexpr int kNarrowLeaves = 15;             // leaves one thread combines; more take a warp

struct SoloSmem {  // byte offsets into the dynamic shared memory
    uint32_t t, q, x, m, v, leaf, best, lists, total;
};

__host__ __device__ inline uint32_t pad16(uint32_t b) { return (b + 15u) & ~15u; }

__host__ __device__ inline SoloSmem solo_smem(int n, int m, int n_mtask, bool pairs, uint32_t list_bytes) {
    SoloSmem s;
    s.t = 0;
    s.q = pad16(8u * (uint32_t)(n + 1));
    s.x = pad16(s.q + (pairs ? 8u : 4u) * (uint32_t)(m + 1));
    s.m = s.x + pad16(4u * (uint32_t)n);
    s.v = s.m + pad16(4u * (uint32_t)n);
    s.leaf = s.v + pad16(4u * (uint32_t)n);
    s.best = s.leaf + pad16(4u * (uint32_t)n_mtask);
    s.lists = s.best + pad16((uint32_t)n);
    s.total = s.lists + list_bytes;
    return s;
}

// Sum over the warp; every lane receives it.
__device__ __forceinline__ unsigned long long warp_sum_u64(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// The pair {value of the literal x, value of the literal not x} of a
// variable: +-tanh(x) with the sign bit set exactly where the literal is
// false under x > 0 (x = +-0 and NaN are false), so that a clause is unsat
// exactly when the sign bits of all its literals' values are set.
__device__ __forceinline__ float2 literal_pair(float x) {
    const uint32_t t = __float_as_uint(tanh_fixed(x)) | (x > 0.0f ? 0u : 0x80000000u);
    return make_float2(__uint_as_float(t), __uint_as_float(t ^ 0x80000000u));
}

}  // namespace

// KIND 0: every clause has 3 literals; 1: at most 32; 2: any length.
// LS: the lists are copied to shared memory.  QP: w*f is held as {q, -q}, so
// an occurrence word addresses its signed value; otherwise the signs are in
// a 32-bit word per leaf task.  WT: clause weights (else all 1).
template <int KIND, bool LS, bool QP, bool WT>
__global__ void __launch_bounds__(kSoloMaxThreads, 1)
    k_solo_steps(SoloDev V, int n, int m, int B, DevState S, DevStep D, int n_steps, int final_eval) {
    extern __shared__ __align__(16) unsigned char solo_smem_raw[];
    __shared__ unsigned long long s_part[32];
    __shared__ float s_at[2][kSoloRing], s_rt[2][kSoloRing];
    __shared__ double s_run[2], s_fin[2];  // running Adam products; those of the call's end
    __shared__ long long s_bstep;  // step of the best cost
    __shared__ int s_improved, s_last;

    const SoloSmem L = solo_smem(n, m, V.n_mtask, QP, 0);
    float2 *st = reinterpret_cast<float2 *>(solo_smem_raw);  // [n+1] literal values
    const float *stf = reinterpret_cast<const float *>(solo_smem_raw);
    float *sq = reinterpret_cast<float *>(solo_smem_raw + L.q);  // [m+1] w*f (or pairs)
    float *sx = reinterpret_cast<float *>(solo_smem_raw + L.x);
    float *smo = reinterpret_cast<float *>(solo_smem_raw + L.m);
    float *sve = reinterpret_cast<float *>(solo_smem_raw + L.v);
    float *sleaf = reinterpret_cast<float *>(solo_smem_raw + L.leaf);
    uint8_t *sbest = solo_smem_raw + L.best;

    const int b = blockIdx.x;
    const int T = (int)blockDim.x - 32;  // work threads; the last warp makes the Adam scalars
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nwarps = T >> 5;
    const bool worker = tid < T;
    StepScalars *sc = D.sc;
    // every cost fits 32 bits
    const bool narrow = !WT || sc->wsum < (1LL << 32);
    // the loss normaliser where it is not the unsat weight (0)
    const float fixed_den = sc->loss_norm == 1 ? 1.0f : sc->loss_norm == 2 ? (float)sc->wsum : 0.0f;
    const AdamView A0 = adam_view(sc);

    // lists to shared memory
    const unsigned char *lists = V.lists;
    if constexpr (LS) {
        const uint4 *src = reinterpret_cast<const uint4 *>(V.lists);
        uint4 *dst = reinterpret_cast<uint4 *>(solo_smem_raw + L.lists);
        for (uint32_t k = tid; k < V.list_bytes / 16; k += blockDim.x) dst[k] = __ldg(src + k);
        lists = solo_smem_raw + L.lists;
    }
    const uint2 *lit = reinterpret_cast<const uint2 *>(lists + V.off_lit) + lane;
    const int *lit_base = reinterpret_cast<const int *>(lists + V.off_lit_base);
    const uint2 *occ = reinterpret_cast<const uint2 *>(lists + V.off_occ) + lane;
    const int *occ_base = reinterpret_cast<const int *>(lists + V.off_occ_base);
    const uint32_t *sgn = reinterpret_cast<const uint32_t *>(lists + V.off_sgn);
    const int *mbeg = reinterpret_cast<const int *>(lists + V.off_mbeg);
    const int *perm = V.perm;
    auto ld2 = [](const uint2 *p) { return LS ? *p : __ldg(p); };
    auto ld1 = [](const int *p) { return LS ? *p : __ldg(p); };

    for (int i = tid; i < n; i += blockDim.x) {
        const int64_t q0 = (int64_t)__ldg(perm + i) * B + b;
        const float xv = S.x[q0];
        sx[i] = xv;
        st[i] = literal_pair(xv);  // tanh of x as the per-pass kernels hold it
        if (n_steps > 0) {
            smo[i] = S.mom[q0];
            sve[i] = S.vel[q0];
        }
    }
    if (tid == 0) {
        // the dummy variable (false, adds nothing) and the dummy clause
        st[n] = make_float2(-0.0f, -0.0f);
        sq[QP ? 2 * m : m] = 0.0f;
        if (QP) sq[2 * m + 1] = 0.0f;
    }
    long long best = D.best[b];
    if (tid == 0) {
        s_bstep = D.best_step[b];
        s_improved = 0;
    }

    // the scalar warp: Adam scalars of kSoloRing steps at a time, one chunk
    // ahead; the products run in step order (in double, as the clause pass's
    // last block computes them), the divisions and roots one step a lane
    auto make_chunk = [&](int first, int buf) {
        const double b1 = sc->beta1, b2 = sc->beta2;
        double p1 = s_run[0], p2 = s_run[1], q1 = p1, q2 = p2;
#pragma unroll 1
        for (int l = 0; l < kSoloRing; ++l) {
            p1 = p1 * b1;
            p2 = p2 * b2;
            if (l == lane) {
                q1 = p1;
                q2 = p2;
            }
            if (first + l + 1 == n_steps && lane == 0) {
                s_fin[0] = p1;
                s_fin[1] = p2;
            }
        }
        s_at[buf][lane] = (float)(sc->lr / (1.0 - q1));
        s_rt[buf][lane] = (float)(1.0 / sqrt(1.0 - q2));
        __syncwarp();
        if (lane == 0) {
            s_run[0] = p1;
            s_run[1] = p2;
        }
        __syncwarp();
    };
    int made = 0;  // steps whose scalars the scalar warp has made
    if (!worker) {
        if (lane == 0) {
            s_run[0] = sc->p1;
            s_run[1] = sc->p2;
        }
        __syncwarp();
        if (n_steps > 0) {
            make_chunk(0, 0);
            made = kSoloRing;
        }
    }
    __syncthreads();

    const int nslice = (m + 31) >> 5;
    const int n_task = V.n_mtask + V.n_single;
    const int ntslice = (n_task + 31) >> 5;
    float lpart = 0.0f;  // of the loss of the last updated x, and its normaliser
    double lden = 0.0;
    int imp = 0;
    float cs = 0.0f;
    long long cost = 0;

    // clause pass: f, exact unsat test (um: the and of the literals' values,
    // negative where all are false), w*f (+0 where satisfied)
    auto clause_pass = [&](bool want_loss) {
        unsigned cacc = 0;           // unsat clauses of this thread
        unsigned long long wacc = 0;  // their weight
        auto finish = [&](int s, float f, int um) {
            const bool unsat = um < 0;
            float q = f;
            if constexpr (WT) {
                const long long wj = __ldg(V.w + s);
                q = (float)wj * f;
                if (unsat) wacc += (unsigned long long)wj;
            } else {
                cacc += (unsigned)um >> 31;
            }
            if (want_loss && unsat) lpart += q * f;
            // f of an unsat clause is a sum of values <= 0; a NaN in it reads
            // as satisfied in the gradient
            q = unsat && f <= 0.0f ? q : 0.0f;
            if constexpr (QP) reinterpret_cast<float2 *>(sq)[s] = make_float2(q, -q);
            else sq[s] = q;
        };
        if constexpr (KIND == 0) {
            // full slices two at a time, the last ones with a bound check
            auto lits = [&](uint2 wd, float (&u)[3]) {
                u[0] = stf[wd.x & 0xffffu];
                u[1] = stf[wd.x >> 16];
                u[2] = stf[wd.y & 0xffffu];
            };
            const int nfull = m >> 5;
            int sl = warp;
            uint2 wa = make_uint2(0u, 0u), wb = wa;  // one pair of slices ahead
            if (sl < nslice) wa = ld2(lit + sl * 32);
            if (sl + nwarps < nslice) wb = ld2(lit + (sl + nwarps) * 32);
#pragma unroll 1
            for (; sl + nwarps < nfull; sl += 2 * nwarps) {
                float ua[3], ub[3];
                lits(wa, ua);
                lits(wb, ub);
                if (sl + 2 * nwarps < nslice) wa = ld2(lit + (sl + 2 * nwarps) * 32);
                if (sl + 3 * nwarps < nslice) wb = ld2(lit + (sl + 3 * nwarps) * 32);
                const float2 f = add2(add2(make_float2(ua[0], ub[0]), make_float2(ua[1], ub[1])),
                                      make_float2(ua[2], ub[2]));
                finish(sl * 32 + lane, f.x, __float_as_int(ua[0]) & __float_as_int(ua[1]) & __float_as_int(ua[2]));
                finish((sl + nwarps) * 32 + lane, f.y,
                       __float_as_int(ub[0]) & __float_as_int(ub[1]) & __float_as_int(ub[2]));
            }
            // at most two slices left
#pragma unroll 1
            for (; sl < nslice; sl += nwarps) {
                const int s = sl * 32 + lane;
                float u[3];
                lits(wa, u);
                wa = wb;
                if (s < m) finish(s, (u[0] + u[1]) + u[2], __float_as_int(u[0]) & __float_as_int(u[1]) & __float_as_int(u[2]));
            }
        } else {
#pragma unroll 1
            for (int sl = warp; sl < nslice; sl += nwarps) {
                const int g0 = ld1(lit_base + sl), g1 = ld1(lit_base + sl + 1);
                float f = -0.0f;
                int um = -1;
                LeafCounter<kClauseLevels> lc;
                if constexpr (KIND == 2) lc.init();
                uint2 wd = ld2(lit + g0 * 32);  // every slice has a row
#pragma unroll 1
                for (int g = g0; g < g1; ++g) {
                    if constexpr (KIND == 2) {
                        if (g > g0 && ((g - g0) & 7) == 0) {
                            lc.push(f);
                            f = -0.0f;
                        }
                    }
                    const float u0 = stf[wd.x & 0xffffu], u1 = stf[wd.x >> 16];
                    const float u2 = stf[wd.y & 0xffffu], u3 = stf[wd.y >> 16];
                    if (g + 1 < g1) wd = ld2(lit + (g + 1) * 32);
                    f = (((f + u0) + u1) + u2) + u3;
                    um &= __float_as_int(u0) & __float_as_int(u1);
                    um &= __float_as_int(u2) & __float_as_int(u3);
                }
                if constexpr (KIND == 2) {
                    if (lc.cnt) {
                        lc.push(f);
                        f = lc.finish();
                    }
                }
                const int s = sl * 32 + lane;
                if (s < m) finish(s, f, um);
            }
        }
        // integer sums: any order is exact
        if constexpr (!WT) {
            const unsigned r = __reduce_add_sync(0xffffffffu, cacc);
            if (lane == 0) s_part[warp] = r;
        } else if (narrow) {
            const unsigned r = __reduce_add_sync(0xffffffffu, (unsigned)wacc);
            if (lane == 0) s_part[warp] = r;
        } else {
            const unsigned long long r = warp_sum_u64(wacc);
            if (lane == 0) s_part[warp] = r;
        }
    };
    // after the barrier: the block's sum in every thread, then the
    // per-restart scalars as the clause pass's last block computes them
    auto clause_scalars = [&](int step) {
        const unsigned long long part = lane < nwarps ? s_part[lane] : 0ull;
        float costf;
        if (narrow) {
            const unsigned c = __reduce_add_sync(0xffffffffu, (unsigned)part);
            cost = (long long)c;
            costf = (float)c;
        } else {
            cost = (long long)warp_sum_u64(part);
            costf = (float)cost;
        }
        imp = cost < best;
        if (imp) {
            best = cost;
            if (tid == 0) {
                s_bstep = sc->steps_done + step;
                s_improved = 1;
            }
        }
        const float den = fixed_den > 0.0f ? fixed_den : costf;
        cs = cost > 0 ? 2.0f / den : 0.0f;
        if (step == n_steps - 1 && cost > 0)
            lden = sc->loss_norm == 1 ? 1.0 : (double)(sc->loss_norm == 2 ? sc->wsum : cost);
    };
    auto update = [&](int i, float sum, float a_t, float r_t) {
        AdamView A = A0;
        A.a_t = a_t;
        A.r_t = r_t;
        const float tv = stf[2 * i];
        const float gr = (sum + 0.0f) * fmaf(-tv, tv, 1.0f);
        float xv = sx[i], mv = smo[i], vv = sve[i];
        if (imp) sbest[i] = xv > 0.0f;
        xv = adam_update(A, xv, mv, vv, gr);
        sx[i] = xv;
        smo[i] = mv;
        sve[i] = vv;
        st[i] = literal_pair(xv);
    };

    bool capture = false;  // the last evaluation's improvement is still to be captured
    const int n_eval = n_steps + final_eval;
#pragma unroll 1
    for (int step = 0; step < n_eval; ++step) {
        if (worker) {
            clause_pass(step == n_steps - 1);
        } else if ((step & (kSoloRing - 1)) == 0 && made < n_steps) {
            make_chunk(made, (made / kSoloRing) & 1);
            made += kSoloRing;
        }
        __syncthreads();
        clause_scalars(step);
        if (cost == 0 || step == n_steps) {
            // solved (the state stays as it is from here on), or the
            // evaluation of the final x
            capture = imp;
            if (step < n_steps && final_eval) imp = 0;
            break;
        }
        const float a_t = s_at[(step / kSoloRing) & 1][step & (kSoloRing - 1)];
        const float r_t = s_rt[(step / kSoloRing) & 1][step & (kSoloRing - 1)];
        if (worker) {
            const float2 cc = make_float2(cs, cs);
#pragma unroll 1
            for (int sl = warp; sl < ntslice; sl += nwarps) {
                const int k = sl * 32 + lane;
                const int g0 = ld1(occ_base + sl), g1 = ld1(occ_base + sl + 1);
                uint32_t bits = 0u;
                if constexpr (!QP) bits = k < n_task ? __ldg(sgn + k) : 0u;
                float sum = 0.0f;
                uint2 wd = ld2(occ + g0 * 32);  // every slice has a row
#pragma unroll 1
                for (int g = g0; g < g1; ++g) {
                    const float q0 = sq[wd.x & 0xffffu], q1 = sq[wd.x >> 16];
                    const float q2 = sq[wd.y & 0xffffu], q3 = sq[wd.y >> 16];
                    if (g + 1 < g1) wd = ld2(occ + (g + 1) * 32);
                    float2 ca = cc, cb = cc;
                    if constexpr (!QP) {
                        const uint32_t c = __float_as_uint(cs);
                        ca = make_float2(__uint_as_float(c ^ ((bits << 31) & 0x80000000u)),
                                         __uint_as_float(c ^ ((bits << 30) & 0x80000000u)));
                        cb = make_float2(__uint_as_float(c ^ ((bits << 29) & 0x80000000u)),
                                         __uint_as_float(c ^ ((bits << 28) & 0x80000000u)));
                        bits >>= 4;
                    }
                    const float2 a = mul2(make_float2(q0, q1), ca), e = mul2(make_float2(q2, q3), cb);
                    sum = (((sum + a.x) + a.y) + e.x) + e.y;
                }
                if (k < V.n_mtask) sleaf[k] = sum;
                else if (k < n_task) update(k - V.n_mtask, sum, a_t, r_t);
            }
        }
        if (V.n_mtask > 0) {  // variables of several leaves: the dyadic tree over their sums
            __syncthreads();
            if (worker) {
                for (int h = warp; h < V.n_wide; h += nwarps) {
                    // lane l: the aligned block of bs leaves from bs * l
                    const int k0 = mbeg[h], K = mbeg[h + 1] - k0;
                    int bs = 1;
                    while (bs * 32 < K) bs <<= 1;
                    LeafCounter<6> lc;
                    lc.init();
                    for (int r = lane * bs; r < min(K, lane * bs + bs); ++r) lc.push(sleaf[k0 + r]);
                    const float sum = warp_dyadic(lc.finish(), (K + bs - 1) / bs, lane);
                    if (lane == 0) update(V.n_single + h, sum, a_t, r_t);
                }
                for (int h = V.n_wide + tid; h < V.n_multi; h += T) {
                    const int k0 = mbeg[h], k1 = mbeg[h + 1];
                    LeafCounter<4> lc;
                    lc.init();
                    for (int r = k0; r < k1; ++r) lc.push(sleaf[r]);
                    update(V.n_single + h, lc.finish(), a_t, r_t);
                }
            }
        }
        __syncthreads();
    }
    // the loss of the last updated x (the terms of the last step's clause pass)
    if (n_steps > 0) {
        double lsum = lpart;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
        __syncthreads();
        if (worker && lane == 0) s_part[warp] = (unsigned long long)__double_as_longlong(lsum);
        __syncthreads();
        if (warp == 0) {
            lsum = lane < nwarps ? __longlong_as_double((long long)s_part[lane]) : 0.0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
            if (lane == 0) D.loss[b] = lden > 0.0 ? (float)(lsum / lden) : 0.0f;
        }
    }
    if (capture)
        for (int i = tid; i < n; i += blockDim.x) sbest[i] = sx[i] > 0.0f;
    // read before the barrier that every thread passes ahead of the block's
    // count: the block that counts last writes the step scalars
    const long long steps_end = sc->steps_done + n_steps;
    __syncthreads();
    const bool improved = s_improved != 0;
    float *t_out = (steps_end & 1) ? S.t1 : S.t0;
    for (int i = tid; i < n; i += blockDim.x) {
        const int64_t q0 = (int64_t)__ldg(perm + i) * B + b;
        if (n_steps > 0) {
            const float xv = sx[i];
            S.x[q0] = xv;
            S.mom[q0] = smo[i];
            S.vel[q0] = sve[i];
            t_out[q0] = copysignf(stf[2 * i], xv);  // the sign tanh itself gives +-0
        }
        if (improved) S.bestx[q0] = sbest[i];
    }
    if (!worker && lane == 0 && made < n_steps) {  // a solved restart: the products of the steps left
        double p1 = s_run[0], p2 = s_run[1];
        for (; made < n_steps; ++made) {
            p1 = p1 * sc->beta1;
            p2 = p2 * sc->beta2;
        }
        s_fin[0] = p1;
        s_fin[1] = p2;
    }
    if (tid == 0) {
        D.cost[b] = cost;
        D.best[b] = best;
        D.best_step[b] = s_bstep;
        D.improved[b] = imp;
        D.cscale[b] = cs;
        __threadfence();
        // the last block to finish leaves the step scalars of the call's end;
        // every thread of every block has read steps_done by then (its read
        // lies before its block's last barrier, the count after it)
        s_last = atomicAdd(&sc->counter, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last || tid >= 32) return;
    __threadfence();
    unsigned long long tot = 0;
    for (int k = lane; k < B; k += 32) tot += (unsigned long long)__ldcg(D.cost + k);
    tot = warp_sum_u64(tot);
    if (lane == 0) {
        sc->counter = 0;
        sc->dense = (double)tot * 16.0 > (double)sc->wsum * (double)B;
        if (n_steps > 0) {
            sc->p1 = s_fin[0];
            sc->p2 = s_fin[1];
            sc->steps_done = steps_end;
        }
    }
}

// --------------------------------------------------------------- host side

namespace {

struct SoloShape {
    int64_t lit_rows = 0, occ_rows = 0;  // 32-lane rows of four words
    int n_single = 0, n_multi = 0, n_wide = 0, n_mtask = 0;
};

}  // namespace

bool solo_fits(int32_t n, int64_t m, int32_t max_deg) {
    // 16-bit words: var << 1 | neg with the dummy variable n, slots up to the
    // dummy clause m
    return n <= 32766 && m <= 65534 && max_deg <= 32 * 1024 &&
           solo_smem(n, (int)m, 0, false, 0).total <= kSoloSmemMax;
}

bool build_solo(int32_t n, int64_t m, int32_t kfix, int32_t max_len, int32_t max_deg, const HostCnf &hc,
                const int64_t *w, const std::function<bool(const SoloDev &)> &pays, SoloHost &out) {
    if (!solo_fits(n, m, max_deg)) return false;
    SoloDev &V = out.dev;
    V = SoloDev{};
    const int32_t *coff = hc.coff.data(), *lit = hc.lit.data(), *voff = hc.voff.data();

    // variables: one leaf first (longest first), then several leaves (those a
    // warp combines first)
    auto leaves = [&](int32_t i) { return (voff[i + 1] - voff[i] + 31) / 32; };
    std::vector<int32_t> perm((size_t)n);
    SoloShape sh;
    {
        int32_t cnt[10] = {0};
        for (int32_t i = 0; i < n; ++i) {
            const int32_t d = voff[i + 1] - voff[i];
            if (d <= 32) ++cnt[8 - (d + 3) / 4];
            else {
                ++sh.n_multi;
                sh.n_mtask += leaves(i);
                if (leaves(i) > kNarrowLeaves) ++sh.n_wide;
            }
        }
        sh.n_single = n - sh.n_multi;
        int32_t at[10], wide = sh.n_single, narrow = sh.n_single + sh.n_wide;
        at[0] = 0;
        for (int k = 0; k < 9; ++k) at[k + 1] = at[k] + cnt[k];
        for (int32_t i = 0; i < n; ++i) {
            const int32_t d = voff[i + 1] - voff[i];
            const int32_t id = d <= 32 ? at[8 - (d + 3) / 4]++ : leaves(i) > kNarrowLeaves ? wide++ : narrow++;
            perm[(size_t)id] = i;
        }
    }
    if (solo_smem(n, (int)m, sh.n_mtask, false, 0).total > kSoloSmemMax) return false;

    // clauses: slots by falling length (all equal: clause order)
    I32Buf slot;  // clause -> slot
    const int64_t nsl = (m + 31) / 32;
    std::vector<int32_t> lbase((size_t)nsl + 1, 0);
    if (kfix == 0 && m > 0) {
        slot.alloc((size_t)m);
        const int32_t top = (max_len + 3) / 4;  // bucket k: clauses of top - k rows
        std::vector<int32_t> at((size_t)top + 2, 0);
        for (int64_t j = 0; j < m; ++j) ++at[(size_t)(top - (hc.clen[(size_t)j] + 3) / 4) + 1];
        for (int32_t k = 0; k <= top; ++k) at[(size_t)k + 1] += at[(size_t)k];
        int32_t k = 0;
        for (int64_t s = 0; s < nsl; ++s) {  // a slice's first clause is its longest
            while (at[(size_t)k + 1] <= 32 * s) ++k;
            lbase[(size_t)s + 1] = lbase[(size_t)s] + std::max(1, top - k);
        }
        for (int64_t j = 0; j < m; ++j)
            slot[(size_t)j] = at[(size_t)(top - (hc.clen[(size_t)j] + 3) / 4)]++;
    } else {
        for (int64_t s = 0; s < nsl; ++s) lbase[(size_t)s + 1] = lbase[(size_t)s] + std::max(1, (kfix + 3) / 4);
    }
    V.kind = kfix == 3 ? 0 : max_len <= 32 ? 1 : 2;
    // signed pairs of w*f where they fit: an occurrence word is then slot <<
    // 1 | neg, else the slot, with the signs apart (m + 1 pairs fit only for
    // m < 32767)
    V.pairs = V.kind < 2 && solo_smem(n, (int)m, sh.n_mtask, true, 0).total <= kSoloSmemMax;
    sh.lit_rows = lbase[(size_t)nsl];

    // leaf tasks: those of the variables of several leaves in (variable,
    // leaf) order, then the variables of one leaf
    const int32_t n_task = sh.n_mtask + sh.n_single;
    std::vector<int32_t> tfirst((size_t)n);  // internal id -> first task
    std::vector<uint8_t> tlen((size_t)n_task);
    std::vector<int32_t> mbeg((size_t)sh.n_multi + 1, 0);
    {
        int32_t k = 0;
        for (int32_t h = 0; h < sh.n_multi; ++h) {
            const int32_t i = perm[(size_t)(sh.n_single + h)];
            const int32_t d = voff[i + 1] - voff[i];
            tfirst[(size_t)(sh.n_single + h)] = k;
            mbeg[(size_t)h] = k;
            for (int32_t r = 0; r < d; r += 32) tlen[(size_t)k++] = (uint8_t)std::min(32, d - r);
        }
        mbeg[(size_t)sh.n_multi] = k;
        for (int32_t id = 0; id < sh.n_single; ++id) {
            const int32_t i = perm[(size_t)id];
            tfirst[(size_t)id] = k;
            tlen[(size_t)k++] = (uint8_t)(voff[i + 1] - voff[i]);
        }
    }
    const int64_t ntsl = (n_task + 31) / 32;
    std::vector<int32_t> obase((size_t)ntsl + 1, 0);
    for (int64_t s = 0; s < ntsl; ++s) {
        int32_t mx = 0;
        for (int64_t k = 32 * s; k < std::min<int64_t>(n_task, 32 * s + 32); ++k) mx = std::max<int32_t>(mx, tlen[(size_t)k]);
        obase[(size_t)s + 1] = obase[(size_t)s] + std::max(1, (mx + 3) / 4);
    }
    sh.occ_rows = obase[(size_t)ntsl];
    V.n_single = sh.n_single;
    V.n_multi = sh.n_multi;
    V.n_wide = sh.n_wide;
    V.n_mtask = sh.n_mtask;
    V.rows = (int)(sh.lit_rows + sh.occ_rows);
    if (!pays(V)) return false;

    // one array: literal rows, occurrence rows, then the small tables
    uint32_t at = 0;
    auto place = [&](uint32_t &off, size_t bytes) {
        off = at;
        at = pad16(at + (uint32_t)bytes);
    };
    place(V.off_lit, (size_t)sh.lit_rows * 256);
    place(V.off_occ, (size_t)sh.occ_rows * 256);
    place(V.off_lit_base, sizeof(int32_t) * lbase.size());
    place(V.off_occ_base, sizeof(int32_t) * obase.size());
    place(V.off_sgn, sizeof(uint32_t) * (size_t)n_task);
    place(V.off_mbeg, sizeof(int32_t) * mbeg.size());
    V.list_bytes = at;
    uint32_t perm_at = 0, w_at = 0;
    place(perm_at, sizeof(int32_t) * (size_t)n);
    if (w && slot.size() > 0) place(w_at, sizeof(int64_t) * (size_t)m);
    out.perm_at = perm_at;
    out.w_at = w_at;
    out.bytes = at;
    out.lists.reset(new unsigned char[at]);
    // every byte but the gaps between the tables is written below
    uint16_t *lw = reinterpret_cast<uint16_t *>(out.lists.get() + V.off_lit);
    uint16_t *ow = reinterpret_cast<uint16_t *>(out.lists.get() + V.off_occ);
    uint32_t *sg = reinterpret_cast<uint32_t *>(out.lists.get() + V.off_sgn);
    std::copy(lbase.begin(), lbase.end(), reinterpret_cast<int32_t *>(out.lists.get() + V.off_lit_base));
    std::copy(obase.begin(), obase.end(), reinterpret_cast<int32_t *>(out.lists.get() + V.off_occ_base));
    std::copy(mbeg.begin(), mbeg.end(), reinterpret_cast<int32_t *>(out.lists.get() + V.off_mbeg));
    // the words of the clauses, by a thread of their own where they are many
    // (a thread costs about 25 us, the words 1 to 2 ns each)
    constexpr int64_t kApart = 1 << 15;
    std::vector<int32_t> id_of((size_t)n);
    for (int32_t id = 0; id < n; ++id) id_of[(size_t)perm[(size_t)id]] = id;
    auto slot_at = [&](int64_t j) { return (uint32_t)(kfix > 0 ? j : slot[(size_t)j]); };
    auto lit_words = [&] {
        std::fill(lw, lw + sh.lit_rows * 128, (uint16_t)(n << 1));
        for (int64_t j = 0; j < m; ++j) {
            const uint32_t s = slot_at(j);
            uint16_t *l0 = lw + ((size_t)lbase[s >> 5] * 32 + (s & 31u)) * 4;
            const int32_t *c = lit + coff[j];
            const int32_t len = coff[j + 1] - coff[j];
            for (int32_t r = 0; r < len; ++r)
                l0[(r >> 2) * 128 + (r & 3)] = (uint16_t)((id_of[(size_t)(c[r] >> 1)] << 1) | (c[r] & 1));
        }
    };
    std::future<void> apart;
    if (hc.nnz >= kApart) {
        try {
            apart = std::async(std::launch::async, lit_words);
        } catch (const std::system_error &) {  // no more threads
        }
    }
    if (!apart.valid()) lit_words();
    // per variable: where its current leaf's words go, the leaf task and the
    // occurrences and signs placed in it
    struct Fill {
        uint32_t at, task, cnt, sgn;
    };
    std::vector<Fill> fill((size_t)n);
    auto leaf_at = [&](uint32_t k) { return ((uint32_t)obase[k >> 5] * 32u + (k & 31u)) * 4u; };
    for (int32_t id = 0; id < n; ++id) {
        const uint32_t k = (uint32_t)tfirst[(size_t)id];
        fill[(size_t)perm[(size_t)id]] = Fill{leaf_at(k), k, 0u, 0u};
    }
    const uint32_t pairs = V.pairs ? 1u : 0u;
    std::fill(ow, ow + sh.occ_rows * 128, (uint16_t)(V.pairs ? 2 * m : m));
    for (int64_t j = 0; j < m; ++j) {
        const uint32_t s = slot_at(j);
        for (int32_t p = coff[j]; p < coff[j + 1]; ++p) {
            const uint32_t neg = (uint32_t)lit[p] & 1u;
            Fill &F = fill[(size_t)(lit[p] >> 1)];
            if (F.cnt == 32u) {
                sg[F.task] = F.sgn;
                ++F.task;
                F.at = leaf_at(F.task);
                F.cnt = F.sgn = 0u;
            }
            ow[F.at + (F.cnt >> 2) * 128u + (F.cnt & 3u)] = (uint16_t)((s << pairs) | (neg & pairs));
            F.sgn |= neg << F.cnt;
            ++F.cnt;
        }
    }
    for (const Fill &F : fill) sg[F.task] = F.sgn;
    std::copy(perm.begin(), perm.end(), reinterpret_cast<int32_t *>(out.lists.get() + perm_at));
    if (w_at) {
        int64_t *sw = reinterpret_cast<int64_t *>(out.lists.get() + w_at);
        for (int64_t j = 0; j < m; ++j) sw[slot[(size_t)j]] = w[j];
    }
    return true;
}

// Shape of a launch: blocks per SM, where the lists lie, and work threads.
// Blocks beyond one wave share SMs (their barriers and latencies overlap)
// where shared memory allows it; the lists go to shared memory where that
// does not cost a block.  A block of up to 160 slices runs on 512 threads
// (n=301: 1.9 us a step, 2.0 with 992; n=1000: 3.7 / 4.0), a larger one on
// 992 (n=2500: 8.0, 9.5 with 512; n=5000: 14.5 / 17.7); two blocks of an SM
// on 480 each (n=301, B=256: 2.6, 4.1 in two waves of 992).
struct SoloShapeAt {
    bool lists_in_smem;
    int threads;
    size_t smem;
};

static SoloShapeAt solo_shape(const SoloDev &V, const DevInst &I) {
    constexpr size_t kSm = 227 * 1024, kStatic = 2048;  // of one SM; static and reserved, per block
    const size_t base = solo_smem(I.n, I.m, V.n_mtask, V.pairs, 0).total;
    const size_t with = base + V.list_bytes;
    int w = std::min(4, (I.B + V.sms - 1) / V.sms);
    SoloShapeAt r{};
    for (; w >= 1; --w) {
        r.lists_in_smem = V.pairs && with <= kSoloSmemMax && w * (with + kStatic) <= kSm;
        if (r.lists_in_smem || w == 1 || w * (base + kStatic) <= kSm) break;
    }
    if (w == 1) r.lists_in_smem = V.pairs && with <= kSoloSmemMax;
    r.smem = r.lists_in_smem ? with : base;
    const int items = std::max(I.m, V.n_mtask + V.n_single);
    const int slices = (items + 31) / 32;
    // 64 registers a thread: 1024 threads fill an SM's register file
    const int most = w > 1 ? kSoloMaxThreads / w / 32 * 32 - 32 : slices <= 160 ? 512 : kSoloMaxThreads - 32;
    r.threads = std::min(most, std::max(64, 32 * slices)) + 32;
    return r;
}

template <int KIND, bool LS, bool QP, bool WT>
static cudaError_t launch_solo_k(const SoloDev &V, const DevInst &I, const DevState &S, const DevStep &D,
                                 int n_steps, int final_eval, const SoloShapeAt &sh, cudaStream_t st) {
    const cudaError_t e = cudaFuncSetAttribute(k_solo_steps<KIND, LS, QP, WT>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSoloSmemMax);
    if (e) return e;
    k_solo_steps<KIND, LS, QP, WT><<<I.B, sh.threads, sh.smem, st>>>(V, I.n, I.m, I.B, S, D, n_steps, final_eval);
    return cudaGetLastError();
}

template <int KIND, bool WT>
static cudaError_t launch_solo_kw(const SoloDev &V, const DevInst &I, const DevState &S, const DevStep &D,
                                  int n_steps, int final_eval, cudaStream_t st) {
    const SoloShapeAt sh = solo_shape(V, I);
    if constexpr (KIND < 2) {
        if (sh.lists_in_smem) return launch_solo_k<KIND, true, true, WT>(V, I, S, D, n_steps, final_eval, sh, st);
        if (V.pairs) return launch_solo_k<KIND, false, true, WT>(V, I, S, D, n_steps, final_eval, sh, st);
    }
    return launch_solo_k<KIND, false, false, WT>(V, I, S, D, n_steps, final_eval, sh, st);
}

cudaError_t launch_solo_steps(const SoloDev &V, const DevInst &I, const DevState &S, const DevStep &D,
                              int n_steps, bool final_eval, cudaStream_t st) {
    if (n_steps <= 0 && !final_eval) return cudaSuccess;
    const int fe = final_eval ? 1 : 0;
    switch (V.kind * 2 + (V.w ? 1 : 0)) {
        case 0: return launch_solo_kw<0, false>(V, I, S, D, n_steps, fe, st);
        case 1: return launch_solo_kw<0, true>(V, I, S, D, n_steps, fe, st);
        case 2: return launch_solo_kw<1, false>(V, I, S, D, n_steps, fe, st);
        case 3: return launch_solo_kw<1, true>(V, I, S, D, n_steps, fe, st);
        case 4: return launch_solo_kw<2, false>(V, I, S, D, n_steps, fe, st);
        default: return launch_solo_kw<2, true>(V, I, S, D, n_steps, fe, st);
    }
}

// Whether `steps` steps are taken faster by this kernel than by the per-pass
// kernels, from what both measured on one GB300 (microseconds a step).  A
// block takes 1 + 0.0115 per list row (n=301 1.9, n=5000 14.5, ordering
// principle on 31 elements 18.9), 1.4 times that with variables a warp
// combines (weighted Zipf n=3000 20.6) and 1.6 with clauses of more than 32
// literals (PHP(40) 30), one wave of SMs at a time (n=5000, B=256: 29), and
// once a call loads its lists and gathers and scatters its column of the
// state (8 + 7e-5 per variable and restart: n=5000, B=256 90).  The two passes take 10 (dependent latency;
// n=5000, B=1: 10.7), 1.5 per million literal evaluations (n=5000, B=256:
// 36), for clauses that are not all of three literals 2 + 0.15 per literal of
// the longest, or 0.3 with four or more restarts (ordering principle, B=8:
// 20.5), and then 12 for a launch of heavy variables (Zipf n=3000, B=4: 37).
// An evaluation alone (no steps) is half a step here, reads one of the three
// state arrays and writes none, and the two passes may cost 1.1 times their
// estimate, which counts none of the host's launches.  Whole calls, passes /
// here: 5-SAT n=1200, B=16 35.7 / 46.6 us, weighted Zipf n=3000, B=1 38.0 /
// 46.2, 4-SAT n=800, B=1024 92.8 / 76.5, 3-SAT n=1000, B=16 37.2 / 35.1.
// slack: factor allowed to this kernel.
bool solo_pays(const SoloDev &V, const DevInst &I, int64_t nnz, int max_len, int64_t steps, double slack) {
    const double waves = (I.B + V.sms - 1) / V.sms;
    const double solo = 1.0 + 0.0115 * V.rows * waves * (V.n_wide > 0 ? 1.4 : 1.0) * (V.kind == 2 ? 1.6 : 1.0);
    const double passes = 10.0 + 1.5e-6 * (double)nnz * I.B +
                          (I.kfix == 3 ? 0.0 : 2.0 + (I.B < 4 ? 0.15 : 0.3) * max_len) +
                          (I.n_heavy > 0 && I.B >= 4 ? 12.0 : 0.0);
    if (steps == 0) return 0.5 * solo + 8.0 + 2e-5 * (double)I.n * I.B <= 1.1 * slack * passes;
    return (double)steps * solo + 8.0 + 7e-5 * (double)I.n * I.B <= slack * (double)steps * passes;
}

}  // namespace msat

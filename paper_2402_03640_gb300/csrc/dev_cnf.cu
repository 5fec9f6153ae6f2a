// Device side of msat_create for large instances whose clauses are already
// canonical: the checks, the packed clause list, the transposed CSR and the
// grouped row order, from the caller's arrays as they are.
//
// The arrays are those the host path builds (host_cnf.cu), element for
// element.  The host path needs stable passes because its threads scatter in
// clause order; here atomics place the occurrences of a variable (and the
// clauses of a row group) in any order, and a rank sort of each short list by
// clause index restores the order: clause indices are distinct within a list,
// so the sorted list is unique.  A list longer than the sorts' reach, and
// anything that is not a clean CNF, goes to the host path.
//
// What bounds it: the upload of the caller's arrays (86 MB at n=1e6,
// m=4.3e6) and one host pass over the occurrence offsets (the partition into
// light blocks); the kernels are random 4-byte atomics and gathers, about 13
// million a pass, 0.9 ms in all (k_row_sort 0.21, k_occ_sort 0.19, k_occ_scatter
// 0.16 ms).  3-SAT n=1e6, m=4.3e6, B=1: msat_create 32 -> 5.3 ms.

#include <cuda_runtime.h>
#include <limits.h>
#include <stdint.h>

#include <algorithm>
#include <vector>

#include "dev_cnf.cuh"
#include "msat_internal.cuh"

namespace msat {

namespace {

constexpr int kMaxCleanLen = 32;     // literals of a clause compared pairwise
constexpr int kMaxSortDeg = 1024;    // occurrences a warp sorts
constexpr int kMaxGroup = 4096;      // clauses of a row group a block sorts
constexpr int kScanItems = 16;       // items a thread scans
constexpr int kScanBlock = kThreads * kScanItems;

struct CnfStat {
    unsigned flags;  // 1: a violation, 2: not canonical or too long
    int max_len, min_len, max_count;
    unsigned long long wsum, wor;
};

unsigned grid_for(int64_t items) {
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>((items + kThreads - 1) / kThreads, 152 * 32));
}

}  // namespace

// A thread a clause: offsets never decreasing (the host has seen the first, 0,
// and the last, raw) and clause lengths.  Before
// anything reads a literal: the last offset says how many the caller has
// only if no offset before it is larger.  On the host this pass costs more
// than its kernel and the wait for it (n=3e5, m=1.3e6, msat_create: 2.2 ms;
// with the host's threads 3.1).
__global__ void __launch_bounds__(kThreads)
    k_off_check(int64_t m, const int64_t *__restrict__ off, CnfStat *__restrict__ stat) {
    unsigned flags = 0;
    int max_len = 0, min_len = INT_MAX;
    for (int64_t j = (int64_t)blockIdx.x * kThreads + threadIdx.x; j < m; j += (int64_t)gridDim.x * kThreads) {
        const int64_t beg = __ldg(off + j), end = __ldg(off + j + 1);
        if (end < beg) flags |= 1u;
        else if (end - beg > kMaxCleanLen) flags |= 2u;
        else {
            max_len = max(max_len, (int)(end - beg));
            min_len = min(min_len, (int)(end - beg));
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        flags |= __shfl_xor_sync(0xffffffffu, flags, o);
        max_len = max(max_len, __shfl_xor_sync(0xffffffffu, max_len, o));
        min_len = min(min_len, __shfl_xor_sync(0xffffffffu, min_len, o));
    }
    if ((threadIdx.x & 31) == 0) {
        if (flags) atomicOr(&stat->flags, flags);
        atomicMax(&stat->max_len, max_len);
        atomicMin(&stat->min_len, min_len);
    }
}

// A thread a clause (of at most kMaxCleanLen literals, offsets checked):
// literals and weights checked, offsets and literals packed, variable counts
// added up.
__global__ void __launch_bounds__(kThreads)
    k_cnf_check(int n, int64_t m, const int64_t *__restrict__ off, const int32_t *__restrict__ lits,
                const int64_t *__restrict__ w, int32_t *__restrict__ coff, int32_t *__restrict__ lit,
                int32_t *__restrict__ deg, CnfStat *__restrict__ stat) {
    unsigned flags = 0;
    unsigned long long wsum = 0, wor = 0;
    for (int64_t j = (int64_t)blockIdx.x * kThreads + threadIdx.x; j < m; j += (int64_t)gridDim.x * kThreads) {
        const int beg = (int)__ldg(off + j), end = (int)__ldg(off + j + 1), len = end - beg;
        if (j == 0) coff[0] = 0;
        coff[j + 1] = end;
        for (int p = 0; p < len; ++p) {
            const int l = __ldg(lits + beg + p);
            if (l == 0 || l > n || l < -n) {
                flags |= 1u;
                break;
            }
            const int v = (l < 0 ? -l : l) - 1;
            for (int r = 0; r < p; ++r) {
                const int o = __ldg(lits + beg + r);
                if ((o < 0 ? -o : o) - 1 == v) flags |= 2u;
            }
            lit[beg + p] = (v << 1) | (l < 0 ? 1 : 0);
            atomicAdd(deg + v, 1);
        }
        if (w) {
            const int64_t wj = __ldg(w + j);
            if (wj < 1) flags |= 1u;
            wsum += (unsigned long long)wj;
            wor |= (unsigned long long)wj;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        flags |= __shfl_xor_sync(0xffffffffu, flags, o);
        wsum += __shfl_xor_sync(0xffffffffu, wsum, o);
        wor |= __shfl_xor_sync(0xffffffffu, wor, o);
    }
    if ((threadIdx.x & 31) == 0) {
        if (flags) atomicOr(&stat->flags, flags);
        if (w) {
            atomicAdd(&stat->wsum, wsum);
            atomicOr(&stat->wor, wor);
        }
    }
}

// ------------------------------------------------------------------- scan
// Exclusive prefix sums of count int32 values in three launches: block sums,
// their prefix by one block, the values.

__device__ __forceinline__ int block_exclusive(int v, int &total) {
    __shared__ int s_w[kThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int inc = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, inc, d);
        if (lane >= d) inc += y;
    }
    __syncthreads();
    if (lane == 31) s_w[warp] = inc;
    __syncthreads();
    int before = 0;
    total = 0;
#pragma unroll
    for (int k = 0; k < kThreads / 32; ++k) {
        before += k < warp ? s_w[k] : 0;
        total += s_w[k];
    }
    return before + inc - v;
}

__global__ void __launch_bounds__(kThreads)
    k_scan_sums(const int32_t *__restrict__ in, int64_t count, int32_t *__restrict__ part, CnfStat *__restrict__ stat) {
    int sum = 0, mx = 0;
    for (int u = 0; u < kScanItems; ++u) {
        const int64_t i = (int64_t)blockIdx.x * kScanBlock + u * kThreads + threadIdx.x;
        if (i < count) {
            const int v = in[i];
            sum += v;
            mx = max(mx, v);
        }
    }
    int total;
    block_exclusive(sum, total);
    if (threadIdx.x == 0) part[blockIdx.x] = total;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0) atomicMax(&stat->max_count, mx);
}

__global__ void __launch_bounds__(kThreads) k_scan_top(int32_t *__restrict__ part, int nblk) {
    int carry = 0;
    for (int b0 = 0; b0 < nblk; b0 += kThreads) {
        const int i = b0 + threadIdx.x;
        const int v = i < nblk ? part[i] : 0;
        int total;
        const int ex = block_exclusive(v, total);
        if (i < nblk) part[i] = carry + ex;
        carry += total;
    }
}

// out[i] = sum of in[0 .. i), out[count] the total; cur (nullable): a copy.
__global__ void __launch_bounds__(kThreads)
    k_scan_apply(const int32_t *__restrict__ in, int64_t count, const int32_t *__restrict__ part,
                 int32_t *__restrict__ out, int32_t *__restrict__ cur) {
    const int64_t i0 = (int64_t)blockIdx.x * kScanBlock + (int64_t)threadIdx.x * kScanItems;
    int v[kScanItems];
    int sum = 0;
#pragma unroll
    for (int u = 0; u < kScanItems; ++u) {
        v[u] = i0 + u < count ? in[i0 + u] : 0;
        sum += v[u];
    }
    int total;
    int at = part[blockIdx.x] + block_exclusive(sum, total);
#pragma unroll
    for (int u = 0; u < kScanItems; ++u) {
        if (i0 + u < count) {
            out[i0 + u] = at;
            if (cur) cur[i0 + u] = at;
            at += v[u];
            if (i0 + u == count - 1) out[count] = at;
        }
    }
}

static cudaError_t scan(const int32_t *in, int64_t count, int32_t *out, int32_t *cur, int32_t *part, CnfStat *stat,
                        cudaStream_t st) {
    const int nblk = (int)((count + kScanBlock - 1) / kScanBlock);
    k_scan_sums<<<nblk, kThreads, 0, st>>>(in, count, part, stat);
    k_scan_top<<<1, kThreads, 0, st>>>(part, nblk);
    k_scan_apply<<<nblk, kThreads, 0, st>>>(in, count, part, out, cur);
    return cudaGetLastError();
}

static size_t scan_parts(int64_t count) { return (size_t)((count + kScanBlock - 1) / kScanBlock); }

// ------------------------------------------------------------ occurrences

// clause << 1 | neg of every literal into its variable's list, in any order.
__global__ void __launch_bounds__(kThreads)
    k_occ_scatter(int64_t m, const int32_t *__restrict__ coff, const int32_t *__restrict__ lit,
                  int32_t *__restrict__ cur, int32_t *__restrict__ occ) {
    for (int64_t j = (int64_t)blockIdx.x * kThreads + threadIdx.x; j < m; j += (int64_t)gridDim.x * kThreads) {
        const int beg = __ldg(coff + j), end = __ldg(coff + j + 1);
        for (int p = beg; p < end; ++p) {
            const int L = __ldg(lit + p);
            occ[atomicAdd(cur + (L >> 1), 1)] = (int)(j << 1) | (L & 1);
        }
    }
}

// A warp sorts one variable's list by clause (each word's rank is the number
// of smaller words) and writes row << 1 | neg in place.
__global__ void __launch_bounds__(kThreads)
    k_occ_sort(int n, const int32_t *__restrict__ voff, const int32_t *__restrict__ row, int32_t *__restrict__ occ) {
    __shared__ int s_list[kThreads / 32][kMaxSortDeg];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto word = [&](int x) { return row ? (__ldg(row + (x >> 1)) << 1) | (x & 1) : x; };
    for (int64_t i = (int64_t)blockIdx.x * (kThreads / 32) + warp; i < n; i += (int64_t)gridDim.x * (kThreads / 32)) {
        const int beg = __ldg(voff + i), d = __ldg(voff + i + 1) - beg;
        if (d <= 32) {
            const int x = lane < d ? occ[beg + lane] : INT_MAX;
            int rank = 0;
            for (int k = 0; k < d; ++k) rank += __shfl_sync(0xffffffffu, x, k) < x;
            if (lane < d) occ[beg + rank] = word(x);
        } else if (d <= kMaxSortDeg) {
            int *s = s_list[warp];
            for (int k = lane; k < d; k += 32) s[k] = occ[beg + k];
            __syncwarp();
            for (int k0 = 0; k0 < d; k0 += 32) {
                const int k = k0 + lane;
                const int x = k < d ? s[k] : INT_MAX;
                int rank = 0;
                for (int q = 0; q < d; ++q) rank += s[q] < x;
                if (k < d) occ[beg + rank] = word(x);
            }
            __syncwarp();
        }
    }
}

// -------------------------------------------------------------- row order

// Light block of every variable (-1, set before: heavy).
__global__ void __launch_bounds__(kThreads) k_var_block(const int2 *__restrict__ lblk, int nb, int32_t *__restrict__ vblk) {
    for (int b = blockIdx.x; b < nb; b += gridDim.x) {
        const int2 r = __ldg(lblk + b);
        for (int v = r.x + threadIdx.x; v < r.y; v += kThreads) vblk[v] = b;
    }
}

// Row group of every clause: its first light variable's block counted from
// the last, nb for clauses of heavy variables alone.
__global__ void __launch_bounds__(kThreads)
    k_row_group(int64_t m, int nb, const int32_t *__restrict__ coff, const int32_t *__restrict__ lit,
                const int32_t *__restrict__ vblk, int32_t *__restrict__ group, int32_t *__restrict__ count) {
    for (int64_t j = (int64_t)blockIdx.x * kThreads + threadIdx.x; j < m; j += (int64_t)gridDim.x * kThreads) {
        const int beg = __ldg(coff + j), end = __ldg(coff + j + 1);
        int g = nb;
        for (int p = beg; p < end; ++p) {
            const int b = __ldg(vblk + (__ldg(lit + p) >> 1));
            if (b >= 0) {
                g = nb - 1 - b;
                break;
            }
        }
        group[j] = g;
        atomicAdd(count + g, 1);
    }
}

__global__ void __launch_bounds__(kThreads)
    k_row_scatter(int64_t m, const int32_t *__restrict__ group, int32_t *__restrict__ cur, int32_t *__restrict__ list) {
    for (int64_t j = (int64_t)blockIdx.x * kThreads + threadIdx.x; j < m; j += (int64_t)gridDim.x * kThreads)
        list[atomicAdd(cur + __ldg(group + j), 1)] = (int32_t)j;
}

// A block sorts one group's clauses (at most kMaxGroup) and writes each
// clause's row with its literals (common length), weight or length.
__global__ void __launch_bounds__(kThreads)
    k_row_sort(int ngroups, const int32_t *__restrict__ start, const int32_t *__restrict__ list, int kfix,
               const int32_t *__restrict__ coff, const int32_t *__restrict__ lit, const int64_t *__restrict__ w,
               int32_t *__restrict__ row, int32_t *__restrict__ plit, int64_t *__restrict__ pw, int32_t *__restrict__ rlen) {
    __shared__ int s[kMaxGroup];
    for (int g = blockIdx.x; g < ngroups; g += gridDim.x) {
        const int beg = __ldg(start + g), c = __ldg(start + g + 1) - beg;
        __syncthreads();
        for (int k = threadIdx.x; k < c; k += kThreads) s[k] = __ldg(list + beg + k);
        __syncthreads();
        for (int k = threadIdx.x; k < c; k += kThreads) {
            const int j = s[k];
            int rank = 0;
            for (int q = 0; q < c; ++q) rank += s[q] < j;
            const int64_t r = beg + rank;
            row[j] = (int32_t)r;
            if (kfix > 0)
                for (int p = 0; p < kfix; ++p) plit[r * kfix + p] = __ldg(lit + (int64_t)j * kfix + p);
            else
                rlen[r] = __ldg(coff + j + 1) - __ldg(coff + j);
            if (w) pw[r] = __ldg(w + j);
        }
    }
}

__global__ void __launch_bounds__(kThreads)
    k_row_lits(int64_t m, const int32_t *__restrict__ coff, const int32_t *__restrict__ lit,
               const int32_t *__restrict__ row, const int32_t *__restrict__ pcoff, int32_t *__restrict__ plit) {
    for (int64_t j = (int64_t)blockIdx.x * kThreads + threadIdx.x; j < m; j += (int64_t)gridDim.x * kThreads) {
        int q = __ldg(pcoff + __ldg(row + j));
        for (int p = __ldg(coff + j); p < __ldg(coff + j + 1); ++p) plit[q++] = __ldg(lit + p);
    }
}

// --------------------------------------------------------------- host side

namespace {

// Temporary device arrays, allocated and freed in order on the stream.
struct Temps {
    cudaStream_t st;
    std::vector<void *> p;
    explicit Temps(cudaStream_t s) : st(s) {}
    ~Temps() {
        for (void *q : p) cudaFreeAsync(q, st);
    }
    template <typename T>
    cudaError_t get(T **out, size_t count) {
        const cudaError_t e = cudaMallocAsync(reinterpret_cast<void **>(out), std::max<size_t>(16, count * sizeof(T)), st);
        if (e == cudaSuccess) p.push_back(*out);
        else *out = nullptr;
        return e;
    }
};

// Up to this many clauses the host looks at the offsets: the pass costs 0.6 us
// per thousand clauses, the device's its launch, a wait and, where the host
// path follows, an upload.  msat_create with the host's look / the device's:
// weighted Zipf m=1e5 4.20 / 4.36 ms, m=3e5 7.42 / 7.55, m=1e6 12.8 / 12.4,
// 3-SAT m=51600 0.56 / 0.56, m=258000 1.06 / 0.93; in either case the host
// path then skips its own (Zipf m=1e5 4.15, m=1e6 11.6, m=2e6 17.5 ms; 4.08,
// 11.9 and 18.3 before there was a device path).
constexpr int64_t kHostOffsets = 1 << 17;

// Whether every clause has 0 to kMaxCleanLen literals, and the shortest and
// longest.  off[0] is 0, so differences within that range (taken modulo 2^64)
// say that the offsets are their sums, below 2^31, and never decrease.
bool lengths_in_range(int64_t m, const int64_t *off, int &min_len, int &max_len) {
    int64_t lo = INT_MAX, hi = 0;
    for (int64_t j = 0; j < m; ++j) {
        const int64_t d = (int64_t)((uint64_t)off[j + 1] - (uint64_t)off[j]);
        lo = std::min(lo, d);
        hi = std::max(hi, d);
    }
    min_len = (int)lo;
    max_len = (int)hi;
    return lo >= 0 && hi <= kMaxCleanLen;
}

// Whether a look at a few clauses (offsets checked, at most kMaxCleanLen
// literals each) already says that the instance is for the host path: a
// variable twice in one of them, or one so frequent that it has about twice
// the occurrences a warp sorts.  The two are found for certain only by the
// kernels, after the upload of every literal and, for a frequent variable,
// atomics that all go to its counter.  msat_create of weighted Zipf n=2e5,
// m=1e6 12.9 -> 12.2 ms, n=2e4, m=1e5 4.7 -> 4.4; 3-SAT n=3e5, m=1.3e6, which
// it passes, 2.19 -> 2.25.
bool sample_unfit(int64_t m, const int64_t *off, const int32_t *lits) {
    constexpr int kClauses = 256, kSlots = 1 << 14;  // more slots than literals
    const int k = (int)std::min<int64_t>(m, kClauses);
    int64_t beg[kClauses], total = 0;
    int len[kClauses];
    for (int s = 0; s < k; ++s) {
        const int64_t j = m * s / k;
        beg[s] = off[j];
        len[s] = (int)(off[j + 1] - off[j]);
        total += len[s];
    }
    for (int s = 0; s < k; ++s) __builtin_prefetch(lits + beg[s]);
    uint32_t var[kSlots];
    uint16_t cnt[kSlots] = {0};
    int top = 0;
    for (int s = 0; s < k; ++s)
        for (int p = 0; p < len[s]; ++p) {
            const int32_t l = lits[beg[s] + p];
            const uint32_t v = l < 0 ? 0u - (uint32_t)l : (uint32_t)l;
            for (int r = 0; r < p; ++r) {
                const int32_t o = lits[beg[s] + r];
                if ((o < 0 ? 0u - (uint32_t)o : (uint32_t)o) == v) return true;
            }
            uint32_t h = (v * 2654435761u) >> 18;
            while (cnt[h] && var[h] != v) h = (h + 1) & (kSlots - 1);
            var[h] = v;
            top = std::max<int>(top, ++cnt[h]);
        }
    return top >= 12 && (double)top * (double)off[m] > 2.0 * kMaxSortDeg * (double)total;
}

// An array that outlives the preparation.
template <typename T>
cudaError_t own(const DevCnf &d, T **out, size_t count) {
    const size_t bytes = std::max<size_t>(16, count * sizeof(T));
    const cudaError_t e = d.pool ? cudaMallocAsync(reinterpret_cast<void **>(out), bytes, d.st)
                                 : cudaMalloc(reinterpret_cast<void **>(out), bytes);
    if (e != cudaSuccess) *out = nullptr;
    return e;
}

}  // namespace

void DevCnf::clear() {
    // pending kernels may still use them: cudaFree waits for the device
    auto drop = [&](auto *&p) {
        if (p) {
            if (pool) cudaFreeAsync(p, st);
            else cudaFree(p);
        }
        p = nullptr;
    };
    drop(coff);
    drop(lit);
    drop(voff);
    drop(occ);
    drop(w);
    drop(plit);
    drop(pcoff);
    drop(pw);
    if (row) cudaFreeAsync(row, st);
    row = nullptr;
}

bool DevCnf::check(int32_t n_vars, int64_t n_clauses, const int64_t *off, const int32_t *lits, const int64_t *weights,
                   cudaStream_t stream, HostCnf &out) {
    n = n_vars;
    m = n_clauses;
    st = stream;
    const int64_t raw = off[m];
    if (off[0] != 0 || raw < 1 || raw >= (1LL << 31) || !lits || m < 1) return false;
    Temps T(st);
    int64_t *d_off = nullptr;
    int32_t *d_raw = nullptr, *deg = nullptr, *part = nullptr;
    CnfStat *stat = nullptr;
    CnfStat h{0u, 0, INT_MAX, 0, 0ull, 0ull};
    const bool host_off = m <= kHostOffsets;
    if (host_off) {
        if (!lengths_in_range(m, off, h.min_len, h.max_len)) return false;
        off_checked = true;
        if (sample_unfit(m, off, lits)) return false;
    }
    cudaError_t e = T.get(&d_off, (size_t)m + 1);
    if (!e) e = T.get(&stat, 1);
    if (!e) e = cudaMemcpyAsync(stat, &h, sizeof(h), cudaMemcpyHostToDevice, st);
    if (!e) e = cudaMemcpyAsync(d_off, off, sizeof(int64_t) * (size_t)(m + 1), cudaMemcpyHostToDevice, st);
    if (!host_off) {
        if (!e) {
            k_off_check<<<grid_for(m), kThreads, 0, st>>>(m, d_off, stat);
            e = cudaGetLastError();
        }
        if (!e) e = cudaMemcpyAsync(&h, stat, sizeof(h), cudaMemcpyDeviceToHost, st);
        if (!e) e = cudaStreamSynchronize(st);
    }
    if (e) {
        cudaGetLastError();
        return false;
    }
    if (!host_off) {
        off_checked = (h.flags & 1u) == 0;
        if (h.flags || sample_unfit(m, off, lits)) return false;
    }
    read_lits = true;
    e = own(*this, &coff, (size_t)m + 1);
    if (!e) e = own(*this, &lit, (size_t)raw);
    if (!e) e = own(*this, &voff, (size_t)n + 1);
    if (!e && weights) e = own(*this, &w, (size_t)m);
    if (!e) e = T.get(&d_raw, (size_t)raw);
    if (!e) e = T.get(&deg, (size_t)n);
    if (!e) e = T.get(&part, scan_parts(n));
    if (!e) e = cudaMemsetAsync(deg, 0, sizeof(int32_t) * (size_t)n, st);
    if (!e) e = cudaMemcpyAsync(d_raw, lits, sizeof(int32_t) * (size_t)raw, cudaMemcpyHostToDevice, st);
    if (!e && weights) e = cudaMemcpyAsync(w, weights, sizeof(int64_t) * (size_t)m, cudaMemcpyHostToDevice, st);
    if (!e) {
        k_cnf_check<<<grid_for(m), kThreads, 0, st>>>(n, m, d_off, d_raw, w, coff, lit, deg, stat);
        e = cudaGetLastError();
    }
    if (!e) e = scan(deg, n, voff, nullptr, part, stat, st);
    out.voff.alloc((size_t)n + 1);
    if (!e) e = cudaMemcpyAsync(&h, stat, sizeof(h), cudaMemcpyDeviceToHost, st);
    if (!e) e = cudaMemcpyAsync(out.voff.data(), voff, sizeof(int32_t) * ((size_t)n + 1), cudaMemcpyDeviceToHost, st);
    const cudaError_t s = cudaStreamSynchronize(st);
    if (!e) e = s;
    if (e) {
        cudaGetLastError();
        return false;
    }
    if (h.flags || h.max_count > kMaxSortDeg) return false;
    nnz = raw;
    kfix = h.min_len == h.max_len ? h.max_len : 0;
    out.nnz = raw;
    out.kfix = kfix;
    out.max_len = h.max_len;
    out.max_deg = h.max_count;
    out.wsum = weights ? (int64_t)h.wsum : m;
    out.wor = weights ? (int64_t)h.wor : 0;
    return true;
}

bool DevCnf::rows(const std::vector<int2> &lblk) {
    const int nb = (int)lblk.size();
    Temps T(st);
    int2 *d_lblk = nullptr;
    int32_t *vblk = nullptr, *group = nullptr, *count = nullptr, *start = nullptr, *cur = nullptr, *list = nullptr;
    int32_t *part = nullptr, *rlen = nullptr;
    CnfStat *stat = nullptr;
    cudaError_t e = own(*this, &plit, (size_t)nnz);
    if (!e && kfix == 0) e = own(*this, &pcoff, (size_t)m + 1);
    if (!e && w) e = own(*this, &pw, (size_t)m);
    if (!e) e = cudaMallocAsync(reinterpret_cast<void **>(&row), sizeof(int32_t) * (size_t)m, st);
    if (!e) e = T.get(&d_lblk, (size_t)nb);
    if (!e) e = T.get(&vblk, (size_t)n);
    if (!e) e = T.get(&group, (size_t)m);
    if (!e) e = T.get(&count, (size_t)nb + 1);
    if (!e) e = T.get(&start, (size_t)nb + 2);
    if (!e) e = T.get(&cur, (size_t)nb + 1);
    if (!e) e = T.get(&list, (size_t)m);
    if (!e) e = T.get(&part, scan_parts(std::max<int64_t>(m, nb + 1)));
    if (!e && kfix == 0) e = T.get(&rlen, (size_t)m);
    if (!e) e = T.get(&stat, 1);
    CnfStat h{};
    if (!e) e = cudaMemcpyAsync(stat, &h, sizeof(h), cudaMemcpyHostToDevice, st);
    if (!e && nb > 0) e = cudaMemcpyAsync(d_lblk, lblk.data(), sizeof(int2) * (size_t)nb, cudaMemcpyHostToDevice, st);
    if (!e) e = cudaMemsetAsync(vblk, 0xff, sizeof(int32_t) * (size_t)n, st);
    if (!e) e = cudaMemsetAsync(count, 0, sizeof(int32_t) * ((size_t)nb + 1), st);
    if (!e) {
        if (nb > 0) k_var_block<<<std::min(nb, 152 * 8), kThreads, 0, st>>>(d_lblk, nb, vblk);
        k_row_group<<<grid_for(m), kThreads, 0, st>>>(m, nb, coff, lit, vblk, group, count);
        e = cudaGetLastError();
    }
    if (!e) e = scan(count, nb + 1, start, cur, part, stat, st);
    if (!e) e = cudaMemcpyAsync(&h, stat, sizeof(h), cudaMemcpyDeviceToHost, st);
    const cudaError_t s = cudaStreamSynchronize(st);
    if (!e) e = s;
    if (!e && h.max_count > kMaxGroup) return false;
    if (!e) {
        k_row_scatter<<<grid_for(m), kThreads, 0, st>>>(m, group, cur, list);
        k_row_sort<<<std::min(nb + 1, 152 * 8), kThreads, 0, st>>>(nb + 1, start, list, kfix, coff, lit, w, row, plit, pw, rlen);
        e = cudaGetLastError();
    }
    if (!e && kfix == 0) {
        e = scan(rlen, m, pcoff, nullptr, part, stat, st);
        if (!e) {
            k_row_lits<<<grid_for(m), kThreads, 0, st>>>(m, coff, lit, row, pcoff, plit);
            e = cudaGetLastError();
        }
    }
    if (e) cudaGetLastError();
    return e == cudaSuccess;
}

bool DevCnf::occurrences() {
    Temps T(st);
    int32_t *cur = nullptr;
    cudaError_t e = own(*this, &occ, (size_t)nnz);
    if (!e) e = T.get(&cur, (size_t)n);
    if (!e) e = cudaMemcpyAsync(cur, voff, sizeof(int32_t) * (size_t)n, cudaMemcpyDeviceToDevice, st);
    if (!e) {
        k_occ_scatter<<<grid_for(m), kThreads, 0, st>>>(m, coff, lit, cur, occ);
        k_occ_sort<<<grid_for((int64_t)n * 32), kThreads, 0, st>>>(n, voff, row, occ);
        e = cudaGetLastError();
    }
    if (e) cudaGetLastError();
    return e == cudaSuccess;
}

}  // namespace msat

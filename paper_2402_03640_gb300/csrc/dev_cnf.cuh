// Device-side CNF preparation of msat_create (dev_cnf.cu).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "host_cnf.cuh"

namespace msat {

// The arrays of a checked CNF on the device, built there from the caller's
// host arrays.  Owns them until release(); temporaries are freed in order on
// the stream.
struct DevCnf {
    int32_t n = 0;
    int64_t m = 0, nnz = 0;
    int32_t kfix = 0;
    cudaStream_t st = nullptr;
    bool pool = false;  // arrays from the stream-ordered pool (contexts of the server)
    int32_t *coff = nullptr, *lit = nullptr, *voff = nullptr, *occ = nullptr;
    int64_t *w = nullptr;
    int32_t *row = nullptr;  // temporary: clause -> row of the store
    int32_t *plit = nullptr, *pcoff = nullptr;
    int64_t *pw = nullptr;
    bool off_checked = false;  // check() has seen that the offsets never decrease
    bool read_lits = false;  // the literals were uploaded

    explicit DevCnf(bool pool_alloc) : pool(pool_alloc) {}
    DevCnf(const DevCnf &) = delete;
    DevCnf &operator=(const DevCnf &) = delete;
    ~DevCnf() { clear(); }

    // Frees every array still held here.
    void clear();

    // Checks and packs the clauses and makes the occurrence offsets; fills
    // the sizes, kfix, max_len, max_deg, wsum, wor and voff of `out`.  False:
    // the instance is for the host path (a violation, whose message that path
    // gives; a repeated variable in a clause; a clause of more than 32
    // literals; a variable of more than 1024 occurrences; no memory).
    bool check(int32_t n_vars, int64_t n_clauses, const int64_t *off, const int32_t *lits, const int64_t *weights,
               cudaStream_t stream, HostCnf &out);
    // Rows of the store grouped by light block (RowOrder): row, plit, pcoff, pw.
    bool rows(const std::vector<int2> &lblk);
    // The occurrence list in (clause, position) order, with rows if rows() ran.
    bool occurrences();
    // Hands an array over to the caller.
    template <typename T>
    static T *release(T *&p) {
        T *q = p;
        p = nullptr;
        return q;
    }
};

// Instances worth the device path: below this many literals the host's cores
// are as fast, and an instance that may fit the one-block-per-restart kernel
// (its 21 bytes a variable and 4 a clause within an SM's shared memory) needs
// the host's clause list for that kernel's lists.
inline bool dev_cnf_worth(int32_t n, int64_t m, int64_t raw) {
    return raw >= (1 << 17) && 21LL * n + 4LL * m > 227 * 1024;
}

// Upper bound of the device bytes that DevCnf::check holds at a time: the
// uploaded offsets and literals and the variables' counts beside the arrays
// that stay.  Nothing else of a context is allocated before they are freed;
// DevCnf::occurrences (without rows) holds less than the context does later.
inline size_t dev_cnf_check_bytes(int32_t n, int64_t m, int64_t raw, bool weighted) {
    return 12 * (size_t)(m + 1) + 8 * (size_t)raw + 9 * (size_t)(n + 1) + (weighted ? 8 * (size_t)m : 0) + 16 * 512;
}

}  // namespace msat

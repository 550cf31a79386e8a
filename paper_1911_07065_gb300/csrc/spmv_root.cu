// Fused CSR SpMV + root update: one pass over A per root of the GMRES
// polynomial (Algorithm 1: phi(A) v, Algorithm 3: p(A) v), plus the plain
// SpMV and the residual b - A x.  Two kernels with the same arithmetic (one fused
// multiply-add per nonzero, acc = fma(val, x[col], acc); a row of up to LONG_ROW
// entries summed in stored order, a longer one by a warp, long_rows; then the same
// epilogue), so their results are bit-identical:
//
// k_spmv_step, for a matrix streamed from HBM: a CTA owns a tile of rows
// (256 in FP64, 512 in FP32: two per thread).  It copies the tile's column
// indices and values into shared memory with asynchronous, coalesced
// 16-byte copies (consecutive threads take consecutive granules, so short
// rows of 5-7 entries leave no lane idle), then each thread walks its rows
// and applies the root update in the epilogue, reading and writing the
// row-aligned vectors once, coalesced.  Tiles whose nonzeros exceed the
// staging buffer are processed in chunks, so any row length is handled.
//
// k_spmv_direct, for small systems and for a matrix held in L2: one row per
// thread, its first entries read straight into registers before the wait on
// the previous step (no staging round trip).
//
// GB300 executes about two FP64 operations per clock per SM, so in FP64 the
// multiply-adds, not only the bytes, bound these kernels: one FMA per
// nonzero is the minimum and the epilogues use fused forms.
//
// Consecutive steps overlap: each is launched as a programmatic dependent of
// the previous one and reads its share of the matrix before it waits for the
// previous step's vectors.
//
// L2 policy: when the matrix and the chain's vectors fit in L2, the matrix is
// read with an evict-last hint into a set-aside and stays resident across
// the roots of a chain (every root reads the same A).  Otherwise a chain
// holds the nonzeros of its leading rows that way in a 48 MB set-aside and
// streams the rest with evict-first, prefetching it into L2 half a resident
// wave ahead.
#include <algorithm>
#include <atomic>

#include "ppg_common.cuh"

namespace ppg {

constexpr int SPMV_ROWS = 256;      // threads per CTA

__device__ __forceinline__ uint64_t l2_policy(int keep) {
    uint64_t p;
    if (keep)
        asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
    else
        asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}

template <int BYTES>
__device__ __forceinline__ void cp_async(void* smem, const void* gmem, uint64_t pol) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global.L2::cache_hint [%0], [%1], %2, %3;" ::"r"(s),
                 "l"(gmem), "n"(BYTES), "l"(pol)
                 : "memory");
}

// Hint: bring [b, e) into L2 (16-byte granules inside the range; nothing
// waits on it).  Both ends are rounded down to 16 bytes, which stays inside
// the (at least 256-byte aligned) allocation that holds the range.
__device__ __forceinline__ void prefetch_l2(const void* b, const void* e) {
    const uintptr_t lo = (uintptr_t)b & ~(uintptr_t)15;
    const uintptr_t hi = (uintptr_t)e & ~(uintptr_t)15;
    if (hi > lo)
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(lo), "r"((unsigned)(hi - lo))
                     : "memory");
}

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem, uint64_t pol) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2;" ::"r"(s), "l"(gmem),
                 "l"(pol)
                 : "memory");
}

// Stage elements [c0, c1) of src into shared memory as dst[k - base], with
// base = c0 rounded down to a multiple of 4 elements.  With src 16-byte
// aligned, the 16-byte granules of [base, c1 rounded down to 4) move with one
// cp.async each (the few elements before c0 come along) and the ragged end
// per element, so nothing at or past c1 is read; otherwise every element of
// [c0, c1) is copied alone.  dst (16-byte aligned) holds c1 - base elements.
template <typename E>
__device__ __forceinline__ void stage_async(E* dst, const E* src, int32_t base, int32_t c0,
                                            int32_t c1, int tid, int nthr, uint64_t pol) {
    constexpr int PER = 16 / (int)sizeof(E);
    int32_t t0 = c0;
    if (((uintptr_t)src & 15) == 0) {
        const int32_t vend = c1 & ~3;
        const int32_t nvec = vend > base ? (vend - base) / PER : 0;
        for (int32_t q = tid; q < nvec; q += nthr) cp_async16(dst + q * PER, src + base + q * PER, pol);
        t0 = max(vend, c0);
    }
    for (int32_t k = t0 + tid; k < c1; k += nthr) cp_async<sizeof(E)>(dst + (k - base), src + k, pol);
}

// Stage a chunk of values and column indices by 16-byte granules from
// base = c0 & ~3 (measured faster than per-element copies in both precisions:
// FP64 2-D 1000^2 chains -2.6 %, 3-D 160^3 -5 %; FP32 3-D 160^3 chains -8 %).
template <typename T>
__device__ __forceinline__ void stage_chunk(T* sval, int32_t* scol, const T* vals,
                                            const int32_t* colind, int32_t base, int32_t c0,
                                            int32_t c1, int tid, int nthr, uint64_t pol) {
    stage_async<T>(sval, vals, base, c0, c1, tid, nthr, pol);
    stage_async<int32_t>(scol, colind, base, c0, c1, tid, nthr, pol);
}

__device__ __forceinline__ void cp_async_wait_all() {
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
}

// The epilogue of one row: the root update of the step, given s = (A x)[r]
// and the row's inputs e0 = a0[r], e1 = a1[r], e2 = a2[r].
template <typename T, int OP>
__device__ __forceinline__ void step_epilogue(const StepArgs<T>& a, int64_t r, T s, T e0, T e1,
                                              T e2, double& sq) {
    if constexpr (OP == OP_SPMV) {
        a.o0[r] = s;
    } else if constexpr (OP == OP_RESID) {
        const T v = e0 - s;
        a.o0[r] = v;
        sq += (double)v * (double)v;
    } else if constexpr (OP == OP_PHI_REAL) {
        const T pin = fma(-a.c1, s, e0);
        a.o0[r] = (a.flags & F_FINAL) ? e2 - pin : pin;
    } else if constexpr (OP == OP_PHI_PAIR2) {
        // pi' = pi + c2 (A prod - 2a prod)
        const T t = fma(-a.c1, e0, s);
        const T pin = fma(a.c2, t, e1);
        a.o0[r] = (a.flags & F_FINAL) ? e2 - pin : pin;
    } else if constexpr (OP == OP_P_REAL) {
        const T pnew = (a.flags & F_PZERO) ? a.c1 * e0 : fma(a.c1, e0, e1);
        const T prodn = fma(-a.c1, s, e0);
        if (a.flags & F_FINAL) {
            a.o0[r] = fma(a.c3, prodn, pnew);
        } else {
            a.o0[r] = pnew;
            a.o1[r] = prodn;
        }
    } else if constexpr (OP == OP_P_PAIR1) {
        const T tmp = fma(a.c1, e0, -s);
        a.o0[r] = (a.flags & F_PZERO) ? a.c2 * tmp : fma(a.c2, tmp, e1);
        if (!(a.flags & F_NO_O1)) a.o1[r] = tmp;
    } else if constexpr (OP == OP_P_PAIR2) {
        const T prodn = fma(-a.c2, s, e0);
        if (a.flags & F_FINAL) {
            a.o0[r] = fma(a.c3, prodn, e1);
        } else {
            a.o0[r] = prodn;
        }
    }
}

// The rows of more than LONG_ROW entries (is_long: this lane's row r is one), a
// warp for each: on one thread such a row is a chain of dependent multiply-adds
// and gathers that the whole step waits for.  Lane l takes entries l, l + 32,
// ...; the lanes' sums meet in a fixed order.  19 FP64 steps over 198,907 rows
// of about six entries and four of 2,500: 6.10 -> 0.39 ms, FP32 2.52 -> 0.26 ms.
// (The whole CTA on a row is faster still, but the code for it cost every other
// matrix 3 % in registers.)
template <typename T, int OP>
__device__ __forceinline__ void long_rows(const StepArgs<T>& a, int64_t r, bool is_long,
                                          double& sq) {
    const int lane = threadIdx.x & 31;
    unsigned todo = __ballot_sync(0xffffffffu, is_long);
    while (todo) {
        const int src = __ffs(todo) - 1;
        todo &= todo - 1;
        const int32_t* rp = a.rowptr + __shfl_sync(0xffffffffu, (int32_t)r, src);
        const int32_t k1 = __ldg(rp + 1);
        T acc = T(0);
#pragma unroll 4
        for (int32_t k = __ldg(rp) + lane; k < k1; k += 32)
            acc = fma(__ldg(a.vals + k), __ldg(a.x + __ldg(a.colind + k)), acc);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
        if (lane == src) {
            const T e0 = a.a0 ? __ldg(a.a0 + r) : T(0);
            const T e1 = (a.a1 && !(a.flags & F_PZERO)) ? a.a1[r] : T(0);
            const T e2 = (a.a2 && (a.flags & F_FINAL)) ? __ldg(a.a2 + r) : T(0);
            step_epilogue<T, OP>(a, r, acc, e0, e1, e2, sq);
        }
    }
}

// The same as a call, eight entries a lane at a time, for small systems: inlined,
// code that few of them need costs a chain of short steps instruction fetches
// (as a graph, 40 FP64 steps of p(A) at 100^2: 63 us without it, 76 with long_rows,
// 68 with the call).
template <typename T, int OP>
__device__ __noinline__ double long_rows_call(const StepArgs<T>& a, int32_t r, unsigned todo) {
    constexpr int U = 8;
    const int lane = threadIdx.x & 31;
    double sq = 0.0;
    while (todo) {
        const int src = __ffs(todo) - 1;
        todo &= todo - 1;
        const int32_t row = __shfl_sync(0xffffffffu, r, src);
        const int32_t k1 = __ldg(a.rowptr + row + 1);
        T acc = T(0);
        for (int32_t k = __ldg(a.rowptr + row) + lane; k < k1; k += 32 * U) {
            int32_t c[U];
            T v[U], g[U];
            // (past the end: the last entry again, so that the loads need no branch)
#pragma unroll
            for (int u = 0; u < U; ++u) {
                c[u] = __ldg(a.colind + min(k + 32 * u, k1 - 1));
                v[u] = __ldg(a.vals + min(k + 32 * u, k1 - 1));
            }
#pragma unroll
            for (int u = 0; u < U; ++u) g[u] = __ldg(a.x + c[u]);
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (k + 32 * u < k1) acc = fma(v[u], g[u], acc);
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
        if (lane == src) {
            const T e0 = a.a0 ? __ldg(a.a0 + r) : T(0);
            const T e1 = (a.a1 && !(a.flags & F_PZERO)) ? a.a1[r] : T(0);
            const T e2 = (a.a2 && (a.flags & F_FINAL)) ? __ldg(a.a2 + r) : T(0);
            step_epilogue<T, OP>(a, r, acc, e0, e1, e2, sq);
        }
    }
    return sq;
}

// The tile's long rows with entries in a staged chunk, entries [c0, c1) at sval /
// scol [k], in long_rows' order, into sum[row].  The rows are dealt to the CTA's NW
// warps (a chunk holds some 26 rows of 135 entries, which are neighbours: with a
// warp on its own 32 rows, one warp would have them all), by a hash, so that every
// second or fourth row being long leaves none idle.  One row at most is left
// unfinished, and its warp has it again in the next chunk: its lanes' sums go to
// `left`, and come from `from`, which another warp's row may have to itself by then.
template <typename T, int NW, int ROWS>
__device__ __forceinline__ void long_rows_staged(const int32_t* srp, const T* sval, const int32_t* scol,
                                                 const T* __restrict__ x, int nrows, int32_t c0,
                                                 int32_t c1, T* sum, const T* from, T* left) {
    constexpr int B = NW == 8 ? 3 : 2;
    static_assert(NW == 1 << B, "the hash");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i0 = 0; i0 < ROWS / NW; i0 += 32) {
        const int i = i0 + lane;
        const int t = NW * i + (warp ^ ((i ^ (i >> B) ^ (i >> 2 * B)) & (NW - 1)));
        bool has = false;
        if (t < nrows) {
            const int32_t lo = srp[t], hi = srp[t + 1];
            has = hi - lo > LONG_ROW && lo < c1 && hi > c0;
        }
        unsigned todo = __ballot_sync(0xffffffffu, has);
        while (todo) {
            const int row = __shfl_sync(0xffffffffu, t, __ffs(todo) - 1);
            todo &= todo - 1;
            const int32_t lo = srp[row], hi = srp[row + 1], e = min(hi, c1);
            int32_t k = lo + lane;
            T part = T(0);
            if (lo < c0) {
                part = from[lane];
                k += (c0 - lo - lane + 31) / 32 * 32;   // (0 where the lane has had none)
            }
            for (; k < e; k += 128) {
                T v[4], g[4];
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (k + 32 * u < e) {
                        v[u] = sval[k + 32 * u];
                        g[u] = __ldg(x + scol[k + 32 * u]);
                    }
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (k + 32 * u < e) part = fma(v[u], g[u], part);
            }
            if (hi > c1) {
                left[lane] = part;
            } else {
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) part += __shfl_xor_sync(0xffffffffu, part, off);
                if (lane == 0) sum[row] = part;
            }
        }
    }
}

// part[block] = the sum of sq over the CTA's NT threads, in a fixed order
template <int NT>
__device__ __forceinline__ void block_sq(double sq, double* sred, double* part) {
    const int tid = threadIdx.x;
    for (int off = 16; off > 0; off >>= 1) sq += __shfl_down_sync(0xffffffffu, sq, off);
    if ((tid & 31) == 0) sred[tid >> 5] = sq;
    __syncthreads();
    if (tid == 0) {
        double t = 0.0;
        for (int w = 0; w < NT / 32; ++w) t += sred[w];
        part[blockIdx.x] = t;
    }
}

// Rows per thread: FP32 tiles take two rows per thread (512 rows per CTA),
// so each CTA's latency-bound phases (row pointers, staging, gathers) serve
// twice the bytes; FP64 keeps one (at 32 registers, 2048 threads per SM).
template <typename T>
__host__ __device__ constexpr int step_rpt() { return sizeof(T) == 4 ? 2 : 1; }

// Threads per CTA of the staged step: FP64 128 (tiles of 128 rows, 16 CTAs
// per SM; 3-D 160^3 FP64 chains 6220 -> 6390 GB/s against 256, 6070 with
// 64), FP32 256 (tiles of 512 rows; 128 threads measured the same)
template <typename T>
__host__ __device__ constexpr int step_threads() { return sizeof(T) == 4 ? 256 : 128; }

// Nonzeros staged per chunk: FP64 1024 (128 rows of up to 8); FP32 3584, so
// that a tile of 512 rows of a 7-point stencil is one chunk and the CTA's
// 30.7 KB of shared memory lets 7 CTAs share an SM (with 4096, 6 fit:
// 3-D 160^3 FP32 chains 1 % slower).  Longer tiles take several chunks.
template <typename T>
__host__ __device__ constexpr int step_chunk() { return sizeof(T) == 4 ? 3584 : 1024; }

// CTAs per SM the register budget must allow (FP32: 32 registers instead
// of 40; FP64: 16 CTAs of 128 threads, 32 registers).  The FP32 second step of a pair of
// Algorithm 1 (not on the precision form's path, which applies p(A) only)
// keeps 40 registers and 6 CTAs: at 32 it spills.
template <typename T, int OP>
__host__ __device__ constexpr int step_min_ctas() {
    return sizeof(T) == 4 ? (OP == OP_PHI_PAIR2 ? 6 : 7) : 16;
}

// ... and of the forms that also know the diagonal steps, or rows of many entries:
// 40 registers, for the sake of their CSR part (seven random entries per row, 60
// steps, 2e6 rows: 2.12 ms with 7 CTAs, 1.89 with 6; the plain kernel 2.05.  Rows
// of 130 - 140 entries, 400,000 of them: 172 us a step with 7 CTAs, 135 with 6).
constexpr int WIDE_CTAS = 6;

// FP32 matrices of more entries than this in the average row take the form that
// sums long rows from the staged chunks: of such a matrix they may be most of the
// bytes, and read twice (long_rows) they made a step up to 1.5 times as long as with
// one thread to a row.  400,000 rows of 130 - 140 entries: one thread 162 us a
// step, read twice 235, from the chunks 135; every fourth row of 140, the others of
// 3: 107, 153 and 82; every eighth 103, 113 and 65; every sixteenth (11.6 in the
// average row) 96 and 55, read twice.  Without long rows the form costs its two
// registers: 30 entries in every row 90.7 -> 92.1 us, 45 99.9 -> 102.2, 100 112 ->
// 99.  In FP64 a long row is bound by its multiply-adds, and reading it twice is
// faster than one thread throughout (the same matrices: 583 -> 350, 485 -> 237, 518
// -> 164 us), so FP64 has no such form: it cost the steps of grids 10 %.
constexpr double LONG_AVG = 16.0;

// one row's multiply-adds over its staged nonzeros [lo, hi): four gathers in
// flight, then the last 1-3 (FP32: issued together; FP64: one at a time)
template <typename T, bool WIDE_TAIL>
__device__ __forceinline__ T row_dot(const T* sval, const int32_t* scol, const T* __restrict__ x,
                                     int32_t k, int32_t hi, T acc) {
    for (; k + 4 <= hi; k += 4) {
        const T v0 = sval[k], v1 = sval[k + 1], v2 = sval[k + 2], v3 = sval[k + 3];
        const T x0 = __ldg(x + scol[k]), x1 = __ldg(x + scol[k + 1]);
        const T x2 = __ldg(x + scol[k + 2]), x3 = __ldg(x + scol[k + 3]);
        acc = fma(v0, x0, acc);
        acc = fma(v1, x1, acc);
        acc = fma(v2, x2, acc);
        acc = fma(v3, x3, acc);
    }
    const int rem = hi - k;
    if constexpr (!WIDE_TAIL) {
#pragma unroll 1
        for (; k < hi; ++k) acc = fma(sval[k], __ldg(x + scol[k]), acc);
    } else if (rem > 0) {
        const T v0 = sval[k];
        const T x0 = __ldg(x + scol[k]);
        T v1 = T(0), x1 = T(0), v2 = T(0), x2 = T(0);
        if (rem > 1) {
            v1 = sval[k + 1];
            x1 = __ldg(x + scol[k + 1]);
        }
        if (rem > 2) {
            v2 = sval[k + 2];
            x2 = __ldg(x + scol[k + 2]);
        }
        acc = fma(v0, x0, acc);
        if (rem > 1) acc = fma(v1, x1, acc);
        if (rem > 2) acc = fma(v2, x2, acc);
    }
    return acc;
}

// ---------------------------------------------------------------------------
// Diagonal form (FP32)
// ---------------------------------------------------------------------------
//
// A matrix from a grid has few distinct column - row offsets.  Stored by these
// diagonals -- a sorted list of offsets, a bit per row and offset, the values
// diagonal by diagonal -- a step reads no column indices and no row pointers,
// a diagonal with one value throughout is not read at all, and all that a tile
// of rows needs of x is a few contiguous windows, which the bulk-copy engine
// brings to shared memory in one round trip.  Rows are still summed entry by
// entry in stored order (the form is built only where the columns of every row
// increase, as the offsets then do), so the results are those of the CSR steps
// bit for bit.
//
// Building it is two passes over the matrix, inside the call.  Whether the
// matrix has the form is known on the device alone: the steps read it from
// the head and take the CSR path if not, so the host waits for nothing, and
// the call stays asynchronous and can be captured.  (A solve waits between cycles
// anyway, asks, and launches the plain steps without a form.)  An FP32 matrix
// without the form pays for the search, as below, and for CSR steps at 40
// registers: seven random entries in a row 102 -> 63 us a step, narrow bands of
// three, five and seven 28.4 -> 31.5, 33.3 -> 35.5 and 40.3 -> 41.1.
//
// 160^3, FP32, 60 steps of p(A): 2.94 -> 1.48 ms (one value per diagonal), 2.92
// -> 2.23 ms (values of their own), against 49 us a step at 0.91 of the copy
// bandwidth by CSR.  What is left is the issue of instructions and the life of a CTA
// (head, copies, arithmetic: three trips).
// Tried and slower: reading x and the values straight from global memory (27 -
// 35 us a step, five dependent trips per CTA), and CTAs that stay and loop over
// tiles without copies in flight (26 - 37 us).
//
// FP64 steps have no use for it: their multiply-adds bound them (529 G FMA/s
// measured, 1.68 per clock and SM; the chains run at 0.79 - 0.84 of that).

constexpr int DIAG_TILE = step_threads<float>() * step_rpt<float>();   // rows of a tile
constexpr int DIAG_CAP = 2 * (step_chunk<float>() + 4);   // elements of its shared memory
constexpr int32_t DIAG_NONE = INT32_MAX;   // no offset: columns are below n

// the head and, behind it, the finder's list
struct DiagHead {
    int32_t w[DIAG_HEAD];
    int32_t off[DIAG_MAX];            // unsorted, DIAG_NONE: free
    uint32_t ref[DIAG_MAX];           // bits of the first value seen, DIAG_UNSET: none yet
    uint32_t mixed;                   // bit i: list entry i has several values
};
constexpr uint32_t DIAG_UNSET = 0x7fb4deadu;   // a NaN that no arithmetic returns

// The list starts with the middle row's offsets (of a grid, all of them), so that
// the CTAs of k_diag_find, which end together, have little to add to it.
__global__ void k_diag_init(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ colind,
                            const float* __restrict__ vals, int32_t n, int32_t most, DiagHead* H) {
    const int i = threadIdx.x;
    const int32_t r = n / 2, k = __ldg(rowptr + r), len = __ldg(rowptr + r + 1) - k;
    if (i < DIAG_HEAD) H->w[i] = i == 0 && len > most ? 1 : 0;
    if (i < DIAG_MAX) {
        const bool has = i < len && len <= most;
        // (not increasing: k_diag_find sees it; no offset is in the list twice)
        const int32_t o = has ? __ldg(colind + k + i) - r : DIAG_NONE;
        const bool first = i == 0 || !has || o > __ldg(colind + k + i - 1) - r;
        H->off[i] = first ? o : DIAG_NONE;
        H->ref[i] = has && first ? __float_as_uint(__ldg(vals + k + i)) : DIAG_UNSET;
    }
    if (i == 0) H->mixed = 0;
}

// Every offset of the matrix into the list, and whether its values are all the
// same.  A CTA takes tiles of DIAG_ROWS rows in turn, copies their entries to
// shared memory (coalesced) and walks them there, one row per thread, beside its
// own sorted list of the offsets so far; what the list lacks is merged into it and
// the tile walked again, which for a grid happens once or twice in all.  At the
// end one warp compares that list with the matrix's and adds what is new.  Latency
// bounds it (a tile's three dependent trips, ten CTAs per SM): 4.1e6 rows of seven
// entries 97 us, 1e6 of thirty 70 where the first tiles show that there is no form;
// a CTA per 128 rows with a round of barriers and reads a row apart per entry took
// 109 and 690.
constexpr int DIAG_ROWS = 128;
constexpr int DIAG_STAGE = 2048;   // entries in shared memory at once
__device__ __forceinline__ int diag_at(int i) { return i + (i >> 5); }   // (no bank conflicts)

__global__ void __launch_bounds__(DIAG_ROWS, 10)
k_diag_find(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ colind,
            const float* __restrict__ vals, int32_t n, int32_t most, DiagHead* H) {
    __shared__ int32_t s_col[DIAG_STAGE + DIAG_STAGE / 32];
    __shared__ int32_t s_val[DIAG_STAGE + DIAG_STAGE / 32];   // (bits)
    __shared__ int2 s_list[DIAG_MAX + 1];                     // offset, bits of its first value
    __shared__ int2 s_new[DIAG_MAX];
    __shared__ int s_to[DIAG_MAX];                            // where the list's entries went
    __shared__ int32_t s_first, s_end, s_bad, s_longest;
    __shared__ uint32_t s_mixed;
    const int tid = threadIdx.x, lane = tid & 31;
    if (tid <= DIAG_MAX) s_list[tid].x = DIAG_NONE;
    if (tid == 0) {
        s_mixed = 0;
        s_longest = 0;
    }
    uint32_t mixed = 0;   // bit q: entry q of the list has several values, by this thread's rows
    bool ok = true;
    // the next tile's row, and whether another CTA has seen that there is no such
    // form, are read a tile ahead
    const int32_t step = gridDim.x * DIAG_ROWS;   // (n and step: below 2^31 together)
    int32_t row0 = blockIdx.x * DIAG_ROWS, next_k = 0, next_e = 0, next_bad = 0;
    auto ahead = [&](int32_t row) {
        if (row + tid < n) {
            next_k = __ldg(rowptr + row + tid);
            next_e = __ldg(rowptr + row + tid + 1);
        }
        if (tid == 0) next_bad = *(volatile int32_t*)&H->w[0];
    };
    ahead(row0);
    for (; row0 < n; row0 += step) {
        const int32_t r = row0 + tid;
        const bool opening = row0 == (int32_t)blockIdx.x * DIAG_ROWS;
        int32_t k = 0, e = 0;
        if (tid == 0) s_bad = next_bad;
        if (r < n) {
            k = next_k;
            e = next_e;
            ok = ok && e - k <= most;
            if (tid == 0) s_first = k;
            if (tid == DIAG_ROWS - 1 || r == n - 1) s_end = e;
        }
        ahead(row0 + step);
        if (__syncthreads_or(!ok)) break;
        if (s_bad) return;
        const int32_t first = s_first, end = s_end;
        if (opening) {   // the list to start with: the longest row's
            atomicMax(&s_longest, (e - k) << 7 | tid);
            __syncthreads();
            const int len = s_longest >> 7;
            if (tid < len) {
                const int32_t rr = row0 + (s_longest & 127), kk = __ldg(rowptr + rr) + tid;
                s_list[tid] = {__ldg(colind + kk) - rr, __float_as_int(__ldg(vals + kk))};
            }
        }
        for (;;) {
            int32_t before = INT32_MIN, miss = DIAG_NONE, miss_v = 0;
            int q = 0;
            int32_t kk = k;
            __syncthreads();
            for (int32_t c0 = first, c1; c0 < end; c0 = c1) {
                c1 = c0 + min(end - c0, DIAG_STAGE);
#pragma unroll 4
                for (int32_t i = tid; i < c1 - c0; i += DIAG_ROWS) {
                    s_col[diag_at(i)] = __ldg(colind + c0 + i);
                    s_val[diag_at(i)] = __float_as_int(__ldg(vals + c0 + i));
                }
                __syncthreads();
                const int32_t stop = min(e, c1);
                for (; kk < stop; ++kk) {
                    const int i = diag_at(kk - c0);
                    const int32_t o = s_col[i] - r;
                    if (o <= before) {   // columns increase within the row
                        ok = false;
                        kk = e;
                        break;
                    }
                    before = o;
                    int2 w = s_list[q];
                    while (w.x < o) w = s_list[++q];   // (ends at DIAG_NONE)
                    if (w.x == o) {
                        if (w.y != s_val[i]) mixed |= 1u << q;
                    } else if (miss == DIAG_NONE) {
                        miss = o;
                        miss_v = s_val[i];
                    }
                }
                __syncthreads();
            }
            if (!__syncthreads_or(miss != DIAG_NONE || !ok)) break;
            if (tid < DIAG_MAX) s_new[tid].x = DIAG_NONE;
            __syncthreads();
            if (miss != DIAG_NONE) {
                int slot = 0;
                for (; slot < DIAG_MAX; ++slot) {
                    const int32_t old = atomicCAS(&s_new[slot].x, DIAG_NONE, miss);
                    if (old == DIAG_NONE || old == miss) break;
                }
                if (slot < DIAG_MAX) s_new[slot].y = miss_v;   // any of them
                ok = ok && slot < DIAG_MAX;
            }
            __syncthreads();
            if (tid < 32) {
                const int2 a = s_list[lane], b = s_new[lane];
                int to_a = lane, to_b = 0;
                for (int i = 0; i < 32; ++i) {
                    const int32_t ai = __shfl_sync(0xffffffffu, a.x, i), bi = __shfl_sync(0xffffffffu, b.x, i);
                    to_a += bi < a.x;
                    to_b += (ai < b.x) + (bi < b.x);
                }
                ok = ok && !(b.x != DIAG_NONE && to_b >= most) && !(a.x != DIAG_NONE && to_a >= most);
                if (__all_sync(0xffffffffu, ok)) {   // (most <= DIAG_MAX)
                    if (a.x != DIAG_NONE) s_list[to_a] = a;
                    if (b.x != DIAG_NONE) s_list[to_b] = b;
                    s_to[lane] = to_a;
                }
            }
            if (__syncthreads_or(!ok)) break;
            uint32_t was = mixed;
            for (mixed = 0; was; was &= was - 1) mixed |= 1u << s_to[__ffs(was) - 1];
        }
    }
    static_assert(DIAG_MAX == 32, "a bit, and a lane, for each");
    mixed = __reduce_or_sync(0xffffffffu, mixed);
    if (lane == 0) atomicOr(&s_mixed, mixed);
    if (__syncthreads_or(!ok)) {
        if (tid == 0) atomicExch(&H->w[0], 1);
        return;
    }
    if (tid >= 32) return;
    // lane i: this CTA's offset i against the list (one load), then whatever the
    // list does not have yet
    const int32_t have = *(volatile int32_t*)&H->off[lane];
    const uint32_t gmixed = *(volatile uint32_t*)&H->mixed;
    const int32_t mine = s_list[lane].x;
    int slot = -1;
    for (int i = 0; i < DIAG_MAX; ++i)
        if (__shfl_sync(0xffffffffu, have, i) == mine && mine != DIAG_NONE) slot = i;
    if (mine != DIAG_NONE && slot < 0)
        for (int i = 0; i < DIAG_MAX && slot < 0; ++i) {
            int32_t old = *(volatile int32_t*)&H->off[i];
            if (old == DIAG_NONE) old = atomicCAS(&H->off[i], DIAG_NONE, mine);
            if (old == DIAG_NONE || old == mine) slot = i;
        }
    uint32_t add = 0;
    if (mine != DIAG_NONE) {
        if (slot < 0) {
            atomicExch(&H->w[0], 1);
        } else if (!((gmixed >> slot) & 1)) {
            const uint32_t v = (uint32_t)s_list[lane].y;
            uint32_t ref = *(volatile uint32_t*)&H->ref[slot];
            if (ref == DIAG_UNSET) {
                ref = atomicCAS(&H->ref[slot], DIAG_UNSET, v);
                if (ref == DIAG_UNSET) ref = v;
            }
            if (((s_mixed >> lane) & 1) || ref != v || v == DIAG_UNSET) add = 1u << slot;
        }
    }
    add = __reduce_or_sync(0xffffffffu, add);
    if (lane == 0 && add) atomicOr(&H->mixed, add);
}

// elements of shared memory that `rows` rows of a matrix with nq offsets, `owns` of
// them with values of their own, take in diag_tile
__device__ __forceinline__ int diag_room(const int32_t* off, int nq, int owns, int rows) {
    int at = owns * rows, open = 0;
    for (int q = 0; q < nq; ++q) {
        if (q == 0 || off[q] - off[q - 1] > 16) open = q;
        if (q == nq - 1 || off[q + 1] - off[q] > 16)
            at += (rows + (off[q] - off[open]) + 8 + 3) / 4 * 4;
    }
    return at;
}

// The form itself, one row per thread, from the finished list.  A matrix whose
// tiles would not fit in shared memory (fifteen diagonals with values of their
// own) keeps the CSR steps: reading those from global memory took twice their
// time.
__global__ void __launch_bounds__(256)
k_diag_fill(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ colind,
            const float* __restrict__ vals, int32_t n, int32_t most, DiagHead* H, float* same, float* out,
            int32_t ld, void* mask, int32_t mask_bytes) {
    __shared__ int32_t s_off[DIAG_MAX];
    __shared__ unsigned s_same;
    __shared__ bool s_bad;
    const int tid = threadIdx.x;
    if (tid < 32) {
        const int32_t o = H->off[tid];
        const bool used = o != DIAG_NONE;
        const int nq = __popc(__ballot_sync(0xffffffffu, used));
        int rank = 0;
        for (int i = 0; i < DIAG_MAX; ++i) rank += __shfl_sync(0xffffffffu, o, i) < o;
        const bool one = used && !((H->mixed >> tid) & 1);
        const unsigned bits = __reduce_or_sync(0xffffffffu, one ? 1u << rank : 0u);
        if (used) s_off[rank] = o;
        __syncwarp();
        const int owns = nq - __popc(bits);
        const bool bad = nq > most || *(volatile int32_t*)&H->w[0] != 0 ||
                         diag_room(s_off, nq, owns, DIAG_TILE) > DIAG_CAP;
        if (tid == 0) {
            s_same = bits;
            s_bad = bad;
        }
        if (blockIdx.x == 0) {
            if (used) {
                H->w[4 + rank] = o;
                if (one) same[rank] = __int_as_float((int)H->ref[tid]);
            }
            if (tid == 0) {
                H->w[1] = nq;
                H->w[2] = (int32_t)bits;
                H->w[3] = diag_room(s_off, nq, owns, 2 * DIAG_TILE) <= DIAG_CAP;   // two tiles at once
                if (bad) H->w[0] = 1;
            }
        }
    }
    __syncthreads();
    if (s_bad) return;
    const unsigned same_bits = s_same;
    for (int64_t r = (int64_t)blockIdx.x * 256 + tid; r < n; r += (int64_t)gridDim.x * 256) {
        const int32_t e = __ldg(rowptr + r + 1);
        unsigned bits = 0;
        int q = 0;
        for (int32_t k = __ldg(rowptr + r); k < e; ++k, ++q) {
            const int32_t o = __ldg(colind + k) - (int32_t)r;
            while (s_off[q] != o) ++q;
            bits |= 1u << q;
            if (!((same_bits >> q) & 1)) out[(int64_t)q * ld + r] = __ldg(vals + k);
        }
        if (mask_bytes == 1)
            ((uint8_t*)mask)[r] = (uint8_t)bits;
        else if (mask_bytes == 2)
            ((uint16_t*)mask)[r] = (uint16_t)bits;
        else
            ((uint32_t*)mask)[r] = bits;
    }
}

// where a tile's diagonals lie in its shared memory, in bytes
constexpr int32_t DIAG_SAME = INT32_MIN;
struct DiagSlot {
    int32_t x;       // the first row's entry of x
    int32_t v;       // the first row's value; DIAG_SAME: the value is `same`
    float same;
    int32_t off;
};

__device__ __forceinline__ unsigned diag_bits(const DiagForm& f, int32_t r) {
    return f.mask_bytes == 1 ? __ldg((const uint8_t*)f.mask + r)
           : f.mask_bytes == 2 ? __ldg((const uint16_t*)f.mask + r)
                               : __ldg((const uint32_t*)f.mask + r);
}

__device__ __forceinline__ void bulk_to_shared(uint32_t dst, const void* src, uint32_t bytes,
                                               uint32_t bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            dst),
        "l"(src), "r"(bytes), "r"(bar)
        : "memory");
}

constexpr uint32_t DIAG_SPIN_LIMIT = 1u << 20;   // polls of a copy's barrier (some 0.1 s)

__device__ __forceinline__ bool diag_arrived(uint32_t bar) {
    for (uint32_t it = 0; it < DIAG_SPIN_LIMIT; ++it) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(bar)
            : "memory");
        if (ok) return true;
    }
    return false;
}

// A tile, or two (halves), of a step by diagonals: ROWS rows from row0, NT
// threads, thread tid on rows tid + i NT of each half.  Two at once double the
// bytes in flight and halve what a CTA pays before its copies leave (160^3 p(A)
// of 60 steps 1.63 -> 1.50 ms, 1500^2 0.81 -> 0.75 ms).  Warp 0 merges offsets less than 16 apart into windows
// of x, lays windows and values out in `sm`, and issues
// the copies: values before the wait on the previous step, windows after it
// (k_diag_fill has seen to it that they fit).
template <typename T, int OP, int NT, int RPT>
__device__ __forceinline__ void diag_tile(const StepArgs<T>& a, int32_t row0, int nrows, float* sm,
                                          DiagSlot* slot, uint64_t* bar, double& sq,
                                          const int halves) {
    constexpr int HALF = NT * RPT;
    const int ROWS = HALF * halves;
    const DiagForm& f = a.diag;
    const int tid = threadIdx.x;
    const uint32_t mb = (uint32_t)__cvta_generic_to_shared(bar);
    unsigned b[RPT];
#pragma unroll
    for (int i = 0; i < RPT; ++i)
        b[i] = tid + i * NT < nrows ? diag_bits(f, row0 + tid + i * NT) : 0;
    const int nq = __ldg(f.head + 1);
    if (tid < 32) {
        const int lane = tid;
        const unsigned same = (unsigned)__ldg(f.head + 2);
        const bool used = lane < nq;
        const int32_t o = used ? __ldg(f.head + 4 + lane) : 0;
        const int32_t before = __shfl_up_sync(0xffffffffu, o, 1);
        const bool opens = used && (lane == 0 || o - before > 16);
        const unsigned heads = __ballot_sync(0xffffffffu, opens);
        const unsigned upto = 0xffffffffu >> (31 - lane);
        const int first = 31 - __clz(heads & upto | 1u);
        const unsigned later = heads & ~upto;
        const int last = later ? __ffs(later) - 2 : nq - 1;
        const int32_t ws = __shfl_sync(0xffffffffu, o, first);
        const int32_t we = __shfl_sync(0xffffffffu, o, max(last, 0));
        // the window's elements [lo, hi) of x, on 16-byte boundaries
        const int32_t lo = max(row0 + ws, 0), hi = min(row0 + nrows + we, a.n);
        const unsigned skew = ((unsigned)(uintptr_t)(a.x + lo) & 15u) / 4;
        const unsigned bytes_to = ((unsigned)(hi - lo) + skew + 3) / 4 * 16;
        // places: windows first, then the diagonals with values of their own
        const int32_t room = opens ? (ROWS + (we - ws) + 8 + 3) / 4 * 4 : 0;
        int32_t end = room;
#pragma unroll
        for (int s = 1; s < 32; s <<= 1) {
            const int32_t v = __shfl_up_sync(0xffffffffu, end, s);
            if (lane >= s) end += v;
        }
        const int32_t at = __shfl_sync(0xffffffffu, end - room, first);
        const int32_t xs = __shfl_sync(0xffffffffu, end, 31);
        const bool own = used && !((same >> lane) & 1);
        const unsigned owns = __ballot_sync(0xffffffffu, own);
        const int32_t vat = xs + __popc(owns & (upto >> 1)) * ROWS;
        if (used)
            slot[lane] = {(at + (int32_t)skew + (row0 + o - lo)) * 4, own ? vat * 4 : DIAG_SAME,
                          own ? 0.0f : __ldg(f.same + lane), o};
        const uint32_t bytes = opens && hi > lo ? bytes_to : 0;
        const uint32_t total = __reduce_add_sync(0xffffffffu, bytes) + __popc(owns) * (ROWS * 4u);
        if (lane == 0) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mb) : "memory");
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mb),
                         "r"(total)
                         : "memory");
        }
        __syncwarp();
        const uint32_t base = (uint32_t)__cvta_generic_to_shared(sm);
        if (own)
            bulk_to_shared(base + vat * 4, f.vals + (int64_t)lane * f.ld + row0, ROWS * 4, mb);
        // the vectors written by the previous step are complete and visible
        asm volatile("griddepcontrol.wait;" ::: "memory");
        if (bytes) bulk_to_shared(base + at * 4, a.x + lo - (int)skew, bytes, mb);
    } else {
        asm volatile("griddepcontrol.wait;" ::: "memory");
    }
    bool ready = false;
    for (int h = 0;;) {
        T e0[RPT], e1[RPT], e2[RPT], acc[RPT];
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
            e0[i] = e1[i] = e2[i] = acc[i] = T(0);
            const int64_t r = (int64_t)row0 + tid + i * NT;
            if (tid + i * NT < nrows) {
                if (a.a0) e0[i] = __ldg(a.a0 + r);
                if (a.a1 && !(a.flags & F_PZERO)) e1[i] = a.a1[r];
                if (a.a2 && (a.flags & F_FINAL)) e2[i] = __ldg(a.a2 + r);
            }
        }
        // rows that lack a diagonal only where a grid ends: most warps have none
        const unsigned all = 0xffffffffu >> (32 - nq);
        bool whole = true;
#pragma unroll
        for (int i = 0; i < RPT; ++i) whole = whole && b[i] == all;
        whole = __all_sync(0xffffffffu, whole);
        if (h == 0) {
            __syncthreads();
            // (one answer for the warp: its lanes poll apart, the sums below are the warp's)
            ready = __all_sync(0xffffffffu, diag_arrived(mb));
        }
        if (ready) {
            const char* me = reinterpret_cast<const char*>(sm + tid);
            auto at = [&](int32_t off, int i) {
                return *reinterpret_cast<const float*>(me + off + i * NT * (int)sizeof(float));
            };
            if (whole) {
#pragma unroll 4
                for (int q = 0; q < nq; ++q) {
                    const DiagSlot s = slot[q];
#pragma unroll
                    for (int i = 0; i < RPT; ++i)
                        acc[i] = fma(s.v == DIAG_SAME ? s.same : at(s.v, i), at(s.x, i), acc[i]);
                }
            } else {
#pragma unroll 4
                for (int q = 0; q < nq; ++q) {
                    const DiagSlot s = slot[q];
#pragma unroll
                    for (int i = 0; i < RPT; ++i)
                        if ((b[i] >> q) & 1)
                            acc[i] = fma(s.v == DIAG_SAME ? s.same : at(s.v, i), at(s.x, i), acc[i]);
                }
            }
        } else {   // the copies did not arrive: from global memory
            for (int q = 0; q < nq; ++q) {
                const DiagSlot s = slot[q];
#pragma unroll
                for (int i = 0; i < RPT; ++i)
                    if ((b[i] >> q) & 1) {
                        const int64_t r = (int64_t)row0 + tid + i * NT;
                        acc[i] = fma(s.v == DIAG_SAME ? s.same : __ldg(f.vals + (int64_t)q * f.ld + r),
                                     __ldg(a.x + r + s.off), acc[i]);
                    }
            }
            diag_arrived(mb);   // nothing may land in this CTA's memory after it
        }
#pragma unroll
        for (int i = 0; i < RPT; ++i)
            if (tid + i * NT < nrows)
                step_epilogue<T, OP>(a, (int64_t)row0 + tid + i * NT, acc[i], e0[i], e1[i], e2[i], sq);
        if (++h == halves) break;
        row0 += HALF;
        nrows -= HALF;
        sm += HALF;
#pragma unroll
        for (int i = 0; i < RPT; ++i)
            b[i] = tid + i * NT < nrows ? diag_bits(f, row0 + tid + i * NT) : 0;
    }
}

// A tile of k_spmv_step that has long rows, its row pointers in srp: ordinary rows
// by a thread each, long rows from the staged chunks.
template <typename T, int OP>
__device__ __forceinline__ double long_tile(const StepArgs<T>& a, int64_t row0, int nrows, T* sval,
                                            int32_t* scol, const int32_t* srp) {
    constexpr int NT = step_threads<T>(), RPT = step_rpt<T>(), ROWS = NT * RPT;
    constexpr int CHUNK = step_chunk<T>() - ROWS - 64;   // the long rows' sums lie behind it
    static_assert(CHUNK % 4 == 0, "16-byte granules");
    T* const sum = sval + CHUNK + 4;
    const int tid = threadIdx.x;
    const int32_t k0 = srp[0], k1 = srp[nrows];
    T acc[RPT];
#pragma unroll
    for (int q = 0; q < RPT; ++q) acc[q] = T(0);
    T *from = sum + ROWS, *left = from + 32;
    for (int32_t c0 = k0, c1; c0 < k1; c0 = c1) {
        c1 = c0 + min(k1 - c0, CHUNK);
        const int32_t base = c0 & ~3;
        if (c0 != k0) __syncthreads();
        stage_chunk<T>(sval, scol, a.vals, a.colind, base, c0, c1, tid, NT,
                       l2_policy((a.flags & F_KEEP_A) || row0 < a.keep_rows));
        // the vectors written by the previous step are complete and visible
        if (c0 == k0) asm volatile("griddepcontrol.wait;" ::: "memory");
        cp_async_wait_all();
        __syncthreads();
#pragma unroll
        for (int q = 0; q < RPT; ++q) {
            const int t = tid + q * NT;
            if (t < nrows && srp[t + 1] - srp[t] <= LONG_ROW)
                acc[q] = row_dot<T, true>(sval, scol, a.x, max(srp[t], c0) - base,
                                          min(srp[t + 1], c1) - base, acc[q]);
        }
        long_rows_staged<T, NT / 32, ROWS>(srp, sval - base, scol - base, a.x, nrows, c0, c1, sum, from, left);
        T* const was = from;
        from = left;
        left = was;
    }
    __syncthreads();
    double sq = 0.0;
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
        const int t = tid + q * NT;
        if (t < nrows) {
            const int64_t r = row0 + t;
            const T e0 = a.a0 ? __ldg(a.a0 + r) : T(0);
            const T e1 = (a.a1 && !(a.flags & F_PZERO)) ? a.a1[r] : T(0);
            const T e2 = (a.a2 && (a.flags & F_FINAL)) ? __ldg(a.a2 + r) : T(0);
            step_epilogue<T, OP>(a, r, srp[t + 1] - srp[t] > LONG_ROW ? sum[t] : acc[q], e0, e1, e2, sq);
        }
    }
    return sq;
}

// DG: the (FP32) matrix is at hand by its diagonals too, if it has that form
// LR: a tile with long rows sums them from its staged chunks (long_tile), else they
// are read a second time (long_rows)
template <typename T, int OP, bool DG, bool LR>
__global__ void __launch_bounds__(step_threads<T>(), DG || LR ? WIDE_CTAS : step_min_ctas<T, OP>())
k_spmv_step(const StepArgs<T> a) {
    constexpr int NT = step_threads<T>();      // threads per CTA
    // staging copies start at a chunk base rounded down to 4 elements
    constexpr int PAD = 4;
    constexpr int RPT = step_rpt<T>();
    constexpr int ROWS = NT * RPT;      // rows per CTA
    constexpr int CHUNK = step_chunk<T>();     // nonzeros staged per chunk
    __shared__ __align__(16) unsigned char stage[(CHUNK + PAD) * (sizeof(T) + 4)];
    T* sval = reinterpret_cast<T*>(stage);
    int32_t* scol = reinterpret_cast<int32_t*>(stage + (CHUNK + PAD) * sizeof(T));
    __shared__ int32_t srp[ROWS + 1];
    __shared__ double sred[NT / 32];

    const int64_t row0 = (int64_t)blockIdx.x * ROWS;
    const int tid = threadIdx.x;
    const int nrows = (int)(((int64_t)a.n - row0) < ROWS ? ((int64_t)a.n - row0) : ROWS);
    // L2 hint of the staging copies: evict-last for a matrix held in L2 (all
    // of it, or the leading rows), else evict-first (the policy is created
    // at each use, so that it holds no registers across the kernel)
    const bool keep = (a.flags & F_KEEP_A) || row0 < a.keep_rows;
    // Programmatic dependent launch: the next step in the stream may start
    // now; everything up to griddepcontrol.wait reads only the matrix, which
    // no step writes, so it overlaps the previous step's tail.
    asm volatile("griddepcontrol.launch_dependents;");
    static_assert(!DG || OP != OP_RESID, "residuals take the matrix in FP64");
    if constexpr (DG) {
        if (__ldg(a.diag.head) == 0) {   // uniform over the grid
            __shared__ __align__(16) DiagSlot slot[DIAG_MAX];
            __shared__ uint64_t bar;
            double sq = 0.0;
            int halves = 1, rows = nrows;
            if (__ldg(a.diag.head + 3)) {   // two tiles on every other CTA
                if (blockIdx.x & 1) return;
                halves = (int64_t)a.n - row0 > ROWS ? 2 : 1;
                rows = (int)min((int64_t)a.n - row0, (int64_t)2 * ROWS);
            }
            diag_tile<T, OP, NT, RPT>(a, (int32_t)row0, rows, (float*)stage, slot, &bar, sq, halves);
            return;
        }
    }
    // the tile that a CTA half a resident wave later stages: its nonzero
    // range is read now, beside this tile's row pointers.  CTAs near the end
    // of the grid prefetch the matrix tiles at the start of the next step
    // instead (a chain's next step reads the same matrix).
    int64_t prow = row0 + (int64_t)a.pf_ahead * ROWS;
    const bool wrap = prow >= a.n;
    if (wrap) prow -= (int64_t)gridDim.x * ROWS;
    const bool pf = tid == 0 && a.pf_ahead > 0 && prow >= 0 && prow < a.n;
    const int64_t prow1 = min(prow + ROWS, (int64_t)a.n);
    int32_t pk0 = 0, pk1 = 0;
    if (pf) {
        pk0 = __ldg(a.rowptr + prow);
        pk1 = __ldg(a.rowptr + prow1);
    }
    if constexpr (LR) {
        bool any = false;
        for (int i = tid; i <= nrows; i += NT) {
            const int32_t k = __ldg(a.rowptr + row0 + i);
            srp[i] = k;
            any = any || (i < nrows && __ldg(a.rowptr + row0 + i + 1) - k > LONG_ROW);
        }
        if (__syncthreads_or(any)) {
            const double sq = long_tile<T, OP>(a, row0, nrows, sval, scol, srp);
            if constexpr (OP == OP_RESID) block_sq<NT>(sq, sred, a.part);
            return;
        }
    } else {
        for (int i = tid; i <= nrows; i += NT) srp[i] = __ldg(a.rowptr + row0 + i);
        __syncthreads();
    }
    const int32_t k0 = srp[0];
    const int32_t k1 = srp[nrows];
    // thread tid owns rows tid and (RPT = 2) tid + NT of the tile
    int32_t my_lo[RPT], my_hi[RPT];
    bool is_long[RPT];
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
        const int t = tid + q * NT;
        my_lo[q] = (t < nrows) ? srp[t] : k1;
        my_hi[q] = (t < nrows) ? srp[t + 1] : k1;
        is_long[q] = !LR && my_hi[q] - my_lo[q] > LONG_ROW;
        if (is_long[q]) my_hi[q] = my_lo[q];   // (long_rows below)
    }
    // element k of the current chunk sits at sval / scol [k - base], base =
    // c0 & ~3
    {
        const int32_t c1 = min(k1, k0 + CHUNK);
        const int32_t base = k0 & ~3;
        stage_chunk<T>(sval, scol, a.vals, a.colind, base, k0, c1, tid, NT,
                       l2_policy(keep));
    }
    if (pf) {
        if (prow >= a.keep_rows) {   // (the leading rows' nonzeros are held in L2)
            prefetch_l2(a.vals + pk0, a.vals + pk1);
            prefetch_l2(a.colind + pk0, a.colind + pk1);
        }
        // and its row pointers, which the CTA reads first, before anything
        // else can start (3-D 160^3 FP32 chains -4 %)
        prefetch_l2(a.rowptr + prow, a.rowptr + prow1 + 1);
    }
    // the vectors written by the previous step are complete and visible
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (pf && !wrap) {
        prefetch_l2(a.x + prow, a.x + prow1);
        if (a.a0) prefetch_l2(a.a0 + prow, a.a0 + prow1);
        if (a.a1 && !(a.flags & F_PZERO)) prefetch_l2(a.a1 + prow, a.a1 + prow1);
        if (a.a2 && (a.flags & F_FINAL)) prefetch_l2(a.a2 + prow, a.a2 + prow1);
    }

    // The epilogue's row-aligned inputs do not depend on the product: load
    // them now, so their latency overlaps the staging and the gathers.
    T e0[RPT], e1[RPT], e2[RPT], acc[RPT];
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
        e0[q] = e1[q] = e2[q] = acc[q] = T(0);
        const int t = tid + q * NT;
        if (t < nrows) {
            const int64_t rr = row0 + t;
            if (a.a0) e0[q] = __ldg(a.a0 + rr);
            if (a.a1 && !(a.flags & F_PZERO)) e1[q] = a.a1[rr];
            if (a.a2 && (a.flags & F_FINAL)) e2[q] = __ldg(a.a2 + rr);
        }
    }

    for (int32_t c0 = k0; c0 < k1; c0 += CHUNK) {
        const int32_t c1 = min(k1, c0 + CHUNK);
        const int32_t base = c0 & ~3;
        if (c0 != k0) {   // the first chunk was issued before the wait
            stage_chunk<T>(sval, scol, a.vals, a.colind, base, c0, c1, tid, NT,
                           l2_policy(keep));
        }
        cp_async_wait_all();
        __syncthreads();
        // exactly one FMA per nonzero (GB300 issues two FP64 operations per
        // clock per SM); summation stays in column order within each row.
        // The last 1-3 nonzeros: FP32 issues their gathers together; FP64
        // takes them one at a time (the wider form took 40 registers, 6
        // instead of 8 CTAs per SM, and measured 13 % slower on 2-D chains).
        if constexpr (RPT == 1) {
            const int32_t lo = max(my_lo[0], c0) - base;
            const int32_t hi = min(my_hi[0], c1) - base;
            acc[0] = row_dot<T, sizeof(T) == 4>(sval, scol, a.x, lo, hi, acc[0]);
        } else {
            // two rows: their four-wide batches in lockstep (eight gathers
            // in flight), then each row's remainder
            int32_t ka = max(my_lo[0], c0) - base, kb = max(my_lo[1], c0) - base;
            const int32_t ha = min(my_hi[0], c1) - base, hb = min(my_hi[1], c1) - base;
            for (; ka + 4 <= ha && kb + 4 <= hb; ka += 4, kb += 4) {
                const T va0 = sval[ka], va1 = sval[ka + 1], va2 = sval[ka + 2], va3 = sval[ka + 3];
                const T vb0 = sval[kb], vb1 = sval[kb + 1], vb2 = sval[kb + 2], vb3 = sval[kb + 3];
                const T xa0 = __ldg(a.x + scol[ka]), xa1 = __ldg(a.x + scol[ka + 1]);
                const T xa2 = __ldg(a.x + scol[ka + 2]), xa3 = __ldg(a.x + scol[ka + 3]);
                const T xb0 = __ldg(a.x + scol[kb]), xb1 = __ldg(a.x + scol[kb + 1]);
                const T xb2 = __ldg(a.x + scol[kb + 2]), xb3 = __ldg(a.x + scol[kb + 3]);
                acc[0] = fma(va3, xa3, fma(va2, xa2, fma(va1, xa1, fma(va0, xa0, acc[0]))));
                acc[1] = fma(vb3, xb3, fma(vb2, xb2, fma(vb1, xb1, fma(vb0, xb0, acc[1]))));
            }
            acc[0] = row_dot<T, true>(sval, scol, a.x, ka, ha, acc[0]);
            acc[1] = row_dot<T, true>(sval, scol, a.x, kb, hb, acc[1]);
        }
        // the staged chunk is read by every thread: a barrier before it is
        // overwritten, none after the last one (3-D 160^3 chains +0.2 %)
        if (c0 + CHUNK < k1) __syncthreads();
    }

    double sq = 0.0;
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
        const int t = tid + q * NT;
        if (t < nrows && !is_long[q])
            step_epilogue<T, OP>(a, row0 + t, acc[q], e0[q], e1[q], e2[q], sq);
    }
    if constexpr (!LR) {
#pragma unroll
        for (int q = 0; q < RPT; ++q) long_rows<T, OP>(a, row0 + tid + q * NT, is_long[q], sq);
    }
    if constexpr (OP == OP_RESID) block_sq<NT>(sq, sred, a.part);
}

// Direct-read step: the same step, one row per thread, the row's matrix
// entries read straight into registers (up to PRE of them) before the wait
// on the previous step -- no shared-memory staging round, so the latency
// chain of a step is row pointers -> (wait) -> gathers -> epilogue.  The
// sums and the epilogue are k_spmv_step's: bit-identical results.  Two uses:
// * small systems (PRE = 8, no register bound): a step is a handful of CTAs,
//   and latency, not bytes, sets its time;
// * a matrix held in L2 (F_KEEP_A; the preloads carry the evict-last hint):
//   the staging round trip is then the longer path.  2-D 1000^2 FP64 chains
//   57.3 -> 55.2 ms.  launch_step chooses PRE and the registers.
// MINB: minimum CTAs per SM given to __launch_bounds__ (0: no register bound).
// One row per thread of any CTA size up to SPMV_ROWS; the residual's partial
// sums are one per CTA.
template <typename T>
__device__ __forceinline__ T ld_hint(const T* p, uint64_t pol);
template <>
__device__ __forceinline__ double ld_hint<double>(const double* p, uint64_t pol) {
    double v;
    asm volatile("ld.global.nc.L2::cache_hint.f64 %0, [%1], %2;" : "=d"(v) : "l"(p), "l"(pol));
    return v;
}
template <>
__device__ __forceinline__ float ld_hint<float>(const float* p, uint64_t pol) {
    float v;
    asm volatile("ld.global.nc.L2::cache_hint.f32 %0, [%1], %2;" : "=f"(v) : "l"(p), "l"(pol));
    return v;
}
template <>
__device__ __forceinline__ int32_t ld_hint<int32_t>(const int32_t* p, uint64_t pol) {
    int32_t v;
    asm volatile("ld.global.nc.L2::cache_hint.s32 %0, [%1], %2;" : "=r"(v) : "l"(p), "l"(pol));
    return v;
}

constexpr int DIRECT_SMALL_ROWS = 64;   // rows (threads) per CTA, up to one such CTA per SM
constexpr int DIRECT_L2_ROWS = 128;     // ... above that
// Rows of many entries in a small system: SPREAD_ROWS of them to a warp, so that
// there are more warps, and that a warp with long rows has fewer to sum in turn (40
// FP64 steps, 32 rows to a warp / 4: 400 rows of 150 1450 / 346 us, with one thread
// to a row 477; 1,000 of 60 232 / 199; 2,500 of 24 142 / 116; below that it loses: FP32,
// 10,000 of 18 89 / 110).
constexpr int SPREAD_ROWS = 4;
constexpr double SPREAD_AVG = 22.0;
constexpr int LATE_MAX = 6, EVEN_MAX = 10;   // CTAs per SM (launch_step)

// LATE: lets the next step in when the previous one is done (launch_step); chosen
// inside the kernel it cost 40 steps at 1000^2 0.2 %
template <typename T, int OP, int PRE, int MINB, bool HINT, bool LATE>
__global__ void __launch_bounds__(SPMV_ROWS, MINB)
k_spmv_direct(const __grid_constant__ StepArgs<T> a) {
    __shared__ double sred[SPMV_ROWS / 32];
    const int tid = threadIdx.x;
    // a row to a lane; rows of many entries, in a small system, to the first few
    // lanes of a warp (launch_step)
    int64_t r = (int64_t)blockIdx.x * blockDim.x + tid;
    bool live = r < a.n;
    if (!HINT && OP != OP_RESID && (a.flags & F_SPREAD)) {
        r = (r >> 5) * SPREAD_ROWS + (tid & 31);
        live = (tid & 31) < SPREAD_ROWS && r < a.n;
    }
    if constexpr (!LATE) asm volatile("griddepcontrol.launch_dependents;");
    int32_t k0 = 0, k1 = 0;
    T pv[PRE];
    int32_t pc[PRE];
    if (live) {
        k0 = __ldg(a.rowptr + r);
        k1 = __ldg(a.rowptr + r + 1);
#pragma unroll
        for (int q = 0; q < PRE; ++q) {
            if (k0 + q < k1) {
                if constexpr (HINT) {
                    pv[q] = ld_hint<T>(a.vals + k0 + q, l2_policy(1));
                    pc[q] = ld_hint<int32_t>(a.colind + k0 + q, l2_policy(1));
                } else {
                    pv[q] = __ldg(a.vals + k0 + q);
                    pc[q] = __ldg(a.colind + k0 + q);
                }
            }
        }
    }
    const unsigned longs = HINT ? 0 : __ballot_sync(0xffffffffu, k1 - k0 > LONG_ROW);
    // the vectors written by the previous step are complete and visible
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if constexpr (LATE) asm volatile("griddepcontrol.launch_dependents;");
    double sq = 0.0;
    const bool is_long = k1 - k0 > LONG_ROW;
    if (live) {
        if (is_long) k1 = k0;   // (long_rows below)
        const T e0 = a.a0 ? __ldg(a.a0 + r) : T(0);
        const T e1 = (a.a1 && !(a.flags & F_PZERO)) ? a.a1[r] : T(0);
        const T e2 = (a.a2 && (a.flags & F_FINAL)) ? __ldg(a.a2 + r) : T(0);
        T xg[PRE];
#pragma unroll
        for (int q = 0; q < PRE; ++q)
            if (k0 + q < k1) xg[q] = __ldg(a.x + pc[q]);
        T acc = T(0);
#pragma unroll
        for (int q = 0; q < PRE; ++q)
            if (k0 + q < k1) acc = fma(pv[q], xg[q], acc);
        // (entries past PRE without the hint: mostly in the lines the hinted
        // loads already brought in)
        for (int32_t k = k0 + PRE; k < k1; ++k)
            acc = fma(__ldg(a.vals + k), __ldg(a.x + __ldg(a.colind + k)), acc);
        if (!is_long) step_epilogue<T, OP>(a, r, acc, e0, e1, e2, sq);
    }
    if constexpr (HINT) {
        long_rows<T, OP>(a, r, is_long, sq);
    } else {
        if (longs) sq += long_rows_call<T, OP>(a, (int32_t)r, longs);
    }
    if constexpr (OP == OP_RESID) {
        for (int off = 16; off > 0; off >>= 1) sq += __shfl_down_sync(0xffffffffu, sq, off);
        if ((tid & 31) == 0) sred[tid >> 5] = sq;
        __syncthreads();
        if (tid == 0) {
            double t = 0.0;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sred[w];
            a.part[blockIdx.x] = t;
        }
    }
}

// A root step whose operator product s = (M x)[r] was computed beforehand
// (M a composite operator such as phi_1(A)): the same epilogue as the
// fused kernel, one thread per row.
template <typename T, int OP>
__global__ void __launch_bounds__(SPMV_ROWS)
k_ew_step(const StepArgs<T> a, const T* __restrict__ prodv) {
    __shared__ double sred[SPMV_ROWS / 32];
    const int tid = threadIdx.x;
    const int64_t r = (int64_t)blockIdx.x * SPMV_ROWS + tid;
    const bool live = r < a.n;
    double sq = 0.0;
    if (live) {
        const T e0 = a.a0 ? __ldg(a.a0 + r) : T(0);
        const T e1 = (a.a1 && !(a.flags & F_PZERO)) ? a.a1[r] : T(0);
        const T e2 = (a.a2 && (a.flags & F_FINAL)) ? __ldg(a.a2 + r) : T(0);
        step_epilogue<T, OP>(a, r, __ldg(prodv + r), e0, e1, e2, sq);
    }
    if constexpr (OP == OP_RESID) {
        for (int off = 16; off > 0; off >>= 1) sq += __shfl_down_sync(0xffffffffu, sq, off);
        if ((tid & 31) == 0) sred[tid >> 5] = sq;
        __syncthreads();
        if (tid == 0) {
            double t = 0.0;
            for (int w = 0; w < SPMV_ROWS / 32; ++w) t += sred[w];
            a.part[blockIdx.x] = t;
        }
    }
}

template <typename T>
int32_t launch_ew_step(int op, const StepArgs<T>& a, const T* prodv, cudaStream_t s) {
    if (a.n <= 0) return 0;
    const int grid = (a.n + SPMV_ROWS - 1) / SPMV_ROWS;
    switch (op) {
        case OP_RESID: k_ew_step<T, OP_RESID><<<grid, SPMV_ROWS, 0, s>>>(a, prodv); break;
        case OP_PHI_REAL: k_ew_step<T, OP_PHI_REAL><<<grid, SPMV_ROWS, 0, s>>>(a, prodv); break;
        case OP_PHI_PAIR2: k_ew_step<T, OP_PHI_PAIR2><<<grid, SPMV_ROWS, 0, s>>>(a, prodv); break;
        case OP_P_REAL: k_ew_step<T, OP_P_REAL><<<grid, SPMV_ROWS, 0, s>>>(a, prodv); break;
        case OP_P_PAIR1: k_ew_step<T, OP_P_PAIR1><<<grid, SPMV_ROWS, 0, s>>>(a, prodv); break;
        case OP_P_PAIR2: k_ew_step<T, OP_P_PAIR2><<<grid, SPMV_ROWS, 0, s>>>(a, prodv); break;
        default: return PPG_ERR_ARG;
    }
    ++g_launches;
    int32_t rc = check_launch("k_ew_step");
    return rc < 0 ? rc : grid;
}

template int32_t launch_ew_step<double>(int, const StepArgs<double>&, const double*,
                                        cudaStream_t);

// An upper bound on the partial sums a residual step of n rows writes (one
// per CTA): the smallest tile of any kernel that computes one (the staged
// FP64 step's 128 rows; the direct step's residual keeps 256-row CTAs)
int32_t spmv_grid_blocks(int32_t n) {
    constexpr int r64 = step_threads<double>() * step_rpt<double>();
    constexpr int r32 = step_threads<float>() * step_rpt<float>();
    constexpr int rmin = r64 < r32 ? (r64 < SPMV_ROWS ? r64 : SPMV_ROWS) : (r32 < SPMV_ROWS ? r32 : SPMV_ROWS);
    return (int32_t)(((int64_t)n + rmin - 1) / rmin);
}

// Reserve L2 for evict-last (persisting) lines on the current device: without
// a set-aside the evict-last hint is treated as normal.  This is a limit of
// this process's context on that device; it ends with the process.  A
// chain over a matrix too large for L2 sets it to kPartialL2 instead
// (set_l2_exact).  Returns the set-aside now in place.
constexpr int kL2Devices = 64;
static std::atomic<size_t> g_l2_reserved[kL2Devices];   // set-aside in place
static std::atomic<size_t> g_l2_asked[kL2Devices];      // what set_l2_exact asked for
static std::atomic<int> g_l2_bytes[kL2Devices];

static int current_device() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kL2Devices) {
        cudaGetLastError();
        return -1;
    }
    return dev;
}

static size_t reserve_l2_for(int dev, size_t bytes, cudaStream_t s) {
    const size_t have = g_l2_reserved[dev].load(std::memory_order_relaxed);
    if (bytes <= have || stream_capturing(s)) return have;
    int maxp = 0;
    if (cudaDeviceGetAttribute(&maxp, cudaDevAttrMaxPersistingL2CacheSize, dev) != cudaSuccess ||
        maxp <= 0) {
        cudaGetLastError();
        return have;
    }
    const size_t want = bytes < (size_t)maxp ? bytes : (size_t)maxp;
    size_t got = have;
    if (want > have && cudaDeviceSetLimit(cudaLimitPersistingL2CacheSize, want) == cudaSuccess &&
        cudaDeviceGetLimit(&got, cudaLimitPersistingL2CacheSize) == cudaSuccess) {
        g_l2_reserved[dev].store(got, std::memory_order_relaxed);
        g_l2_asked[dev].store(0, std::memory_order_relaxed);
    }
    cudaGetLastError();
    return g_l2_reserved[dev].load(std::memory_order_relaxed);
}

// Set the set-aside to `bytes` exactly (shrinking or growing it; persisting
// lines back to normal first).  Returns the set-aside now in place (the
// driver rounds the request to its granularity).
static size_t set_l2_exact(int dev, size_t bytes, cudaStream_t s) {
    const size_t have = g_l2_reserved[dev].load(std::memory_order_relaxed);
    if (g_l2_asked[dev].load(std::memory_order_relaxed) == bytes || stream_capturing(s)) return have;
    int maxp = 0;
    if (cudaDeviceGetAttribute(&maxp, cudaDevAttrMaxPersistingL2CacheSize, dev) != cudaSuccess ||
        maxp <= 0) {
        cudaGetLastError();
        return have;
    }
    const size_t want = bytes < (size_t)maxp ? bytes : (size_t)maxp;
    cudaCtxResetPersistingL2Cache();
    size_t got = have;
    if (cudaDeviceSetLimit(cudaLimitPersistingL2CacheSize, want) == cudaSuccess &&
        cudaDeviceGetLimit(&got, cudaLimitPersistingL2CacheSize) == cudaSuccess) {
        g_l2_reserved[dev].store(got, std::memory_order_relaxed);
        g_l2_asked[dev].store(bytes, std::memory_order_relaxed);
    }
    cudaGetLastError();
    return g_l2_reserved[dev].load(std::memory_order_relaxed);
}

// Set-aside a chain over a matrix too large for L2 holds its leading rows in.
// Measured on the 3-D 160^3 chains with an unused set-aside (FP32 / FP64
// GB/s): none 6032 / 6150, 48 MB 6018 / 6147, 67 MB 5357 / 6032, 80 MB
// 4646 / 5604: up to about 48 MB the streamed part loses next to nothing.
constexpr size_t kPartialL2 = (size_t)48 << 20;

static int l2_bytes(int dev) {
    int l2 = g_l2_bytes[dev].load(std::memory_order_relaxed);
    if (l2 == 0) {
        int v = 0;
        if (cudaDeviceGetAttribute(&v, cudaDevAttrL2CacheSize, dev) != cudaSuccess || v <= 0) {
            cudaGetLastError();
            v = -1;
        }
        g_l2_bytes[dev].store(v, std::memory_order_relaxed);
        l2 = v;
    }
    return l2;
}

// a chain's matrix and vectors fit comfortably in L2
static bool fits_l2(double bytes, int l2) { return bytes <= 0.8 * (double)l2; }

int row_flags(int64_t n, int64_t nnz) {
    return ((double)nnz > 5.5 * (double)n ? F_WIDE : 0) | ((double)nnz > LONG_AVG * (double)n ? F_LONG : 0) |
           ((double)nnz > SPREAD_AVG * (double)n ? F_SPREAD : 0);
}

int keep_a_flag(int64_t n, int64_t nnz, int elem, int nvec, cudaStream_t s, bool may_reserve,
                int32_t* keep_rows) {
    if (keep_rows) *keep_rows = 0;
    const int dev = current_device();
    if (dev < 0) return 0;
    const int l2 = l2_bytes(dev);
    if (l2 <= 0 || n <= 0) return 0;
    const double a_bytes = (double)nnz * (elem + 4) + 4.0 * (n + 1);
    const double bytes = a_bytes + (double)nvec * n * elem;
    const int rows = row_flags(n, nnz);
    if (!fits_l2(bytes, l2)) {
        // streaming: a chain holds the nonzeros of its leading rows in a
        // set-aside of kPartialL2 (shrinking a larger one that an L2-resident
        // workload left: an unused 76 MB set-aside cost the 160^3 FP32 chains
        // 11 %), and streams the rest
        if (!keep_rows) return rows;
        const size_t have = may_reserve ? set_l2_exact(dev, kPartialL2, s)
                                        : g_l2_reserved[dev].load(std::memory_order_relaxed);
        const double held = 0.9 * (double)have / (a_bytes / (double)n);
        *keep_rows = (int32_t)(held < (double)n ? held : (double)n);
        return rows;
    }
    const size_t need = (size_t)(a_bytes * 1.05);
    if (may_reserve) {
        reserve_l2_for(dev, need, s);
        return F_KEEP_A | rows;
    }
    // no change to the context: the hint only where a set-aside exists
    return rows | (g_l2_reserved[dev].load(std::memory_order_relaxed) >= need ? F_KEEP_A : 0);
}

// CTAs of the root-step kernel resident at once (occupancy x SMs), per
// device and form of the kernel
template <typename T, bool DG, bool LR>
static int step_resident_ctas() {
    static std::atomic<int> cached[16];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 16) dev = 0;
    int v = cached[dev].load(std::memory_order_relaxed);
    if (v == 0) {
        int occ = 0, sms = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_spmv_step<T, OP_P_REAL, DG, LR>,
                                                          step_threads<T>(), 0) != cudaSuccess ||
            occ < 1)
            occ = 1;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
            sms < 1)
            sms = 1;
        cudaGetLastError();
        v = occ * sms;
        cached[dev].store(v, std::memory_order_relaxed);
    }
    return v;
}

// The diagonal form is tried with at most as many diagonals as keep it below
// the CSR's bytes (an entry without its column index), where the steps to come
// repay building it: two passes over the matrix, 135 us at 160^3 (165 us with values
// of their own to write).  Per step, CSR against diagonals (one value per diagonal /
// values of their own):
//   160^3:     49 us   22.5 us / 34 us   (repaid by 5 and 11 steps)
// A matrix held in L2 stays with the direct steps: by diagonals a grid would gain
// (1000^2, 60 steps: 0.53 -> 0.38 ms), but whether it is one is known on the device
// alone, and a matrix that is not would lose more than the direct steps' gain
// (1.2e6 rows of seven random entries, 60 steps: 0.76 -> 1.07 ms).
constexpr int64_t DIAG_MIN_STEPS = 20;

// Scratch that a call can do without: out of what the pool holds, or at most an
// eighth of the device's free memory, since the pool keeps what it has once taken
// and another allocator's next request would go without.  (In a capture the memory
// is the graph's, and the device must not be asked.)
static bool scratch_at_hand(int dev, size_t need, cudaStream_t s) {
    if (stream_capturing(s)) return true;
    cudaMemPool_t pool;
    uint64_t held = 0, used = 0;
    size_t free_bytes = 0, total = 0;
    const bool ok = cudaDeviceGetDefaultMemPool(&pool, dev) == cudaSuccess &&
                    cudaMemPoolGetAttribute(pool, cudaMemPoolAttrReservedMemCurrent, &held) == cudaSuccess &&
                    cudaMemPoolGetAttribute(pool, cudaMemPoolAttrUsedMemCurrent, &used) == cudaSuccess &&
                    (held - used >= need ||
                     (cudaMemGetInfo(&free_bytes, &total) == cudaSuccess && need <= free_bytes / 8));
    cudaGetLastError();
    return ok;
}

int32_t DiagStore::build(const int32_t* rowptr, const int32_t* colind, const float* vals, int32_t n,
                         int64_t nnz, int64_t steps, cudaStream_t stream) {
    if (n <= DIRECT_MAX_N || n > (1 << 30) || steps < DIAG_MIN_STEPS || nnz < n) return PPG_OK;
    const int dev = current_device();
    if (dev < 0) return PPG_OK;
    if (fits_l2(8.0 * nnz + 16.0 * n, l2_bytes(dev))) return PPG_OK;
    const double avg = (double)nnz / (double)n;
    const int most = (int)std::min<double>(DIAG_MAX, 2.0 * avg + 0.5);
    if (avg > most) return PPG_OK;
    const int32_t ld = (n + DIAG_PAD - 1) / DIAG_PAD * DIAG_PAD;
    f.mask_bytes = most <= 8 ? 1 : most <= 16 ? 2 : 4;
    const size_t b_vals = (size_t)most * ld * sizeof(float);
    const size_t need = 1024 + b_vals + (size_t)ld * f.mask_bytes;
    if (!scratch_at_hand(dev, need, stream) || cudaMallocAsync(&mem, need, stream) != cudaSuccess) {
        cudaGetLastError();   // the CSR steps need none of it
        mem = nullptr;
        return PPG_OK;
    }
    static_assert(sizeof(DiagHead) <= 768, "the head's place");
    s = stream;
    char* m = (char*)mem;
    DiagHead* H = (DiagHead*)m;
    f.same = (const float*)(m + 768);
    f.vals = (const float*)(m + 1024);
    f.mask = m + 1024 + b_vals;
    f.ld = ld;
    k_diag_init<<<1, 64, 0, stream>>>(rowptr, colind, vals, n, most, H);
    // CTAs that stay: where there is no such form, all leave at once
    const int sms = device_sm_count();
    const int find = std::min((n + DIAG_ROWS - 1) / DIAG_ROWS, 10 * sms);
    const int fill = std::min((n + 255) / 256, 8 * sms);
    k_diag_find<<<find, DIAG_ROWS, 0, stream>>>(rowptr, colind, vals, n, most, H);
    k_diag_fill<<<fill, 256, 0, stream>>>(rowptr, colind, vals, n, most, H, (float*)f.same,
                                                        (float*)f.vals, ld, (void*)f.mask, f.mask_bytes);
    g_launches += 3;
    PPG_TRY(check_launch("k_diag_fill"));
    f.head = H->w;
    fresh = true;
    return PPG_OK;
}

int32_t DiagStore::settle(void* pinned) {
    if (!f.head) return PPG_OK;
    PPG_CUDA(cudaMemcpyAsync(pinned, f.head, 3 * sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    PPG_CUDA(cudaStreamSynchronize(s));
    const int32_t* head = (const int32_t*)pinned;
    own = head[1];
    for (uint32_t one = (uint32_t)head[2]; one; one &= one - 1) --own;
    if (head[0] != 0) drop();
    return PPG_OK;
}

template <typename T, int OP, int PRE, int MINB, bool HINT>
static cudaError_t launch_late(cudaLaunchConfig_t& cfg, const StepArgs<T>& a, bool late) {
    return late ? cudaLaunchKernelEx(&cfg, k_spmv_direct<T, OP, PRE, MINB, HINT, true>, a)
                : cudaLaunchKernelEx(&cfg, k_spmv_direct<T, OP, PRE, MINB, HINT, false>, a);
}

template <typename T, int PRE, int MINB, bool HINT>
static cudaError_t launch_direct(cudaLaunchConfig_t& cfg, int op, const StepArgs<T>& a, bool late) {
    switch (op) {
        case OP_SPMV: return launch_late<T, OP_SPMV, PRE, MINB, HINT>(cfg, a, late);
        case OP_RESID: return cudaLaunchKernelEx(&cfg, k_spmv_direct<T, OP_RESID, PRE, MINB, HINT, false>, a);
        case OP_PHI_REAL: return launch_late<T, OP_PHI_REAL, PRE, MINB, HINT>(cfg, a, late);
        case OP_PHI_PAIR2: return launch_late<T, OP_PHI_PAIR2, PRE, MINB, HINT>(cfg, a, late);
        case OP_P_REAL: return launch_late<T, OP_P_REAL, PRE, MINB, HINT>(cfg, a, late);
        case OP_P_PAIR1: return launch_late<T, OP_P_PAIR1, PRE, MINB, HINT>(cfg, a, late);
        case OP_P_PAIR2: return launch_late<T, OP_P_PAIR2, PRE, MINB, HINT>(cfg, a, late);
        default: return cudaErrorInvalidValue;
    }
}

template <typename T, bool DG, bool LR>
static cudaError_t launch_op(cudaLaunchConfig_t& cfg, int op, const StepArgs<T>& a) {
    switch (op) {
        case OP_SPMV: return cudaLaunchKernelEx(&cfg, k_spmv_step<T, OP_SPMV, DG, LR>, a);
        case OP_RESID:
            if constexpr (DG) return cudaErrorInvalidValue;
            else return cudaLaunchKernelEx(&cfg, k_spmv_step<T, OP_RESID, DG, LR>, a);
        case OP_PHI_REAL: return cudaLaunchKernelEx(&cfg, k_spmv_step<T, OP_PHI_REAL, DG, LR>, a);
        case OP_PHI_PAIR2: return cudaLaunchKernelEx(&cfg, k_spmv_step<T, OP_PHI_PAIR2, DG, LR>, a);
        case OP_P_REAL: return cudaLaunchKernelEx(&cfg, k_spmv_step<T, OP_P_REAL, DG, LR>, a);
        case OP_P_PAIR1: return cudaLaunchKernelEx(&cfg, k_spmv_step<T, OP_P_PAIR1, DG, LR>, a);
        case OP_P_PAIR2: return cudaLaunchKernelEx(&cfg, k_spmv_step<T, OP_P_PAIR2, DG, LR>, a);
        default: return cudaErrorInvalidValue;
    }
}

template <typename T>
int32_t launch_step(int op, const StepArgs<T>& a_in, cudaStream_t s) {
    if (a_in.n <= 0) return 0;
    const int rows = step_threads<T>() * step_rpt<T>();
    const int grid = (int)(((int64_t)a_in.n + rows - 1) / rows);
    StepArgs<T> a = a_in;
    // prefetch half a resident wave ahead, unless the matrix is held in an
    // L2 set-aside (measured: the prefetches then cost more than they save).
    // 3-D 160^3 chains (FP32 / FP64) by distance in resident waves:
    // 1/4 5860 / 6121 GB/s, 1/3 6017 / 6141, 1/2 6041 / 6151, 1 5969 / 6142,
    // 3/2 5836 / 6123, 2 5218 / 5982.
    constexpr bool F32 = sizeof(T) == 4;
    const bool dg = F32 && a.diag.head != nullptr, lr = F32 && (a.flags & F_LONG);
    a.pf_ahead = (a.flags & F_KEEP_A) ? 0
                 : ((lr ? (dg ? step_resident_ctas<T, F32, F32>() : step_resident_ctas<T, false, F32>())
                        : (dg ? step_resident_ctas<T, F32, false>() : step_resident_ctas<T, false, false>())) +
                    1) / 2;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(step_threads<T>());
    cfg.dynamicSmemBytes = 0;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = (a.flags & F_SERIAL) ? 0 : 1;
    if (op < OP_SPMV || op > OP_P_PAIR2) return PPG_ERR_ARG;
    const bool small = a_in.n <= DIRECT_MAX_N;
    if (small || ((a_in.flags & F_KEEP_A) && !dg)) {
        // one row per thread, no staging round (small system, or matrix in L2)
        const int dgrid = (int)(((int64_t)a_in.n + SPMV_ROWS - 1) / SPMV_ROWS);
        cfg.gridDim = dim3(dgrid);
        cfg.blockDim = dim3(SPMV_ROWS);
        // CTAs of 64 rows while an SM each is enough (a step then spreads over
        // more of them: 2-D 50^2 p(A) v 37.9 -> 32.7 us against 256 rows; 128
        // rows 35.6, 32 rows 36.8), else of 128 (1000^2 FP64 chains 55.22 ->
        // 54.88 ms against 256 rows; 64 rows 69.5 ms); the residual keeps 256:
        // one partial sum per 256 rows
        const int sms = a.sms = a.sms ? a.sms : device_sm_count();
        bool late = false;
        if (op != OP_RESID) {
            const int rows_d = a_in.n <= sms * DIRECT_SMALL_ROWS ? DIRECT_SMALL_ROWS : DIRECT_L2_ROWS;
            cfg.blockDim = dim3(rows_d);
            int64_t threads = a_in.n;
            if (small && (a.flags & F_SPREAD))   // more warps for the same rows
                threads = ((int64_t)a_in.n + SPREAD_ROWS - 1) / SPREAD_ROWS * 32;
            cfg.gridDim = dim3((unsigned)((threads + rows_d - 1) / rows_d));
            // The next steps' CTAs take places wherever there is room before a step's own
            // are done, to wait there, and a step of a few CTAs per SM then runs with
            // several on some SMs and none on others.  So a grid of at most LATE_MAX
            // CTAs per SM lets the next one in only when the previous one is done, so
            // that at most one waits: 40 FP64 steps, let in at once / so, 2-D 150^2 155 /
            // 85 us, 240^2 217 / 101, 300^2 216 / 135; four such chains on four streams, as
            // graphs, 240^2 153 / 131, 300^2 182 / 178.  A larger one, up to EVEN_MAX, takes
            // shared memory that nothing uses, which leaves an SM room for its share only:
            // 350^2 211 us at once, 161 let in late, 131 so, the four 242, 241 and 273; 400^2
            // 220, 163 and 148, the four 316, 315 and 317.  (Smaller grids gain by that too,
            // 300^2 104 us, but shut other streams out: the four 260 us, at 240^2 251.)
            // Above, neither pays (500^2 in FP32, 13 CTAs per SM, let in late 116 -> 121 us).
            const int per = (int)((cfg.gridDim.x + sms - 1) / sms);
            late = per <= LATE_MAX;
            // 228 KB per SM, 1 KB of it taken by each CTA beside its own; a share and
            // one CTA more must not fit (eight of 64 registers a thread do not)
            const bool by_registers = (a_in.flags & F_WIDE) && !F32 && a_in.n <= sms * 8 * DIRECT_L2_ROWS;
            if (!small && !late && per <= EVEN_MAX && !by_registers)
                cfg.dynamicSmemBytes = (size_t)(228 / per - 2) * 1024;
        }
        // matrix in L2: entries preloaded before the dependency wait.
        // Up to 5.5 in the average row, five: FP64 at 40 registers (1536 threads
        // per SM), the plain SpMV step at 32 (2048 threads; it fits), FP32 at 40
        // (2-D 1000^2 FP64 chains: staged kernel 57.3 ms; direct with four
        // preloads at 32 registers 55.8 ms, without the evict-last hint 56.3 ms;
        // with 128-row CTAs 54.7 ms; five for the plain SpMV step 53.4 ms; five
        // for the pair step at 40 registers 52.5 ms, four there 52.8 ms; 40 steps
        // of p(A) with four at 32 registers 586 us, five at 40 580 us.  FP32, 40
        // steps: 400^2 105 -> 94 us, 512^2 137 -> 124 us, 700^2 194 -> 184 us).
        // Above, a seven-entry row whole at 40 registers (FP64 60 x 70 x 80 phi
        // chains of 40 295 -> 268 us, FP32 p chains of 20 100 -> 79 us; 48
        // registers 279 and 80 us, six entries 287 and 88 us), and eight at 64
        // registers in FP64 while those 8 CTAs per SM hold the whole matrix
        // (45^3 201 -> 137 us, seven 146 us; 53^3 247 -> 168 us, seven 203 us).
        cudaError_t ed;
        if (small)
            ed = launch_direct<T, 8, 0, false>(cfg, op, a, late);
        else if ((a_in.flags & F_WIDE) && !F32 && a_in.n <= sms * 8 * DIRECT_L2_ROWS)
            ed = launch_direct<T, 8, 4, true>(cfg, op, a, late);
        else if (a_in.flags & F_WIDE)
            ed = launch_direct<T, 7, 6, true>(cfg, op, a, late);
        else if (!F32 && op == OP_SPMV)
            ed = launch_late<T, OP_SPMV, 5, 8, true>(cfg, a, late);
        else
            ed = launch_direct<T, 5, 6, true>(cfg, op, a, late);
        ++g_launches;
        if (ed != cudaSuccess) {
            set_cuda_error(ed, "cudaLaunchKernelEx(k_spmv_direct)");
            cudaGetLastError();
            return PPG_ERR_CUDA;
        }
        return dgrid;
    }
    const cudaError_t e =
        lr ? (dg ? launch_op<T, F32, F32>(cfg, op, a) : launch_op<T, false, F32>(cfg, op, a))
           : (dg ? launch_op<T, F32, false>(cfg, op, a) : launch_op<T, false, false>(cfg, op, a));
    ++g_launches;
    if (e != cudaSuccess) {
        set_cuda_error(e, "cudaLaunchKernelEx(k_spmv_step)");
        return PPG_ERR_CUDA;
    }
    int32_t rc = check_launch("k_spmv_step");
    return rc < 0 ? rc : grid;
}

template int32_t launch_step<double>(int, const StepArgs<double>&, cudaStream_t);
template int32_t launch_step<float>(int, const StepArgs<float>&, cudaStream_t);

// Unique bytes a step must move: the CSR (values, column indices, row
// pointers) once, and each distinct length-n vector it reads or writes once.
double step_bytes(int op, int flags, int64_t n, int64_t nnz, int elem) {
    double M = (double)nnz * (elem + 4) + 4.0 * (double)(n + 1);
    int vec = 0;
    switch (op) {
        case OP_SPMV: vec = 2; break;
        case OP_RESID: vec = 3; break;
        case OP_PHI_REAL: vec = (flags & F_FINAL) ? 3 : 2; break;
        case OP_PHI_PAIR2: vec = (flags & F_FINAL) ? 4 : 3; break;
        case OP_P_REAL:
            vec = 2 + ((flags & F_PZERO) ? 0 : 1) + ((flags & F_FINAL) ? 0 : 1);
            break;
        case OP_P_PAIR1:
            vec = 2 + ((flags & F_PZERO) ? 0 : 1) + ((flags & F_NO_O1) ? 0 : 1);
            break;
        case OP_P_PAIR2: vec = (flags & F_FINAL) ? 4 : 3; break;
        default: break;
    }
    return M + (double)vec * (double)elem * (double)n;
}

}  // namespace ppg

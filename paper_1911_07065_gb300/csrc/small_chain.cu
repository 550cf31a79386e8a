// A whole chain of root steps (Algorithm 1 or 3) of a small system in one
// launch: one thread-block cluster, the vector that a step gathers from in its
// CTAs' shared memory, everything else of a row in its thread's registers.
//
// Step by step, a small chain is bound by its launches: about 2 us each on the
// host, and at least as much on the device from one step's stores to the next
// step's gathers through L2, for some 0.3 us of arithmetic.  Here a step is a
// gather from (mostly the own, else a neighbouring) CTA's shared memory, the
// row's multiply-adds, and a hardware barrier of the cluster: 0.45 us in FP32, 0.9
// us in FP64 at n = 2,500 (p(A) v of degree 10: 34 -> 17 us with its launch).  Each row
// keeps the step kernels' arithmetic -- entries in stored order, rows of more
// than LONG_ROW entries by a warp, the same epilogue forms -- so the results
// are those bits.
//
// The cluster is CHAIN_CTAS SMs of the chip, so FP64 multiply-adds (1.6 per
// clock and SM) end its range: see chain_cluster_fits.
#include <atomic>

#include "ppg_common.cuh"

namespace ppg {

namespace {

constexpr int CHAIN_CTAS = 16;
constexpr int CHAIN_THREADS = 512;   // at most
constexpr int CHAIN_ROWS = 2;        // rows per thread at most
constexpr int CHAIN_STEPS = 112;     // what fits in the kernel's arguments
constexpr int CHAIN_E = 8;           // entries of a row in registers

template <typename T>
struct ChainStep {
    T c1, c2, c3;
    int32_t op;      // StepOp | StepFlag << 8
};

template <typename T>
struct ChainArgs {
    const int32_t* rowptr;
    const int32_t* colind;
    const T* vals;
    int32_t n, chunk, nsteps;
    uint32_t recip;      // ceil(2^32 / chunk)
    int32_t from_p;      // Algorithm 3 adds to what `out` holds
    int32_t phi;         // Algorithm 1
    const T* in;
    T* out;
    ChainStep<T> st[CHAIN_STEPS];
};
static_assert(sizeof(ChainArgs<double>) <= 4096, "kernel arguments");

__device__ __forceinline__ uint32_t cta_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t map_to(uint32_t addr, uint32_t rank) {
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(addr), "r"(rank));
    return a;
}
__device__ __forceinline__ void ld_cluster(double& v, uint32_t a) {
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
}
__device__ __forceinline__ void ld_cluster(float& v, uint32_t a) {
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
}
__device__ __forceinline__ void cluster_arrive() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <typename T, int R>
__global__ void __launch_bounds__(CHAIN_THREADS, R == 1 ? 1 : 0)
k_chain_cluster(const __grid_constant__ ChainArgs<T> a) {
    extern __shared__ __align__(16) unsigned char chain_x[];   // 2 x chunk of T
    T* const xs = reinterpret_cast<T*>(chain_x);
    const int tid = threadIdx.x, lane = tid & 31, NT = blockDim.x;
    const uint32_t rank = cta_rank();
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(chain_x);
    const uint32_t flip = (uint32_t)a.chunk * sizeof(T);   // second buffer behind the first
    PPG_PDL_TRIGGER();
    auto at = [&](int32_t col) {
        // col / chunk: exact below 2^32 / chunk, and n * chunk is at most 2^24
        const uint32_t owner = __umulhi((uint32_t)col, a.recip);
        return map_to(base, owner) + ((uint32_t)col - owner * (uint32_t)a.chunk) * (uint32_t)sizeof(T);
    };
    int32_t k0[R], len[R];
    T v[R][CHAIN_E];
    uint32_t x_at[R][CHAIN_E];
    int most = 0;   // entries in the warp's longest ordinary row
    unsigned longs[R];
#pragma unroll
    for (int i = 0; i < R; ++i) {
        const int32_t t = tid + i * NT;
        const int32_t r = (int32_t)rank * a.chunk + t;
        k0[i] = len[i] = 0;
        if (t < a.chunk && r < a.n) {
            k0[i] = __ldg(a.rowptr + r);
            len[i] = __ldg(a.rowptr + r + 1) - k0[i];
        }
        longs[i] = __ballot_sync(0xffffffffu, len[i] > LONG_ROW);
        const int ordinary = len[i] > LONG_ROW ? 0 : len[i];
        most = max(most, ordinary);
#pragma unroll
        for (int e = 0; e < CHAIN_E; ++e)
            if (e < ordinary) {
                v[i][e] = __ldg(a.vals + k0[i] + e);
                x_at[i][e] = at(__ldg(a.colind + k0[i] + e));
            }
    }
    most = __reduce_max_sync(0xffffffffu, most);
    PPG_PDL_WAIT();
    // prod: the running product (Algorithm 1: pi); aux: the pair's A pi or tmp
    T first[R], prod[R], aux[R], p[R];
#pragma unroll
    for (int i = 0; i < R; ++i) {
        const int32_t t = tid + i * NT;
        const int32_t r = (int32_t)rank * a.chunk + t;
        first[i] = prod[i] = aux[i] = p[i] = T(0);
        if (t < a.chunk && r < a.n) {
            first[i] = prod[i] = a.in[r];
            if (a.from_p) p[i] = a.out[r];
        }
        if (t < a.chunk) xs[t] = prod[i];
    }
    cluster_arrive();
    cluster_wait();
    uint32_t cur = 0;
    for (int k = 0; k < a.nsteps; ++k) {
        const T c1 = a.st[k].c1, c2 = a.st[k].c2, c3 = a.st[k].c3;
        const int op = a.st[k].op & 0xff, flags = a.st[k].op >> 8;
        T s[R];
#pragma unroll
        for (int i = 0; i < R; ++i) {
            T x[CHAIN_E];
            const int ordinary = len[i] > LONG_ROW ? 0 : len[i];
#pragma unroll
            for (int e = 0; e < CHAIN_E; ++e)
                if (e < ordinary) ld_cluster(x[e], x_at[i][e] + cur);
            T acc = T(0);
#pragma unroll
            for (int e = 0; e < CHAIN_E; ++e)
                if (e < most) {   // uniform: no FP64 issue for what no lane has
                    if (e < ordinary) acc = fma(v[i][e], x[e], acc);
                }
            if constexpr (R == 1) {
                for (int e = CHAIN_E; e < ordinary; e += 4) {
                    // (past the end: the last entry again, so that the loads need no branch)
                    int32_t c[4];
                    T w[4], xe[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        c[u] = __ldg(a.colind + k0[i] + min(e + u, ordinary - 1));
                        w[u] = __ldg(a.vals + k0[i] + min(e + u, ordinary - 1));
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) ld_cluster(xe[u], at(c[u]) + cur);
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (e + u < ordinary) acc = fma(w[u], xe[u], acc);
                }
            } else {   // (no registers for four at a time beside two rows)
#pragma unroll 4
                for (int e = CHAIN_E; e < ordinary; ++e) {
                    T xe;
                    ld_cluster(xe, at(__ldg(a.colind + k0[i] + e)) + cur);
                    acc = fma(__ldg(a.vals + k0[i] + e), xe, acc);
                }
            }
            // rows of more than LONG_ROW entries, a warp for each
            for (unsigned todo = longs[i]; todo; todo &= todo - 1) {
                const int src = __ffs(todo) - 1;
                const int32_t b = __shfl_sync(0xffffffffu, k0[i], src);
                const int32_t e1 = b + __shfl_sync(0xffffffffu, len[i], src);
                T part = T(0);
#pragma unroll 4
                for (int32_t e = b + lane; e < e1; e += 32) {
                    T xe;
                    ld_cluster(xe, at(__ldg(a.colind + e)) + cur);
                    part = fma(__ldg(a.vals + e), xe, part);
                }
#pragma unroll
                for (int off = 16; off > 0; off >>= 1)
                    part += __shfl_xor_sync(0xffffffffu, part, off);
                if (lane == src) acc = part;
            }
            s[i] = acc;
        }
        const uint32_t next = flip - cur;
#pragma unroll
        for (int i = 0; i < R; ++i) {
            T x_new;
            switch (op) {   // the epilogues of the step kernels
                case OP_PHI_REAL:
                    x_new = prod[i] = fma(-c1, s[i], prod[i]);
                    break;
                case OP_SPMV:
                    x_new = aux[i] = s[i];
                    break;
                case OP_PHI_PAIR2:
                    x_new = prod[i] = fma(c2, fma(-c1, aux[i], s[i]), prod[i]);
                    break;
                case OP_P_REAL: {
                    const T pn = (flags & F_PZERO) ? c1 * prod[i] : fma(c1, prod[i], p[i]);
                    const T prodn = fma(-c1, s[i], prod[i]);
                    p[i] = (flags & F_FINAL) ? fma(c3, prodn, pn) : pn;
                    x_new = prod[i] = prodn;
                    break;
                }
                case OP_P_PAIR1:
                    x_new = aux[i] = fma(c1, prod[i], -s[i]);
                    p[i] = (flags & F_PZERO) ? c2 * aux[i] : fma(c2, aux[i], p[i]);
                    break;
                default: {   // OP_P_PAIR2
                    const T prodn = fma(-c2, s[i], prod[i]);
                    if (flags & F_FINAL) p[i] = fma(c3, prodn, p[i]);
                    x_new = prod[i] = prodn;
                    break;
                }
            }
            const int32_t t = tid + i * NT;
            if (t < a.chunk) *reinterpret_cast<T*>(chain_x + next + t * sizeof(T)) = x_new;
        }
        // every CTA is done with this step's gathers and sees the new vector
        cluster_arrive();
        cluster_wait();
        cur = next;
    }
    const bool final_phi = a.phi && ((a.st[a.nsteps - 1].op >> 8) & F_FINAL);
#pragma unroll
    for (int i = 0; i < R; ++i) {
        const int32_t t = tid + i * NT;
        const int32_t r = (int32_t)rank * a.chunk + t;
        if (t < a.chunk && r < a.n)
            a.out[r] = !a.phi ? p[i] : final_phi ? first[i] - prod[i] : prod[i];
    }
}

template <typename T, int R>
cudaError_t launch_cluster(const ChainArgs<T>& a, int threads, size_t smem, bool probe, int* clusters,
                           cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(CHAIN_CTAS);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CHAIN_CTAS;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = probe ? 1 : 2;
    if (probe) {
        const cudaError_t e = cudaFuncSetAttribute(
            k_chain_cluster<T, R>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
        return cudaOccupancyMaxActiveClusters(clusters, k_chain_cluster<T, R>, &cfg);
    }
    return cudaLaunchKernelEx(&cfg, k_chain_cluster<T, R>, a);
}

// can the current device run the kernel's clusters?  (asked once per device)
template <typename T>
bool cluster_possible() {
    static std::atomic<int> known[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
        cudaGetLastError();
        return false;
    }
    int k = known[dev].load(std::memory_order_relaxed);
    if (k == 0) {
        int c1 = 0, c2 = 0;
        const size_t smem = 2 * (size_t)CHAIN_THREADS * CHAIN_ROWS * sizeof(T);
        const ChainArgs<T> none{};
        const bool ok =
            launch_cluster<T, 1>(none, CHAIN_THREADS, smem, true, &c1, nullptr) == cudaSuccess &&
            launch_cluster<T, 2>(none, CHAIN_THREADS, smem, true, &c2, nullptr) == cudaSuccess &&
            c1 > 0 && c2 > 0;
        cudaGetLastError();
        k = ok ? 1 : -1;
        known[dev].store(k, std::memory_order_relaxed);
    }
    return k > 0;
}

}  // namespace

// The line, from 40 steps of p(A), launch by launch / in one cluster.  FP64: where
// the cluster's multiply-adds (nnz + n a step) take less than a step's launch: 2-D
// 50^2 78 / 41 us, 85^2 79 / 68, 95^2 79 / 78, 98^2 78 / 83; short chains, where what a
// call costs beside its launches counts, a little further (98^2, 20 steps of phi 45 /
// 41).  As a graph the launches cost less: 70^2 64 / 57, 80^2 64 / 66.  FP32: up to two
// rows a thread (50^2 76 / 21, as a graph 45 / 25; 128^2 78 / 35 and 47 / 39).  And at
// most CHAIN_E entries in the average row: what a row has beyond them is read again
// in each step, with the chain of its gathers in the cluster's few warps (FP64, 2,000
// rows of 30: 160 / 236 us, 220 rows of 200: 620 / 2,330; FP32, 3,000 rows of 64: 248 /
// 460).
template <typename T>
bool chain_cluster_fits(size_t steps, int32_t n, int64_t nnz, cudaStream_t s) {
    if (n > CHAIN_CTAS * CHAIN_THREADS * CHAIN_ROWS || nnz > (int64_t)CHAIN_E * n) return false;
    const int64_t work = nnz + n;
    if (sizeof(T) == 8 && work > (steps <= 20 ? 60000 : 54000)) return false;
    if (sizeof(T) == 8 && work > 36000 && stream_capturing(s)) return false;
    if (steps < 2 || steps > (size_t)CHAIN_STEPS) return false;
    return cluster_possible<T>();
}
template bool chain_cluster_fits<double>(size_t, int32_t, int64_t, cudaStream_t);
template bool chain_cluster_fits<float>(size_t, int32_t, int64_t, cudaStream_t);

double chain_cluster_bytes(const std::vector<Step>& plan, int64_t n, int64_t nnz, int elem) {
    const Step& head = plan[0];
    const bool phi = head.op == OP_PHI_REAL || head.op == OP_SPMV;
    const int vec = !phi && !(head.flags & F_PZERO) ? 3 : 2;   // in, out (read too where it adds to it)
    return (double)nnz * (elem + 4) + 4.0 * (double)(n + 1) + (double)vec * elem * (double)n;
}

template <typename T>
bool launch_chain_cluster(const std::vector<Step>& plan, const int32_t* rowptr,
                             const int32_t* colind, const T* vals, int32_t n, const Buffers& bufs,
                             cudaStream_t s) {
    ChainArgs<T> a;
    a.rowptr = rowptr;
    a.colind = colind;
    a.vals = vals;
    a.n = n;
    a.nsteps = (int32_t)plan.size();
    const Step& head = plan[0];
    const bool phi = head.op == OP_PHI_REAL || head.op == OP_SPMV;
    a.phi = phi;
    a.from_p = !phi && !(head.flags & F_PZERO);
    a.in = (const T*)bufs.ptr[B_IN];
    a.out = (T*)bufs.ptr[phi ? B_OUT : B_P];
    for (size_t k = 0; k < plan.size(); ++k)
        a.st[k] = {(T)plan[k].c1, (T)plan[k].c2, (T)plan[k].c3, plan[k].op | plan[k].flags << 8};
    a.chunk = ((n + CHAIN_CTAS - 1) / CHAIN_CTAS + 31) / 32 * 32;
    a.recip = (uint32_t)((((uint64_t)1 << 32) + a.chunk - 1) / a.chunk);
    const size_t smem = 2 * (size_t)a.chunk * sizeof(T);
    cudaError_t e;
    if (a.chunk <= CHAIN_THREADS)
        e = launch_cluster<T, 1>(a, a.chunk, smem, false, nullptr, s);
    else
        e = launch_cluster<T, 2>(a, (a.chunk / 2 + 31) / 32 * 32, smem, false, nullptr, s);
    if (e != cudaSuccess) {   // (fewer SMs at hand than when the device was asked)
        cudaGetLastError();
        return false;
    }
    ++g_launches;
    return true;
}
template bool launch_chain_cluster<double>(const std::vector<Step>&, const int32_t*,
                                              const int32_t*, const double*, int32_t,
                                              const Buffers&, cudaStream_t);
template bool launch_chain_cluster<float>(const std::vector<Step>&, const int32_t*,
                                             const int32_t*, const float*, int32_t, const Buffers&,
                                             cudaStream_t);

}  // namespace ppg

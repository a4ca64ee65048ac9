// paco_cluster.cu -- the whole PACO transform of a small size in one launch,
// with the paper's p processors as groups of CTAs of one thread-block cluster.
//
// N1 = N2 = 256, p in {4, 8}.  The transform runs on a cluster of K CTAs
// (K = 16 where the GPU allows that cluster size, else 8; K is a multiple of
// p): processor q of Sect. 2 is the group of K/p consecutive CTAs, and CTA r
// owns 256/K of its slab's columns on both sides, so that more SMs share the
// work of one transform.  CTA r:
//   Phase I    owns input columns c in [r 256/K, (r+1) 256/K) of X = x viewed
//              N1 x N2 (processor q = floor(r p / K) owns slab q, Eq.
//              input-slab-owner) and computes their length-256 DFTs in shared
//              memory (radix 16 x 16);
//   middle     each result A[v][c] goes to the CTA that owns output column v (its
//              processor owns v by Eq. (3)): one all-to-all through distributed shared memory
//              (PARA-CO-DRP, Sect. 4.2, App. C.5), one block of N/K^2 items per
//              ordered pair of CTAs, N/p^2 per ordered pair of processors; a
//              CTA's block for itself stays in its own shared memory.  Row
//              pi_m2(c) of W = Z-hat (Eq. (17)) is kept as row c mod 256/K of
//              the block from c's owner;
//   Phase III  computes the length-256 DFTs of its output columns over the
//              digit-reversed rows pi_m2(j) (Lemma 1, input layout), that is
//              over c = j, with the top-level twiddle w_N^{-vc} folded into their
//              butterflies (paco_fold.cuh), and writes columns k1 in [r 256/K, (r+1) 256/K) of
//              Y = y viewed N2 x N1.
// The blocks travel as one bulk copy each (2 KiB for K = 16), which counts its
// bytes on the destination's transaction barrier.  Item by item (st.async of 8
// bytes) the exchange kept each SM's port busy for 4096 packets a side: the
// transform took 6.7 us in a replayed graph, and 6.05 us so (4.3 with the folded
// butterflies as well).
// Synchronisation: one split cluster barrier (arrive at entry, wait before the
// first copy) makes sure every CTA of the cluster runs and has set up its
// barrier; a CTA starts Phase III as soon as its own N/K items have landed; a
// second split barrier (arrive there, wait at the end) keeps each CTA's blocks
// in place until all of them have been read.  The wait for the items is bounded
// (2 s): a CTA that gives up sets the plan's status word to PACO_ERR_TIMEOUT and
// finishes the launch with whatever landed.
#include <cuda_runtime.h>

#include <atomic>
#include <cstring>

#include "../../include/paco.h"
#include "paco_fold.cuh"
#include "paco_plan.h"

namespace paco {

struct ClusterArgs {
    const float2 *in;
    float2 *out;
    long long N;                 // 65536
    int p;                       // processors (counts are kept per pair of processors)
    int conj;                    // dir = +1: conjugate on load and store
    const float2 *tau;           // the factors of paco_fold.cuh: Phase I's F2 (128), Phase III's F1 and F2 (136 x 256)
    int *status;                 // device status word (PACO_ERR_TIMEOUT)
    unsigned *pair_count;        // p x p counts of items sent (test hook), or nullptr
    unsigned long long wait_ns;  // limit of the bounded wait
    unsigned extra_tx;           // test hook: bytes expected beyond the N/K items (0 in use)
};

namespace {

constexpr int L = 256;

__device__ __forceinline__ cx<float> ld_cx(const float2 *p)
{
    const float2 v = *p;
    return make_cx<float>(v.x, v.y);
}
__device__ __forceinline__ unsigned smem_u32(const void *p)
{
    return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// address of the same shared variable in CTA `rank` of the cluster
__device__ __forceinline__ unsigned map_rank(unsigned addr, int rank)
{
    unsigned r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
// bulk copy into another CTA's shared memory that counts its bytes on that
// CTA's transaction barrier
__device__ __forceinline__ void bulk_copy(unsigned dst, unsigned src, unsigned bytes, unsigned bar)
{
    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 :: "r"(dst), "r"(src), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned bar, unsigned parity)
{
    unsigned ok;
    asm volatile("{\n\t.reg .pred p;\n\t"
                 "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}

// One length-256 DFT per column of a W-column block, as radix 16 x 16 with
// one exchange through buf.  Pass 1: thread (col, t16) -- col = tid % W,
// t16 = tid / W -- brings the DFT of its 16 inputs x[t16 + 16 s] in v.  Pass 2:
// thread (col2, u) -- (tid % W, tid / W) when T16_FAST is false, else
// (tid / 16, tid % 16) -- gets outputs u + 16 k', k' < 16, of column col2 in
// v, with the factors f of its folded butterflies.  buf holds the intermediate
// (k16, t16) of column col at row 16 k16 + t16, column col ^ k16:
// conflict-free for both pass-2 roles.
template <bool T16_FAST>
__device__ __forceinline__ void dft256_finish(cx<float> *v, float2 *buf, int W, int col, int t16, const float2 *f)
{
#pragma unroll
    for (int s = 0; s < 16; ++s) buf[(s * 16 + t16) * W + (col ^ s)] = make_float2(v[s].x, v[s].y);
    __syncthreads();
    const int tid = threadIdx.x;
    const int col2 = T16_FAST ? tid / 16 : tid % W, u = T16_FAST ? tid % 16 : tid / W;
#pragma unroll
    for (int t = 0; t < 16; ++t) v[t] = ld_cx(&buf[(u * 16 + t) * W + (col2 ^ u)]);
    fold_dft<DIRECT, float, 16>(v, [&](int q) { return make_cx<float>(f[q].x, f[q].y); });
}

} // namespace

// K CTAs per transform (a cluster), 4096 / K threads each.
template <int K>
__global__ void __launch_bounds__(4096 / K, K == 16 ? 2 : 1) paco_cluster_kernel(const ClusterArgs a)
{
    extern __shared__ __align__(16) float2 smem[];
    constexpr int NK = 65536 / K;                             // items per CTA
    float2 *bufA = smem;                                      // the in-CTA exchanges of the length-256 DFTs
    float2 *bufB = smem + NK;                                 // this CTA's part of W, [source CTA][c][v], filled by the all-to-all
    float2 *bufC = smem + 2 * NK;                             // what it sends, [destination CTA][c][v]
    __shared__ __align__(8) unsigned long long full;          // counts the bytes that land in bufB
    __shared__ unsigned cnt[16];
    constexpr int W1 = L / K, W2 = L / K;                     // input and output columns of a CTA
    unsigned q;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(q));  // this CTA
    const long long tr = (long long)(blockIdx.x / K);         // the transform of this cluster
    const int tid = threadIdx.x;
    const int col = tid % W1, t16 = tid / W1;                 // Phase I pass 1; Phase III: (vl, u16) = (col, t16)
    const int colB = tid / 16, tB = tid % 16;                 // Phase I pass 2: column q W1 + colB, outputs tB + 16 k
    const int cglob = (int)q * W1 + col;
    const unsigned fullA = smem_u32(&full);

    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(fullA) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
                     :: "r"(fullA), "r"((unsigned)(NK * sizeof(float2)) + a.extra_tx) : "memory");
    }
    if (a.pair_count && tid < 16) cnt[tid] = 0;
    // (the barrier's initialisation is ordered by the fence above)
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");

    // Factors first: the plan's tables are not written by the preceding
    // kernels, so their loads overlap the wait for those kernels.
    const int k1 = (int)q * W2 + col;                         // Phase III's column
    float2 f1[8], f3a[8], f3b[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        f1[i] = __ldg(&a.tau[i * 16 + tB]);
        f3a[i] = __ldg(&a.tau[128 + i * L + k1]);
        f3b[i] = __ldg(&a.tau[128 + (8 + i * 16 + t16) * L + k1]);
    }
    // Programmatic dependent launch: wait for the kernels before this one
    // (they may write x or read y), then let the next kernel start its CTAs.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    const float2 *x = a.in + tr * a.N;
    float2 *y = a.out + tr * a.N;

    // ---- Phase I on input columns c = q W1 + col
    cx<float> v[16];
#pragma unroll
    for (int s = 0; s < 16; ++s) {
        v[s] = ld_cx(x + (long long)(t16 + 16 * s) * L + cglob);   // row t16 + 16 s of X
        if (a.conj) v[s].y = -v[s].y;
    }
    dft16(v);
    dft256_finish<true>(v, bufA, W1, col, t16, f1);
    // k-th result: column v = tB + 16 k of Y, row colB of the block for v's owner
    // (16 lanes fill 16 consecutive places)
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const int vf = tB + 16 * k, qd = vf / W2, vl = vf % W2;
        bufC[(qd * W1 + colB) * W2 + vl] = make_float2(v[k].x, v[k].y);
        if (a.pair_count) atomicAdd(&cnt[qd], 1u);
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");          // the copies below read these stores
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");   // all CTAs run, barriers set up
    __syncthreads();
    if (tid < K) {
        const int qd = ((int)q + tid) % K;                    // spread over the destinations
        constexpr unsigned block = W1 * W2 * sizeof(float2);
        bulk_copy(map_rank(smem_u32(bufB) + q * block, qd), smem_u32(bufC) + qd * block, block, map_rank(fullA, qd));
    }
    // every item of this CTA's part has landed (bounded wait)
    if (!mbar_try_wait(fullA, 0)) {
        const unsigned long long t0 = global_ns();
        while (!mbar_try_wait(fullA, 0)) {
            if (global_ns() - t0 > a.wait_ns) {                // give up: flag it, finish the launch
                atomicExch(a.status, (int)PACO_ERR_TIMEOUT);
                break;
            }
        }
    }
    __syncwarp();
    // this CTA has what the others sent it (or gave up waiting)
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    if (a.pair_count) {                                       // per ordered pair of processors
        __syncthreads();
        if (tid < K) {
            const int g = K / a.p;
            atomicAdd(&a.pair_count[((int)q / g) * a.p + tid / g], cnt[tid]);
        }
    }

    // ---- Phase III on output columns v = q W2 + vl, logical rows j = c
    const int vl = col, u16 = t16;
#pragma unroll
    for (int s = 0; s < 16; ++s) {
        const int j = u16 + 16 * s;
        v[s] = ld_cx(&bufB[j * W2 + vl]);                     // row j mod W1 of the block from CTA j / W1
    }
    fold_dft<DIRECT, float, 16>(v, [&](int i) { return make_cx<float>(f3a[i].x, f3a[i].y); });
    dft256_finish<false>(v, bufA, W2, vl, u16, f3b);          // (every read of bufA was before the exchange)
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const int k2 = u16 + 16 * k;
        y[(long long)k2 * L + k1] = make_float2(v[k].x, a.conj ? -v[k].y : v[k].y);   // Y[k2][k1] = y[k1 + k2 N1]
    }
    asm volatile("barrier.cluster.wait.aligned;" ::: "memory");   // every block of this CTA has been read
}

const void *cluster_kernel_fn(int K)
{
    return K == 16 ? reinterpret_cast<const void *>(&paco_cluster_kernel<16>)
                   : reinterpret_cast<const void *>(&paco_cluster_kernel<8>);
}

// The one-launch form applies to complex64 plans with N1 = N2 = 256 and p = 4
// or 8, up to 16 transforms.  It keeps one transform on one cluster of K SMs, which
// is latency-bound; the alternative is two passes over all SMs.  us in a replayed
// graph, this form and the passes: 1 transform 4.3 and 4.9, 4 4.4 and 5.2, 8 6.8 and
// 6.4, 12 7.2 and 10.0, 16 9.9 and 10.6.  (The limit of 16 dates from the stage
// launches before the passes, which were faster at 32.)
bool cluster_eligible(const paco_plan *pl)
{
    return pl->dtype == PACO_C64 && pl->N1 == 256 && pl->N2 == 256 && (pl->p == 4 || pl->p == 8) &&
           pl->batch <= 16;
}

// CTAs per transform on the current device: 16 when a 16-CTA cluster of this
// kernel can be resident, else 8 (queried once per device; concurrent first
// calls compute the same answer).
int cluster_size()
{
    static std::atomic<int> cache[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) dev = 0;
    const int known = cache[dev].load(std::memory_order_relaxed);
    if (known) return known;
    int k = 8;
    if (cudaFuncSetAttribute(cluster_kernel_fn(16), cudaFuncAttributeNonPortableClusterSizeAllowed, 1) ==
        cudaSuccess) {
        cudaLaunchConfig_t cfg;
        memset(&cfg, 0, sizeof(cfg));
        cfg.gridDim = dim3(16, 1, 1);
        cfg.blockDim = dim3(256, 1, 1);
        cfg.dynamicSmemBytes = 3 * 4096 * sizeof(float2);
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 16;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, cluster_kernel_fn(16), &cfg) == cudaSuccess && n > 0) k = 16;
    }
    cudaGetLastError();                                       // a refused query leaves no error behind
    cache[dev].store(k, std::memory_order_relaxed);
    return k;
}

paco_status_t launch_cluster(const paco_plan *pl, const void *in, void *out, int dir, unsigned *pair_count,
                             cudaStream_t stream)
{
    ClusterArgs a;
    memset(&a, 0, sizeof(a));
    a.in = static_cast<const float2 *>(in);
    a.out = static_cast<float2 *>(out);
    a.N = pl->N;
    a.p = pl->p;
    a.conj = (dir == 1);
    a.tau = static_cast<const float2 *>(pl->cluster_tau);
    a.status = pl->d_status;
    a.pair_count = pair_count;
    a.wait_ns = 2000000000ull;
    a.extra_tx = 8u * pl->dbg_wait_bias;          // paco_debug_set_waits: a wait that runs out
    const int K = pl->fused_k;                    // chosen at plan creation on the plan's device
    const int threads = (int)(pl->N / K / 16);
    const size_t smem = 3 * (size_t)(pl->N / K) * sizeof(float2);
    for (int64_t b0 = 0; b0 < pl->batch; b0 += 8192) {
        const int64_t nb = (pl->batch - b0 < 8192) ? pl->batch - b0 : 8192;
        ClusterArgs ab = a;
        ab.in = a.in + b0 * pl->N;
        ab.out = a.out + b0 * pl->N;
        cudaLaunchConfig_t cfg;
        memset(&cfg, 0, sizeof(cfg));
        cfg.gridDim = dim3((unsigned)(nb * K), 1, 1);
        cfg.blockDim = dim3((unsigned)threads, 1, 1);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = stream;
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)K;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // the kernel waits (griddepcontrol)
        attr[1].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 2;
        void *params[] = {&ab};
        PACO_CUDA_TRY(cudaLaunchKernelExC(&cfg, cluster_kernel_fn(K), params));
    }
    return PACO_OK;
}

// Kernel attributes and the plan's table of factors (273 KiB).
paco_status_t cluster_setup(paco_plan *pl)
{
    PACO_CUDA_TRY(cudaFuncSetAttribute(cluster_kernel_fn(8), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       3 * 8192 * (int)sizeof(float2)));
    PACO_CUDA_TRY(cudaFuncSetAttribute(cluster_kernel_fn(16), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       3 * 4096 * (int)sizeof(float2)));
    pl->fused_k = cluster_size();
    // the factors of two passes of 16 x 16 points, in one table
    FoldKernel k;
    k.lgA = k.lgB = 4;
    const paco_status_t st = fold_table<float>(&pl->cluster_tau, k, 1, 8, pl->dims >= 2,    // (the 2-D DFT has no top-level twiddle)
                                               128 * sizeof(float2));
    if (st != PACO_OK) return st;
    fold_levels(pl->cluster_tau, k);
    PACO_CUDA_TRY(cudaGetLastError());
    return PACO_OK;
}

} // namespace paco

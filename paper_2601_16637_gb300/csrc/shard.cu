// Row-block sigma for alpha-row sharding (paper Sec. III: the alpha rows of C and sigma are
// distributed over processes and the C blocks travel around a ring, so each process adds, block
// after block, the contribution of every block to its own rows).
//
// A plan fixes the output alpha rows [r0, r1) and the source alpha rows [j0, j1).  It holds the
// alpha excitation lists of the output rows restricted to targets in [j0, j1), with the targets
// renumbered from j0, in the layouts the passes read: canonical singles for the alpha-beta pass;
// padded, bank-ordered singles and doubles for the alpha pass, with the values of the arithmetics the
// plan is for (a solve takes only its own).  The beta lists of the output rows inside the block are
// the handle's.  sigma_block_apply (sigma.cu) then runs the three passes on the block: beta pass on the
// output rows that lie inside the block, alpha pass on the transposed block, alpha-beta pass on the
// block's rows.
#include <algorithm>
#include <vector>

#include "common.cuh"

namespace sbd {

namespace {

constexpr int kThreadsB = 128;

int grid_for(int64_t n) { return (int)std::max<int64_t>(1, std::min<int64_t>(65535, (n + kThreadsB - 1) / kThreadsB)); }

// per output row: entries of the canonical singles list with target in [j0, j1)
__global__ void count_canon_kernel(const int64_t *__restrict__ ptr, const int32_t *__restrict__ tgt, int64_t r0,
                                   int64_t nr, int64_t j0, int64_t j1, int64_t *cnt)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nr; i += (int64_t)gridDim.x * blockDim.x) {
        int64_t k = 0;
        for (int64_t e = ptr[r0 + i]; e < ptr[r0 + i + 1]; ++e) k += tgt[e] >= j0 && tgt[e] < j1;
        cnt[i] = k;
    }
}

__global__ void fill_canon_kernel(const int64_t *__restrict__ ptr, const int32_t *__restrict__ tgt,
                                  const uint32_t *__restrict__ pk, int64_t r0, int64_t nr, int64_t j0, int64_t j1,
                                  const int64_t *__restrict__ optr, uint32_t *opk)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nr; i += (int64_t)gridDim.x * blockDim.x) {
        int64_t o = optr[i];
        for (int64_t e = ptr[r0 + i]; e < ptr[r0 + i + 1]; ++e)
            if (tgt[e] >= j0 && tgt[e] < j1) opk[o++] = (pk[e] & ~kPackJMask) | (uint32_t)(tgt[e] - j0);
    }
}

// exclusive prefix sum of n counts into out[0..n] (single CTA, sequential blocks of the block size)
__global__ void scan_counts_kernel(const int64_t *cnt, int64_t n, int64_t *out)
{
    __shared__ int64_t part[1024];
    __shared__ int64_t carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int64_t b = 0; b < n; b += blockDim.x) {
        const int64_t i = b + threadIdx.x;
        part[threadIdx.x] = i < n ? cnt[i] : 0;
        __syncthreads();
        for (int off = 1; off < (int)blockDim.x; off <<= 1) {
            const int64_t v = threadIdx.x >= (unsigned)off ? part[threadIdx.x - off] : 0;
            __syncthreads();
            part[threadIdx.x] += v;
            __syncthreads();
        }
        if (i < n) out[i + 1] = carry + part[threadIdx.x];
        __syncthreads();
        if (threadIdx.x == blockDim.x - 1) carry += part[threadIdx.x];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[0] = 0;
}

}  // namespace

BlockPlan *block_plan_create(Ctx &c, int64_t r0, int64_t r1, int64_t j0, int64_t j1, int mask)
{
    if (r0 < 0 || r1 <= r0 || r1 > c.nA || j0 < 0 || j1 <= j0 || j1 > c.nA)
        fail(SBD_ERR_INVALID_ARG, "block plan: row ranges must be non-empty and inside [0, nA)");
    const size_t held = c.allocs.size();
    const SigLists beta = c.sp[1].sig;
    auto *p = new BlockPlan();
    p->c = &c;
    p->r0 = r0;
    p->r1 = r1;
    p->j0 = j0;
    p->j1 = j1;
    const SpinTables &ta = c.sp[0];
    const int64_t nr = r1 - r0;
    cudaStream_t s = c.stream;
    try {
        int64_t *cnt = dalloc_n<int64_t>(c, (size_t)nr);
        // canonical singles (alpha-beta pass)
        p->s_ptr = dalloc_n<int64_t>(c, (size_t)nr + 1);
        count_canon_kernel<<<grid_for(nr), kThreadsB, 0, s>>>(ta.s_ptr, ta.s_j, r0, nr, j0, j1, cnt);
        SBD_LAUNCH("count_canon_kernel");
        scan_counts_kernel<<<1, 1024, 0, s>>>(cnt, nr, p->s_ptr);
        SBD_LAUNCH("scan_counts_kernel");
        dfree(c, cnt);
        int64_t ns = 0;
        SBD_CUDA(cudaMemcpyAsync(&ns, p->s_ptr + nr, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
        SBD_CUDA(cudaStreamSynchronize(s));
        p->s_pk = dalloc_n<uint32_t>(c, (size_t)ns);
        fill_canon_kernel<<<grid_for(nr), kThreadsB, 0, s>>>(ta.s_ptr, ta.s_j, ta.s_pk, r0, nr, j0, j1, p->s_ptr,
                                                             p->s_pk);
        SBD_LAUNCH("fill_canon_kernel");
        // padded lists of the alpha pass
        build_sig_lists(c, ta, r0, nr, j0, j1, mask, p->sig);
        // transposed source block, doubles
        p->work_t = dalloc(c, sizeof(double) * (size_t)(j1 - j0) * (size_t)c.nB);
        p->rowmax = dalloc_n<float>(c, (size_t)(j1 - j0));
        for (size_t i = held; i < c.allocs.size(); ++i) p->allocs.push_back(c.allocs[i].first);
        // the beta lists that the output rows inside the block read, made with the first such plan
        if (std::max(r0, j0) < std::min(r1, j1)) build_sig_lists(c, c.sp[1], 0, c.nB, 0, c.nB, mask, c.sp[1].sig);
        SBD_CUDA(cudaStreamSynchronize(s));
    } catch (...) {  // an allocation was refused: the handle is as it was
        while (c.allocs.size() > held) dfree(c, c.allocs.back().first);
        c.sp[1].sig = beta;
        delete p;
        throw;
    }
    return p;
}

void ring_sigma(ShardCtx &sh, Ctx &c, const void *x_rows, double *y_rows, sbd_precision prec, cudaStream_t s,
                const double *x64_rows)
{
    const size_t elem = prec == SBD_MIXED ? sizeof(float) : sizeof(double);
    const int W = sh.world, r = sh.rank;
    SBD_CUDA(cudaMemsetAsync(y_rows, 0, sizeof(double) * (size_t)sh.rows() * (size_t)c.nB, s));
    // the rank's own block is complete before the first transfer reads it
    SBD_CUDA(cudaStreamSynchronize(s));
    const void *cur = x_rows;
    for (int step = 0; step < W; ++step) {
        const int b = ((r - step) % W + W) % W;
        sigma_block_apply(*sh.plans[b], cur, y_rows, prec, s, b == r ? x64_rows : nullptr);
        void *nxt = nullptr;
        if (step + 1 < W) {
            // double buffering (Sec. III-E): the transfer runs while the products above are in flight.
            // Both only read cur; nxt was last read by the previous step's products, which have completed.
            const int nb = ((r - step - 1) % W + W) % W;
            nxt = sh.ring[step % 2];
            const size_t sb = (size_t)(sh.bounds[b + 1] - sh.bounds[b]) * (size_t)c.nB * elem;
            const size_t rb = (size_t)(sh.bounds[nb + 1] - sh.bounds[nb]) * (size_t)c.nB * elem;
            if (sh.comm.ring_exchange(sh.comm.ctx, cur, sb, nxt, rb, (void *)s) != 0)
                fail(SBD_ERR_CUDA, "ring_exchange callback failed");
        }
        SBD_CUDA(cudaStreamSynchronize(s));  // this block's products are done before its buffer is reused
        if (nxt) cur = nxt;
    }
}

void block_plan_destroy(BlockPlan *p)
{
    if (!p) return;
    for (void *q : p->allocs) dfree(*p->c, q);
    delete p;
}

}  // namespace sbd

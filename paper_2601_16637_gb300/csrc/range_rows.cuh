// Row passes of the sigma product: same-spin excitation lists against ranges of C staged in shared
// memory (see RangeLists for the lists).
//
// The pass computes, for `nrow` independent rows (the strings of the other spin) and every string i
// of the list spin,
//   Y[i][r] (+)= sum_{j in doubles(i)} H(i,j) X[j][r]
//              + sum_{j in singles(i), pair rs, phase t} [H(i,j) + t J_r[rs]] X[j][r],
// with the rows contiguous in X and Y: the alpha pass reads C and adds into sigma as they are, the
// beta pass reads the transpose of C and writes the transpose of its part of sigma.
//
// What bounds it and why it is laid out this way: every multiply-add takes one operand of C from
// shared memory, and what a load brings into registers passes at 128 bytes per SM clock, whether the
// bytes differ between the lanes or not.  In FP32 the pass is bound by that, in FP64 by the FP64 pipe.
// A CTA stages 128 bytes of every string j of a range: 32 rows in FP32, 16 in FP64 or FP32 pairs.
// Four lanes walk one list together, each owning two 16-byte chunks of the staged line (8 rows in
// FP32), so that a list entry, 6 bytes in FP32, feeds 8 multiply-adds; with eight lanes and one chunk
// each, the entries took 27 % of the bytes instead of 16 %.  Chunk c holds rows c, c + 8, ...; the two
// lists that share a 128-bit phase read their chunks in opposite order, so the phase covers all 32
// banks whatever strings they read.  Every lane works on every entry (on the FP64 pipe an idle lane
// costs as much as a busy one), no sum crosses lanes, and the four lanes' loads and stores of Y are
// contiguous without asking anything of its alignment or row length.
//
// Measured, beta + alpha pass of one product (CUDA events, before: whole rows of C staged, one list
// per eight lanes and one entry per lane): 1.0e8 determinants, FP32 25.1 -> 17.6 ms; 3.6e7
// determinants (norb 29), FP32 7.0 -> 5.0, FP64 64.2 -> 49.6, FP32 pairs 20.8 -> 15.5 ms; 2.5e7
// determinants at norb 58, FP32 about 12 -> 6.4 ms.
// Steps on the way (FP32, 3.6e7 determinants): an octet per list with separate lists 6.0 ms, with
// interleaved lists 6.2 (padding costs more than the contiguous loads save while every octet still
// reads 24 bytes of entries per 64 of C), four lanes per list 5.5; 24 warps with 80 registers instead
// of 32 with 64 (which spilled) 5.1, 16 warps 5.9; entries loaded two blocks ahead 5.0.
#pragma once

#include "common.cuh"
#include "pair.cuh"

namespace sbd {

constexpr int kRangeThreads = 768;
constexpr int kRangeRowBytes = 128;

// The table of J_r[rs] of the staged rows sits in shared memory while it leaves at least half of it
// to the ranges (norb <= 43); above that the few singles read J from global memory, because shorter
// ranges would mean more passes over Y.
__host__ __device__ inline size_t range_j_bytes(int norb) { return (size_t)(norb * (norb - 1) / 2 + 1) * kRangeRowBytes; }
__host__ __device__ inline size_t range_smem(int optin) { return ((size_t)optin - 1024) / kRangeRowBytes * kRangeRowBytes; }
__host__ __device__ inline bool range_j_staged(int optin, int norb) { return 2 * range_j_bytes(norb) <= range_smem(optin); }
// most strings of one range (behind them: the table, whose last line is zero, or one line of zeros)
inline int range_width_max(int optin, int norb)
{
    const size_t room = range_smem(optin) - (range_j_staged(optin, norb) ? range_j_bytes(norb) : kRangeRowBytes);
    return (int)(room / kRangeRowBytes);
}
// the line of zeros that padding entries point to, for ranges of w strings and np pairs in the table
inline int range_pad(int optin, int norb, int w, int np) { return w + (range_j_staged(optin, norb) ? np : 0); }

// list value type of an arithmetic (pairs: the high parts; the low parts are an array of their own)
template <typename T>
struct RangeVal {
    using type = T;
};
template <>
struct RangeVal<F2> {
    using type = float;
};
// element type of the vectors (the pair arithmetic reads FP64 vectors)
template <typename T>
struct RangeIn {
    using type = T;
};
template <>
struct RangeIn<F2> {
    using type = double;
};

template <typename T>
struct RangeArgs {
    const typename RangeIn<T>::type *X;  // [n][nrow]
    double *Y;                           // [n][nrow]
    int64_t n, nrow;
    int accumulate;  // add to Y (0: the first range writes)
    float *rowmax;   // FP32 only, optional: [nrow] max_j |X[j][r]|
    int npair, jstaged, w, ng;  // npair: orbital pairs of the lists
    int q;             // batched launches: pieces a row block is cut into (a divisor of kParts)
    const double *jg;  // [npair][nrow]
    const int32_t *zi;
    const uint32_t *qd, *qs;
    const uint16_t *dt;
    const typename RangeVal<T>::type *dv;
    const uint32_t *sm;
    const typename RangeVal<T>::type *sv;
    const float *dlo, *slo;  // pairs: low parts
};

template <typename T>
constexpr int kRangeRows = kRangeRowBytes / (int)sizeof(T);


// Packed FP32 arithmetic on two rows at a time: the same roundings as two scalar operations in half
// the instructions (the pass issues in 73 % of the cycles with scalar ones).
__device__ __forceinline__ uint64_t pk_fma(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t pk_mul(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t pk_add(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t pk_dup(float v)
{
    uint64_t d;
    asm("mov.b64 %0, {%1, %1};" : "=l"(d) : "f"(v));
    return d;
}
__device__ __forceinline__ uint64_t pk_pair(float a, float b)
{
    uint64_t d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(a), "f"(b));
    return d;
}
__device__ __forceinline__ float pk_get(uint64_t p, int i)
{
    return __uint_as_float(i ? (unsigned)(p >> 32) : (unsigned)p);
}
// x - y as one rounded operation per half
__device__ __forceinline__ uint64_t pk_sub(uint64_t x, uint64_t y) { return pk_fma(y, pk_dup(-1.f), x); }

// f2_mac on two pairs at once: (hi, lo) += (ah + al) * (b.x + b.y), an = -ah (which saves negating the
// product for its error term)
__device__ __forceinline__ void pk_f2_mac(uint64_t &hi, uint64_t &lo, uint64_t ah, uint64_t an, uint64_t al, ulonglong2 b)
{
    const uint64_t pn = pk_mul(an, b.x);
    uint64_t e = pk_fma(ah, b.x, pn);
    e = pk_fma(ah, b.y, e);
    e = pk_fma(al, b.x, e);
    const uint64_t s = pk_sub(hi, pn);
    const uint64_t bb = pk_sub(s, hi);
    const uint64_t t = pk_sub(pk_sub(hi, pk_sub(s, bb)), pk_add(pn, bb));
    hi = s;
    lo = pk_add(lo, pk_add(t, e));
}
// (hi, lo) = (ah + al) * (b.x + b.y)
__device__ __forceinline__ void pk_f2_mul(uint64_t &hi, uint64_t &lo, uint64_t ah, uint64_t an, uint64_t al, ulonglong2 b)
{
    hi = pk_mul(ah, b.x);
    uint64_t e = pk_fma(ah, b.x, pk_mul(an, b.x));
    e = pk_fma(ah, b.y, e);
    lo = pk_fma(al, b.x, e);
}
// (hi, lo) += (bh, bl), the low part back below the rounding of the high part
__device__ __forceinline__ void pk_f2_add(uint64_t &hi, uint64_t &lo, uint64_t bh, uint64_t bl)
{
    const uint64_t s = pk_add(hi, bh), bb = pk_sub(s, hi);
    const uint64_t t = pk_add(pk_sub(hi, pk_sub(s, bb)), pk_sub(bh, bb));
    lo = pk_add(lo, pk_add(t, bl));
    hi = pk_add(s, lo);
    lo = pk_sub(lo, pk_sub(hi, s));
}

// The sums of one lane: NH chunks of a staged line.  A chunk's 16 bytes are two words:
// two packed pairs of rows (FP32), two FP64 rows, or the high and the low parts of two pair rows.
template <typename T, int NH = 2>
struct RangeAcc;

template <int NH>
struct RangeAcc<float, NH> {
    static constexpr int kRowsPerChunk = 4;
    using Val = float;
    uint64_t blk[2 * NH], acc[2 * NH], sum[2 * NH];
    __device__ __forceinline__ void zero()
    {
#pragma unroll
        for (int i = 0; i < 2 * NH; ++i) acc[i] = sum[i] = 0ull;
    }
    static __device__ __forceinline__ Val val(const float *p, const float *) { return __ldg(p); }
    static __device__ __forceinline__ void load(const float *p, const float *, float (&v)[4])
    {
        const float4 a = __ldg(reinterpret_cast<const float4 *>(p));
        v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w;
    }
    // entry u of a block; the block's products are summed by themselves, and the blocks on two
    // levels (eight blocks, then all): short chains keep the rounding error of a long list down
    __device__ __forceinline__ void mac(int u, float v, const ulonglong2 (&x)[NH])
    {
        const uint64_t vv = pk_dup(v);
#pragma unroll
        for (int h = 0; h < NH; ++h) {
            blk[2 * h] = u == 0 ? pk_mul(vv, x[h].x) : pk_fma(vv, x[h].x, blk[2 * h]);
            blk[2 * h + 1] = u == 0 ? pk_mul(vv, x[h].y) : pk_fma(vv, x[h].y, blk[2 * h + 1]);
        }
    }
    __device__ __forceinline__ void end_block(unsigned count)
    {
#pragma unroll
        for (int i = 0; i < 2 * NH; ++i) acc[i] = pk_add(acc[i], blk[i]);
        if ((count & 7u) == 0u) {
#pragma unroll
            for (int i = 0; i < 2 * NH; ++i) sum[i] = pk_add(sum[i], acc[i]), acc[i] = 0ull;
        }
    }
    // (v + sg*j) x, the entries of a block in two chains
    __device__ __forceinline__ void single(int u, float v, float sg, const ulonglong2 (&j)[NH], const ulonglong2 (&x)[NH])
    {
        const uint64_t vv = pk_dup(v), ss = pk_dup(sg);
        uint64_t(&s)[2 * NH] = u == 0 ? acc : sum;
#pragma unroll
        for (int h = 0; h < NH; ++h) {
            s[2 * h] = pk_fma(pk_fma(ss, j[h].x, vv), x[h].x, s[2 * h]);
            s[2 * h + 1] = pk_fma(pk_fma(ss, j[h].y, vv), x[h].y, s[2 * h + 1]);
        }
    }
    __device__ __forceinline__ void end_singles()
    {
#pragma unroll
        for (int i = 0; i < 2 * NH; ++i) sum[i] = pk_add(sum[i], acc[i]), acc[i] = 0ull;
    }
    __device__ __forceinline__ double value(int h, int i) const
    {
        return (double)(pk_get(acc[2 * h + i / 2], i & 1) + pk_get(sum[2 * h + i / 2], i & 1));
    }
    static __device__ __forceinline__ void store(unsigned char *line, int row, double x)
    {
        reinterpret_cast<float *>(line)[(row & 7) * 4 + (row >> 3)] = (float)x;
    }
    static __device__ __forceinline__ ulonglong2 chunk(const double (&x)[4])
    {
        return make_ulonglong2(pk_pair((float)x[0], (float)x[1]), pk_pair((float)x[2], (float)x[3]));
    }
};

template <int NH>
struct RangeAcc<double, NH> {
    static constexpr int kRowsPerChunk = 2;
    using Val = double;
    double acc[2 * NH];
    __device__ __forceinline__ void zero()
    {
#pragma unroll
        for (int i = 0; i < 2 * NH; ++i) acc[i] = 0.0;
    }
    static __device__ __forceinline__ Val val(const double *p, const float *) { return __ldg(p); }
    static __device__ __forceinline__ void load(const double *p, const float *, double (&v)[4])
    {
        const double2 a = __ldg(reinterpret_cast<const double2 *>(p)), b = __ldg(reinterpret_cast<const double2 *>(p) + 1);
        v[0] = a.x, v[1] = a.y, v[2] = b.x, v[3] = b.y;
    }
    __device__ __forceinline__ void mac(int, double v, const ulonglong2 (&x)[NH])
    {
#pragma unroll
        for (int h = 0; h < NH; ++h) {
            acc[2 * h] = fma(v, __longlong_as_double((long long)x[h].x), acc[2 * h]);
            acc[2 * h + 1] = fma(v, __longlong_as_double((long long)x[h].y), acc[2 * h + 1]);
        }
    }
    __device__ __forceinline__ void end_block(unsigned) {}
    __device__ __forceinline__ void single(int, double v, float sg, const ulonglong2 (&j)[NH], const ulonglong2 (&x)[NH])
    {
        const uint64_t flip = sg < 0.f ? 0x8000000000000000ull : 0ull;
#pragma unroll
        for (int h = 0; h < NH; ++h) {
            acc[2 * h] = fma(v + __longlong_as_double((long long)(j[h].x ^ flip)),
                             __longlong_as_double((long long)x[h].x), acc[2 * h]);
            acc[2 * h + 1] = fma(v + __longlong_as_double((long long)(j[h].y ^ flip)),
                                 __longlong_as_double((long long)x[h].y), acc[2 * h + 1]);
        }
    }
    __device__ __forceinline__ void end_singles() {}
    __device__ __forceinline__ double value(int h, int i) const { return acc[2 * h + i]; }
    static __device__ __forceinline__ void store(unsigned char *line, int row, double x)
    {
        reinterpret_cast<double *>(line)[(row & 7) * 2 + (row >> 3)] = x;
    }
    static __device__ __forceinline__ ulonglong2 chunk(const double (&x)[2])
    {
        return make_ulonglong2((uint64_t)__double_as_longlong(x[0]), (uint64_t)__double_as_longlong(x[1]));
    }
};

template <int NH>
struct RangeAcc<F2, NH> {
    static constexpr int kRowsPerChunk = 2;
    using Val = float2;
    uint64_t bh[NH], bl[NH], hi[NH], lo[NH];  // a block's sum, and the sum of the blocks
    __device__ __forceinline__ void zero()
    {
#pragma unroll
        for (int h = 0; h < NH; ++h) hi[h] = lo[h] = 0ull;
    }
    static __device__ __forceinline__ Val val(const float *hi, const float *lo) { return make_float2(__ldg(hi), __ldg(lo)); }
    static __device__ __forceinline__ void load(const float *hi, const float *lo, float2 (&v)[4])
    {
        const float4 a = __ldg(reinterpret_cast<const float4 *>(hi)), b = __ldg(reinterpret_cast<const float4 *>(lo));
        v[0] = make_float2(a.x, b.x), v[1] = make_float2(a.y, b.y);
        v[2] = make_float2(a.z, b.z), v[3] = make_float2(a.w, b.w);
    }
    __device__ __forceinline__ void mac2(bool first, int h, uint64_t ah, uint64_t an, uint64_t al, ulonglong2 b)
    {
        if (first) pk_f2_mul(bh[h], bl[h], ah, an, al, b);
        else pk_f2_mac(bh[h], bl[h], ah, an, al, b);
    }
    __device__ __forceinline__ void mac(int u, float2 v, const ulonglong2 (&x)[NH])
    {
        const uint64_t ah = pk_dup(v.x), an = pk_dup(-v.x), al = pk_dup(v.y);
#pragma unroll
        for (int h = 0; h < NH; ++h) mac2(u == 0, h, ah, an, al, x[h]);
    }
    // A block is summed by itself and then added: one chain over a list rounds its low part at the size of
    // the whole sum with every entry (error of products of 300 x 300 strings, norb 24: 1.10e-15, 0.93e-15 with
    // eight lanes to a list; this costs no more, the first product of a block needs no sum).
    __device__ __forceinline__ void end_block(unsigned)
    {
#pragma unroll
        for (int h = 0; h < NH; ++h) pk_f2_add(hi[h], lo[h], bh[h], bl[h]);
    }
    __device__ __forceinline__ void single(int, float2 v, float sg, const ulonglong2 (&j)[NH], const ulonglong2 (&x)[NH])
    {
        const uint64_t ss = pk_dup(sg), sn = pk_dup(-sg);
        mac(0, v, x);
#pragma unroll
        for (int h = 0; h < NH; ++h)
            mac2(false, h, pk_mul(ss, j[h].x), pk_mul(sn, j[h].x), pk_mul(ss, j[h].y), x[h]);
        end_block(0);
    }
    __device__ __forceinline__ void end_singles() {}
    __device__ __forceinline__ double value(int h, int i) const
    {
        return (double)pk_get(hi[h], i) + (double)pk_get(lo[h], i);
    }
    static __device__ __forceinline__ void store(unsigned char *line, int row, double x)
    {
        const F2 s = f2_split(x);
        float *f = reinterpret_cast<float *>(line) + (row & 7) * 4 + (row >> 3);
        f[0] = s.hi;
        f[2] = s.lo;
    }
    static __device__ __forceinline__ ulonglong2 chunk(const double (&x)[2])
    {
        const F2 a = f2_split(x[0]), b = f2_split(x[1]);
        return make_ulonglong2(pk_pair(a.hi, b.hi), pk_pair(a.lo, b.lo));
    }
};

// Rows row0 .. row0 + kRangeRows - 1, output strings of the parts [p0, p1).
template <typename T>
__device__ __forceinline__ void range_rows(const RangeArgs<T> &a, int64_t row0, int p0, int p1, unsigned char *smem)
{
    using Acc = RangeAcc<T>;
    using In = typename RangeIn<T>::type;
    constexpr int ROWS = kRangeRows<T>, RPC = Acc::kRowsPerChunk, LPW = 32 / ROWS;  // LPW: lines a warp stages at once
    constexpr int kWarps = kRangeThreads / 32;
    // the FP64-accurate arithmetics have no registers left for a second block (pairs: 7.8 -> 7.9 ms)
    constexpr int kAhead = sizeof(T) == 4 ? 2 : 1;
    unsigned char *Js = smem + (size_t)a.w * kRangeRowBytes;  // [npair + 1] lines, or a line of zeros, behind the w lines
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int lst = lane >> 2, l = lane & 3;  // list of the group, lane of the list
    const int nr = (int)min((int64_t)ROWS, a.nrow - row0);
    const int sr = lane & (ROWS - 1), sub = lane / ROWS;  // staging: row and line of the lane
    const bool srow = sr < nr;
    // the lane's chunks of a line and its first rows in them
    const int c0 = l + 4 * (lst & 1), c1 = c0 ^ 4;
    unsigned rmax = 0u;
    __shared__ unsigned rmax_s[ROWS];
    __shared__ unsigned next_s;
    __syncthreads();  // the previous rows are finished with shared memory
    if (threadIdx.x < ROWS) rmax_s[threadIdx.x] = 0u;
    if (a.jstaged) {
        for (int p = warp * LPW + sub; p <= a.npair; p += kWarps * LPW)
            Acc::store(Js + (size_t)p * kRangeRowBytes, sr,
                       p < a.npair && srow ? __ldg(a.jg + (int64_t)p * a.nrow + row0 + sr) : 0.0);
    } else if (threadIdx.x < kRangeRowBytes / 16) {
        reinterpret_cast<float4 *>(Js)[threadIdx.x] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    const int64_t groups = part_group(a.n, kParts);
    // Groups are taken from a counter (their lengths differ, and the range ends with a barrier) in the
    // order: the first (longest) of every part, the second of every part, ...
    const unsigned np = p1 - p0, most = (unsigned)(part_group(a.n, p0 + 1) - part_group(a.n, p0)) * np;
    auto group_of = [&](unsigned i, unsigned &q) {  // the i-th to be taken; false where a part has one less
        const unsigned gi = i / np, p = p0 + (i - gi * np);
        q = (unsigned)part_group(a.n, (int)p) + gi;
        return i < most && q < (unsigned)part_group(a.n, (int)p + 1);
    };
    for (int g = 0; g < a.ng; ++g) {
        if (g) __syncthreads();  // every warp is finished with the previous range
        if (threadIdx.x == 0) next_s = kWarps;
        const int64_t j0 = (int64_t)g * a.w;
        const int wj = (int)min((int64_t)a.w, a.n - j0);
        const In *src = a.X + j0 * a.nrow + row0 + sr;
        for (int jb = warp * LPW + sub; jb < wj; jb += 8 * kWarps * LPW) {
            In v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int j = jb + u * kWarps * LPW;
                v[u] = (j < wj && srow) ? src[(int64_t)j * a.nrow] : In(0);
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int j = jb + u * kWarps * LPW;
                if (j < wj) Acc::store(smem + (size_t)j * kRangeRowBytes, sr, (double)v[u]);
                if constexpr (sizeof(T) == 4) rmax = max(rmax, __float_as_uint(fabsf(v[u])));
            }
        }
        __syncthreads();
        const unsigned char *x0 = smem + c0 * 16, *x1 = smem + c1 * 16;
        const bool add = g > 0 || a.accumulate;
        const int32_t *zi_g = a.zi + (int64_t)g * groups * kListGroup + lst;
        const uint32_t *qd_g = a.qd + (int64_t)g * groups, *qs_g = a.qs + (int64_t)g * groups;
        unsigned i = warp, q = 0;
        int zi = -1;
        uint32_t db = 0, de = 0, sb = 0, se = 0;
        if (group_of(i, q)) zi = zi_g[(int64_t)q * kListGroup], db = qd_g[q], de = qd_g[q + 1], sb = qs_g[q], se = qs_g[q + 1];
        while (i < most) {  // uniform over the warp
            if (lane == 0) i = atomicAdd(&next_s, 1u);
            i = __shfl_sync(0xffffffffu, i, 0);
            int zi_n = -1;
            uint32_t db_n = 0, de_n = 0, sb_n = 0, se_n = 0;  // the next group's bounds
            if (group_of(i, q))
                zi_n = zi_g[(int64_t)q * kListGroup], db_n = qd_g[q], de_n = qd_g[q + 1], sb_n = qs_g[q], se_n = qs_g[q + 1];
            if (!add || db < de || sb < se) {
                Acc acc;
                acc.zero();
                for (uint32_t b = sb; b < se; ++b) {
                    const size_t at = (size_t)b * kListGroup + lst;
                    const uint2 m2 = __ldg(reinterpret_cast<const uint2 *>(a.sm) + at);
                    const uint32_t m[2] = {m2.x, m2.y};
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        const typename Acc::Val v = Acc::val(a.sv + at * 2 + u, a.slo + at * 2 + u);
                        const uint32_t jo = (m[u] & 0xffffu) * kRangeRowBytes;
                        const int pr = (int)((m[u] >> 16) & 0x7fffu);
                        const ulonglong2 x[2] = {*reinterpret_cast<const ulonglong2 *>(x0 + jo),
                                                 *reinterpret_cast<const ulonglong2 *>(x1 + jo)};
                        ulonglong2 jv[2];
                        if (a.jstaged) {
                            jv[0] = *reinterpret_cast<const ulonglong2 *>(Js + pr * kRangeRowBytes + c0 * 16);
                            jv[1] = *reinterpret_cast<const ulonglong2 *>(Js + pr * kRangeRowBytes + c1 * 16);
                        } else {
                            double t[2][RPC];
#pragma unroll
                            for (int h = 0; h < 2; ++h)
#pragma unroll
                                for (int i = 0; i < RPC; ++i) {
                                    const int r = (h ? c1 : c0) + 8 * i;
                                    t[h][i] = pr < a.npair && r < nr ? __ldg(a.jg + (int64_t)pr * a.nrow + row0 + r) : 0.0;
                                }
                            jv[0] = Acc::chunk(t[0]);
                            jv[1] = Acc::chunk(t[1]);
                        }
                        acc.single(u, v, (m[u] >> 31) ? -1.f : 1.f, jv, x);
                    }
                }
                acc.end_singles();
                // doubles, a block of four entries at a time, loaded kAhead blocks ahead
                if (db < de) {
                    typename Acc::Val v[kAhead][4];
                    uint2 t4[kAhead];
                    const uint2 *tp = reinterpret_cast<const uint2 *>(a.dt) + (size_t)db * kListGroup + lst;
                    const typename RangeVal<T>::type *vp = a.dv + ((size_t)db * kListGroup + lst) * 4;
                    const float *lp = a.dlo + ((size_t)db * kListGroup + lst) * 4;
                    const unsigned nb = de - db;
#pragma unroll
                    for (int s = 0; s < kAhead; ++s)
                        if (s < nb) {
                            t4[s] = __ldg(tp + s * kListGroup);
                            Acc::load(vp + s * kListGroup * 4, lp + s * kListGroup * 4, v[s]);
                        }
                    for (unsigned b = 0; b < nb; b += kAhead) {
#pragma unroll
                        for (int s = 0; s < kAhead; ++s) {
                            if (b + s >= nb) break;
                            const uint2 t = t4[s];
                            const typename Acc::Val c[4] = {v[s][0], v[s][1], v[s][2], v[s][3]};
                            if (b + s + kAhead < nb) {
                                t4[s] = __ldg(tp + (s + kAhead) * kListGroup);
                                Acc::load(vp + (s + kAhead) * kListGroup * 4, lp + (s + kAhead) * kListGroup * 4, v[s]);
                            }
                            const uint32_t j[4] = {t.x & 0xffffu, t.x >> 16, t.y & 0xffffu, t.y >> 16};
#pragma unroll
                            for (int u = 0; u < 4; ++u) {
                                const uint32_t jo = j[u] * kRangeRowBytes;
                                const ulonglong2 x[2] = {*reinterpret_cast<const ulonglong2 *>(x0 + jo),
                                                         *reinterpret_cast<const ulonglong2 *>(x1 + jo)};
                                acc.mac(u, c[u], x);
                            }
                            acc.end_block(b + s + 1);
                        }
                        tp += kAhead * kListGroup;
                        vp += kAhead * kListGroup * 4;
                        lp += kAhead * kListGroup * 4;
                    }
                }
                if (zi >= 0 && (!add || (zi & kListHas))) {  // the string's sum changes Y
                    double *y = a.Y + (int64_t)(zi & ~kListHas) * a.nrow + row0;
                    double yo[2][RPC];
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int i = 0; i < RPC; ++i) {
                            const int r = (h ? c1 : c0) + 8 * i;
                            yo[h][i] = add && r < nr ? y[r] : 0.0;
                        }
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int i = 0; i < RPC; ++i) {
                            const int r = (h ? c1 : c0) + 8 * i;
                            if (r < nr) y[r] = (zi & kListHas) ? yo[h][i] + acc.value(h, i) : 0.0;
                        }
                }
            }
            zi = zi_n, db = db_n, de = de_n, sb = sb_n, se = se_n;
        }
    }
    if constexpr (sizeof(T) == 4) {
        if (a.rowmax && p0 == 0) {  // uniform over the CTA
            atomicMax(rmax_s + sr, rmax);
            __syncthreads();
            if (threadIdx.x < nr) a.rowmax[row0 + threadIdx.x] = __uint_as_float(rmax_s[threadIdx.x]);
        }
    }
}

// The same sums for lists of one range and few strings: two warps share a group, each with one chunk of a line
// per lane (half of the rows).  With one or two groups to a CTA a pass takes as long as one warp takes for its
// lists (FP64 product of 100 x 100 strings, norb 12: 119 -> 99 us).
// DIRECT: X and Y have the rows outside, [nrow][n], and the diagonal term hd x64 (null: hd X) is added.  The two
// transposes of a small product cost more as launches (8 us) than the scattered accesses.
template <typename T, bool DIRECT>
__device__ __forceinline__ void range_small(const RangeArgs<T> &a, const double *__restrict__ hd,
                                            const double *__restrict__ x64, int64_t row0, int p0, int p1,
                                            unsigned char *smem)
{
    using Acc = RangeAcc<T, 1>;
    using In = typename RangeIn<T>::type;
    constexpr int ROWS = kRangeRows<T>, RPC = Acc::kRowsPerChunk, LPW = 32 / ROWS;
    constexpr int kWarps = kRangeThreads / 32;
    unsigned char *Js = smem + (size_t)a.w * kRangeRowBytes;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int lst = lane >> 2, l = lane & 3;
    const int nr = (int)min((int64_t)ROWS, a.nrow - row0);
    const int sr = lane & (ROWS - 1), sub = lane / ROWS;
    const bool srow = sr < nr;
    unsigned rmax = 0u;
    __shared__ unsigned rmax_s[ROWS];
    __syncthreads();  // the previous rows are finished with shared memory
    if (threadIdx.x < ROWS) rmax_s[threadIdx.x] = 0u;
    if (a.jstaged) {
        for (int p = warp * LPW + sub; p <= a.npair; p += kWarps * LPW)
            Acc::store(Js + (size_t)p * kRangeRowBytes, sr,
                       p < a.npair && srow ? __ldg(a.jg + (int64_t)p * a.nrow + row0 + sr) : 0.0);
    } else if (threadIdx.x < kRangeRowBytes / 16) {
        reinterpret_cast<float4 *>(Js)[threadIdx.x] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    const In *src = a.X + (DIRECT ? (row0 + sr) * a.n : row0 + sr);
    const int64_t sj = DIRECT ? 1 : a.nrow;  // between the amplitudes of a row
    for (int jb = warp * LPW + sub; jb < a.n; jb += 8 * kWarps * LPW) {
        In v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int j = jb + u * kWarps * LPW;
            v[u] = (j < a.n && srow) ? src[j * sj] : In(0);
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int j = jb + u * kWarps * LPW;
            if (j < a.n) Acc::store(smem + (size_t)j * kRangeRowBytes, sr, (double)v[u]);
            if constexpr (sizeof(T) == 4) rmax = max(rmax, __float_as_uint(fabsf(v[u])));
        }
    }
    __syncthreads();
    const int q0 = (int)part_group(a.n, p0), q1 = (int)part_group(a.n, p1);
    for (int task = warp; task < 2 * (q1 - q0); task += kWarps) {
        const int q = q0 + (task >> 1);
        const int c = (l + 4 * (lst & 1)) ^ (4 * (task & 1));
        const unsigned char *x0 = smem + c * 16;
        const int zi = a.zi[(int64_t)q * kListGroup + lst];
        const uint32_t db = a.qd[q], de = a.qd[q + 1], sb = a.qs[q], se = a.qs[q + 1];
        Acc acc;
        acc.zero();
        uint2 m_n = make_uint2(0u, 0u);  // the next block of singles
        typename Acc::Val v_n[2] = {};
        const auto load_singles = [&](uint32_t b) {
            const size_t at = (size_t)b * kListGroup + lst;
            m_n = __ldg(reinterpret_cast<const uint2 *>(a.sm) + at);
            v_n[0] = Acc::val(a.sv + at * 2, a.slo + at * 2), v_n[1] = Acc::val(a.sv + at * 2 + 1, a.slo + at * 2 + 1);
        };
        if (sb < se) load_singles(sb);
        for (uint32_t b = sb; b < se; ++b) {
            const uint32_t m[2] = {m_n.x, m_n.y};
            const typename Acc::Val v[2] = {v_n[0], v_n[1]};
            if (b + 1 < se) load_singles(b + 1);
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int pr = (int)((m[u] >> 16) & 0x7fffu);
                const ulonglong2 x[1] = {*reinterpret_cast<const ulonglong2 *>(x0 + (m[u] & 0xffffu) * kRangeRowBytes)};
                ulonglong2 j[1];
                if (a.jstaged) {
                    j[0] = *reinterpret_cast<const ulonglong2 *>(Js + pr * kRangeRowBytes + c * 16);
                } else {
                    double t[RPC];
#pragma unroll
                    for (int i = 0; i < RPC; ++i) {
                        const int r = c + 8 * i;
                        t[i] = pr < a.npair && r < nr ? __ldg(a.jg + (int64_t)pr * a.nrow + row0 + r) : 0.0;
                    }
                    j[0] = Acc::chunk(t);
                }
                acc.single(u, v[u], (m[u] >> 31) ? -1.f : 1.f, j, x);
            }
        }
        acc.end_singles();
        const uint2 *tp = reinterpret_cast<const uint2 *>(a.dt) + (size_t)db * kListGroup + lst;
        const typename RangeVal<T>::type *vp = a.dv + ((size_t)db * kListGroup + lst) * 4;
        const float *lp = a.dlo + ((size_t)db * kListGroup + lst) * 4;
        const unsigned nb = de - db;
        constexpr int kAhead = 2;
        typename Acc::Val v[kAhead][4];
        uint2 t4[kAhead];
#pragma unroll
        for (int s = 0; s < kAhead; ++s)
            if (s < nb) {
                t4[s] = __ldg(tp + s * kListGroup);
                Acc::load(vp + s * kListGroup * 4, lp + s * kListGroup * 4, v[s]);
            }
        for (unsigned b = 0; b < nb; b += kAhead) {
#pragma unroll
            for (int s = 0; s < kAhead; ++s) {
                if (b + s >= nb) break;
                const uint2 t = t4[s];
                const typename Acc::Val val[4] = {v[s][0], v[s][1], v[s][2], v[s][3]};
                if (b + s + kAhead < nb) {
                    t4[s] = __ldg(tp + (s + kAhead) * kListGroup);
                    Acc::load(vp + (s + kAhead) * kListGroup * 4, lp + (s + kAhead) * kListGroup * 4, v[s]);
                }
                const uint32_t j[4] = {t.x & 0xffffu, t.x >> 16, t.y & 0xffffu, t.y >> 16};
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const ulonglong2 x[1] = {*reinterpret_cast<const ulonglong2 *>(x0 + j[u] * kRangeRowBytes)};
                    acc.mac(u, val[u], x);
                }
                acc.end_block(b + s + 1);
            }
            tp += kAhead * kListGroup;
            vp += kAhead * kListGroup * 4;
            lp += kAhead * kListGroup * 4;
        }
        if (zi < 0) continue;
        const bool has = zi & kListHas;
        const int64_t i = zi & ~kListHas;
#pragma unroll
        for (int k = 0; k < RPC; ++k) {
            const int r = c + 8 * k;
            if (r >= nr) continue;
            const int64_t at = DIRECT ? (row0 + r) * a.n + i : i * a.nrow + row0 + r;
            double y = has ? acc.value(0, k) : 0.0;
            if (DIRECT) y = fma(hd[at], x64 ? x64[at] : (double)a.X[at], y);
            if (DIRECT || has || !a.accumulate) a.Y[at] = a.accumulate ? a.Y[at] + y : y;
        }
    }
    if constexpr (sizeof(T) == 4) {
        if (a.rowmax && p0 == 0) {  // uniform over the CTA
            atomicMax(rmax_s + sr, rmax);
            __syncthreads();
            if (threadIdx.x < nr) a.rowmax[row0 + threadIdx.x] = __uint_as_float(rmax_s[threadIdx.x]);
        }
    }
}

}  // namespace sbd

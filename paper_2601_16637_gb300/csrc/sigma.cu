// Matrix-free sigma product s = H c on the selected space A x B (paper
// Sec. II-A/B, Eq. 4; the three task types of Sec. III-B).
//
// With E_pq split by spin, H = H_alpha (x) 1 + 1 (x) H_beta + V_ab where
//   H_alpha(I,J) = <I| sum h_pq E_pq + 1/2 sum (pq|rs)(E_pq E_rs - d_qr E_ps) |J>
// evaluated by the same-spin Slater-Condon rules between alpha strings, and
//   V_ab = sum_pqrs (pq|rs) E^alpha_pq E^beta_rs.
// Because every alpha operator pair commutes with the beta creators, the
// phases factorise: <Ia Ib|E^a_pq E^b_rs|Ja Jb> = <Ia|E_pq|Ja><Ib|E_rs|Jb>.
// With J_x[uv] = sum_{k in x} (uv|kk) this gives, for output (ia, ib):
//   s = Hd(ia,ib) c(ia,ib)                                          diagonal
//     + sum_{jb in doubles(ib)} Hb(ib,jb) c(ia,jb)
//     + sum_{jb in singles(ib), code rs, phase t} [Hb(ib,jb) + t J_ia[rs]] c(ia,jb)
//     + sum_{ja in doubles(ia)} Ha(ia,ja) c(ja,ib)
//     + sum_{ja in singles(ia), code pq, phase u} [Ha(ia,ja) + u J_ib[pq]] c(ja,ib)
//     + sum_{ja in singles(ia)} sum_{jb in singles(ib)} u t (pq|rs) c(ja,jb)
// The second and third line are a gather inside row ia of C ("beta pass"), the next two the same
// gather inside column ib ("alpha pass", same kernel: range_rows.cuh), and the last line is the
// alpha-beta pass.  The beta pass runs on the transpose of C and leaves its result transposed; the
// pass that transposes it back adds the diagonal term (in FP64 and pairs last of all: the sums of the other
// passes are then rounded at their own size, error of an FP64 product 4.7e-16 -> 4.2e-16 at norb 29).
//
// Every output element is owned by one thread group in each pass and each pass adds into it in
// program order, so results are deterministic.
//
// Row-block products (alpha-row sharding), the engine's mixed row passes and the two-operand alpha-beta
// pass stage whole rows of C in shared memory, R rows interleaved per column so one vector load fetches the same column of all
// R rows; each lane of an 8-lane group fetches 4 entries of the padded sigma copies of the lists with
// 16-byte loads, and the next column's list bounds are prefetched.  The phase of a single is folded
// into the shared-memory coefficient tables, which are indexed by 2*code + (phase<0).
// Precision T = double (FP64), float (mixed: FP32 amplitudes, integrals,
// products and per-list sums, each list sum and the diagonal term accumulated
// into the FP64 output), or F2 (FP64-accurate arithmetic on the FP32 pipe:
// every amplitude, integral and matrix element is an unevaluated sum hi + lo
// of two floats, products are exact hi*hi (a fused multiply-add recovers the
// rounding error, Dekker's product) plus the two cross terms, and sums use
// Knuth's two-sum; on GB300 the FP32 pipe is ~64x the FP64 pipe).
#include <string.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "pair.cuh"
#include "range_rows.cuh"

namespace sbd {

namespace {

constexpr int kGroup = 8;  // lanes cooperating on one output column
constexpr int kGroupsPerWarp = 32 / kGroup;

template <typename T>
constexpr bool kIsF2 = std::is_same<T, F2>::value;

// element type of the vectors a pass reads (the pair precision reads FP64 vectors)
template <typename T>
struct In {
    using type = T;
};
template <>
struct In<F2> {
    using type = double;
};

template <typename T>
__device__ __forceinline__ T conv(double x)
{
    if constexpr (kIsF2<T>) return f2_split(x);
    else return (T)x;
}
template <typename T>
__device__ __forceinline__ T conv(float x)
{
    return (T)x;
}

template <typename T>
struct Threads;
template <>
struct Threads<F2> {
    static constexpr int value = 1024;  // latency-bound at 512 (209 vs 292 ms per sigma at 1.0e8 dets)
};
template <>
struct Threads<float> {
    static constexpr int value = 1024;
};
template <>
struct Threads<double> {
    static constexpr int value = 512;
};

template <typename T, int R>
struct VecIO;
template <>
struct VecIO<float, 4> {
    __device__ static void ld(const float *p, float (&v)[4])
    {
        const float4 x = *reinterpret_cast<const float4 *>(p);
        v[0] = x.x;
        v[1] = x.y;
        v[2] = x.z;
        v[3] = x.w;
    }
    __device__ static void st(float *p, const float (&v)[4])
    {
        *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
    }
};
template <>
struct VecIO<float, 2> {
    __device__ static void ld(const float *p, float (&v)[2])
    {
        const float2 x = *reinterpret_cast<const float2 *>(p);
        v[0] = x.x;
        v[1] = x.y;
    }
    __device__ static void st(float *p, const float (&v)[2])
    {
        *reinterpret_cast<float2 *>(p) = make_float2(v[0], v[1]);
    }
};
template <>
struct VecIO<double, 2> {
    __device__ static void ld(const double *p, double (&v)[2])
    {
        const double2 x = *reinterpret_cast<const double2 *>(p);
        v[0] = x.x;
        v[1] = x.y;
    }
    __device__ static void st(double *p, const double (&v)[2])
    {
        *reinterpret_cast<double2 *>(p) = make_double2(v[0], v[1]);
    }
};
template <>
struct VecIO<F2, 2> {
    __device__ static void ld(const F2 *p, F2 (&v)[2])
    {
        const float4 x = *reinterpret_cast<const float4 *>(p);
        v[0] = F2(x.x, x.y);
        v[1] = F2(x.z, x.w);
    }
    __device__ static void st(F2 *p, const F2 (&v)[2])
    {
        *reinterpret_cast<float4 *>(p) = make_float4(v[0].hi, v[0].lo, v[1].hi, v[1].lo);
    }
};
template <>
struct VecIO<F2, 1> {
    __device__ static void ld(const F2 *p, F2 (&v)[1])
    {
        const float2 x = *reinterpret_cast<const float2 *>(p);
        v[0] = F2(x.x, x.y);
    }
    __device__ static void st(F2 *p, const F2 (&v)[1]) { *reinterpret_cast<float2 *>(p) = make_float2(v[0].hi, v[0].lo); }
};
template <typename T>
struct VecIO<T, 1> {
    __device__ static void ld(const T *p, T (&v)[1]) { v[0] = *p; }
    __device__ static void st(T *p, const T (&v)[1]) { *p = v[0]; }
};

template <int R, typename T>
__device__ __forceinline__ T pick(const T (&v)[R], int i)
{
    T out = v[0];
#pragma unroll
    for (int r = 1; r < R; ++r)
        if (i == r) out = v[r];
    return out;
}

__host__ __device__ constexpr size_t round16(size_t b) { return (b + 15) & ~(size_t)15; }

__device__ __forceinline__ int pk_j(uint32_t pk) { return (int)(pk & kPackJMask); }
__device__ __forceinline__ int pk_key(uint32_t pk) { return (int)(pk >> kPackKeyShift); }  // 2*code + neg
__device__ __forceinline__ int pk_code(uint32_t pk) { return (int)(pk >> (kPackKeyShift + 1)); }
__device__ __forceinline__ bool pk_neg(uint32_t pk) { return ((pk >> kPackKeyShift) & 1u) != 0u; }

// Excitation lists of the column spin (SigLists), as each precision reads them.  Every list starts at a
// multiple of kListPad entries.  The 8 lanes of a group read a list in chunks of up to 32 slots: in a
// chunk, lane l takes slots 4l..4l+3, and entry u of the lane is the slot the u-th 128-bit shared-memory
// phase of the pass gathers for that lane.
__device__ __forceinline__ void load4(const uint32_t *p, uint32_t (&v)[4])
{
    const uint4 a = __ldg(reinterpret_cast<const uint4 *>(p));
    v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w;
}
__device__ __forceinline__ void load4(const int32_t *p, int (&v)[4])
{
    const int4 a = __ldg(reinterpret_cast<const int4 *>(p));
    v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w;
}
__device__ __forceinline__ void load4(const float *p, const float *, float (&v)[4])
{
    const float4 a = __ldg(reinterpret_cast<const float4 *>(p));
    v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w;
}
__device__ __forceinline__ void load4(const double *p, const float *, double (&v)[4])
{
    const double2 a = __ldg(reinterpret_cast<const double2 *>(p)), b = __ldg(reinterpret_cast<const double2 *>(p) + 1);
    v[0] = a.x, v[1] = a.y, v[2] = b.x, v[3] = b.y;
}
__device__ __forceinline__ void load4(const float *p, const float *q, F2 (&v)[4])
{
    const float4 a = __ldg(reinterpret_cast<const float4 *>(p)), b = __ldg(reinterpret_cast<const float4 *>(q));
    v[0] = F2(a.x, b.x), v[1] = F2(a.y, b.y), v[2] = F2(a.z, b.z), v[3] = F2(a.w, b.w);
}

template <typename T>
struct Lists {
    using V = typename RangeVal<T>::type;
    const uint32_t *spk;
    const V *sv;
    const float *slo;
    const int32_t *dj;
    const V *dv;
    const float *dlo;
    __device__ void singles4(int64_t e, uint32_t (&pk)[4], T (&v)[4]) const
    {
        load4(spk + e, pk);
        load4(sv + e, slo + e, v);
    }
    __device__ void doubles4(int64_t e, int (&j)[4], T (&v)[4]) const
    {
        load4(dj + e, j);
        load4(dv + e, dlo + e, v);
    }
};

template <typename T>
struct RowArgs {
    const typename In<T>::type *X;  // [nrow][ncol]
    int64_t nrow, ncol;
    int64_t ncol_out;  // output columns (list sources); ncol except for row-block sigma
    double *Y;  // output element (row r, column c) at r*y_rs + c*y_cs
    int64_t y_rs, y_cs;
    int accumulate;
    const double *hd;    // optional diagonal, indexed like Y
    const double *xd64;  // optional FP64 amplitudes [nrow][ncol] for the diagonal term
    float *rowmax;       // optional (FP32 only): rowmax[r] = max_c |X[r][c]| of every row of the pass
    const uint64_t *row_strings;
    int norb;
    const double *eri;  // FP64 integrals, for the J vectors of the staged rows
    const int64_t *s_ptr, *d_ptr;
    Lists<T> lists;
    // mixed passes over column halves (row_halves): the column spin's lists split at `half`
    const int64_t *hls_ptr, *hld_ptr;  // singles, doubles: [2n + 1]
    const uint2 *hls;                  // (packed single, FP32 value bits)
    const float *hldv;                 // doubles: FP32 values
    const uint16_t *hldt;              // doubles: targets relative to their column half
    int64_t half;
};

// Gather pass over rows of X: each CTA stages R consecutive rows, then every
// output column c sums its excitation list (column spin) inside those rows.
// row_group() does one group of rows starting at r0; the single-instance
// kernel strides over the groups, the batched kernel takes (instance, group)
// items from a work counter.
template <typename T, int R, bool STAGED>
__device__ __forceinline__ void row_group(const RowArgs<T> &a, int64_t r0, unsigned char *smem)
{
    constexpr int kThreads = Threads<T>::value;
    const int n2 = a.norb * a.norb;
    const size_t xs_bytes = STAGED ? round16((size_t)a.ncol * R * sizeof(T)) : 0;
    T *Xs = reinterpret_cast<T *>(smem);
    T *Js = reinterpret_cast<T *>(smem + xs_bytes);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int gi = lane / kGroup, lig = lane % kGroup;
    const int64_t ngroups = (kThreads / 32) * kGroupsPerWarp;
    {
        const int nr = (int)min((int64_t)R, a.nrow - r0);
        __syncthreads();
        // row maxima (FP32 pass only): largest |x| as the bit pattern of a non-negative float, so a
        // NaN amplitude leaves a NaN maximum
        unsigned rmax[R];
#pragma unroll
        for (int r = 0; r < R; ++r) rmax[r] = 0u;
        constexpr bool kMax = std::is_same<T, float>::value;
        if (STAGED) {
            for (int64_t c = tid; c < a.ncol; c += kThreads) {
                T v[R];
#pragma unroll
                for (int r = 0; r < R; ++r) v[r] = r < nr ? conv<T>(a.X[(r0 + r) * a.ncol + c]) : T(0);
                VecIO<T, R>::st(Xs + c * R, v);
                if constexpr (kMax) {
#pragma unroll
                    for (int r = 0; r < R; ++r) rmax[r] = max(rmax[r], __float_as_uint(fabsf(v[r])));
                }
            }
        } else if constexpr (kMax) {
            if (a.rowmax)
                for (int64_t c = tid; c < a.ncol; c += kThreads) rmax[0] = max(rmax[0], __float_as_uint(fabsf(a.X[r0 * a.ncol + c])));
        }
        __shared__ unsigned red_max[kMax ? R : 1][kMax ? kThreads / 32 : 1];
        if constexpr (kMax) {
            if (a.rowmax) {
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const unsigned w = __reduce_max_sync(0xffffffffu, rmax[r]);
                    if (lane == 0) red_max[r][warp] = w;
                }
            }
        }
        // sign-folded J table: row key = 2*code + neg holds (neg ? -1 : 1) * J_r[code]; code 0 rows
        // stay zero (no single has code 0; padding entries point there)
        for (int key = tid; key < 2 * n2; key += kThreads) {
            const int code = key >> 1;
            T v[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                double s = 0.0;
                if (r < nr && code != 0)
                    for (uint64_t m = a.row_strings[r0 + r]; m; m &= m - 1ull) {
                        const int k = __ffsll((long long)m) - 1;
                        s += __ldg(a.eri + (size_t)code * n2 + (size_t)k * (a.norb + 1));
                    }
                v[r] = conv<T>((key & 1) ? -s : s);
            }
            VecIO<T, R>::st(Js + (size_t)key * R, v);
        }
        __syncthreads();
        if constexpr (kMax) {
            if (a.rowmax && tid < nr) {
                unsigned m = 0u;
                for (int w = 0; w < kThreads / 32; ++w) m = max(m, red_max[tid][w]);
                a.rowmax[r0 + tid] = __uint_as_float(m);
            }
        }

        int64_t cb = (int64_t)warp * kGroupsPerWarp;
        int64_t nxt_s0 = 0, nxt_s1 = 0, nxt_d0 = 0, nxt_d1 = 0;
        if (cb + gi < a.ncol_out) {
            nxt_s0 = a.s_ptr[cb + gi];
            nxt_s1 = a.s_ptr[cb + gi + 1];
            nxt_d0 = a.d_ptr[cb + gi];
            nxt_d1 = a.d_ptr[cb + gi + 1];
        }
        for (; cb < a.ncol_out; cb += ngroups) {
            const int64_t c = cb + gi;
            const bool valid = c < a.ncol_out;
            const int64_t s0 = nxt_s0, s1 = nxt_s1, d0 = nxt_d0, d1 = nxt_d1;
            if (c + ngroups < a.ncol_out) {  // prefetch the next column's list bounds
                nxt_s0 = a.s_ptr[c + ngroups];
                nxt_s1 = a.s_ptr[c + ngroups + 1];
                nxt_d0 = a.d_ptr[c + ngroups];
                nxt_d1 = a.d_ptr[c + ngroups + 1];
            }
            T acc[R];
#pragma unroll
            for (int r = 0; r < R; ++r) acc[r] = T(0);
            if (valid) {
                const int ls = (int)(s1 - s0), ld = (int)(d1 - d0);
                for (int cb = 0; cb < ls; cb += kGroup * kListPad) {
                    const int lc = min(kGroup * kListPad, ls - cb);
                    if (kListPad * lig >= lc) break;
                    uint32_t pk[4];
                    T v[4];
                    a.lists.singles4(s0 + cb + kListPad * lig, pk, v);
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        T xj[R], jv[R];
                        if (STAGED) VecIO<T, R>::ld(Xs + (size_t)pk_j(pk[u]) * R, xj);
                        else xj[0] = conv<T>(a.X[r0 * a.ncol + pk_j(pk[u])]);
                        VecIO<T, R>::ld(Js + (size_t)pk_key(pk[u]) * R, jv);
#pragma unroll
                        for (int r = 0; r < R; ++r) {
                            if constexpr (kIsF2<T>) {
                                f2_mac(acc[r], v[u], xj[r]);
                                f2_mac(acc[r], jv[r], xj[r]);
                            } else {
                                acc[r] += (v[u] + jv[r]) * xj[r];
                            }
                        }
                    }
                }
                for (int cb = 0; cb < ld; cb += kGroup * kListPad) {
                    const int lc = min(kGroup * kListPad, ld - cb);
                    if (kListPad * lig >= lc) break;
                    int jj[4];
                    T v[4];
                    a.lists.doubles4(d0 + cb + kListPad * lig, jj, v);
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        T xj[R];
                        if (STAGED) VecIO<T, R>::ld(Xs + (size_t)jj[u] * R, xj);
                        else xj[0] = conv<T>(a.X[r0 * a.ncol + jj[u]]);
#pragma unroll
                        for (int r = 0; r < R; ++r) {
                            if constexpr (kIsF2<T>) f2_mac(acc[r], v[u], xj[r]);
                            else acc[r] += v[u] * xj[r];
                        }
                    }
                }
            }
#pragma unroll
            for (int off = kGroup / 2; off > 0; off >>= 1)
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    if constexpr (kIsF2<T>) {
                        const F2 o(__shfl_xor_sync(0xffffffffu, acc[r].hi, off, kGroup),
                                   __shfl_xor_sync(0xffffffffu, acc[r].lo, off, kGroup));
                        acc[r] = f2_add(acc[r], o);
                    } else {
                        acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], off, kGroup);
                    }
                }
            if (valid && lig < nr) {
                double out;
                if constexpr (kIsF2<T>) out = f2_value(pick<R>(acc, lig));
                else out = (double)pick<R>(acc, lig);
                const int64_t idx = (r0 + lig) * a.y_rs + c * a.y_cs;
                if (a.hd) {
                    double xc;
                    if constexpr (kIsF2<T>) xc = a.X[(r0 + lig) * a.ncol + c];  // the FP64 input itself
                    else xc = a.xd64 ? a.xd64[(r0 + lig) * a.ncol + c]
                                     : (double)(STAGED ? Xs[(size_t)c * R + lig] : a.X[(r0 + lig) * a.ncol + c]);
                    out += a.hd[idx] * xc;
                }
                a.Y[idx] = a.accumulate ? a.Y[idx] + out : out;
            }
        }
    }
}

template <typename T, int R, bool STAGED>
__global__ void __launch_bounds__(Threads<T>::value) row_pass_kernel(const RowArgs<T> a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    for (int64_t r0 = (int64_t)blockIdx.x * R; r0 < a.nrow; r0 += (int64_t)gridDim.x * R) row_group<T, R, STAGED>(a, r0, smem);
}

// Mixed-precision gather pass over 8 rows, one column half at a time (the engine's 8-row setting).  With 4 rows the whole row
// range fits shared memory; staging 8 rows of one half ([0, half) or [half, ncol)) in the same space
// lets every excitation-list entry, loaded once from L2, feed 8 multiply-adds instead of 4.  Each
// output column sums its entries with targets in the staged half (the split lists of the column
// spin), writes that half's sum (with the diagonal term), and adds the other half's sum after the
// second staging.  The 8 rows are kept as two 4-row interleaved arrays, so a 16-byte gather per
// array has the bank pattern of the 4-row pass; the coefficient table of the singles likewise.
constexpr int kHalfRows = 8;

__host__ __device__ inline size_t halves_smem(int64_t half, int norb)
{
    return (size_t)32 * half + (size_t)64 * norb * norb;
}

__device__ __forceinline__ void row_halves(const RowArgs<float> &a, int64_t r0, unsigned char *smem)
{
    constexpr int kThreads = Threads<float>::value;
    const int n2 = a.norb * a.norb;
    const int64_t hw = a.half;  // rows of the staged arrays: the lower half is the wider one
    float *Xa = reinterpret_cast<float *>(smem);                   // [hw][4]  rows 0-3
    float *Xb = Xa + 4 * hw;                                        // [hw][4]  rows 4-7
    float *Ja = Xb + 4 * hw;                                        // [2 n2][4]
    float *Jb = Ja + 8 * n2;                                        // [2 n2][4]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int gi = lane / kGroup, lig = lane % kGroup;
    const int64_t ngroups = (kThreads / 32) * kGroupsPerWarp;
    const int nr = (int)min((int64_t)kHalfRows, a.nrow - r0);
    unsigned rmax[kHalfRows];
#pragma unroll
    for (int r = 0; r < kHalfRows; ++r) rmax[r] = 0u;
    __shared__ unsigned red_h[kHalfRows];
    __syncthreads();  // the previous row group is finished with shared memory
    if (tid < kHalfRows) red_h[tid] = 0u;
    // sign-folded J table of the 8 rows (row key = 2*code + neg; code 0 rows zero)
    for (int key = tid; key < 2 * n2; key += kThreads) {
        const int code = key >> 1;
        float v[kHalfRows];
#pragma unroll
        for (int r = 0; r < kHalfRows; ++r) {
            double sj = 0.0;
            if (r < nr && code != 0)
                for (uint64_t m = a.row_strings[r0 + r]; m; m &= m - 1ull) {
                    const int k = __ffsll((long long)m) - 1;
                    sj += __ldg(a.eri + (size_t)code * n2 + (size_t)k * (a.norb + 1));
                }
            v[r] = (float)((key & 1) ? -sj : sj);
        }
        *reinterpret_cast<float4 *>(Ja + (size_t)key * 4) = make_float4(v[0], v[1], v[2], v[3]);
        *reinterpret_cast<float4 *>(Jb + (size_t)key * 4) = make_float4(v[4], v[5], v[6], v[7]);
    }
    for (int h = 0; h < 2; ++h) {
        const int64_t c0 = h ? a.half : 0, c1 = h ? a.ncol : a.half;
        if (h) __syncthreads();  // every column is finished with the first half
        for (int64_t c = c0 + tid; c < c1; c += kThreads) {
            float v[kHalfRows];
#pragma unroll
            for (int r = 0; r < kHalfRows; ++r) v[r] = r < nr ? a.X[(r0 + r) * a.ncol + c] : 0.f;
            *reinterpret_cast<float4 *>(Xa + (c - c0) * 4) = make_float4(v[0], v[1], v[2], v[3]);
            *reinterpret_cast<float4 *>(Xb + (c - c0) * 4) = make_float4(v[4], v[5], v[6], v[7]);
#pragma unroll
            for (int r = 0; r < kHalfRows; ++r) rmax[r] = max(rmax[r], __float_as_uint(fabsf(v[r])));
        }
        __syncthreads();
        for (int64_t cb = (int64_t)warp * kGroupsPerWarp; cb < a.ncol_out; cb += ngroups) {
            const int64_t c = cb + gi;
            const bool valid = c < a.ncol_out;
            float acc[kHalfRows];
#pragma unroll
            for (int r = 0; r < kHalfRows; ++r) acc[r] = 0.f;
            if (valid) {
                const int64_t s0 = a.hls_ptr[2 * c + h], s1 = a.hls_ptr[2 * c + h + 1];
                const int64_t d0 = a.hld_ptr[2 * c + h], d1 = a.hld_ptr[2 * c + h + 1];
                const int ls = (int)(s1 - s0), ld = (int)(d1 - d0);
                for (int cb2 = 0; cb2 < ls; cb2 += kGroup * kListPad) {
                    const int lc = min(kGroup * kListPad, ls - cb2);
                    if (kListPad * lig >= lc) break;
                    const int64_t e0 = s0 + cb2 + kListPad * lig;
                    const uint4 p0 = __ldg(reinterpret_cast<const uint4 *>(a.hls + e0));
                    const uint4 p1 = __ldg(reinterpret_cast<const uint4 *>(a.hls + e0 + 2));
                    const uint32_t pk[4] = {p0.x, p0.z, p1.x, p1.z};
                    const float vv[4] = {__uint_as_float(p0.y), __uint_as_float(p0.w), __uint_as_float(p1.y),
                                         __uint_as_float(p1.w)};
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int64_t jl = (pk[u] ? (int64_t)pk_j(pk[u]) - c0 : 0);
                        const float4 xa = *reinterpret_cast<const float4 *>(Xa + jl * 4);
                        const float4 xb = *reinterpret_cast<const float4 *>(Xb + jl * 4);
                        const float4 ja = *reinterpret_cast<const float4 *>(Ja + (size_t)pk_key(pk[u]) * 4);
                        const float4 jb = *reinterpret_cast<const float4 *>(Jb + (size_t)pk_key(pk[u]) * 4);
                        acc[0] += (vv[u] + ja.x) * xa.x;
                        acc[1] += (vv[u] + ja.y) * xa.y;
                        acc[2] += (vv[u] + ja.z) * xa.z;
                        acc[3] += (vv[u] + ja.w) * xa.w;
                        acc[4] += (vv[u] + jb.x) * xb.x;
                        acc[5] += (vv[u] + jb.y) * xb.y;
                        acc[6] += (vv[u] + jb.z) * xb.z;
                        acc[7] += (vv[u] + jb.w) * xb.w;
                    }
                }
                for (int cb2 = 0; cb2 < ld; cb2 += kGroup * kListPad) {
                    const int lc = min(kGroup * kListPad, ld - cb2);
                    if (kListPad * lig >= lc) break;
                    const int64_t e0 = d0 + cb2 + kListPad * lig;
                    // entries e0 .. e0 + 3: four values (16 bytes) and four 16-bit targets (8 bytes)
                    const float4 v4 = __ldg(reinterpret_cast<const float4 *>(a.hldv + e0));
                    const uint2 t4 = __ldg(reinterpret_cast<const uint2 *>(a.hldt + e0));
                    const uint32_t jj[4] = {t4.x & 0xFFFFu, t4.x >> 16, t4.y & 0xFFFFu, t4.y >> 16};
                    const float vv[4] = {v4.x, v4.y, v4.z, v4.w};
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        // targets are relative to the staged half; padding entries: target 0, value 0
                        const int64_t jl = (int64_t)jj[u];
                        const float4 xa = *reinterpret_cast<const float4 *>(Xa + jl * 4);
                        const float4 xb = *reinterpret_cast<const float4 *>(Xb + jl * 4);
                        acc[0] += vv[u] * xa.x;
                        acc[1] += vv[u] * xa.y;
                        acc[2] += vv[u] * xa.z;
                        acc[3] += vv[u] * xa.w;
                        acc[4] += vv[u] * xb.x;
                        acc[5] += vv[u] * xb.y;
                        acc[6] += vv[u] * xb.z;
                        acc[7] += vv[u] * xb.w;
                    }
                }
            }
#pragma unroll
            for (int off = kGroup / 2; off > 0; off >>= 1)
#pragma unroll
                for (int r = 0; r < kHalfRows; ++r) acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], off, kGroup);
            if (valid && lig < nr) {
                double out = (double)pick<kHalfRows>(acc, lig);
                const int64_t idx = (r0 + lig) * a.y_rs + c * a.y_cs;
                if (h == 0) {
                    if (a.hd) {
                        const double xc = a.xd64 ? a.xd64[(r0 + lig) * a.ncol + c] : (double)a.X[(r0 + lig) * a.ncol + c];
                        out += a.hd[idx] * xc;
                    }
                    a.Y[idx] = a.accumulate ? a.Y[idx] + out : out;
                } else {
                    a.Y[idx] += out;
                }
            }
        }
    }
    if (a.rowmax) {  // uniform
#pragma unroll
        for (int r = 0; r < kHalfRows; ++r) {
            const unsigned w = __reduce_max_sync(0xffffffffu, rmax[r]);
            if (lane == 0) atomicMax(red_h + r, w);
        }
        __syncthreads();
        if (tid < nr) a.rowmax[r0 + tid] = __uint_as_float(red_h[tid]);
    }
}

// Row passes of whole instances (range_rows.cuh).  A unit is (row block, part): a CTA takes a run of
// consecutive units, so that all CTAs get the same number (+-1) and a row block's staging is shared
// by the units of a run.
template <typename T>
__global__ void __launch_bounds__(kRangeThreads, 1) range_rows_kernel(const RangeArgs<T> a, int64_t units)
{
    extern __shared__ __align__(16) unsigned char smem[];
    int64_t u = units * blockIdx.x / gridDim.x;
    const int64_t end = units * (blockIdx.x + 1) / gridDim.x;
    while (u < end) {
        const int p0 = (int)(u % kParts), p1 = (int)min((int64_t)kParts, p0 + (end - u));
        range_rows<T>(a, u / kParts * kRangeRows<T>, p0, p1, smem);
        u += p1 - p0;
    }
}

template <typename T, bool DIRECT>
__global__ void __launch_bounds__(kRangeThreads, 1) range_small_kernel(const RangeArgs<T> a, const double *hd,
                                                                      const double *x64, int64_t units)
{
    extern __shared__ __align__(16) unsigned char smem[];
    int64_t u = units * blockIdx.x / gridDim.x;
    const int64_t end = units * (blockIdx.x + 1) / gridDim.x;
    while (u < end) {
        const int p0 = (int)(u % kParts), p1 = (int)min((int64_t)kParts, p0 + (end - u));
        range_small<T, DIRECT>(a, hd, x64, u / kParts * kRangeRows<T>, p0, p1, smem);
        u += p1 - p0;
    }
}

template <typename T>
struct AbArgs {
    const typename In<T>::type *C;  // [nA][nB]
    double *S;                       // [nA][nB], accumulated
    int64_t nA, nB;
    int norb;
    const typename In<T>::type *eri;  // (pq|rs): FP32 [npair][npair], else [norb^2][norb^2]
    const int64_t *as_ptr;
    const uint32_t *as_pk;
    const int32_t *sl_col;  // beta singles in slices (SpinTables::sl_*)
    const uint32_t *sl_off, *sl_ent;
};

// R elements of one staged column or coefficient row, and a lane's sum over its entries.
template <typename T, int R>
struct AbVec {
    T v[R];
    __device__ static void st(T *p, const T (&v)[R]) { VecIO<T, R>::st(p, v); }
    __device__ __forceinline__ void ld(const T *p) { VecIO<T, R>::ld(p, v); }
};
// two pairs as (hi, hi, lo, lo): the packed arithmetic takes both at once
template <>
struct AbVec<F2, 2> {
    ulonglong2 v;
    __device__ static void st(F2 *p, const F2 (&x)[2])
    {
        *reinterpret_cast<float4 *>(p) = make_float4(x[0].hi, x[1].hi, x[0].lo, x[1].lo);
    }
    __device__ __forceinline__ void ld(const F2 *p) { v = *reinterpret_cast<const ulonglong2 *>(p); }
};

template <typename T, int R>
struct AbSum {  // FP64: one chain per row k
    T s[R];
    __device__ __forceinline__ void zero()
    {
#pragma unroll
        for (int k = 0; k < R; ++k) s[k] = T(0);
    }
    __device__ __forceinline__ void mac(int, const AbVec<T, R> &w, const AbVec<T, R> &c)
    {
#pragma unroll
        for (int k = 0; k < R; ++k) s[k] = fma(w.v[k], c.v[k], s[k]);
    }
    __device__ __forceinline__ void end_block() {}
    __device__ __forceinline__ double value() const
    {
        double t = (double)s[0];
#pragma unroll
        for (int k = 1; k < R; ++k) t += (double)s[k];
        return t;
    }
    __device__ __forceinline__ void add_lane(int off)
    {
#pragma unroll
        for (int k = 0; k < R; ++k) s[k] += __shfl_xor_sync(0xffffffffu, s[k], off);
    }
};
template <int R>
struct AbSum<float, R> {  // FP32: a short chain per block of entries
    float s, blk;
    __device__ __forceinline__ void zero() { s = blk = 0.f; }
    __device__ __forceinline__ void mac(int, const AbVec<float, R> &w, const AbVec<float, R> &c)
    {
#pragma unroll
        for (int k = 0; k < R; ++k) blk = fmaf(w.v[k], c.v[k], blk);
    }
    __device__ __forceinline__ void end_block()
    {
        s += blk;
        blk = 0.f;
    }
    __device__ __forceinline__ double value() const { return (double)s; }
    __device__ __forceinline__ void add_lane(int off) { s += __shfl_xor_sync(0xffffffffu, s, off); }
};
// pairs: a block of entries by itself, then added (as in the row passes)
template <>
struct AbSum<F2, 1> {
    F2 s, blk;
    __device__ __forceinline__ void zero() { s = F2(0.f); }
    __device__ __forceinline__ void mac(int i, const AbVec<F2, 1> &w, const AbVec<F2, 1> &c)
    {
        if (i == 0) blk = F2(0.f);
        f2_mac(blk, w.v[0], c.v[0]);
    }
    __device__ __forceinline__ void end_block() { s = f2_add(s, blk); }
    __device__ __forceinline__ double value() const { return f2_value(s); }
    __device__ __forceinline__ void add_lane(int off)
    {
        const F2 o(__shfl_xor_sync(0xffffffffu, s.hi, off), __shfl_xor_sync(0xffffffffu, s.lo, off));
        s = f2_add(s, o);
    }
};
template <>
struct AbSum<F2, 2> {
    uint64_t bh, bl, hi, lo;
    __device__ __forceinline__ void zero() { hi = lo = 0ull; }
    __device__ __forceinline__ void mac(int i, const AbVec<F2, 2> &w, const AbVec<F2, 2> &c)
    {
        const uint64_t an = pk_mul(w.v.x, pk_dup(-1.f));
        if (i == 0) pk_f2_mul(bh, bl, w.v.x, an, w.v.y, c.v);
        else pk_f2_mac(bh, bl, w.v.x, an, w.v.y, c.v);
    }
    __device__ __forceinline__ void end_block() { pk_f2_add(hi, lo, bh, bl); }
    __device__ __forceinline__ void add_lane(int off)
    {
        const uint64_t oh = __shfl_xor_sync(0xffffffffu, hi, off), ol = __shfl_xor_sync(0xffffffffu, lo, off);
        pk_f2_add(hi, lo, oh, ol);
    }
    __device__ __forceinline__ double value() const
    {
        // (the halves added as pairs: an FP64 instruction takes 64 clocks, however few of its lanes work)
        return f2_value(f2_add(F2(pk_get(hi, 0), pk_get(lo, 0)), F2(pk_get(hi, 1), pk_get(lo, 1))));
    }
};

// Two-operand alpha-beta pass: CTA per output row ia.  The alpha singles of ia are taken R at a
// time: their rows C[ja,:] are staged interleaved, W[2*pair + neg][k] = +-u_k (p_k q_k|rs) is
// tabulated, and every lane walks the beta singles of one output column ib (slices of 32 columns
// with lists of nearly equal length, so that the lanes of a warp stay busy: on the FP64 pipe an idle
// lane costs as much as a busy one): acc += sum_k W[rs][k] C[ja_k, jb], added to s(ia, ib) with a
// fire-and-forget reduction.  Warps take the slices from a counter, longest lists first (dealt out in
// a fixed pattern, the warp with the longest list held up the barrier of every group).  A column is
// added to once per group, and the groups are separated by a barrier, so its adds land in order.
//
// Bound by the FP64 pipe (FP64) or by the two 16-byte gathers per entry (pairs: L1/shared pipe 84 %,
// 43 % of the wavefronts are bank conflicts left by the ordering of the entries).  Measured
// against eight lanes per column (each column's list padded to 32 slots), 3.6e7 determinants, norb 29:
// FP64 84.1 -> 34 ms, pairs 33.1 -> 19.1 ms; with the slices dealt out in a fixed pattern 36.6 and
// 21.4 ms.
// Pairs: where the longest slice is 3 (8) times a warp's share of all steps or more, it holds up the
// barrier, and two (four) lanes walk a list: 2,000 rows x 150 columns at norb 24 839 -> 569 us, x 700
// columns 1,663 -> 1,430; with equal lists (full space, 495 strings) one lane 397 us, two 451.  FP64 is bound by
// its pipe even then (one lane 727 us, eight 1,686 at 300 columns).
// Where a row of C does not fit shared memory its elements come from L2, and the bounds of the next slice are
// loaded during this one (200 x 60,000 strings, norb 58: FP64 209 -> 111 ms, pairs 96 -> 76; for staged
// FP64 the registers this takes cost a resident CTA: 61 -> 71 ms at 60,000 x 300, norb 40).
template <typename T, int R, bool STAGED>
__device__ __forceinline__ void ab_row(const AbArgs<T> &a, int64_t ia, unsigned char *smem)
{
    constexpr int kThreads = Threads<T>::value, kWarps = kThreads / 32;
    constexpr bool kAhead = !STAGED || kIsF2<T>;  // a slice's bounds loaded during the one before
    const int n2 = a.norb * a.norb, nkey = a.norb * (a.norb - 1);
    // column nB is zero (padding entries); it takes from the room that choose() leaves behind the nkey + 1
    // coefficient rows (2 norb^2 - nkey - 1 more rows of R elements, at least 5 where there is a single)
    const size_t cs_bytes = STAGED ? round16((size_t)(a.nB + 1) * R * sizeof(T)) : 0;
    T *Cs = reinterpret_cast<T *>(smem);
    T *Ws = reinterpret_cast<T *>(smem + cs_bytes);  // [nkey + 1][R]
    __shared__ int next_s;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t e0 = a.as_ptr[ia], nsl = (a.nB + 31) / 32;
    const int K = (int)(a.as_ptr[ia + 1] - e0);
    const unsigned longest = a.sl_off[1], steps = a.sl_off[nsl];  // of one slice, of all
    for (int k0 = 0; k0 < K; k0 += R) {
        const int kr = min(R, K - k0);
        int64_t ja[R];
        int pq[R];
        double u[R];
#pragma unroll
        for (int k = 0; k < R; ++k) {
            const bool ok = k < kr;
            const uint32_t pk = ok ? a.as_pk[e0 + k0 + k] : 0u;
            ja[k] = pk_j(pk);
            pq[k] = pk_code(pk);
            if (std::is_same<T, float>::value) pq[k] = ok ? orbital_pair(pq[k] / a.norb, pq[k] % a.norb) : 0;
            u[k] = ok ? (pk_neg(pk) ? -1.0 : 1.0) : 0.0;
        }
        __syncthreads();
        if (tid == 0) next_s = kWarps;
        if (STAGED) {
            for (int64_t c = tid; c <= a.nB; c += kThreads) {
                T v[R];
#pragma unroll
                for (int k = 0; k < R; ++k) v[k] = k < kr && c < a.nB ? conv<T>(a.C[ja[k] * a.nB + c]) : T(0);
                AbVec<T, R>::st(Cs + c * R, v);
            }
        }
        for (int key = tid; key <= nkey; key += kThreads) {
            const int pair = key >> 1;
            int r = (int)((1.f + sqrtf(8.f * (float)pair + 1.f)) * 0.5f);
            if (r * (r - 1) / 2 > pair) --r;
            if (r * (r + 1) / 2 <= pair) ++r;
            const int rs = r * a.norb + (pair - r * (r - 1) / 2);
            const double sg = (key & 1) ? -1.0 : 1.0;
            T v[R];
#pragma unroll
            for (int k = 0; k < R; ++k) {
                const size_t at = std::is_same<T, float>::value ? (size_t)pq[k] * (nkey / 2) + pair : (size_t)pq[k] * n2 + rs;
                v[k] = key < nkey ? conv<T>((typename In<T>::type)(sg * u[k]) * __ldg(a.eri + at)) : T(0);
            }
            AbVec<T, R>::st(Ws + (size_t)key * R, v);
        }
        __syncthreads();
        // STEP lanes walk a column's list side by side, a warp 32 / STEP columns of a slice
        const auto walk = [&](auto step) {
            constexpr int STEP = decltype(step)::value;
            const int64_t units = nsl * STEP;
            const int sub = lane & (STEP - 1);
            const auto unit_of = [&](int64_t un, int &len, int &col, const uint32_t *&ent) {
                const int64_t sl = un / STEP;
                const int l = (int)(un % STEP) * (32 / STEP) + lane / STEP;
                const uint32_t o0 = a.sl_off[sl];
                len = (int)(a.sl_off[sl + 1] - o0);
                col = a.sl_col[sl * 32 + l];
                ent = a.sl_ent + (size_t)o0 * 32 + l;
            };
            int64_t un = warp;
            int len = 0, col = -1;
            const uint32_t *ent = nullptr;
            if (kAhead && un < units) unit_of(un, len, col, ent);
            while (un < units) {
                if (!kAhead) unit_of(un, len, col, ent);
                if (len == 0) break;  // the lists descend: nothing follows
                int next = 0;
                if (lane == 0) next = atomicAdd(&next_s, 1);
                next = __shfl_sync(0xffffffffu, next, 0);
                int len_n = 0, col_n = -1;
                const uint32_t *ent_n = nullptr;
                if (kAhead && next < units) unit_of(next, len_n, col_n, ent_n);
                AbSum<T, R> acc;
                acc.zero();
                uint32_t nx[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) nx[i] = sub + STEP * i < len ? __ldg(ent + 32 * (sub + STEP * i)) : 0u;
                for (int t = sub; t < len; t += 4 * STEP) {
                    uint32_t e[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) e[i] = nx[i];
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        nx[i] = t + STEP * (4 + i) < len ? __ldg(ent + 32 * (t + STEP * (4 + i))) : 0u;
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (t + STEP * i < len) {
                            AbVec<T, R> c, w;
                            const int jb = pk_j(e[i]);
                            if constexpr (STAGED) c.ld(Cs + (size_t)jb * R);
                            else c.v[0] = jb < a.nB ? conv<T>(a.C[ja[0] * a.nB + jb]) : T(0);
                            w.ld(Ws + (size_t)(e[i] >> kPackKeyShift) * R);
                            acc.mac(i, w, c);
                        }
                    acc.end_block();
                }
                if constexpr (STEP > 1) {
                    __syncwarp();
#pragma unroll
                    for (int off = STEP / 2; off > 0; off >>= 1) acc.add_lane(off);
                }
                if (sub == 0 && col >= 0) atomicAdd(a.S + ia * a.nB + col, acc.value());
                un = next;
                if (kAhead) len = len_n, col = col_n, ent = ent_n;
            }
        };
        if constexpr (STAGED && kIsF2<T>) {
            if (longest * kWarps >= 8 * steps) walk(std::integral_constant<int, 4>());
            else if (longest * kWarps >= 3 * steps) walk(std::integral_constant<int, 2>());
            else walk(std::integral_constant<int, 1>());
        } else {
            walk(std::integral_constant<int, 1>());
        }
    }
}

template <typename T, int R, bool STAGED>
__global__ void __launch_bounds__(Threads<T>::value) ab_pass_kernel(const AbArgs<T> a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    for (int64_t ia = blockIdx.x; ia < a.nA; ia += gridDim.x) ab_row<T, R, STAGED>(a, ia, smem);
}

// ---------------------------------------------------------------------------
// Column-stationary alpha-beta pass of the mixed sigma.
//
// For output row ia with alpha singles (ja_k, pq_k, u_k), k < K, and the beta singles of each
// string (ib <- jb with orbital pair {r, s}, phase t; by Hermiticity the singles list of jb names
// every ib that has jb among its singles, with the same phase):
//   s(ia, ib) += sum_{jb} sum_{ib in singles(jb)} t * sum_k W[{r,s}][k] C(ja_k, jb),
//   W[{r,s}][k] = u_k (p_k q_k|rs)                       ((pq|rs) = (pq|sr) for real orbitals)
// The alpha singles are taken in chunks of KC <= 32.  A lane owns one column jb: it holds the KC
// amplitudes C(ja_k, jb) in registers and walks the singles of jb; for each it gathers one
// 4*KC-byte row of W from shared memory (the only shared-memory operand of the multiply-adds,
// 4 bytes per FMA) and adds the FP32 dot product to the row accumulator of ib.
//
// Bank conflicts: a W row is 128 bytes (eight 16-byte chunks).  With KC = 32 lane l reads chunk
// (step + l) mod 8 at each step, so the 8 lanes of a 128-bit phase hit 8 distinct bank groups
// whatever rows they read; with KC = 16 (8) each row holds 2 (4) copies and lanes read their own
// copy, rotated within it.  The lane's registers hold the amplitudes in the same order.
// Where the rows of all pairs do not fit beside the row accumulator (norb 58: 1,653 pairs, 211 KB), the
// pairs are cut into parts: the table holds one part's rows at a time and the beta singles come part by
// part, so a column's amplitudes are loaded once per part.  (Rows of 64 bytes for chunks of at most 16
// alpha singles, the layout before, had two lanes of a phase in the same bank group half of the time
// and added to the accumulator twice as often: norb 58, 5,000 strings,
// 11.4 -> 8.5 ms; 15,000 strings 164 -> 109 ms.)
//
// Determinism: each FP32 dot product is rounded once onto a fixed-point grid with one scale 2^e per
// output row and added as an integer, and integer addition is exact and order independent, so the
// result does not depend on the order of the shared-memory atomics.  An element of the row receives
// at most m = maxdeg_beta * (chunks of the row) contributions v.  Each v is split as
// v = hi * 2^L + lo with 0 <= lo < 2^L, L = 32 - bitlength(m), and lo and hi are added with 32-bit
// integer atomics into two words per element (random 32-bit shared-memory atomics run several times
// faster than 64-bit ones): the lo word cannot overflow (m * 2^L < 2^32), and e is chosen so that
// the largest possible row sum of |v|,
//   maxdeg_beta * max|(pq|rs)| * sum_k max_jb |C(ja_k, jb)|  (times 2^e),
// stays below 2^(30+L), which keeps the sum of the hi words inside a signed 32-bit word.  The grid
// step is then about 2^-(30+L) >= 2^-52 of that bound, far below FP32 rounding of the products.
// The element is hi_sum * 2^L + lo_sum exactly; the row is added to s(ia, :) in FP64 by the CTA
// that owns the row.

constexpr int kSrcThreads = 1024;  // packed dot products (896: 18.4 ms, 1,024: 18.1 at 1.0e8 determinants)
template <bool PACKED>
constexpr int kSrcThreadsOf = PACKED ? kSrcThreads : 896;  // one chain: more registers a thread

struct AbSrcArgs {
    const float *C;  // [nA][nB] FP32 amplitudes
    double *S;       // [nA][nB], accumulated
    int64_t nA, nB;
    int norb, npair;
    const float *eri;         // FP32 (pq|rs) as [npair][npair]
    const int64_t *as_ptr;    // alpha singles, canonical CSR
    const uint32_t *as_pk;
    const uint32_t *src_item; // beta singles, source-major items (string | entries << 18)
    const uint32_t *src_ent;
    int parts, width;         // parts of the orbital pairs, pairs of a part
    int slice[kSrcParts + 1]; // slices of 32 items of each part
    const float *rowmax;      // [nA] max |C(ja, :)|
    float bound;              // maxdeg_beta * max |(pq|rs)|
    int maxdeg;               // maxdeg_beta: most singles of a beta string
    const int32_t *row_order; // rows by descending number of alpha singles, -1 where there is none; may be null
};

// shared memory of one CTA: W [width][8] float4, accumulator [nB] u64
__host__ __device__ constexpr size_t src_w_bytes(int width) { return (size_t)width * 128; }
__host__ __device__ inline size_t src_smem(int width, int64_t nB) { return src_w_bytes(width) + (size_t)nB * 8; }
// the fewest parts whose table fits `limit` bytes, 0 if kSrcParts do not
inline int src_parts_for(int npair, int64_t nB, size_t limit)
{
    for (int h = 1; h <= kSrcParts; ++h)
        if (src_smem((npair + h - 1) / h, nB) <= limit) return h;
    return 0;
}

// adds t * f to element ib of the row accumulator (words lo[ib], hi[ib]; see above).  scale_hi =
// scale 2^-L and two_l = 2^L: |f| scale_hi is cut into its whole part (hi) and the rest, scaled back
// and rounded to an integer (lo); both steps are exact in FP32 but for that one rounding, so the value
// is the nearest grid point, as a conversion of f scale to a 64-bit integer gives (which runs on the
// FP64 pipe: 37 % of its cycles).
__device__ __forceinline__ void src_add(unsigned *acc_lo, unsigned *acc_hi, uint32_t e, float f, float scale_hi,
                                        float two_l, int lbits)
{
    const float x = fabsf(f) * scale_hi;
    unsigned hi = __float2uint_rz(x);
    unsigned lo = __float2uint_rn((x - __uint2float_rz(hi)) * two_l);
    const unsigned neg = ((__float_as_uint(f) >> 31) ^ (e >> kSrcNegBit)) & 1u;
    if (neg) {  // -(hi 2^L + lo) with the low word in [0, 2^L]
        const unsigned some = lo != 0u ? 1u : 0u;
        hi = 0u - hi - some;
        lo = (some << lbits) - lo;
    }
    const int ib = (int)(e & kPackJMask);
    atomicAdd(acc_lo + ib, lo);
    atomicAdd(acc_hi + ib, hi);
}

// PACKED: two multiply-adds per instruction (even and odd alpha singles in two sums), chunk step xor
// lane instead of (step + lane) mod CPW.  The engine keeps the one chain per dot product that its jobs
// have always summed in: the result of a job stopped by its iteration cap depends on the rounding of
// its products to 1e-9 of the energy.
template <int KC, bool PACKED>
__device__ __forceinline__ void src_chunk(const AbSrcArgs &a, const float4 *__restrict__ Wt, unsigned *acc_lo,
                                          unsigned *acc_hi, const int *ja_s, int kc, float scale_hi, float two_l,
                                          int lbits, int sl1, int *ctr)
{
    constexpr int RS = 8;  // 16-byte chunks of a W row
    constexpr int CPW = KC / 4;  // 16-byte chunks per copy of a W row
    const int lane = threadIdx.x & 31;
    const int rot = lane & (CPW - 1);
    const int base = ((lane / CPW) & (RS / CPW - 1)) * CPW;  // first chunk of this lane's copy
    const uint32_t first = (uint32_t)(base + rot) * 16u;
    const unsigned char *Wb = reinterpret_cast<const unsigned char *>(Wt);
    while (true) {
        int sl = 0;
        if (lane == 0) sl = atomicAdd(ctr, 1);
        sl = __shfl_sync(0xffffffffu, sl, 0);
        if (sl >= sl1) break;
        // one item per lane: a string jb (column of C) and at most kSrcItem of its singles
        const int64_t t = (int64_t)sl * 32 + lane;
        const uint32_t info = __ldg(a.src_item + t);
        const int64_t jb = info & kPackJMask;
        const int cnt = (int)(info >> kSrcPairShift);
        const uint32_t *ent = a.src_ent + (int64_t)sl * 32 * kSrcItem + lane;
        if constexpr (PACKED) {
            // amplitudes of the chunk's alpha singles at column jb (consecutive lanes: consecutive or equal
            // columns), two to a word, then permuted so that register chunk s holds amplitude chunk s xor rot
            uint64_t cv[KC / 2];
#pragma unroll
            for (int k4 = 0; k4 < KC; k4 += 4) {
                const int4 j4 = *reinterpret_cast<const int4 *>(ja_s + k4);  // one broadcast load per 4 rows
                const int jr[4] = {j4.x, j4.y, j4.z, j4.w};
                float v[4];
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    v[i] = (cnt > 0 && k4 + i < kc) ? __ldg(a.C + (int64_t)jr[i] * a.nB + jb) : 0.f;
                cv[k4 / 2] = pk_pair(v[0], v[1]);
                cv[k4 / 2 + 1] = pk_pair(v[2], v[3]);
            }
#pragma unroll
            for (int b = 1; b < CPW; b <<= 1) {
                const bool swap = rot & b;
#pragma unroll
                for (int s = 0; s < CPW; ++s)
                    if (!(s & b)) {
#pragma unroll
                        for (int i = 0; i < 2; ++i) {
                            const uint64_t x = cv[2 * s + i], y = cv[2 * (s ^ b) + i];
                            cv[2 * s + i] = swap ? y : x;
                            cv[2 * (s ^ b) + i] = swap ? x : y;
                        }
                    }
            }
            uint32_t n0 = cnt > 0 ? __ldg(ent) : 0u, n1 = cnt > 1 ? __ldg(ent + 32) : 0u;
#pragma unroll
            for (int i = 0; i < kSrcItem; i += 2) {  // two singles per round for independent chains
                const uint32_t e0 = n0, e1 = n1;
                ent += 64;
                n0 = i + 2 < cnt ? __ldg(ent) : 0u;
                n1 = i + 3 < cnt ? __ldg(ent + 32) : 0u;
                if (i < cnt) {
                    const bool two = i + 1 < cnt;
                    const uint32_t o0 = ((e0 >> kSrcPairShift) & 0x7ffu) * (RS * 16u) + first;
                    const uint32_t o1 = ((e1 >> kSrcPairShift) & 0x7ffu) * (RS * 16u) + first;
                    uint64_t f0 = 0ull, f1 = 0ull;
#pragma unroll
                    for (int s = 0; s < CPW; ++s) {  // chunk s xor rot of the row: 8 lanes, 8 bank groups
                        const ulonglong2 x0 = *reinterpret_cast<const ulonglong2 *>(Wb + (o0 ^ (s * 16u)));
                        // where there is no second single, entry 0 reads the table's first row: unused
                        const ulonglong2 x1 = *reinterpret_cast<const ulonglong2 *>(Wb + (o1 ^ (s * 16u)));
                        f0 = pk_fma(x0.x, cv[2 * s], f0);
                        f1 = pk_fma(x1.x, cv[2 * s], f1);
                        f0 = pk_fma(x0.y, cv[2 * s + 1], f0);
                        f1 = pk_fma(x1.y, cv[2 * s + 1], f1);
                    }
                    src_add(acc_lo, acc_hi, e0, pk_get(f0, 0) + pk_get(f0, 1), scale_hi, two_l, lbits);
                    if (two) src_add(acc_lo, acc_hi, e1, pk_get(f1, 0) + pk_get(f1, 1), scale_hi, two_l, lbits);
                }
            }
        } else {
            uint32_t e[kSrcItem];
#pragma unroll
            for (int i = 0; i < kSrcItem; ++i) e[i] = i < cnt ? __ldg(ent + 32 * i) : 0u;
            // amplitudes of the chunk's alpha singles at column jb (consecutive lanes: consecutive or equal
            // columns), then rotated by `rot` chunks so that register chunk s holds amplitude chunk
            // (s + rot) mod CPW
            float cv[KC];
#pragma unroll
            for (int k4 = 0; k4 < KC; k4 += 4) {
                const int4 j4 = *reinterpret_cast<const int4 *>(ja_s + k4);  // one broadcast load per 4 rows
                const int jr[4] = {j4.x, j4.y, j4.z, j4.w};
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    cv[k4 + i] = (cnt > 0 && k4 + i < kc) ? __ldg(a.C + (int64_t)jr[i] * a.nB + jb) : 0.f;
            }
#pragma unroll
            for (int b = 1; b < CPW; b <<= 1) {
                if (rot & b) {
                    float tmp[KC];
#pragma unroll
                    for (int s = 0; s < CPW; ++s)
#pragma unroll
                        for (int i = 0; i < 4; ++i) tmp[4 * s + i] = cv[4 * ((s + b) % CPW) + i];
#pragma unroll
                    for (int k = 0; k < KC; ++k) cv[k] = tmp[k];
                }
            }
#pragma unroll
            for (int i = 0; i < kSrcItem; i += 2) {  // two singles per round for independent chains
                if (i < cnt) {
                    const bool two = i + 1 < cnt;
                    const float4 *w0 = Wt + ((e[i] >> kSrcPairShift) & 0x7ffu) * RS + base;
                    const float4 *w1 = Wt + ((e[i + 1] >> kSrcPairShift) & 0x7ffu) * RS + base;
                    float f0 = 0.f, f1 = 0.f;
#pragma unroll
                    for (int s = 0; s < CPW; ++s) {
                        const int q = (s + rot) & (CPW - 1);
                        const float4 x0 = w0[q];
                        const float4 x1 = w1[q];  // where there is no second single: the first row, unused
                        f0 = fmaf(x0.x, cv[4 * s], f0);
                        f1 = fmaf(x1.x, cv[4 * s], f1);
                        f0 = fmaf(x0.y, cv[4 * s + 1], f0);
                        f1 = fmaf(x1.y, cv[4 * s + 1], f1);
                        f0 = fmaf(x0.z, cv[4 * s + 2], f0);
                        f1 = fmaf(x1.z, cv[4 * s + 2], f1);
                        f0 = fmaf(x0.w, cv[4 * s + 3], f0);
                        f1 = fmaf(x1.w, cv[4 * s + 3], f1);
                    }
                    src_add(acc_lo, acc_hi, e[i], f0, scale_hi, two_l, lbits);
                    if (two) src_add(acc_lo, acc_hi, e[i + 1], f1, scale_hi, two_l, lbits);
                }
            }
        }
    }
}

// W[x][position p] for the chunk's alpha singles, position p holding amplitude chunk p mod CPW
template <int KC>
__device__ __forceinline__ void src_build_w(const AbSrcArgs &a, float4 *Wt, int p0, int width, const int *pq_s,
                                            const float *u_s, int kc)
{
    constexpr int CPW = KC / 4, RS = 8;
    const int p = threadIdx.x % RS, c = p & (CPW - 1);  // RS divides the block size
    float u[4];
    const float *row[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int k = 4 * c + i;
        u[i] = k < kc ? u_s[k] : 0.f;
        row[i] = a.eri + (size_t)(k < kc ? pq_s[k] : 0) * a.npair + p0;
    }
#pragma unroll 4
    for (int x = threadIdx.x / RS; x < width; x += blockDim.x / RS)
        Wt[(size_t)x * RS + p] = make_float4(u[0] * __ldg(row[0] + x), u[1] * __ldg(row[1] + x),
                                             u[2] * __ldg(row[2] + x), u[3] * __ldg(row[3] + x));
}

template <bool PACKED>
__device__ __forceinline__ void src_row(const AbSrcArgs &a, int64_t ia, unsigned char *smem)
{
    constexpr int KMAX = 32;  // alpha singles per chunk
    float4 *Wt = reinterpret_cast<float4 *>(smem);
    unsigned *acc_lo = reinterpret_cast<unsigned *>(smem + src_w_bytes(a.width));
    unsigned *acc_hi = acc_lo + a.nB;
    __shared__ __align__(16) int ja_s[32];
    __shared__ int pq_s[32];
    __shared__ float u_s[32];
    __shared__ int ctr;
    __shared__ float s_scale;
    __shared__ double s_inv;
    __shared__ int s_lbits;
    __shared__ int s_state;  // 0 skip the row, 1 accumulate, 2 non-finite amplitudes
    const int tid = threadIdx.x;
    const int64_t e0 = a.as_ptr[ia];
    const int K = (int)(a.as_ptr[ia + 1] - e0);
    __syncthreads();  // the previous row is finished with shared memory
    for (int64_t ib = tid; ib < a.nB; ib += blockDim.x) acc_lo[ib] = acc_hi[ib] = 0u;
    if (tid < 32) {
        float m = 0.f;
        for (int k = tid; k < K; k += 32) m += __ldg(a.rowmax + (a.as_pk[e0 + k] & kPackJMask));
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) m += __shfl_xor_sync(0xffffffffu, m, off);
        if (tid == 0) {
            const double bnd = (double)m * (double)a.bound;
            if (!(bnd <= 1e300)) {
                s_state = 2;
            } else if (bnd == 0.0) {
                s_state = 0;
            } else {
                // contributions per element: at most maxdeg per chunk of the row
                const long long m = (long long)max(a.maxdeg, 1) * ((K + KMAX - 1) / KMAX);
                const int lbits = max(1, 32 - (64 - __clzll(m)));
                int e = 30 + lbits - ilogb(bnd) - 1;  // bnd < 2^(ilogb+1), so bnd * 2^e < 2^(30+lbits)
                e = max(-120, min(120, e));
                s_scale = ldexpf(1.f, e - lbits);
                s_inv = ldexp(1.0, -e);
                s_lbits = lbits;
                s_state = 1;
            }
        }
    }
    __syncthreads();
    const int state = s_state;
    if (state == 0) return;
    if (state == 2) {
        for (int64_t ib = tid; ib < a.nB; ib += blockDim.x) a.S[ia * a.nB + ib] = __longlong_as_double(0x7ff8000000000000ll);
        return;
    }
    const int lbits = s_lbits;
    const float two_l = __uint_as_float((unsigned)(127 + lbits) << 23), scale_hi = s_scale;
    for (int k0 = 0; k0 < K; k0 += KMAX) {
        const int kc = min(KMAX, K - k0);
        __syncthreads();  // the previous chunk is finished with W and the chunk arrays
        if (tid < kc) {
            const uint32_t pk = a.as_pk[e0 + k0 + tid];
            ja_s[tid] = (int)(pk & kPackJMask);
            const int code = (int)(pk >> (kPackKeyShift + 1));
            pq_s[tid] = orbital_pair(code / a.norb, code % a.norb);
            u_s[tid] = ((pk >> kPackKeyShift) & 1u) ? -1.f : 1.f;
        }
        for (int h = 0; h < a.parts; ++h) {
            const int p0 = h * a.width, width = min(a.width, a.npair - p0);
            if (h) __syncthreads();  // the previous part is finished with W
            if (tid == 0) ctr = a.slice[h];
            __syncthreads();
            if (kc <= 8) src_build_w<8>(a, Wt, p0, width, pq_s, u_s, kc);
            else if (kc <= 16) src_build_w<16>(a, Wt, p0, width, pq_s, u_s, kc);
            else src_build_w<32>(a, Wt, p0, width, pq_s, u_s, kc);
            __syncthreads();
            const int sl1 = a.slice[h + 1];
            if (kc <= 8) src_chunk<8, PACKED>(a, Wt, acc_lo, acc_hi, ja_s, kc, scale_hi, two_l, lbits, sl1, &ctr);
            else if (kc <= 16) src_chunk<16, PACKED>(a, Wt, acc_lo, acc_hi, ja_s, kc, scale_hi, two_l, lbits, sl1, &ctr);
            else src_chunk<32, PACKED>(a, Wt, acc_lo, acc_hi, ja_s, kc, scale_hi, two_l, lbits, sl1, &ctr);
        }
    }
    __syncthreads();
    const double inv = s_inv;
    double *s = a.S + ia * a.nB;
    for (int64_t b = tid; b < a.nB; b += 4 * (int64_t)blockDim.x) {  // four loads of sigma in flight
        double y[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) y[u] = b + u * blockDim.x < a.nB ? s[b + u * blockDim.x] : 0.0;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int64_t ib = b + u * blockDim.x;
            if (ib < a.nB) {
                const long long v = (long long)(int)acc_hi[ib] * (1ll << lbits) + (long long)acc_lo[ib];
                s[ib] = y[u] + (double)v * inv;
            }
        }
    }
}

__global__ void __launch_bounds__(kSrcThreads, 1) ab_src_kernel(const AbSrcArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    // A row costs as much as it has alpha singles (none to several times the mean).  The rows are dealt
    // out in descending order, back and forth over the CTAs, which evens out their sums; in ascending
    // order of the strings the last CTA ended a tenth later than the mean.
    for (int64_t i = 0; i * gridDim.x < a.nA; ++i) {
        const int64_t x = i * gridDim.x + ((i & 1) ? gridDim.x - 1 - blockIdx.x : blockIdx.x);
        const int64_t ia = x >= a.nA ? -1 : a.row_order ? a.row_order[x] : x;
        if (ia >= 0) src_row<true>(a, ia, smem);
    }
}

// out[c][r] = in[r][c]; with rowmax (FP32 only, zeroed beforehand): rowmax[r] = max_c |in[r][c]|,
// accumulated as the bit patterns of non-negative floats (a NaN row stays NaN)
template <typename T>
__global__ void transpose_kernel(const T *__restrict__ in, T *__restrict__ out, int64_t rows, int64_t cols,
                                 float *rowmax = nullptr)
{
    __shared__ T tile[32][33];
    const int64_t bx = (int64_t)blockIdx.x * 32, by = (int64_t)blockIdx.y * 32;
    for (int j = threadIdx.y; j < 32; j += 8) {
        const int64_t r = by + j, c = bx + threadIdx.x;
        T v = T(0);
        if (r < rows && c < cols) {
            v = in[r * cols + c];
            tile[j][threadIdx.x] = v;
        }
        if constexpr (sizeof(T) == 4) {
            if (rowmax) {  // uniform per launch
                const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(fabsf((float)v)));
                if (threadIdx.x == 0 && r < rows) atomicMax(reinterpret_cast<unsigned *>(rowmax) + r, m);
            }
        }
    }
    __syncthreads();
    for (int j = threadIdx.y; j < 32; j += 8) {
        const int64_t c = bx + j, r = by + threadIdx.x;
        if (r < rows && c < cols) out[c * rows + r] = tile[threadIdx.x][j];
    }
}

// One 32 x 32 tile of sigma[r][c] (+)= st[c][r] + hd[r][c] x[r][c]: the beta pass' transposed result
// and the diagonal term (x: the FP64 amplitudes where the caller has them).  The FP64-accurate products add it
// last (ADD): the diagonal term is the largest, and every sum that comes after it is rounded at its size.
template <typename E, bool ADD>
__device__ __forceinline__ void untranspose_tile(double (&tile)[32][33], const double *__restrict__ st,
                                                 const double *__restrict__ hd, const E *__restrict__ x,
                                                 const double *__restrict__ x64, double *__restrict__ sigma,
                                                 int64_t rows, int64_t cols, int64_t by, int64_t bx)
{
    for (int j = threadIdx.y; j < 32; j += 8) {
        const int64_t c = bx + j, r = by + threadIdx.x;
        if (r < rows && c < cols) tile[j][threadIdx.x] = st[c * rows + r];
    }
    __syncthreads();
    for (int j = threadIdx.y; j < 32; j += 8) {
        const int64_t r = by + j, c = bx + threadIdx.x;
        if (r < rows && c < cols) {
            const int64_t i = r * cols + c;
            const double v = fma(hd[i], x64 ? x64[i] : (double)x[i], tile[threadIdx.x][j]);
            sigma[i] = ADD ? sigma[i] + v : v;
        }
    }
}

template <typename E, bool ADD>
__global__ void untranspose_kernel(const double *__restrict__ st, const double *__restrict__ hd,
                                   const E *__restrict__ x, const double *__restrict__ x64, double *__restrict__ sigma,
                                   int64_t rows, int64_t cols)
{
    __shared__ double tile[32][33];
    untranspose_tile<E, ADD>(tile, st, hd, x, x64, sigma, rows, cols, (int64_t)blockIdx.y * 32, (int64_t)blockIdx.x * 32);
}

struct PassCfg {
    int R = 1;
    bool staged = false;
    size_t smem = 0;
};

PassCfg choose(int64_t ncol, int n2, size_t elem, int rmax, size_t limit)
{
    PassCfg p;
    for (int R = rmax; R >= 1; R /= 2) {
        size_t b = round16((size_t)ncol * R * elem) + (size_t)2 * n2 * R * elem;
        if (b <= limit) {
            p.R = R;
            p.staged = true;
            p.smem = b;
            return p;
        }
    }
    p.R = 1;
    p.staged = false;
    p.smem = (size_t)2 * n2 * elem;
    return p;
}

size_t smem_limit(const Ctx &c) { return (size_t)c.smem_optin - 1024; }

// max |FP32 of x| over n values, as the bit pattern of a non-negative float (out zeroed beforehand)
__global__ void absmax_kernel(const double *__restrict__ x, int64_t n, unsigned *out)
{
    unsigned m = 0u;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        m = max(m, __float_as_uint(fabsf((float)x[i])));
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) atomicMax(out, m);
}

int npairs(int norb) { return norb * (norb - 1) / 2; }

// the column-stationary alpha-beta pass applies when a part of its W table and the row accumulator fit
bool src_fits(const Ctx &c) { return c.norb >= 2 && c.sp[1].src_parts > 0; }

AbSrcArgs src_args(const Ctx &c, const float *C, double *S, const float *rowmax)
{
    const SpinTables &ta = c.sp[0], &tb = c.sp[1];
    AbSrcArgs a{};
    a.C = C;
    a.S = S;
    a.nA = c.nA;
    a.nB = c.nB;
    a.norb = c.norb;
    a.npair = npairs(c.norb);
    a.eri = c.eri32;
    a.as_ptr = ta.s_ptr;
    a.as_pk = ta.s_pk;
    a.src_item = tb.src_item;
    a.src_ent = tb.src_ent;
    a.parts = tb.src_parts;
    a.width = tb.src_width;
    std::copy(tb.src_slice, tb.src_slice + kSrcParts + 1, a.slice);
    a.rowmax = rowmax;
    a.bound = (float)((double)tb.src_maxdeg * (double)c.eri_absmax);
    a.maxdeg = tb.src_maxdeg;
    a.row_order = ta.sl_col;
    return a;
}

// CTAs that share an SM: two of half the threads where both fit and have a few rows each.  Between its
// rows and chunks a CTA tabulates W and adds its sums to sigma while its gathers idle, and the other's
// rows fill that (one product at norb 20, 1,703 x 2,381 strings: one CTA 1.52 ms, two 1.46, four 1.56;
// norb 24, 300 strings: one 88 us, two 92 us).
int src_ctas(size_t smem, int sm_bytes, int64_t rows, int num_sms)
{
    return 2 * (smem + 2048) <= (size_t)sm_bytes && rows >= 4 * (int64_t)num_sms ? 2 : 1;
}

void launch_ab_src(const AbSrcArgs &a, const Ctx &c, cudaStream_t s)
{
    const size_t smem = src_smem(a.width, a.nB);
    const int f = src_ctas(smem, c.smem_optin, a.nA, c.num_sms);
    const int grid = (int)std::min<int64_t>(a.nA, (int64_t)c.num_sms * f);
    ab_src_kernel<<<grid, kSrcThreads / f, smem, s>>>(a);
    SBD_LAUNCH("ab_src_kernel");
}

template <typename T>
void set_attrs(int optin)
{
    SBD_CUDA(cudaFuncSetAttribute(range_rows_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin));
    SBD_CUDA(cudaFuncSetAttribute(range_small_kernel<T, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin));
    SBD_CUDA(cudaFuncSetAttribute(range_small_kernel<T, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin));
    if constexpr (sizeof(T) == 4) {
        SBD_CUDA(cudaFuncSetAttribute(row_pass_kernel<T, 4, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin));
        SBD_CUDA(cudaFuncSetAttribute(ab_pass_kernel<T, 4, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin));
    }
    SBD_CUDA(cudaFuncSetAttribute(row_pass_kernel<T, 2, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin));
    SBD_CUDA(cudaFuncSetAttribute(row_pass_kernel<T, 1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin));
    SBD_CUDA(cudaFuncSetAttribute(row_pass_kernel<T, 1, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin));
    SBD_CUDA(cudaFuncSetAttribute(ab_pass_kernel<T, 2, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin));
    SBD_CUDA(cudaFuncSetAttribute(ab_pass_kernel<T, 1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin));
    SBD_CUDA(cudaFuncSetAttribute(ab_pass_kernel<T, 1, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin));
}

// Lists of few strings: range_small (at most six groups to a part, so that half of a CTA's warps would idle).
// Products of n x n strings without and with it, pairs, norb 24: n = 300 211 -> 183 us, 800 811 -> 768,
// 1,200 1,835 -> 1,882.
constexpr int kSmallStrings = 768;
bool small_range(int64_t n, int ng) { return ng == 1 && n <= kSmallStrings; }

template <typename T>
void launch_direct(const Ctx &c, const RangeArgs<T> &a, const double *x64, cudaStream_t s)
{
    const int64_t units = (a.nrow + kRangeRows<T> - 1) / kRangeRows<T> * kParts;
    const int grid = (int)std::min<int64_t>(units, c.num_sms);
    range_small_kernel<T, true><<<grid, kRangeThreads, range_smem(c.smem_optin), s>>>(a, c.hd, x64, units);
    SBD_LAUNCH("range_small_kernel");
}

template <typename T>
void launch_range(const Ctx &c, const RangeArgs<T> &a, cudaStream_t s)
{
    const int64_t units = (a.nrow + kRangeRows<T> - 1) / kRangeRows<T> * kParts;
    const int grid = (int)std::min<int64_t>(units, c.num_sms);
    if (small_range(a.n, a.ng)) {
        range_small_kernel<T, false><<<grid, kRangeThreads, range_smem(c.smem_optin), s>>>(a, nullptr, nullptr, units);
        SBD_LAUNCH("range_small_kernel");
        return;
    }
    range_rows_kernel<T><<<grid, kRangeThreads, range_smem(c.smem_optin), s>>>(a, units);
    SBD_LAUNCH("range_rows_kernel");
}

template <typename T>
void launch_row(const RowArgs<T> &a, const PassCfg &p, cudaStream_t s)
{
    constexpr int kThreads = Threads<T>::value;
    const int64_t groups = (a.nrow + p.R - 1) / p.R;
    const int grid = (int)(groups < 65535 ? groups : 65535);
    if (!p.staged) row_pass_kernel<T, 1, false><<<grid, kThreads, p.smem, s>>>(a);
    else if (p.R == 4) row_pass_kernel<T, (sizeof(T) == 4 ? 4 : 2), true><<<grid, kThreads, p.smem, s>>>(a);
    else if (p.R == 2) row_pass_kernel<T, 2, true><<<grid, kThreads, p.smem, s>>>(a);
    else row_pass_kernel<T, 1, true><<<grid, kThreads, p.smem, s>>>(a);
    SBD_LAUNCH("row_pass_kernel");
}

template <typename T>
void launch_ab(const AbArgs<T> &a, const PassCfg &p, cudaStream_t s)
{
    constexpr int kThreads = Threads<T>::value;
    const int grid = (int)(a.nA < 65535 ? a.nA : 65535);
    if (!p.staged) ab_pass_kernel<T, 1, false><<<grid, kThreads, p.smem, s>>>(a);
    else if (p.R == 4) ab_pass_kernel<T, (sizeof(T) == 4 ? 4 : 2), true><<<grid, kThreads, p.smem, s>>>(a);
    else if (p.R == 2) ab_pass_kernel<T, 2, true><<<grid, kThreads, p.smem, s>>>(a);
    else ab_pass_kernel<T, 1, true><<<grid, kThreads, p.smem, s>>>(a);
    SBD_LAUNCH("ab_pass_kernel");
}

template <typename T>
void transpose(const T *in, T *out, int64_t rows, int64_t cols, cudaStream_t s, float *rowmax = nullptr)
{
    const int64_t gy = (rows + 31) / 32;
    if (gy > 65535) fail(SBD_ERR_UNSUPPORTED, "alpha string set too large for the transpose");
    dim3 grid((unsigned)((cols + 31) / 32), (unsigned)gy);
    if (rowmax) SBD_CUDA(cudaMemsetAsync(rowmax, 0, (size_t)rows * sizeof(float), s));
    transpose_kernel<T><<<grid, dim3(32, 8), 0, s>>>(in, out, rows, cols, rowmax);
    SBD_LAUNCH("transpose_kernel");
}

template <typename T>
Lists<T> lists_of(const SigLists &l)
{
    if constexpr (std::is_same<T, double>::value) return Lists<double>{l.s_pk, l.s_v, nullptr, l.d_j, l.d_v, nullptr};
    else return Lists<T>{l.s_pk, l.s_hi, l.s_lo, l.d_j, l.d_hi, l.d_lo};
}

// timing slot of the first sigma kernel of a precision (transpose, beta, alpha, alpha-beta follow)
template <typename T>
constexpr int kSlotBase = kIsF2<T> ? 8 : (sizeof(T) == 4 ? 4 : 0);
template <typename T>
constexpr int kRowsMax = sizeof(T) == 4 ? 4 : 2;

// Runs launch(); when timing is on, brackets it with events on stream s and
// queues the pair for sbd_kernel_times (slot: kernel kind, +4 for FP32).
template <typename F>
void timed(Ctx &c, int slot, cudaStream_t s, F &&launch)
{
    if (!c.opt.timing) {
        launch();
        return;
    }
    cudaEvent_t a = take_event(c), b = take_event(c);
    SBD_CUDA(cudaEventRecord(a, s));
    launch();
    SBD_CUDA(cudaEventRecord(b, s));
    c.pending.push_back({slot, a, b});
}

// Arguments of the two-operand alpha-beta pass.
template <typename T>
void make_ab_args(const Ctx &c, const typename In<T>::type *C, double *S, AbArgs<T> &ab)
{
    const SpinTables &ta = c.sp[0], &tb = c.sp[1];
    ab = AbArgs<T>{};
    ab.C = C;
    ab.S = S;
    ab.nA = c.nA;
    ab.nB = c.nB;
    ab.norb = c.norb;
    using E = typename In<T>::type;
    ab.eri = sizeof(E) == 4 ? (const E *)(const void *)c.eri32 : (const E *)(const void *)c.eri64;
    ab.as_ptr = ta.s_ptr;      // canonical alpha lists: exact counts for the row groups
    ab.as_pk = ta.s_pk;
    ab.sl_col = tb.sl_col;
    ab.sl_off = tb.sl_off;
    ab.sl_ent = tb.sl_ent;
}

// Arguments of the engine's mixed row passes: beta pass on C, alpha pass on its transpose Ct.
void make_row_args(const Ctx &c, const float *C, double *S, const double *c64, const float *Ct, RowArgs<float> &rb,
                   RowArgs<float> &ra)
{
    const SpinTables &ta = c.sp[0], &tb = c.sp[1];
    auto lists = [](RowArgs<float> &r, const SpinTables &t) {
        r.s_ptr = t.sig.s_ptr;
        r.d_ptr = t.sig.d_ptr;
        r.lists = lists_of<float>(t.sig);
        r.hls_ptr = t.hs_ptr;
        r.hld_ptr = t.hd_ptr;
        r.hls = t.hs;
        r.hldv = t.hdv;
        r.hldt = t.hdt;
        r.half = t.half;
    };
    rb = RowArgs<float>{};
    rb.norb = c.norb;
    rb.eri = c.eri64;
    ra = rb;
    rb.X = C;
    rb.nrow = c.nA;
    rb.ncol = rb.ncol_out = c.nB;
    rb.Y = S;
    rb.y_rs = c.nB;
    rb.y_cs = 1;
    rb.hd = c.hd;
    rb.xd64 = c64;
    rb.row_strings = ta.strings;
    lists(rb, tb);
    ra.X = Ct;
    ra.nrow = c.nB;
    ra.ncol = ra.ncol_out = c.nA;
    ra.Y = S;
    ra.y_rs = 1;
    ra.y_cs = c.nB;
    ra.accumulate = 1;
    ra.row_strings = tb.strings;
    lists(ra, ta);
}

template <typename T>
const typename RangeVal<T>::type *range_vals(const float *hi, const double *v64)
{
    if constexpr (std::is_same<T, double>::value) return v64;
    else return hi;
}

// Row pass over the lists of spin `ls` of a handle: X and Y have that spin's strings as rows of
// the other spin's length.
template <typename T>
RangeArgs<T> range_args(const Ctx &c, int ls, const typename In<T>::type *X, double *Y, int accumulate)
{
    const SpinTables &t = c.sp[ls], &o = c.sp[1 - ls];
    const RangeLists &r = t.rl;
    RangeArgs<T> a{};
    a.X = X;
    a.Y = Y;
    a.n = t.n;
    a.nrow = o.n;
    a.accumulate = accumulate;
    a.npair = r.np;
    a.jstaged = range_j_staged(c.smem_optin, c.norb);
    a.w = r.w;
    a.ng = r.ng;
    a.q = 1;
    a.jg = r.jg;
    a.zi = r.zi;
    a.qd = r.qd;
    a.qs = r.qs;
    a.dt = r.dt;
    a.sm = r.sm;
    a.dv = range_vals<T>(r.dhi, r.dv64);
    a.sv = range_vals<T>(r.shi, r.sv64);
    a.dlo = r.dlo;
    a.slo = r.slo;
    return a;
}

// Whether the beta pass takes the rows of C as they are (range_small, DIRECT).  Mixed products, norb 12: 100 x 100
// strings 45 -> 36 us without the transposes, 495 x 200 87 -> 78, 495 x 495 the same; pairs 303 -> 298, 503 -> 509.
bool direct_beta(const Ctx &c) { return small_range(c.nB, c.sp[1].rl.ng) && c.N <= (int64_t)1 << 17; }

// The transposed copy of C is kept in the output buffer until the beta pass has read it, and the
// beta pass' transposed result in the handle's work vector, so the row passes need no memory of
// their own.
template <typename T>
void apply(Ctx &c, const typename In<T>::type *C, double *S, const double *c64, cudaStream_t s)
{
    using E = typename In<T>::type;
    const int n2 = c.norb * c.norb;
    const size_t lim = smem_limit(c);
    const int base = kSlotBase<T>;
    E *Ct = reinterpret_cast<E *>(S);
    double *St = static_cast<double *>(c.work_t);
    constexpr bool kLast = !std::is_same<T, float>::value;  // beta part and diagonal added last (untranspose_tile)
    const bool direct = direct_beta(c);
    RangeArgs<T> rb = range_args<T>(c, 1, direct ? C : Ct, direct ? S : St, direct && kLast);
    RangeArgs<T> ra = range_args<T>(c, 0, C, S, !kLast);
    // the mixed alpha-beta pass takes the row maxima of C from the beta pass
    const bool src = !kLast && src_fits(c);
    if (src) rb.rowmax = c.rowmax;
    const auto back = [&] {
        if (direct) {
            launch_direct<T>(c, rb, c64, s);
            return;
        }
        const dim3 grid((unsigned)((c.nB + 31) / 32), (unsigned)((c.nA + 31) / 32));
        untranspose_kernel<E, kLast><<<grid, dim3(32, 8), 0, s>>>(St, c.hd, C, c64, S, c.nA, c.nB);
        SBD_LAUNCH("untranspose_kernel");
    };
    if (!direct) timed(c, base + 0, s, [&] { transpose<E>(C, Ct, c.nA, c.nB, s); });
    if (!direct || !kLast) {
        timed(c, base + 1, s, [&] {
            if (!direct) launch_range<T>(c, rb, s);
            if (!kLast) back();
        });
    }
    timed(c, base + 2, s, [&] { launch_range<T>(c, ra, s); });
    timed(c, base + 3, s, [&] {
        if constexpr (!kLast) {
            if (src) {
                launch_ab_src(src_args(c, C, S, c.rowmax), c, s);
                return;
            }
        }
        AbArgs<T> ab;
        make_ab_args<T>(c, C, S, ab);
        launch_ab<T>(ab, choose(c.nB, n2, sizeof(T), kRowsMax<T>, lim), s);
        if (kLast && !direct) back();
    });
    if (kLast && direct) timed(c, base + 1, s, back);
}

// ---------------------------------------------------------------------------
// Batched sigma.  One descriptor block holds, for every slot, the arguments of its passes and
// the prefix sums of its work items (transpose tiles, beta row groups, alpha row groups, alpha-beta
// rows).  Persistent CTAs take items from a counter and run the same per-item device functions as
// the single-instance kernels, so every output element is computed by the same arithmetic.

template <typename T>
struct TDesc {
    const T *x;         // amplitudes [rows][cols]
    const double *x64;  // FP64 amplitudes for the diagonal term, or null
    double *y;          // sigma; holds the transposed amplitudes until the beta pass has read them
    double *st;         // the beta pass' transposed result
    const double *hd;
    int64_t rows, cols;
};

struct Layout {
    size_t n, off_t, off_b, off_a, off_ab, td, rb, ra, ab, src, total;
};

template <typename T>
Layout layout_for(int m)
{
    Layout L{};
    size_t o = 0;
    auto take = [&](size_t bytes) {
        const size_t at = o;
        o = (o + bytes + 255) & ~(size_t)255;
        return at;
    };
    L.n = take(sizeof(int));
    L.off_t = take(sizeof(int64_t) * (m + 1));
    L.off_b = take(sizeof(int64_t) * (m + 1));
    L.off_a = take(sizeof(int64_t) * (m + 1));
    L.off_ab = take(sizeof(int64_t) * (m + 1));
    L.td = take(sizeof(TDesc<typename In<T>::type>) * m);
    L.rb = take(std::max(sizeof(RangeArgs<T>), sizeof(RowArgs<T>)) * m);
    L.ra = take(std::max(sizeof(RangeArgs<T>), sizeof(RowArgs<T>)) * m);
    L.ab = take(sizeof(AbArgs<T>) * m);
    L.src = take(sizeof(AbSrcArgs) * m);
    L.total = o;
    return L;
}

// slot s with off[s] <= item < off[s + 1] (empty slots are skipped)
__device__ __forceinline__ int find_slot(const int64_t *off, int n, int64_t item)
{
    int lo = 0, hi = n;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (off[mid] <= item) lo = mid;
        else hi = mid;
    }
    return lo;
}

// BACK 0: the transposed amplitudes of every slot; 1: sigma = the beta pass' result transposed back
// plus the diagonal term (FP64-accurate products: added to sigma)
template <typename T, bool BACK>
__global__ void transpose_batch_kernel(const int *pn, const int64_t *off, const TDesc<T> *td)
{
    __shared__ double tile[32][33];
    const int n = *pn;
    const int64_t total = off[n];
    for (int64_t it = blockIdx.x; it < total; it += gridDim.x) {
        const int sl = find_slot(off, n, it);
        const TDesc<T> d = td[sl];
        const int64_t lt = it - off[sl], tx = (d.cols + 31) / 32;
        const int64_t by = (lt / tx) * 32, bx = (lt % tx) * 32;
        __syncthreads();
        if constexpr (BACK) {
            untranspose_tile<T, sizeof(T) == 8>(tile, d.st, d.hd, d.x, d.x64, d.y, d.rows, d.cols, by, bx);
        } else {
            T *out = reinterpret_cast<T *>(d.y);
            for (int j = threadIdx.y; j < 32; j += 8) {
                const int64_t r = by + j, c = bx + threadIdx.x;
                if (r < d.rows && c < d.cols) tile[j][threadIdx.x] = (double)d.x[r * d.cols + c];
            }
            __syncthreads();
            for (int j = threadIdx.y; j < 32; j += 8) {
                const int64_t c = bx + j, r = by + threadIdx.x;
                if (r < d.rows && c < d.cols) out[c * d.rows + r] = (T)tile[threadIdx.x][j];
            }
        }
    }
}

// Work-item loop of the persistent pass kernels: thread 0 takes the next item from the counter,
// the CTA copies the slot's arguments to shared memory when the slot changes, then runs body().
template <typename Args, typename F>
__device__ __forceinline__ void item_loop(const int *pn, const int64_t *off, const Args *args,
                                          unsigned long long *counter, Args &sa, F &&body)
{
    __shared__ int64_t s_item;
    __shared__ int s_slot;
    const int n = *pn;
    const int64_t total = off[n];
    int cur = -1;
    while (true) {
        __syncthreads();  // the previous item is finished with shared memory
        if (threadIdx.x == 0) {
            const int64_t it = (int64_t)atomicAdd(counter, 1ull);
            s_item = it;
            s_slot = it < total ? find_slot(off, n, it) : -1;
        }
        __syncthreads();
        const int64_t it = s_item;
        const int sl = s_slot;
        if (it >= total) break;
        if (sl != cur) {
            const uint32_t *src = reinterpret_cast<const uint32_t *>(args + sl);
            uint32_t *dst = reinterpret_cast<uint32_t *>(&sa);
            for (int i = threadIdx.x; i < (int)(sizeof(Args) / 4); i += blockDim.x) dst[i] = src[i];
            cur = sl;
            __syncthreads();
        }
        body(it - off[sl]);
    }
}

// The engine's mixed row passes: whole rows of C staged, R at a time (8: one column half at a time)
template <typename T, int R>
__global__ void __launch_bounds__(Threads<T>::value) row_batch_kernel(const int *pn, const int64_t *off,
                                                                      const RowArgs<T> *args,
                                                                      unsigned long long *counter)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ RowArgs<T> sa;
    item_loop(pn, off, args, counter, sa, [&](int64_t li) { row_group<T, R, true>(sa, li * R, smem); });
}

__global__ void __launch_bounds__(Threads<float>::value) row_halves_batch_kernel(const int *pn, const int64_t *off,
                                                                               const RowArgs<float> *args,
                                                                               unsigned long long *counter)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ RowArgs<float> sa;
    item_loop(pn, off, args, counter, sa, [&](int64_t li) { row_halves(sa, li * kHalfRows, smem); });
}

template <typename T>
__global__ void __launch_bounds__(kRangeThreads, 1) range_batch_kernel(const int *pn, const int64_t *off,
                                                                      const RangeArgs<T> *args,
                                                                      unsigned long long *counter)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ RangeArgs<T> sa;
    item_loop(pn, off, args, counter, sa, [&](int64_t li) {
        const int per = kParts / sa.q, p0 = (int)(li % sa.q) * per;
        range_rows<T>(sa, li / sa.q * kRangeRows<T>, p0, p0 + per, smem);
    });
}

template <typename T, int R>
__global__ void __launch_bounds__(Threads<T>::value) ab_batch_kernel(const int *pn, const int64_t *off,
                                                                     const AbArgs<T> *args,
                                                                     unsigned long long *counter)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ AbArgs<T> sa;
    item_loop(pn, off, args, counter, sa, [&](int64_t li) { ab_row<T, R, true>(sa, li, smem); });
}

template <bool PACKED>
__global__ void __launch_bounds__(kSrcThreadsOf<PACKED>, 1) ab_src_batch_kernel(const int *pn, const int64_t *off,
                                                                      const AbSrcArgs *args,
                                                                      unsigned long long *counter)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ AbSrcArgs sa;
    item_loop(pn, off, args, counter, sa, [&](int64_t li) { src_row<PACKED>(sa, li, smem); });
}

size_t batch_smem(size_t elem, int R, int max_strings, int max_norb)
{
    if (R == kHalfRows) return halves_smem((max_strings + 1) / 2, max_norb);
    return round16((size_t)max_strings * R * elem) + (size_t)2 * max_norb * max_norb * R * elem;
}

}  // namespace

struct SigmaBatch {
    sbd_precision prec = SBD_MIXED;
    int max_slots = 0, R = 1, device = 0, grid_range = 0, grid_ab = 0, grid_t = 0, grid_src = 0;
    size_t smem = 0, range_smem = 0;  // alpha-beta pass, row passes
    bool rows = false;    // the row passes over whole staged rows (engine, mixed)
    int grid_rows = 0;
    bool src = false;     // mixed: the column-stationary alpha-beta pass (when its table and accumulator fit)
    size_t src_smem = 0;
    int src_threads = 0;
    Layout L{};
    unsigned char *dev = nullptr, *host = nullptr;
    unsigned long long *counters = nullptr;  // [3]: beta, alpha, alpha-beta
};

namespace {

template <typename T>
void batch_set(SigmaBatch *b, const SigmaSlot *slots, int n)
{
    const Layout &L = b->L;
    unsigned char *h = b->host;
    *reinterpret_cast<int *>(h + L.n) = n;
    int64_t *ot = reinterpret_cast<int64_t *>(h + L.off_t), *ob = reinterpret_cast<int64_t *>(h + L.off_b);
    int64_t *oa = reinterpret_cast<int64_t *>(h + L.off_a), *oab = reinterpret_cast<int64_t *>(h + L.off_ab);
    using E = typename In<T>::type;
    TDesc<E> *td = reinterpret_cast<TDesc<E> *>(h + L.td);
    RangeArgs<T> *rb = reinterpret_cast<RangeArgs<T> *>(h + L.rb), *ra = reinterpret_cast<RangeArgs<T> *>(h + L.ra);
    AbArgs<T> *ab = reinterpret_cast<AbArgs<T> *>(h + L.ab);
    ot[0] = ob[0] = oa[0] = oab[0] = 0;
    // row blocks are cut into q pieces, enough for about eight work items per CTA
    int64_t blocks = 0;
    for (int i = 0; i < n; ++i) blocks += (std::min(slots[i].c->nA, slots[i].c->nB) + kRangeRows<T> - 1) / kRangeRows<T>;
    int q = 1;
    while (q < kParts && blocks * q < (int64_t)8 * b->grid_range) q *= 2;
    for (int i = 0; i < n; ++i) {
        const SigmaSlot &sl = slots[i];
        const Ctx &c = *sl.c;
        const E *x = static_cast<const E *>(sl.x);
        double *st = static_cast<double *>(sl.xt);
        make_ab_args<T>(c, x, sl.y, ab[i]);
        td[i] = TDesc<E>{x, sl.x64, sl.y, st, c.hd, c.nA, c.nB};
        ob[i + 1] = ob[i] + (c.nA + kRangeRows<T> - 1) / kRangeRows<T> * q;
        oa[i + 1] = oa[i] + (c.nB + kRangeRows<T> - 1) / kRangeRows<T> * q;
        float *rowmax = nullptr;
        if constexpr (std::is_same<T, float>::value) rowmax = b->src ? c.rowmax : nullptr;
        if (std::is_same<T, float>::value && b->rows) {
            RowArgs<float> *wb = reinterpret_cast<RowArgs<float> *>(h + L.rb), *wa = reinterpret_cast<RowArgs<float> *>(h + L.ra);
            make_row_args(c, static_cast<const float *>(sl.x), sl.y, sl.x64, static_cast<const float *>(sl.xt), wb[i], wa[i]);
            wb[i].rowmax = rowmax;
            td[i].y = st;  // the transposed amplitudes stay in the work vector
            ob[i + 1] = ob[i] + (c.nA + b->R - 1) / b->R;
            oa[i + 1] = oa[i] + (c.nB + b->R - 1) / b->R;
        } else {
            rb[i] = range_args<T>(c, 1, reinterpret_cast<const E *>(sl.y), st, 0);
            ra[i] = range_args<T>(c, 0, x, sl.y, std::is_same<T, float>::value);
            rb[i].q = ra[i].q = q;
            rb[i].rowmax = rowmax;
        }
        if constexpr (std::is_same<T, float>::value) {
            if (b->src) reinterpret_cast<AbSrcArgs *>(h + L.src)[i] = src_args(c, x, sl.y, c.rowmax);
        }
        ot[i + 1] = ot[i] + ((c.nA + 31) / 32) * ((c.nB + 31) / 32);
        oab[i + 1] = oab[i] + c.nA;
    }
}

template <typename T, int R>
void batch_launch_r(SigmaBatch *b, cudaStream_t s)
{
    const Layout &L = b->L;
    unsigned char *d = b->dev;
    const int *pn = reinterpret_cast<const int *>(d + L.n);
    using E = typename In<T>::type;
    const int64_t *off_t = reinterpret_cast<const int64_t *>(d + L.off_t);
    const TDesc<E> *td = reinterpret_cast<const TDesc<E> *>(d + L.td);
    transpose_batch_kernel<E, false><<<b->grid_t, dim3(32, 8), 0, s>>>(pn, off_t, td);
    SBD_LAUNCH("transpose_batch_kernel");
    const int64_t *off_b = reinterpret_cast<const int64_t *>(d + L.off_b), *off_a = reinterpret_cast<const int64_t *>(d + L.off_a);
    if (std::is_same<T, float>::value && b->rows) {
        if constexpr (std::is_same<T, float>::value) {
            const RowArgs<float> *wb = reinterpret_cast<const RowArgs<float> *>(d + L.rb);
            const RowArgs<float> *wa = reinterpret_cast<const RowArgs<float> *>(d + L.ra);
            constexpr int kThreads = Threads<float>::value;
            if constexpr (R == kHalfRows) {
                row_halves_batch_kernel<<<b->grid_rows, kThreads, b->smem, s>>>(pn, off_b, wb, b->counters);
                SBD_LAUNCH("row_halves_batch_kernel");
                row_halves_batch_kernel<<<b->grid_rows, kThreads, b->smem, s>>>(pn, off_a, wa, b->counters + 1);
                SBD_LAUNCH("row_halves_batch_kernel");
            } else {
                row_batch_kernel<float, R><<<b->grid_rows, kThreads, b->smem, s>>>(pn, off_b, wb, b->counters);
                SBD_LAUNCH("row_batch_kernel");
                row_batch_kernel<float, R><<<b->grid_rows, kThreads, b->smem, s>>>(pn, off_a, wa, b->counters + 1);
                SBD_LAUNCH("row_batch_kernel");
            }
        }
    } else {
        range_batch_kernel<T><<<b->grid_range, kRangeThreads, b->range_smem, s>>>(
            pn, off_b, reinterpret_cast<const RangeArgs<T> *>(d + L.rb), b->counters);
        SBD_LAUNCH("range_batch_kernel");
        if (std::is_same<T, float>::value) {  // the other precisions add it last
            transpose_batch_kernel<E, true><<<b->grid_t, dim3(32, 8), 0, s>>>(pn, off_t, td);
            SBD_LAUNCH("transpose_batch_kernel");
        }
        range_batch_kernel<T><<<b->grid_range, kRangeThreads, b->range_smem, s>>>(
            pn, off_a, reinterpret_cast<const RangeArgs<T> *>(d + L.ra), b->counters + 1);
        SBD_LAUNCH("range_batch_kernel");
    }
    if (std::is_same<T, float>::value && b->src) {
        const int64_t *off_ab = reinterpret_cast<const int64_t *>(d + L.off_ab);
        const AbSrcArgs *src_args_d = reinterpret_cast<const AbSrcArgs *>(d + L.src);
        if (b->rows)
            ab_src_batch_kernel<false><<<b->grid_src, b->src_threads, b->src_smem, s>>>(pn, off_ab, src_args_d, b->counters + 2);
        else
            ab_src_batch_kernel<true><<<b->grid_src, b->src_threads, b->src_smem, s>>>(pn, off_ab, src_args_d, b->counters + 2);
        SBD_LAUNCH("ab_src_batch_kernel");
        return;
    }
    if constexpr (R != kHalfRows) {  // 8 rows per item only come with the column-stationary pass
        ab_batch_kernel<T, R><<<b->grid_ab, Threads<T>::value, b->smem, s>>>(
            pn, reinterpret_cast<const int64_t *>(d + L.off_ab), reinterpret_cast<const AbArgs<T> *>(d + L.ab),
            b->counters + 2);
        SBD_LAUNCH("ab_batch_kernel");
    }
    if (!std::is_same<T, float>::value) {
        transpose_batch_kernel<E, true><<<b->grid_t, dim3(32, 8), 0, s>>>(pn, off_t, td);
        SBD_LAUNCH("transpose_batch_kernel");
    }
}

template <typename T, int R>
void batch_attrs(SigmaBatch *b)
{
    int sms = 0;
    SBD_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, b->device));
    SBD_CUDA(cudaFuncSetAttribute(range_batch_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)b->range_smem));
    b->grid_range = sms;
    if constexpr (std::is_same<T, float>::value) {
        if (b->rows) {
            int occ = 0;
            if constexpr (R == kHalfRows) {
                SBD_CUDA(cudaFuncSetAttribute(row_halves_batch_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)b->smem));
                SBD_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, row_halves_batch_kernel, Threads<T>::value,
                                                                       b->smem));
            } else {
                SBD_CUDA(cudaFuncSetAttribute(row_batch_kernel<T, R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)b->smem));
                SBD_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, row_batch_kernel<T, R>, Threads<T>::value,
                                                                       b->smem));
            }
            b->grid_rows = sms * std::max(1, occ);
        }
    }
    if constexpr (R != kHalfRows) {
        int occ_ab = 0;
        SBD_CUDA(cudaFuncSetAttribute(ab_batch_kernel<T, R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)b->smem));
        SBD_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ_ab, ab_batch_kernel<T, R>, Threads<T>::value,
                                                               b->smem));
        b->grid_ab = sms * std::max(1, occ_ab);
    }
    b->grid_t = sms * 8;
    if (b->src) {
        int occ_src = 0, optin = 0;
        SBD_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, b->device));
        b->src_threads = (b->rows ? kSrcThreadsOf<false> : kSrcThreads) / src_ctas(b->src_smem, optin, INT64_MAX, sms);
        auto *kernel = b->rows ? ab_src_batch_kernel<false> : ab_src_batch_kernel<true>;
        SBD_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)b->src_smem));
        SBD_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ_src, kernel, b->src_threads, b->src_smem));
        b->grid_src = sms * std::max(1, occ_src);
    }
}

}  // namespace

int src_parts(int norb, int64_t n, int smem_optin)
{
    return norb >= 2 ? src_parts_for(npairs(norb), n, (size_t)smem_optin - 1024) : 0;
}

void sigma_prepare(Ctx &c)
{
    // dynamic shared memory up to smem_limit(): the kernels' static shared memory (at most 1 KB) and
    // the dynamic part must stay within the opt-in maximum together
    const int lim = (int)smem_limit(c);
    set_attrs<double>(lim);
    set_attrs<float>(lim);
    set_attrs<F2>(lim);
    SBD_CUDA(cudaFuncSetAttribute(ab_src_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, lim));
    // max |(pq|rs)| of the FP32 integrals, for the fixed-point scale of the alpha-beta pass
    const int64_t n4 = (int64_t)c.norb * c.norb * c.norb * c.norb;
    unsigned *m = reinterpret_cast<unsigned *>(c.dstat);  // status words are free after create
    SBD_CUDA(cudaMemsetAsync(m, 0, sizeof(unsigned), c.stream));
    absmax_kernel<<<(int)std::min<int64_t>((n4 + 255) / 256, 1024), 256, 0, c.stream>>>(c.eri64, n4, m);
    SBD_LAUNCH("absmax_kernel");
    unsigned bits = 0;
    SBD_CUDA(cudaMemcpyAsync(&bits, m, sizeof(unsigned), cudaMemcpyDeviceToHost, c.stream));
    SBD_CUDA(cudaStreamSynchronize(c.stream));
    memcpy(&c.eri_absmax, &bits, sizeof(float));
    c.rowmax = dalloc_n<float>(c, (size_t)c.nA);
}

size_t sigma_batch_smem(sbd_precision prec, int R, int max_strings, int max_norb)
{
    return batch_smem(prec == SBD_MIXED ? 4 : 8, R, max_strings, max_norb);
}

bool sigma_batch_fits(sbd_precision prec, int R, int max_strings, int max_norb, int device)
{
    const size_t lim = sigma_batch_smem_limit(device);
    if (R == kHalfRows)
        return prec == SBD_MIXED && max_norb >= 2 && sigma_batch_smem(prec, R, max_strings, max_norb) <= lim &&
               src_parts_for(npairs(max_norb), max_strings, lim) > 0;
    if (R == 4 && prec != SBD_MIXED) return false;
    return sigma_batch_smem(prec, R, max_strings, max_norb) <= lim;
}

size_t sigma_batch_smem_limit(int device)
{
    int optin = 0;
    SBD_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device));
    return (size_t)optin - 1024;  // headroom for the kernels' static shared memory
}

SigmaBatch *sigma_batch_create(int max_slots, sbd_precision prec, int R, int max_strings, int max_norb, int device,
                               bool rows)
{
    if (max_slots < 1) fail(SBD_ERR_INVALID_ARG, "batched sigma needs at least one slot");
    if (!(R == 1 || R == 2 || ((R == 4 || R == kHalfRows) && prec == SBD_MIXED)) || prec < SBD_FP64 ||
        prec > SBD_F32X2)
        fail(SBD_ERR_INVALID_ARG, "rows per work item must be 1, 2 or (mixed only) 4 or 8");
    const size_t smem = sigma_batch_smem(prec, R, max_strings, max_norb);
    if (smem > sigma_batch_smem_limit(device))
        fail(SBD_ERR_UNSUPPORTED, "batched sigma: staged rows do not fit in shared memory");
    auto *b = new SigmaBatch();
    b->prec = prec;
    b->max_slots = max_slots;
    b->R = R;
    b->rows = rows && prec == SBD_MIXED;
    b->device = device;
    b->smem = smem;
    int optin = 0;
    if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device) != cudaSuccess) {
        delete b;
        fail(SBD_ERR_CUDA, "batched sigma: the device does not report its shared memory");
    }
    b->range_smem = range_smem(optin);
    const size_t lim = sigma_batch_smem_limit(device);
    const int mp = npairs(max_norb), h = max_norb >= 2 ? src_parts_for(mp, max_strings, lim) : 0;
    // one part for the largest instance is one part for all; else a smaller one may take up to the limit
    b->src_smem = h == 1 ? src_smem(mp, max_strings) : lim;
    b->src = prec == SBD_MIXED && h > 0;
    if (R == kHalfRows && !b->src) {
        delete b;
        fail(SBD_ERR_UNSUPPORTED, "batched sigma: 8 rows per item need the column-stationary alpha-beta pass, "
                                  "whose table and accumulator do not fit shared memory here");
    }
    b->L = prec == SBD_FP64 ? layout_for<double>(max_slots)
                            : (prec == SBD_F32X2 ? layout_for<F2>(max_slots) : layout_for<float>(max_slots));
    try {
        SBD_CUDA(cudaMalloc(&b->dev, b->L.total));
        SBD_CUDA(cudaMallocHost(&b->host, b->L.total));
        SBD_CUDA(cudaMalloc(&b->counters, 3 * sizeof(unsigned long long)));
        memset(b->host, 0, b->L.total);
        if (prec == SBD_FP64) {
            if (R == 2) batch_attrs<double, 2>(b);
            else batch_attrs<double, 1>(b);
        } else if (prec == SBD_F32X2) {
            if (R == 2) batch_attrs<F2, 2>(b);
            else batch_attrs<F2, 1>(b);
        } else {
            if (R == kHalfRows) batch_attrs<float, kHalfRows>(b);
            else if (R == 4) batch_attrs<float, 4>(b);
            else if (R == 2) batch_attrs<float, 2>(b);
            else batch_attrs<float, 1>(b);
        }
    } catch (...) {
        sigma_batch_destroy(b);
        throw;
    }
    return b;
}

void sigma_batch_set(SigmaBatch *b, const SigmaSlot *slots, int n)
{
    if (n < 0 || n > b->max_slots) fail(SBD_ERR_INVALID_ARG, "batched sigma: too many slots");
    for (int i = 0; i < n; ++i) {
        const Ctx &c = *slots[i].c;
        if (sigma_batch_smem(b->prec, b->R, (int)std::max(c.nA, c.nB), c.norb) > b->smem)
            fail(SBD_ERR_UNSUPPORTED, "batched sigma: an instance exceeds the string or orbital limit of the batch");
    }
    if (b->prec == SBD_FP64) batch_set<double>(b, slots, n);
    else if (b->prec == SBD_F32X2) batch_set<F2>(b, slots, n);
    else batch_set<float>(b, slots, n);
}

void sigma_batch_launch(SigmaBatch *b, cudaStream_t s)
{
    SBD_CUDA(cudaMemcpyAsync(b->dev, b->host, b->L.total, cudaMemcpyHostToDevice, s));
    SBD_CUDA(cudaMemsetAsync(b->counters, 0, 3 * sizeof(unsigned long long), s));
    if (b->prec == SBD_FP64) {
        if (b->R == 2) batch_launch_r<double, 2>(b, s);
        else batch_launch_r<double, 1>(b, s);
    } else if (b->prec == SBD_F32X2) {
        if (b->R == 2) batch_launch_r<F2, 2>(b, s);
        else batch_launch_r<F2, 1>(b, s);
    } else {
        if (b->R == kHalfRows) batch_launch_r<float, kHalfRows>(b, s);
        else if (b->R == 4) batch_launch_r<float, 4>(b, s);
        else if (b->R == 2) batch_launch_r<float, 2>(b, s);
        else batch_launch_r<float, 1>(b, s);
    }
}

void sigma_batch_destroy(SigmaBatch *b)
{
    if (!b) return;
    if (b->dev) (void)cudaFree(b->dev);
    if (b->host) (void)cudaFreeHost(b->host);
    if (b->counters) (void)cudaFree(b->counters);
    delete b;
}

namespace {

// The three passes of one source block for the output rows of a plan (see BlockPlan).
template <typename T>
void apply_block(BlockPlan &p, const typename In<T>::type *Cb, double *S, cudaStream_t s, const double *x64)
{
    using E = typename In<T>::type;
    Ctx &c = *p.c;
    const int n2 = c.norb * c.norb;
    const int rmax = kRowsMax<T>;
    const size_t lim = smem_limit(c);
    const int64_t nj = p.j1 - p.j0, nr = p.r1 - p.r0;
    const SpinTables &ta = c.sp[0], &tb = c.sp[1];
    E *Ct = static_cast<E *>(p.work_t);
    // mixed: the column-stationary alpha-beta pass takes the source rows' maxima from the transpose
    const bool src = std::is_same<T, float>::value && src_fits(c);
    transpose<E>(Cb, Ct, nj, c.nB, s, src ? p.rowmax : nullptr);
    // beta pass: the output rows inside the block
    const int64_t lo = std::max(p.r0, p.j0), hi = std::min(p.r1, p.j1);
    RowArgs<T> row{};
    row.norb = c.norb;
    row.eri = c.eri64;
    row.accumulate = 1;
    if (lo < hi) {
        RowArgs<T> b = row;
        b.X = Cb + (lo - p.j0) * c.nB;
        b.nrow = hi - lo;
        b.ncol = b.ncol_out = c.nB;
        b.Y = S + (lo - p.r0) * c.nB;
        b.y_rs = c.nB;
        b.y_cs = 1;
        b.hd = c.hd + lo * c.nB;
        b.xd64 = x64 ? x64 + (lo - p.r0) * c.nB : nullptr;
        b.row_strings = ta.strings + lo;
        b.s_ptr = tb.sig.s_ptr;
        b.d_ptr = tb.sig.d_ptr;
        b.lists = lists_of<T>(tb.sig);
        launch_row<T>(b, choose(c.nB, n2, sizeof(T), rmax, lim), s);
    }
    // alpha pass: rows of the transposed block, output columns r0..r1, lists restricted to the block
    RowArgs<T> ra = row;
    ra.X = Ct;
    ra.nrow = c.nB;
    ra.ncol = nj;
    ra.ncol_out = nr;
    ra.Y = S;
    ra.y_rs = 1;
    ra.y_cs = c.nB;
    ra.row_strings = tb.strings;
    ra.s_ptr = p.sig.s_ptr;
    ra.d_ptr = p.sig.d_ptr;
    ra.lists = lists_of<T>(p.sig);
    launch_row<T>(ra, choose(nj, n2, sizeof(T), rmax, lim), s);
    // alpha-beta pass: output rows r0..r1, their alpha singles inside the block
    if constexpr (std::is_same<T, float>::value) {
        if (src) {
            AbSrcArgs a = src_args(c, Cb, S, p.rowmax);
            a.nA = nr;
            a.as_ptr = p.s_ptr;
            a.as_pk = p.s_pk;
            a.row_order = nullptr;
            launch_ab_src(a, c, s);
            return;
        }
    }
    AbArgs<T> ab;
    make_ab_args<T>(c, Cb, S, ab);
    ab.nA = nr;
    ab.as_ptr = p.s_ptr;
    ab.as_pk = p.s_pk;
    launch_ab<T>(ab, choose(c.nB, n2, sizeof(T), rmax, lim), s);
}

}  // namespace

void sigma_block_apply(BlockPlan &p, const void *cblock, double *sigma_rows, sbd_precision prec, cudaStream_t s,
                       const double *x64_rows)
{
    if (value_mask(prec) & ~p.sig.mask) fail(SBD_ERR_INVALID_ARG, "block plan: not made for this precision");
    if (prec == SBD_FP64) apply_block<double>(p, static_cast<const double *>(cblock), sigma_rows, s, nullptr);
    else if (prec == SBD_F32X2) apply_block<F2>(p, static_cast<const double *>(cblock), sigma_rows, s, nullptr);
    else apply_block<float>(p, static_cast<const float *>(cblock), sigma_rows, s, x64_rows);
}

void sigma_apply(Ctx &c, const void *cvec, double *svec, sbd_precision prec, cudaStream_t s, const double *c64)
{
    if (prec == SBD_FP64) apply<double>(c, static_cast<const double *>(cvec), svec, nullptr, s);
    else if (prec == SBD_F32X2) apply<F2>(c, static_cast<const double *>(cvec), svec, nullptr, s);
    else apply<float>(c, static_cast<const float *>(cvec), svec, c64, s);
}

}  // namespace sbd

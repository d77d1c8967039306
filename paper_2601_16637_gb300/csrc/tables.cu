// Excitation tables, same-spin string matrix elements and the Hamiltonian
// diagonal.
//
// For one spin's sorted string set S, the singles and doubles tables list,
// for every source string S_i, the strings S_j of the set that differ from
// it by moving one (single) or two (double) electrons -- the per-string
// excitation lists the sigma product iterates over (paper Sec. III-B,
// Listing 3) -- in canonical CSR form (targets ascending).  Two builders
// produce identical tables:
//   all-pairs  : XOR-popcount of S_i against every S_j (popcount 2 -> single,
//                4 -> double), a warp per source, ballots place the hits;
//   enumerate  : every single/double move of S_i is generated and looked up
//                with the warp-cooperative search; hits are marked in a
//                per-warp bitmap that is then read back in ascending order.
// Fermionic phases are popcount masks over the ket string (Jordan-Wigner
// order within one spin):
//   single q -> p : (-1)^popcount(S_j & bits strictly between p and q)
//                 = <S_i| a+_p a_q |S_j>;
//   double q1<q2 -> p1<p2 : phase(S_j, q2->p2) * phase(S_j', q1->p1), S_j' =
//                 S_j with q2 -> p2, which equals <S_i|a+_p1 a+_p2 a_q2 a_q1|S_j>.
// Matrix elements (Slater-Condon rules, Sec. II-B Eq. 4, for one spin):
//   diagonal  sum_{i in S} h_ii + 1/2 sum_{i,j in S} [(ii|jj) - (ij|ji)]
//   single    phase * [h_pq + sum_{k in S_j} ((pq|kk) - (pk|kq))]
//   double    phase * [(p1 q1|p2 q2) - (p1 q2|p2 q1)]
#include <string.h>

#include <algorithm>

#include "common.cuh"
#include "range_rows.cuh"

namespace sbd {

namespace {

__device__ __forceinline__ double eri_at(const double *__restrict__ eri, int norb, int p, int q, int r, int s)
{
    return __ldg(eri + ((((size_t)p * norb + q) * norb + r) * norb + s));
}

// bits strictly between positions a and b
__device__ __forceinline__ uint64_t between_mask(int a, int b)
{
    const int lo = min(a, b), hi = max(a, b);
    const uint64_t below_hi = (1ull << hi) - 1ull;  // hi <= 63
    const uint64_t upto_lo = (lo >= 63) ? ~0ull : ((1ull << (lo + 1)) - 1ull);
    return below_hi & ~upto_lo;
}

__device__ __forceinline__ int move_phase(uint64_t ket, int from, int to)
{
    return (__popcll(ket & between_mask(from, to)) & 1) ? -1 : 1;
}

// p1, p2 (occupied in si only), q1, q2 (in sj only), each ascending, 255 where there is none; and the phase
struct Move {
    uint8_t orb[4];
    int8_t sign;
};
struct Entry : Move {
    int32_t j;
    double val;
};

__device__ __forceinline__ Move single_move(uint64_t si, uint64_t sj)
{
    const uint64_t x = si ^ sj;
    const int p = __ffsll((long long)(x & si)) - 1, q = __ffsll((long long)(x & sj)) - 1;
    return Move{{(uint8_t)p, 255, (uint8_t)q, 255}, (int8_t)move_phase(sj, q, p)};
}

__device__ __forceinline__ Move double_move(uint64_t si, uint64_t sj)
{
    const uint64_t x = si ^ sj, pb = x & si, qb = x & sj;
    const int p1 = __ffsll((long long)pb) - 1, p2 = 63 - __clzll((long long)pb);
    const int q1 = __ffsll((long long)qb) - 1, q2 = 63 - __clzll((long long)qb);
    const uint64_t sj2 = sj ^ (1ull << q2) ^ (1ull << p2);
    return Move{{(uint8_t)p1, (uint8_t)p2, (uint8_t)q1, (uint8_t)q2},
                (int8_t)(move_phase(sj, q2, p2) * move_phase(sj2, q1, p1))};
}

__device__ Entry make_single(uint64_t si, uint64_t sj, int32_t j, int norb, const double *__restrict__ h,
                             const double *__restrict__ eri)
{
    Entry e;
    static_cast<Move &>(e) = single_move(si, sj);
    const int p = e.orb[0], q = e.orb[2];
    double v = __ldg(h + (size_t)p * norb + q);
    for (uint64_t m = sj; m; m &= m - 1ull) {
        const int k = __ffsll((long long)m) - 1;
        v += eri_at(eri, norb, p, q, k, k) - eri_at(eri, norb, p, k, k, q);
    }
    e.j = j;
    e.val = e.sign * v;
    return e;
}

__device__ Entry make_double(uint64_t si, uint64_t sj, int32_t j, int norb, const double *__restrict__ eri)
{
    Entry e;
    static_cast<Move &>(e) = double_move(si, sj);
    const int p1 = e.orb[0], p2 = e.orb[1], q1 = e.orb[2], q2 = e.orb[3];
    const double v = eri_at(eri, norb, p1, q1, p2, q2) - eri_at(eri, norb, p1, q2, p2, q1);
    e.j = j;
    e.val = e.sign * v;
    return e;
}

// orbitals and phases of `m` entries of a table from entry e0 on (either output may be null)
__global__ void moves_kernel(const uint64_t *__restrict__ S, int64_t n, const int64_t *__restrict__ ptr,
                             const int32_t *__restrict__ tgt, bool singles, int64_t e0, int64_t m, uint32_t *orbs, int8_t *sign)
{
    for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < m; x += (int64_t)gridDim.x * blockDim.x) {
        int64_t lo = 0, hi = n;  // the row: ptr[lo] <= e0 + x < ptr[hi]
        while (hi - lo > 1) {
            const int64_t mid = (lo + hi) / 2;
            if (ptr[mid] <= e0 + x) lo = mid;
            else hi = mid;
        }
        const uint64_t si = S[lo], sj = S[tgt[e0 + x]];
        const Move v = singles ? single_move(si, sj) : double_move(si, sj);
        if (orbs)
            orbs[x] = (uint32_t)v.orb[0] | (uint32_t)v.orb[1] << 8 | (uint32_t)v.orb[2] << 16 | (uint32_t)v.orb[3] << 24;
        if (sign) sign[x] = v.sign;
    }
}

struct TableOut {
    const int64_t *s_ptr, *d_ptr;
    int32_t *s_j, *d_j;
    uint32_t *s_pk;
    double *s_v, *d_v;
};

__device__ __forceinline__ void store_single(const TableOut &o, int64_t pos, const Entry &e, int norb)
{
    o.s_j[pos] = e.j;
    o.s_v[pos] = e.val;
    const uint32_t key = 2u * (uint32_t)(e.orb[0] * norb + e.orb[2]) + (e.sign < 0 ? 1u : 0u);
    o.s_pk[pos] = (uint32_t)e.j | (key << kPackKeyShift);
}

__device__ __forceinline__ void store_double(const TableOut &o, int64_t pos, const Entry &e)
{
    o.d_j[pos] = e.j;
    o.d_v[pos] = e.val;
}

// ---- all-pairs builder -----------------------------------------------------

__global__ void pairs_count_kernel(const uint64_t *__restrict__ S, int64_t n, int64_t *cnt_s, int64_t *cnt_d)
{
    const int lane = threadIdx.x & 31;
    const int64_t nw = (int64_t)gridDim.x * (blockDim.x / 32);
    for (int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / 32; i < n; i += nw) {
        const uint64_t si = S[i];
        int64_t cs = 0, cd = 0;
        for (int64_t j0 = 0; j0 < n; j0 += 32) {
            const int64_t j = j0 + lane;
            const int pc = j < n ? __popcll(si ^ __ldg(S + j)) : 0;
            cs += __popc(__ballot_sync(0xffffffffu, pc == 2));
            cd += __popc(__ballot_sync(0xffffffffu, pc == 4));
        }
        if (lane == 0) {
            cnt_s[i] = cs;
            cnt_d[i] = cd;
        }
    }
}

// A warp collects its hits in shared memory and works them out 32 at a time: one or two hits in a
// window of 32 strings would leave the warp waiting for their integrals with the other lanes idle
// (580 us at 10,000 strings of norb 29).
constexpr int kFillWarps = 8;
__global__ void __launch_bounds__(32 * kFillWarps) pairs_fill_kernel(const uint64_t *__restrict__ S, int64_t n, int norb,
                                                                     const double *__restrict__ h,
                                                                     const double *__restrict__ eri, TableOut o)
{
    __shared__ int32_t queue[kFillWarps][2][64];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    int32_t *qs = queue[wib][0], *qd = queue[wib][1];
    const int64_t nw = (int64_t)gridDim.x * kFillWarps;
    for (int64_t i = blockIdx.x * (int64_t)kFillWarps + wib; i < n; i += nw) {
        const uint64_t si = S[i];
        int64_t ps = o.s_ptr[i], pd = o.d_ptr[i];
        int cs = 0, cd = 0;  // hits waiting
        auto flush_s = [&](int m) {
            if (lane < m) {
                const int32_t j = qs[lane];
                store_single(o, ps + lane, make_single(si, __ldg(S + j), j, norb, h, eri), norb);
            }
            ps += m;
        };
        auto flush_d = [&](int m) {
            if (lane < m) {
                const int32_t j = qd[lane];
                store_double(o, pd + lane, make_double(si, __ldg(S + j), j, norb, eri));
            }
            pd += m;
        };
        for (int64_t j0 = 0; j0 < n; j0 += 32) {
            const int64_t j = j0 + lane;
            const uint64_t sj = j < n ? __ldg(S + j) : si;
            const int pc = __popcll(si ^ sj);
            const unsigned bs = __ballot_sync(0xffffffffu, pc == 2);
            const unsigned bd = __ballot_sync(0xffffffffu, pc == 4);
            if (!(bs | bd)) continue;  // most windows of a large set
            if (pc == 2) qs[cs + __popc(bs & lt)] = (int32_t)j;
            if (pc == 4) qd[cd + __popc(bd & lt)] = (int32_t)j;
            cs += __popc(bs);
            cd += __popc(bd);
            __syncwarp();
            if (cs >= 32) {  // uniform
                flush_s(32);
                cs -= 32;
                const int32_t r = qs[32 + lane];
                __syncwarp();
                qs[lane] = r;
                __syncwarp();
            }
            if (cd >= 32) {
                flush_d(32);
                cd -= 32;
                const int32_t r = qd[32 + lane];
                __syncwarp();
                qd[lane] = r;
                __syncwarp();
            }
        }
        flush_s(cs);
        flush_d(cd);
        __syncwarp();  // the next string's hits reuse the queues
    }
}

// ---- enumerate + lookup builder ---------------------------------------------

constexpr int kEnumWarps = 4;

// pair index k in [0, m(m-1)/2) -> (x, y), x < y, in lexicographic order
__device__ __forceinline__ void unrank_pair(int k, int m, int &x, int &y)
{
    x = 0;
    while (k >= m - 1 - x) {
        k -= m - 1 - x;
        ++x;
    }
    y = x + 1 + k;
}

__device__ void mark_hits(const uint64_t *__restrict__ S, int64_t n, uint64_t t, bool valid, unsigned *bitmap)
{
    const int lane = threadIdx.x & 31;
    unsigned todo = __ballot_sync(0xffffffffu, valid);
    while (todo) {
        const int src = __ffs(todo) - 1;
        todo &= todo - 1u;
        const uint64_t key = __shfl_sync(0xffffffffu, t, src);
        const int64_t idx = warp_find(S, n, key);
        if (lane == 0 && idx >= 0) atomicOr(bitmap + (idx >> 5), 1u << (idx & 31));
    }
}

// mode 0: counts, mode 1: fill
__global__ void enum_kernel(const uint64_t *__restrict__ S, int64_t n, int norb, int nel, int mode,
                            int64_t *cnt_s, int64_t *cnt_d, const double *__restrict__ h,
                            const double *__restrict__ eri, TableOut o)
{
    extern __shared__ unsigned smem_u[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int64_t words = (n + 31) / 32;
    unsigned *bitmap = smem_u + (size_t)wib * words;
    __shared__ uint8_t occ_s[kEnumWarps][64], vir_s[kEnumWarps][64];
    uint8_t *occ = occ_s[wib], *vir = vir_s[wib];
    const unsigned lt = (1u << lane) - 1u;
    const int64_t nw = (int64_t)gridDim.x * kEnumWarps;
    const int no = nel, nv = norb - nel;
    for (int64_t i = blockIdx.x * (int64_t)kEnumWarps + wib; i < n; i += nw) {
        const uint64_t si = S[i];
        int oseen = 0, vseen = 0;
        for (int half = 0; half < 2; ++half) {
            const int m = lane + 32 * half;
            const bool inr = m < norb;
            const bool isocc = inr && ((si >> m) & 1ull);
            const unsigned mo = __ballot_sync(0xffffffffu, isocc);
            const unsigned mv = __ballot_sync(0xffffffffu, inr && !isocc);
            if (isocc) occ[oseen + __popc(mo & lt)] = (uint8_t)m;
            if (inr && !isocc) vir[vseen + __popc(mv & lt)] = (uint8_t)m;
            oseen += __popc(mo);
            vseen += __popc(mv);
        }
        for (int64_t w = lane; w < words; w += 32) bitmap[w] = 0u;
        __syncwarp();
        const int nsc = no * nv;
        for (int c0 = 0; c0 < nsc; c0 += 32) {
            const int cidx = c0 + lane;
            const bool valid = cidx < nsc;
            uint64_t t = 0;
            if (valid) t = si ^ (1ull << occ[cidx / nv]) ^ (1ull << vir[cidx % nv]);
            mark_hits(S, n, t, valid, bitmap);
        }
        const int npo = no * (no - 1) / 2, npv = nv * (nv - 1) / 2;
        const int64_t ndc = (int64_t)npo * npv;
        for (int64_t c0 = 0; c0 < ndc; c0 += 32) {
            const int64_t cidx = c0 + lane;
            const bool valid = cidx < ndc;
            uint64_t t = 0;
            if (valid) {
                int a1, a2, b1, b2;
                unrank_pair((int)(cidx / npv), no, a1, a2);
                unrank_pair((int)(cidx % npv), nv, b1, b2);
                t = si ^ (1ull << occ[a1]) ^ (1ull << occ[a2]) ^ (1ull << vir[b1]) ^ (1ull << vir[b2]);
            }
            mark_hits(S, n, t, valid, bitmap);
        }
        __syncwarp();
        int64_t ps = mode ? o.s_ptr[i] : 0, pd = mode ? o.d_ptr[i] : 0;
        for (int64_t w0 = 0; w0 < words; w0 += 32) {
            const int64_t w = w0 + lane;
            const unsigned bits = w < words ? bitmap[w] : 0u;
            int cs = 0, cd = 0;
            for (unsigned b = bits; b; b &= b - 1u) {
                const int64_t j = w * 32 + (__ffs(b) - 1);
                const int pc = __popcll(si ^ __ldg(S + j));
                cs += pc == 2;
                cd += pc == 4;
            }
            // exclusive warp prefix of (cs, cd)
            int xs = cs, xd = cd;
            for (int off = 1; off < 32; off <<= 1) {
                const int ys = __shfl_up_sync(0xffffffffu, xs, off);
                const int yd = __shfl_up_sync(0xffffffffu, xd, off);
                if (lane >= off) {
                    xs += ys;
                    xd += yd;
                }
            }
            const int ts = __shfl_sync(0xffffffffu, xs, 31), td = __shfl_sync(0xffffffffu, xd, 31);
            if (mode) {
                int64_t qs = ps + xs - cs, qd = pd + xd - cd;
                for (unsigned b = bits; b; b &= b - 1u) {
                    const int64_t j = w * 32 + (__ffs(b) - 1);
                    const uint64_t sj = __ldg(S + j);
                    const int pc = __popcll(si ^ sj);
                    if (pc == 2) store_single(o, qs++, make_single(si, sj, (int32_t)j, norb, h, eri), norb);
                    else if (pc == 4) store_double(o, qd++, make_double(si, sj, (int32_t)j, norb, eri));
                }
            }
            ps += ts;
            pd += td;
        }
        if (!mode && lane == 0) {
            cnt_s[i] = ps;
            cnt_d[i] = pd;
        }
        __syncwarp();
    }
    (void)lt;
}

// ---- scan, diagonal energies, conversions, Hamiltonian diagonal ---------------

// ptr[0] = 0, ptr[i+1] = ptr[i] + cnt[i]; one CTA, each thread a contiguous chunk
__global__ void __launch_bounds__(1024) scan_kernel(const int64_t *cnt, int64_t n, int64_t *ptr)
{
    __shared__ int64_t part[1024];
    const int tid = threadIdx.x;
    const int64_t chunk = (n + 1023) / 1024;
    const int64_t b = tid * chunk, e = min(n, b + chunk);
    int64_t s = 0;
    for (int64_t i = b; i < e; ++i) s += cnt[i];
    part[tid] = s;
    __syncthreads();
    if (tid == 0) {
        int64_t run = 0;
        for (int t = 0; t < 1024; ++t) {
            const int64_t v = part[t];
            part[t] = run;
            run += v;
        }
    }
    __syncthreads();
    int64_t run = part[tid];
    if (tid == 0) ptr[0] = 0;
    for (int64_t i = b; i < e; ++i) {
        run += cnt[i];
        ptr[i + 1] = run;
    }
}

// The same over many elements, in tiles: sums of the tiles, their scan (scan_kernel), the tiles' scans.
constexpr int kScanPer = 8, kScanTile = 1024 * kScanPer;
__device__ __forceinline__ int64_t scan_block(int64_t v, int64_t &total)  // exclusive, over 1024 threads
{
    __shared__ int64_t wsum[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int64_t x = v;
    for (int off = 1; off < 32; off <<= 1) {
        const int64_t y = __shfl_up_sync(0xffffffffu, x, off);
        if (lane >= off) x += y;
    }
    if (lane == 31) wsum[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int64_t w = wsum[lane];
        for (int off = 1; off < 32; off <<= 1) {
            const int64_t y = __shfl_up_sync(0xffffffffu, w, off);
            if (lane >= off) w += y;
        }
        wsum[lane] = w;
    }
    __syncthreads();
    total = wsum[31];
    return x - v + (warp ? wsum[warp - 1] : 0);
}
__global__ void __launch_bounds__(1024) scan_sums_kernel(const int64_t *__restrict__ cnt, int64_t n, int64_t *sums)
{
    int64_t s = 0, total;
    for (int u = 0; u < kScanPer; ++u) {
        const int64_t i = (int64_t)blockIdx.x * kScanTile + u * 1024 + threadIdx.x;
        if (i < n) s += cnt[i];
    }
    scan_block(s, total);
    if (threadIdx.x == 0) sums[blockIdx.x] = total;
}
__global__ void __launch_bounds__(1024) scan_tiles_kernel(const int64_t *__restrict__ cnt, int64_t n,
                                                          const int64_t *__restrict__ off, int64_t *ptr)
{
    const int64_t b = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanPer;
    int64_t v[kScanPer], s = 0, total;
    for (int u = 0; u < kScanPer; ++u) s += v[u] = b + u < n ? cnt[b + u] : 0;
    int64_t run = off[blockIdx.x] + scan_block(s, total);
    if (b == 0) ptr[0] = 0;
    for (int u = 0; u < kScanPer; ++u) {
        run += v[u];
        if (b + u < n) ptr[b + u + 1] = run;
    }
}

__global__ void ediag_kernel(const uint64_t *S, int64_t n, int norb, const double *__restrict__ h,
                             const double *__restrict__ eri, double *out)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t s = S[i];
        double one = 0.0, two = 0.0;
        for (uint64_t a = s; a; a &= a - 1ull) {
            const int p = __ffsll((long long)a) - 1;
            one += __ldg(h + (size_t)p * norb + p);
            for (uint64_t b = s; b; b &= b - 1ull) {
                const int q = __ffsll((long long)b) - 1;
                two += eri_at(eri, norb, p, p, q, q) - eri_at(eri, norb, p, q, q, p);
            }
        }
        out[i] = one + 0.5 * two;
    }
}

// Sigma order of each source's list.  The list is padded with empty slots to a multiple of
// kListPad and laid out for 16-byte loads: lane l of an 8-lane group fetches slots 4l..4l+3 of
// each 32-slot chunk, and one 128-bit shared-memory phase gathers slot 4l+u of every lane.
// Entries are first ranked as rounds "rank 0 of every target residue mod 8, rank 1 of every
// residue, ...", so that consecutive entries in that order have distinct residues where the
// residue counts allow; each phase then receives a run of consecutive positions.
// round-order position q of a list of Lp slots -> slot: in a chunk of Lc slots (32, or what is left of
// a short list) m = Lc/4 lanes each fetch 4 slots, and phase u gathers slot 4*l + u of every lane l;
// position m*u + l goes to slot 4*l + u, so each phase reads m consecutive round-order positions
__device__ __forceinline__ int slot_of(int q, int Lp)
{
    const int chunk = q / 32, within = q % 32;
    const int m = min(32, Lp - chunk * 32) / 4;
    return chunk * 32 + 4 * (within % m) + within / m;
}

// Singles lists, where the gathers read two tables: staged amplitudes by target j and coefficient
// rows by key = 2*code + neg (16-byte rows, bank group = index mod 8).  Each phase of m positions is
// filled one entry at a time with the untaken entry that scores highest: residues new to the phase
// first (both sides, then one), and among those the residues most frequent among the untaken
// entries, since the busiest residue classes bound the number of conflict-free phases.  Lists longer
// than kJointMax keep the target-only order.
// The picks follow one another; a warp scores a list's entries at once (one thread per list: up to 1.3 ms
// for a few thousand strings).
constexpr int kJointMax = 1024;
__global__ void joint_order_kernel(const int64_t *__restrict__ beg, const int64_t *__restrict__ end,
                                   const int64_t *__restrict__ sig_ptr, int64_t n, const int32_t *__restrict__ j_src,
                                   const uint32_t *__restrict__ pk, int32_t *perm)
{
    const int lane = threadIdx.x & 31;
    for (int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / 32; i < n;
         i += (int64_t)gridDim.x * blockDim.x / 32) {
        const int64_t b = beg[i], e = end[i], sb = sig_ptr[i];
        const int L = (int)(e - b), Lp = (int)(sig_ptr[i + 1] - sb);
        if (L > kJointMax) continue;  // sigma_order_kernel orders these
        for (int q = lane; q < Lp; q += 32) perm[sb + q] = -1;  // slots no entry lands on stay padding
        // entry x = lane + 32 y: residues of its target (3 bits) and coefficient row (3 bits), taken when
        // bit y of `taken` is set; lane r < 8 counts the untaken entries of target residue r, lane 8 + r of
        // row residue r
        unsigned taken = 0u;
        int count = 0;
        for (int x0 = 0; x0 < L; x0 += 32) {
            const int x = x0 + lane;
            const bool in = x < L;
            const int rj = in ? j_src[b + x] & 7 : -1, rk = in ? (int)(pk[b + x] >> kPackKeyShift) & 7 : -1;
            for (int r = 0; r < 8; ++r) {
                const int cj = __popc(__ballot_sync(0xffffffffu, rj == r)), ck = __popc(__ballot_sync(0xffffffffu, rk == r));
                if (lane == r) count += cj;
                if (lane == 8 + r) count += ck;
            }
        }
        __syncwarp();
        int q = 0;
        while (q < L) {
            const int chunk = q / 32;
            const int m = min(32, Lp - chunk * 32) / 4;
            const int phase_end = min(L, q + m - (q - chunk * 32) % m);  // end of the phase q lies in
            unsigned used_j = 0u, used_k = 0u;
            for (; q < phase_end; ++q) {
                int best = -1;  // (score << 10 | 1023 - x): the largest score, the first entry among equals
                for (int x0 = 0, y = 0; x0 < L; x0 += 32, ++y) {
                    const int x = x0 + lane;
                    const bool in = x < L && !((taken >> y) & 1u);
                    const int rj = x < L ? j_src[b + x] & 7 : 0, rk = x < L ? (int)(pk[b + x] >> kPackKeyShift) & 7 : 0;
                    const int cj = __shfl_sync(0xffffffffu, count, rj), ck = __shfl_sync(0xffffffffu, count, 8 + rk);
                    const int fresh = (int)!((used_j >> rj) & 1u) + (int)!((used_k >> rk) & 1u);
                    if (in) best = max(best, ((fresh * 4096 + cj + ck) << 10) | (kJointMax - 1 - x));
                }
                best = __reduce_max_sync(0xffffffffu, best);
                const int x = kJointMax - 1 - (best & (kJointMax - 1));
                const int rj = j_src[b + x] & 7, rk = (int)(pk[b + x] >> kPackKeyShift) & 7;
                if ((x & 31) == lane) taken |= 1u << (x >> 5);
                if (lane == rj || lane == 8 + rk) --count;
                used_j |= 1u << rj;
                used_k |= 1u << rk;
                if (lane == 0) perm[sb + slot_of(q, Lp)] = (int32_t)(b + x);
            }
        }
    }
}

// perm[sig_ptr[i] + slot] = index of the canonical entry (of [beg[i], end[i])), or -1 for padding.  One thread per
// source.
// joint: lists of at most kJointMax entries are joint_order_kernel's.
__global__ void sigma_order_kernel(const int64_t *__restrict__ beg, const int64_t *__restrict__ end,
                                   const int64_t *__restrict__ sig_ptr, int64_t n, const int32_t *__restrict__ j_src,
                                   bool joint, int32_t *perm)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t b = beg[i], e = end[i], sb = sig_ptr[i], se = sig_ptr[i + 1];
        const int Lp = (int)(se - sb);
        if (joint && e - b <= kJointMax) continue;
        for (int q = 0; q < Lp; ++q) perm[sb + q] = -1;  // slots no entry lands on stay padding
        int count[kBankGroups] = {0, 0, 0, 0, 0, 0, 0, 0};
        for (int64_t x = b; x < e; ++x) ++count[j_src[x] & (kBankGroups - 1)];
        int seen[kBankGroups] = {0, 0, 0, 0, 0, 0, 0, 0};
        for (int64_t x = b; x < e; ++x) {
            const int r = j_src[x] & (kBankGroups - 1);
            const int t = seen[r]++;
            int q = 0;  // position in round order
#pragma unroll
            for (int w = 0; w < kBankGroups; ++w) q += min(count[w], t) + ((w < r && count[w] > t) ? 1 : 0);
            perm[sb + slot_of(q, Lp)] = (int32_t)x;
        }
    }
}

// first entry of [lo, hi) with target >= key (targets ascend)
__device__ __forceinline__ int64_t first_at_least(const int32_t *__restrict__ tgt, int64_t lo, int64_t hi, int64_t key)
{
    while (lo < hi) {
        const int64_t mid = (lo + hi) / 2;
        if (tgt[mid] < key) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// x = hi + lo with hi the FP32 rounding of x and lo the FP32 rounding of the remainder
__device__ __forceinline__ float2 split2(double x)
{
    const float hi = __double2float_rn(x);
    return make_float2(hi, __double2float_rn(x - (double)hi));
}

// entries of list r0 + i with targets in [j0, j1): [beg[i], end[i])
__global__ void row_bounds_kernel(const int64_t *__restrict__ ptr, const int32_t *__restrict__ tgt, int64_t r0, int64_t nr,
                                  int64_t j0, int64_t j1, int64_t *beg, int64_t *end)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nr; i += (int64_t)gridDim.x * blockDim.x) {
        beg[i] = first_at_least(tgt, ptr[r0 + i], ptr[r0 + i + 1], j0);
        end[i] = first_at_least(tgt, beg[i], ptr[r0 + i + 1], j1);
    }
}

// The entries perm names, zeros for padding: key (a packed single or, pk null, a target; from j0) and values; a
// null output is left out
__global__ void sig_gather_kernel(const int32_t *__restrict__ perm, int64_t m, const int32_t *__restrict__ j,
                                  const uint32_t *__restrict__ pk, const double *__restrict__ val, int64_t j0, uint32_t *key,
                                  float *hi, float *lo, double *v64)
{
    for (int64_t o = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; o < m; o += (int64_t)gridDim.x * blockDim.x) {
        const int32_t e = perm[o];
        const double v = e >= 0 ? val[e] : 0.0;
        if (key) key[o] = e >= 0 ? (uint32_t)(j[e] - j0) | (pk ? pk[e] & ~kPackJMask : 0u) : 0u;
        const float2 x = split2(v);
        if (hi) hi[o] = x.x;
        if (lo) lo[o] = x.y;
        if (v64) v64[o] = v;
    }
}

// padded counts: cnt[i] = ceil((end[i]-beg[i]) / kListPad) * kListPad
__global__ void padded_count_kernel(const int64_t *__restrict__ beg, const int64_t *__restrict__ end, int64_t n, int64_t *cnt)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t L = end[i] - beg[i];
        cnt[i] = (L + kListPad - 1) / kListPad * kListPad;
    }
}

// Source-major singles (column-stationary alpha-beta pass): cnt[i] = items of string i (its singles
// with a pair in [p0, p1), in pieces of kSrcItem); *maxdeg = largest singles count.
// index of the unordered pair of the orbital code of a packed single
__device__ __forceinline__ int single_pair(uint32_t pk, int norb)
{
    const int code = (int)(pk >> (kPackKeyShift + 1)), p = code / norb;
    return orbital_pair(p, code - p * norb);
}

__global__ void src_count_kernel(const int64_t *__restrict__ ptr, const uint32_t *__restrict__ pk, int64_t n, int norb,
                                 int p0, int p1, int64_t *cnt, int *maxdeg)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        int d = 0;
        for (int64_t x = ptr[i]; x < ptr[i + 1]; ++x) {
            const int pair = single_pair(pk[x], norb);
            d += pair >= p0 && pair < p1;
        }
        cnt[i] = (d + kSrcItem - 1) / kSrcItem;
        atomicMax(maxdeg, (int)(ptr[i + 1] - ptr[i]));
    }
}

// items of string i from item ioff[i] on; each entry keeps the target and phase of the canonical
// single and replaces its orbital code p*norb+q by the index r(r-1)/2 + s - p0 of the pair r = max, s = min
__global__ void src_fill_kernel(const int64_t *__restrict__ ptr, const uint32_t *__restrict__ pk, int64_t n,
                                int norb, int p0, int p1, const int64_t *__restrict__ ioff, uint32_t *item, uint32_t *ent)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t b = ptr[i], e = ptr[i + 1];
        int d = 0;
        for (int64_t x = b; x < e; ++x) {
            const uint32_t v = pk[x];
            const int pair = single_pair(v, norb);
            if (pair < p0 || pair >= p1) continue;
            const int64_t t = ioff[i] + d / kSrcItem;
            const int slot = d % kSrcItem;
            ++d;
            item[t] = (uint32_t)i | ((uint32_t)(slot + 1) << kSrcPairShift);  // the last entry leaves the count
            const uint32_t neg = (v >> kPackKeyShift) & 1u;
            ent[(t / 32) * 32 * kSrcItem + 32 * slot + (t % 32)] =
                (v & kPackJMask) | ((uint32_t)(pair - p0) << kSrcPairShift) | (neg << kSrcNegBit);
        }
    }
}

// Order of the items inside each slice of 32: full items first, then the partial ones by decreasing
// length (stable), so that in every round of the alpha-beta pass the lanes that still have a single
// form a prefix of the warp and whole quarter-warps go idle together.  One warp per slice.
__global__ void src_slice_order_kernel(const uint32_t *__restrict__ item_in, const uint32_t *__restrict__ ent_in,
                                       int64_t nsl, uint32_t *item_out, uint32_t *ent_out)
{
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    for (int64_t s = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / 32; s < nsl;
         s += (int64_t)gridDim.x * blockDim.x / 32) {
        const uint32_t it = item_in[s * 32 + lane];
        const int key = (int)(it >> kSrcPairShift);  // entries of the item, 0 for an empty slot
        int rank = 0;
        for (int c = kSrcItem; c >= 0; --c) {
            const unsigned m = __ballot_sync(0xffffffffu, key == c);
            if (c > key) rank += __popc(m);
            else if (c == key) rank += __popc(m & lt);
        }
        item_out[s * 32 + rank] = it;
        const int64_t base = s * 32 * kSrcItem;
        for (int i = 0; i < kSrcItem; ++i) ent_out[base + 32 * i + rank] = ent_in[base + 32 * i + lane];
    }
}

// Split of each source list at target `half`: ptr2[2i] = start of list i, ptr2[2i+1] = its first
// entry with target >= half (targets ascend in the canonical lists), ptr2[2n] = end of the last list
__global__ void half_split_kernel(const int64_t *__restrict__ ptr, const int32_t *__restrict__ tgt, int64_t n,
                                  int64_t half, int64_t *ptr2)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        int64_t lo = ptr[i], hi = ptr[i + 1];
        ptr2[2 * i] = lo;
        while (lo < hi) {
            const int64_t mid = (lo + hi) / 2;
            if (tgt[mid] < half) lo = mid + 1;
            else hi = mid;
        }
        ptr2[2 * i + 1] = lo;
        if (i == n - 1) ptr2[2 * n] = ptr[n];
    }
}

// Doubles of the half-split lists: val[o] = FP32 of v[perm[o]], tgt[o] = its target relative to
// the column half it lies in (target - half for targets >= half); zeros for padding
__global__ void gather_half_doubles_kernel(const int32_t *__restrict__ perm, int64_t m,
                                           const int32_t *__restrict__ j, const double *__restrict__ v,
                                           int64_t half, float *val, uint16_t *tgt)
{
    for (int64_t o = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; o < m; o += (int64_t)gridDim.x * blockDim.x) {
        const int64_t e = perm[o];
        const int64_t jj = e >= 0 ? (int64_t)j[e] : 0;
        val[o] = e >= 0 ? __double2float_rn(v[e]) : 0.f;
        tgt[o] = (uint16_t)(jj >= half ? jj - half : jj);
    }
}

// out[o] = (key[perm[o]], FP32 of val[perm[o]]), zeros for padding
__global__ void gather_pair_kernel(const int32_t *__restrict__ perm, int64_t m, const uint32_t *__restrict__ key,
                                   const double *__restrict__ val, uint2 *out)
{
    for (int64_t o = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; o < m; o += (int64_t)gridDim.x * blockDim.x) {
        const int64_t e = perm[o];
        out[o] = e >= 0 ? make_uint2(key[e], __float_as_uint(__double2float_rn(val[e]))) : make_uint2(0u, 0u);
    }
}

// ---- range lists of the row passes (RangeLists) --------------------------------

// cnt[g*n + i] = blocks of `pad` entries that string i's list needs for the targets of range g
__global__ void range_count_kernel(const int64_t *__restrict__ ptr, const int32_t *__restrict__ tgt, int64_t n, int w,
                                   int ng, int pad, uint32_t *cnt)
{
    for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < n * ng; x += (int64_t)gridDim.x * blockDim.x) {
        const int64_t g = x / n, i = x - g * n;
        const int64_t lo = first_at_least(tgt, ptr[i], ptr[i + 1], g * w);
        const int64_t hi = first_at_least(tgt, lo, ptr[i + 1], (g + 1) * w);
        cnt[x] = (uint32_t)((hi - lo + pad - 1) / pad);
    }
}

// One CTA per (range, part): counting sort of the part's strings by descending doubles blocks (cd, by
// string) into zi.  (The order of equal lengths is left to the atomics: a list's sum does not depend
// on its position.)
constexpr int kOrderKeys = 1024;
__global__ void __launch_bounds__(256) range_order_kernel(int64_t n, const uint32_t *__restrict__ cd,
                                                          int32_t *zi)
{
    __shared__ unsigned hist[kOrderKeys];
    __shared__ unsigned wsum[8];
    const int64_t g = blockIdx.x / kParts, p = blockIdx.x % kParts;
    const int tid = threadIdx.x;
    for (int k = tid; k < kOrderKeys; k += 256) hist[k] = 0u;
    __syncthreads();
    for (int64_t i = p + (int64_t)kParts * tid; i < n; i += (int64_t)kParts * 256)
        atomicAdd(hist + (kOrderKeys - 1 - min(cd[g * n + i], (unsigned)kOrderKeys - 1u)), 1u);
    __syncthreads();
    // exclusive prefix over the keys, four per thread
    unsigned v[4], s = 0u;
    for (int k = 0; k < 4; ++k) v[k] = hist[4 * tid + k], s += v[k];
    unsigned x = s;
    for (int off = 1; off < 32; off <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, x, off);
        if ((tid & 31) >= off) x += y;
    }
    if ((tid & 31) == 31) wsum[tid >> 5] = x;
    __syncthreads();
    unsigned run = x - s;
    for (int q = 0; q < (tid >> 5); ++q) run += wsum[q];
    for (int k = 0; k < 4; ++k) {
        hist[4 * tid + k] = run;
        run += v[k];
    }
    __syncthreads();
    const int64_t nq = part_group(n, kParts);
    const int64_t z0 = kListGroup * (g * nq + part_group(n, (int)p));
    const int64_t z1 = kListGroup * (g * nq + part_group(n, (int)p + 1));
    for (int64_t i = p + (int64_t)kParts * tid; i < n; i += (int64_t)kParts * 256)
        zi[z0 + atomicAdd(hist + (kOrderKeys - 1 - min(cd[g * n + i], (unsigned)kOrderKeys - 1u)), 1u)] = (int32_t)i;
    for (int64_t z = z0 + (n - p + kParts - 1) / kParts + tid; z < z1; z += 256) zi[z] = -1;
}

// Blocks of each group (the longest of its lists), and the kListHas mark of its strings
__global__ void range_group_kernel(int64_t n, int64_t groups, int64_t total, const uint32_t *__restrict__ cd,
                                  const uint32_t *__restrict__ cs, int32_t *zi, int64_t *nd, int64_t *ns)
{
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < total; q += (int64_t)gridDim.x * blockDim.x) {
        const int64_t g = q / groups;
        uint32_t md = 0, ms = 0;
        for (int o = 0; o < kListGroup; ++o) {
            const int32_t i = zi[kListGroup * q + o];
            if (i < 0) continue;
            const uint32_t d = cd[g * n + i], s = cs[g * n + i];
            md = max(md, d);
            ms = max(ms, s);
            if (d | s) zi[kListGroup * q + o] = i | kListHas;
        }
        nd[q] = md;
        ns[q] = ms;
    }
}

// One warp per list (group q, place o): copies its entries (KIND 1 singles, 2 doubles) to their blocks.
template <int KIND>
__global__ void range_fill_kernel(const int64_t *__restrict__ ptr, const int32_t *__restrict__ tgt,
                                  const uint32_t *__restrict__ pk, const double *__restrict__ val, int64_t groups,
                                  int norb, const int *__restrict__ used, RangeLists r)
{
    constexpr int B = KIND == 1 ? kRangeSingles : kRangeDoubles;
    const uint32_t *qp = KIND == 1 ? r.qs : r.qd;
    const int lane = threadIdx.x & 31;
    const int64_t lists = kListGroup * groups * r.ng;
    for (int64_t z = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / 32; z < lists;
         z += (int64_t)gridDim.x * blockDim.x / 32) {
        const int64_t q = z / kListGroup, g = q / groups;
        const int o = (int)(z % kListGroup);
        const int64_t b0 = qp[q];
        const int len = (int)(qp[q + 1] - qp[q]) * B;
        int64_t lo = 0, hi = 0;
        if (r.zi[z] >= 0 && len > 0) {
            const int64_t i = r.zi[z] & ~kListHas;
            lo = first_at_least(tgt, ptr[i], ptr[i + 1], g * r.w);
            hi = first_at_least(tgt, lo, ptr[i + 1], (g + 1) * r.w);
        }
        for (int x = lane; x < len; x += 32) {
            const int64_t e = lo + x, at = ((b0 + x / B) * kListGroup + o) * B + x % B;
            const bool real = e < hi;
            const uint32_t t = real ? (uint32_t)(tgt[e] - g * r.w) : (uint32_t)r.pad;
            const double v = real ? val[e] : 0.0;
            if constexpr (KIND == 1) {
                // padding: value 0 and pair index np, whose row of the coefficient table is zero
                const uint32_t pair = real ? (uint32_t)used[single_pair(pk[e], norb)] : (uint32_t)r.np;
                const uint32_t neg = real ? (pk[e] >> kPackKeyShift) & 1u : 0u;
                r.sm[at] = t | (pair << 16) | (neg << 31);
                const float2 x = split2(v);
                r.shi[at] = x.x;
                r.slo[at] = x.y;
                if (r.sv64) r.sv64[at] = v;
            } else {
                const float2 x = split2(v);
                r.dt[at] = (uint16_t)t;
                r.dhi[at] = x.x;
                r.dlo[at] = x.y;
                if (r.dv64) r.dv64[at] = v;
            }
        }
    }
}

// flag[pair] = 1 for the pairs of the singles
__global__ void pair_mark_kernel(const uint32_t *__restrict__ pk, int64_t ns, int norb, int *flag)
{
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < ns; e += (int64_t)gridDim.x * blockDim.x) {
        int *f = flag + single_pair(pk[e], norb);
        if (*f == 0) *f = 1;
    }
}

// used[pair] = index of a marked pair among them (in: its mark), list[index] = pair, *np = their number; one
// CTA of 1024 threads, two pairs (of at most 2016) each
__global__ void __launch_bounds__(1024) pair_list_kernel(int *used, int npair, int *list, int *np)
{
    const int x = 2 * threadIdx.x;
    const int f0 = x < npair ? used[x] : 0, f1 = x + 1 < npair ? used[x + 1] : 0;
    int64_t total;
    const int at = (int)scan_block(f0 + f1, total);
    if (f0) used[x] = at, list[at] = x;
    if (f1) used[x + 1] = at + f0, list[at + f0] = x + 1;
    if (threadIdx.x == 0) *np = (int)total;
}

// jg[x][i] = sum_{k in string i} (rs|kk), rs = pair list[x]
__global__ void pair_j_kernel(const uint64_t *__restrict__ S, int64_t n, int norb, const double *__restrict__ eri,
                              const int *__restrict__ list, int np, double *jg)
{
    const int64_t n2 = (int64_t)norb * norb;
    for (int x = blockIdx.y; x < np; x += gridDim.y) {
        const int pair = list[x];
        int r = (int)((1.f + sqrtf(8.f * (float)pair + 1.f)) * 0.5f);
        if (r * (r - 1) / 2 > pair) --r;
        if (r * (r + 1) / 2 <= pair) ++r;
        const double *row = eri + ((int64_t)r * norb + (pair - r * (r - 1) / 2)) * n2;
        for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
            double v = 0.0;
            for (uint64_t m = S[i]; m; m &= m - 1ull) v += __ldg(row + (int64_t)(__ffsll((long long)m) - 1) * (norb + 1));
            jg[(int64_t)x * n + i] = v;
        }
    }
}

// out[pq][rs] = FP32 of (pq|rs), p > q, r > s
__global__ void pack_integrals_kernel(const double *__restrict__ eri, int norb, float *out)
{
    const int npair = norb * (norb - 1) / 2;
    for (int r = 1; r < norb; ++r)
        for (int x = blockIdx.x; x < npair; x += gridDim.x) {
            int p = (int)((1.f + sqrtf(8.f * (float)x + 1.f)) * 0.5f);
            if (p * (p - 1) / 2 > x) --p;
            if (p * (p + 1) / 2 <= x) ++p;
            const int q = x - p * (p - 1) / 2;
            for (int s = threadIdx.x; s < r; s += blockDim.x)
                out[(size_t)x * npair + r * (r - 1) / 2 + s] = (float)eri_at(eri, norb, p, q, r, s);
        }
}

// ---- slices of the two-operand alpha-beta pass -----------------------------------

// sort key of string i: descending number of singles in the low 16 bits, i above
__global__ void slice_key_kernel(const int64_t *__restrict__ ptr, int64_t n, uint64_t *keys)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        keys[i] = ((uint64_t)i << 16) | (uint64_t)(0xffff - min((int64_t)0xffff, ptr[i + 1] - ptr[i]));
}

// strings of the slices, and each slice's steps (its first list is the longest)
__global__ void slice_col_kernel(const uint64_t *__restrict__ keys, int64_t n, int64_t nsl, int32_t *col, int64_t *len)
{
    for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < 32 * nsl; x += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t k = x < n ? keys[x] : 0xffffull;
        const int64_t l = 0xffff - (int64_t)(k & 0xffffull);
        col[x] = l > 0 ? (int32_t)(k >> 16) : -1;
        if ((x & 31) == 0) len[x / 32] = l;
    }
}

__global__ void slice_fill_kernel(const int64_t *__restrict__ ptr, const uint32_t *__restrict__ pk, int64_t n, int norb,
                                  int64_t nsl, const int32_t *__restrict__ col, const uint32_t *__restrict__ off, uint32_t *ent)
{
    for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < 32 * nsl; x += (int64_t)gridDim.x * blockDim.x) {
        const int64_t s = x / 32;
        const int lane = (int)(x % 32), steps = (int)(off[s + 1] - off[s]);
        const int64_t b = col[x] >= 0 ? ptr[col[x]] : 0, e = col[x] >= 0 ? ptr[col[x] + 1] : 0;
        const uint32_t zero = (uint32_t)n | ((uint32_t)(norb * (norb - 1)) << kPackKeyShift);
        for (int t = 0; t < steps; ++t) {
            uint32_t v = zero;
            if (b + t < e) {
                const uint32_t w = pk[b + t], key = w >> kPackKeyShift;
                const int p = (int)(key >> 1) / norb, q = (int)(key >> 1) % norb;
                const int r = max(p, q), m = min(p, q);
                v = (w & kPackJMask) | ((2u * (uint32_t)(r * (r - 1) / 2 + m) + (key & 1u)) << kPackKeyShift);
            }
            ent[((int64_t)off[s] + t) * 32 + lane] = v;
        }
    }
}

// Order inside the lists of one 128-bit phase (8 lanes of a slice; one warp): step by step, each list
// takes from its next kSliceWindow entries the one whose target and coefficient row, modulo 8, no
// earlier list of the step has taken (both, else one, else the first).  The steps follow one another;
// the warp looks at a window at once, in shared memory (one thread per phase in global memory: 945 us
// at 10,000 strings of norb 29, 168 singles in the longest list).
constexpr int kSliceWindow = 16;
constexpr int kSliceSteps = 1024;  // most singles of a string: 32 * 32
__global__ void __launch_bounds__(32) slice_order_kernel(const int64_t *__restrict__ ptr, int64_t nsl,
                                                         const int32_t *__restrict__ col,
                                                         const uint32_t *__restrict__ off, uint32_t *ent)
{
    __shared__ uint32_t w[kSliceSteps * 8];
    const int lane = threadIdx.x;
    for (int64_t x = blockIdx.x; x < 4 * nsl; x += gridDim.x) {
        const int64_t s = x / 4;
        uint32_t *e = ent + (int64_t)off[s] * 32 + 8 * (x % 4);
        const int32_t i = lane < 8 ? col[s * 32 + 8 * (x % 4) + lane] : -1;
        const int len = i >= 0 ? (int)(ptr[i + 1] - ptr[i]) : 0;
        const int most = __reduce_max_sync(0xffffffffu, len);
        for (int z = lane; z < most * 8; z += 32) w[z] = e[32 * (z / 8) + z % 8];
        __syncwarp();
        for (int t = 0; t < most; ++t) {
            unsigned used_j = 0u, used_k = 0u;
            for (int l = 0; l < 8; ++l) {
                const int ll = __shfl_sync(0xffffffffu, len, l);
                if (t >= ll) continue;
                const int y = t + lane;
                const bool in = lane < kSliceWindow && y < ll;
                const uint32_t v = in ? w[8 * y + l] : 0u;
                const bool fj = in && !((used_j >> (v & 7u)) & 1u), fk = in && !((used_k >> ((v >> kPackKeyShift) & 7u)) & 1u);
                const unsigned two = __ballot_sync(0xffffffffu, fj && fk), one = __ballot_sync(0xffffffffu, fj || fk);
                const int best = two ? __ffs(two) - 1 : one ? __ffs(one) - 1 : 0;
                const uint32_t take = __shfl_sync(0xffffffffu, v, best), head = __shfl_sync(0xffffffffu, v, 0);
                if (lane == 0) {
                    w[8 * (t + best) + l] = head;
                    w[8 * t + l] = take;
                }
                __syncwarp();
                used_j |= 1u << (take & 7u);
                used_k |= 1u << ((take >> kPackKeyShift) & 7u);
            }
        }
        for (int z = lane; z < most * 8; z += 32) e[32 * (z / 8) + z % 8] = w[z];
        __syncwarp();
    }
}

// out[i] = in[i] (a scan of block counts that fits 32 bits)
__global__ void narrow_kernel(const int64_t *__restrict__ in, uint32_t *out, int64_t n)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = (uint32_t)in[i];
}

// Order of the entries inside the items of each slice: in round i every lane of the warp adds the
// dot product of its item's i-th entry into the row accumulator at the entry's target (32-bit shared
// atomics, bank = target mod 32).  A local search, one warp per slice: lane after lane, the exchange of
// two of the lane's entries that removes most pairs of lanes with equal banks in a round is made, a few
// times over.  Any order gives the same sums.  (Picking each round's entries greedily in lane order left
// 2.0 wavefronts per atomic, this 1.6; one thread per slice took 167 us of a create, this takes a tenth.)
constexpr int kEntryPasses = 6;
constexpr int kEntryWarps = 4;
__global__ void src_entry_order_kernel(const uint32_t *__restrict__ item, uint32_t *ent, int64_t nsl)
{
    __shared__ uint32_t es[kEntryWarps][kSrcItem * 32];
    __shared__ int cs[kEntryWarps][kSrcItem * 32];  // lanes of a round with the bank
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    uint32_t *e = es[wib];
    int *cnt = cs[wib];
    static_assert(kSrcItem * (kSrcItem - 1) / 2 <= 32, "one pair of entries per lane");
    int pb = 1, pa = lane;  // lane's pair of places pa < pb
    while (pa >= pb) pa -= pb++;
    for (int64_t s = blockIdx.x * (int64_t)kEntryWarps + wib; s < nsl; s += (int64_t)gridDim.x * kEntryWarps) {
        uint32_t *es_g = ent + s * 32 * kSrcItem;
        const int n = (int)(item[s * 32 + lane] >> kSrcPairShift);
        for (int i = 0; i < kSrcItem; ++i) {
            e[32 * i + lane] = es_g[32 * i + lane];
            cnt[32 * i + lane] = 0;
        }
        __syncwarp();
        for (int i = 0; i < n; ++i) atomicAdd(cnt + 32 * i + (int)(e[32 * i + lane] & 31u), 1);
        __syncwarp();
        for (int pass = 0; pass < kEntryPasses; ++pass) {
            bool any = false;
            for (int l = 0; l < 32; ++l) {
                const int nl = __shfl_sync(0xffffffffu, n, l);
                int best = 0;  // (pairs of equal banks added + 64) << 5 | lane, the smallest
                if (pb < nl) {
                    const int x = (int)(e[32 * pa + l] & 31u), y = (int)(e[32 * pb + l] & 31u);
                    best = x == y ? 0 : (cnt[32 * pb + x] + cnt[32 * pa + y]) - (cnt[32 * pa + x] + cnt[32 * pb + y] - 2);
                }
                best = __reduce_min_sync(0xffffffffu, ((best + 64) << 5) | lane);
                if ((best >> 5) - 64 < 0) {  // uniform
                    any = true;
                    if (lane == (best & 31)) {
                        const uint32_t u = e[32 * pa + l], v = e[32 * pb + l];
                        e[32 * pa + l] = v;
                        e[32 * pb + l] = u;
                        --cnt[32 * pa + (u & 31u)];
                        ++cnt[32 * pb + (u & 31u)];
                        --cnt[32 * pb + (v & 31u)];
                        ++cnt[32 * pa + (v & 31u)];
                    }
                    __syncwarp();
                }
            }
            if (!any) break;
        }
        __syncwarp();
        for (int i = 0; i < kSrcItem; ++i) es_g[32 * i + lane] = e[32 * i + lane];
        __syncwarp();
    }
}

__global__ void to_float_kernel(const double *in, float *out, int64_t n)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = __double2float_rn(in[i]);
}

// Hd[ia, ib] = E_alpha(ia) + E_beta(ib) + sum_{p in ia, r in ib} (pp|rr)   (Sec. II-E).  Bound by the FP64
// pipe, one addition per electron.  (Looking the sum up byte by byte halves the time, but rounds
// differently: determinants of equal energy then take another order, and a solve that starts from the
// lowest of them can take another path.)
__global__ void hdiag_kernel(const uint64_t *__restrict__ A, const uint64_t *__restrict__ B,
                             const double *__restrict__ eA, const double *__restrict__ eB,
                             const double *__restrict__ eri, int norb, int64_t nA, int64_t nB, double *hd)
{
    __shared__ double jd[64];
    for (int64_t ia = blockIdx.x; ia < nA; ia += gridDim.x) {
        const uint64_t a = A[ia];
        if (threadIdx.x < norb) {
            const int r = threadIdx.x;
            double s = 0.0;
            for (uint64_t m = a; m; m &= m - 1ull) {
                const int p = __ffsll((long long)m) - 1;
                s += eri_at(eri, norb, p, p, r, r);
            }
            jd[r] = s;
        }
        __syncthreads();
        const double ea = eA[ia];
        for (int64_t ib = threadIdx.x; ib < nB; ib += blockDim.x) {
            double v = ea + eB[ib];
            for (uint64_t m = B[ib]; m; m &= m - 1ull) v += jd[__ffsll((long long)m) - 1];
            hd[ia * nB + ib] = v;
        }
        __syncthreads();
    }
}

int blocks_for(int64_t n, int threads, int cap = 65535)
{
    int64_t g = (n + threads - 1) / threads;
    if (g < 1) g = 1;
    if (g > cap) g = cap;
    return (int)g;
}

}  // namespace

void table_moves(const Ctx &c, int spin, bool singles, uint8_t *orbs_host, int8_t *sign_host)
{
    constexpr int64_t kPiece = 1 << 20;
    const SpinTables &t = c.sp[spin];
    const int64_t total = singles ? t.ns : t.nd;
    if (!total || (!orbs_host && !sign_host)) return;
    struct Staging {  // pinned: the kernel writes to it
        unsigned char *p = nullptr;
        ~Staging() { (void)cudaFreeHost(p); }
    } st;
    const int64_t piece = std::min(total, kPiece);
    if (cudaHostAlloc((void **)&st.p, (size_t)piece * 5, cudaHostAllocMapped) != cudaSuccess) {
        (void)cudaGetLastError();
        fail(SBD_ERR_OUT_OF_MEMORY, "pinned staging for the tables");
    }
    uint32_t *orbs = orbs_host ? reinterpret_cast<uint32_t *>(st.p) : nullptr;
    int8_t *sign = sign_host ? reinterpret_cast<int8_t *>(st.p + 4 * piece) : nullptr;
    for (int64_t e = 0; e < total; e += piece) {
        const int64_t m = std::min(piece, total - e);
        moves_kernel<<<blocks_for(m, 256), 256, 0, c.stream>>>(t.strings, t.n, singles ? t.s_ptr : t.d_ptr,
                                                               singles ? t.s_j : t.d_j, singles, e, m, orbs, sign);
        SBD_LAUNCH("moves_kernel");
        SBD_CUDA(cudaStreamSynchronize(c.stream));
        if (orbs) memcpy(orbs_host + 4 * e, orbs, (size_t)m * 4);
        if (sign) memcpy(sign_host + e, sign, (size_t)m);
    }
}

// One CTA up to kScanOne elements (its time grows with them: 0.12 ms at 60,000, 11 ms at 5.6e6 list groups)
constexpr int64_t kScanOne = 1 << 14;
static void scan(Ctx &c, const int64_t *cnt, int64_t n, int64_t *ptr)
{
    if (n <= kScanOne) {
        scan_kernel<<<1, 1024, 0, c.stream>>>(cnt, n, ptr);
        SBD_LAUNCH("scan_kernel");
        return;
    }
    const int64_t tiles = (n + kScanTile - 1) / kScanTile;
    int64_t *sums = dalloc_n<int64_t>(c, 2 * (size_t)tiles + 1);
    scan_sums_kernel<<<(unsigned)tiles, 1024, 0, c.stream>>>(cnt, n, sums);
    SBD_LAUNCH("scan_sums_kernel");
    scan_kernel<<<1, 1024, 0, c.stream>>>(sums, tiles, sums + tiles);
    SBD_LAUNCH("scan_kernel");
    scan_tiles_kernel<<<(unsigned)tiles, 1024, 0, c.stream>>>(cnt, n, sums + tiles, ptr);
    SBD_LAUNCH("scan_tiles_kernel");
    dfree(c, sums);
}

void to_float(const double *in, float *out, int64_t n, cudaStream_t s)
{
    if (n <= 0) return;
    to_float_kernel<<<blocks_for(n, 256, 16384), 256, 0, s>>>(in, out, n);
    SBD_LAUNCH("to_float_kernel");
}

void build_tables(Ctx &c, int spin)
{
    SpinTables &t = c.sp[spin];
    const int64_t n = t.n;
    const int norb = c.norb;
    if (n >= kMaxStringsPerSpin) fail(SBD_ERR_UNSUPPORTED, "at most 262143 strings per spin are supported");
    int64_t *cnt = dalloc_n<int64_t>(c, 2 * (size_t)n);
    t.s_ptr = dalloc_n<int64_t>(c, n + 1);
    t.d_ptr = dalloc_n<int64_t>(c, n + 1);

    int algo = c.opt.table_algo;
    if (algo == 0) {
        // all-pairs costs n^2/32 warp steps; enumeration about n * moves * (log32 n + 1)
        double moves = (double)t.nel * (norb - t.nel) +
                       0.25 * t.nel * (t.nel - 1.0) * (norb - t.nel) * (norb - t.nel - 1.0);
        double steps = 1.0;
        for (double r = (double)n; r > 32.0; r /= 32.0) steps += 1.0;
        algo = ((double)n / 32.0 > moves * steps && n <= (1 << 17)) ? 2 : 1;
    }
    if (algo == 2 && n > (1 << 17)) fail(SBD_ERR_UNSUPPORTED, "enumerate+lookup tables need |S| <= 131072");
    const int64_t words = (n + 31) / 32;
    const size_t enum_smem = (size_t)kEnumWarps * words * sizeof(unsigned);
    int warps_per_block = 8, threads = 256;
    int grid = blocks_for(n, warps_per_block, 4 * 65535);
    grid = grid > 65535 ? 65535 : grid;
    TableOut o{};
    if (algo == 1) {
        pairs_count_kernel<<<grid, threads, 0, c.stream>>>(t.strings, n, cnt, cnt + n);
        SBD_LAUNCH("pairs_count_kernel");
    } else {
        SBD_CUDA(cudaFuncSetAttribute(enum_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)enum_smem));
        int eg = blocks_for(n, kEnumWarps, 65535);
        enum_kernel<<<eg, 32 * kEnumWarps, enum_smem, c.stream>>>(t.strings, n, norb, t.nel, 0, cnt, cnt + n,
                                                                  c.h64, c.eri64, o);
        SBD_LAUNCH("enum_kernel(count)");
    }
    scan(c, cnt, n, t.s_ptr);
    scan(c, cnt + n, n, t.d_ptr);
    SBD_CUDA(cudaMemcpyAsync(&t.ns, t.s_ptr + n, sizeof(int64_t), cudaMemcpyDeviceToHost, c.stream));
    SBD_CUDA(cudaMemcpyAsync(&t.nd, t.d_ptr + n, sizeof(int64_t), cudaMemcpyDeviceToHost, c.stream));
    SBD_CUDA(cudaStreamSynchronize(c.stream));
    if (t.ns > 0x7fffffffLL || t.nd > 0x7fffffffLL) fail(SBD_ERR_UNSUPPORTED, "excitation table too large");

    t.s_j = dalloc_n<int32_t>(c, t.ns);
    t.s_pk = dalloc_n<uint32_t>(c, t.ns);
    t.s_v64 = dalloc_n<double>(c, t.ns);
    t.d_j = dalloc_n<int32_t>(c, t.nd);
    t.d_v64 = dalloc_n<double>(c, t.nd);
    o.s_ptr = t.s_ptr;
    o.d_ptr = t.d_ptr;
    o.s_j = t.s_j;
    o.d_j = t.d_j;
    o.s_pk = t.s_pk;
    o.s_v = t.s_v64;
    o.d_v = t.d_v64;
    if (algo == 1) {
        pairs_fill_kernel<<<grid, threads, 0, c.stream>>>(t.strings, n, norb, c.h64, c.eri64, o);
        SBD_LAUNCH("pairs_fill_kernel");
    } else {
        int eg = blocks_for(n, kEnumWarps, 65535);
        enum_kernel<<<eg, 32 * kEnumWarps, enum_smem, c.stream>>>(t.strings, n, norb, t.nel, 1, nullptr, nullptr,
                                                                  c.h64, c.eri64, o);
        SBD_LAUNCH("enum_kernel(fill)");
    }
    t.ediag = dalloc_n<double>(c, n);
    ediag_kernel<<<blocks_for(n, 128), 128, 0, c.stream>>>(t.strings, n, norb, c.h64, c.eri64, t.ediag);
    SBD_LAUNCH("ediag_kernel");
    dfree(c, cnt);
}

// sigma order of n lists; pk (singles only): packed entries, for the joint target/row order
static void order_lists(Ctx &c, const int64_t *beg, const int64_t *end, const int64_t *sig_ptr, int64_t n, const int32_t *j,
                        const uint32_t *pk, int32_t *perm)
{
    if (pk) {
        joint_order_kernel<<<blocks_for(n, 4, 65535), 128, 0, c.stream>>>(beg, end, sig_ptr, n, j, pk, perm);
        SBD_LAUNCH("joint_order_kernel");
    }
    sigma_order_kernel<<<blocks_for(n, 128), 128, 0, c.stream>>>(beg, end, sig_ptr, n, j, pk != nullptr, perm);
    SBD_LAUNCH("sigma_order_kernel");
}

void build_sig_lists(Ctx &c, const SpinTables &t, int64_t r0, int64_t nr, int64_t j0, int64_t j1, int mask, SigLists &out)
{
    const int add = mask & ~out.mask;
    if (!add) return;
    int64_t *beg = dalloc_n<int64_t>(c, (size_t)nr), *end = dalloc_n<int64_t>(c, (size_t)nr);
    for (int kind = 1; kind <= 2; ++kind) {
        const bool singles = kind == 1;
        const int32_t *j = singles ? t.s_j : t.d_j;
        const uint32_t *pk = singles ? t.s_pk : nullptr;
        int64_t *&ptr = singles ? out.s_ptr : out.d_ptr;
        int64_t &m = singles ? out.ns : out.nd;
        row_bounds_kernel<<<blocks_for(nr, 256), 256, 0, c.stream>>>(singles ? t.s_ptr : t.d_ptr, j, r0, nr, j0, j1, beg, end);
        SBD_LAUNCH("row_bounds_kernel");
        if (!out.mask) {
            int64_t *cnt = dalloc_n<int64_t>(c, (size_t)nr);
            ptr = dalloc_n<int64_t>(c, (size_t)nr + 1);
            padded_count_kernel<<<blocks_for(nr, 256), 256, 0, c.stream>>>(beg, end, nr, cnt);
            SBD_LAUNCH("padded_count_kernel");
            scan(c, cnt, nr, ptr);
            SBD_CUDA(cudaMemcpyAsync(&m, ptr + nr, sizeof(int64_t), cudaMemcpyDeviceToHost, c.stream));
            SBD_CUDA(cudaStreamSynchronize(c.stream));
            dfree(c, cnt);
        }
        uint32_t *key = nullptr;
        if (!out.mask) {
            key = dalloc_n<uint32_t>(c, (size_t)m);
            if (singles) out.s_pk = key;
            else out.d_j = reinterpret_cast<int32_t *>(key);
        }
        float *hi = add & kValHi ? dalloc_n<float>(c, (size_t)m) : nullptr;
        float *lo = add & kValLo ? dalloc_n<float>(c, (size_t)m) : nullptr;
        double *v = add & kValF64 ? dalloc_n<double>(c, (size_t)m) : nullptr;
        if (hi) (singles ? out.s_hi : out.d_hi) = hi;
        if (lo) (singles ? out.s_lo : out.d_lo) = lo;
        if (v) (singles ? out.s_v : out.d_v) = v;
        if (m) {
            int32_t *perm = dalloc_n<int32_t>(c, (size_t)m);
            order_lists(c, beg, end, ptr, nr, j, pk, perm);
            sig_gather_kernel<<<blocks_for(m, 256, 16384), 256, 0, c.stream>>>(perm, m, j, pk, singles ? t.s_v64 : t.d_v64, j0,
                                                                              key, hi, lo, v);
            SBD_LAUNCH("sig_gather_kernel");
            dfree(c, perm);
        }
    }
    dfree(c, beg);
    dfree(c, end);
    out.mask |= add;
}

// Lists split at the middle of the string set
static void build_half_lists(Ctx &c, SpinTables &t)
{
    const int64_t n = t.n;
    // mixed-sigma lists split at the middle of the set (row passes over column halves); their
    // 16-bit doubles targets need half <= 65536 (the staged halves fit shared memory only far below)
    if ((n + 1) / 2 <= 65536) {
        t.half = (n + 1) / 2;
        int64_t *ptr2 = dalloc_n<int64_t>(c, 2 * (size_t)n + 1);
        int64_t *cnt2 = dalloc_n<int64_t>(c, 2 * (size_t)n);
        for (int kind = 0; kind < 2; ++kind) {
            const int64_t *ptr = kind == 0 ? t.s_ptr : t.d_ptr;
            const int32_t *tgt = kind == 0 ? t.s_j : t.d_j;
            int64_t *&hptr = kind == 0 ? t.hs_ptr : t.hd_ptr;
            half_split_kernel<<<blocks_for(n, 256), 256, 0, c.stream>>>(ptr, tgt, n, t.half, ptr2);
            SBD_LAUNCH("half_split_kernel");
            hptr = dalloc_n<int64_t>(c, 2 * (size_t)n + 1);
            padded_count_kernel<<<blocks_for(2 * n, 256), 256, 0, c.stream>>>(ptr2, ptr2 + 1, 2 * n, cnt2);
            SBD_LAUNCH("padded_count_kernel(halves)");
            scan(c, cnt2, 2 * n, hptr);
            int64_t m = 0;
            SBD_CUDA(cudaMemcpyAsync(&m, hptr + 2 * n, sizeof(int64_t), cudaMemcpyDeviceToHost, c.stream));
            SBD_CUDA(cudaStreamSynchronize(c.stream));
            const size_t mm = (size_t)std::max<int64_t>(m, 1);
            if (kind == 0) {
                t.hs = dalloc_n<uint2>(c, mm);
            } else {
                t.hdv = dalloc_n<float>(c, mm);
                t.hdt = dalloc_n<uint16_t>(c, mm);
            }
            if (m) {
                int32_t *hperm = dalloc_n<int32_t>(c, (size_t)m);
                order_lists(c, ptr2, ptr2 + 1, hptr, 2 * n, tgt, kind == 0 ? t.s_pk : nullptr, hperm);
                SBD_LAUNCH("sigma_order_kernel(halves)");
                if (kind == 0) {
                    gather_pair_kernel<<<blocks_for(m, 256, 16384), 256, 0, c.stream>>>(hperm, m, t.s_pk, t.s_v64,
                                                                                         t.hs);
                    SBD_LAUNCH("gather_pair_kernel(halves)");
                } else {
                    gather_half_doubles_kernel<<<blocks_for(m, 256, 16384), 256, 0, c.stream>>>(
                        hperm, m, t.d_j, t.d_v64, t.half, t.hdv, t.hdt);
                    SBD_LAUNCH("gather_half_doubles_kernel");
                }
                dfree(c, hperm);
            }
        }
        dfree(c, cnt2);
        dfree(c, ptr2);
    }
}

void build_engine_lists(Ctx &c, int rows)
{
    for (int spin = 0; spin < 2; ++spin) {
        SpinTables &t = c.sp[spin];
        if (t.alias) {
            const SpinTables o = c.sp[0];
            uint64_t *own = t.strings;
            const int parts = t.src_parts, width = t.src_width, deg = t.src_maxdeg;
            uint32_t *item = t.src_item, *ent = t.src_ent;
            int slice[kSrcParts + 1];
            std::copy(t.src_slice, t.src_slice + kSrcParts + 1, slice);
            t = o;
            t.strings = own;
            t.alias = true;
            t.src_parts = parts, t.src_width = width, t.src_maxdeg = deg;
            t.src_item = item, t.src_ent = ent;
            std::copy(slice, slice + kSrcParts + 1, t.src_slice);
            continue;
        }
        if (rows == 0 || rows == 8) build_half_lists(c, t);
        if (rows != 8) build_sig_lists(c, t, 0, t.n, 0, t.n, kValHi, t.sig);
    }
    SBD_CUDA(cudaStreamSynchronize(c.stream));
}

void build_src_lists(Ctx &c, int spin)
{
    SpinTables &t = c.sp[spin];
    const int64_t n = t.n;
    const int norb = c.norb, npair = norb * (norb - 1) / 2;
    const int parts = t.src_parts = src_parts(norb, n, c.smem_optin);
    t.src_width = 1;
    if (!parts) return;  // the two-operand pass runs instead
    t.src_width = std::max(1, (npair + parts - 1) / parts);
    int64_t *cnt = dalloc_n<int64_t>(c, (size_t)n);
    int64_t *ioff = dalloc_n<int64_t>(c, (size_t)parts * (n + 1));
    int *dmax = dalloc_n<int>(c, 1);
    SBD_CUDA(cudaMemsetAsync(dmax, 0, sizeof(int), c.stream));
    int64_t items[kSrcParts] = {0};
    for (int h = 0; h < parts; ++h) {
        src_count_kernel<<<blocks_for(n, 128), 128, 0, c.stream>>>(t.s_ptr, t.s_pk, n, norb, h * t.src_width,
                                                                   (h + 1) * t.src_width, cnt, dmax);
        SBD_LAUNCH("src_count_kernel");
        scan(c, cnt, n, ioff + h * (n + 1));
        SBD_CUDA(cudaMemcpyAsync(&items[h], ioff + h * (n + 1) + n, sizeof(int64_t), cudaMemcpyDeviceToHost, c.stream));
    }
    SBD_CUDA(cudaMemcpyAsync(&t.src_maxdeg, dmax, sizeof(int), cudaMemcpyDeviceToHost, c.stream));
    SBD_CUDA(cudaStreamSynchronize(c.stream));
    t.src_slice[0] = 0;
    for (int h = 0; h < parts; ++h) t.src_slice[h + 1] = t.src_slice[h] + (int)((items[h] + 31) / 32);
    const int64_t nsl = std::max(t.src_slice[parts], 1);
    uint32_t *item = dalloc_n<uint32_t>(c, (size_t)nsl * 32), *ent = dalloc_n<uint32_t>(c, (size_t)nsl * 32 * kSrcItem);
    t.src_item = dalloc_n<uint32_t>(c, (size_t)nsl * 32);
    t.src_ent = dalloc_n<uint32_t>(c, (size_t)nsl * 32 * kSrcItem);
    SBD_CUDA(cudaMemsetAsync(item, 0, (size_t)nsl * 32 * sizeof(uint32_t), c.stream));
    SBD_CUDA(cudaMemsetAsync(ent, 0, (size_t)nsl * 32 * kSrcItem * sizeof(uint32_t), c.stream));
    for (int h = 0; h < parts; ++h) {
        const size_t s0 = (size_t)t.src_slice[h] * 32;
        src_fill_kernel<<<blocks_for(n, 128), 128, 0, c.stream>>>(t.s_ptr, t.s_pk, n, norb, h * t.src_width,
                                                                  (h + 1) * t.src_width, ioff + h * (n + 1), item + s0,
                                                                  ent + s0 * kSrcItem);
        SBD_LAUNCH("src_fill_kernel");
    }
    src_slice_order_kernel<<<blocks_for(nsl * 32, 256), 256, 0, c.stream>>>(item, ent, nsl, t.src_item, t.src_ent);
    SBD_LAUNCH("src_slice_order_kernel");
    src_entry_order_kernel<<<blocks_for(nsl, kEntryWarps), 32 * kEntryWarps, 0, c.stream>>>(t.src_item, t.src_ent, nsl);
    SBD_LAUNCH("src_entry_order_kernel");
    dfree(c, item);
    dfree(c, ent);
    dfree(c, cnt);
    dfree(c, ioff);
    dfree(c, dmax);
}

// Slices of the two-operand alpha-beta pass (SpinTables::sl_*); without `entries`, only the order of the
// strings (in which the column-stationary pass takes its rows).
static void build_slices(Ctx &c, SpinTables &t, bool entries)
{
    const int64_t n = t.n, nsl = (n + 31) / 32;
    uint64_t *keys = dalloc_n<uint64_t>(c, (size_t)n);
    int64_t *len = dalloc_n<int64_t>(c, (size_t)nsl), *off = dalloc_n<int64_t>(c, (size_t)nsl + 1);
    t.sl_col = dalloc_n<int32_t>(c, 32 * (size_t)nsl);
    t.sl_off = dalloc_n<uint32_t>(c, (size_t)nsl + 1);
    slice_key_kernel<<<blocks_for(n, 256), 256, 0, c.stream>>>(t.s_ptr, n, keys);
    SBD_LAUNCH("slice_key_kernel");
    radix_sort_strings(c, keys, n, 16);  // stable, by the low 16 bits: descending length
    slice_col_kernel<<<blocks_for(32 * nsl, 256), 256, 0, c.stream>>>(keys, n, nsl, t.sl_col, len);
    SBD_LAUNCH("slice_col_kernel");
    if (!entries) {
        dfree(c, keys);
        dfree(c, len);
        dfree(c, off);
        return;
    }
    scan(c, len, nsl, off);
    narrow_kernel<<<blocks_for(nsl + 1, 256), 256, 0, c.stream>>>(off, t.sl_off, nsl + 1);
    SBD_LAUNCH("narrow_kernel(slices)");
    int64_t steps = 0;
    SBD_CUDA(cudaMemcpyAsync(&steps, off + nsl, sizeof(int64_t), cudaMemcpyDeviceToHost, c.stream));
    SBD_CUDA(cudaStreamSynchronize(c.stream));
    t.sl_ent = dalloc_n<uint32_t>(c, 32 * (size_t)steps);
    if (steps) {
        slice_fill_kernel<<<blocks_for(32 * nsl, 128, 65535), 128, 0, c.stream>>>(t.s_ptr, t.s_pk, n, c.norb, nsl,
                                                                                t.sl_col, t.sl_off, t.sl_ent);
        SBD_LAUNCH("slice_fill_kernel");
        slice_order_kernel<<<blocks_for(4 * nsl, 1, 65535), 32, 0, c.stream>>>(t.s_ptr, nsl, t.sl_col, t.sl_off, t.sl_ent);
        SBD_LAUNCH("slice_order_kernel");
    }
    dfree(c, keys);
    dfree(c, len);
    dfree(c, off);
}

void build_range_lists(Ctx &c, int spin, bool beta)
{
    SpinTables &t = c.sp[spin];
    RangeLists &r = t.rl;
    const int64_t n = t.n;
    const int wmax = range_width_max(c.smem_optin, c.norb);
    r.ng = (int)((n + wmax - 1) / wmax);
    r.w = (int)((n + r.ng - 1) / r.ng);
    const int64_t groups = part_group(n, kParts), nq = groups * r.ng;
    uint32_t *cd = dalloc_n<uint32_t>(c, (size_t)(n * r.ng)), *cs = dalloc_n<uint32_t>(c, (size_t)(n * r.ng));
    int64_t *cnt = dalloc_n<int64_t>(c, 2 * (size_t)nq);
    int64_t *sum = dalloc_n<int64_t>(c, (size_t)nq + 1);
    r.zi = dalloc_n<int32_t>(c, kListGroup * (size_t)nq);
    r.qd = dalloc_n<uint32_t>(c, (size_t)nq + 1);
    r.qs = dalloc_n<uint32_t>(c, (size_t)nq + 1);
    const int cb = blocks_for(n * r.ng, 256, 16384), qb = blocks_for(nq + 1, 256, 16384);
    range_count_kernel<<<cb, 256, 0, c.stream>>>(t.d_ptr, t.d_j, n, r.w, r.ng, kRangeDoubles, cd);
    range_count_kernel<<<cb, 256, 0, c.stream>>>(t.s_ptr, t.s_j, n, r.w, r.ng, kRangeSingles, cs);
    SBD_LAUNCH("range_count_kernel");
    range_order_kernel<<<r.ng * kParts, 256, 0, c.stream>>>(n, cd, r.zi);
    SBD_LAUNCH("range_order_kernel");
    range_group_kernel<<<qb, 256, 0, c.stream>>>(n, groups, nq, cd, cs, r.zi, cnt, cnt + nq);
    SBD_LAUNCH("range_group_kernel");
    int64_t total[2] = {0, 0};
    for (int kind = 0; kind < 2; ++kind) {
        scan(c, kind == 0 ? cnt + nq : cnt, nq, sum);
        narrow_kernel<<<qb, 256, 0, c.stream>>>(sum, kind == 0 ? r.qs : r.qd, nq + 1);
        SBD_LAUNCH("narrow_kernel");
        SBD_CUDA(cudaMemcpyAsync(&total[kind], sum + nq, sizeof(int64_t), cudaMemcpyDeviceToHost, c.stream));
    }
    // the orbital pairs that the singles need J of (few of them in a sparse set of many orbitals)
    const int npair = c.norb * (c.norb - 1) / 2;
    int *used = dalloc_n<int>(c, (size_t)npair), *list = dalloc_n<int>(c, (size_t)npair + 1);
    SBD_CUDA(cudaMemsetAsync(used, 0, sizeof(int) * (size_t)npair, c.stream));
    pair_mark_kernel<<<blocks_for(t.ns, 256, 2048), 256, 0, c.stream>>>(t.s_pk, t.ns, c.norb, used);
    SBD_LAUNCH("pair_mark_kernel");
    pair_list_kernel<<<1, 1024, 0, c.stream>>>(used, npair, list, list + npair);
    SBD_LAUNCH("pair_list_kernel");
    SBD_CUDA(cudaMemcpyAsync(&r.np, list + npair, sizeof(int), cudaMemcpyDeviceToHost, c.stream));
    SBD_CUDA(cudaStreamSynchronize(c.stream));
    r.pad = range_pad(c.smem_optin, c.norb, r.w, r.np);
    const size_t ms = (size_t)total[0] * kListGroup * kRangeSingles, md = (size_t)total[1] * kListGroup * kRangeDoubles;
    if (total[0] > 0xffffffffLL || total[1] > 0xffffffffLL) fail(SBD_ERR_UNSUPPORTED, "excitation lists too large");
    r.sm = dalloc_n<uint32_t>(c, ms);
    r.shi = dalloc_n<float>(c, ms);
    r.slo = dalloc_n<float>(c, ms);
    r.sv64 = c.job ? nullptr : dalloc_n<double>(c, ms);
    r.dt = dalloc_n<uint16_t>(c, md);
    r.dhi = dalloc_n<float>(c, md);
    r.dlo = dalloc_n<float>(c, md);
    r.dv64 = c.job ? nullptr : dalloc_n<double>(c, md);
    const int fb = blocks_for(nq * kListGroup * 32, 256, 16384);
    if (ms) {
        range_fill_kernel<1><<<fb, 256, 0, c.stream>>>(t.s_ptr, t.s_j, t.s_pk, t.s_v64, groups, c.norb, used, r);
        SBD_LAUNCH("range_fill_kernel(singles)");
    }
    if (md) {
        range_fill_kernel<2><<<fb, 256, 0, c.stream>>>(t.d_ptr, t.d_j, nullptr, t.d_v64, groups, c.norb, nullptr, r);
        SBD_LAUNCH("range_fill_kernel(doubles)");
    }
    build_slices(c, t, beta);
    const SpinTables &o = c.sp[1 - spin];
    r.jg = dalloc_n<double>(c, (size_t)r.np * o.n);
    if (r.np) {
        const dim3 jb((unsigned)blocks_for(o.n, 256, 1024), (unsigned)std::min(r.np, 256));
        pair_j_kernel<<<jb, 256, 0, c.stream>>>(o.strings, o.n, c.norb, c.eri64, list, r.np, r.jg);
        SBD_LAUNCH("pair_j_kernel");
    }
    dfree(c, used);
    dfree(c, list);
    dfree(c, cd);
    dfree(c, cs);
    dfree(c, cnt);
    dfree(c, sum);
}

void pack_integrals(Ctx &c)
{
    const int npair = c.norb * (c.norb - 1) / 2;
    c.eri32 = dalloc_n<float>(c, (size_t)npair * npair);
    if (!npair) return;
    pack_integrals_kernel<<<npair, 64, 0, c.stream>>>(c.eri64, c.norb, c.eri32);
    SBD_LAUNCH("pack_integrals_kernel");
}

void build_diagonal(Ctx &c)
{
    c.hd = dalloc_n<double>(c, (size_t)c.N);
    int grid = (int)(c.nA < 65535 ? c.nA : 65535);
    hdiag_kernel<<<grid, 256, 0, c.stream>>>(c.sp[0].strings, c.sp[1].strings, c.sp[0].ediag, c.sp[1].ediag,
                                             c.eri64, c.norb, c.nA, c.nB, c.hd);
    SBD_LAUNCH("hdiag_kernel");
}

}  // namespace sbd

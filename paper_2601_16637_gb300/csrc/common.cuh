// Internal declarations of the SBD CUDA library (not part of the C ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "sbd.h"

namespace sbd {

// ---------------------------------------------------------------------------
// errors: thrown inside the library, converted to status codes at the ABI

struct Error {
    int code;
    std::string msg;
};

[[noreturn]] void fail(int code, const std::string &msg);
void set_thread_error(const std::string &msg);  // sbd_last_error(NULL) on this thread
void check_cuda(cudaError_t e, const char *what, const char *file, int line);
void count_launch();
#define SBD_CUDA(call) ::sbd::check_cuda((call), #call, __FILE__, __LINE__)
#define SBD_LAUNCH(what) (::sbd::count_launch(), ::sbd::check_cuda(cudaGetLastError(), what, __FILE__, __LINE__))

// Packed single-excitation entry: target j in bits 0-17, phase -1 in bit 18, code p*norb+q in
// bits 19-30, so pk >> 18 = 2*code + (phase < 0) indexes sign-folded coefficient tables.  A
// single always has p != q, so code 0 never occurs: pk = 0 is the padding entry, and the
// coefficient-table rows of code 0 are kept zero.  Strings per spin must stay below 2^18.
constexpr int kPackJBits = 18;
constexpr uint32_t kPackJMask = (1u << kPackJBits) - 1u;
constexpr int kPackKeyShift = 18;  // pk >> 18 = 2*code + neg
constexpr int64_t kMaxStringsPerSpin = (int64_t)1 << kPackJBits;
constexpr int kSrcPairShift = 18;  // source-major singles: orbital-pair index at bits 18-28
constexpr int kSrcNegBit = 29;     // and the phase at bit 29
constexpr int kSrcItem = 8;        // source-major singles per work item
constexpr int kSrcParts = 8;      // most parts the orbital pairs of the alpha-beta pass are cut into
constexpr int kBankGroups = 8;     // 16-byte bank groups of shared memory (32 banks x 4 bytes)
constexpr int kListPad = 4;        // sigma lists are padded to multiples of 4 entries (16-byte loads)

// ---------------------------------------------------------------------------
// device status words written by validation kernels

struct DevStatus {
    unsigned long long first_bad;  // smallest index of a malformed string (~0 if none)
    unsigned long long first_dup;  // smallest index i with sorted[i] == sorted[i-1]
    int nonfinite;                 // nonzero if h or eri hold NaN/Inf
    int differ;                    // nonzero if two sorted sets differ
};

// ---------------------------------------------------------------------------
// per-spin tables, all device memory

// Same-spin excitation lists of one string set as the row passes read them (range_rows.cuh).  The
// targets are cut into ng ranges of w strings (the part of C that a CTA stages at a time).  The
// strings are dealt to kParts parts (part = string mod kParts); inside a range the parts follow each
// other, and inside a part the lists descend in length and are taken kListGroup at a time.  Such a
// group is what a warp walks side by side, so its lists are padded to the longest of them and stored
// interleaved, block by block: a warp's load of one block of all its lists is one contiguous piece.
// Padding entries have value zero and the target `pad`, a staged line of zeros: an amplitude that is no
// number must not reach the sum of a string that it is not connected to (0 x inf is no zero).
constexpr int kParts = 16;
constexpr int kRangeDoubles = 4;  // entries of one list in a block of doubles
constexpr int kRangeSingles = 2;  // and in a block of singles
constexpr int kListGroup = 8;     // lists of a group
constexpr int32_t kListHas = 1 << 30;  // the string's list has entries in this range
struct RangeLists {
    int w = 0, ng = 0, pad = 0;
    int32_t *zi = nullptr;                     // [ng*groups*8] string | kListHas, or -1 (no string)
    uint32_t *qd = nullptr, *qs = nullptr;     // [ng*groups + 1] first block of a group's doubles, singles
    uint16_t *dt = nullptr;                    // doubles: target inside the range
    float *dhi = nullptr, *dlo = nullptr;      // and matrix element: its FP32 rounding, FP32 of the remainder,
    double *dv64 = nullptr;                    // FP64 (mixed products read the first, pair products two)
    uint32_t *sm = nullptr;  // singles: target inside the range | used pair << 16 | phase -1 << 31
    float *shi = nullptr, *slo = nullptr;
    double *sv64 = nullptr;
    // the orbital pairs {r, s} that occur in the singles, and for the strings i of the other spin
    // J_i[rs] = sum_{k in i} (rs|kk), [np][other n]
    int np = 0;
    double *jg = nullptr;
};
// first group of part p (p = kParts: groups of a range) for n strings
__host__ __device__ __forceinline__ int64_t part_group(int64_t n, int p)
{
    const int64_t a = n / kParts, rest = n % kParts;  // parts below `rest` hold a + 1 strings, the others a
    const int64_t big = a / kListGroup + 1, small = (a + kListGroup - 1) / kListGroup;
    return p < rest ? p * big : rest * big + (p - rest) * small;
}

// Copies of the same-spin lists in the order that the passes over whole staged rows read them (row-block
// products, engine jobs): each list is padded with zero entries to a multiple of kListPad and
// reordered so that the 8 entries one 128-bit shared-memory phase gathers have distinct targets modulo 8
// where possible (kBankGroups).  Values are held as `mask` says.
enum { kValHi = 1, kValLo = 2, kValF64 = 4 };  // FP32 rounding, FP32 of the remainder, FP64
struct SigLists {
    int mask = 0;                                // 0: not built
    int64_t *s_ptr = nullptr, *d_ptr = nullptr;  // [rows + 1], padded CSR offsets
    int64_t ns = 0, nd = 0;
    uint32_t *s_pk = nullptr;  // packed single (SpinTables::s_pk)
    int32_t *d_j = nullptr;    // target of a double
    float *s_hi = nullptr, *s_lo = nullptr, *d_hi = nullptr, *d_lo = nullptr;
    double *s_v = nullptr, *d_v = nullptr;
};

// index of the unordered orbital pair {p, q}
__host__ __device__ __forceinline__ int orbital_pair(int p, int q)
{
    const int r = p > q ? p : q, s = p > q ? q : p;
    return r * (r - 1) / 2 + s;
}

struct SpinTables {
    int nel = 0;                 // electrons of this spin
    int64_t n = 0;               // |S|
    uint64_t *strings = nullptr; // sorted ascending
    // canonical CSR excitation tables (kind 1 singles, kind 2 doubles)
    int64_t *s_ptr = nullptr, *d_ptr = nullptr;  // [n+1]
    int64_t ns = 0, nd = 0;                      // total entries
    int32_t *s_j = nullptr, *d_j = nullptr;      // target index
    // packed single: target j (bits 0-17) | code p*norb+q (bits 18-29) | phase -1 (bit 30)
    uint32_t *s_pk = nullptr;
    double *s_v64 = nullptr, *d_v64 = nullptr;   // same-spin matrix elements
    SigLists sig;  // of the whole set: for engine jobs, and of the beta spin for block plans
    // Engine jobs: the mixed row passes' lists split at the middle of the string set (half = (n + 1) / 2):
    // virtual list 2i holds the entries of source i with target < half, list 2i + 1 those with target
    // >= half, each padded to kListPad and in sigma order.
    int64_t half = 0;
    int64_t *hs_ptr = nullptr, *hd_ptr = nullptr;  // [2n + 1]
    uint2 *hs = nullptr;  // (packed single, FP32 value bits)
    // doubles as two arrays with the same entry index: FP32 values, and targets relative to the
    // list's column half, which fit 16 bits: the split lists are built only for half <= 65536
    float *hdv = nullptr;
    uint16_t *hdt = nullptr;
    // Singles for the two-operand alpha-beta pass, one lane per string: the strings in descending order
    // of their number of singles (ties ascending), cut into slices of 32; a slice holds as many steps as
    // its longest list, entry t of lane l at sl_ent[(sl_off[slice] + t)*32 + l].  An entry is the target
    // (bits 0-17) and the coefficient row 2*pair + (phase < 0) at bits 18-29; padding has the target n,
    // a column of zeros, and the row 2*npair, which is zero too.  Inside a list the entries are ordered so that the 8
    // lanes of a 128-bit phase read distinct targets and rows modulo 8 where they can.
    int32_t *sl_col = nullptr;   // [slices*32] string, -1: none or no singles
    uint32_t *sl_off = nullptr;  // [slices + 1]
    uint32_t *sl_ent = nullptr;
    RangeLists rl;  // same-spin lists of the row passes
    // Source-major singles for the column-stationary alpha-beta pass, of the spin that is the beta spin
    // of the pass.  The orbital pairs {p, q} are cut into src_parts ranges of src_width pairs (one where
    // the pass' table of all pairs fits shared memory).  For each part, the canonical singles list
    // of each string, restricted to the part's pairs, is cut into items of at most kSrcItem entries
    // (strings in ascending order,
    // each string's items consecutive, then inside each slice of 32 items the full ones first and
    // the partial ones by decreasing length), so that the lanes of a warp, one item each, walk
    // lists of nearly equal length; part h has the slices [src_slice[h], src_slice[h + 1]);
    // item t = string | entries << 18 (src_item[t]); entry i of item t is
    // src_ent[(t / 32) * 32 * kSrcItem + 32 * i + t % 32] (coalesced for the 32 items of a warp):
    // target (bits 0-17) | index of the pair inside its part (bits 18-28) | phase -1 (bit 29).
    uint32_t *src_item = nullptr;
    uint32_t *src_ent = nullptr;
    int src_parts = 0, src_width = 0;  // 0: the pass does not fit for this many strings
    int src_slice[kSrcParts + 1] = {0};
    int src_maxdeg = 0;          // largest singles count of a string
    double *ediag = nullptr;     // [n] same-spin diagonal energies
    bool alias = false;          // storage owned by the other spin (A == B)
};

struct Ctx {
    int device = 0;
    cudaStream_t stream = nullptr;
    sbd_options opt{};
    bool job = false;  // an engine job: mixed products over whole staged rows, pair products for the check
    int norb = 0, na = 0, nb = 0;
    int64_t nA = 0, nB = 0, N = 0;
    double *h64 = nullptr, *eri64 = nullptr;
    float *eri32 = nullptr;  // (pq|rs) of orbital pairs p > q, r > s, [npair][npair], pair p(p-1)/2 + q
    SpinTables sp[2];
    double *hd = nullptr;   // [N] Hamiltonian diagonal
    void *work_t = nullptr; // [N] doubles: the beta pass' transposed result
    float *rowmax = nullptr; // [nA] max |c(ia, :)| of the last mixed-precision vector (written by its beta pass)
    float eri_absmax = 0.f;  // max |(pq|rs)| of the FP32 integrals
    size_t bytes_held = 0;
    std::vector<std::pair<void *, size_t>> allocs;
    std::string last_error;
    DevStatus *dstat = nullptr;  // device
    int smem_optin = 0;          // max dynamic shared memory per block
    int num_sms = 0;
    // kernel timing (sbd_options.timing)
    struct Pending {
        int slot;
        cudaEvent_t a, b;
    };
    std::vector<Pending> pending;
    std::vector<cudaEvent_t> event_pool;
    double kernel_ms[12] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
    int64_t kernel_n[12] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
};

// the context inside a C-ABI handle (api.cu)
Ctx &ctx_of(sbd_handle h);
// sbd_create; job: see Ctx
int create_handle(sbd_handle *out, int norb, int nalpha, int nbeta, const double *h, const double *eri, const uint64_t *A,
                  int64_t nA, const uint64_t *B, int64_t nB, const sbd_options *opt, void *stream, bool job);

// kernel timing helpers (api.cu)
cudaEvent_t take_event(Ctx &c);
void harvest_timing(Ctx &c);

// device memory through the handle's allocator, with budget accounting
void *dalloc(Ctx &c, size_t bytes);
void dfree(Ctx &c, void *p);
template <typename T>
T *dalloc_n(Ctx &c, size_t n)
{
    return static_cast<T *>(dalloc(c, n * sizeof(T) > 0 ? n * sizeof(T) : 16));
}

// ---------------------------------------------------------------------------
// Diagonal preconditioner of Davidson (paper Eq. 7): t = r / (sign(d) max(|d|, delta)),
// d = Hd - theta.  The factor multiplying r is formed as an FP32 reciprocal: a preconditioner only
// shapes the correction direction (which is then orthogonalised and normalised in FP64), and the
// FP64 division would cost the FP64 pipe as much as a fifth of the Ritz pass.
__device__ __forceinline__ double precond_factor(double d, double delta)
{
    const double den = (d >= 0.0 ? 1.0 : -1.0) * fmax(fabs(d), delta);
    return (double)__frcp_rn((float)den);
}

// ---------------------------------------------------------------------------
// warp-cooperative search, shared by the lookup entry point and the table builder

// Position of `key` in sorted[0, n), or -1.  All 32 lanes call it with the
// same key; each step samples 32 evenly spaced elements of the remaining
// range and narrows it to one gap between samples (a 32-ary search).
__device__ __forceinline__ int64_t warp_find(const uint64_t *__restrict__ sorted, int64_t n, uint64_t key)
{
    const int lane = threadIdx.x & 31;
    int64_t lo = 0, hi = n;  // first element >= key lies in [lo, hi]
    while (hi - lo > 32) {
        const int64_t step = (hi - lo + 31) / 32;
        const int64_t pos = lo + lane * step;
        const bool below = pos < hi && __ldg(sorted + pos) < key;
        const int c = __popc(__ballot_sync(0xffffffffu, below));
        const int64_t nlo = c == 0 ? lo : lo + (int64_t)(c - 1) * step + 1;
        const int64_t nhi = min(hi, lo + (int64_t)c * step + 1);
        lo = nlo;
        hi = nhi;
    }
    const int64_t pos = lo + lane;
    const bool hit = pos < hi && pos < n && __ldg(sorted + pos) == key;
    const unsigned m = __ballot_sync(0xffffffffu, hit);
    return m ? lo + (__ffs(m) - 1) : -1;
}

// ---------------------------------------------------------------------------
// launchers (each enqueues on c.stream unless a stream is given)

// strings.cu
void validate_strings(Ctx &c, const uint64_t *s, int64_t n, int norb, int nel);
void radix_sort_strings(Ctx &c, uint64_t *keys, int64_t n, int nbits);
void check_duplicates(Ctx &c, const uint64_t *sorted, int64_t n);
void compare_sets(Ctx &c, const uint64_t *a, const uint64_t *b, int64_t n);
void check_finite(Ctx &c, const double *x, int64_t n);
void lookup_strings(const uint64_t *sorted, int64_t n, const uint64_t *keys, int64_t nq, int64_t *idx,
                    cudaStream_t s);
void sort_validate_into(const uint64_t *in, int64_t n, int norb, int nel, uint64_t *out, uint64_t *tmp,
                        DevStatus *st, cudaStream_t s);

// tables.cu
void build_tables(Ctx &c, int spin);
// beta: also what the alpha-beta passes read of their beta spin
void build_range_lists(Ctx &c, int spin, bool beta);
// copies of the lists of rows [r0, r0 + nr) with targets in [j0, j1), renumbered from j0; where `out` is built
// already, the values of `mask` that it lacks
void build_sig_lists(Ctx &c, const SpinTables &t, int64_t r0, int64_t nr, int64_t j0, int64_t j1, int mask, SigLists &out);
// lists of the engine's mixed row passes with `rows` rows per item (0: any)
void build_engine_lists(Ctx &c, int rows);
void build_diagonal(Ctx &c);
// orbitals (4 per entry) and phases of a spin's singles or doubles, worked out from the strings into host memory
void table_moves(const Ctx &c, int spin, bool singles, uint8_t *orbs_host, int8_t *sign_host);
void pack_integrals(Ctx &c);  // eri32 from eri64
void to_float(const double *in, float *out, int64_t n, cudaStream_t s);

// sigma.cu
void sigma_prepare(Ctx &c);
// parts the orbital pairs are cut into by the column-stationary alpha-beta pass for n beta strings
// (0: does not fit), within the shared memory of the device
int src_parts(int norb, int64_t n, int smem_optin);
void build_src_lists(Ctx &c, int spin);

// ---------------------------------------------------------------------------
// row-block sigma for alpha-row sharding (shard.cu, sigma.cu)

// The alpha lists of output rows [r0, r1) restricted to sources in [j0, j1), targets renumbered
// from j0: canonical singles, and padded singles and doubles in the arithmetics of sig.mask.
struct BlockPlan {
    Ctx *c = nullptr;
    int64_t r0 = 0, r1 = 0, j0 = 0, j1 = 0;
    int64_t *s_ptr = nullptr;
    uint32_t *s_pk = nullptr;
    SigLists sig;
    void *work_t = nullptr;  // [nB][j1 - j0] doubles: the transposed source block
    float *rowmax = nullptr; // [j1 - j0] max |c| of each source row (mixed alpha-beta pass)
    std::vector<void *> allocs;
};
// mask: values of the arithmetics that the plan is for (value_mask)
BlockPlan *block_plan_create(Ctx &c, int64_t r0, int64_t r1, int64_t j0, int64_t j1, int mask);
inline int value_mask(sbd_precision p) { return p == SBD_MIXED ? kValHi : p == SBD_F32X2 ? kValHi | kValLo : kValF64; }
void block_plan_destroy(BlockPlan *p);
// sigma_rows[(ia - r0)*nB + ib] += sum over (ja, jb), ja in [j0, j1), of H[(ia,ib),(ja,jb)] cblock[(ja - j0)*nB + jb]
// x64_rows (optional, mixed precision): FP64 amplitudes of the output rows, for the diagonal term
void sigma_block_apply(BlockPlan &p, const void *cblock, double *sigma_rows, sbd_precision prec, cudaStream_t s,
                       const double *x64_rows = nullptr);

// ---------------------------------------------------------------------------
// batched sigma: many instances in one set of persistent launches (sigma.cu)

// One instance of a batched sigma (host side).
struct SigmaSlot {
    const Ctx *c;
    const void *x;       // amplitudes [nA][nB]: float (mixed) or double (FP64)
    double *y;           // sigma [nA][nB], overwritten; scratch until the last pass, must not overlap x or x64
    const double *x64;   // mixed only: FP64 amplitudes for the diagonal term, or null
    void *xt;            // work space of nA*nB doubles: the beta pass' transposed result, or (passes over whole
                         // staged rows) the transposed amplitudes
};
struct SigmaBatch;
// Device descriptors for up to max_slots instances whose string sets have at most max_strings
// entries per spin and norb <= max_norb; R = rows staged per work item (1, 2, or for the mixed
// precision 4, or 8 over column halves).
// rows: mixed row passes over whole staged rows, R per work item (the handles need build_engine_lists)
SigmaBatch *sigma_batch_create(int max_slots, sbd_precision prec, int R, int max_strings, int max_norb, int device,
                               bool rows = false);
// Shared memory one work item needs with R staged rows; compare with sigma_batch_smem_limit().
size_t sigma_batch_smem(sbd_precision prec, int R, int max_strings, int max_norb);
size_t sigma_batch_smem_limit(int device);
// whether R rows per item (8: mixed only, over column halves, with the column-stationary alpha-beta
// pass) fits shared memory for max_strings and max_norb
bool sigma_batch_fits(sbd_precision prec, int R, int max_strings, int max_norb, int device);
// Fills the host staging copy of the descriptors (no device work).
void sigma_batch_set(SigmaBatch *b, const SigmaSlot *slots, int n);
// Copies the staged descriptors to the device and runs transpose, beta, alpha and alpha-beta
// passes over every slot: fixed grids and device-resident counts, so the sequence can be
// captured in a CUDA graph once and replayed after each sigma_batch_set.
void sigma_batch_launch(SigmaBatch *b, cudaStream_t s);
void sigma_batch_destroy(SigmaBatch *b);
// c64 (mixed only, may be NULL): the FP64 amplitudes, used for the diagonal term
void sigma_apply(Ctx &c, const void *cvec, double *svec, sbd_precision prec, cudaStream_t s,
                 const double *c64 = nullptr);

// davidson.cu
// A rank of an alpha-row-sharded solve: its rows [bounds[rank], bounds[rank+1]) of every vector,
// one block plan per source block, two ring buffers and the caller's communication callbacks.
struct ShardCtx {
    int rank = 0, world = 1;
    std::vector<int64_t> bounds;    // world + 1 alpha-row boundaries
    std::vector<BlockPlan *> plans; // plans[b]: this rank's rows, source block b
    void *ring[2] = {nullptr, nullptr};
    sbd_comm comm{};
    int64_t row0() const { return bounds[rank]; }
    int64_t rows() const { return bounds[rank + 1] - bounds[rank]; }
};

int davidson(Ctx &c, int nroots, double tol, sbd_precision prec, double *energies, double *vecs,
             double *resid, sbd_report *rep, ShardCtx *shard = nullptr);
// sigma of this rank's rows: the source blocks pass around the ring of ranks (shard.cu)
void ring_sigma(ShardCtx &sh, Ctx &c, const void *x_rows, double *y_rows, sbd_precision prec, cudaStream_t s,
                const double *x64_rows = nullptr);

}  // namespace sbd

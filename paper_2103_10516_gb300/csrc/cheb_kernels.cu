// Chebyshev moment engine: a block of Rademacher probes pushed through the
// three-term recurrence V_{k+1} = 2 At V_k - V_{k-1} (Section 2.2,
// Eq. recurrence), At = alpha A + beta I, with the per-probe dot products that
// give the moments fused into the same pass over the matrix.
//
// Data layout (device, row-major): V[i * ldv + c] is entry i of probe c, so a
// gathered row of V is ldv contiguous values and each probe's column is strided.
// Probes are sorted by degree, descending; at step k only the first act_k
// columns are live, so retired probes cost nothing.
//
// Doubling mode (the symmetric quadratic-form trick the paper cites in
// Section 2.2): with T_{2k} = 2 T_k^2 - 1 and T_{2k+1} = 2 T_{k+1} T_k - T_1,
//   mu_{2k+2} = 2 V_{k+1}.V_{k+1} - mu_0,   mu_{2k+1} = 2 V_{k+1}.V_k - mu_1,
// so degree n needs ceil(n/2) operator applications.  Direct mode keeps
// mu_{k+1} = z . V_{k+1} (n applications).
//
// Work split (plan.cu; fixed per matrix, so every result is reproducible): rows
// cost kPlanRowCost units plus one per entry; the unit axis is cut into chunks
// of Uc units.  A row of degree <= Ul (>= Uc) belongs to the chunk holding its
// first unit.  Longer rows are cut into fixed segments of Ul entries whose
// partial products go to a scratch table; a second kernel adds each row's
// segments in order and applies the recurrence there.  Work items are dealt
// round-robin to groups of G lanes on a grid no larger than the resident one; a
// group always owns the same columns.  An item is a chunk, a few rows a group
// (row_items), or a chunk a group with rows in step (ordered_items), then the
// segments; items are small (about a thousand chunks per SM), so at any moment
// the groups work on one narrow band of rows and the rows of V gathered by
// neighbouring rows are still in L2.
//
// Reductions are deterministic: each CTA merges its groups' sums in a fixed
// tree and writes per-column partial sums, and a separate kernel adds the CTA
// partials in CTA order.  Each thread's running dot products are FP64 for FP64
// vectors.  For FP32 vectors they are compensated (Kahan) FP32 sums, whose
// error is at most 2^-23 times the sum of |terms| (below the rounding already
// in the FP32 vectors), because FP64 arithmetic on GB300 runs at 1/64 of the
// FP32 rate and a per-row FP64 update would cost more than streaming the
// vectors; a CTA merges them as double-float pairs, and double-float sums to the
// precision of FP64 (see Merge); from the CTA partials on everything is FP64.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>
#include <vector>

#include "df64.cuh"
#include "mlt_internal.h"
#include "rng.cuh"


namespace mlt {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kFp32Blocks = 5;      // CTAs per SM over which FP32 steps deal their chunks (see ordered_items)
constexpr int64_t kRowsPerGroup = 8, kUnitsPerGroup = 96;   // a narrow group's share of a work item
constexpr int64_t kLargePattern = 4000000;   // entries from which narrower pattern steps walk (see walks)
constexpr int64_t kDependentWork = 16000000;   // see pdl_trigger
constexpr int kNarrowBatch = 8;     // entries a lane of a narrow group takes at a time
constexpr int kSlots = 16;          // steps whose partials are buffered before a reduction

// Programmatic dependent launch (PTX griddepcontrol).  On small operators a
// step takes a few microseconds, of which the launch and the kernel's set-up
// are a third.  A step kernel therefore lets the next kernel of the group start
// when its rows are done, while it reduces its dot products; the next kernel
// sets itself up and waits for it to complete (pdl_wait) before it reads or
// writes anything but its parameters and shared memory.  Used when a launch
// handles at most kDependentWork row slices (launch_step_g): the log-det of
// the 64^2 grid took 828 -> 738 us, the 48^3 host estimate 5.78 -> 5.71 ms
// (thresholds of 1 and 4 million: 761 and 749 us), while on large operators the
// same launches measured 1.3% (100^3 stencil) and 5% (scale-20 R-MAT) slower,
// and letting the next kernel start earlier, before the rows are done, 6%
// slower on the grid as well.
//
// A kernel launched this way is resident while the one before it still writes
// its results, so those are not read-only for its lifetime: it must not take
// them through a const __restrict__ parameter or __ldg, whose loads may use
// the non-coherent path, which the wait does not order.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename... P, typename... A>
cudaError_t launch_dependent(bool dependent, void (*kernel)(P...), dim3 grid, int threads, cudaStream_t s, A... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.stream = s;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = dependent ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

template <typename T> struct Lanes;
template <> struct Lanes<double> { static constexpr int N = 2; };   // 16-byte vectors
template <> struct Lanes<float> { static constexpr int N = 4; };
template <> struct Lanes<df64> { static constexpr int N = 2; };     // 16-byte vectors of pairs

// A lane's 16-byte slice of a vector row.  Double-float slices hold the high
// parts of their two entries, then the two low parts, so that a slice loads as
// two packed FP32 pairs (see the f32x2 operations below).
template <typename T, int N> struct alignas(sizeof(T) * N) Pack {
    T v[N];
    __device__ __forceinline__ T get(int q) const { return v[q]; }
    __device__ __forceinline__ void set(int q, T x) { v[q] = x; }
};
template <> struct alignas(16) Pack<df64, 2> {
    float h[2], l[2];
    __device__ __forceinline__ df64 get(int q) const { return df64(h[q], l[q]); }
    __device__ __forceinline__ void set(int q, df64 x) { h[q] = x.hi; l[q] = x.lo; }
};

// Per vector type: the resident CTAs per SM the step kernel is compiled for
// (C), the unroll depth of its gather loop (U), whether its gathers carry an
// L2 evict-last policy (E), whether long-row segments are dealt out in
// column-window order (W, see plan.cu), predicated gather blocks (PR),
// the column-index prefetch on pattern matrices (PF) and the widest group that
// takes row_product_narrow (NG).  More unrolled gathers keep more row
// reads outstanding but need registers, which lowers the resident CTAs; the
// evict-last policy keeps the gathered V_k rows in L2 against the streams of
// V_{k-1}, V_{k+1} and the column indices.  Measured on the scale-22 R-MAT
// graph (gather-bound) and the 100^3 diffusion operator (streaming): FP32 and
// FP64 gain from the deeper unroll (FP32 9.5 -> 8.1 ms a step on the graph)
// and FP32 from the policy (8.1 -> 7.5 ms).  The double-float step on packed
// pairs (row_sum_df2, epilogue_df2) needs few enough registers for eight
// unrolled gathers at five CTAs: 8.4 -> 7.2 ms on the graph, against 8.3 at
// six CTAs and unroll 8 and 8.1 at five and unroll 12 (3% slower on the
// streaming operator).  The column-window order takes FP32 and double-float
// steps on the graph 3-4% lower and the FP64 step, bound by FP64 arithmetic,
// 2% higher.
//
// PR shapes the gather loop for rows whose length is not a multiple of the
// unroll depth: predicated gathers go in blocks of
// unroll-depth slots, each slot switched off past the row's end, so that a
// short row's gathers are all in flight together; without PR the compiler's
// remainder loop takes them one at a time.  Predicated blocks took the FP32
// step on the 100^3 diffusion operator (7 entries a row) from 0.569 to
// 0.516 ms and the Gram operator's X^T step from 0.201 to 0.182 ms, left FP32
// on the graph unchanged (6.18 -> 6.14 ms), and slowed the double-float and
// FP64 steps by 2-9%.  They apply to groups of at least unroll-depth lanes:
// a narrower group (few live probes) takes at most G entries a batch, and a
// block of mostly idle slots cost the learned estimator's FP32 moments, whose
// last steps run 1-2 live probes, 16% of their time.
//
// PF: on pattern matrices, a batch's column indices are loaded one batch
// ahead, so that their latency overlaps the previous batch's gathers.  That
// took the FP32 step on the graph from 6.12 to 5.87 ms; the double-float step
// went from 7.17 to 7.60 ms and FP64 1% slower, and on valued FP32 matrices
// (stencil, Gram) it lost 1-5%, so it is on for FP32 patterns only.
template <int C, int U, bool E, bool W, bool PR, bool PF, int NG> struct TuneOf {
    static constexpr int kNarrow = NG;
    static constexpr int kCtas = C, kUnroll = U;
    static constexpr bool kEvictLast = E, kWindowSegs = W, kPredicated = PR, kPrefetchPattern = PF;
};
template <typename T> struct StepTuning;
template <> struct StepTuning<float> : TuneOf<5, 8, true, true, true, true, 4> {};
template <> struct StepTuning<double> : TuneOf<4, 8, false, false, false, false, 2> {};
template <> struct StepTuning<df64> : TuneOf<5, 8, false, true, false, false, 4> {};

// An L2 access policy that marks lines evict-last (createpolicy, PTX ISA).
__device__ __forceinline__ uint64_t evict_last_policy()
{
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}

// A gathered 16-byte row slice, under the L2 policy `pol` when E.
template <bool E, typename P>
__device__ __forceinline__ P ld_gather(const P* p, uint64_t pol)
{
    static_assert(sizeof(P) == 16, "16-byte packs");
    if constexpr (E) {
        uint4 u;
        asm volatile("ld.global.L2::cache_hint.v4.u32 {%0,%1,%2,%3}, [%4], %5;"
                     : "=r"(u.x), "=r"(u.y), "=r"(u.z), "=r"(u.w)
                     : "l"(p), "l"(pol));
        P r;
        memcpy(&r, &u, 16);
        return r;
    } else {
        (void)pol;
        return *p;
    }
}

// The same 16-byte load as two 64-bit words (the operands of packed pair
// arithmetic).
template <bool E>
__device__ __forceinline__ ulonglong2 ld_gather2(const void* p, uint64_t pol)
{
    if constexpr (E) {
        ulonglong2 u;
        asm volatile("ld.global.L2::cache_hint.v2.u64 {%0,%1}, [%2], %3;"
                     : "=l"(u.x), "=l"(u.y)
                     : "l"(p), "l"(pol));
        return u;
    } else {
        (void)pol;
        return *reinterpret_cast<const ulonglong2*>(p);
    }
}

// A thread's running dot product.  The kernels keep these in shared memory
// (one slot per thread, see DotSlots): held in registers beside a row's
// gathers they pushed the step kernel past the six-CTA register budget, and
// the spilled copies went through L1 to L2.
template <typename T> struct DotAcc;
template <> struct DotAcc<double> {
    double s;
    __device__ __forceinline__ void clear() { s = 0.0; }
    __device__ __forceinline__ void add_prod(double a, double b) { s = fma(a, b, s); }
    __device__ __forceinline__ void add(double x) { s += x; }
};
template <> struct DotAcc<float> {
    float s, c;   // Kahan: s - c is the running sum
    __device__ __forceinline__ void clear() { s = c = 0.0f; }
    __device__ __forceinline__ void add(float x)
    {
        const float y = x - c;
        const float t = s + y;
        c = (t - s) - y;
        s = t;
    }
    __device__ __forceinline__ void add_prod(float a, float b)
    {
        const float y = fmaf(a, b, -c);   // the product enters unrounded
        const float t = s + y;
        c = (t - s) - y;
        s = t;
    }
};
template <> struct DotAcc<df64> {
    df64 s;
    __device__ __forceinline__ void clear() { s = df64(0); }
    __device__ __forceinline__ void add_prod(df64 a, df64 b) { s = a * b + s; }
    __device__ __forceinline__ void add(df64 x) { s = s + x; }
};

// The CTA's running dots: kind [0] V_{k+1}.V_{k+1} (unused in direct mode),
// [1] V_{k+1}.V_k or z.V_{k+1}, for the thread's columns c0 + q.  Each thread
// only touches its own slots, and a warp's accesses are consecutive.
template <typename T>
struct DotSlots {
    DotAcc<T> d[2][Lanes<T>::N][kThreads];
    __device__ __forceinline__ DotAcc<T> load(int kind, int q, int t) const { return d[kind][q][t]; }
    __device__ __forceinline__ void store(int kind, int q, int t, DotAcc<T> x) { d[kind][q][t] = x; }
};
// FP32: the Kahan sums of columns (c0, c0 + 1) and (c0 + 2, c0 + 3) as packed
// pairs, (sums, compensations), so that epilogue_f2 updates two columns with
// each packed instruction.
template <>
struct DotSlots<float> {
    ulonglong2 d[2][2][kThreads];
    __device__ __forceinline__ DotAcc<float> load(int kind, int q, int t) const
    {
        const ulonglong2 v = d[kind][q >> 1][t];
        DotAcc<float> x;
        x.s = (q & 1) ? hi_half(v.x) : lo_half(v.x);
        x.c = (q & 1) ? hi_half(v.y) : lo_half(v.y);
        return x;
    }
    __device__ __forceinline__ void store(int kind, int q, int t, DotAcc<float> x)
    {
        ulonglong2 v = d[kind][q >> 1][t];
        if (q & 1) {
            v.x = pack2(lo_half(v.x), x.s);
            v.y = pack2(lo_half(v.y), x.c);
        } else {
            v.x = pack2(x.s, hi_half(v.x));
            v.y = pack2(x.c, hi_half(v.y));
        }
        d[kind][q >> 1][t] = v;
    }
};

// A matrix value through the read-only cache.
template <typename T>
__device__ __forceinline__ T ldg_val(const T* p) { return __ldg(p); }
template <>
__device__ __forceinline__ df64 ldg_val<df64>(const df64* p)
{
    const float2 v = __ldg(reinterpret_cast<const float2*>(p));
    return df64(v.x, v.y);
}

// A register value from lane src of the group.
template <typename T>
__device__ __forceinline__ T shfl_val(unsigned mask, T v, int src, int width)
{
    return __shfl_sync(mask, v, src, width);
}
template <>
__device__ __forceinline__ df64 shfl_val<df64>(unsigned mask, df64 v, int src, int width)
{
    return df64(__shfl_sync(mask, v.hi, src, width), __shfl_sync(mask, v.lo, src, width));
}

// The operand's values in precision T (null for a pattern matrix).
template <typename T>
const T* vals_of(const DevCSR& C)
{
    if (std::is_same<T, double>::value) return reinterpret_cast<const T*>(C.val64);
    if (std::is_same<T, float>::value) return reinterpret_cast<const T*>(C.val32);
    return reinterpret_cast<const T*>(C.valdf);
}

template <typename T>
struct StepArgs {
    const int64_t* rowptr;
    const int32_t* col;
    const T* val;          // null: pattern (all ones)
    int64_t nrows;         // rows handled by this launch
    int64_t nnz;           // stored entries
    int vec;               // col starts on a 16-byte boundary
    int ldv;               // row stride of every vector buffer
    int nvec;              // live vectors per row: ceil(act / N)
    int nchunks;           // vector chunks of width G per row
    const T* vgather;      // gathered operand (V_k, or W = X V_k for a Gram step)
    const T* vcur;         // V_k at the row itself
    T* vprev_out;          // in: V_{k-1} (unless first); out: V_{k+1}
    T alpha, beta;         // At = alpha A + beta I
    T ua, ub;              // the update's coefficients: 2 alpha, 2 beta in a recurrence step, alpha, beta in a first one
    int mode;              // 0 first step, 1 recurrence step, 2 plain product, 3 Clenshaw step
    const T* addv;         // mode 3: out = m1 * At V_k - V_{k-1} + coef * addv (no dots)
    T coef, m1;
    int direct;            // dots are z . V_{k+1} instead of V.V and V.V_k
    int B;                 // probes in the group (columns >= B are padding)
    uint64_t seedmix;
    const int64_t* ids;    // global id of each column's probe (direct mode)
    const int32_t* orig;   // original id of each row (relabelled operator), or null
    double* partials;      // [gridDim.x][2][ldv] for this launch
    // work split of this operand
    int64_t nch, Uc, Ul, nseg;
    int rb;                // rows of a work item of groups narrower than a warp (0: chunks)
    int even;              // neighbouring rows are of about equal length
    int walk;              // each group walks its own chunks (see may_walk)
    int nlong, nhuge;
    int long_ctas;         // CTAs of the long-row kernel that deal out its rows to groups
    int by_cta;            // rows of kHugeSegs segments or more take a CTA each (see cta_rows)
    const int32_t* first;      // [nch + 1] the first row whose first unit lies in chunk c or later
    const int32_t* seg_row;
    const int64_t* seg_k0;
    const int32_t* long_rows;
    const int64_t* long_seg0;
    const int32_t* huge;        // the long rows of kHugeSegs segments or more (indices of long_rows)
    const int32_t* seg_order;   // dealing order of the segments, or null (segment order)
    T* segpart;            // [nseg][ldv] partial products of long-row segments
};

template <typename T, int G>
struct Lane {
    static constexpr int N = Lanes<T>::N;
    int glane;
    unsigned gmask;
    bool vok;
    int c0;
    long long gcls, ncls;   // group index within its column class, groups per class
    bool active;

    __device__ Lane(const StepArgs<T>& a)
    {
        const int tid = threadIdx.x;
        const int lane = tid & 31;
        glane = lane & (G - 1);
        gmask = (G == 32) ? 0xFFFFFFFFu : (((1u << G) - 1u) << (lane & ~(G - 1)));
        // Both branches give the same for full warps.  In the second form ptxas
        // allocates the full-warp kernels' registers differently: FP32 at 128
        // probes took 6% (graphs) to 19% longer (stencils), double-float up to 7%.
        int chunk;
        if constexpr (G == 32) {
            const int gpb = kThreads / G;
            const long long gg = (long long)blockIdx.x * gpb + tid / G;
            const long long total = (long long)gridDim.x * gpb;
            ncls = total / a.nchunks;
            gcls = gg / a.nchunks;
            chunk = (int)(gg % a.nchunks);
            active = gg < ncls * a.nchunks;
        } else {
            // a warp's groups share one column class
            const int gw = blockIdx.x * kWarps + (tid >> 5);
            const int wcls = (int)(gridDim.x * kWarps) / a.nchunks;
            chunk = gw % a.nchunks;
            gcls = (long long)(gw / a.nchunks) * (32 / G) + lane / G;
            ncls = (long long)wcls * (32 / G);
            active = gw < wcls * a.nchunks;
        }
        const int vidx = chunk * G + glane;
        vok = vidx < a.nvec;
        c0 = vidx * N;
    }
};


// What a step kernel computes with a row sum.
enum StepKind {
    kRecurrence = 0,   // the recurrence update and its dot products (modes 0 and 1)
    kClenshaw = 1,     // a Clenshaw step (mode 3)
    kProduct = 2,      // the plain product (mode 2)
};

// Running sums of one row over the lane's N columns: add() takes one gathered
// row slice (and the entry's value, for valued matrices), close() ends a batch
// of at most G entries, out() gives the N sums.  Three forms:
//  - SumScalar: any vector type, acc = fma(a_ij, x, acc) for valued matrices
//    and acc + x for patterns (every a_ij = 1; for FP32 and FP64 that equals
//    fma(1, x, acc) bit for bit);
//  - SumF2, FP32 patterns: the four sums as two packed pairs, each packed add
//    the scalar add on both halves, so the sums are the same bit for bit (on
//    valued matrices the packed form, with a_ij broadcast into a pair,
//    measured slower);
//  - SumDf2, double-float patterns: the two sums as packed pairs of high and
//    low parts, added as df_add_lazy does (the rounding error of the high
//    parts into the low parts, left unnormalised) and renormalised as df_norm
//    does at the end of each batch.  That cuts the arithmetic from 11 to 8
//    FP32 operations per value, each packed instruction doing two, and the
//    deferred error stays below 2^-38 of the sum.  A double-float slice loads
//    as (high parts, low parts), the two packed operands.
template <typename T, bool PAT>
struct SumScalar {
    static constexpr int N = Lanes<T>::N;
    using P = Pack<T, N>;
    T s[N];
    __device__ __forceinline__ void init()
    {
#pragma unroll
        for (int q = 0; q < N; ++q) s[q] = T(0);
    }
    template <bool E>
    __device__ __forceinline__ void add(const T* p, T v, uint64_t pol)
    {
        const P x = ld_gather<E>(reinterpret_cast<const P*>(p), pol);
#pragma unroll
        for (int q = 0; q < N; ++q) {
            if constexpr (PAT) s[q] = s[q] + x.get(q);
            else s[q] = fma(v, x.get(q), s[q]);
        }
    }
    __device__ __forceinline__ void close() {}
    __device__ __forceinline__ void out(T (&acc)[N]) const
    {
#pragma unroll
        for (int q = 0; q < N; ++q) acc[q] = s[q];
    }
};

struct SumF2 {
    uint64_t A0, A1;
    __device__ __forceinline__ void init() { A0 = A1 = 0; }
    template <bool E>
    __device__ __forceinline__ void add(const float* p, float, uint64_t pol)
    {
        const ulonglong2 x = ld_gather2<E>(p, pol);
        A0 = add2(A0, x.x);
        A1 = add2(A1, x.y);
    }
    __device__ __forceinline__ void close() {}
    __device__ __forceinline__ void out(float (&acc)[4]) const
    {
        acc[0] = lo_half(A0);
        acc[1] = hi_half(A0);
        acc[2] = lo_half(A1);
        acc[3] = hi_half(A1);
    }
};

struct SumDf2 {
    uint64_t H, Lo;
    __device__ __forceinline__ void init() { H = Lo = 0; }
    template <bool E>
    __device__ __forceinline__ void add(const df64* p, df64, uint64_t pol)
    {
        const ulonglong2 x = ld_gather2<E>(p, pol);
        const uint64_t s = add2(H, x.x);
        const uint64_t bb = sub2(s, H);
        const uint64_t e = add2(sub2(H, sub2(s, bb)), sub2(x.x, bb));
        Lo = add2(Lo, add2(e, x.y));
        H = s;
    }
    __device__ __forceinline__ void close()
    {
        const uint64_t s = add2(H, Lo);
        Lo = sub2(Lo, sub2(s, H));
        H = s;
    }
    __device__ __forceinline__ void out(df64 (&acc)[2]) const
    {
        acc[0] = df64(lo_half(H), lo_half(Lo));
        acc[1] = df64(hi_half(H), hi_half(Lo));
    }
};

template <typename T, bool PAT> struct SumOf { using type = SumScalar<T, PAT>; };
template <> struct SumOf<float, true> { using type = SumF2; };
template <> struct SumOf<df64, true> { using type = SumDf2; };

// The sum over entries [k0, k1) for groups of a few lanes (few live probes):
// every lane loads its row's next kNarrowBatch column indices itself (the same
// addresses within a group), so that the gathers of a batch are in flight
// together; the loop over batches of G entries below would load one index,
// then its row slice, one latency after the other.  On FP32 and FP64 patterns
// (graphs: the rows are long enough) the indices come as two aligned 16-byte
// loads where the array allows it (a.vec: it starts on such a boundary), as
// lanes on different rows touch a sector each, whatever the width of the load;
// on valued matrices (short rows: the aligned start wastes slots) and for
// double-float that measured 4-40% slower.  Entries are added in order, as
// everywhere.  Per step, relabelled scale-20 R-MAT graph: FP32, 2 probes 412 ->
// 281 us, 16 probes 442 -> 280; double-float, 2 probes 392 -> 349, 8 probes 556
// -> 379; FP64, 2 probes 419 -> 349.  Wider groups share the index loads
// better: FP64 at 8 probes (G = 4) and double-float at 16 (G = 8) were up to
// 10% slower on stencils and Gram operators, so they keep the loop (kNarrow).
template <typename T, int G, bool PAT, typename Sum>
__device__ __forceinline__ void row_product_narrow(const StepArgs<T>& a, const Lane<T, G>& L, int k0, int k1, Sum& S,
                                                   uint64_t pol)
{
    constexpr bool E = StepTuning<T>::kEvictLast;
    const bool vec = PAT && !std::is_same<T, df64>::value && a.vec;
    // a batch may reach past 2^31 - 1: its slots are compared with the entries left
    const int first = vec ? k0 & ~3 : k0;
    int lead = k0 - first;
    const int32_t* col = a.col + first;
    const T* val = PAT ? nullptr : a.val + first;
    const int tail = (int)min(a.nnz - k1, (int64_t)kNarrowBatch);   // entries after the row
    for (int left = k1 - first; left > 0; left -= kNarrowBatch, lead = 0, col += kNarrowBatch) {
        int c[kNarrowBatch];
        T v[kNarrowBatch];
        if (vec && left + tail >= kNarrowBatch) {
#pragma unroll
            for (int u = 0; u < kNarrowBatch; u += 4) {
                const int4 x = __ldg(reinterpret_cast<const int4*>(col + u));
                c[u] = x.x;
                c[u + 1] = x.y;
                c[u + 2] = x.z;
                c[u + 3] = x.w;
            }
        } else {
#pragma unroll
            for (int u = 0; u < kNarrowBatch; ++u) c[u] = __ldg(col + min(u, left - 1));
        }
#pragma unroll
        for (int u = 0; u < kNarrowBatch; ++u) {
            v[u] = T(1);
            if constexpr (!PAT) v[u] = ldg_val(val + min(u, left - 1));
        }
        if constexpr (!PAT) val += kNarrowBatch;
#pragma unroll
        for (int u = 0; u < kNarrowBatch; ++u)
            if (u >= lead && u < left && L.vok)
                S.template add<E>(a.vgather + (size_t)c[u] * a.ldv + L.c0, v[u], pol);
        S.close();
    }
}

// acc = sum over entries [k0, k1) of a_ij * V[j, c0 .. c0+N), the column
// indices (and values) loaded G at a time from the row's first entry.  Row
// and entry indices fit in 32 bits (nnz < 2^31 is checked when the handle is
// made).
template <typename T, int G, bool PAT>
__device__ __forceinline__ void row_product_t(const StepArgs<T>& a, const Lane<T, G>& L, int k0, int k1,
                                              T (&acc)[Lanes<T>::N], uint64_t pol)
{
    constexpr int kGatherUnroll = StepTuning<T>::kUnroll;
    constexpr bool E = StepTuning<T>::kEvictLast;
    typename SumOf<T, PAT>::type S;
    S.init();
    if constexpr (G <= StepTuning<T>::kNarrow) {
        row_product_narrow<T, G, PAT>(a, L, k0, k1, S, pol);
        S.out(acc);
        return;
    }
    // the batch's column indices (and values); with PF the next batch's are
    // loaded while this batch's gathers are in flight
    constexpr bool PF = PAT && StepTuning<T>::kPrefetchPattern;
    int cj = 0;
    T vj = T(0);
    if (PF && k0 + L.glane < k1) cj = __ldg(a.col + k0 + L.glane);
    for (unsigned base = k0; base < (unsigned)k1; base += G) {   // unsigned: may reach past 2^31 - 1
        int cn = 0;
        if constexpr (PF) {
            if (base + G + L.glane < (unsigned)k1) cn = __ldg(a.col + base + G + L.glane);
        } else {
            const unsigned k = base + L.glane;
            if (k < (unsigned)k1) {
                cj = __ldg(a.col + k);
                if constexpr (!PAT) vj = ldg_val(a.val + k);
            }
        }
        const int cnt = min(G, k1 - (int)base);
        if constexpr (StepTuning<T>::kPredicated && G >= kGatherUnroll) {
            // blocks of kGatherUnroll predicated slots: every gather of a block
            // is issued before the first of them is consumed, also in the
            // last, partial block (groups narrower than a block, which take
            // at most G entries a batch, keep the plain loop)
            for (int t0 = 0; t0 < cnt; t0 += kGatherUnroll) {
#pragma unroll
                for (int u = 0; u < kGatherUnroll; ++u) {
                    const int t = t0 + u;
                    const int c = __shfl_sync(L.gmask, cj, t, G);
                    T v = T(1);
                    if constexpr (!PAT) v = shfl_val(L.gmask, vj, t, G);
                    if (t < cnt && L.vok) S.template add<E>(a.vgather + (size_t)c * a.ldv + L.c0, v, pol);
                }
            }
        } else {
#pragma unroll kGatherUnroll
            for (int t = 0; t < cnt; ++t) {
                const int c = __shfl_sync(L.gmask, cj, t, G);
                T v = T(1);
                if constexpr (!PAT) v = shfl_val(L.gmask, vj, t, G);
                if (L.vok) S.template add<E>(a.vgather + (size_t)c * a.ldv + L.c0, v, pol);
            }
        }
        S.close();
        if constexpr (PF) cj = cn;
    }
    S.out(acc);
}

template <typename T, int G, bool VALUED>
__device__ __forceinline__ void row_product(const StepArgs<T>& a, const Lane<T, G>& L, int k0, int k1,
                                            T (&acc)[Lanes<T>::N], uint64_t pol)
{
    if (VALUED || a.val) row_product_t<T, G, false>(a, L, k0, k1, acc, pol);
    else row_product_t<T, G, true>(a, L, k0, k1, acc, pol);
}

// row_product on a pattern.  The double-float step keeps the test of a.val: with
// the pattern form alone ptxas allocates its gather loop differently and the
// step measures 9-20% slower on graphs (relabelled scale-20 R-MAT, 64 probes,
// 1.78 against 1.63 ms); the FP32 step measures 3% faster without it (128
// probes, 1.28 against 1.31).
template <typename T, int G>
__device__ __forceinline__ void pattern_product(const StepArgs<T>& a, const Lane<T, G>& L, int k0, int k1,
                                                T (&acc)[Lanes<T>::N], uint64_t pol)
{
    if constexpr (std::is_same<T, df64>::value) row_product<T, G, false>(a, L, k0, k1, acc, pol);
    else row_product_t<T, G, true>(a, L, k0, k1, acc, pol);
}

// The row's operands of the epilogue, loaded before its gathers (they do not
// depend on them): V_k at the row and, in a recurrence step, V_{k-1}.
template <typename T>
struct RowOperands {
    Pack<T, Lanes<T>::N> xc, xp;
};

template <typename T>
__device__ __forceinline__ RowOperands<T> load_operands(const StepArgs<T>& a, int64_t r, int c0)
{
    using P = Pack<T, Lanes<T>::N>;
    RowOperands<T> o;
    const size_t off = (size_t)r * a.ldv + c0;
    if (a.mode != 2) o.xc = *reinterpret_cast<const P*>(a.vcur + off);
    if constexpr (std::is_same<T, double>::value) {   // a first step's update takes V_{k-1} = 0
        o.xp.set(0, 0.0);
        o.xp.set(1, 0.0);
    }
    if (a.mode == 1 || a.mode == 3) o.xp = *reinterpret_cast<const P*>(a.vprev_out + off);
    return o;
}

// The recurrence update and the V.V, V.V_k dot products of epilogue (below)
// for double-float vectors, on packed pairs: the lane's two entries go through
// the df64 operations of the generic code side by side.  A recurrence step
// folds its factor 2 into alpha and beta (doubling is exact), so
// out = (2 alpha) acc + (2 beta) xc - xp equals 2 (alpha acc + beta xc) - xp.
__device__ __forceinline__ void epilogue_df2(const StepArgs<df64>& a, size_t off, const df64 (&acc)[2],
                                             const RowOperands<df64>& ops, DotSlots<df64>& dots)
{
    df2 xc;
    memcpy(&xc, &ops.xc, sizeof(df2));
    df2 al = df2_of(a.alpha, a.alpha), be = df2_of(a.beta, a.beta);
    if (a.mode != 0) {
        al = df2_twice(al);
        be = df2_twice(be);
    }
    df2 out = al * df2_of(acc[0], acc[1]) + be * xc;
    if (a.mode != 0) {
        df2 xp;
        memcpy(&xp, &ops.xp, sizeof(df2));
        out = out + (-xp);
    }
    *reinterpret_cast<ulonglong2*>(a.vprev_out + off) = make_ulonglong2(out.h, out.l);
    const int tid = threadIdx.x;
    const df2 s0 = out * out + df2_of(dots.d[0][0][tid].s, dots.d[0][1][tid].s);
    dots.d[0][0][tid].s = df2_first(s0);
    dots.d[0][1][tid].s = df2_second(s0);
    const df2 s1 = out * xc + df2_of(dots.d[1][0][tid].s, dots.d[1][1][tid].s);
    dots.d[1][0][tid].s = df2_first(s1);
    dots.d[1][1][tid].s = df2_second(s1);
}

// A packed Kahan step on two columns: sc = (sums, compensations) takes the
// products a * b, each as DotAcc<float>::add_prod does.
__device__ __forceinline__ void kahan_prod2(ulonglong2& sc, uint64_t a, uint64_t b)
{
    ulonglong2 v = sc;
    const uint64_t y = fma2(a, b, neg2(v.y));
    const uint64_t t = add2(v.x, y);
    v.y = sub2(sub2(t, v.x), y);
    v.x = t;
    sc = v;
}

// The recurrence update and the V.V, V.V_k dot products of epilogue (below)
// for FP32 vectors, on packed pairs: out = alpha' acc + beta' xc (- xp), the
// product beta' xc rounded and alpha' acc fused into the sum, with the factor
// 2 of a recurrence step folded into alpha' and beta' (doubling is exact).
__device__ __forceinline__ void epilogue_f2(const StepArgs<float>& a, size_t off, const float (&acc)[4],
                                            const RowOperands<float>& ops, DotSlots<float>& dots)
{
    ulonglong2 xc;
    memcpy(&xc, &ops.xc, sizeof(xc));
    const float al = a.mode != 0 ? 2.0f * a.alpha : a.alpha;
    const float be = a.mode != 0 ? 2.0f * a.beta : a.beta;
    const uint64_t al2 = pack2(al, al), be2 = pack2(be, be);
    uint64_t o0 = fma2(al2, pack2(acc[0], acc[1]), mul2(be2, xc.x));
    uint64_t o1 = fma2(al2, pack2(acc[2], acc[3]), mul2(be2, xc.y));
    if (a.mode != 0) {
        ulonglong2 xp;
        memcpy(&xp, &ops.xp, sizeof(xp));
        o0 = sub2(o0, xp.x);
        o1 = sub2(o1, xp.y);
    }
    *reinterpret_cast<ulonglong2*>(a.vprev_out + off) = make_ulonglong2(o0, o1);
    const int tid = threadIdx.x;
    kahan_prod2(dots.d[0][0][tid], o0, o0);
    kahan_prod2(dots.d[0][1][tid], o1, o1);
    kahan_prod2(dots.d[1][0][tid], o0, xc.x);
    kahan_prod2(dots.d[1][1][tid], o1, xc.y);
}

// V_{k+1}[r] from acc = (A V_k)[r], and the fused dot products.
template <typename T, int K>
__device__ __forceinline__ void epilogue(const StepArgs<T>& a, int64_t r, int c0, const T (&acc)[Lanes<T>::N],
                                         const RowOperands<T>& ops, DotSlots<T>& dots)
{
    constexpr int N = Lanes<T>::N;
    using P = Pack<T, N>;
    const size_t off = (size_t)r * a.ldv + c0;
    P out;
    if constexpr (K == kProduct) {
#pragma unroll
        for (int q = 0; q < N; ++q) out.set(q, acc[q]);
        *reinterpret_cast<P*>(a.vprev_out + off) = out;
        return;
    }
    const P& xc = ops.xc;
    if constexpr (K == kClenshaw) {
        const P& xp = ops.xp;
        const P xa = *reinterpret_cast<const P*>(a.addv + off);
#pragma unroll
        for (int q = 0; q < N; ++q)
            out.set(q, a.m1 * (a.alpha * acc[q] + a.beta * xc.get(q)) - xp.get(q) + a.coef * xa.get(q));
        *reinterpret_cast<P*>(a.vprev_out + off) = out;
        return;
    }
    if constexpr (std::is_same<T, df64>::value) {
        if (!a.direct) {
            epilogue_df2(a, off, acc, ops, dots);
            return;
        }
    }
    if constexpr (std::is_same<T, float>::value) {
        if (!a.direct) {
            epilogue_f2(a, off, acc, ops, dots);
            return;
        }
    }
    if constexpr (std::is_same<T, double>::value) {
        // two FP64 operations a value for both modes: a recurrence step's factor
        // 2 is folded into the coefficients (doubling is exact), a first step has
        // no V_{k-1}.  (Doubled here, the coefficients cost two more operations a
        // row: 18% on the 72^3 stencil, whose step is bound by the FP64 pipe.)
        const P& xp = ops.xp;
#pragma unroll
        for (int q = 0; q < N; ++q) out.set(q, ::fma(a.ua, acc[q], ::fma(a.ub, xc.get(q), -xp.get(q))));
    } else if (a.mode == 0) {
#pragma unroll
        for (int q = 0; q < N; ++q) out.set(q, a.alpha * acc[q] + a.beta * xc.get(q));
    } else {
        const P& xp = ops.xp;
#pragma unroll
        for (int q = 0; q < N; ++q) out.set(q, T(2) * (a.alpha * acc[q] + a.beta * xc.get(q)) - xp.get(q));
    }
    *reinterpret_cast<P*>(a.vprev_out + off) = out;
    const int tid = threadIdx.x;
    if (!a.direct) {
#pragma unroll
        for (int q = 0; q < N; ++q) {
            DotAcc<T> s0 = dots.load(0, q, tid), s1 = dots.load(1, q, tid);
            const T o = out.get(q);
            s0.add_prod(o, o);
            s1.add_prod(o, xc.get(q));
            dots.store(0, q, tid, s0);
            dots.store(1, q, tid, s1);
        }
    } else {
#pragma unroll
        for (int q = 0; q < N; ++q) {
            if (c0 + q >= a.B) break;
            const bool neg = probe_negative(a.seedmix, (uint64_t)a.ids[c0 + q], (uint64_t)(a.orig ? a.orig[r] : r));
            DotAcc<T> s1 = dots.load(1, q, tid);
            s1.add(neg ? -out.get(q) : out.get(q));
            dots.store(1, q, tid, s1);
        }
    }
}

// Zero the thread's dot slots (each thread only ever touches its own).
template <typename T>
__device__ __forceinline__ void clear_dots(DotSlots<T>& dots)
{
#pragma unroll
    for (int q = 0; q < Lanes<T>::N; ++q) {
        DotAcc<T> z;
        z.clear();
        dots.store(0, q, threadIdx.x, z);
        dots.store(1, q, threadIdx.x, z);
    }
}

// What running dots are merged in across a CTA: FP64 sums in FP64; double-float
// ones as sums with two error terms (sum3: closer than FP64 additions, on the
// FP32 pipes); FP32 ones (sum and compensation) as double-float pairs, whose
// additions lose 2^-47 of the larger operand, against the 2^-23 of the sums
// themselves.  Measured over 240 combinations of operator, width and form,
// against FP64 moments: the errors of FP32 ones are the same to four digits
// with a merge in FP64, in pairs or in sum3; those of double-float ones were up
// to 1.4 times larger with pairs, and are the same with FP64 and sum3 (mean
// ratio to FP64 0.995).  A double-float step merged in FP64 took 3.6% longer
// than with sum3 (geometric mean over stencils, grids, Gram operators and graphs; 48^3
// stencil, one probe, 14.9 against 12.3 us; 64^2 grid, 128 probes, 17.4 against
// 15.0); an FP32 step merged in FP64 took up to 7 us longer (72^3 stencil, one
// probe, 27.9 -> 35.0), and in sum3 1% (geometric mean) than with pairs.
template <typename T> struct Merge {
    using In = df64;   // a thread's sum
    using M = sum3;
    static __device__ __forceinline__ double out(sum3 x) { return to_double(x); }
};
template <> struct Merge<float> {
    using In = df64;
    using M = df64;
    static __device__ __forceinline__ double out(df64 x) { return df_to_double(x); }
};
template <> struct Merge<double> {
    using In = double;
    using M = double;
    static __device__ __forceinline__ double out(double x) { return x; }
};
__device__ __forceinline__ double merge_in(DotAcc<double> x) { return x.s; }
__device__ __forceinline__ df64 merge_in(DotAcc<float> x) { return df64(x.s, -x.c); }
__device__ __forceinline__ df64 merge_in(DotAcc<df64> x) { return x.s; }
__device__ __forceinline__ double shfl_xor_val(double v, int m) { return __shfl_xor_sync(0xFFFFFFFFu, v, m); }
__device__ __forceinline__ df64 shfl_xor_val(df64 v, int m)
{
    return df64(__shfl_xor_sync(0xFFFFFFFFu, v.hi, m), __shfl_xor_sync(0xFFFFFFFFu, v.lo, m));
}
__device__ __forceinline__ sum3 shfl_xor_val(sum3 v, int m)
{
    return sum3(__shfl_xor_sync(0xFFFFFFFFu, v.a, m), __shfl_xor_sync(0xFFFFFFFFu, v.b, m),
                __shfl_xor_sync(0xFFFFFFFFu, v.c, m));
}

// CTA reduction in a fixed order.  A warp has one column class, so its 32/G
// groups hold 2 N G sums (kind, column of the lane, lane of the group) that
// are first merged within the warp, then across the warps of the class.
//
// With G lanes a group the CTA holds 256/G running sums per column.  Adding
// those one after another (one thread per column) is a serial chain of up to
// 256 dependent FP64 additions: it set a floor of 50 us (FP64) to 100 us (FP32,
// with its conversions) under every step of 1 to 4 live probes, whatever the
// operator's size.  Here each lane adds 2 N of them (or the 32/G of its
// outputs) and a shuffle tree the rest, at most 2 N + 5 + 8 additions deep.
// Measured, per step: 64^2 grid, 2 probes, FP32 99.5 -> 10.5 us, FP64 51.7 ->
// 12.2; 72^3 stencil, 2 probes, FP32 125 -> 32 us, FP64 85 -> 46; 20^3 stencil,
// 128 probes, FP32 22.9 -> 14.3.  Steps bound elsewhere did not move.
template <typename T, int G>
__device__ __forceinline__ void cta_partials(double* partials, int ldv, int nvec, int nchunks, DotSlots<T>& dots)
{
    constexpr int N = Lanes<T>::N;
    using In = typename Merge<T>::In;
    using M = typename Merge<T>::M;
    using W = std::conditional_t<G == 32, In, M>;   // a warp's sums (of full-warp groups: as they come)
    constexpr int O = 2 * N * G;                    // a warp's outputs: (kind * N + q) * G + lane of the group
    constexpr int V = O > 32 ? O / 32 : 1;          // outputs per lane
    static_assert(sizeof(W) * O * kWarps <= sizeof(DotSlots<T>), "the warp sums overlay the dot slots");
    __syncwarp();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, t0 = threadIdx.x & ~31;
    W v[V];
    if constexpr (O <= 32) {
        const int o = lane % O, part = lane / O;    // 32/O parts of 2N groups each
        const int kind = o / (N * G), q = (o / G) % N, gl = o % G;
        v[0] = W(merge_in(dots.load(kind, q, t0 + part * (2 * N) * G + gl)));
#pragma unroll
        for (int g = 1; g < 2 * N; ++g) v[0] = v[0] + W(merge_in(dots.load(kind, q, t0 + (part * 2 * N + g) * G + gl)));
#pragma unroll
        for (int m = O; m < 32; m <<= 1) v[0] = v[0] + shfl_xor_val(v[0], m);
    } else {
#pragma unroll
        for (int i = 0; i < V; ++i) {
            const int o = i * 32 + lane;
            const int kind = o / (N * G), q = (o / G) % N, gl = o % G;
            v[i] = W(merge_in(dots.load(kind, q, t0 + gl)));
#pragma unroll
            for (int g = 1; g < 32 / G; ++g) v[i] = v[i] + W(merge_in(dots.load(kind, q, t0 + g * G + gl)));
        }
    }
    __syncthreads();
    W* wsum = reinterpret_cast<W*>(&dots);          // [warp][O]
    if constexpr (O <= 32) {
        if (lane < O) wsum[warp * O + lane] = v[0];
    } else {
#pragma unroll
        for (int i = 0; i < V; ++i) wsum[warp * O + i * 32 + lane] = v[i];
    }
    __syncthreads();
    const int ncols = nvec * N;
    double* part = partials + (size_t)blockIdx.x * 2 * ldv;
    const int w0 = blockIdx.x * kWarps;
    const int nact = ((int)(gridDim.x * kWarps) / nchunks) * nchunks;   // warps that work
    for (int i = threadIdx.x; i < 2 * ncols; i += kThreads) {
        const int kind = i >= ncols, c = i - kind * ncols;
        const int vi = c / N, q = c % N;
        const int ch = vi / G, gl = vi % G;
        int w = (ch - w0 % nchunks + nchunks) % nchunks;   // the first warp of this class in the CTA
        M s = M(0);
        for (; w < kWarps && w0 + w < nact; w += nchunks) s = s + M(wsum[w * O + (kind * N + q) * G + gl]);
        part[kind * ldv + c] = Merge<T>::out(s);
    }
}

// The product of segment sidx, to the segment table (of a matrix that is VALUED or
// a PATTERN for certain, or either).
template <typename T, int G, bool VALUED, bool PATTERN = false>
__device__ __forceinline__ void segment_product(const StepArgs<T>& a, const Lane<T, G>& L, int64_t sidx, uint64_t pol)
{
    constexpr int N = Lanes<T>::N;
    T acc[N];
    const int64_t r = __ldg(a.seg_row + sidx);
    const int k0 = (int)__ldg(a.seg_k0 + sidx);
    const int k1 = (int)min((int64_t)k0 + a.Ul, __ldg(a.rowptr + r + 1));
    if constexpr (PATTERN) pattern_product<T, G>(a, L, k0, k1, acc, pol);
    else row_product<T, G, VALUED>(a, L, k0, k1, acc, pol);
    if (!L.vok) return;
    Pack<T, N> p;
#pragma unroll
    for (int q = 0; q < N; ++q) p.set(q, acc[q]);
    *reinterpret_cast<Pack<T, N>*>(a.segpart + (size_t)sidx * a.ldv + L.c0) = p;
}

// The work items of a warp whose lanes form R = 32/G groups: a run of rows,
// dealt to the groups in turn, so that the groups do a row each in step.  (With
// a chunk per group the groups of a warp drift apart: a chunk holds six or
// seven rows of a stencil, and its first row may belong to the one before; the
// warp then issues the union of their work.)  The run is a.rb rows, or R
// chunks where a.rb = 0 (see launch_step_g).
//
// Full-warp groups (R = 1) take their rows this way on valued matrices: the
// 48^3 stencil's double-float step at 128 probes 217 -> 165 us, the 2^18 x 2^16
// Gram operator's 937 -> 731.  Pattern steps (graphs: long rows) measured 5%
// slower and keep the chunk loop of the kernel below.
template <typename T, int G, int K>
__device__ __forceinline__ void row_items(const StepArgs<T>& a, const Lane<T, G>& L, DotSlots<T>& dots, uint64_t pol)
{
    constexpr int N = Lanes<T>::N;
    constexpr int R = 32 / G;
    const int sub = (threadIdx.x & 31) / G;
    const int nrows = (int)a.nrows;
    const int64_t nblk = a.rb ? (nrows - 1) / a.rb + 1 : (a.nch + R - 1) / R;
    const int64_t nitems = nblk + (a.nseg + R - 1) / R;
    const int64_t w0 = L.gcls / R, wstride = L.ncls / R;
    for (int64_t it = w0; it < nitems; it += wstride) {
        T acc[N];
        if (it < nblk) {
            int r0 = (int)it * a.rb, n = min(a.rb, nrows - r0);
            if (!a.rb) {
                r0 = __ldg(a.first + it * R);
                n = __ldg(a.first + min(it * R + R, a.nch)) - r0;
            }
            // rows are counted from the run's first: a group's next row may lie
            // past 2^31 - 1
            const int64_t* rp = a.rowptr + r0;
            int i = sub;
            int beg = i < n ? (int)__ldg(rp + i) : 0, end = i < n ? (int)__ldg(rp + i + 1) : 0;
            for (int ib = 0; ib < n; ib += R) {
                const int in = i + R;      // this group's next row, loaded one row ahead
                const int nbeg = in < n ? (int)__ldg(rp + in) : 0;
                const int nend = in < n ? (int)__ldg(rp + in + 1) : 0;
                if (i < n && end - beg <= a.Ul) {
                    const int r = r0 + i;
                    RowOperands<T> ops;
                    if (L.vok) ops = load_operands(a, r, L.c0);
                    row_product<T, G, G == 32>(a, L, beg, end, acc, pol);
                    if (L.vok) epilogue<T, K>(a, r, L.c0, acc, ops, dots);
                }
                i = in;
                beg = nbeg;
                end = nend;
            }
        } else {
            const int64_t i = (it - nblk) * R + sub;
            if (i < a.nseg)
                segment_product<T, G, G == 32>(a, L, a.seg_order ? (int64_t)__ldg(a.seg_order + i) : i, pol);
        }
    }
}

// The work items of FP32 recurrence steps.  A compensated FP32 sum rounds each
// product together with the running compensation, so the moments' last digits
// (1e-9 of the moments on a few thousand rows) depend on which rows a group
// adds and in which order.  That assignment is therefore fixed: group g of ncls
// takes chunks g, g + ncls, ... in order, and ncls follows from the operand,
// the width and the SM count alone (kFp32Blocks).  The groups of a warp still
// do a row each in step, each walking its own chunks.  Per step at 128 probes,
// against a loop that tests each row's units against its chunk's: 72^3 stencil
// 196 -> 175 us, 48^3 80 -> 64; at 32 probes 48^3 47 -> 25, 2^18 x 2^16 Gram 138 ->
// 101; relabelled scale-20 R-MAT 1321 -> 1250 at 128 probes, 470 -> 445 at 32,
// 793 -> 830 at 64.  Holding the chunks' rows in the lanes (no dependent loads)
// spilled and measured 14% slower, loading the next chunk's rows ahead 1-15%.
template <int G>
__device__ __forceinline__ void ordered_items(const StepArgs<float>& a, const Lane<float, G>& L,
                                              DotSlots<float>& dots, uint64_t pol)
{
    const int nch = (int)a.nch, ncls = (int)L.ncls;
    const auto do_row = [&](int r, int beg, int end) {
        if (end - beg > a.Ul) return;
        RowOperands<float> ops;
        float acc[Lanes<float>::N];
        if (L.vok) ops = load_operands(a, r, L.c0);
        row_product<float, G, G == 32>(a, L, beg, end, acc, pol);
        if (L.vok) epilogue<float, kRecurrence>(a, r, L.c0, acc, ops, dots);
    };
    if constexpr (G == 32) {
        for (int c = (int)L.gcls; c < nch; c += ncls) {
            int r = __ldg(a.first + c);
            const int rend = __ldg(a.first + c + 1);
            if (r >= rend) continue;
            int beg = (int)__ldg(a.rowptr + r), end = (int)__ldg(a.rowptr + r + 1);
            for (; r < rend; ++r) {
                // the next row's end, one row ahead of its use
                const int nxt = r + 1 < rend ? (int)__ldg(a.rowptr + r + 2) : end;
                do_row(r, beg, end);
                beg = end;
                end = nxt;
            }
        }
    } else {
        int c = (int)L.gcls, r = 0, rend = 0, beg = 0, end = 0;
        if (c < nch) {
            r = __ldg(a.first + c);
            rend = __ldg(a.first + c + 1);
        }
        bool fresh = true;             // the row's pointers are not loaded yet
        for (;;) {
            while (r >= rend && c < nch) {
                c += ncls;
                fresh = true;
                if (c < nch) {
                    r = __ldg(a.first + c);
                    rend = __ldg(a.first + c + 1);
                }
            }
            const bool have = c < nch;
            if (!__any_sync(0xFFFFFFFFu, have)) break;
            if (have) {
                if (fresh) {
                    beg = (int)__ldg(a.rowptr + r);
                    end = (int)__ldg(a.rowptr + r + 1);
                }
                const int nxt = r + 1 < rend ? (int)__ldg(a.rowptr + r + 2) : end;
                do_row(r, beg, end);
                ++r;
                beg = end;
                end = nxt;
                fresh = false;
            }
        }
    }
    for (int64_t i = L.gcls; i < a.nseg; i += L.ncls)
        segment_product<float, G, G == 32>(a, L, a.seg_order ? (int64_t)__ldg(a.seg_order + i) : i, pol);
}

// Whether a kernel has the loop in which each group walks its own chunks, out of
// step with the groups beside it: pattern steps of full-warp groups always take
// it, FP32 and double-float ones of 8 and 16 lanes where walks() says so.
template <typename T, int G>
constexpr bool may_walk() { return G == 32 || (G >= 8 && !std::is_same<T, double>::value); }

// On graphs the gathers of a group's row leave little for rows in step to save,
// and a long row holds up its neighbours.  Measured per step, in step against
// walking: relabelled scale-20 R-MAT, FP32, 64 probes 830 -> 709 us, 32 probes
// 444 -> 382, double-float, 32 probes 988 -> 932; scale 18, FP32, 64 probes 275 ->
// 254, double-float, 32 probes 354 -> 327; scale 16, FP32, 64 probes 112 -> 96,
// double-float, 32 probes 157 -> 142.  In step stays faster for FP32 groups of
// 8 lanes at scale 16 (32 probes 79 against 83), for double-float on relabelled
// small graphs (scale 16, 32 probes 75 against 103), and for FP64 (scale 20, 32
// probes 2.44 against 2.52 ms).
template <typename T, int G>
bool walks(const StepArgs<T>& a)
{
    if (a.val) return false;
    if (G == 32) return true;
    if (!may_walk<T, G>()) return false;
    const bool large = a.nnz >= kLargePattern;
    return std::is_same<T, float>::value ? G == 16 || large : !a.even || large;
}

// How the walking loop finds a chunk's end: from the next chunk's first row, or,
// for full-warp double-float groups, by each row's units.  Both give the same
// rows; the second has no second load that the first row's must wait with.
// Measured per step, first rows against units: double-float, 64 probes,
// relabelled scale-22 R-MAT 7181 -> 7069 us (calls as a whole differ by more than
// that from run to run), scale 20 1633 -> 1632, scale 16 within 0.5%; but FP32 64
// probes at scale 20 713 -> 759, 128 probes 1266 -> 1296, and double-float groups
// of 16 lanes (32 probes) at scale 20 939 -> 1013.
template <typename T, int G>
constexpr bool ends_by_units() { return std::is_same<T, df64>::value && G == 32; }

// Resident CTAs per SM a step kernel is compiled for.  The narrow kernels hold
// eight gathers of a lane in registers and run at four, but for the FP32
// recurrence, whose work is dealt to five per SM (ordered_items).
template <typename T, int G, int K>
constexpr int step_ctas()
{
    const bool ordered = std::is_same<T, float>::value && K == kRecurrence;
    return G <= StepTuning<T>::kNarrow && !ordered ? 4 : StepTuning<T>::kCtas;
}

template <typename T, int G, int K>
__global__ void __launch_bounds__(kThreads, step_ctas<T, G, K>()) cheb_step_kernel(StepArgs<T> a)
{
    constexpr int N = Lanes<T>::N;
    const Lane<T, G> L(a);
    __shared__ DotSlots<T> dots;
    if constexpr (K == kRecurrence) clear_dots<T>(dots);
    pdl_wait();
    const uint64_t pol = StepTuning<T>::kEvictLast ? evict_last_policy() : 0;

    if (!may_walk<T, G>() || !a.walk) {
        if (L.active) {
            if constexpr (std::is_same<T, float>::value && K == kRecurrence) ordered_items<G>(a, L, dots, pol);
            else row_items<T, G, K>(a, L, dots, pol);
        }
        pdl_trigger();
        if constexpr (K != kRecurrence) return;
        cta_partials<T, G>(a.partials, a.ldv, a.nvec, a.nchunks, dots);
        return;
    }
    if (L.active) {
        const int64_t nitems = a.nch + a.nseg;
        for (int64_t it = L.gcls; it < nitems; it += L.ncls) {
            T acc[N];
            if (it < a.nch) {
                // row and entry indices fit in 32 bits (nnz < 2^31)
                const int nrows = (int)a.nrows;
                int r = __ldg(a.first + it);
                constexpr bool BU = ends_by_units<T, G>();
                const int64_t u1 = (it + 1) * a.Uc;
                const int rend = BU ? nrows : __ldg(a.first + it + 1);
                int beg = r < nrows ? (int)__ldg(a.rowptr + r) : 0;
                int end = r < nrows ? (int)__ldg(a.rowptr + r + 1) : 0;
                for (; r < rend; ++r) {
                    if (BU && (int64_t)beg + kPlanRowCost * r >= u1) break;
                    // the row after next's end, one row ahead of its use
                    const int nxt = r <= nrows - 2 ? (int)__ldg(a.rowptr + r + 2) : end;
                    if (end - beg <= a.Ul) {   // long rows are done by segments
                        RowOperands<T> ops;
                        if (L.vok) ops = load_operands(a, r, L.c0);
                        pattern_product<T, G>(a, L, beg, end, acc, pol);
                        if (L.vok) epilogue<T, K>(a, r, L.c0, acc, ops, dots);
                    }
                    beg = end;
                    end = nxt;
                }
            } else {
                const int64_t sidx = a.seg_order ? (int64_t)__ldg(a.seg_order + (it - a.nch)) : it - a.nch;
                segment_product<T, G, false, true>(a, L, sidx, pol);
            }
        }
    }
    pdl_trigger();
    if constexpr (K != kRecurrence) return;
    cta_partials<T, G>(a.partials, a.ldv, a.nvec, a.nchunks, dots);
}

// Long rows: add the segment products in segment order, then the recurrence.
// Bound by latency: a row's products come one after another, and the hub rows
// of a power-law graph have hundreds (283 on the scale-20 R-MAT graph).  Rows
// of kHugeSegs segments or more therefore take a whole CTA: 82 -> 33 us a launch
// on that graph (FP32, relabelled), 95 -> 29 (double-float) and 39 -> 17 us (FP32
// Clenshaw) at scale 18; thresholds of 8 and 16 segments are within 8 us of
// that.  Several loads in flight per row instead measured slower on FP32 (70 to
// 142 us).  With more such rows than CTAs all rows go to groups (cta_rows).
template <typename T, int G, int K>
__global__ void __launch_bounds__(kThreads) cheb_long_kernel(StepArgs<T> a)
{
    constexpr int N = Lanes<T>::N;
    using P = Pack<T, N>;
    const Lane<T, G> L(a);
    __shared__ DotSlots<T> dots;
    pdl_trigger();
    if constexpr (K == kRecurrence) clear_dots<T>(dots);
    pdl_wait();
    // the rows of many segments, by CTA: every group brings its share of
    // the products to shared memory, the first group adds them in order
    if (a.by_cta) {
        constexpr int kGroups = kThreads / G, kRound = 4 * kGroups;
        __shared__ P prod[4 * kThreads];
        const int grp = threadIdx.x / G;
        for (int64_t h = blockIdx.x; h < a.nhuge; h += gridDim.x) {
            const int i = a.huge[h];
            const int s0 = (int)a.long_seg0[i], s1 = (int)a.long_seg0[i + 1];
            const int64_t r = a.long_rows[i];
            T acc[N];
#pragma unroll
            for (int q = 0; q < N; ++q) acc[q] = T(0);
            RowOperands<T> ops;
            if (grp == 0 && L.vok) ops = load_operands(a, r, L.c0);
            for (int base = s0; base < s1; base += kRound) {
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int s = base + u * kGroups + grp;
                    if (s < s1 && L.vok)
                        prod[u * kThreads + threadIdx.x] =
                            *reinterpret_cast<const P*>(a.segpart + (size_t)s * a.ldv + L.c0);
                }
                __syncthreads();
                if (grp == 0 && L.vok) {
                    const int n = min(kRound, s1 - base);
#pragma unroll 8
                    for (int j = 0; j < n; ++j) {
                        const P p = prod[j * G + threadIdx.x];   // group j % kGroups of load j / kGroups
#pragma unroll
                        for (int q = 0; q < N; ++q) acc[q] += p.get(q);
                    }
                }
                __syncthreads();
            }
            if (grp == 0 && L.vok) epilogue<T, K>(a, r, L.c0, acc, ops, dots);
        }
    }
    // with one column class, the groups of the first long_ctas CTAs (the others
    // are there for the rows above)
    const long long ncls = a.nchunks == 1 ? (long long)a.long_ctas * (kThreads / G) : L.ncls;
    if (L.active && L.gcls < ncls) {
        for (int64_t i = L.gcls; i < a.nlong; i += ncls) {
            if (!L.vok) continue;
            const int s0 = (int)a.long_seg0[i], s1 = (int)a.long_seg0[i + 1];
            if (a.by_cta && s1 - s0 >= kHugeSegs) continue;   // done above
            T acc[N];
#pragma unroll
            for (int q = 0; q < N; ++q) acc[q] = T(0);
            const int64_t r = a.long_rows[i];
            const RowOperands<T> ops = load_operands(a, r, L.c0);
            for (int s = s0; s < s1; ++s) {
                const P p = *reinterpret_cast<const P*>(a.segpart + (size_t)s * a.ldv + L.c0);
#pragma unroll
                for (int q = 0; q < N; ++q) acc[q] += p.get(q);
            }
            epilogue<T, K>(a, r, L.c0, acc, ops, dots);
        }
    }
    if constexpr (K != kRecurrence) return;
    cta_partials<T, G>(a.partials, a.ldv, a.nvec, a.nchunks, dots);
}

struct ReduceArgs {
    int nslots;
    int step0;
    int nblocks[kSlots];
    int act[kSlots];
};

// One warp per (slot, kind, column): lane l adds CTAs l, l+32, ... in order, then
// a fixed shuffle tree; the summation order never depends on timing.
__global__ void reduce_partials_kernel(const double* part, int max_blocks, int ldv, ReduceArgs ra, double* dots, int B)
{
    pdl_trigger();
    pdl_wait();
    const int slot = blockIdx.y;
    const int act = ra.act[slot];
    const int lane = threadIdx.x & 31;
    const int idx = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (idx >= 2 * act) return;
    const int kind = idx / act, c = idx % act;
    const double* p = part + (size_t)slot * max_blocks * 2 * ldv + (size_t)kind * ldv + c;
    double s = 0.0;
    const int nb = ra.nblocks[slot];
    for (int b = lane; b < nb; b += 32) s += p[(size_t)b * 2 * ldv];
#pragma unroll
    for (int o = 16; o; o >>= 1) s += __shfl_down_sync(0xFFFFFFFFu, s, o);
    if (lane == 0) dots[(size_t)(ra.step0 + slot) * 2 * B + (size_t)kind * B + c] = s;
}

// V_0 = z: row i of a relabelled operator holds the probe entry of original
// row orig[i].  A thread writes one 16-byte slice (N columns), hashing once per
// 64 consecutive probe ids.  Bound by the write (0.5 GB for 128 FP32 probes on
// 2^20 rows, 80 us at the copy rate); with one hash, one 64-bit division and one
// element a thread at a time it took 390 us there, now 198.
template <typename T>
__global__ void init_probes_kernel(T* v0, int64_t d, int ldv, int B, const int64_t* __restrict__ ids,
                                   uint64_t seedmix, const int32_t* __restrict__ orig)
{
    constexpr int N = Lanes<T>::N;
    using P = Pack<T, N>;
    const unsigned nv = ldv / N;       // ldv is a multiple of 8
    const int64_t total = d * (int64_t)nv;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = total <= 0xFFFFFFFFLL ? (int64_t)((unsigned)e / nv) : e / nv;
        const int c0 = (int)(e - i * nv) * N;
        const uint64_t row = (uint64_t)(orig ? orig[i] : i);
        uint64_t q = ~(uint64_t)0, w = 0;
        P z;
#pragma unroll
        for (int k = 0; k < N; ++k) {
            bool neg = false;
            if (c0 + k < B) {
                const uint64_t p = (uint64_t)ids[c0 + k];
                if ((p >> 6) != q) {
                    q = p >> 6;
                    w = probe_word(seedmix, q, row);
                }
                neg = (w >> (p & 63)) & 1u;
            }
            z.set(k, c0 + k < B ? (neg ? T(-1) : T(1)) : T(0));
        }
        *reinterpret_cast<P*>(v0 + i * ldv + c0) = z;
    }
}

__global__ void finalize_moments_kernel(const double* __restrict__ dots, int B,
                                        const int32_t* __restrict__ deg,
                                        const int64_t* __restrict__ row, double* mu, int64_t ld,
                                        double d, int direct, int* err)
{
    const int c = blockIdx.y;
    const int dg = deg[c];
    double* out = mu + row[c] * ld;
    const double x0 = dg >= 1 ? dots[B + c] : 0.0;
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < ld;
         j += (int64_t)gridDim.x * blockDim.x) {
        double v;
        if (j > dg) {
            v = 0.0;
        } else if (j == 0) {
            v = d;
        } else if (direct) {
            v = dots[(size_t)(j - 1) * 2 * B + B + c];
        } else if (j == 1) {
            v = x0;
        } else if ((j & 1) == 0) {
            v = 2.0 * dots[(size_t)(j / 2 - 1) * 2 * B + c] - d;
        } else {
            v = 2.0 * dots[(size_t)((j - 1) / 2) * 2 * B + B + c] - x0;
        }
        if (!(fabs(v) <= d * (1.0 + 1e-6))) atomicOr(err, 1);
        out[j] = v;
    }
}

__global__ void to_float_kernel(const double* __restrict__ in, float* __restrict__ out, int64_t n)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        out[i] = (float)in[i];
}

int pow2_at_least(int v)
{
    int g = 1;
    while (g < v && g < 32) g <<= 1;
    return g;
}

// Lanes a group of a step with nvec 16-byte vectors a row.  A power of two that
// covers them in one class (at most 32) leaves up to half of the lanes idle,
// and an FP64 step, bound by the FP64 pipe, pays for every idle lane: 36 live
// probes (18 lanes of 32) cost what 64 do.  Several classes of narrower groups
// waste fewer, but the groups of a warp wait for the longest of their rows
// (imb, from the plan) and repeat the per-row work.  The narrower group is
// taken when lanes x imbalance x 1.35 is below the single class's lanes: the
// factor is what class splitting cost at most where rows are equal (72^3 and
// 48^3 stencils: 1.2 to 1.35; 36 probes 513 -> 420 us and 162 -> 141, 70
// probes 1045 -> 757; 46 and 50 probes stay at one class, where splitting
// measured 0.96 to 1.2 x).  Operators with uneven neighbouring rows (unsorted
// R-MAT, Gram) keep one class: 36 probes at scale 18 1293 against 1495 us,
// X^T X of 2^18 x 2^16 524 against 740.  FP32 and double-float steps are not
// bound by that pipe and keep one class.
template <typename T>
int lanes_per_group(int nvec, const SpmmPlan& P, const SpmmPlan* Q)
{
    const int full = pow2_at_least(std::min(nvec, 32));
    if (!std::is_same<T, double>::value || full < 8) return full;
    int best = full;
    double cost = (double)((nvec + full - 1) / full * full);
    for (int g = full / 2; g >= 4; g >>= 1) {
        const int i = g == 16 ? 0 : (g == 8 ? 1 : 2);
        const double imb = Q ? std::max(P.imb[i], Q->imb[i]) : P.imb[i];
        const double c = (double)((nvec + g - 1) / g * g) * imb * 1.35;
        if (c < cost) {
            best = g;
            cost = c;
        }
    }
    return best;
}

// Resident CTAs per SM of one instance of the step kernel.
template <typename T, int G, int K>
int resident_ctas()
{
    static const int occ = [] {
        int o = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, cheb_step_kernel<T, G, K>, kThreads, 0) !=
            cudaSuccess) {
            cudaGetLastError();
            o = 0;
        }
        return o;
    }();
    return occ;
}

// Whether a step's kernels are launched dependent on the one before (see
// pdl_trigger): row slices (16-byte vectors) gathered, plus 4 a row.
template <typename T>
bool dependent_launch(const StepArgs<T>& a)
{
    return (a.nnz + kPlanRowCost * a.nrows) * (int64_t)a.nvec <= kDependentWork;
}

// Whether the rows of kHugeSegs segments or more take a CTA each: where there is
// one for each of them.  A CTA's rows follow one another at 1 to 4 us a row,
// while groups take theirs side by side.  Per launch, one FP64 probe, with the
// CTAs counted for the groups (one for 256 rows) against this rule: 20 rows of
// 40 segments 80 -> 10 us, 200 rows 736 -> 11, 5,000 rows of 32 segments 860 -> 17
// (by groups); 128 FP32 probes, 200 rows 32 -> 10; R-MAT scale 18 (172 such rows
// among 12,616 long ones), one FP64 probe 37 -> 27, 128 FP32 probes 37 -> 30.
template <typename T>
bool cta_rows(const StepArgs<T>& a, int max_long)
{
    return a.nchunks == 1 && a.nhuge > 0 && a.nhuge <= max_long;
}

// Launch the step (and, with long rows, the kernel that adds their segments after
// it).  The CTA partials of the two kernels sit next to each other in `part`.
template <typename T, int G>
int launch_step_g(StepArgs<T> a, int max_main, int max_long, int num_sms, int* nblocks_out, cudaStream_t s)
{
    const int gpb = kThreads / G;
    const int min_blocks = (a.nchunks + kWarps - 1) / kWarps;    // a warp per column class at least
    const int occ = a.mode == 3   ? resident_ctas<T, G, kClenshaw>()
                    : a.mode == 2 ? resident_ctas<T, G, kProduct>()
                                  : resident_ctas<T, G, kRecurrence>();
    if (occ > 0) max_main = std::min(max_main, occ * num_sms);   // one resident wave
    long long ctas;
    const bool ordered = std::is_same<T, float>::value && a.mode < 2;   // see ordered_items
    if (ordered) max_main = std::min(max_main, kFp32Blocks * num_sms);
    a.walk = walks<T, G>(a);
    if (ordered || a.walk) {
        ctas = ((a.nch + a.nseg) * (long long)a.nchunks + gpb - 1) / gpb;
    } else {
        // Where neighbouring rows are about equal, a work item is a few rows a
        // group (a warp is one group on valued matrices at full width): about
        // kUnitsPerGroup units, at most kRowsPerGroup rows, fewer where a warp
        // would get less than four items.  Against R chunks (per step): 48^3
        // FP64, 32 probes 112 -> 87 us, 36 probes 141 -> 111; 72^3 FP64, 8 probes
        // 94 -> 78; 2^18 x 2^16 Gram FP64, 8 probes 169 -> 106; relabelled scale-16
        // R-MAT FP64, 32 probes 242 -> 170.  Rows of uneven length are better
        // dealt by units: unsorted scale-18 R-MAT FP64, 32 probes 838 us by
        // chunks, 967 by rows.
        constexpr int R = 32 / G;
        if (a.even) {
            const int64_t warps = std::max<int64_t>(1, (int64_t)max_main * kWarps / a.nchunks);
            const int64_t mean = (a.nnz + kPlanRowCost * a.nrows) / std::max<int64_t>(a.nrows, 1) + 1;
            const int64_t m = std::min<int64_t>({kUnitsPerGroup / mean, kRowsPerGroup, a.nrows / (4 * R * warps)});
            a.rb = R * (int)std::max<int64_t>(1, m);
        }
        const int64_t blocks = a.even ? (a.nrows + a.rb - 1) / a.rb : (a.nch + R - 1) / R;
        ctas = ((blocks + (a.nseg + R - 1) / R) * a.nchunks + kWarps - 1) / kWarps;
    }
    int nb = (int)std::max<long long>(1, std::min<long long>(ctas, max_main));
    nb = std::max(nb, min_blocks);
    const bool dep = dependent_launch(a);
    {
        ProfScope ps(a.mode == 2 ? "gram_spmm" : (a.mode == 3 ? "clenshaw_step" : "cheb_step"), s);
        auto* kernel = a.mode == 3   ? cheb_step_kernel<T, G, kClenshaw>
                       : a.mode == 2 ? cheb_step_kernel<T, G, kProduct>
                                     : cheb_step_kernel<T, G, kRecurrence>;
        MLT_CUDA_TRY(launch_dependent(dep, kernel, dim3(nb), kThreads, s, a));
    }
    int nl = 0;
    if (a.nlong > 0) {
        const long long litems = (long long)a.nlong * a.nchunks;
        nl = (int)std::max<long long>(1, std::min<long long>((litems + gpb - 1) / gpb, max_long));
        nl = std::max(nl, min_blocks);
        StepArgs<T> b = a;
        b.long_ctas = nl;
        b.by_cta = cta_rows(a, max_long);
        if (b.by_cta) nl = std::max(nl, a.nhuge);
        if (b.partials) b.partials += (size_t)nb * 2 * a.ldv;
        ProfScope ps(a.mode == 2 ? "gram_spmm_long" : (a.mode == 3 ? "clenshaw_step_long" : "cheb_step_long"), s);
        auto* kernel = a.mode == 3   ? cheb_long_kernel<T, G, kClenshaw>
                       : a.mode == 2 ? cheb_long_kernel<T, G, kProduct>
                                     : cheb_long_kernel<T, G, kRecurrence>;
        MLT_CUDA_TRY(launch_dependent(dep, kernel, dim3(nl), kThreads, s, b));
    }
    *nblocks_out = nb + nl;
    return MLT_OK;
}

template <typename T>
int launch_step(int G, const StepArgs<T>& a, int max_main, int max_long, int num_sms, int* nb, cudaStream_t s)
{
    switch (G) {
    case 1: return launch_step_g<T, 1>(a, max_main, max_long, num_sms, nb, s);
    case 2: return launch_step_g<T, 2>(a, max_main, max_long, num_sms, nb, s);
    case 4: return launch_step_g<T, 4>(a, max_main, max_long, num_sms, nb, s);
    case 8: return launch_step_g<T, 8>(a, max_main, max_long, num_sms, nb, s);
    case 16: return launch_step_g<T, 16>(a, max_main, max_long, num_sms, nb, s);
    default: return launch_step_g<T, 32>(a, max_main, max_long, num_sms, nb, s);
    }
}

template <typename T>
void set_operand(StepArgs<T>& a, const DevCSR& C, const T* val)
{
    a.rowptr = C.rowptr;
    a.col = C.col;
    a.val = val;
    a.nrows = C.nrows;
    a.nnz = C.nnz;
    a.vec = (reinterpret_cast<uintptr_t>(C.col) & 15) == 0;
}

template <typename T>
void set_split(StepArgs<T>& a, const SpmmPlan& P, T* segpart)
{
    a.nch = P.nch;
    a.Uc = P.Uc;
    a.Ul = P.Ul;
    a.nseg = P.nseg;
    a.even = P.imb[2] <= kEvenRows;
    a.nlong = P.nlong;
    a.nhuge = P.nhuge;
    a.huge = P.huge;
    a.first = P.first;
    a.seg_row = P.seg_row;
    a.seg_k0 = P.seg_k0;
    a.long_rows = P.long_rows;
    a.long_seg0 = P.long_seg0;
    a.seg_order = StepTuning<T>::kWindowSegs ? P.seg_order : nullptr;
    a.segpart = segpart;
}

// State shared by the recurrence steps of one probe group.
struct GroupCtx {
    bool gram;
    const int32_t* orig;    // relabelled operator (MLT_REORDER): original row ids, else null
    int64_t d;
    int ldv;
    double alpha, beta;
    uint64_t seedmix;
    double* part;
    double* dots;
    int max_main, max_long, max_blocks;
    ReduceArgs ra;
};

// Recurrence steps k0 <= k < k1 in precision T: V[k & 1] holds V_k and
// V[(k + 1) & 1] holds V_{k-1} on entry to step k.
template <typename T>
int run_steps(mlt_matrix* M, const MomentPlan& plan, GroupCtx& g, int k0, int k1, T* const* V, T* W,
              T* segpart, cudaStream_t s)
{
    constexpr int N = Lanes<T>::N;
    const DevCSR& A = g.orig ? M->P : M->A;
    const DevCSR& AT = M->AT;
    SpmmPlan& planA = g.orig ? M->plan_P : M->plan_A;
    const T* valA = vals_of<T>(A);
    const T* valAT = vals_of<T>(AT);
    int rc;
    for (int k = k0; k < k1; ++k) {
        const int act = plan.act[k];
        const int nvec = (act + N - 1) / N;
        const int G = lanes_per_group<T>(nvec, g.gram ? M->plan_A : planA, g.gram ? &M->plan_AT : nullptr);
        const int nchunks = (nvec + G - 1) / G;
        T* cur = V[k & 1];
        T* out = V[(k + 1) & 1];
        StepArgs<T> sa{};
        sa.ldv = g.ldv;
        sa.nvec = nvec;
        sa.nchunks = nchunks;
        sa.alpha = (T)g.alpha;
        sa.beta = (T)g.beta;
        sa.direct = plan.direct;
        sa.B = plan.B;
        sa.seedmix = g.seedmix;
        sa.ids = plan.ids_dev;
        sa.orig = g.orig;
        int nb = 0;
        if (g.gram) {
            StepArgs<T> pa = sa;
            set_operand(pa, A, valA);
            pa.vgather = cur; pa.vcur = nullptr; pa.vprev_out = W; pa.mode = 2;
            pa.partials = nullptr;
            set_split(pa, M->plan_A, segpart);
            if ((rc = launch_step<T>(G, pa, g.max_main, g.max_long, M->num_sms, &nb, s))) return rc;
            set_operand(sa, AT, valAT);
            sa.vgather = W;
            set_split(sa, M->plan_AT, segpart);
        } else {
            set_operand(sa, A, valA);
            sa.vgather = cur;
            set_split(sa, planA, segpart);
        }
        sa.vcur = cur;
        sa.vprev_out = out;
        sa.mode = (k == 0) ? 0 : 1;
        sa.ua = (T)(sa.mode ? 2.0 * g.alpha : g.alpha);
        sa.ub = (T)(sa.mode ? 2.0 * g.beta : g.beta);
        ReduceArgs& ra = g.ra;
        const int slot = k - ra.step0;
        sa.partials = g.part + (size_t)slot * g.max_blocks * 2 * g.ldv;
        if ((rc = launch_step<T>(G, sa, g.max_main, g.max_long, M->num_sms, &nb, s))) return rc;
        ra.nblocks[slot] = nb;
        ra.act[slot] = act;
        ra.nslots = slot + 1;
        if (ra.nslots == kSlots || k == plan.K - 1) {
            int amax = 0;
            for (int i = 0; i < ra.nslots; ++i) amax = std::max(amax, ra.act[i]);
            dim3 grid((2 * amax + 3) / 4, ra.nslots);
            ProfScope ps("reduce_partials", s);
            const bool dep = dependent_launch(sa);
            MLT_CUDA_TRY(launch_dependent(dep, reduce_partials_kernel, grid, 128, s, g.part, g.max_blocks, g.ldv, ra, g.dots,
                                          plan.B));
            ra.step0 = k + 1;
            ra.nslots = 0;
        }
    }
    return MLT_OK;
}

__global__ void widen_kernel(const float* __restrict__ in, double* __restrict__ out, int64_t n)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = (double)in[i];
}

// One probe group: steps [0, ks) in FP32 (when the group starts in FP32) and
// [ks, K) in FP64; ks = 0 is all FP64, ks >= K all FP32.  At the switch the
// two live vectors V_k, V_{k-1} are widened to FP64 and the recurrence goes on.
int run_group(mlt_matrix* M, const MomentPlan& plan, int ks, double a, double b, uint64_t seed,
              double* mu_dev, int64_t ld_mu, int* err_flag, cudaStream_t s, bool alloc_only)
{
    GroupCtx g;
    g.gram = (M->flags & MLT_GRAM) != 0;
    g.orig = M->perm;
    g.d = plan.dim;
    g.ldv = plan.ldv;
    ks = std::max(0, std::min(ks, plan.K));
    const bool f32 = ks > 0;
    const bool f64 = ks < plan.K || !f32;
    const size_t n = (size_t)g.d * g.ldv;
    const size_t wrows = g.gram ? (size_t)M->A.nrows * g.ldv : 0;
    int rc;
    if ((rc = ensure_spmm_plan(M, g.orig ? M->P : M->A, g.orig ? M->plan_P : M->plan_A, s))) return rc;
    if (g.gram && (rc = ensure_spmm_plan(M, M->AT, M->plan_AT, s))) return rc;
    if (f32 && (rc = ensure_fp32_values(M, s))) return rc;
    // V buffers: FP32 pair in ws_v (when used), FP64 pair in ws_v (all-FP64) or ws_v2 (mixed)
    float* Vf[2] = {nullptr, nullptr};
    double* Vd[2] = {nullptr, nullptr};
    if (f32) {
        if ((rc = M->ws_v[0].ensure(n * sizeof(float), s)) || (rc = M->ws_v[1].ensure(n * sizeof(float), s))) return rc;
        Vf[0] = M->ws_v[0].as<float>();
        Vf[1] = M->ws_v[1].as<float>();
    }
    if (f64) {
        DevBuf* vb = f32 ? M->ws_v2 : M->ws_v;
        if ((rc = vb[0].ensure(n * sizeof(double), s)) || (rc = vb[1].ensure(n * sizeof(double), s))) return rc;
        Vd[0] = vb[0].as<double>();
        Vd[1] = vb[1].as<double>();
    }
    const size_t tsz = f64 ? sizeof(double) : sizeof(float);
    if (g.gram && (rc = M->ws_w.ensure(wrows * tsz, s))) return rc;
    const int64_t nseg = std::max((g.orig ? M->plan_P : M->plan_A).nseg, g.gram ? M->plan_AT.nseg : (int64_t)0);
    if ((rc = M->ws_seg.ensure((size_t)std::max<int64_t>(nseg, 1) * g.ldv * tsz, s))) return rc;
    g.max_main = 8 * M->num_sms;
    g.max_long = 2 * M->num_sms;
    g.max_blocks = g.max_main + g.max_long;
    if ((rc = M->ws_part.ensure((size_t)kSlots * g.max_blocks * 2 * g.ldv * sizeof(double), s))) return rc;
    if ((rc = M->ws_dots.ensure((size_t)std::max(plan.K, 1) * 2 * plan.B * sizeof(double), s))) return rc;
    g.part = M->ws_part.as<double>();
    g.dots = M->ws_dots.as<double>();
    g.seedmix = seed * kGolden;
    g.ra = ReduceArgs{};
    // At = alpha A + beta I; the stored entries carry `scale` (squared for X^T X).
    const double sc = g.gram ? M->scale * M->scale : M->scale;
    g.alpha = 2.0 / (b - a) * sc;
    g.beta = -(a + b) / (b - a);
    if (alloc_only) return MLT_OK;
    {
        const int nb = (int)std::min<int64_t>(((int64_t)n + 255) / 256, 16LL * M->num_sms);
        ProfScope ps("init_probes", s);
        if (f32)
            init_probes_kernel<float><<<std::max(nb, 1), 256, 0, s>>>(Vf[0], g.d, g.ldv, plan.B, plan.ids_dev,
                                                                      g.seedmix, g.orig);
        else
            init_probes_kernel<double><<<std::max(nb, 1), 256, 0, s>>>(Vd[0], g.d, g.ldv, plan.B, plan.ids_dev,
                                                                       g.seedmix, g.orig);
    }
    MLT_CUDA_TRY(cudaGetLastError());
    if (f32) {
        if ((rc = run_steps<float>(M, plan, g, 0, ks, Vf, M->ws_w.as<float>(), M->ws_seg.as<float>(), s))) return rc;
    }
    if (f32 && f64 && ks < plan.K) {
        const int nb = (int)std::min<int64_t>(((int64_t)n + 255) / 256, 16LL * M->num_sms);
        ProfScope ps("widen_vectors", s);
        widen_kernel<<<std::max(nb, 1), 256, 0, s>>>(Vf[0], Vd[0], (int64_t)n);
        widen_kernel<<<std::max(nb, 1), 256, 0, s>>>(Vf[1], Vd[1], (int64_t)n);
        MLT_CUDA_TRY(cudaGetLastError());
    }
    if (f64) {
        if ((rc = run_steps<double>(M, plan, g, f32 ? ks : 0, plan.K, Vd, M->ws_w.as<double>(),
                                    M->ws_seg.as<double>(), s))) return rc;
    }
    {
        dim3 grid((unsigned)std::min<int64_t>((ld_mu + 127) / 128, 64), plan.B);
        ProfScope ps("finalize_moments", s);
        finalize_moments_kernel<<<grid, 128, 0, s>>>(g.dots, plan.B, plan.deg_dev, plan.row_dev, mu_dev,
                                                     ld_mu, (double)g.d, plan.direct, err_flag);
        MLT_CUDA_TRY(cudaGetLastError());
    }
    return MLT_OK;
}

// One probe group in double-float arithmetic throughout (MLT_PREC_DF64): the
// steps of run_group with df64 vectors, SpMM and per-thread dot products, the
// CTA partials and everything after them in FP64.
int run_group_df(mlt_matrix* M, const MomentPlan& plan, double a, double b, uint64_t seed, double* mu_dev,
                 int64_t ld_mu, int* err_flag, cudaStream_t s, bool alloc_only)
{
    GroupCtx g;
    g.gram = (M->flags & MLT_GRAM) != 0;
    g.orig = M->perm;
    g.d = plan.dim;
    g.ldv = plan.ldv;
    const size_t n = (size_t)g.d * g.ldv;
    const size_t wrows = g.gram ? (size_t)M->A.nrows * g.ldv : 0;
    int rc;
    if ((rc = ensure_spmm_plan(M, g.orig ? M->P : M->A, g.orig ? M->plan_P : M->plan_A, s))) return rc;
    if (g.gram && (rc = ensure_spmm_plan(M, M->AT, M->plan_AT, s))) return rc;
    if ((rc = ensure_df_values(M, s))) return rc;
    if ((rc = M->ws_v[0].ensure(n * sizeof(df64), s)) || (rc = M->ws_v[1].ensure(n * sizeof(df64), s))) return rc;
    df64* V[2] = {M->ws_v[0].as<df64>(), M->ws_v[1].as<df64>()};
    if (g.gram && (rc = M->ws_w.ensure(wrows * sizeof(df64), s))) return rc;
    const int64_t nseg = std::max((g.orig ? M->plan_P : M->plan_A).nseg, g.gram ? M->plan_AT.nseg : (int64_t)0);
    if ((rc = M->ws_seg.ensure((size_t)std::max<int64_t>(nseg, 1) * g.ldv * sizeof(df64), s))) return rc;
    g.max_main = 8 * M->num_sms;
    g.max_long = 2 * M->num_sms;
    g.max_blocks = g.max_main + g.max_long;
    if ((rc = M->ws_part.ensure((size_t)kSlots * g.max_blocks * 2 * g.ldv * sizeof(double), s))) return rc;
    if ((rc = M->ws_dots.ensure((size_t)std::max(plan.K, 1) * 2 * plan.B * sizeof(double), s))) return rc;
    g.part = M->ws_part.as<double>();
    g.dots = M->ws_dots.as<double>();
    g.seedmix = seed * kGolden;
    g.ra = ReduceArgs{};
    const double sc = g.gram ? M->scale * M->scale : M->scale;
    g.alpha = 2.0 / (b - a) * sc;
    g.beta = -(a + b) / (b - a);
    if (alloc_only) return MLT_OK;
    {
        const int nb = (int)std::min<int64_t>(((int64_t)n + 255) / 256, 16LL * M->num_sms);
        ProfScope ps("init_probes", s);
        init_probes_kernel<df64><<<std::max(nb, 1), 256, 0, s>>>(V[0], g.d, g.ldv, plan.B, plan.ids_dev, g.seedmix, g.orig);
    }
    MLT_CUDA_TRY(cudaGetLastError());
    if ((rc = run_steps<df64>(M, plan, g, 0, plan.K, V, M->ws_w.as<df64>(), M->ws_seg.as<df64>(), s))) return rc;
    {
        dim3 grid((unsigned)std::min<int64_t>((ld_mu + 127) / 128, 64), plan.B);
        ProfScope ps("finalize_moments", s);
        finalize_moments_kernel<<<grid, 128, 0, s>>>(g.dots, plan.B, plan.deg_dev, plan.row_dev, mu_dev, ld_mu,
                                                     (double)g.d, plan.direct, err_flag);
        MLT_CUDA_TRY(cudaGetLastError());
    }
    return MLT_OK;
}

// Matrix values as double-float pairs, entry by entry (values are read one
// entry at a time, not as vector slices).
__global__ void to_df_values_kernel(const double* __restrict__ in, df64* __restrict__ out, int64_t n)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = df64(in[i]);
}

// In place: the n (even) doubles at v become n double-float entries in the
// slice layout of Pack<df64, 2>; one thread per pair reads both before writing.
__global__ void to_df_kernel(double* v, int64_t n)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n / 2;
         i += (int64_t)gridDim.x * blockDim.x) {
        const double2 x = reinterpret_cast<const double2*>(v)[i];
        const df64 p(x.x), q(x.y);
        reinterpret_cast<float4*>(v)[i] = make_float4(p.hi, q.hi, p.lo, q.lo);
    }
}

// out[i] = coef * x[i] over n elements (x null: zeros).
template <typename T>
__global__ void scaled_copy_kernel(T* __restrict__ out, const T* __restrict__ x, T coef, int64_t n)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = x ? coef * x[i] : T(0);
}

// The context of FP64 steps over an explicit block of `cols` vectors with row
// stride ldv (buffers sized, map At = alpha A + beta I set).
int block_ctx(mlt_matrix* M, int ldv, int cols, int K, double a, double b, GroupCtx& g, cudaStream_t s)
{
    g.gram = (M->flags & MLT_GRAM) != 0;
    g.orig = nullptr;   // explicit vector blocks are in original row order
    g.d = g.gram ? M->A.ncols : M->A.nrows;
    g.ldv = ldv;
    int rc;
    if ((rc = ensure_spmm_plan(M, M->A, M->plan_A, s))) return rc;
    if (g.gram && (rc = ensure_spmm_plan(M, M->AT, M->plan_AT, s))) return rc;
    if (g.gram && (rc = M->ws_w.ensure((size_t)M->A.nrows * ldv * sizeof(double), s))) return rc;
    const int64_t nseg = std::max(M->plan_A.nseg, g.gram ? M->plan_AT.nseg : (int64_t)0);
    if ((rc = M->ws_seg.ensure((size_t)std::max<int64_t>(nseg, 1) * ldv * sizeof(double), s))) return rc;
    g.max_main = 8 * M->num_sms;
    g.max_long = 2 * M->num_sms;
    g.max_blocks = g.max_main + g.max_long;
    if ((rc = M->ws_part.ensure((size_t)kSlots * g.max_blocks * 2 * ldv * sizeof(double), s))) return rc;
    if ((rc = M->ws_dots.ensure((size_t)std::max(K, 1) * 2 * cols * sizeof(double), s))) return rc;
    g.part = M->ws_part.as<double>();
    g.dots = M->ws_dots.as<double>();
    g.seedmix = 0;
    g.ra = ReduceArgs{};
    const double sc = g.gram ? M->scale * M->scale : M->scale;
    g.alpha = 2.0 / (b - a) * sc;
    g.beta = -(a + b) / (b - a);
    return MLT_OK;
}

}  // namespace

// Y = p(At) X by Clenshaw's recurrence for p = sum_k c_k T_k (in FP64, or in
// FP32 with the handle's FP32 values): b_{n+1} = 0,
// b_n = c_n X, b_k = 2 At b_{k+1} - b_{k+2} + c_k X (k = n-1 .. 1), and
// p(At) X = At b_1 - b_2 + c_0 X: n operator applications.  b_j lives in
// P[(n + 1 - j) & 1], so each step overwrites b_{k+2} in place.
template <typename T>
int poly_apply_block_t(mlt_matrix* M, double a, double b, const double* c, int n, const T* X, T* Y, int ldv,
                       int ncols, T* P0, T* P1, cudaStream_t s)
{
    GroupCtx g;
    int rc;
    if ((rc = block_ctx(M, ldv, ncols, 1, a, b, g, s))) return rc;
    if (std::is_same<T, float>::value && (rc = ensure_fp32_values(M, s))) return rc;
    if (std::is_same<T, df64>::value && (rc = ensure_df_values(M, s))) return rc;
    const T* valA = vals_of<T>(M->A);
    const T* valAT = vals_of<T>(M->AT);
    const int64_t total = g.d * (int64_t)ldv;
    const int nbk = (int)std::max<int64_t>(1, std::min<int64_t>((total + 255) / 256, 16LL * M->num_sms));
    T* P[2] = {P0, P1};
    {
        ProfScope ps("clenshaw_init", s);
        scaled_copy_kernel<T><<<nbk, 256, 0, s>>>(P[0], nullptr, T(0), total);
        scaled_copy_kernel<T><<<nbk, 256, 0, s>>>(P[1], X, (T)c[n], total);
    }
    MLT_CUDA_TRY(cudaGetLastError());
    const int nvec = (ncols + Lanes<T>::N - 1) / Lanes<T>::N;
    const int G = lanes_per_group<T>(nvec, M->plan_A, g.gram ? &M->plan_AT : nullptr);
    const DevCSR& A = M->A;
    const DevCSR& AT = M->AT;
    for (int k = n - 1; k >= 0; --k) {
        T* cur = P[(n - k) & 1];               // b_{k+1}
        T* out = P[(n + 1 - k) & 1];           // in: b_{k+2}; out: b_k (or the result at k = 0)
        StepArgs<T> sa{};
        sa.ldv = ldv;
        sa.nvec = nvec;
        sa.nchunks = (nvec + G - 1) / G;
        sa.alpha = (T)g.alpha;
        sa.beta = (T)g.beta;
        sa.B = ncols;
        int nb = 0;
        if (g.gram) {
            StepArgs<T> pa = sa;
            set_operand(pa, A, valA);
            pa.vgather = cur; pa.vcur = nullptr; pa.vprev_out = M->ws_w.as<T>(); pa.mode = 2;
            set_split(pa, M->plan_A, M->ws_seg.as<T>());
            if ((rc = launch_step<T>(G, pa, g.max_main, g.max_long, M->num_sms, &nb, s))) return rc;
            set_operand(sa, AT, valAT);
            sa.vgather = M->ws_w.as<T>();
            set_split(sa, M->plan_AT, M->ws_seg.as<T>());
        } else {
            set_operand(sa, A, valA);
            sa.vgather = cur;
            set_split(sa, M->plan_A, M->ws_seg.as<T>());
        }
        sa.vcur = cur;
        sa.vprev_out = out;
        sa.mode = 3;
        sa.addv = X;
        sa.coef = (T)c[k];
        sa.m1 = k > 0 ? T(2) : T(1);
        if ((rc = launch_step<T>(G, sa, g.max_main, g.max_long, M->num_sms, &nb, s))) return rc;
    }
    T* res = P[(n + 1) & 1];
    if (res != Y) MLT_CUDA_TRY(cudaMemcpyAsync(Y, res, (size_t)total * sizeof(T), cudaMemcpyDeviceToDevice, s));
    return MLT_OK;
}

int poly_apply_block(mlt_matrix* M, double a, double b, const double* c, int n, const double* X, double* Y, int ldv,
                     int ncols, double* P0, double* P1, cudaStream_t s)
{
    return poly_apply_block_t<double>(M, a, b, c, n, X, Y, ldv, ncols, P0, P1, s);
}

int poly_apply_block_f32(mlt_matrix* M, double a, double b, const double* c, int n, const float* X, float* Y,
                         int ldv, int ncols, float* P0, float* P1, cudaStream_t s)
{
    return poly_apply_block_t<float>(M, a, b, c, n, X, Y, ldv, ncols, P0, P1, s);
}

// Doubling moments of an explicit FP64 block: V0 holds the start vectors (row
// stride ldv, columns >= cols zero) and V1 is scratch of the same size, both
// overwritten; with df the steps run in double-float pairs.  After K steps dots[k][0][c] = V_{k+1}.V_{k+1} and
// dots[k][1][c] = V_{k+1}.V_k for column c (device, in the handle's scratch).
int moments_block(mlt_matrix* M, double a, double b, double* V0, double* V1, int ldv, int cols, int K,
                  const double** dots_dev, bool df, cudaStream_t s)
{
    GroupCtx g;
    int rc;
    if ((rc = block_ctx(M, ldv, cols, K, a, b, g, s))) return rc;
    std::vector<int> act(std::max(K, 1), cols);
    MomentPlan plan{};
    plan.dim = g.d;
    plan.B = cols;
    plan.ldv = ldv;
    plan.K = K;
    plan.act = act.data();
    plan.direct = 0;
    if (df) {
        // the start block becomes double-float pairs in place (both 8 bytes an entry)
        if ((rc = ensure_df_values(M, s))) return rc;
        const int64_t n = g.d * (int64_t)ldv;
        const int nb = (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 16LL * M->num_sms));
        if (ldv & 1) return MLT_EINVAL;
        df64* W0 = reinterpret_cast<df64*>(V0);
        {
            ProfScope ps("to_df", s);
            to_df_kernel<<<nb, 256, 0, s>>>(V0, n);
        }
        MLT_CUDA_TRY(cudaGetLastError());
        df64* V[2] = {W0, reinterpret_cast<df64*>(V1)};
        if ((rc = run_steps<df64>(M, plan, g, 0, K, V, M->ws_w.as<df64>(), M->ws_seg.as<df64>(), s))) return rc;
    } else {
        double* V[2] = {V0, V1};
        if ((rc = run_steps<double>(M, plan, g, 0, K, V, M->ws_w.as<double>(), M->ws_seg.as<double>(), s)))
            return rc;
    }
    *dots_dev = g.dots;
    return MLT_OK;
}

int ensure_df_values(mlt_matrix* M, cudaStream_t s)
{
    auto conv = [&](DevCSR& C, void*& own) -> int {
        if (C.valdf || !C.val64 || C.nnz == 0) return MLT_OK;
        df64* p = nullptr;
        cudaError_t e = pool_malloc((void**)&p, (size_t)C.nnz * sizeof(df64), s);
        if (e != cudaSuccess) return fail(MLT_ENOMEM, "device allocation (double-float values) failed");
        const int nb = (int)std::min<int64_t>((C.nnz + 255) / 256, 16LL * M->num_sms);
        ProfScope ps("to_df", s);
        to_df_values_kernel<<<std::max(nb, 1), 256, 0, s>>>(C.val64, p, C.nnz);
        MLT_CUDA_TRY(cudaGetLastError());
        own = p;
        C.valdf = p;
        return MLT_OK;
    };
    int rc = conv(M->A, M->own_val_df);
    if (rc) return rc;
    if (M->perm && (rc = conv(M->P, M->own_p_val_df))) return rc;
    if (M->flags & MLT_GRAM) rc = conv(M->AT, M->own_t_val_df);
    return rc;
}

int ensure_fp32_values(mlt_matrix* M, cudaStream_t s)
{
    auto conv = [&](DevCSR& C, void*& own) -> int {
        if (C.val32 || !C.val64 || C.nnz == 0) return MLT_OK;
        float* p = nullptr;
        cudaError_t e = pool_malloc((void**)&p, (size_t)C.nnz * sizeof(float), s);
        if (e != cudaSuccess) return fail(MLT_ENOMEM, "device allocation (fp32 values) failed");
        const int nb = (int)std::min<int64_t>((C.nnz + 255) / 256, 16LL * M->num_sms);
        ProfScope ps("to_float", s);
        to_float_kernel<<<std::max(nb, 1), 256, 0, s>>>(C.val64, p, C.nnz);
        MLT_CUDA_TRY(cudaGetLastError());
        own = p;
        C.val32 = p;
        return MLT_OK;
    };
    int rc = conv(M->A, M->own_val32);
    if (rc) return rc;
    if (M->perm && (rc = conv(M->P, M->own_p_val32))) return rc;
    if (M->flags & MLT_GRAM) rc = conv(M->AT, M->own_t_val32);
    return rc;
}

int run_moments_group(mlt_matrix* M, int precision, const MomentPlan& plan, double a, double b,
                      uint64_t seed, double* mu_dev, int64_t ld_mu, int* err_flag, cudaStream_t s,
                      bool alloc_only)
{
    if (precision == MLT_PREC_DF64)
        return run_group_df(M, plan, a, b, seed, mu_dev, ld_mu, err_flag, s, alloc_only);
    // FP64: no FP32 steps; FP32: all steps FP32; mixed: FP32 for the first k steps
    int ks = 0;
    if (precision == MLT_PREC_FP32) ks = plan.K;
    else if ((precision & 0xFF) == MLT_PREC_MIXED) ks = precision >> 8;
    return run_group(M, plan, ks, a, b, seed, mu_dev, ld_mu, err_flag, s, alloc_only);
}

}  // namespace mlt

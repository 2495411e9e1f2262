// The fixed work split of one CSR operand for the moment engine (SpmmPlan),
// built on the device once per operand.
//
// Rows cost kPlanRowCost units plus one per entry; the unit axis is cut into about
// kChunksPerSm chunks per SM of Uc units each (8 to 4096): with the resident
// grid dealing them round-robin, the rows being worked on at any moment form a
// band of about 1/(kChunksPerSm/32) of the matrix.  The plan holds the first
// row of every chunk, and the segment table of rows longer than Ul = max(Uc,
// kPlanLongRow).
//
// Segments are dealt out in the order of their first column, in windows of
// kSegWindow columns (row order within a window).  Where a row's columns are
// sorted, the segments in flight at any moment gather from one narrow band of
// columns, and a vector row that several long rows share is read from L2
// rather than DRAM by all but the first.  (The relabelled operator keeps each
// row's entries in their original order, so there the bands are wider; the
// order still measured 3-4% faster for FP32 and double-float steps on the
// scale-22 graph.)  The order only decides when a segment runs; its partial
// product, and the order in which a row's segments are added, do not change.
//
// One prefix scan over the rows numbers the long rows and their segments, each
// chunk finds its first row by bisection, a stable radix sort orders the
// segments.  0.07 ms of kernels for the 48^3 stencil, where the same plan built
// on the host from a copy of the row pointers took 0.34 ms of the first call on
// a handle.  Two synchronisations, for the sizes and before the plan is marked
// ready; the second costs 0.02 ms of that call (4.20 -> 4.22 ms).
#include <cuda_runtime.h>

#include <cub/cub.cuh>
#include <thrust/iterator/counting_iterator.h>

#include <algorithm>

#include "mlt_internal.h"

namespace mlt {
namespace {

constexpr int kSegBits = 40;              // scan words: long rows above, segments below
constexpr uint64_t kSegMask = (1ull << kSegBits) - 1;
constexpr int kImbBlocks = 2048;          // row blocks sampled per imbalance figure
constexpr int32_t kSegWindow = 16384;     // column window of the segment dealing order
constexpr int kSegKeyBits = 17;           // columns are below 2^31

// Units of a work chunk.
int64_t chunk_units(int64_t nnz, int64_t nrows, int num_sms)
{
    return std::max<int64_t>(8, std::min<int64_t>(4096, (nnz + kPlanRowCost * nrows) / (kChunksPerSm * num_sms)));
}

struct PlanCounts {
    unsigned long long worst[3], total[3];   // imbalance sums (see imbalance_kernel)
    unsigned long long nhuge;
};

// x[r] = (1, number of segments) of a long row, 0 of another and of r = n.
__global__ void long_rows_kernel(const int64_t* __restrict__ rp, int64_t n, int64_t Ul, uint64_t* __restrict__ x,
                                 PlanCounts* counts)
{
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r <= n; r += (int64_t)gridDim.x * blockDim.x) {
        const int64_t deg = r < n ? rp[r + 1] - rp[r] : 0;
        const int64_t segs = deg > Ul ? (deg - 1) / Ul + 1 : 0;
        x[r] = segs ? (1ull << kSegBits) | (uint64_t)segs : 0ull;
        if (segs >= kHugeSegs) atomicAdd(&counts->nhuge, 1ull);
    }
}

// For R = 2, 4, 8 neighbouring rows (blockIdx.y): the sums over up to
// kImbBlocks evenly spaced blocks of R times the longest row and of all rows,
// in FP64 instructions (entries + 4 for the update and the dots); rows cut into
// segments do not count.  Integer sums, so the atomics' order does not matter.
__global__ void imbalance_kernel(const int64_t* __restrict__ rp, int64_t n, int64_t Ul, PlanCounts* counts)
{
    const int R = 2 << blockIdx.y;
    const int64_t blocks = n / R, step = max((int64_t)1, blocks / kImbBlocks);
    const int64_t q = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) * step;
    if (q >= blocks) return;
    int64_t mx = 0, sum = 0;
    for (int64_t r = q * R; r < q * R + R; ++r) {
        const int64_t deg = rp[r + 1] - rp[r], c = deg <= Ul ? deg + 4 : 0;
        mx = max(mx, c);
        sum += c;
    }
    atomicAdd(&counts->worst[blockIdx.y], (unsigned long long)(mx * R));
    atomicAdd(&counts->total[blockIdx.y], (unsigned long long)sum);
}

// first[c]: the first row whose first unit lies in chunk c or later (n past the last).
__global__ void chunk_first_kernel(const int64_t* __restrict__ rp, int64_t n, int64_t nch, int64_t Uc,
                                   int32_t* __restrict__ first)
{
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c <= nch; c += (int64_t)gridDim.x * blockDim.x) {
        int64_t lo = 0, hi = n;
        if (c == nch) lo = n;
        while (lo < hi) {
            const int64_t mid = (lo + hi) >> 1;
            if (rp[mid] + kPlanRowCost * mid < c * Uc) lo = mid + 1;
            else hi = mid;
        }
        first[c] = (int32_t)lo;
    }
}

// The tables of the long rows from the scanned words x: row, first segment, and
// per segment its row, first entry, and sort key and value for the dealing order.
__global__ void segments_kernel(const int64_t* __restrict__ rp, const int32_t* __restrict__ col, int64_t n, int64_t Ul,
                                const uint64_t* __restrict__ x, SpmmPlan P, uint32_t* __restrict__ key,
                                int32_t* __restrict__ id)
{
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r <= n; r += (int64_t)gridDim.x * blockDim.x) {
        const int64_t li = (int64_t)(x[r] >> kSegBits);
        int64_t s = (int64_t)(x[r] & kSegMask);
        if (r == n) {
            P.long_seg0[li] = s;
            continue;
        }
        const int64_t beg = rp[r], end = rp[r + 1];
        if (end - beg <= Ul) continue;
        P.long_rows[li] = (int32_t)r;
        P.long_seg0[li] = s;
        for (int64_t k = beg; k < end; k += Ul, ++s) {
            P.seg_row[s] = (int32_t)r;
            P.seg_k0[s] = k;
            key[s] = (uint32_t)(col[k] / kSegWindow);
            id[s] = (int32_t)s;
        }
    }
}

struct IsHuge {
    const int64_t* long_seg0;
    __device__ bool operator()(int32_t i) const { return long_seg0[i + 1] - long_seg0[i] >= kHugeSegs; }
};

}  // namespace

int ensure_spmm_plan(mlt_matrix* M, const DevCSR& C, SpmmPlan& P, cudaStream_t s)
{
    if (P.ready) return MLT_OK;
    const int64_t n = C.nrows, units = C.nnz + kPlanRowCost * n;
    const int64_t Uc = chunk_units(C.nnz, n, M->num_sms), Ul = std::max<int64_t>(Uc, kPlanLongRow);
    const int64_t nch = std::max<int64_t>(1, (units + Uc - 1) / Uc);
    const int grid = (int)std::min<int64_t>((std::max(n, nch) + 1 + 255) / 256, 16LL * M->num_sms);
    void *scan = nullptr, *sort = nullptr;   // scratch of the two phases, freed in stream order
    auto done = [&](int rc) {
        if (scan) cudaFreeAsync(scan, s);
        if (sort) cudaFreeAsync(sort, s);
        return rc;
    };
    auto oom = [&]() {
        cudaGetLastError();
        return done(fail(MLT_ENOMEM, "device allocation (work split) failed"));
    };
    auto check = [&](cudaError_t e, const char* what) { return e == cudaSuccess ? MLT_OK : done(cuda_fail(e, what)); };
    int rc;
    // sizes: the long rows and their segments, the imbalance figures
    size_t tmp = 0;
    if ((rc = check(cub::DeviceScan::ExclusiveSum(nullptr, tmp, (uint64_t*)nullptr, (uint64_t*)nullptr, n + 1, s),
                    "work split")))
        return rc;
    const size_t xb = ((size_t)(n + 1) * sizeof(uint64_t) + 255) & ~(size_t)255;
    if (pool_malloc(&scan, 2 * xb + 256 + tmp, s) != cudaSuccess) return oom();
    uint64_t* x = static_cast<uint64_t*>(scan);
    uint64_t* xs = reinterpret_cast<uint64_t*>(static_cast<char*>(scan) + xb);
    PlanCounts* counts = reinterpret_cast<PlanCounts*>(static_cast<char*>(scan) + 2 * xb);
    void* ct = static_cast<char*>(scan) + 2 * xb + 256;
    PlanCounts h{};
    uint64_t last = 0;
    {
        ProfScope ps("work_split", s);
        cudaError_t e = cudaMemsetAsync(counts, 0, sizeof(PlanCounts), s);
        long_rows_kernel<<<grid, 256, 0, s>>>(C.rowptr, n, Ul, x, counts);
        imbalance_kernel<<<dim3((2 * kImbBlocks + 255) / 256, 3), 256, 0, s>>>(C.rowptr, n, Ul, counts);
        if (e == cudaSuccess) e = cudaGetLastError();
        if (e == cudaSuccess) e = cub::DeviceScan::ExclusiveSum(ct, tmp, x, xs, n + 1, s);
        if (e == cudaSuccess) e = cudaMemcpyAsync(&h, counts, sizeof(h), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaMemcpyAsync(&last, xs + n, sizeof(last), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if ((rc = check(e, "work split"))) return rc;
    }
    const int64_t nseg = (int64_t)(last & kSegMask), nlong = (int64_t)(last >> kSegBits), nhuge = (int64_t)h.nhuge;
    const size_t bytes = (size_t)(nseg + nlong + 1) * sizeof(int64_t) +
                         (size_t)(2 * nseg + nlong + nch + 1 + nhuge) * sizeof(int32_t) + 64;
    if (!P.mem && pool_malloc(&P.mem, bytes, s) != cudaSuccess) {
        P.mem = nullptr;
        return oom();
    }
    P.seg_k0 = static_cast<int64_t*>(P.mem);
    P.long_seg0 = P.seg_k0 + nseg;
    P.seg_row = reinterpret_cast<int32_t*>(P.long_seg0 + nlong + 1);
    P.long_rows = P.seg_row + nseg;
    P.seg_order = P.long_rows + nlong;
    P.first = P.seg_order + nseg;
    P.huge = P.first + nch + 1;
    // tables, the dealing order, the list of huge rows
    size_t tsort = 0, tsel = 0;
    int32_t* none = nullptr;
    cudaError_t e = cudaSuccess;
    if (nseg)
        e = cub::DeviceRadixSort::SortPairs(nullptr, tsort, (uint32_t*)nullptr, (uint32_t*)nullptr, none, none, (int)nseg,
                                            0, kSegKeyBits, s);
    if (e == cudaSuccess && nhuge)
        e = cub::DeviceSelect::If(nullptr, tsel, thrust::counting_iterator<int32_t>(0), none, none, (int)nlong,
                                  IsHuge{nullptr}, s);
    if ((rc = check(e, "work split"))) return rc;
    const size_t kb = ((size_t)std::max<int64_t>(nseg, 1) * sizeof(uint32_t) + 255) & ~(size_t)255;
    if (pool_malloc(&sort, 3 * kb + 256 + std::max(tsort, tsel), s) != cudaSuccess) return oom();
    uint32_t* key = static_cast<uint32_t*>(sort);
    uint32_t* key2 = reinterpret_cast<uint32_t*>(static_cast<char*>(sort) + kb);
    int32_t* id = reinterpret_cast<int32_t*>(static_cast<char*>(sort) + 2 * kb);
    int32_t* nsel = reinterpret_cast<int32_t*>(static_cast<char*>(sort) + 3 * kb);
    ct = static_cast<char*>(sort) + 3 * kb + 256;
    {
        ProfScope ps("work_split", s);
        chunk_first_kernel<<<grid, 256, 0, s>>>(C.rowptr, n, nch, Uc, P.first);
        segments_kernel<<<grid, 256, 0, s>>>(C.rowptr, C.col, n, Ul, xs, P, key, id);
        e = cudaGetLastError();
        if (e == cudaSuccess && nseg)
            e = cub::DeviceRadixSort::SortPairs(ct, tsort, key, key2, id, P.seg_order, (int)nseg, 0, kSegKeyBits, s);
        if (e == cudaSuccess && nhuge)
            e = cub::DeviceSelect::If(ct, tsel, thrust::counting_iterator<int32_t>(0), P.huge, nsel, (int)nlong,
                                      IsHuge{P.long_seg0}, s);
    }
    // a later call may use the plan on another stream: complete before it is ready
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if ((rc = check(e, "work split"))) return rc;
    for (int i = 0; i < 3; ++i) P.imb[i] = h.total[i] ? (double)h.worst[i] / (double)h.total[i] : 1.0;
    P.nch = nch;
    P.Uc = Uc;
    P.Ul = Ul;
    P.nseg = nseg;
    P.nlong = (int)nlong;
    P.nhuge = (int)nhuge;
    P.ready = true;
    return done(MLT_OK);
}

}  // namespace mlt

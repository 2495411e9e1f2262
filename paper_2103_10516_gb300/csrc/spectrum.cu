// Spectrum interval by Lanczos.  The affine map of Section 2.2 needs an
// interval containing the spectrum, and the paper only asks for a rough
// estimate of the extreme eigenvalues.  k steps of the Lanczos recurrence
//   w = A q_j - alpha_j q_j - beta_{j-1} q_{j-1},  beta_j = |w|,  q_{j+1} = w / beta_j
// give a tridiagonal T_k whose extreme eigenvalues (Ritz values) theta approach
// those of A from inside; each Ritz pair's residual |A y - theta y| equals
// beta_k |s_k| (s the eigenvector of T_k, s_k its last entry), and an interval
// of half-width |residual| around theta holds an eigenvalue of A.  The bounds
// returned are theta_min - r_min and theta_max + r_max, widened by 1% of their
// magnitude.  The T_k eigenvalues come from Sturm-sequence bisection and their
// eigenvectors from inverse iteration, both on the host (k is small).
#include <cuda_runtime.h>

#include <cub/cub.cuh>

#include <algorithm>
#include <cmath>
#include <vector>

#include "mlt_internal.h"
#include "rng.cuh"

namespace mlt {
namespace {

constexpr int kLzThreads = 256;
constexpr int kLzBatch = 8;      // entries a thread has in flight
constexpr double kSortWork = 64e6;   // see sorted_rows

__global__ void start_vector_kernel(double* q, int64_t d, uint64_t seedmix, double inv_norm)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < d; i += (int64_t)gridDim.x * blockDim.x)
        q[i] = probe_negative(seedmix, 0, (uint64_t)i) ? -inv_norm : inv_norm;
}

// The block's sum of s, in lane order then warp order, to part[blockIdx.x].
__device__ __forceinline__ void block_partial(double s, double* __restrict__ part)
{
    __shared__ double sh[32];
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sh[w];
        part[blockIdx.x] = t;
    }
}

// part[block] = partial sum of x[i] y[i] over this block's indices
__global__ void dot_kernel(const double* __restrict__ x, const double* __restrict__ y, int64_t d,
                           double* __restrict__ part)
{
    double s = 0.0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < d; i += (int64_t)gridDim.x * blockDim.x)
        s = fma(x[i], y[i], s);
    block_partial(s, part);
}

// w = w - alpha q - beta p and part[block] = partial sum of the new w[i]^2
__global__ void axpy_dot_kernel(double* __restrict__ w, const double* __restrict__ q, const double* __restrict__ p,
                                int64_t d, double alpha, double beta, double* __restrict__ part)
{
    double s = 0.0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < d; i += (int64_t)gridDim.x * blockDim.x) {
        const double v = fma(-beta, p[i], fma(-alpha, q[i], w[i]));
        w[i] = v;
        s = fma(v, v, s);
    }
    block_partial(s, part);
}

__global__ void scale_kernel(double* __restrict__ dst, const double* __restrict__ src, int64_t d, double f)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < d; i += (int64_t)gridDim.x * blockDim.x)
        dst[i] = src[i] * f;
}

// ---- y = C x for one FP64 vector ----------------------------------------------
//
// A thread sums one row (or one segment of the operand's work split, of a row
// longer than a segment), entry by entry in storage order.  Bound: FP64
// additions (1/64 of the FP32 rate: 59 us for the 31 M entries of a scale-20
// R-MAT graph, if every lane of a warp adds) and one L1 lookup per gathered
// entry (31 M / 152 SMs, about 110 us); the vectors stay in L2.  Lanes of one
// warp must therefore sum equal lengths, which the rows of a graph in storage
// order do not have: there, with a lane per run of rows (the moment step's
// kernel at one column), the same product took 966 us; in order of decreasing
// length (sorted_rows) it takes 140 us.  A tree over several lanes per row would
// spend 32 FP64 lanes on each level, and would change the sums: the residuals of
// converged Ritz pairs are rounding noise, so the interval's last digits follow
// the order of every sum, and storage order is kept.
struct LzOperand {
    const int64_t* rowptr = nullptr;
    const int32_t* col = nullptr;
    const double* val = nullptr;
    int64_t n = 0, nnz = 0;
    int vec = 0;                     // col is 16-byte aligned
    const int32_t* order = nullptr;  // rows by decreasing length, or null (storage order)
    // the work split's long rows and their segments
    int64_t Ul = 0, nseg = 0, nlong = 0;
    const int32_t* seg_row = nullptr;
    const int64_t* seg_k0 = nullptr;
    const int32_t* long_rows = nullptr;
    const int64_t* long_seg0 = nullptr;
    double* part = nullptr;          // [nseg] segment sums
};

template <bool PAT>
__device__ __forceinline__ double span_sum(const LzOperand& C, const double* __restrict__ x, int k0, int k1)
{
    double s = 0.0;
    const bool vec = PAT && C.vec;
    // a batch may reach past 2^31 - 1: its slots are compared with the entries left
    const int first = vec ? k0 & ~3 : k0;
    const int tail = (int)min(C.nnz - k1, (int64_t)kLzBatch);   // entries after the span
    const int32_t* col = C.col + first;
    const double* val = PAT ? nullptr : C.val + first;
    int lead = k0 - first;
    for (int left = k1 - first; left > 0; left -= kLzBatch, lead = 0, col += kLzBatch) {
        int c[kLzBatch];
        double v[kLzBatch], xv[kLzBatch];
        if (vec && left + tail >= kLzBatch) {
#pragma unroll
            for (int u = 0; u < kLzBatch; u += 4) {
                const int4 t = __ldg(reinterpret_cast<const int4*>(col + u));
                c[u] = t.x;
                c[u + 1] = t.y;
                c[u + 2] = t.z;
                c[u + 3] = t.w;
            }
        } else {
#pragma unroll
            for (int u = 0; u < kLzBatch; ++u) c[u] = __ldg(col + min(u, left - 1));
        }
#pragma unroll
        for (int u = 0; u < kLzBatch; ++u) {
            const bool in = u >= lead && u < left;
            xv[u] = in ? __ldg(x + c[u]) : 0.0;
            v[u] = !PAT && in ? __ldg(val + u) : 1.0;
        }
        if constexpr (!PAT) val += kLzBatch;
#pragma unroll
        for (int u = 0; u < kLzBatch; ++u)
            if (u >= lead && u < left) s = PAT ? s + xv[u] : fma(v[u], xv[u], s);
    }
    return s;
}

template <bool PAT>
__global__ void __launch_bounds__(kLzThreads) lz_segments_kernel(LzOperand C, const double* __restrict__ x)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= C.nseg) return;
    const int64_t k0 = C.seg_k0[i];
    C.part[i] = span_sum<PAT>(C, x, (int)k0, (int)min(k0 + C.Ul, C.rowptr[C.seg_row[i] + 1]));
}

// The first nlong threads add a long row's segments each, the others take a row.
template <bool PAT>
__global__ void __launch_bounds__(kLzThreads) lz_rows_kernel(LzOperand C, const double* __restrict__ x,
                                                             double* __restrict__ y)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x - C.nlong;
    if (i >= C.n) return;
    if (i >= 0) {
        const int64_t r = C.order ? C.order[i] : i;
        const int k0 = (int)C.rowptr[r], k1 = (int)C.rowptr[r + 1];
        if (k1 - k0 <= C.Ul) y[r] = span_sum<PAT>(C, x, k0, k1);
        return;
    }
    const int64_t l = i + C.nlong;
    const int s0 = (int)C.long_seg0[l], s1 = (int)C.long_seg0[l + 1];
    double acc = 0.0;
    for (int s = s0; s < s1; s += kLzBatch) {
        double p[kLzBatch];
#pragma unroll
        for (int u = 0; u < kLzBatch; ++u) p[u] = s + u < s1 ? C.part[s + u] : 0.0;
#pragma unroll
        for (int u = 0; u < kLzBatch; ++u)
            if (s + u < s1) acc += p[u];
    }
    y[C.long_rows[l]] = acc;
}

__global__ void lz_keys_kernel(const int64_t* __restrict__ rp, int64_t n, uint32_t* __restrict__ key,
                               int32_t* __restrict__ id)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        key[i] = ~(uint32_t)(rp[i + 1] - rp[i]);
        id[i] = (int32_t)i;
    }
}

// Whether a call of k products sorts the operand's rows by length: where the
// lanes that would wait for longer rows (entries x (imbalance - 1), of 8
// neighbouring rows) over the call outweigh a sort of 20 to 60 us.  Sorted
// against storage order, R-MAT graphs: that product at 7 million (scale 14, 10
// steps) 802 against 744 us a call, 52 (scale 15, 40 steps) 3042 against 2958,
// 62 (scale 18, 5 steps) 626 against 605, 65 (scale 17, 10 steps) 1020 against
// 1069, 114 (scale 16, 40 steps) 3074 against 3290, 2175 (scale 20, 40 steps)
// 7870 against 11724.  Even rows are never sorted: 2 steps on the 48^3 stencil
// 175 against 109.
bool sorted_rows(const DevCSR& C, const SpmmPlan& P, int k)
{
    return P.imb[2] > kEvenRows && (double)k * C.nnz * (P.imb[2] - 1.0) > kSortWork;
}

cudaError_t lz_temp_bytes(int n, size_t* bytes)
{
    return cub::DeviceRadixSort::SortPairs(nullptr, *bytes, (uint32_t*)nullptr, (uint32_t*)nullptr, (int32_t*)nullptr,
                                           (int32_t*)nullptr, n);
}

size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }

// Workspace of one operand: segment sums and, when its rows are sorted, their
// order; the sort's keys, ids and temporary storage share one region (`tmp`)
// between operands.
size_t lz_operand_bytes(const DevCSR& C, const SpmmPlan& P, bool sorted)
{
    return align256((size_t)P.nseg * 8) + (sorted ? align256((size_t)C.nrows * 4) : 0);
}

int lz_setup(mlt_matrix* M, const DevCSR& C, const SpmmPlan& P, const int32_t* order, bool sorted, LzOperand& L,
             char* mem, char* tmp, size_t cub_bytes, cudaStream_t s)
{
    const int64_t n = C.nrows;
    L.rowptr = C.rowptr;
    L.col = C.col;
    L.val = C.val64;
    L.n = n;
    L.nnz = C.nnz;
    L.vec = (reinterpret_cast<uintptr_t>(C.col) & 15) == 0;
    L.Ul = P.Ul;
    L.nseg = P.nseg;
    L.nlong = P.nlong;
    L.seg_row = P.seg_row;
    L.seg_k0 = P.seg_k0;
    L.long_rows = P.long_rows;
    L.long_seg0 = P.long_seg0;
    L.part = reinterpret_cast<double*>(mem);
    L.order = order;
    if (!sorted) return MLT_OK;
    int32_t* ord = reinterpret_cast<int32_t*>(mem + align256((size_t)P.nseg * 8));
    uint32_t* key = reinterpret_cast<uint32_t*>(tmp);
    uint32_t* key2 = reinterpret_cast<uint32_t*>(tmp + align256((size_t)n * 4));
    int32_t* id = reinterpret_cast<int32_t*>(tmp + 2 * align256((size_t)n * 4));
    void* ct = tmp + 3 * align256((size_t)n * 4);
    const int g = (int)std::min<int64_t>((n + 255) / 256, 16LL * M->num_sms);
    ProfScope ps("lanczos_setup", s);
    lz_keys_kernel<<<g, 256, 0, s>>>(C.rowptr, n, key, id);
    MLT_CUDA_TRY(cudaGetLastError());
    MLT_CUDA_TRY(cub::DeviceRadixSort::SortPairs(ct, cub_bytes, key, key2, id, ord, (int)n, 0, 32, s));
    L.order = ord;
    return MLT_OK;
}

int lz_product(const LzOperand& C, const double* x, double* y, cudaStream_t s)
{
    if (C.n == 0) return MLT_OK;
    const unsigned gs = (unsigned)((C.nseg + kLzThreads - 1) / kLzThreads);
    const unsigned gr = (unsigned)((C.n + C.nlong + kLzThreads - 1) / kLzThreads);
    ProfScope ps("lanczos_product", s);
    if (C.val) {
        if (gs) lz_segments_kernel<false><<<gs, kLzThreads, 0, s>>>(C, x);
        lz_rows_kernel<false><<<gr, kLzThreads, 0, s>>>(C, x, y);
    } else {
        if (gs) lz_segments_kernel<true><<<gs, kLzThreads, 0, s>>>(C, x);
        lz_rows_kernel<true><<<gr, kLzThreads, 0, s>>>(C, x, y);
    }
    MLT_CUDA_TRY(cudaGetLastError());
    return MLT_OK;
}

// Number of eigenvalues of the tridiagonal (dg, e) below x (Sturm sequence).
int count_below(const std::vector<double>& dg, const std::vector<double>& e, double x)
{
    const int n = (int)dg.size();
    int cnt = 0;
    double q = dg[0] - x;
    if (q < 0) ++cnt;
    for (int i = 1; i < n; ++i) {
        if (q == 0.0) q = 1e-300;
        q = (dg[i] - x) - e[i - 1] * e[i - 1] / q;
        if (q < 0) ++cnt;
    }
    return cnt;
}

// The j-th smallest eigenvalue (0-based) by bisection on the Gershgorin interval.
double bisect_eigenvalue(const std::vector<double>& dg, const std::vector<double>& e, int j)
{
    const int n = (int)dg.size();
    double lo = 1e300, hi = -1e300;
    for (int i = 0; i < n; ++i) {
        const double r = (i > 0 ? std::fabs(e[i - 1]) : 0.0) + (i < n - 1 ? std::fabs(e[i]) : 0.0);
        lo = std::min(lo, dg[i] - r);
        hi = std::max(hi, dg[i] + r);
    }
    for (int it = 0; it < 200 && hi - lo > 1e-15 * std::max(std::fabs(lo), std::fabs(hi)) + 1e-300; ++it) {
        const double mid = 0.5 * (lo + hi);
        if (count_below(dg, e, mid) > j) hi = mid;
        else lo = mid;
    }
    return 0.5 * (lo + hi);
}

// Last entry of the unit eigenvector for eigenvalue theta (inverse iteration
// with a tridiagonal solve of (T - theta I) v = b, three sweeps).
double eigvec_last(const std::vector<double>& dg, const std::vector<double>& e, double theta)
{
    const int n = (int)dg.size();
    std::vector<double> v(n, 1.0), c(n), dd(n);
    const double shift = theta + 1e-12 * (std::fabs(theta) + 1.0);
    for (int sweep = 0; sweep < 3; ++sweep) {
        // forward elimination (Thomas), tiny pivots replaced by a small number
        for (int i = 0; i < n; ++i) {
            double piv = dg[i] - shift - (i > 0 ? e[i - 1] * c[i - 1] : 0.0);
            if (std::fabs(piv) < 1e-300) piv = 1e-300;
            c[i] = i < n - 1 ? e[i] / piv : 0.0;
            dd[i] = (v[i] - (i > 0 ? e[i - 1] * dd[i - 1] : 0.0)) / piv;
        }
        for (int i = n - 1; i >= 0; --i) v[i] = dd[i] - (i < n - 1 ? c[i] * v[i + 1] : 0.0);
        double nrm = 0.0;
        for (double x : v) nrm += x * x;
        nrm = std::sqrt(nrm);
        if (!(nrm > 0.0) || !std::isfinite(nrm)) return 1.0;
        for (double& x : v) x /= nrm;
    }
    return v[n - 1];
}

// The sum of the nblk block partials, in block order.
double sum_sync(const double* part, int nblk, std::vector<double>& h, cudaStream_t s, int* rc)
{
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(h.data(), part, nblk * sizeof(double), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) {
        *rc = cuda_fail(e, "lanczos dot");
        return 0.0;
    }
    double t = 0.0;
    for (int b = 0; b < nblk; ++b) t += h[b];
    return t;
}

}  // namespace

int lanczos_bounds(mlt_matrix* M, int steps, uint64_t seed, double* lo, double* hi, cudaStream_t s)
{
    const bool gram = (M->flags & MLT_GRAM) != 0;
    const int64_t d = M->dim();
    if (d < 1) return fail(MLT_EINVAL, "mlt_spectrum_bounds: empty operator");
    const int k = (int)std::min<int64_t>(std::max(steps, 2), d);
    int rc;
    const size_t vb = align256((size_t)d * sizeof(double));
    const size_t tb = gram ? align256((size_t)M->A.nrows * sizeof(double)) : 0;
    const int nblk = (int)std::max<int64_t>(1, std::min<int64_t>((d + 255) / 256, 4LL * M->num_sms));
    if ((rc = ensure_spmm_plan(M, M->A, M->plan_A, s))) return rc;
    if (gram && (rc = ensure_spmm_plan(M, M->AT, M->plan_AT, s))) return rc;
    // a relabelled handle's permutation is the order of decreasing length
    const bool sort_a = !M->perm && sorted_rows(M->A, M->plan_A, k);
    const bool sort_t = gram && sorted_rows(M->AT, M->plan_AT, k);
    const int64_t nsort = std::max(sort_a ? M->A.nrows : (int64_t)0, sort_t ? M->AT.nrows : (int64_t)0);
    size_t cub_bytes = 0;
    if (nsort) MLT_CUDA_TRY(lz_temp_bytes((int)nsort, &cub_bytes));
    const size_t ob = lz_operand_bytes(M->A, M->plan_A, sort_a);
    const size_t obt = gram ? lz_operand_bytes(M->AT, M->plan_AT, sort_t) : 0;
    if ((rc = M->ws_v[0].ensure(3 * vb + tb + align256(nblk * sizeof(double)) + ob + obt +
                                    3 * align256((size_t)nsort * 4) + align256(cub_bytes),
                                s)))
        return rc;
    char* mem = M->ws_v[0].as<char>();
    double* q_prev = reinterpret_cast<double*>(mem);
    double* q = reinterpret_cast<double*>(mem + vb);
    double* w = reinterpret_cast<double*>(mem + 2 * vb);
    double* t = reinterpret_cast<double*>(mem + 3 * vb);
    double* part = reinterpret_cast<double*>(mem + 3 * vb + tb);
    char* om = mem + 3 * vb + tb + align256(nblk * sizeof(double));
    LzOperand A, AT;
    char* tmp = om + ob + obt;
    if ((rc = lz_setup(M, M->A, M->plan_A, M->perm, sort_a, A, om, tmp, cub_bytes, s))) return rc;
    if (gram && (rc = lz_setup(M, M->AT, M->plan_AT, nullptr, sort_t, AT, om + ob, tmp, cub_bytes, s))) return rc;
    MLT_CUDA_TRY(cudaMemsetAsync(q_prev, 0, vb, s));
    const int g = (int)std::min<int64_t>((d + 255) / 256, 16LL * M->num_sms);
    {
        ProfScope ps("lanczos_vectors", s);
        start_vector_kernel<<<g, 256, 0, s>>>(q, d, seed * kGolden, 1.0 / std::sqrt((double)d));
    }
    MLT_CUDA_TRY(cudaGetLastError());
    std::vector<double> alpha, beta, h(nblk);
    double bprev = 0.0;
    for (int j = 0; j < k; ++j) {
        if (gram) {
            if ((rc = lz_product(A, q, t, s))) return rc;
            if ((rc = lz_product(AT, t, w, s))) return rc;
        } else {
            if ((rc = lz_product(A, q, w, s))) return rc;
        }
        rc = MLT_OK;
        {
            ProfScope ps("lanczos_vectors", s);
            dot_kernel<<<nblk, 256, 0, s>>>(q, w, d, part);
        }
        const double a = sum_sync(part, nblk, h, s, &rc);
        if (rc) return rc;
        {
            ProfScope ps("lanczos_vectors", s);
            axpy_dot_kernel<<<nblk, 256, 0, s>>>(w, q, q_prev, d, a, bprev, part);
        }
        const double b2 = sum_sync(part, nblk, h, s, &rc);
        if (rc) return rc;
        alpha.push_back(a);
        const double b = std::sqrt(std::max(b2, 0.0));
        beta.push_back(b);
        if (!(b > 1e-12 * (std::fabs(a) + bprev + 1e-300))) break;   // invariant subspace found
        {
            ProfScope ps("lanczos_vectors", s);
            scale_kernel<<<g, 256, 0, s>>>(q_prev, w, d, 1.0 / b);    // the next q, over q_prev
        }
        MLT_CUDA_TRY(cudaGetLastError());
        std::swap(q, q_prev);
        bprev = b;
    }
    const int n = (int)alpha.size();
    std::vector<double> e(beta.begin(), beta.begin() + (n - 1));
    const double tmin = bisect_eigenvalue(alpha, e, 0);
    const double tmax = bisect_eigenvalue(alpha, e, n - 1);
    const double blast = beta[n - 1];
    const double rmin = std::fabs(blast * eigvec_last(alpha, e, tmin));
    const double rmax = std::fabs(blast * eigvec_last(alpha, e, tmax));
    const double sc = gram ? M->scale * M->scale : M->scale;
    double a0 = (tmin - rmin) * sc, b0 = (tmax + rmax) * sc;
    if (sc < 0) std::swap(a0, b0);
    a0 -= 0.01 * std::fabs(a0);
    b0 += 0.01 * std::fabs(b0);
    if (gram) a0 = std::max(a0, 1e-6 * b0);
    *lo = a0;
    *hi = b0;
    return MLT_OK;
}

}  // namespace mlt

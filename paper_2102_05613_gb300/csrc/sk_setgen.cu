// sk_setgen.cu -- generation probabilities of sets of configurations
// (App. D.1, D.2): Pt(M) = P_gen(S | S \ M) for every subset M of an
// n-element set S, where the set grows by adding one element at a time,
// generated from a parent chosen uniformly in the current set.
//
// The recursion on the first addition,
//   Pt(M) = (1/|S \ M|) sum_{e in M} c(M, e) Pt(M \ {e}),
//   c(M, e) = sum_{p in S \ M} P_gen(e | p),
// needs only subsets with one element fewer, so the masks are processed one
// cardinality at a time, one thread per mask; a thread finds its mask by
// unranking its index in the combinatorial number system.  Three forms:
// direct (each c(M, e) summed afresh, O(n^2 2^n)), the paper's cumulative
// form (Eq. eq_rec_set_short: c(M, e) = c(M \ {f}, e) - P_gen(e | f) from
// the previous cardinality's table, f the lowest other element of M;
// O(n 2^n) work and a table of n 2^n doubles) and the block form below
// (setgen_block), the default.  Double precision (the values are products of
// up to n-1 probabilities).
#include <cuda_runtime.h>
#include <stdint.h>

#include <cstring>
#include <vector>

#include "sk_internal.h"
#include "sk_mcmcmc.h"

namespace sk {
namespace {

constexpr uint32_t kMaxSetN = 28;

__global__ void setgen_level(const double* __restrict__ Pg, const unsigned long long* __restrict__ binom, uint32_t n,
                             uint32_t m, unsigned long long count, double* __restrict__ out) {
    __shared__ double P[kMaxSetN * kMaxSetN];
    __shared__ unsigned long long C[(kMaxSetN + 1) * (kMaxSetN + 1)];
    for (uint32_t i = threadIdx.x; i < n * n; i += blockDim.x) P[i] = Pg[i];
    for (uint32_t i = threadIdx.x; i < (n + 1) * (n + 1); i += blockDim.x) C[i] = binom[i];
    __syncthreads();
    const unsigned long long idx = blockIdx.x * static_cast<unsigned long long>(blockDim.x) + threadIdx.x;
    if (idx >= count) return;
    // the idx-th m-subset in colexicographic order
    uint32_t M = 0;
    unsigned long long r = idx;
    uint32_t left = m;
    for (int b = static_cast<int>(n) - 1; b >= 0 && left; --b) {
        const unsigned long long c = C[b * (n + 1) + left];  // binom(b, left)
        if (c <= r) {
            M |= 1u << b;
            r -= c;
            --left;
        }
    }
    const uint32_t all = (n == 32u) ? 0xFFFFFFFFu : ((1u << n) - 1u);
    const uint32_t cur = all & ~M;
    double tot = 0.0;
    for (uint32_t e = 0; e < n; ++e) {
        if (!((M >> e) & 1u)) continue;
        double a = 0.0;
        for (uint32_t p = 0; p < n; ++p)
            if ((cur >> p) & 1u) a += P[e * n + p];
        tot = fma(a, out[M & ~(1u << e)], tot);
    }
    out[M] = tot / static_cast<double>(n - m);
}

// The cumulative form: as setgen_level, with c(M, e) kept at c[M n + e].
__global__ void setgen_level_cum(const double* __restrict__ Pg, const unsigned long long* __restrict__ binom,
                                 uint32_t n, uint32_t m, unsigned long long count, double* __restrict__ out,
                                 double* __restrict__ c) {
    __shared__ double P[kMaxSetN * kMaxSetN];
    __shared__ unsigned long long C[(kMaxSetN + 1) * (kMaxSetN + 1)];
    for (uint32_t i = threadIdx.x; i < n * n; i += blockDim.x) P[i] = Pg[i];
    for (uint32_t i = threadIdx.x; i < (n + 1) * (n + 1); i += blockDim.x) C[i] = binom[i];
    __syncthreads();
    const unsigned long long idx = blockIdx.x * static_cast<unsigned long long>(blockDim.x) + threadIdx.x;
    if (idx >= count) return;
    uint32_t M = 0;
    unsigned long long r = idx;
    uint32_t left = m;
    for (int b = static_cast<int>(n) - 1; b >= 0 && left; --b) {
        const unsigned long long cb = C[b * (n + 1) + left];  // binom(b, left)
        if (cb <= r) {
            M |= 1u << b;
            r -= cb;
            --left;
        }
    }
    double tot = 0.0;
    for (uint32_t e = 0; e < n; ++e) {
        if (!((M >> e) & 1u)) continue;
        const uint32_t rest = M & ~(1u << e);
        double ce;
        if (!rest) {  // c({e}, e): every other element is a parent
            ce = 0.0;
            for (uint32_t p = 0; p < n; ++p)
                if (p != e) ce += P[e * n + p];
        } else {
            const uint32_t f = static_cast<uint32_t>(__ffs(rest) - 1);
            ce = c[static_cast<size_t>(M & ~(1u << f)) * n + e] - P[e * n + f];
        }
        c[static_cast<size_t>(M) * n + e] = ce;
        tot = fma(ce, out[rest], tot);
    }
    out[M] = tot / static_cast<double>(n - m);
}

// The block form: M = (h << L) | l, L = min(n, kLow).  A CTA takes the 2^L
// masks of eight high parts h, a warp each; c(M, e) = A_e(h) + B_e(l), with A_e
// the parents among the high elements not in h (summed by the warp) and B_e
// those among the low elements not in l (a table of n 2^L doubles, copied to
// shared memory).  The elements of h come first: their terms need only out[]
// of parts with one element fewer (earlier launches: one per cardinality of
// h), read along l, so coalesced, four elements' loads at a time; then the
// elements of l, one cardinality of l at a time, the masks of all eight parts
// spread over the CTA's threads (a warp per part would issue FP64
// instructions with 1 to 20 lanes in use).  Bound: FP64 issue, an add and a
// fused multiply-add per mask and member (n = 22: 9.2e7 of them, 0.16 ms at
// 2 per clock and SM).  The cumulative form moves its n 2^n table through HBM
// twice instead, and allocates it: n = 22 2.13 ms a call (1.31 ms of kernels),
// against 0.44 ms for this one.  (L = 10 with a CTA per h: 0.52 ms, every
// launch at least 31 us of dependent table loads.)
constexpr uint32_t kLow = 6;
constexpr uint32_t kParts = 8;                     // high parts per CTA
constexpr uint32_t kBlockThreads = 32u * kParts;
constexpr uint32_t kValStride = (1u << kLow) + 2u;  // parts on different banks

// The tables: B[e 2^L + l] = sum of P[e n + p] over the low elements p not in
// l; and, with the high elements in two halves of H1 and H - H1, the same sums
// over each half, T[h n + e] and, after those 2^H1 n, T2[h n + e].  (Summed
// by every warp for itself, A cost 16 dependent FP64 adds at n = 22, a
// quarter of a warp's FP64 work.)
__global__ void setgen_tables(const double* __restrict__ P, uint32_t n, uint32_t L, uint32_t H1, double* __restrict__ B,
                              double* __restrict__ T) {
    const uint32_t H2 = n - L - H1, nB = n << L, n1 = n << H1, n2 = n << H2;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < nB + n1 + n2; i += gridDim.x * blockDim.x) {
        uint32_t e, mask, p0, bits;
        double* dst;
        if (i < nB) {
            e = i >> L, mask = i & ((1u << L) - 1u), p0 = 0u, bits = L;
            dst = B + i;
        } else {
            const uint32_t q = i - nB, second = q >= n1;
            const uint32_t x = second ? q - n1 : q;
            e = x % n, mask = x / n, p0 = second ? L + H1 : L, bits = second ? H2 : H1;
            dst = T + q;
        }
        double a = 0.0;
        for (uint32_t b = 0; b < bits; ++b)
            if (!((mask >> b) & 1u)) a += __ldg(&P[e * n + p0 + b]);
        *dst = a;
    }
}

// x / k for an integer k of at most 28 with r = 1 / k rounded: the product
// and one correction from its remainder (Markstein, IBM J. Res. Dev. 34, 1990),
// three FP64 operations; infinities pass through.  (The product alone is 5 %
// faster and rounds once more: rms error at n = 8 1.4e-16 against 1.0e-16 here
// and 1.3e-16 in the cumulative form; at n = 14 1.2e-16 here, 4.2e-16 there.)
__device__ __forceinline__ double div_small(double x, double k, double r) {
    const double q = x * r;
    if ((__double2hiint(q) & 0x7FF00000) == 0x7FF00000) return q;
    return fma(fma(-q, k, x), r, q);
}

// The `parts` = binom(n - L, k) high parts of k elements, kParts per CTA.
// order: the low masks by cardinality; binom: 29 x 29; inv[k] = 1 / k.
__global__ void __launch_bounds__(kBlockThreads) setgen_block(const double* __restrict__ T, uint32_t H1,
                                                               const double* __restrict__ Bg,
                                                               const double* __restrict__ inv,
                                                               const uint16_t* __restrict__ order,
                                                               const uint32_t* __restrict__ binom, uint32_t n,
                                                               uint32_t L, uint32_t k, uint32_t parts,
                                                               double* __restrict__ out) {
    __shared__ double B[kMaxSetN << kLow];
    __shared__ double A[kParts][kMaxSetN];
    __shared__ double val[kParts][kValStride];  // terms of h, then the part's values
    __shared__ uint16_t ord[1u << kLow];
    const uint32_t tid = threadIdx.x, lane = tid & 31u, w = tid >> 5, S = 1u << L, H = n - L;
    for (uint32_t i = tid; i < n << L; i += kBlockThreads) B[i] = __ldg(Bg + i);
    if (tid < S) ord[tid] = __ldg(order + tid);
    const uint32_t part = blockIdx.x * kParts + w;
    const bool own = part < parts;
    // the part-th k-subset of the high elements in colexicographic order
    uint32_t h = 0, r = part, left = own ? k : 0u;
    for (int b = static_cast<int>(H) - 1; b >= 0 && left; --b) {
        const uint32_t c = __ldg(&binom[b * (kMaxSetN + 1) + left]);
        if (c <= r) {
            h |= 1u << b;
            r -= c;
            --left;
        }
    }
    if (lane < n)
        A[w][lane] = __ldg(&T[(h & ((1u << H1) - 1u)) * n + lane]) + __ldg(&T[(n << H1) + (h >> H1) * n + lane]);
    __syncthreads();
    double acc0 = 0.0, acc1 = 0.0;  // masks l = lane and lane + 32
    if (own) {
        const bool on0 = lane < S, on1 = lane + 32u < S;
        uint32_t m = h;
        for (uint32_t i = 0; i < k; i += 4u) {
            uint32_t e[4];
            double x0[4], x1[4];
#pragma unroll
            for (uint32_t q = 0; q < 4u; ++q) {
                e[q] = m ? static_cast<uint32_t>(__ffs(static_cast<int>(m)) - 1) : 0u;
                x0[q] = x1[q] = 0.0;
                if (m) {
                    const double* __restrict__ x = out + (static_cast<size_t>(h ^ (1u << e[q])) << L) + lane;
                    if (on0) x0[q] = x[0];
                    if (on1) x1[q] = x[32];
                }
                m &= m - 1u;
            }
#pragma unroll
            for (uint32_t q = 0; q < 4u; ++q)
                if (i + q < k) {
                    const double a = A[w][e[q] + L];
                    const double* be = B + ((e[q] + L) << L) + lane;
                    if (on0) acc0 = fma(a + be[0], x0[q], acc0);
                    if (on1) acc1 = fma(a + be[32], x1[q], acc1);
                }
        }
        if (on0) val[w][lane] = acc0;
        if (on1) val[w][lane + 32u] = acc1;
    }
    uint32_t first = 0;
    const uint32_t pw = tid & (kParts - 1u);  // this thread's part below
    const bool pown = blockIdx.x * kParts + pw < parts;
    for (uint32_t j = 0; j <= L; ++j) {  // the low masks of j elements
        __syncthreads();
        const uint32_t cnt = __ldg(&binom[L * (kMaxSetN + 1) + j]);
        const uint32_t left_in = n - k - j;  // elements of the current set
        const uint32_t i = tid / kParts;     // binom(6, j) <= 20 masks of 32
        if (pown && i < cnt) {
            const uint32_t l = ord[first + i];
            double tot = val[pw][l];
            for (uint32_t m = l; m; m &= m - 1u) {
                const uint32_t e = static_cast<uint32_t>(__ffs(static_cast<int>(m)) - 1);
                tot = fma(A[pw][e] + B[(e << L) + l], val[pw][l ^ (1u << e)], tot);
            }
            // no element missing: 1; every element missing: 0
            val[pw][l] = k + j == 0u ? 1.0 : left_in == 0u ? 0.0 : div_small(tot, static_cast<double>(left_in), __ldg(&inv[left_in]));
        }
        first += cnt;
    }
    __syncthreads();
    if (own)
        for (uint32_t l = lane; l < S; l += 32u) out[(static_cast<size_t>(h) << L) + l] = val[w][l];
}

__global__ void setgen_ends(double* out, uint32_t all) {
    if (threadIdx.x == 0) {
        out[0] = 1.0;
        out[all] = 0.0;
    }
}

// The block form on the host side; out: 2^n doubles on the host or the device.
cudaError_t setgen_blocks(uint32_t n, const double* P, double* out, bool host, cudaStream_t st) {
    const uint32_t L = n < kLow ? n : kLow, S = 1u << L, H = n - L;
    constexpr uint32_t D = kMaxSetN + 1;
    // one upload: P, the binomials, the low masks by cardinality
    const size_t o_binom = n * n * sizeof(double), o_order = o_binom + D * D * sizeof(uint32_t);
    const uint32_t H1 = H / 2;
    const size_t o_inv = (o_order + S * sizeof(uint16_t) + 15u) & ~static_cast<size_t>(15u);
    const size_t o_B = (o_inv + D * sizeof(double) + 255u) & ~static_cast<size_t>(255u);
    std::vector<unsigned char> up(o_B, 0);
    std::memcpy(up.data(), P, o_binom);
    uint32_t* C = reinterpret_cast<uint32_t*>(up.data() + o_binom);
    for (uint32_t a = 0; a < D; ++a) {
        C[a * D] = 1;
        for (uint32_t b = 1; b <= a; ++b) C[a * D + b] = C[(a - 1) * D + b - 1] + (b < a ? C[(a - 1) * D + b] : 0);
    }
    for (uint32_t k = 1; k < D; ++k) reinterpret_cast<double*>(up.data() + o_inv)[k] = 1.0 / k;
    uint16_t* order = reinterpret_cast<uint16_t*>(up.data() + o_order);
    uint32_t at[kLow + 2] = {0};
    for (uint32_t j = 0; j <= L; ++j) at[j + 1] = at[j] + C[L * D + j];
    for (uint32_t l = 0; l < S; ++l) order[at[__builtin_popcount(l)]++] = static_cast<uint16_t>(l);
    unsigned char* d = nullptr;
    double* dout = host ? nullptr : out;
    cudaError_t e = workspace_alloc(reinterpret_cast<void**>(&d), o_B + n * (static_cast<size_t>(S) + (1u << H1) + (1u << (H - H1))) * sizeof(double), st);
    if (e == cudaSuccess && host) e = cudaMalloc(&dout, sizeof(double) << n);
    if (e == cudaSuccess) e = cudaMemcpyAsync(d, up.data(), o_B, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) {
        const double* dP = reinterpret_cast<const double*>(d);
        double* dB = reinterpret_cast<double*>(d + o_B);
        double* dT = dB + (static_cast<size_t>(n) << L);
        const uint32_t entries = n * (S + (1u << H1) + (1u << (H - H1)));
        setgen_tables<<<(entries + 127u) / 128u, 128, 0, st>>>(dP, n, L, H1, dB, dT);
        for (uint32_t k = 0; k <= H; ++k)
            setgen_block<<<(C[H * D + k] + kParts - 1u) / kParts, kBlockThreads, 0, st>>>(
                dT, H1, dB, reinterpret_cast<const double*>(d + o_inv), reinterpret_cast<const uint16_t*>(d + o_order), reinterpret_cast<const uint32_t*>(d + o_binom), n,
                L, k, C[H * D + k], dout);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess && host) e = cudaMemcpyAsync(out, dout, sizeof(double) << n, cudaMemcpyDeviceToHost, st);
    if (d) cudaFreeAsync(d, st);
    const cudaError_t e2 = cudaStreamSynchronize(st);
    if (host) cudaFree(dout);
    return e != cudaSuccess ? e : e2;
}

}  // namespace
}  // namespace sk

extern "C" sk_status sk_set_generation(uint32_t n, const double* P, double* out, uint32_t mem, uint32_t method,
                                       void* stream) {
    if (!P || !out) {
        sk::set_error_message("sk_set_generation: NULL argument");
        return SK_ERR_INVALID_ARG;
    }
    if (n < 1 || n > sk::kMaxSetN) {
        sk::set_error_message("sk_set_generation: n must be 1..28");
        return SK_ERR_INVALID_ARG;
    }
    if (mem != SK_MEM_HOST && mem != SK_MEM_DEVICE) {
        sk::set_error_message("sk_set_generation: mem must be SK_MEM_HOST or SK_MEM_DEVICE");
        return SK_ERR_INVALID_ARG;
    }
    if (method > SK_SETGEN_CUMULATIVE) {
        sk::set_error_message("sk_set_generation: method must be SK_SETGEN_AUTO, _DIRECT or _CUMULATIVE");
        return SK_ERR_INVALID_ARG;
    }
    for (uint32_t i = 0; i < n * n; ++i)
        if (!(P[i] >= 0.0) || P[i] == INFINITY) {
            sk::set_error_message("sk_set_generation: P must be finite and >= 0");
            return SK_ERR_INVALID_ARG;
        }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const size_t nmask = static_cast<size_t>(1) << n;
    if (method == SK_SETGEN_AUTO) {
        const cudaError_t e = sk::setgen_blocks(n, P, out, mem == SK_MEM_HOST, st);
        if (e == cudaSuccess) return SK_OK;
        cudaGetLastError();
        sk::set_error_message(cudaGetErrorString(e));
        return e == cudaErrorMemoryAllocation ? SK_ERR_OOM : SK_ERR_CUDA;
    }
    std::vector<unsigned long long> C((n + 1) * (n + 1), 0ull);
    for (uint32_t a = 0; a <= n; ++a) {
        C[a * (n + 1)] = 1;
        for (uint32_t b = 1; b <= a; ++b) C[a * (n + 1) + b] = C[(a - 1) * (n + 1) + b - 1] + (b < a ? C[(a - 1) * (n + 1) + b] : 0);
    }
    double* dP = nullptr;
    unsigned long long* dC = nullptr;
    double* dc = nullptr;  // the cumulative table, n 2^n doubles
    double* dout = mem == SK_MEM_DEVICE ? out : nullptr;
    cudaError_t e = cudaSuccess;
    if (method == SK_SETGEN_CUMULATIVE && n > 1) {
        e = cudaMalloc(&dc, nmask * n * sizeof(double));
        if (e != cudaSuccess) {
            cudaGetLastError();
            sk::set_error_message("sk_set_generation: no room for the cumulative table (n 2^n doubles)");
            return SK_ERR_OOM;
        }
    }
    if (e == cudaSuccess) e = cudaMalloc(&dP, n * n * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc(&dC, C.size() * sizeof(unsigned long long));
    if (e == cudaSuccess && !dout) e = cudaMalloc(&dout, nmask * sizeof(double));
    if (e == cudaSuccess) e = cudaMemcpyAsync(dP, P, n * n * sizeof(double), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(dC, C.data(), C.size() * sizeof(unsigned long long), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) {
        sk::setgen_ends<<<1, 32, 0, st>>>(dout, static_cast<uint32_t>(nmask - 1));
        e = cudaGetLastError();
    }
    for (uint32_t m = 1; m < n && e == cudaSuccess; ++m) {
        const unsigned long long count = C[n * (n + 1) + m];
        const unsigned long long blocks = (count + 255) / 256;
        if (dc)
            sk::setgen_level_cum<<<static_cast<unsigned>(blocks), 256, 0, st>>>(dP, dC, n, m, count, dout, dc);
        else
            sk::setgen_level<<<static_cast<unsigned>(blocks), 256, 0, st>>>(dP, dC, n, m, count, dout);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess && mem == SK_MEM_HOST)
        e = cudaMemcpyAsync(out, dout, nmask * sizeof(double), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    cudaFree(dP);
    cudaFree(dC);
    cudaFree(dc);
    if (mem == SK_MEM_HOST) cudaFree(dout);
    if (e != cudaSuccess) {
        cudaGetLastError();
        sk::set_error_message(cudaGetErrorString(e));
        return e == cudaErrorMemoryAllocation ? SK_ERR_OOM : SK_ERR_CUDA;
    }
    return SK_OK;
}

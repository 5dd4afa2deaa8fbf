// Device side of the coarse solve by substructuring (plan: fronts.cu).
//
// With E = R_0 A R_0^T in the plan's order, every part p with interior I and
// boundary B keeps, once the earlier stages are eliminated into its front,
//   Ainv = (S_II)^{-1}     and     W = S_II^{-1} S_IB
// as dense blocks, and E e = c is solved exactly by
//   down, stage by stage:  c_B -= W^T c_I
//   up, in reverse:        e_I  = Ainv c_I - W e_B.
// The parts of a stage are independent, so a solve is one launch per stage and
// direction (the last stage has no boundary) instead of a chain over the
// blocks of a banded factor.  What bounds it: the launches (2 x stages) and, with
// several vectors, the FP64 rate (one multiply-add per stored entry and vector,
// two per clock and SM); a warp per row keeps every load coalesced and fills
// the chip from about a thousand rows on.  Measured against the banded factor
// with 512-wide blocks and a grid barrier per block: PCG iteration on 24^3
// (n_C = 13,824, 4 stages, 5.5 M entries) 1.07 -> 0.26 ms; with eight vectors
// on 20^3 2.83 -> 0.59 ms; apply on 64^2 301 -> 117 us.
#include "amdd_internal.h"

namespace amdd {
namespace {

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// s[k] += sum over columns j = lane, lane + 32, ... < m of row[j] x_k[j] (x_k
// ldv apart): eight loads of the row in flight per lane.
template <int NB>
__device__ __forceinline__ void row_dot(const double* __restrict__ row, const double* x, int64_t ldv, int m, int nb,
                                        int lane, double* s) {
    constexpr int U = NB == 1 ? 8 : 4;
    int j = lane;
    for (; j + 32 * (U - 1) < m; j += 32 * U) {
        double a[U];
#pragma unroll
        for (int u = 0; u < U; ++u) a[u] = __ldg(row + j + 32 * u);
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int k = 0; k < NB; ++k)
                if (NB == 1 || k < nb) s[k] = fma(a[u], x[k * ldv + j + 32 * u], s[k]);
    }
    for (; j < m; j += 32) {
        const double a = __ldg(row + j);
#pragma unroll
        for (int k = 0; k < NB; ++k)
            if (NB == 1 || k < nb) s[k] = fma(a, x[k * ldv + j], s[k]);
    }
}

}  // namespace

// Lower triangle of the front of part p, columns of its interior, from the
// dense lower triangle of E (subdomain order): F[r][c] = E[max][min] of the
// two coarse unknowns.  F is zero on entry (its boundary block stays zero).
__global__ void __launch_bounds__(256) front_gather_kernel(const FrontDev* __restrict__ fr,
                                                           const int32_t* __restrict__ bnd,
                                                           const int32_t* __restrict__ perm,
                                                           const double* __restrict__ E, int64_t nE) {
    const FrontDev f = fr[blockIdx.y];
    const int n = f.m + f.nb;
    for (int r = blockIdx.x; r < n; r += gridDim.x) {
        const int64_t pr = perm[r < f.m ? f.i0 + r : bnd[f.b0 + r - f.m]];
        double* row = f.F + (size_t)r * n;
        const int cend = min(r + 1, f.m);
        for (int c = threadIdx.x; c < cend; c += blockDim.x) {
            const int64_t pc = perm[f.i0 + c];
            row[c] = E[(pr > pc ? pr : pc) * nE + (pr > pc ? pc : pr)];
        }
    }
}

void launch_front_gather(const FrontDev* fr, int nfr, const int32_t* bnd, const int32_t* perm, const double* E,
                         int64_t nE, int maxn, cudaStream_t s) {
    for (int k = 0; k < nfr; k += 32768)  // grid.y is 16 bits wide
        front_gather_kernel<<<dim3(maxn < 512 ? maxn : 512, nfr - k < 32768 ? nfr - k : 32768), 256, 0, s>>>(
            fr + k, bnd, perm, E, nE);
}

// Adds the Schur complements of the children of every front of a stage into it
// (lower triangles).  One CTA per front row; the children one after the other
// in a fixed order, so sums do not depend on the schedule.  inv[r] is the
// child's boundary row of front row r (-1: none), map its inverse.
__global__ void __launch_bounds__(128) front_extend_add_kernel(const FrontDev* __restrict__ fr,
                                                               const FrontChild* __restrict__ kids,
                                                               const int32_t* __restrict__ maps) {
    const FrontDev f = fr[blockIdx.y];
    const int n = f.m + f.nb;
    for (int r = blockIdx.x; r < n; r += gridDim.x) {
        double* row = f.F + (size_t)r * n;
        for (int k = f.kid0; k < f.kid1; ++k) {
            const FrontChild c = kids[k];
            const int lr = maps[c.inv + r];
            if (lr >= 0) {
                const double* src = c.S + (size_t)lr * c.ld;
                const int32_t* mp = maps + c.map;
                for (int j = threadIdx.x; j <= lr; j += blockDim.x) row[mp[j]] += src[j];
            }
            __syncthreads();
        }
    }
}

void launch_front_extend_add(const FrontDev* fr, int nfr, const FrontChild* kids, const int32_t* maps, int maxn,
                             cudaStream_t s) {
    for (int k = 0; k < nfr; k += 32768)
        front_extend_add_kernel<<<dim3(maxn < 1024 ? maxn : 1024, nfr - k < 32768 ? nfr - k : 32768), 128, 0, s>>>(
            fr + k, kids, maps);
}

// With the basis diag(A_II)^{-1/2} everywhere E is A itself, scaled on both
// sides: its entries go straight from the CSR values into the fronts.
__global__ void __launch_bounds__(256) front_scale_kernel(const double* __restrict__ val,
                                                          const int64_t* __restrict__ diag,
                                                          const int32_t* __restrict__ perm,
                                                          double* __restrict__ scale, double* __restrict__ own,
                                                          int64_t n) {
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
        const double d = 1.0 / sqrt(diag[k] >= 0 ? val[diag[k]] : 0.0);
        scale[k] = d;
        own[perm[k]] = d;
    }
}

void launch_front_scale(const double* val, const int64_t* diag, const int32_t* perm, double* scale, double* own,
                        int64_t n, cudaStream_t s) {
    const int64_t want = (n + 255) / 256;
    if (n > 0)
        front_scale_kernel<<<(unsigned)(want < 152 * 16 ? want : 152 * 16), 256, 0, s>>>(val, diag, perm, scale, own, n);
}

__global__ void __launch_bounds__(256) front_scatter_kernel(const double* __restrict__ val,
                                                            const int64_t* __restrict__ src,
                                                            const int64_t* __restrict__ dst,
                                                            const int32_t* __restrict__ a,
                                                            const int32_t* __restrict__ b,
                                                            const double* __restrict__ scale,
                                                            double* __restrict__ F, int64_t cnt) {
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < cnt; t += (int64_t)gridDim.x * blockDim.x)
        F[dst[t]] = val[src[t]] * scale[b[t]] * scale[a[t]];
}

void launch_front_scatter(const double* val, const int64_t* src, const int64_t* dst, const int32_t* a,
                          const int32_t* b, const double* scale, double* F, int64_t cnt, cudaStream_t s) {
    const int64_t want = (cnt + 255) / 256;
    if (cnt > 0)
        front_scatter_kernel<<<(unsigned)(want < 152 * 16 ? want : 152 * 16), 256, 0, s>>>(val, src, dst, a, b, scale,
                                                                                           F, cnt);
}

// v[k] = c[src[k]] (times scale[k] when given) for every plan position (nb vectors)
__global__ void __launch_bounds__(256) front_load_kernel(int64_t n, const int32_t* __restrict__ src,
                                                         const double* __restrict__ scale,
                                                         const double* __restrict__ c, int64_t ldc,
                                                         double* __restrict__ v, int nb) {
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
        const int32_t p = src[k];
        const double d = scale ? scale[k] : 1.0;
        for (int q = 0; q < nb; ++q) v[q * n + k] = d * c[q * ldc + p];
    }
}

// Down: one warp per boundary unknown t of a stage, over the parts next to it
// (refs[ptr[t] .. ptr[t + 1]): a row of W^T and the part's interior).
template <int NB>
__global__ void __launch_bounds__(256) front_down_kernel(int64_t nrow, const int32_t* __restrict__ rows,
                                                         const int32_t* __restrict__ ptr,
                                                         const FrontRef* __restrict__ refs, double* v, int64_t n,
                                                         int nb) {
    const int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (t >= nrow) return;
    double s[NB];
#pragma unroll
    for (int k = 0; k < NB; ++k) s[k] = 0.0;
    for (int e = ptr[t]; e < ptr[t + 1]; ++e) {
        const FrontRef r = refs[e];
        row_dot<NB>(r.row, v + r.i0, n, r.m, nb, lane, s);
    }
    const int64_t at = rows[t];
#pragma unroll
    for (int k = 0; k < NB; ++k) {
        const double q = warp_sum(s[k]);
        if (lane == 0 && (NB == 1 || k < nb)) v[k * n + at] -= q;
    }
}

// Up: one warp per interior row of a stage; e in plan order (read by the
// earlier stages) and, through perm (times scale), in the caller's order.
template <int NB>
__global__ void __launch_bounds__(256) front_up_kernel(const FrontDev* __restrict__ fr,
                                                       const int32_t* __restrict__ row_front, int64_t r0, int64_t r1,
                                                       const int32_t* __restrict__ bnd,
                                                       const int32_t* __restrict__ perm,
                                                       const double* __restrict__ scale,
                                                       const double* __restrict__ v, double* e,
                                                       double* __restrict__ out, int64_t n, int64_t ldo, int nb) {
    const int64_t i = r0 + (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int lane = threadIdx.x & 31;
    if (i >= r1) return;
    const FrontDev f = fr[row_front[i]];
    const int li = (int)(i - f.i0);
    double s[NB];
#pragma unroll
    for (int k = 0; k < NB; ++k) s[k] = 0.0;
    row_dot<NB>(f.Ainv + (size_t)li * f.m, v + f.i0, n, f.m, nb, lane, s);
    const double* w = f.W + (size_t)li * f.nb;
    const int32_t* bl = bnd + f.b0;
#pragma unroll 4
    for (int j = lane; j < f.nb; j += 32) {
        const double a = -__ldg(w + j);
        const int64_t b = bl[j];
#pragma unroll
        for (int k = 0; k < NB; ++k)
            if (NB == 1 || k < nb) s[k] = fma(a, e[k * n + b], s[k]);
    }
    const int64_t o = perm[i];
    const double d = scale ? scale[i] : 1.0;
#pragma unroll
    for (int k = 0; k < NB; ++k) {
        const double q = warp_sum(s[k]);
        if (lane == 0 && (NB == 1 || k < nb)) {
            e[k * n + i] = q;
            out[k * ldo + o] = d * q;
        }
    }
}

void launch_front_solve(const FrontSolve& a, const double* c, int64_t ldc, double* out, int64_t ldo, int nb,
                        cudaStream_t s) {
    const int64_t want = (a.n + 255) / 256;
    front_load_kernel<<<(unsigned)(want < 152 * 16 ? want : 152 * 16), 256, 0, s>>>(a.n, a.src, a.scale, c, ldc,
                                                                                         a.v, nb);
    for (int st = 0; st + 1 < a.stages; ++st) {
        const int64_t nrow = a.down_off[st + 1] - a.down_off[st];
        if (nrow <= 0) continue;
        const unsigned g = (unsigned)((nrow * 32 + 255) / 256);
        const int32_t* rows = a.down_rows + a.down_off[st];
        const int32_t* ptr = a.down_ptr + a.down_off[st];
        if (nb == 1)
            front_down_kernel<1><<<g, 256, 0, s>>>(nrow, rows, ptr, a.refs, a.v, a.n, 1);
        else
            front_down_kernel<MAXB><<<g, 256, 0, s>>>(nrow, rows, ptr, a.refs, a.v, a.n, nb);
    }
    for (int st = a.stages - 1; st >= 0; --st) {
        const int64_t r0 = a.row_off[st], r1 = a.row_off[st + 1];
        if (r1 <= r0) continue;
        const unsigned g = (unsigned)(((r1 - r0) * 32 + 255) / 256);
        if (nb == 1)
            front_up_kernel<1><<<g, 256, 0, s>>>(a.fr, a.row_front, r0, r1, a.bnd, a.perm, a.scale, a.v, a.e, out,
                                                 a.n, ldo, 1);
        else
            front_up_kernel<MAXB><<<g, 256, 0, s>>>(a.fr, a.row_front, r0, r1, a.bnd, a.perm, a.scale, a.v, a.e, out,
                                                    a.n, ldo, nb);
    }
}

}  // namespace amdd

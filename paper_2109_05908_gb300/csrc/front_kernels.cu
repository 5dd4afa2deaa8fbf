// Device side of the exact solves by substructuring (plan: fronts.cu): the coarse
// solve with E (FP64) and the local solves with all A_ii at once, whose graph is
// a forest of one tree per subdomain (FP64, or FP32 in the mixed form).
//
// With the matrix in the plan's order, every part p with interior I and boundary
// B keeps, once the earlier stages are eliminated into its front,
//   Ainv = (S_II)^{-1}     and     W = S_II^{-1} S_IB
// as dense blocks, and M e = c is solved exactly by
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
// on 20^3 2.83 -> 0.59 ms; apply on 64^2 301 -> 117 us.  Local solves against the
// two dense triangles of each L_i^{-1}: one-level apply of 1024 boxes of 324
// unknowns in FP64 526 -> 125 us (a third of the entries, and the shuffle trees
// shared by eight rows); 16 subdomains of 1.7k unknowns in FP32 72 -> 43 us.
#include "amdd_internal.h"

namespace amdd {
namespace {

// s[k] += sum over columns j = sub, sub + G, ... < m of row[j] x_k[j] (x_k ldv
// apart), four to eight loads of the row in flight per lane
template <typename T, int NB, int G>
__device__ __forceinline__ void row_dot(const T* __restrict__ row, const T* x, int64_t ldv, int m, int nb, int sub,
                                        T* s) {
    constexpr int U = NB == 1 ? 8 : 4;
    int j = sub;
    for (; j + G * (U - 1) < m; j += G * U) {
        T a[U];
#pragma unroll
        for (int u = 0; u < U; ++u) a[u] = __ldg(row + j + G * u);
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int k = 0; k < NB; ++k)
                if (NB == 1 || k < nb) s[k] = fma(a[u], x[k * ldv + j + G * u], s[k]);
    }
    for (; j < m; j += G) {
        const T a = __ldg(row + j);
#pragma unroll
        for (int k = 0; k < NB; ++k)
            if (NB == 1 || k < nb) s[k] = fma(a, x[k * ldv + j], s[k]);
    }
}

template <typename T, int G>
__device__ __forceinline__ T lane_sum(T v) {
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

}  // namespace

// Lower triangle of the front of part p, columns of its interior, from the lower
// triangle of its dense matrix A (E, or the A_ii of its subdomain): F[r][c] =
// A[max][min] of the two unknowns.  F is zero on entry (its boundary block stays zero).
__global__ void __launch_bounds__(256) front_gather_kernel(const FrontDevT<double>* __restrict__ fr,
                                                           const FrontSrc* __restrict__ src,
                                                           const int32_t* __restrict__ bnd,
                                                           const int32_t* __restrict__ perm) {
    const FrontDevT<double> f = fr[blockIdx.y];
    const FrontSrc a = src[blockIdx.y];
    const int n = f.m + f.nb;
    for (int r = blockIdx.x; r < n; r += gridDim.x) {
        const int64_t pr = perm[r < f.m ? f.i0 + r : bnd[f.b0 + r - f.m]] - a.off;
        double* row = f.F + (size_t)r * n;
        const int cend = min(r + 1, f.m);
        for (int c = threadIdx.x; c < cend; c += blockDim.x) {
            const int64_t pc = perm[f.i0 + c] - a.off;
            row[c] = a.A[(pr > pc ? pr : pc) * a.ld + (pr > pc ? pc : pr)];
        }
    }
}

void launch_front_gather(const FrontDevT<double>* fr, const FrontSrc* src, int nfr, const int32_t* bnd,
                         const int32_t* perm, int maxn, cudaStream_t s) {
    for (int k = 0; k < nfr; k += 32768)  // grid.y is 16 bits wide
        front_gather_kernel<<<dim3(maxn < 512 ? maxn : 512, nfr - k < 32768 ? nfr - k : 32768), 256, 0, s>>>(
            fr + k, src + k, bnd, perm);
}

// Adds the Schur complements of the children of every front of a stage into it
// (lower triangles).  One CTA per front row; the children one after the other
// in a fixed order, so sums do not depend on the schedule.  inv[r] is the
// child's boundary row of front row r (-1: none), map its inverse.
__global__ void __launch_bounds__(128) front_extend_add_kernel(const FrontDevT<double>* __restrict__ fr,
                                                               const FrontChild* __restrict__ kids,
                                                               const int32_t* __restrict__ maps) {
    const FrontDevT<double> f = fr[blockIdx.y];
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

void launch_front_extend_add(const FrontDevT<double>* fr, int nfr, const FrontChild* kids, const int32_t* maps,
                             int maxn, cudaStream_t s) {
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
                                                            const double* __restrict__ scale, double* __restrict__ F,
                                                            int64_t cnt) {
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < cnt; t += (int64_t)gridDim.x * blockDim.x) {
        F[dst[t]] = val[src[t]] * scale[b[t]] * scale[a[t]];
    }
}

void launch_front_scatter(const double* val, const int64_t* src, const int64_t* dst, const int32_t* a,
                          const int32_t* b, const double* scale, double* F, int64_t cnt, cudaStream_t s) {
    const int64_t want = (cnt + 255) / 256;
    if (cnt > 0)
        front_scatter_kernel<<<(unsigned)(want < 152 * 16 ? want : 152 * 16), 256, 0, s>>>(val, src, dst, a, b,
                                                                                              scale, F, cnt);
}

// v[k] = c[src[k]] (times scale[k] when given) for every plan position (nb vectors)
template <typename T>
__global__ void __launch_bounds__(256) front_load_kernel(int64_t n, const int32_t* __restrict__ src,
                                                         const double* __restrict__ scale,
                                                         const double* __restrict__ c, int64_t ldc,
                                                         T* __restrict__ v, int nb) {
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
        const int32_t p = src[k];
        const double d = scale ? scale[k] : 1.0;
        for (int q = 0; q < nb; ++q) v[q * n + k] = (T)(d * c[q * ldc + p]);
    }
}

// Small CTAs: the rows of a stage are few, and their work should reach every SM.
constexpr int FRONT_THREADS = 64;

// Down: G lanes per boundary unknown t of a stage, over the parts next to it
// (refs[ptr[t] .. ptr[t + 1]): a row of W^T and the part's interior).
template <typename T, int NB, int G>
__global__ void __launch_bounds__(FRONT_THREADS) front_down_kernel(int64_t nrow, const int32_t* __restrict__ rows,
                                                         const int32_t* __restrict__ ptr,
                                                         const FrontRefT<T>* __restrict__ refs, T* v, int64_t n,
                                                         int nb) {
    const int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / G;
    const int sub = threadIdx.x & (G - 1);
    T s[NB];
#pragma unroll
    for (int k = 0; k < NB; ++k) s[k] = T(0);
    const int e1 = t < nrow ? ptr[t + 1] : 0;
    for (int e = t < nrow ? ptr[t] : 0; e < e1; ++e) {
        const FrontRefT<T> r = refs[e];
        row_dot<T, NB, G>(r.row, v + r.i0, n, r.m, nb, sub, s);
    }
    const int64_t at = t < nrow ? rows[t] : 0;
#pragma unroll
    for (int k = 0; k < NB; ++k) {
        const T q = lane_sum<T, G>(s[k]);
        if (sub == 0 && t < nrow && (NB == 1 || k < nb)) v[k * n + at] -= q;
    }
}

// Up: G lanes per interior row of a stage; e in plan order (read by the earlier
// stages) and, when out is given, through perm (times scale) in the caller's order.
template <typename T, int NB, int G>
__global__ void __launch_bounds__(FRONT_THREADS) front_up_kernel(const FrontDevT<T>* __restrict__ fr,
                                                       const int32_t* __restrict__ row_front, int64_t r0, int64_t r1,
                                                       const int32_t* __restrict__ bnd,
                                                       const int32_t* __restrict__ perm,
                                                       const double* __restrict__ scale,
                                                       const T* __restrict__ v, T* e, T* __restrict__ out, int64_t n,
                                                       int64_t ldo, int nb) {
    const int64_t i = r0 + ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / G;
    const int sub = threadIdx.x & (G - 1);
    T s[NB];
#pragma unroll
    for (int k = 0; k < NB; ++k) s[k] = T(0);
    if (i < r1) {
        const FrontDevT<T> f = fr[row_front[i]];
        const int li = (int)(i - f.i0);
        row_dot<T, NB, G>(f.Ainv + (size_t)li * f.m, v + f.i0, n, f.m, nb, sub, s);
        const T* w = f.W + (size_t)li * f.nb;
        const int32_t* bl = bnd + f.b0;
#pragma unroll 4
        for (int j = sub; j < f.nb; j += G) {
            const T a = -__ldg(w + j);
            const int64_t b = bl[j];
#pragma unroll
            for (int k = 0; k < NB; ++k)
                if (NB == 1 || k < nb) s[k] = fma(a, e[k * n + b], s[k]);
        }
    }
#pragma unroll
    for (int k = 0; k < NB; ++k) {
        const T q = lane_sum<T, G>(s[k]);
        if (sub == 0 && i < r1 && (NB == 1 || k < nb)) {
            e[k * n + i] = q;
            if (out) out[k * ldo + perm[i]] = (T)((scale ? scale[i] : 1.0) * (double)q);
        }
    }
}

namespace {

// Lanes per row: 4 while that fills the chip (FP64 runs at two multiply-adds per
// clock and SM, idle lanes or not, so the shuffle tree is best shared by 8 rows),
// a warp when the rows of the stage are few.  With several vectors each load feeds
// eight independent sums: in FP64 fewer threads then fill the chip, in FP32, whose
// rate is not the limit, more are wanted to hide the loads (local solves in FP32 on
// 19,000 rows of a 27-point matrix with three unknowns a node, one-level apply with
// 2 / 8 vectors: 161 / 199 us with the FP64 line, 90 / 107 so; dense triangles 158 / 174).
template <typename T, int NB>
int lanes_for(int64_t rows) {
    if (sizeof(T) == 4 && NB > 1) {
        const int64_t fill = 152 * 768;
        return rows * 4 >= fill ? 4 : (rows * 8 >= fill ? 8 : (rows * 16 >= fill ? 16 : 32));
    }
    const int64_t fill = 152 * (NB == 1 ? 448 : 128);
    return rows * 4 >= fill ? 4 : (rows * 8 >= fill ? 8 : 32);
}

template <typename T, int NB, int G>
void stage_down(const FrontSolveT<T>& a, int st, int nb, cudaStream_t s) {
    const int64_t nrow = a.down_off[st + 1] - a.down_off[st];
    front_down_kernel<T, NB, G><<<(unsigned)((nrow * G + FRONT_THREADS - 1) / FRONT_THREADS), FRONT_THREADS, 0, s>>>(
        nrow, a.down_rows + a.down_off[st], a.down_ptr + a.down_off[st], a.refs, a.v, a.n, nb);
}
template <typename T, int NB, int G>
void stage_up(const FrontSolveT<T>& a, int st, T* out, int64_t ldo, int nb, cudaStream_t s) {
    const int64_t r0 = a.row_off[st], r1 = a.row_off[st + 1];
    front_up_kernel<T, NB, G><<<(unsigned)(((r1 - r0) * G + FRONT_THREADS - 1) / FRONT_THREADS), FRONT_THREADS, 0, s>>>(
        a.fr, a.row_front, r0, r1, a.bnd, a.perm, a.scale, a.v, a.e, out, a.n, ldo, nb);
}

template <typename T, int NB>
void solve_nb(const FrontSolveT<T>& a, T* out, int64_t ldo, int nb, cudaStream_t s) {
    for (int st = 0; st + 1 < a.stages; ++st) {
        const int64_t nrow = a.down_off[st + 1] - a.down_off[st];
        if (nrow <= 0) continue;
        const int g = lanes_for<T, NB>(nrow);
        if (g == 4)
            stage_down<T, NB, 4>(a, st, nb, s);
        else if (g == 8)
            stage_down<T, NB, 8>(a, st, nb, s);
        else if (g == 16)
            stage_down<T, NB, 16>(a, st, nb, s);
        else
            stage_down<T, NB, 32>(a, st, nb, s);
    }
    for (int st = a.stages - 1; st >= 0; --st) {
        if (a.row_off[st + 1] <= a.row_off[st]) continue;
        const int g = lanes_for<T, NB>(a.row_off[st + 1] - a.row_off[st]);
        if (g == 4)
            stage_up<T, NB, 4>(a, st, out, ldo, nb, s);
        else if (g == 8)
            stage_up<T, NB, 8>(a, st, out, ldo, nb, s);
        else if (g == 16)
            stage_up<T, NB, 16>(a, st, out, ldo, nb, s);
        else
            stage_up<T, NB, 32>(a, st, out, ldo, nb, s);
    }
}

}  // namespace

template <typename T>
void launch_front_solve(const FrontSolveT<T>& a, const double* c, int64_t ldc, T* out, int64_t ldo, int nb,
                        cudaStream_t s) {
    if (a.n <= 0) return;
    const int64_t want = (a.n + 255) / 256;
    front_load_kernel<T><<<(unsigned)(want < 152 * 16 ? want : 152 * 16), 256, 0, s>>>(a.n, a.src, a.scale, c, ldc,
                                                                                       a.v, nb);
    if (nb == 1)
        solve_nb<T, 1>(a, out, ldo, 1, s);
    else
        solve_nb<T, MAXB>(a, out, ldo, nb, s);
}
template void launch_front_solve<double>(const FrontSolveT<double>&, const double*, int64_t, double*, int64_t, int,
                                         cudaStream_t);
template void launch_front_solve<float>(const FrontSolveT<float>&, const double*, int64_t, float*, int64_t, int,
                                        cudaStream_t);

}  // namespace amdd

// Inner eigensolve of the FP32 block-pair Jacobi on the tensor cores: the
// symmetric 64 x 64 Gram matrix G of two row blocks is diagonalised in shared
// memory by two-sided Jacobi on 8 x 8 blocks, the rotations are accumulated in
// Qt (Qt G Qt^T diagonal).
//
// The 64 indices are eight blocks of 8; a sweep is the seven rounds of the
// circle schedule on the blocks, with four disjoint block pairs each.  Per round
//   * warps 0..3 diagonalise one 16 x 16 diagonal submatrix each, in registers:
//     lane i < 16 holds row i of the submatrix, lane 16 + i row i of the
//     accumulated rotation W, so one row operation serves both.  Eight rounds of
//     eight disjoint (first block, second block) pairs; in the first round of a
//     sweep the seven rounds inside the blocks precede them.  Together every two
//     of the 64 indices meet once a sweep;
//   * warps 4..7 meanwhile apply the previous round's W to Qt, which the
//     eigensolves do not read;
//   * then warps 0..3 apply W to the rows and to the columns of G, a thread per two
//     columns (rows) of a block pair: 32 entries in registers, 512 multiply-adds.
// Why: the sweep that rotates G and Qt pair by pair (jpi_solve) needs 63 barriers
// and moves both matrices through shared memory in each of them.  Here a sweep has
// 21 barriers and moves them seven times; the loads of W bound it.  On the 3D
// workload (24^3, 16 subdomains, orders to 1903) an inner solve went from 200 k to
// 124 k cycles, two CTAs to an SM.  The tests are those of jpi_solve.
#pragma once

#include "jacobi_pair_inner.cuh"

namespace amdd {

constexpr int JB_B = 8;                    // indices per inner block
constexpr int JB_R = 4 * 16 * 16;          // the four W of a round

struct JbShared {
    float2 cs[4][16];     // per warp: a round's rotations
    int rot[2][4];        // per warp: rotations of the round
};

struct JbTest {
    float tin, absf, nf;
    JacLoose<float> loose;
    float rel;  // couplings below rel max(a, b) are left alone
};

// the two indices blocks of pair g (0..3) of round ir (0..6)
__device__ __forceinline__ void jb_pair(int g, int ir, int& p, int& q) {
    if (g == 0) {
        p = 7;
        q = ir;
    } else {
        p = (ir + g) % 7;
        q = (ir - g + 7) % 7;
    }
    p *= JB_B;
    q *= JB_B;
}

// rotation of the pair [[a, g], [g, b]] as in jpi_rotation; false (cs = 1, sn = t = 0)
// when the tests leave it
__device__ __forceinline__ bool jb_rotation(float a, float b, float g, const JbTest& ts, float& cs, float& sn, float& t) {
    cs = 1.0f;
    sn = t = 0.0f;
    const float m = fmaxf(a, b), g2 = g * g;
    if (!(g != 0.0f && g2 > jac_tol2(ts.tin, a, b, ts.loose) * a * b && fabsf(g) > ts.absf && g2 > ts.nf * m &&
          fabsf(g) > ts.rel * m))
        return false;
    const float dd = b - a, gg = g + g;
    t = copysignf(1.0f, dd) * gg / (fabsf(dd) + sqrtf(fmaf(dd, dd, gg * gg)));
    cs = jpi_rsqrt(fmaf(t, t, 1.0f));
    sn = cs * t;
    return true;
}

// r[i] of the eight (sixteen) values by the low bits of i
__device__ __forceinline__ float jb_sel8(const float* r, int i) {
    const float a = (i & 1) ? r[1] : r[0], b = (i & 1) ? r[3] : r[2], c = (i & 1) ? r[5] : r[4], d = (i & 1) ? r[7] : r[6];
    const float e = (i & 2) ? b : a, f = (i & 2) ? d : c;
    return (i & 4) ? f : e;
}

// The eight rows pairs (i, i ^ M), M < 8, inside the two blocks
template <int M>
__device__ __forceinline__ int jb_inside(float (&r)[16], float& dg, const JbTest& ts, float2* csn, int lane) {
    constexpr int HB = M >= 4 ? 4 : (M >= 2 ? 2 : 1);
    const int i = lane & 15;
    const bool hi = (i & HB) != 0;
    const int pl = hi ? i ^ M : i;
    float v[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = r[j ^ M];
    const float own = (i & 8) ? jb_sel8(v + 8, i) : jb_sel8(v, i);  // r[i ^ M]
    const float g = __shfl_sync(0xffffffffu, own, pl), a = __shfl_sync(0xffffffffu, dg, pl),
                b = __shfl_sync(0xffffffffu, dg, pl ^ M);
    float cs, sn, t;
    const bool d = jb_rotation(a, b, g, ts, cs, sn, t);
    const unsigned bal = __ballot_sync(0xffffffffu, d && lane < 16 && !hi);
    if (!bal) return 0;
    if (lane < 16 && !hi) csn[i] = make_float2(cs, sn);
    const float ss = hi ? sn : -sn;
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        const float o = __shfl_xor_sync(0xffffffffu, r[j], M);
        v[j] = fmaf(cs, r[j], ss * o);
    }
    dg = hi ? fmaf(t, g, dg) : fmaf(-t, g, dg);
    __syncwarp();
    if (lane < 16) {
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            if (j & HB) continue;
            const float2 c = csn[j];
            const float x = v[j], y = v[j ^ M];
            v[j] = fmaf(c.x, x, -c.y * y);
            v[j ^ M] = fmaf(c.y, x, c.x * y);
        }
    }
#pragma unroll
    for (int j = 0; j < 16; ++j) r[j] = v[j];
    __syncwarp();
    return __popc(bal);
}

// One warp: the Jacobi rounds on the submatrix of blocks p, q (first indices);
// W to Wout (16 x 16, row-major).  Returns the number of rotations.
__device__ __forceinline__ int jb_eig16(const float* G, int p, int q, bool inside, const JbTest& ts, float* Wout,
                                        float2* csn, int lane) {
    float r[16];
    const int i = lane & 15;
    const float* gr = G + ((i & 8) ? q + i - 8 : p + i) * JPI_LDG;
    float dg = gr[(i & 8) ? q + i - 8 : p + i];
#pragma unroll
    for (int j = 0; j < 16; ++j) r[j] = lane < 16 ? gr[j < 8 ? p + j : q + j - 8] : (j == i ? 1.0f : 0.0f);
    int n = 0;
    if (inside) {
        n += jb_inside<1>(r, dg, ts, csn, lane);
        n += jb_inside<2>(r, dg, ts, csn, lane);
        n += jb_inside<3>(r, dg, ts, csn, lane);
        n += jb_inside<4>(r, dg, ts, csn, lane);
        n += jb_inside<5>(r, dg, ts, csn, lane);
        n += jb_inside<6>(r, dg, ts, csn, lane);
        n += jb_inside<7>(r, dg, ts, csn, lane);
    }
    // pairs (k, 8 + (k + t) mod 8): after each round the columns 8..15 move up by
    // one register, so that column k's partner is always register 8 + k; eight
    // rounds bring them back
    const bool hi = (i & 8) != 0;
#pragma unroll 1
    for (int t8 = 0; t8 < 8; ++t8) {
        const int pl = hi ? (i - t8) & 7 : i;
        const int ql = 8 + ((pl + t8) & 7);
        const float own = jb_sel8(r + 8, i);
        const float g = __shfl_sync(0xffffffffu, own, pl), a = __shfl_sync(0xffffffffu, dg, pl),
                    b = __shfl_sync(0xffffffffu, dg, ql);
        float cs, sn, t;
        const bool d = jb_rotation(a, b, g, ts, cs, sn, t);
        const unsigned bal = __ballot_sync(0xffffffffu, d && lane < 8);
        if (bal) {
            if (lane < 8) csn[lane] = make_float2(cs, sn);
            const float ss = hi ? sn : -sn;
            const int other = (hi ? pl : ql) | (lane & 16);
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                const float o = __shfl_sync(0xffffffffu, r[j], other);
                r[j] = fmaf(cs, r[j], ss * o);
            }
            dg = hi ? fmaf(t, g, dg) : fmaf(-t, g, dg);
            __syncwarp();
            if (lane < 16) {
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const float2 c = csn[j];
                    const float x = r[j], y = r[8 + j];
                    r[j] = fmaf(c.x, x, -c.y * y);
                    r[8 + j] = fmaf(c.y, x, c.x * y);
                }
            }
            n += __popc(bal);
            __syncwarp();
        }
        const float r8 = r[8];
#pragma unroll
        for (int j = 8; j < 15; ++j) r[j] = r[j + 1];
        r[15] = r8;
    }
    if (lane >= 16) {
        float4* w = reinterpret_cast<float4*>(Wout + i * 16);
#pragma unroll
        for (int j = 0; j < 4; ++j) w[j] = make_float4(r[4 * j], r[4 * j + 1], r[4 * j + 2], r[4 * j + 3]);
    }
    return n;
}

// x <- W x for the 16 entries of two columns (rows) of a block pair: entries 0..7
// at M, M + step, ..., entries 8..15 at M + off, ..., the second column `next` on.
// Two columns a thread: the loads of W (a 16-byte load of one address still takes
// four cycles of the shared-memory pipe) are what bounds this product, 64 of them
// for 512 multiply-adds instead of 256.
__device__ __forceinline__ void jb_mul16(float* M, int off, int step, int next, const float* W) {
    float x[16], y[16];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        x[j] = M[j * step];
        x[8 + j] = M[off + j * step];
        y[j] = M[next + j * step];
        y[8 + j] = M[next + off + j * step];
    }
    const float4* w4 = reinterpret_cast<const float4*>(W);
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        float s0 = 0.0f, s1 = 0.0f, t0 = 0.0f, t1 = 0.0f;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float4 w = w4[i * 4 + j];
            s0 = fmaf(w.x, x[4 * j], s0);
            t0 = fmaf(w.x, y[4 * j], t0);
            s1 = fmaf(w.y, x[4 * j + 1], s1);
            t1 = fmaf(w.y, y[4 * j + 1], t1);
            s0 = fmaf(w.z, x[4 * j + 2], s0);
            t0 = fmaf(w.z, y[4 * j + 2], t0);
            s1 = fmaf(w.w, x[4 * j + 3], s1);
            t1 = fmaf(w.w, y[4 * j + 3], t1);
        }
        float* o = M + (i < 8 ? i * step : off + (i - 8) * step);
        o[0] = s0 + s1;
        o[next] = t0 + t1;
    }
}

// The whole inner iteration, by all JPI_THREADS threads: G (64 x 64, both
// triangles, leading dimension JPI_LDG), Qt the identity (JPI_LDQ), W two times
// JB_R floats of scratch (16-byte aligned).  Returns the number of sweeps; *nrot_out
// counts each warp's rotations (the same in all its lanes).
__device__ int jb_solve(float* G, float* Qt, float* W, JbShared& sh, JbTest ts, int max_sweeps, unsigned& nrot_out) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int c = lane, g = warp & 3;  // columns (rows) c, c + 32 of block pair g
    unsigned nrot = 0;
    int par = 0, buf = 0, lag = -1, sw = 0;
    const float rel = 8.0f * 1.1920928955078125e-7f;
    for (; sw < max_sweeps; ++sw) {
        bool swrot = false;
        ts.rel = sw ? rel : 0.0f;
        for (int ir = 0; ir < 7; ++ir) {
            if (warp < 4) {
                int p, q;
                jb_pair(warp, ir, p, q);
                const int n = jb_eig16(G, p, q, ir == 0, ts, W + buf * JB_R + warp * 256, sh.cs[warp], lane);
                nrot += n;
                if (lane == 0) sh.rot[par][warp] = n;
            } else if (lag >= 0) {
                int p, q;
                jb_pair(g, lag, p, q);
                jb_mul16(Qt + p * JPI_LDQ + c, (q - p) * JPI_LDQ, JPI_LDQ, 32, W + (buf ^ 1) * JB_R + g * 256);
            }
            __syncthreads();
            const bool any = (sh.rot[par][0] | sh.rot[par][1] | sh.rot[par][2] | sh.rot[par][3]) != 0;
            par ^= 1;
            lag = -1;
            if (any) {
                int p, q;
                jb_pair(g, ir, p, q);
                const float* w = W + buf * JB_R + g * 256;
                if (warp < 4) jb_mul16(G + p * JPI_LDG + c, (q - p) * JPI_LDG, JPI_LDG, 32, w);
                __syncthreads();
                if (warp < 4) jb_mul16(G + c * JPI_LDG + p, q - p, 1, 32 * JPI_LDG, w);
                __syncthreads();
                lag = ir;
                buf ^= 1;
                swrot = true;
            }
        }
        if (!swrot) break;
    }
    if (lag >= 0 && warp >= 4) {
        int p, q;
        jb_pair(g, lag, p, q);
        jb_mul16(Qt + p * JPI_LDQ + c, (q - p) * JPI_LDQ, JPI_LDQ, 32, W + (buf ^ 1) * JB_R + g * 256);
    }
    __syncthreads();
    nrot_out = nrot;
    return min(sw + 1, max_sweeps);
}

}  // namespace amdd

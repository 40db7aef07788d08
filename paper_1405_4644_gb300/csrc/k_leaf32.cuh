// k_leaf32.cuh -- float32 leaves of the low-precision factorisation (steps
// A1/A2 of Section 3.1's Cholesky) and the per-block inverses the
// triangular sweeps use:
//
//   k_potrf_leaf32   factors W[k:k+nb, k:k+nb] = L L^T in four 32-column
//                    steps of four-pivot micro-steps, the rows below the
//                    diagonal block following micro-step by micro-step;
//                    meanwhile the other warps store the previous columns
//                    of L (and their operand mirror) and form the 32x32
//                    inverses.
//   k_trsm_leaf32    panel solve X L^T = B for 64 rows per CTA in four
//                    32-column steps with the same 32x32 inverses.
//   k_block_inverse  after the whole factorisation, off the critical path
//                    and one CTA per block: the full (L_JJ^{-1})^T of every
//                    128x128 diagonal block, for the sweeps.
//
// The float64 baseline keeps the sub-block kernels of k_leaf.cuh.
#pragma once
#include "common.cuh"

#define LDL 132   // the leaf: 16-byte rows, eight consecutive rows in distinct banks

// Dinv32 for block b lives at Dinv32 + b * 4096: four row-major 32x32
// blocks, D_s[i][c] = (L_ss^{-1})[i][c] (lower triangular).
constexpr size_t potrf_leaf32_smem() { return (size_t)(128 * LDL + 8 * 32 * 4 + 128) * sizeof(float); }
constexpr int LEAF_THREADS = 512;

// Entries of L in columns [c0, c0 + 32), rows c0 .. nb - 1, from the leaf's
// shared copy S to W and its mirror, four columns per store; thread t of nt.
__device__ __forceinline__ void leaf_store_cols(const float* S, float* W, long ldw, int k, int nb, int c0,
                                                const Mirror& mir, int t, int nt) {
    for (int e = t; e < (128 - c0) * 8; e += nt) {
        const int r = c0 + (e >> 3), c4 = c0 + (e & 7) * 4;
        if (r >= nb || c4 > r) continue;
        const float4 f = *reinterpret_cast<const float4*>(S + r * LDL + c4);
        float* dst = W + (long)(k + r) * ldw + k + c4;
        if (c4 + 3 <= r) {
            *reinterpret_cast<float4*>(dst) = f;
            mirror_store4(mir, (long)(k + r), (long)(k + c4), f);
        } else {
            const float v[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (c4 + q <= r) {
                    dst[q] = v[q];
                    mirror_store(mir, (long)(k + r), (long)(k + c4 + q), v[q]);
                }
        }
    }
}

// One unit of the leaf's trailing update after the 32-column step at o: rows i
// .. i + NR - 1, columns j, j + 8, j + 16, j + 24: S[i][.] -= sum_{l<32} S[i][o+l]
// S[.][o+l].  The eight lanes of a row group read eight consecutive rows of S,
// 16 bytes each, in distinct banks; the loads from shared memory bound it.
template <int NR>
__device__ __forceinline__ void leaf_tile(float* S, int o, int i, int j) {
    float acc[NR][4] = {};
#pragma unroll 4
    for (int l = 0; l < 32; l += 4) {
        float4 x[NR], y[4];
#pragma unroll
        for (int r = 0; r < NR; ++r) x[r] = *reinterpret_cast<const float4*>(S + (i + r) * LDL + o + l);
#pragma unroll
        for (int q = 0; q < 4; ++q) y[q] = *reinterpret_cast<const float4*>(S + (j + 8 * q) * LDL + o + l);
#pragma unroll
        for (int r = 0; r < NR; ++r)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                acc[r][q] = fmaf(x[r].x, y[q].x, acc[r][q]);
                acc[r][q] = fmaf(x[r].y, y[q].y, acc[r][q]);
                acc[r][q] = fmaf(x[r].z, y[q].z, acc[r][q]);
                acc[r][q] = fmaf(x[r].w, y[q].w, acc[r][q]);
            }
    }
#pragma unroll
    for (int r = 0; r < NR; ++r)
#pragma unroll
        for (int q = 0; q < 4; ++q) S[(i + r) * LDL + j + 8 * q] -= acc[r][q];
}

__device__ __forceinline__ float rsqrt_ftz(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// The Cholesky factor of a 4 x 4 pivot block p (lower triangle by rows: 00 10 11
// 20 21 22 30 31 32 33): rv = the reciprocals of its diagonal, r1.x, r2.xy,
// r3.xyz the entries below it, d the pivots.
template <bool FTZ>
__device__ __forceinline__ void leaf_pivots(const float (&p)[10], float4& rv, float4& r1, float4& r2, float4& r3,
                                            float (&d)[4]) {
    auto rs = [](float x) { return FTZ ? rsqrt_ftz(x) : rsqrtf(x); };
    d[0] = p[0];
    rv.x = rs(d[0]);
    r1.x = p[1] * rv.x;
    r2.x = p[3] * rv.x;
    r3.x = p[6] * rv.x;
    d[1] = fmaf(-r1.x, r1.x, p[2]);
    rv.y = rs(d[1]);
    r2.y = fmaf(-r1.x, r2.x, p[4]) * rv.y;
    r3.y = fmaf(-r1.x, r3.x, p[7]) * rv.y;
    d[2] = fmaf(-r2.y, r2.y, fmaf(-r2.x, r2.x, p[5]));
    rv.z = rs(d[2]);
    r3.z = fmaf(-r2.y, r3.y, fmaf(-r2.x, r3.x, p[8])) * rv.z;
    d[3] = fmaf(-r3.z, r3.z, fmaf(-r3.y, r3.y, fmaf(-r3.x, r3.x, p[9])));
    rv.w = rs(d[3]);
}

// Micro-step B (columns 4 B .. 4 B + 3, four pivots) of a 32-column step for one
// row, a[] = the row's 32 columns.  The diagonal block's warp (DIAG, lane = row)
// broadcasts the ten entries of the 4 x 4 pivot block and every lane factors
// them: the chain is four reciprocal square roots and one exchange through
// shared memory per four pivots, and the rank-4 update reads 16 bytes per
// column.  The warps below follow, one named barrier (1 + B; the diagonal warp
// only arrives) behind.  The square roots flush subnormal pivots; a pivot block
// with one that is not a positive normal number is redone without, where the
// first non-positive pivot is noted.
template <int B, bool DIAG>
__device__ __forceinline__ void leaf_micro(float (&a)[32], int lane, float4* Xs, float* Rs, int nthr, int& badj) {
    constexpr int j = 4 * B;
    float4* X = Xs + B * 32;
    float4 rv, r1, r2, r3;
    if constexpr (DIAG) {
        const unsigned F = 0xffffffffu;
        float p[10], d[4];
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int c = 0; c <= r; ++c) p[r * (r + 1) / 2 + c] = __shfl_sync(F, a[j + c], j + r);
        leaf_pivots<true>(p, rv, r1, r2, r3, d);
        constexpr float MIN = 1.17549435e-38f;
        if (!(d[0] >= MIN && d[1] >= MIN && d[2] >= MIN && d[3] >= MIN)) {  // the same in every lane
            leaf_pivots<false>(p, rv, r1, r2, r3, d);
#pragma unroll
            for (int q = 3; q >= 0; --q)
                if (!(d[q] > 0.f) && badj >= j) badj = j + q;
        }
    } else {
        asm volatile("bar.sync %0, %1;" ::"r"(B + 1), "r"(nthr) : "memory");
        rv = *reinterpret_cast<const float4*>(Rs + j);
        r1 = X[j + 1];
        r2 = X[j + 2];
        r3 = X[j + 3];
    }
    float4 x;  // x L_bb^T = a
    x.x = a[j] * rv.x;
    x.y = fmaf(-x.x, r1.x, a[j + 1]) * rv.y;
    x.z = fmaf(-x.y, r2.y, fmaf(-x.x, r2.x, a[j + 2])) * rv.z;
    x.w = fmaf(-x.z, r3.z, fmaf(-x.y, r3.y, fmaf(-x.x, r3.x, a[j + 3]))) * rv.w;
    if constexpr (DIAG) {
        X[lane] = x;
        if (lane == 0) *reinterpret_cast<float4*>(Rs + j) = rv;
        __syncwarp();
        if (nthr > 32) asm volatile("bar.arrive %0, %1;" ::"r"(B + 1), "r"(nthr) : "memory");
    }
#pragma unroll
    for (int l = j + 4; l < 32; ++l) {
        const float4 t = X[l];
        a[l] = fmaf(-x.w, t.w, fmaf(-x.z, t.z, fmaf(-x.y, t.y, fmaf(-x.x, t.x, a[l]))));
    }
    a[j] = x.x;
    a[j + 1] = x.y;
    a[j + 2] = x.z;
    a[j + 3] = x.w;
}

template <bool DIAG>
__device__ __forceinline__ void leaf_step32(float* row, int lane, float4* Xs, float* Rs, int nthr, int& badj) {
    float a[32];
#pragma unroll
    for (int c = 0; c < 32; c += 4) {
        const float4 f = *reinterpret_cast<const float4*>(row + c);
        a[c] = f.x;
        a[c + 1] = f.y;
        a[c + 2] = f.z;
        a[c + 3] = f.w;
    }
    leaf_micro<0, DIAG>(a, lane, Xs, Rs, nthr, badj);
    leaf_micro<1, DIAG>(a, lane, Xs, Rs, nthr, badj);
    leaf_micro<2, DIAG>(a, lane, Xs, Rs, nthr, badj);
    leaf_micro<3, DIAG>(a, lane, Xs, Rs, nthr, badj);
    leaf_micro<4, DIAG>(a, lane, Xs, Rs, nthr, badj);
    leaf_micro<5, DIAG>(a, lane, Xs, Rs, nthr, badj);
    leaf_micro<6, DIAG>(a, lane, Xs, Rs, nthr, badj);
    leaf_micro<7, DIAG>(a, lane, Xs, Rs, nthr, badj);
#pragma unroll
    for (int c = 0; c < 32; c += 4) {
        float4 f = make_float4(a[c], a[c + 1], a[c + 2], a[c + 3]);
        if (DIAG) {  // zeros above the diagonal
            if (c + 0 > lane) f.x = 0.f;
            if (c + 1 > lane) f.y = 0.f;
            if (c + 2 > lane) f.z = 0.f;
            if (c + 3 > lane) f.w = 0.f;
        }
        *reinterpret_cast<float4*>(row + c) = f;
    }
}

// The inverse of the 32 x 32 diagonal block at o (lane c: column c), to Dout
// (row-major): x_i = (delta_ic - sum_{l<i} L_il x_l) / L_ii.
__device__ __forceinline__ void leaf_inverse32(const float* S, int o, const float* Rs, float* __restrict__ Dout,
                                               int lane) {
    float x[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) {
        float s0 = (i == lane) ? 1.f : 0.f, s1 = 0.f;
#pragma unroll
        for (int l = 0; l < i; l += 4) {
            const float4 t = *reinterpret_cast<const float4*>(S + (o + i) * LDL + o + l);
            s0 = fmaf(-t.x, x[l], s0);
            if (l + 1 < i) s1 = fmaf(-t.y, x[l + 1], s1);
            if (l + 2 < i) s0 = fmaf(-t.z, x[l + 2], s0);
            if (l + 3 < i) s1 = fmaf(-t.w, x[l + 3], s1);
        }
        x[i] = (s0 + s1) * Rs[i];
        Dout[i * 32 + lane] = x[i];
    }
}

// The 128 x 128 leaf.  Bound: the chain of 128 dependent pivots (a warp alone
// issues a 16-byte shared load about every 13 cycles, and a reciprocal square
// root takes 18 cycles without the handling of subnormals, 42 with it).  Four
// 32-column steps, one thread per row (leaf_micro); the sub-panel below the
// diagonal block takes no time of its own and needs no inverse.  After each
// step all warps update the rest of the block; the stores of the finished
// columns and the 32 x 32 inverses are done by the idle warps during the next
// step.  Measured: 18.5 us per leaf launched back to back (of 31k cycles, 17.8k
// in the four steps' pivots, 7k in the updates between them); a whole solve of
// n = 16384 went from 27.96 to 25.26 ms against one pivot at a time, 21 us a leaf.
static __global__ void __launch_bounds__(LEAF_THREADS, 1) k_potrf_leaf32(float* __restrict__ W, long ldw, int k, int nb,
                                                               float* __restrict__ Dinv32, Mirror mir, DevStatus* st) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float* S = reinterpret_cast<float*>(smem_raw);           // [128][132] the block, then L
    float4* Xs = reinterpret_cast<float4*>(S + 128 * LDL);   // [8][32] rows of the micro-steps
    float* Rs = reinterpret_cast<float*>(Xs + 8 * 32);       // [128] reciprocals of the diagonal of L
    __shared__ int s_bad;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    pdl_wait();  // the update of this diagonal block is the previous kernel
    const int flags = *reinterpret_cast<const volatile int*>(&st->flags);
    if (nb == 128) {
        // 8 float4 per thread, all loads in flight before the stores
        float4 v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int e = tid + q * LEAF_THREADS, r = e >> 5, c4 = (e & 31) * 4;
            v[q] = *reinterpret_cast<const float4*>(W + (long)(k + r) * ldw + k + c4);
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int e = tid + q * LEAF_THREADS, r = e >> 5, c4 = (e & 31) * 4;
            float4 f = v[q];
            if (c4 + 0 > r) f.x = 0.f;
            if (c4 + 1 > r) f.y = 0.f;
            if (c4 + 2 > r) f.z = 0.f;
            if (c4 + 3 > r) f.w = 0.f;
            *reinterpret_cast<float4*>(S + r * LDL + c4) = f;
        }
    } else {  // ragged last block: identity beyond nb
        for (int e = tid; e < 128 * 128; e += LEAF_THREADS) {
            int r = e >> 7, c = e & 127;
            float v;
            if (r < nb && c < nb) v = (c <= r) ? W[(long)(k + r) * ldw + k + c] : 0.f;
            else v = (r == c) ? 1.f : 0.f;
            S[r * LDL + c] = v;
        }
    }
    if (tid == 0) s_bad = 0;
    if (flags & (SPD_DEV_BREAKDOWN | SPD_DEV_NONFINITE | SPD_DEV_BADDIAG)) return;  // an earlier block broke down
    __syncthreads();
    float* Dout = Dinv32 + (long)(k / 128) * 4096;

    constexpr int NW = LEAF_THREADS / 32;
    for (int o = 0; o < 128; o += 32) {
        if (o == 64 && tid == 0) pdl_trigger();  // the panel solve may start loading its rows
        const int nthr = 128 - o;                // threads 0 .. nthr - 1 hold rows o ..
        if (tid < nthr) {
            int badj = INT_MAX;
            float* row = S + (o + tid) * LDL + o;
            if (warp == 0) {
                leaf_step32<true>(row, lane, Xs, Rs + o, nthr, badj);
                if (badj < nb - o && lane == 0) {
                    s_bad = 1;
                    atomicMin(&st->info, k + o + badj + 1);
                    dev_raise(st, SPD_DEV_BREAKDOWN);
                }
            } else {
                leaf_step32<false>(row, lane, Xs, Rs + o, nthr, badj);
            }
        } else if (o > 0) {  // the previous step's inverse (the last warp) and its columns' stores
            if (warp == NW - 1) leaf_inverse32(S, o - 32, Rs + o - 32, Dout + (o / 32 - 1) * 1024, lane);
            else leaf_store_cols(S, W, ldw, k, nb, o - 32, mir, tid - nthr, LEAF_THREADS - 32 - nthr);
        }
        __syncthreads();
        if (s_bad) return;
        // the trailing update: groups of 32 columns, rows on or below the group's own
        const int b0 = o + 32;
        if (o == 96) break;
        if (o < 64) {  // 4-row units: 384 and 192 of them
            const int ng = (96 - o) >> 5, e = tid & 7, u = tid >> 3;
            // row quads below: 8 ng in group 0, 8 (ng - 1) in group 1, ...
            int g = 0, q = u;
            while (g < ng && q >= 8 * (ng - g)) q -= 8 * (ng - g), ++g;
            if (g < ng) leaf_tile<4>(S, o, b0 + 32 * g + 4 * q, b0 + 32 * g + e);
        } else if (tid < 256) {
            leaf_tile<1>(S, o, b0 + (tid >> 3), b0 + (tid & 7));
        }
        __syncthreads();
    }
    // the last block column and inverse (the others went out during the next step)
    if (warp == 0) leaf_inverse32(S, 96, Rs + 96, Dout + 3 * 1024, lane);
    else leaf_store_cols(S, W, ldw, k, nb, 96, mir, tid - 32, LEAF_THREADS - 32);
}

// Panel solve for rows [r0, r0 + m) against the factored diagonal block at
// column c0 (order 128): X L^T = B, in four 32-column steps s:
//   X_s = B_s D_s^T,   B_s' -= X_s L_s's^T  (s' > s),
// with D_s the 32x32 inverses the leaf stored.  CTA = 64 rows, two CTAs per SM.
// Bound: the loads from shared memory (16 bytes per thread and 2.4 cycles of the
// SM each) of a 4-row tile: thread (rows tr .. tr + 3, column class cg) owns the
// columns cg, cg + 16, .. of each product, so that eight lanes read eight
// consecutive rows of the right factor in distinct banks, four k at a time.
// Measured from the leaf's end to the solve's (globaltimer stamps): 6.4 us with
// one CTA on an SM (n = 2999; 12.4 us with scalar loads and one k at a time), 9.9
// us with two (n = 16384; 17 us).
#define LDB 132  // rows of B and L: 16-byte aligned, consecutive rows 4 banks apart
#define LDD 36   // rows of D likewise
constexpr size_t trsm_leaf32_smem() { return (size_t)(64 * LDB + 96 * LDB + 4 * 32 * LDD) * sizeof(float); }

// acc[j][q] += sum over four k of x[j] y[q]
template <int NQ>
__device__ __forceinline__ void trsm_fma4(float (&acc)[4][NQ], const float4 (&x)[4], const float4& y, int q) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        acc[j][q] = fmaf(x[j].x, y.x, acc[j][q]);
        acc[j][q] = fmaf(x[j].y, y.y, acc[j][q]);
        acc[j][q] = fmaf(x[j].z, y.z, acc[j][q]);
        acc[j][q] = fmaf(x[j].w, y.w, acc[j][q]);
    }
}

template <int S>
__device__ __forceinline__ void trsm_step(float* Bs, const float* Ls, const float* Ds, int tr, int cg) {
    constexpr int o = 32 * S, NQ = 6 - 2 * S;
    const float* br = Bs + tr * LDB + o;
    {   // X_s, columns o + cg and o + 16 + cg (D_s is lower triangular: the first ends at k = 15)
        float x[4][2] = {};
        const float* d0 = Ds + (o + cg) * LDD;
#pragma unroll
        for (int l = 0; l < 32; l += 4) {
            float4 b[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) b[j] = *reinterpret_cast<const float4*>(br + j * LDB + l);
            if (l < 16) trsm_fma4<2>(x, b, *reinterpret_cast<const float4*>(d0 + l), 0);
            trsm_fma4<2>(x, b, *reinterpret_cast<const float4*>(d0 + 16 * LDD + l), 1);
        }
        __syncthreads();  // every read of B_s done
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            Bs[(tr + j) * LDB + o + cg] = x[j][0];
            Bs[(tr + j) * LDB + o + 16 + cg] = x[j][1];
        }
    }
    __syncthreads();
    if constexpr (S < 3) {  // columns o + 32 + cg + 16 q
        float acc[4][NQ] = {};
        const float* lr = Ls + (o + cg) * LDB + o;  // Ls holds rows 32 .. of L_kk
#pragma unroll 2
        for (int l = 0; l < 32; l += 4) {
            float4 b[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) b[j] = *reinterpret_cast<const float4*>(br + j * LDB + l);
#pragma unroll
            for (int q = 0; q < NQ; ++q)
                trsm_fma4<NQ>(acc, b, *reinterpret_cast<const float4*>(lr + 16 * q * LDB + l), q);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int q = 0; q < NQ; ++q) Bs[(tr + j) * LDB + o + 32 + 16 * q + cg] -= acc[j][q];
        __syncthreads();
    }
}

// b_ready: the previous kernel in the stream (the leaf) does not write B, and
// what does was complete before the leaf passed its own wait, so B is loaded
// before waiting (programmatic dependent launch).
static __global__ void __launch_bounds__(256, 2) k_trsm_leaf32(float* __restrict__ W, long ldw, int r0, int m, int c0,
                                                     const float* __restrict__ Dinv32, Mirror mir,
                                                     const DevStatus* st, int b_ready) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float* Bs = reinterpret_cast<float*>(smem_raw);  // [64][132] B, becoming X
    float* Ls = Bs + 64 * LDB;                       // [96][132] rows 32..127 of L_kk, columns 0..95
    float* Ds = Ls + 96 * LDB;                       // [4][32][36] D_s
    const int tid = threadIdx.x;
    const int rb0 = r0 + blockIdx.x * 64;
    {
        if (!b_ready) pdl_wait();
        float4 vb[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {  // B: 64 rows x 128 columns
            const int e = tid + q * 256, r = e >> 5, c4 = (e & 31) * 4;
            vb[q] = (rb0 + r < r0 + m) ? *reinterpret_cast<const float4*>(W + (long)(rb0 + r) * ldw + c0 + c4)
                                       : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        if (b_ready) pdl_wait();  // L_kk and its inverses come from the previous kernel
        const int flags = *reinterpret_cast<const volatile int*>(&st->flags);
        // rows 32..127 of L_kk, columns 0..95 (the 32-blocks below the diagonal
        // are used) and the four 32x32 inverses: every load in flight first
        float4 vl[9], vd[4];
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            const int e = tid + q * 256, r = e / 24, c4 = (e - r * 24) * 4;
            vl[q] = *reinterpret_cast<const float4*>(W + (long)(c0 + 32 + r) * ldw + c0 + c4);
        }
        const float4* dg = reinterpret_cast<const float4*>(Dinv32 + (long)(c0 / 128) * 4096);
#pragma unroll
        for (int q = 0; q < 4; ++q) vd[q] = dg[tid + q * 256];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int e = tid + q * 256, r = e >> 5, c4 = (e & 31) * 4;
            *reinterpret_cast<float4*>(Bs + r * LDB + c4) = vb[q];
        }
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            const int e = tid + q * 256, r = e / 24, c4 = (e - r * 24) * 4;
            *reinterpret_cast<float4*>(Ls + r * LDB + c4) = vl[q];
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int e = tid + q * 256, r = e >> 3, c4 = (e & 7) * 4;
            *reinterpret_cast<float4*>(Ds + r * LDD + c4) = vd[q];
        }
        if (flags & (SPD_DEV_BREAKDOWN | SPD_DEV_NONFINITE | SPD_DEV_BADDIAG)) return;
    }
    __syncthreads();
    const int tr = (tid >> 4) * 4, cg = tid & 15;
    trsm_step<0>(Bs, Ls, Ds, tr, cg);
    trsm_step<1>(Bs, Ls, Ds, tr, cg);
    trsm_step<2>(Bs, Ls, Ds, tr, cg);
    trsm_step<3>(Bs, Ls, Ds, tr, cg);
    if (tid == 0) pdl_trigger();  // the next block column's update may be scheduled
    for (int e = tid; e < 64 * 32; e += 256) {
        const int rr = e >> 5, c4 = (e & 31) * 4;
        const long row = rb0 + rr;
        if (row >= r0 + m) continue;
        const float4 v = *reinterpret_cast<const float4*>(Bs + rr * LDB + c4);
        *reinterpret_cast<float4*>(W + row * ldw + c0 + c4) = v;
        mirror_store4(mir, row, (long)(c0 + c4), v);
    }
}

// The inverse of every 128x128 diagonal block (one CTA per block, after the
// factorisation), X = L_JJ^{-1} by block rows: X_ii = D_i (the leaf's 32x32
// inverses), X_i,0:i = -D_i (L_i,0:i X_0:i,0:i).  Kept transposed in shared memory,
// so that both products are of rows with rows, four k per load (leaf_tile's
// layout).  LinvT[l][c] = X[c][l]; with Xsb also X itself as diagonal block J mod
// sbb of super-block J / sbb (order 128 sbb).  Rows past n are the identity.
constexpr size_t block_inverse_smem() { return (size_t)(2 * 128 * LDL + 96 * 36 + 4 * 32 * 36) * sizeof(float); }

// 4 x 4 outputs: out[r][q] = sum over k in [k0, k1) (multiples of 4) of A[i + r][k] B[j + 8 q][k]
__device__ __forceinline__ void rowrow_tile(float (&acc)[4][4], const float* A, int lda, const float* B, int ldb, int k0,
                                            int k1) {
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[r][q] = 0.f;
#pragma unroll 2
    for (int k = k0; k < k1; k += 4) {
        float4 x[4], y[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) x[r] = *reinterpret_cast<const float4*>(A + r * lda + k);
#pragma unroll
        for (int q = 0; q < 4; ++q) y[q] = *reinterpret_cast<const float4*>(B + 8 * q * ldb + k);
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                acc[r][q] = fmaf(x[r].x, y[q].x, acc[r][q]);
                acc[r][q] = fmaf(x[r].y, y[q].y, acc[r][q]);
                acc[r][q] = fmaf(x[r].z, y[q].z, acc[r][q]);
                acc[r][q] = fmaf(x[r].w, y[q].w, acc[r][q]);
            }
    }
}

static __global__ void __launch_bounds__(256) k_block_inverse(const float* __restrict__ W, long ldw, int n,
                                                       const float* __restrict__ Dinv32, float* __restrict__ LinvT,
                                                       float* __restrict__ Xsb, int sbb) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float* S = reinterpret_cast<float*>(smem_raw);  // [128][132] L_JJ
    float* XT = S + 128 * LDL;                      // [128][132] (L_JJ^{-1})^T
    float* TT = XT + 128 * LDL;                     // [96][36] (L_i,0:i X_0:i,0:i)^T
    float* Ds = TT + 96 * 36;                       // [4][32][36] D_i
    const int tid = threadIdx.x;
    const int J = blockIdx.x;
    const long k = (long)J * 128;
    const int nb = (int)min((long)128, n - k);
    const float* dg = Dinv32 + (long)J * 4096;
    for (int e = tid; e < 128 * 32; e += 256) {
        const int r = e >> 5, c4 = (e & 31) * 4;
        float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
        if (r < nb && k + c4 < ldw) f = *reinterpret_cast<const float4*>(W + (k + r) * ldw + k + c4);
        float v[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int c = c4 + q;
            if (r >= nb || c >= nb) v[q] = (r == c) ? 1.f : 0.f;
            else if (c > r) v[q] = 0.f;
        }
        *reinterpret_cast<float4*>(S + r * LDL + c4) = make_float4(v[0], v[1], v[2], v[3]);
        *reinterpret_cast<float4*>(XT + r * LDL + c4) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncthreads();
    for (int e = tid; e < 4096; e += 256) {  // D_b[r][c] (zeros above its diagonal)
        const int b = e >> 10, r = (e >> 5) & 31, c = e & 31;
        const float v = dg[e];
        Ds[(b * 32 + r) * 36 + c] = v;
        XT[(32 * b + c) * LDL + 32 * b + r] = v;
    }
    __syncthreads();
    for (int i = 1; i < 4; ++i) {
        const int ri = 32 * i;
        float acc[4][4];
        for (int e = tid; e < 64 * i; e += 256) {  // T[r][c]: 4 rows x columns c, c + 8, ..; k from c's block on
            const int cb = e >> 6, r = ((e >> 3) & 7) * 4, c = 32 * cb + (e & 7);
            rowrow_tile(acc, S + (ri + r) * LDL, LDL, XT + c * LDL, LDL, 32 * cb, ri);
#pragma unroll
            for (int q = 0; q < 4; ++q)
                *reinterpret_cast<float4*>(TT + (c + 8 * q) * 36 + r) =
                    make_float4(acc[0][q], acc[1][q], acc[2][q], acc[3][q]);
        }
        __syncthreads();
        for (int e = tid; e < 64 * i; e += 256) {  // X[ri + r][c] = -sum_q D_i[r][q] T[q][c]
            const int cb = e >> 6, r = ((e >> 3) & 7) * 4, c = 32 * cb + (e & 7);
            rowrow_tile(acc, Ds + (32 * i + r) * 36, 36, TT + c * 36, 36, 0, 32);
#pragma unroll
            for (int q = 0; q < 4; ++q)
                *reinterpret_cast<float4*>(XT + (c + 8 * q) * LDL + ri + r) =
                    make_float4(-acc[0][q], -acc[1][q], -acc[2][q], -acc[3][q]);
        }
        __syncthreads();
    }
    float* out = LinvT + (long)J * 16384;
    for (int e = tid; e < 128 * 32; e += 256) {
        const int l = e >> 5, c4 = (e & 31) * 4;
        *reinterpret_cast<float4*>(out + l * 128 + c4) = *reinterpret_cast<const float4*>(XT + l * LDL + c4);
    }
    if (Xsb) {
        const long ld = (long)sbb * 128;
        float* xo = Xsb + (long)(J / sbb) * ld * ld + (long)(J % sbb) * 128 * (ld + 1);
        for (int e = tid; e < 128 * 128; e += 256) {
            const int r = e >> 7, c = e & 127;
            xo[r * ld + c] = XT[c * LDL + r];
        }
    }
}

// k_batched.cuh -- many independent SPD systems of uneven order (n <= 512)
// solved in one persistent launch: Algorithm 1 (low-precision Cholesky +
// float64 refinement) or Jacobi-preconditioned CG, one system per CTA at a
// time.  CTAs take systems from a shared counter over a list sorted by
// decreasing n, so the long systems start first.  Every system is processed
// by exactly one CTA with a fixed sequence of operations, so its result
// does not depend on the schedule.
//
// Per-CTA scratch in global memory (L2-resident): the scaled working
// matrix W (column-major lower, ld 512, float32).  Shared memory holds the
// 32x32 diagonal-block inverses (packed lower triangles), the current panel, and
// the vectors: 112 KB, so that two CTAs of 256 threads share an SM and one's
// pivots and barriers run beside the other's products.  4096 systems of order 32
// .. 512: 11.9 ms (20.6 with one CTA per SM, single pivots by shuffles, and a warp
// per row in the back substitution).
#pragma once
#include "common.cuh"
#include "k_leaf32.cuh"

#define BMAX 512           // largest system order
#define BLD 512            // leading dimension of the per-CTA working matrix
#define BPANEL 32

struct BatchSys {
    const double* A;  // n x n, column-major, lda
    const double* B;  // n
    double* X;        // n
    int n, lda;
};

struct BatchRep {
    int status;   // SPD_OK, SPD_ERR_NOT_SPD, SPD_ERR_NO_CONVERGENCE
    int info;     // failing column (1-based) on breakdown
    int iters;    // refinement sweeps / CG steps
    int pad;
    double berr;  // final normwise backward error
};

struct BatchArgs {
    const BatchSys* sys;
    const int* order;    // system indices, decreasing n
    int count;
    int* next;           // work counter (zeroed before the launch)
    float* scratch;      // per CTA: BLD * BLD floats
    BatchRep* rep;
    int prec;            // SPD_PREC_FP32 / BF16 / FP16: rounding of the update operands
    double tol;
    int maxit;
    int polish;
};

// The panel's rows transposed: PnT[l * BLDP + i] = L[i][k0 + l] (rounded to the
// update type), rows contiguous so that four rows are one 16-byte load.
#define BLDP 516
#define BTRI 528  // entries of a 32 x 32 lower triangle
__device__ __forceinline__ constexpr int btri(int r) { return r * (r + 1) / 2; }
constexpr size_t batch_smem_bytes() {
    return (size_t)(BMAX / 32) * BTRI * sizeof(float)  // Inv
           + (size_t)32 * BLDP * sizeof(float)         // panel
           + (size_t)3 * BMAX * sizeof(double)         // x, r, d
           + (size_t)BMAX * sizeof(float);             // y
}
constexpr size_t batch_pcg_smem_bytes() { return (size_t)6 * BMAX * sizeof(double); }

__device__ __forceinline__ float round_op(float v, int prec) {
    if (prec == 3) return __bfloat162float(__float2bfloat16_rn(v));  // SPD_PREC_BF16
    if (prec == 4) return __half2float(__float2half_rn(v));          // SPD_PREC_FP16
    return v;
}

template <int NT>
__device__ double block_max(double v, double* red) {
    v = warp_max(v);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    double r = 0.0;
    for (int w = 0; w < NT / 32; ++w) r = fmax(r, red[w]);
    __syncthreads();
    return r;
}
template <int NT>
__device__ double block_sum(double v, double* red) {
    v = warp_sum(v);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    double r = 0.0;
    for (int w = 0; w < NT / 32; ++w) r += red[w];  // fixed order
    __syncthreads();
    return r;
}

// y <- (L L^T)^{-1} y in place (float32, shared memory, zero from n to the next
// multiple of 32) with the factor in W and the diagonal-block inverses in Inv.
// One thread per row for the updates; the row's 32 entries of L (forward: a
// strided row, coalesced across threads; backward: 128 contiguous bytes of its
// column) are in flight while warp 0 applies the block's inverse.
template <int NT>
__device__ void batch_lsolve(const float* W, const float* Inv, float* y, int n) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nb = (n + 31) / 32;
    for (int kb = 0; kb < nb; ++kb) {  // forward
        const int k0 = kb * 32;
        int i = k0 + 32 + tid;
        float w[32];
        if (i < n) {
#pragma unroll
            for (int c = 0; c < 32; ++c) w[c] = W[i + (long)(k0 + c) * BLD];
        }
        if (warp == 0) {
            const float* I = Inv + kb * BTRI + btri(lane);
            float s0 = 0.f, s1 = 0.f;
#pragma unroll
            for (int l = 0; l < 32; l += 2) {
                if (l <= lane) s0 = fmaf(I[l], y[k0 + l], s0);
                if (l + 1 <= lane) s1 = fmaf(I[l + 1], y[k0 + l + 1], s1);
            }
            __syncwarp();
            if (k0 + lane < n) y[k0 + lane] = s0 + s1;
        }
        __syncthreads();
        while (i < n) {
            float s = 0.f;
#pragma unroll
            for (int c = 0; c < 32; ++c) s = fmaf(w[c], y[k0 + c], s);
            y[i] -= s;
            i += NT;
            if (i < n) {
#pragma unroll
                for (int c = 0; c < 32; ++c) w[c] = W[i + (long)(k0 + c) * BLD];
            }
        }
        __syncthreads();
    }
    for (int kb = nb - 1; kb >= 0; --kb) {  // backward
        const int k0 = kb * 32;
        int i = tid;
        float w[32];
        auto load = [&]() {
            const float4* p = reinterpret_cast<const float4*>(W + (long)i * BLD + k0);
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const float4 v = p[q];
                w[4 * q] = v.x;
                w[4 * q + 1] = v.y;
                w[4 * q + 2] = v.z;
                w[4 * q + 3] = v.w;
            }
            if (k0 + 32 > n) {  // rows past n hold another system's values
#pragma unroll
                for (int c = 0; c < 32; ++c)
                    if (k0 + c >= n) w[c] = 0.f;
            }
        };
        if (i < k0) load();
        if (warp == 0) {
            const float* I = Inv + kb * BTRI + lane;
            float s0 = 0.f, s1 = 0.f;
#pragma unroll
            for (int l = 0; l < 32; l += 2) {
                if (l >= lane) s0 = fmaf(I[btri(l)], y[k0 + l], s0);
                if (l + 1 >= lane) s1 = fmaf(I[btri(l + 1)], y[k0 + l + 1], s1);
            }
            __syncwarp();
            if (k0 + lane < n) y[k0 + lane] = s0 + s1;
        }
        __syncthreads();
        while (i < k0) {
            float s = 0.f;
#pragma unroll
            for (int c = 0; c < 32; ++c) s = fmaf(w[c], y[k0 + c], s);
            y[i] -= s;
            i += NT;
            if (i < k0) load();
        }
        __syncthreads();
    }
}

// The Cholesky factor of a 32 x 32 diagonal block by one warp (lane = row, a[] =
// the row's columns; micro-steps of four pivots, k_leaf32.cuh): L back into a[]
// and, four columns at a time, into Xs (8 x 32 float4), the reciprocals of its
// diagonal into Rs.  Returns the first non-positive pivot (INT_MAX: none).
__device__ __forceinline__ int batch_diag32(float (&a)[32], int lane, float4* Xs, float* Rs) {
    int bad = INT_MAX;
    leaf_micro<0, true>(a, lane, Xs, Rs, 32, bad);
    leaf_micro<1, true>(a, lane, Xs, Rs, 32, bad);
    leaf_micro<2, true>(a, lane, Xs, Rs, 32, bad);
    leaf_micro<3, true>(a, lane, Xs, Rs, 32, bad);
    leaf_micro<4, true>(a, lane, Xs, Rs, 32, bad);
    leaf_micro<5, true>(a, lane, Xs, Rs, 32, bad);
    leaf_micro<6, true>(a, lane, Xs, Rs, 32, bad);
    leaf_micro<7, true>(a, lane, Xs, Rs, 32, bad);
    return bad;
}

// Its inverse (lane = column: x_i = (delta - sum_{l<i} L_il x_l) / L_ii): the lower
// triangle packed into I, rows of 36 with zeros above the diagonal into D.
__device__ __forceinline__ void batch_inverse32(int lane, const float4* Xs, const float* Rs, float* I, float* D) {
    float x[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) {
        float s0 = (i == lane) ? 1.f : 0.f, s1 = 0.f;
#pragma unroll
        for (int l = 0; l < i; l += 4) {
            const float4 t = Xs[(l >> 2) * 32 + i];
            s0 = fmaf(-t.x, x[l], s0);
            if (l + 1 < i) s1 = fmaf(-t.y, x[l + 1], s1);
            if (l + 2 < i) s0 = fmaf(-t.z, x[l + 2], s0);
            if (l + 3 < i) s1 = fmaf(-t.w, x[l + 3], s1);
        }
        x[i] = (s0 + s1) * Rs[i];
        if (lane <= i) I[btri(i) + lane] = x[i];
        D[i * 36 + lane] = lane <= i ? x[i] : 0.f;
    }
}

// sum_j A_ij x_j (float64), and with ABS sum_j |A_ij|: four interleaved
// accumulators (column j into j % 4), eight loads in flight, added in a fixed
// order.  (Four threads per row, a column quarter each, so that the four
// schedulers' float64 units have equal work, and loads one group ahead, measured
// no faster.)
template <bool ABS>
__device__ __forceinline__ double batch_row_dot(const BatchSys& S, const double* x, int i, double& abs_sum) {
    const double* Ai = S.A + i;
    double q[4] = {0.0, 0.0, 0.0, 0.0}, a = 0.0;
    int j = 0;
    for (; j + 8 <= S.n; j += 8) {
        double v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = Ai[(long)(j + u) * S.lda];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            q[u & 3] = fma(v[u], x[j + u], q[u & 3]);
            if (ABS) a += fabs(v[u]);
        }
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        if (j + u < S.n) {
            const double v = Ai[(long)(j + u) * S.lda];
            q[u & 3] = fma(v, x[j + u], q[u & 3]);
            if (ABS) a += fabs(v);
        }
    }
    abs_sum = a;
    return (q[0] + q[1]) + (q[2] + q[3]);
}

// |v| for a maximum that decides convergence: NaN counts as infinity (fmax drops it)
__device__ __forceinline__ double abs_or_inf(double v) { return v == v ? fabs(v) : INFINITY; }

// The block's sum of s and maxima of m1 and m2, one pass (red: 3 NT / 32 values)
template <int NT>
__device__ __forceinline__ void block_sum_max2(double& s, double& m1, double& m2, double* red) {
    constexpr int NW = NT / 32;
    s = warp_sum(s);
    m1 = warp_max(m1);
    m2 = warp_max(m2);
    if ((threadIdx.x & 31) == 0) {
        red[threadIdx.x >> 5] = s;
        red[NW + (threadIdx.x >> 5)] = m1;
        red[2 * NW + (threadIdx.x >> 5)] = m2;
    }
    __syncthreads();
    s = m1 = m2 = 0.0;
    for (int w = 0; w < NW; ++w) {  // fixed order
        s += red[w];
        m1 = fmax(m1, red[NW + w]);
        m2 = fmax(m2, red[2 * NW + w]);
    }
    __syncthreads();
}

// r = b - A x (float64) for one system; returns berr = ||r||_inf / (anorm
// ||x||_inf), infinity where r is not finite; with want_anorm anorm = ||A||_inf is
// formed first.  x is complete (a barrier before the call).
template <int NT>
__device__ double batch_residual(const BatchSys& S, const double* x, double* r, bool want_anorm, double* red,
                                 double* anorm) {
    double rmax = 0.0, amax = 0.0, xmax = 0.0, none = 0.0;
    for (int i = threadIdx.x; i < S.n; i += NT) {
        double a = 0.0;
        const double s = S.B[i] - (want_anorm ? batch_row_dot<true>(S, x, i, a) : batch_row_dot<false>(S, x, i, a));
        r[i] = s;
        rmax = fmax(rmax, abs_or_inf(s));
        xmax = fmax(xmax, fabs(x[i]));
        amax = fmax(amax, a);
    }
    block_sum_max2<NT>(none, rmax, xmax, red);
    if (want_anorm) {
        amax = block_max<NT>(amax, red);
        if (threadIdx.x == 0) *anorm = amax;
        __syncthreads();
    }
    const double an = *anorm;
    if (rmax == INFINITY) return INFINITY;
    // (x = 0 solves b = 0 only)
    return (an > 0.0 && xmax > 0.0) ? rmax / (an * xmax) : rmax > 0.0 ? INFINITY : 0.0;
}

template <int NT>
__global__ void __launch_bounds__(NT, 512 / NT) k_batch_chol_ir(BatchArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float* Inv = reinterpret_cast<float*>(smem_raw);           // [16][528]
    float* Pn = Inv + (BMAX / 32) * BTRI;                      // [32][516]
    double* xs = reinterpret_cast<double*>(Pn + 32 * BLDP);    // [512]
    double* rs = xs + BMAX;
    double* ds = rs + BMAX;
    float* ys = reinterpret_cast<float*>(ds + BMAX);           // [512]
    // scratch of the factor: the diagonal block's rows before the panel is
    // formed, its inverse by rows before the solution is
    float4* Xs = reinterpret_cast<float4*>(Pn);                // [8][32]
    float* Rs = Pn + 8 * 32 * 4;                               // [32]
    float* D = reinterpret_cast<float*>(xs);                   // [32][36]
    __shared__ int s_idx, s_bad;
    __shared__ double red[3 * NT / 32];
    __shared__ double s_anorm;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    float* W = a.scratch + (long)blockIdx.x * BLD * BLD;

    for (;;) {
        if (tid == 0) s_idx = atomicAdd(a.next, 1);
        __syncthreads();
        if (s_idx >= a.count) break;
        const int sid = a.order[s_idx];
        const BatchSys S = a.sys[sid];
        const int n = S.n;
        // scaling and conversion (A0): W[i][j] = d_i A_ij d_j, j <= i
        for (int i = tid; i < n; i += NT) {
            const double v = S.A[i + (long)i * S.lda];
            ds[i] = (v > 0.0) ? 1.0 / sqrt(v) : 1.0;
        }
        if (tid == 0) s_bad = 0;
        __syncthreads();
        // (a warp per column of the lower triangle, four loads in flight per lane)
        for (int j = warp; j < n; j += NT / 32) {
            const double dj = ds[j];
            const double* aj = S.A + (long)j * S.lda;
            float* wj = W + (long)j * BLD;
            for (int i0 = j + lane; i0 < n; i0 += 128) {
                double v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) v[u] = i0 + 32 * u < n ? aj[i0 + 32 * u] : 0.0;
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (i0 + 32 * u < n) wj[i0 + 32 * u] = (float)(ds[i0 + 32 * u] * v[u] * dj);
            }
        }
        __syncthreads();
        // factor (A1-A3) by 32-column panels
        const int nb = (n + 31) / 32;
        // (s_bad is read only behind the barrier after the diagonal block: in the loop's
        // condition a late warp could meet this block's value and leave the others there)
        for (int kb = 0; kb < nb; ++kb) {
            const int k0 = kb * 32;
            if (warp == 0) {
                float av[32];
#pragma unroll
                for (int c = 0; c < 32; ++c) {
                    const int r = k0 + lane, cc = k0 + c;
                    av[c] = (r < n && cc < n) ? ((c <= lane) ? W[r + (long)cc * BLD] : 0.f) : (lane == c ? 1.f : 0.f);
                }
                const int badj = batch_diag32(av, lane, Xs, Rs);
#pragma unroll
                for (int c = 0; c < 32; ++c)
                    if (k0 + lane < n && k0 + c < n && c <= lane) W[k0 + lane + (long)(k0 + c) * BLD] = av[c];
                if (badj < n - k0 && lane == 0) {
                    s_bad = 1;
                    a.rep[sid].info = k0 + badj + 1;
                }
                __syncwarp();
                batch_inverse32(lane, Xs, Rs, Inv + kb * BTRI, D);
            }
            __syncthreads();
            if (s_bad) break;
            const int R = n - k0 - 32;
            if (R <= 0) break;
            // panel: rows below, X = B D^T
            for (int i = tid; i < R; i += NT) {
                float b[32];
#pragma unroll
                for (int c = 0; c < 32; ++c) b[c] = W[(k0 + 32 + i) + (long)(k0 + c) * BLD];
#pragma unroll
                for (int g = 0; g < 4; ++g) {  // D is zero above its diagonal
#pragma unroll 2
                    for (int c = 8 * g; c < 8 * g + 8; ++c) {
                        float s0 = 0.f, s1 = 0.f;
#pragma unroll
                        for (int l = 0; l < 8 * g + 8; l += 4) {
                            const float4 d = *reinterpret_cast<const float4*>(D + c * 36 + l);
                            s0 = fmaf(b[l], d.x, s0);
                            s1 = fmaf(b[l + 1], d.y, s1);
                            s0 = fmaf(b[l + 2], d.z, s0);
                            s1 = fmaf(b[l + 3], d.w, s1);
                        }
                        W[(k0 + 32 + i) + (long)(k0 + c) * BLD] = s0 + s1;
                        Pn[c * BLDP + i] = round_op(s0 + s1, a.prec);
                    }
                }
            }
            for (int e = tid; e < 32 * 4; e += NT) Pn[(e >> 2) * BLDP + R + (e & 3)] = 0.f;  // rows R.. of the last group
            __syncthreads();
            // trailing update of the lower part, 4x4 register blocks: consecutive
            // threads take consecutive row groups bi of one column group bj, so
            // that the panel reads are 16-byte broadcasts or contiguous and the
            // updates of W are contiguous rows of a column
            const int Rb = (R + 3) / 4;
            for (int e = tid; e < Rb * Rb; e += NT) {
                const int bj = e / Rb, bi = e - bj * Rb;
                if (bj > bi) continue;
                float acc[4][4] = {};
#pragma unroll 8
                for (int l = 0; l < 32; ++l) {
                    const float4 pi = *reinterpret_cast<const float4*>(Pn + l * BLDP + 4 * bi);
                    const float4 pj = *reinterpret_cast<const float4*>(Pn + l * BLDP + 4 * bj);
                    const float ip[4] = {pi.x, pi.y, pi.z, pi.w}, jq[4] = {pj.x, pj.y, pj.z, pj.w};
#pragma unroll
                    for (int p = 0; p < 4; ++p)
#pragma unroll
                        for (int q = 0; q < 4; ++q) acc[p][q] = fmaf(ip[p], jq[q], acc[p][q]);
                }
                const bool full = (bi > bj) && (4 * bi + 3 < R);  // four rows inside, below the diagonal block
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int j = 4 * bj + q;
                    if (j >= R) break;
                    float* w = W + (k0 + 32 + 4 * bi) + (long)(k0 + 32 + j) * BLD;
                    if (full) {
                        float4 v = *reinterpret_cast<float4*>(w);
                        v.x -= acc[0][q];
                        v.y -= acc[1][q];
                        v.z -= acc[2][q];
                        v.w -= acc[3][q];
                        *reinterpret_cast<float4*>(w) = v;
                    } else {
#pragma unroll
                        for (int p = 0; p < 4; ++p) {
                            const int i = 4 * bi + p;
                            if (i < R && j <= i) w[p] -= acc[p][q];
                        }
                    }
                }
            }
            __syncthreads();
        }
        if (s_bad) {
            if (tid == 0) {
                a.rep[sid].status = SPD_ERR_NOT_SPD;
                a.rep[sid].iters = 0;
                a.rep[sid].berr = INFINITY;
            }
            __syncthreads();
            continue;
        }
        // refinement (Algorithm 1, lines 2-7); it = -1 is line 2's solve
        for (int i = tid; i < n; i += NT) {
            rs[i] = S.B[i];
            xs[i] = 0.0;
        }
        __syncthreads();
        int it = -1, extra = a.polish;
        bool conv = false;
        double berr = 0.0;
        for (;;) {
            for (int i = tid; i < 32 * nb; i += NT) ys[i] = i < n ? (float)(ds[i] * rs[i]) : 0.f;
            __syncthreads();
            batch_lsolve<NT>(W, Inv, ys, n);
            for (int i = tid; i < n; i += NT) xs[i] += ds[i] * (double)ys[i];
            __syncthreads();
            berr = batch_residual<NT>(S, xs, rs, it < 0, red, &s_anorm);
            ++it;
            if (berr <= a.tol) {
                if (extra <= 0) {
                    conv = true;
                    break;
                }
                --extra;
            } else {
                extra = a.polish;
            }
            if (it >= a.maxit) break;
        }
        for (int i = tid; i < n; i += NT) S.X[i] = xs[i];
        if (tid == 0) {
            a.rep[sid].status = conv ? SPD_OK : SPD_ERR_NO_CONVERGENCE;
            a.rep[sid].iters = it;
            a.rep[sid].berr = berr;
        }
        __syncthreads();
    }
}

// Jacobi-preconditioned CG in float64 per system (x0 = 0), restarted from
// the true residual when the recursive one claims convergence but the true
// backward error does not meet the tolerance.  Bound: the float64 rate (n^2
// multiply-adds a step, one SM's float64 units take two a cycle); two CTAs of 256
// threads share an SM to keep them busy through each other's reductions: 512
// systems of order 32 .. 256 take 5.65 ms with one, 5.25 with two, 7.4 with three
// (the systems no longer stay in the SM's L1).
template <int NT>
__global__ void __launch_bounds__(NT, 512 / NT) k_batch_pcg(BatchArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double* xs = reinterpret_cast<double*>(smem_raw);
    double* rs = xs + BMAX;
    double* ps = rs + BMAX;
    double* zs = ps + BMAX;
    double* qs = zs + BMAX;
    double* dinv = qs + BMAX;
    __shared__ int s_idx;
    __shared__ double red[3 * NT / 32];
    __shared__ double s_anorm;
    const int tid = threadIdx.x;
    for (;;) {
        if (tid == 0) s_idx = atomicAdd(a.next, 1);
        __syncthreads();
        if (s_idx >= a.count) break;
        const int sid = a.order[s_idx];
        const BatchSys S = a.sys[sid];
        const int n = S.n;
        for (int i = tid; i < n; i += NT) {
            dinv[i] = 1.0 / S.A[i + (long)i * S.lda];
            xs[i] = 0.0;
        }
        __syncthreads();
        double berr = batch_residual<NT>(S, xs, rs, true, red, &s_anorm);
        int it = 0;
        bool conv = false;
        for (int restart = 0; restart < 4 && !conv; ++restart) {
            double rho = 0.0, xmax = 0.0, rmax = 0.0;
            for (int i = tid; i < n; i += NT) {
                const double r = rs[i], z = dinv[i] * r;
                zs[i] = z;
                ps[i] = z;
                rho += r * z;
                xmax = fmax(xmax, fabs(xs[i]));
                rmax = fmax(rmax, fabs(r));
            }
            block_sum_max2<NT>(rho, xmax, rmax, red);  // its barriers also publish ps
            for (; it < a.maxit; ++it) {
                // (r = 0: b = 0, or nothing left to reduce; alpha would be 0 / 0.  A maximum
                // of nothing but NaN is 0 too, and the residual below tells the two apart; by
                // its bits, since a float64 comparison is on the step's chain)
                if (__double_as_longlong(rmax) == 0ll || (xmax > 0.0 && rmax <= 0.5 * a.tol * s_anorm * xmax)) break;
                double pq = 0.0;
                for (int i = tid; i < n; i += NT) {
                    double none;
                    const double s = batch_row_dot<false>(S, ps, i, none);
                    qs[i] = s;
                    pq += ps[i] * s;
                }
                pq = block_sum<NT>(pq, red);
                const double alpha = rho / pq;
                double rz = 0.0;
                xmax = rmax = 0.0;
                for (int i = tid; i < n; i += NT) {
                    const double x = fma(alpha, ps[i], xs[i]), r = fma(-alpha, qs[i], rs[i]), z = dinv[i] * r;
                    xs[i] = x;
                    rs[i] = r;
                    zs[i] = z;
                    rz += r * z;
                    xmax = fmax(xmax, fabs(x));
                    rmax = fmax(rmax, fabs(r));
                }
                block_sum_max2<NT>(rz, xmax, rmax, red);
                const double beta = rz / rho;
                rho = rz;
                for (int i = tid; i < n; i += NT) ps[i] = fma(beta, ps[i], zs[i]);
                __syncthreads();
            }
            berr = batch_residual<NT>(S, xs, rs, false, red, &s_anorm);
            conv = berr <= a.tol;
            if (it >= a.maxit) break;
        }
        for (int i = tid; i < n; i += NT) S.X[i] = xs[i];
        if (tid == 0) {
            a.rep[sid].status = conv ? SPD_OK : SPD_ERR_NO_CONVERGENCE;
            a.rep[sid].iters = it;
            a.rep[sid].berr = berr;
            a.rep[sid].info = 0;
        }
        __syncthreads();
    }
}

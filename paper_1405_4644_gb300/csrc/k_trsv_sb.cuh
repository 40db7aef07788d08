// k_trsv_sb.cuh -- step A4 (Algorithm 1, lines 2 and 5) over diagonal
// super-blocks: the float32 sweeps y = L^{-1} y and z = L^{-T} z with the
// explicit inverses X_I = L_II^{-1} of the diagonal super-blocks (SBB
// 128-blocks each, S = 128 SBB rows), formed once per factor.
//
// Forward, super-block by super-block (I = 0, 1, ...):
//   y_I = X_I r_I,   then   r_J -= L_JI y_I  for every 128-row block J below,
// backward (I = last, ..., 0):
//   z_I = X_I^T y_I, then   y_K -= L_IK^T z_I  for every 128-row block K above,
// i.e. block substitution with the diagonal solve replaced by a product with
// the inverse.  One persistent cooperative kernel per sweep runs two grid-wide
// phases per super-block, separated by bounded grid barriers (a factor of one
// super-block has phase F alone, no barrier, and is launched as an ordinary kernel):
//   F   the SBB (SBB + 1) / 2 tile products X_I[b][c] r_I[c] (c <= b; for the
//       backward sweep X_I[c][b]^T r_I[c], c >= b) into partial tiles; the
//       last tile of block row b to arrive (an atomic count) adds the row's
//       partials in a fixed order into y_I[b], written to the output vector
//       (never over r_I, which other tiles of the phase may still read); and
//       the fix-up of the previous panel update's split rows (below);
//   B   the panel update: units (J, c) = the tile L_{J, I c} (backward
//       L_{I c, J}^T) times y_I[c], J-major over every remaining 128-row block
//       J, in equal contiguous ranges over all CTAs ("stream-K"), so the
//       panel of L streams through every SM.  A CTA whose range covers a
//       whole block row subtracts its sum from r_J; the pieces of a row shared
//       by several CTAs go to partial slots (2g for CTA g's first piece, 2g+1
//       for its last), which the next phase F adds in CTA order (= c order):
//       folded into the staged rows of the next super-block's tile products,
//       subtracted from r_J for every other row.
// Every result is formed in an order fixed by the launch's grid, not by
// timing.  The chain of the 128-block sweeps (one cross-SM hand-over per 128
// rows) becomes two barriers per S rows.  The right-hand sides Y are reduced
// in place and the result goes to O (forward: Y = the caller's vectors, O =
// scratch; backward: Y = that scratch, O = the caller's vectors).  The product of a 128x128 tile
// with a 128 x MC block uses the register tiles of k_trsv32.cuh.
#pragma once
#include "k_trsv32.cuh"

struct SbArgs {
    const float* W;       // factor rows (row-major, lower), ldw
    long ldw;
    int n, NB;            // order and number of 128-blocks
    const float* X;       // super-block inverses: NS blocks of S x S floats, row-major
    int S, SBB, NS;       // super-block order (= 128 SBB), 128-blocks per super-block, super-blocks
    float* Y;             // right-hand sides, n x m column-major (ld n), reduced in place
    int c0, mc;           // columns [c0, c0 + mc) of Y in this pass
    float* O;             // the sweep's result, column-major (ld n), columns [oc0, oc0 + mc)
    int oc0;
    float* P;             // partial tiles of phase F: SBB (SBB + 1) / 2 x 128 x MC floats
    float* P2;            // partial slots of phase B: 2 gridDim.x x 128 x MC floats
    int* bar;             // [0] barrier arrivals, [1] abort, then NS SBB block-row tile counts (zero at launch)
    unsigned long long wait_ns;
    DevStatus* st;
    const int* gate;      // (may be NULL) return at once when *gate == 0
    // column groups of MC columns swept side by side (blockIdx.y = group): the
    // columns of all groups from c0 / oc0 on, and the groups' strides of P, P2, bar
    int mtot;
    long pstride, p2stride;
    int barstride;
};

// Grid-wide barrier: the k-th barrier of a launch waits for k * gridDim.x
// arrivals (bounded; a CTA that gives up raises SPD_DEV_TIMEOUT and the abort
// flag, which releases the others).  Every write before it is visible after.
__device__ __forceinline__ bool sb_barrier(const SbArgs& a, int k, int* s_abort) {
    __syncthreads();
    if (threadIdx.x == 0 && !*s_abort) {
        __threadfence();
        atomicAdd(a.bar, 1);
        const int target = k * (int)gridDim.x;
        if (ld_acquire(a.bar) < target) {
            const uint64_t t0 = tv_globaltimer();
            while (ld_acquire(a.bar) < target) {
                if (ld_acquire(a.bar + 1)) {
                    *s_abort = 1;
                    break;
                }
                if (tv_globaltimer() - t0 > a.wait_ns) {
                    *s_abort = 1;
                    atomicOr(&a.st->flags, SPD_DEV_TIMEOUT);
                    atomicExch(a.bar + 1, 1);
                    break;
                }
            }
        }
        __threadfence();
    }
    __syncthreads();
    return !*s_abort;
}

// Geometry of one panel update (phase B): units u = (J - J0) nb + c for
// J0 <= J < J0 + rows, c < nb; CTA g < geff takes [g W / geff, (g+1) W / geff).
struct SbPanel {
    int J0, nb, geff;
    long W;
};
__device__ __forceinline__ long sb_ub(int g, long W, int G) { return (long)g * W / G; }

// The partial slots of block row J of panel pn in CTA order (= c order):
// returns their count (0: one CTA covered the row, nothing pending); slots
// are slot_lo, 2 (glo + 1), ..., 2 ghi.
__device__ __forceinline__ int sb_row_slots(const SbPanel& pn, int J, int& slot_lo, int& glo) {
    const long ut0 = (long)(J - pn.J0) * pn.nb, ut1 = ut0 + pn.nb;
    glo = (int)(((ut0 + 1) * pn.geff - 1) / pn.W);  // owner of the row's first unit
    const int ghi = (int)((ut1 * pn.geff - 1) / pn.W);
    if (glo == ghi) return 0;
    slot_lo = 2 * glo + (sb_ub(glo, pn.W, pn.geff) < ut0 ? 1 : 0);
    return ghi - glo + 1;
}

// Block row J's pending partial sum, for this thread's elements e = tid +
// 256 u (row l = e & 127, column c = e >> 7): the row's slots added in CTA
// order, each slot's loads issued together.
template <int MC, int PER>
__device__ __forceinline__ void sb_pending(const SbArgs& a, int ns, int slot_lo, int glo, float (&pend)[PER]) {
#pragma unroll
    for (int u = 0; u < PER; ++u) pend[u] = 0.f;
    for (int k = 0; k < ns; ++k) {
        const float* ps = a.P2 + (long)(k == 0 ? slot_lo : 2 * (glo + k)) * 128 * MC;
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            const int e = threadIdx.x + u * 256, l = e & 127, c = e >> 7;
            if (e < 128 * MC) pend[u] += __ldcg(ps + l * MC + c);
        }
    }
}

// 64 tile entries into registers as tv_tile, in 16-byte loads of whole lines (with
// pieces of lines the sweeps were bound by the passes through L1: busy 43 and 53 % of
// the time at n = 8191, m = 32, the float32 units 20 %; forward 258 -> 189 us,
// backward 313 -> 216, the reductions below included).  Forward, eight adjacent lanes
// are the slices s of a row quad q: thread (q, s) takes the columns 32 l + 4 s + e
// (l, e < 4) of its rows, v[j * 16 + 4 l + e]; sb_pos is where row k of the staged
// right-hand sides goes so that the product finds it at s + 8 (4 l + e).  Backward, a
// warp is a slice s and its lanes the 32 column quads q: a load is one row of the tile.
template <bool FWD>
__device__ __forceinline__ int sb_pos(int k) {
    return FWD ? (k & ~31) | ((k & 3) << 3) | ((k >> 2) & 7) : k;
}
template <bool FWD>
__device__ __forceinline__ void sb_tile(float (&v)[64], const float* W, long ldw, int n, int J, int K, int q, int s) {
    if constexpr (FWD) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const long gr = (long)J * 128 + 4 * q + j;
            const float4* src = reinterpret_cast<const float4*>(W + gr * ldw + (long)K * 128) + s;
#pragma unroll
            for (int l = 0; l < 4; ++l) {
                const float4 t = gr < n ? __ldg(src + 8 * l) : make_float4(0.f, 0.f, 0.f, 0.f);
                v[j * 16 + 4 * l] = t.x;
                v[j * 16 + 4 * l + 1] = t.y;
                v[j * 16 + 4 * l + 2] = t.z;
                v[j * 16 + 4 * l + 3] = t.w;
            }
        }
    } else {
        tv_tile<false>(v, W, ldw, n, J, K, q, s);
    }
}

// Yk[sb_pos(l)][c] = Y[r0 + l, c0 + c] (zero past n or past mc), minus the block
// row's pending partial sum when ns > 0
template <int MC, bool FWD>
__device__ __forceinline__ void sb_stage(float* Yk, const SbArgs& a, long r0, int ns = 0, int slot_lo = 0,
                                         int glo = 0) {
    constexpr int PER = (128 * MC + 255) / 256;
    float v[PER];
#pragma unroll
    for (int u = 0; u < PER; ++u) {
        const int e = threadIdx.x + u * 256, l = e & 127, c = e >> 7;
        const long r = r0 + l;
        v[u] = (e < 128 * MC && c < a.mc && r < a.n) ? __ldcg(a.Y + (long)(a.c0 + c) * a.n + r) : 0.f;
    }
    if (ns > 0) {
        float pend[PER];
        sb_pending<MC>(a, ns, slot_lo, glo, pend);
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            const int e = threadIdx.x + u * 256, l = e & 127, c = e >> 7;
            if (e < 128 * MC && c < a.mc && r0 + l < a.n) v[u] -= pend[u];
        }
    }
#pragma unroll
    for (int u = 0; u < PER; ++u) {
        const int e = threadIdx.x + u * 256, l = e & 127, c = e >> 7;
        if (e < 128 * MC) Yk[sb_pos<FWD>(l) * tv_ys<MC>() + c] = v[u];
    }
}

// Blocks [cs0, cs1) of y_I (from the output vector O) into YI (block c at
// YI + c 128 tv_ys), loads issued eight per thread at a time
template <int MC, bool FWD>
__device__ __forceinline__ void sb_stage_range(float* YI, const SbArgs& a, int jb0, int cs0, int cs1) {
    constexpr int BATCH = 8;
    const int total = (cs1 - cs0) * 128 * MC;
    for (int base = threadIdx.x; base < total; base += 256 * BATCH) {
        float v[BATCH];
#pragma unroll
        for (int k = 0; k < BATCH; ++k) {
            const int e = base + k * 256;
            v[k] = 0.f;
            if (e < total) {
                const int blk = cs0 + e / (128 * MC), rem = e - (blk - cs0) * 128 * MC;
                const int l = rem & 127, c = rem >> 7;
                const long row = (long)(jb0 + blk) * 128 + l;
                if (c < a.mc && row < a.n) v[k] = __ldcg(a.O + (long)(a.oc0 + c) * a.n + row);
            }
        }
#pragma unroll
        for (int k = 0; k < BATCH; ++k) {
            const int e = base + k * 256;
            if (e < total) {
                const int blk = cs0 + e / (128 * MC), rem = e - (blk - cs0) * 128 * MC;
                YI[(blk * 128 + sb_pos<FWD>(rem & 127)) * tv_ys<MC>() + (rem >> 7)] = v[k];
            }
        }
    }
}

// Prefetch into L2 the 128 x 128 tile at rows r0.., columns k0.. of a
// row-major float matrix (ld floats, rows < nrows): 512 lines of 128 bytes,
// two per thread.  Nothing waits for it; the later loads find the lines in L2.
__device__ __forceinline__ void sb_prefetch_tile(const float* M, long ld, long nrows, long r0, long k0) {
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int line = threadIdx.x + k * 256, r = line >> 2, part = line & 3;
        if (r0 + r < nrows) {
            const float* ptr = M + (r0 + r) * ld + k0 + part * 32;
            asm volatile("prefetch.global.L2 [%0];" ::"l"(ptr));
        }
    }
}

// The tile of unit u of panel pn (forward L_{J, jb0 + c}, backward
// L_{jb0 + c, J}), prefetched
template <bool FWD>
__device__ __forceinline__ void sb_prefetch_unit(const SbArgs& a, const SbPanel& pn, int jb0, long u) {
    const int J = pn.J0 + (int)(u / pn.nb), K = jb0 + (int)(u % pn.nb);
    if (FWD) sb_prefetch_tile(a.W, a.ldw, a.n, (long)J * 128, (long)K * 128);
    else sb_prefetch_tile(a.W, a.ldw, a.n, (long)K * 128, (long)J * 128);
}

// Backward: the slices are the eight warps; each writes its sums to red (in the order
// in which lanes hold them) and every thread adds the slices of its share, four columns
// (MC < 4: one) of row 4 q + j at a time, in slice order, and passes it to put(row of
// the tile, first column, sums).
template <int MC, typename Put>
__device__ __forceinline__ void sb_reduce_warps(const float (&acc)[4][MC], float* red, Put put) {
    constexpr int V = MC >= 4 ? 4 : 1, CV = MC / V;
    const int q = threadIdx.x & 31, s = threadIdx.x >> 5;
    __syncthreads();  // the last sums have been read
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int c = 0; c < CV; ++c) {
            float* d = red + (((s * 4 + j) * CV + c) * 32 + q) * V;
            if constexpr (V == 4)
                *reinterpret_cast<float4*>(d) = make_float4(acc[j][4 * c], acc[j][4 * c + 1], acc[j][4 * c + 2], acc[j][4 * c + 3]);
            else
                *d = acc[j][c];
        }
    __syncthreads();
#pragma unroll
    for (int e0 = 0; e0 < 128 * CV; e0 += 256) {
        const int e = e0 + threadIdx.x;
        if (128 * CV < 256 && e >= 128 * CV) break;
        const int r = e >> 5, j = r / CV, c = r % CV;
        float t[V];
#pragma unroll
        for (int i = 0; i < V; ++i) t[i] = 0.f;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const float* d = red + (k * 128 * CV + e) * V;
            if constexpr (V == 4) {
                const float4 x = *reinterpret_cast<const float4*>(d);
                t[0] += x.x;
                t[1] += x.y;
                t[2] += x.z;
                t[3] += x.w;
            } else {
                t[0] += *d;
            }
        }
        put(4 * (e & 31) + j, c * V, t);
    }
}

// Forward: sum over the eight reduction slices (adjacent lanes); each exchange halves the
// values a lane still holds (7 MC / 2 shuffles instead of 12 MC), so that lane s ends
// with row j = s / 2 of the quad, columns (s % 2) MC / 2 .. in acc[0][0 ..] (MC = 1: the
// column, in both lanes of the pair), and the results are written by all lanes.
template <int MC>
__device__ __forceinline__ void sb_reduce(float (&acc)[4][MC], float (&out)[MC > 1 ? MC / 2 : 1], int s) {
    float v[4 * MC];
#pragma unroll
    for (int i = 0; i < 4 * MC; ++i) v[i] = acc[i / MC][i % MC];
#pragma unroll
    for (int b = 4, h = 2 * MC; b >= 1; b >>= 1, h >>= 1) {
        if (h >= 1) {
            const bool hi = s & b;
#pragma unroll
            for (int i = 0; i < h; ++i) {
                const float send = hi ? v[i] : v[i + h];
                const float keep = hi ? v[i + h] : v[i];
                v[i] = keep + __shfl_xor_sync(0xffffffffu, send, b);
            }
        } else {
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], b);
        }
    }
#pragma unroll
    for (int i = 0; i < (MC > 1 ? MC / 2 : 1); ++i) out[i] = v[i];
}

// out of sb_reduce to a 128 x MC partial tile
template <int MC>
__device__ __forceinline__ void sb_put(float* pt, const float (&out)[MC > 1 ? MC / 2 : 1], int q, int s) {
    float* d = pt + (4 * q + (s >> 1)) * MC + (MC > 1 ? (s & 1) * (MC / 2) : 0);
    if constexpr (MC >= 8) {
#pragma unroll
        for (int i = 0; i < MC / 2; i += 4)
            *reinterpret_cast<float4*>(d + i) = make_float4(out[i], out[i + 1], out[i + 2], out[i + 3]);
    } else {
#pragma unroll
        for (int i = 0; i < (MC > 1 ? MC / 2 : 1); ++i) d[i] = out[i];
    }
}

// the slices' sum of acc to a 128 x MC partial tile
template <int MC, bool FWD>
__device__ __forceinline__ void sb_store(float* pt, float (&acc)[4][MC], float* red, int q, int s) {
    if constexpr (FWD) {
        float sum[MC > 1 ? MC / 2 : 1];
        sb_reduce<MC>(acc, sum, s);
        sb_put<MC>(pt, sum, q, s);
    } else {
        sb_reduce_warps<MC>(acc, red, [&](int r, int c, auto& t) {
            if constexpr (MC >= 4)
                *reinterpret_cast<float4*>(pt + r * MC + c) = make_float4(t[0], t[1], t[2], t[3]);
            else
                pt[r * MC + c] = t[0];
        });
    }
}

// shared memory: y_I of one super-block (SPD_SB_BLOCKS staged 128 x MC blocks; one
// where there is no panel to update) and the eight warps' sums of the backward sweep
__host__ __device__ constexpr int sb_staged(int NS) { return NS == 1 ? 1 : SPD_SB_BLOCKS; }
template <int MC>
constexpr size_t trsv_sb_smem(int NS) {
    return (size_t)(sb_staged(NS) * 128 * tv_ys<MC>() + 8 * 128 * MC) * sizeof(float);
}

// tile index of the pair (p, q), q <= p, in the order (0,0), (1,0), (1,1), ...
__device__ __forceinline__ int sb_tri(int p, int q) { return p * (p + 1) / 2 + q; }

// Columns go in groups of MC, up to SB_GROUPS of them side by side in one launch,
// each on its share of the CTAs with barriers of its own: a sweep is mostly its
// chain of grid-wide phases, which the groups then run at the same time, and they
// read the same tiles of L within a short time of each other.
constexpr int SB_GROUPS = 4;
template <int MC, bool FWD>
__global__ void __launch_bounds__(256, 1) k_trsv_sb(SbArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float* YI = reinterpret_cast<float*>(smem_raw);  // [SBB][128][tv_ys] staged blocks of y_I (F: one)
    constexpr int YB = 128 * tv_ys<MC>();           // floats per staged block
    float* red = YI + sb_staged(a.NS) * YB;         // backward: the warps' sums
    __shared__ int s_abort, s_last;
    if (a.gate && *a.gate == 0) return;  // refinement over (capturable solves)
    const int tid = threadIdx.x;
    const int tq = FWD ? tid >> 3 : tid & 31, ts = FWD ? tid & 7 : tid >> 5;  // row quad, reduction slice
    const int G = gridDim.x, g = blockIdx.x;
    if (gridDim.y > 1) {
        const int y = blockIdx.y;
        a.c0 += y * MC;
        a.oc0 += y * MC;
        a.mc = min(MC, a.mtot - y * MC);
        a.P += y * a.pstride;
        a.P2 += y * a.p2stride;
        a.bar += y * a.barstride;
    }
    if (tid == 0) s_abort = 0;
    __syncthreads();
    int nbar = 0;
    float ra[64], rb[64];
    SbPanel prev{0, 1, 1, 0};  // the previous step's panel update (W = 0: none)
    // each phase's first tile is loaded before the barrier in front of it: tiles of L
    // and of the inverses do not change
    auto first_inverse_tile = [&](int I) {
        const int nb = min(a.SBB, a.NB - I * a.SBB);
        if (g >= nb * (nb + 1) / 2) return;
        int p = 0;
        while (sb_tri(p + 1, 0) <= g) ++p;
        const int q = g - sb_tri(p, 0);
        sb_tile<FWD>(ra, a.X + (long)I * a.S * a.S, a.S, a.S, FWD ? p : q, FWD ? q : p, tq, ts);
    };
    first_inverse_tile(FWD ? 0 : a.NS - 1);
    for (int t = 0; t < a.NS; ++t) {
        const int I = FWD ? t : a.NS - 1 - t;
        const int jb0 = I * a.SBB;                    // first 128-block of the super-block
        const int nb = min(a.SBB, a.NB - jb0);        // its 128-blocks
        const float* XI = a.X + (long)I * a.S * a.S;  // its inverse, S x S row-major
        // F: partial tiles, and the previous panel's split rows outside this
        // super-block (forward: below it; backward: above it)
        const int ntile = nb * (nb + 1) / 2;
        const int nfix = prev.W == 0 ? 0 : (FWD ? a.NB - (jb0 + nb) : jb0);
        for (int task = g; task < ntile + nfix; task += G) {
            if (task >= ntile) {
                const int J = FWD ? jb0 + nb + (task - ntile) : task - ntile;
                int slot_lo, glo;
                const int ns = sb_row_slots(prev, J, slot_lo, glo);
                if (ns == 0) continue;  // block-uniform
                constexpr int PER = (128 * MC + 255) / 256;
                float pend[PER];
                sb_pending<MC>(a, ns, slot_lo, glo, pend);
#pragma unroll
                for (int u = 0; u < PER; ++u) {
                    const int e = tid + u * 256, l = e & 127, cc = e >> 7;
                    const long row = (long)J * 128 + l;
                    if (e < 128 * MC && cc < a.mc && row < a.n) {
                        float* y = a.Y + (long)(a.c0 + cc) * a.n + row;
                        *y = __ldcg(y) - pend[u];
                    }
                }
                continue;
            }
            int p = 0;
            while (sb_tri(p + 1, 0) <= task) ++p;
            const int q = task - sb_tri(p, 0);  // q <= p
            // forward: X[b][c] with b = p, c = q; backward: X[c][b]^T with b = q, c = p
            const int b = FWD ? p : q, c = FWD ? q : p;
            if (task != g) sb_tile<FWD>(ra, XI, a.S, a.S, b, c, tq, ts);
            int slot_lo = 0, glo = 0;
            const int ns = prev.W == 0 ? 0 : sb_row_slots(prev, jb0 + c, slot_lo, glo);
            sb_stage<MC, FWD>(YI, a, (long)(jb0 + c) * 128, ns, slot_lo, glo);
            __syncthreads();
            float acc[4][MC];
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int cc = 0; cc < MC; ++cc) acc[j][cc] = 0.f;
            tv_dot<MC>(acc, ra, YI, ts);
            sb_store<MC, FWD>(a.P + (long)task * 128 * MC, acc, red, tq, ts);
            __syncthreads();
            // the last tile of block row b to arrive adds the row's partials
            // in c order (forward c = 0..b, backward c = b..nb-1) into y_I[b]
            // in O, all of a thread's loads in flight together
            if (tid == 0) {
                __threadfence();
                const int cnt = FWD ? b + 1 : nb - b;
                s_last = atomicAdd(a.bar + 2 + t * a.SBB + b, 1) == cnt - 1;
                __threadfence();
            }
            __syncthreads();
            if (s_last) {
                constexpr int EPT = (128 * MC + 255) / 256;
                float v[SPD_SB_BLOCKS][EPT];
#pragma unroll
                for (int k = 0; k < SPD_SB_BLOCKS; ++k)
#pragma unroll
                    for (int i = 0; i < EPT; ++i) {
                        const int e = tid + 256 * i, c2 = FWD ? k : b + k;
                        const bool in = (FWD ? k <= b : c2 < nb) && e < 128 * MC;
                        v[k][i] = in ? __ldcg(a.P + (long)(FWD ? sb_tri(b, c2) : sb_tri(c2, b)) * 128 * MC + e) : 0.f;
                    }
#pragma unroll
                for (int i = 0; i < EPT; ++i) {
                    const int e = tid + 256 * i, r = e / MC, cc = e - r * MC;
                    float s = 0.f;
#pragma unroll
                    for (int k = 0; k < SPD_SB_BLOCKS; ++k)
                        if (FWD ? k <= b : b + k < nb) s += v[k][i];
                    const long row = (long)(jb0 + b) * 128 + r;
                    if (e < 128 * MC && cc < a.mc && row < a.n) a.O[(long)(a.oc0 + cc) * a.n + row] = s;
                }
            }
        }
        if (t + 1 == a.NS) break;  // no rows left to update
        // B: units (J, c) of every remaining 128-row block J (forward: below
        // the super-block, backward: above it), in equal ranges over the CTAs
        SbPanel pn;
        pn.J0 = FWD ? jb0 + nb : 0;
        pn.nb = nb;
        pn.W = (long)((FWD ? a.NB : jb0) - pn.J0) * nb;
        pn.geff = (int)min((long)G, pn.W);
        const long u0 = sb_ub(g, pn.W, pn.geff), u1 = g < pn.geff ? sb_ub(g + 1, pn.W, pn.geff) : u0;
        if (g < pn.geff) {
            sb_tile<FWD>(ra, a.W, a.ldw, a.n, pn.J0 + (int)(u0 / nb), jb0 + (int)(u0 % nb), tq, ts);
            if (u0 + 1 < u1) sb_prefetch_unit<FWD>(a, pn, jb0, u0 + 1);
        }
        if (!sb_barrier(a, ++nbar, &s_abort)) return;
        if (g < pn.geff) {
            // the blocks of y_I this CTA's units multiply, staged once
            const bool all = (u1 - u0 >= nb) || (u0 / nb != (u1 - 1) / nb);
            const int cs0 = all ? 0 : (int)(u0 % nb), cs1 = all ? nb : (int)((u1 - 1) % nb) + 1;
            sb_stage_range<MC, FWD>(YI, a, jb0, cs0, cs1);
            __syncthreads();
            for (long u = u0; u < u1;) {
                const int J = pn.J0 + (int)(u / nb), ca = (int)(u % nb);
                const int ce = (int)min((long)nb, ca + (u1 - u));
                float acc[4][MC];
#pragma unroll
                for (int j = 0; j < 4; ++j)
#pragma unroll
                    for (int cc = 0; cc < MC; ++cc) acc[j][cc] = 0.f;
                // tiles L_{J, jb0 + c} (forward) or L_{jb0 + c, J}^T (backward),
                // two per trip so that the register buffers alternate: the
                // next tile's loads are in flight during this tile's products
                // (tiles two units ahead, across pieces, are prefetched into L2)
                if (u != u0) sb_tile<FWD>(ra, a.W, a.ldw, a.n, J, jb0 + ca, tq, ts);
                for (int c = ca; c < ce; c += 2) {
                    const long uc = u + (c - ca);
                    if (uc + 2 < u1) sb_prefetch_unit<FWD>(a, pn, jb0, uc + 2);
                    if (c + 1 < ce) sb_tile<FWD>(rb, a.W, a.ldw, a.n, J, jb0 + c + 1, tq, ts);
                    tv_dot<MC>(acc, ra, YI + c * YB, ts);
                    if (c + 1 >= ce) break;
                    if (uc + 3 < u1) sb_prefetch_unit<FWD>(a, pn, jb0, uc + 3);
                    if (c + 2 < ce) sb_tile<FWD>(ra, a.W, a.ldw, a.n, J, jb0 + c + 2, tq, ts);
                    tv_dot<MC>(acc, rb, YI + (c + 1) * YB, ts);
                }
                if (ca == 0 && ce == nb) {  // the whole row: subtract in place
                    auto sub = [&](int r, int c, float t) {
                        const long row = (long)J * 128 + r;
                        if (row < a.n && c < a.mc) {
                            float* y = a.Y + (long)(a.c0 + c) * a.n + row;
                            *y = __ldcg(y) - t;
                        }
                    };
                    if constexpr (FWD) {
                        float sum[MC > 1 ? MC / 2 : 1];
                        sb_reduce<MC>(acc, sum, ts);
                        if (MC > 1 || !(ts & 1))
#pragma unroll
                            for (int i = 0; i < (MC > 1 ? MC / 2 : 1); ++i)
                                sub(4 * tq + (ts >> 1), (MC > 1 ? (ts & 1) * (MC / 2) : 0) + i, sum[i]);
                    } else {
                        sb_reduce_warps<MC>(acc, red, [&](int r, int c, auto& t) {
#pragma unroll
                            for (int i = 0; i < (MC >= 4 ? 4 : 1); ++i) sub(r, c + i, t[i]);
                        });
                    }
                } else {  // a piece of a shared row: partial slot
                    sb_store<MC, FWD>(a.P2 + (long)(2 * g + (u == u0 ? 0 : 1)) * 128 * MC, acc, red, tq, ts);
                }
                u += ce - ca;
            }
        }
        {   // the next super-block's other inverse tiles this CTA will multiply in phase F
            const int In = FWD ? I + 1 : I - 1;
            const int nbn = min(a.SBB, a.NB - In * a.SBB), ntn = nbn * (nbn + 1) / 2;
            for (int task = g + G; task < ntn; task += G) {
                int p = 0;
                while (sb_tri(p + 1, 0) <= task) ++p;
                const int q = task - sb_tri(p, 0);
                const int b = FWD ? p : q, c = FWD ? q : p;
                const float* XN = a.X + (long)In * a.S * a.S;
                if (FWD) sb_prefetch_tile(XN, a.S, a.S, (long)b * 128, (long)c * 128);
                else sb_prefetch_tile(XN, a.S, a.S, (long)c * 128, (long)b * 128);
            }
        }
        first_inverse_tile(FWD ? I + 1 : I - 1);
        prev = pn;
        if (!sb_barrier(a, ++nbar, &s_abort)) return;
    }
}

// ---------------------------------------------------------------------------
// the super-block inverses, once per factor
// ---------------------------------------------------------------------------
// X_I = L_II^{-1} by doubling: the 128-row diagonal blocks' inverses come from
// k_block_inverse; with the inverses A^{-1}, C^{-1} of two neighbouring diagonal
// blocks of order h in place, the block below the first is -C^{-1} (B A^{-1}), B
// its block of L, for h = 128, 256, 512: two products per level, T = B A^{-1}
// (kept in the unused block above the diagonal) and -C^{-1} T, over all pairs of
// all super-blocks at once.  Block forward substitution down each column strip
// was a chain of up to 35 products of 128 x 128 x 32 in one CTA: 282 us whatever
// the order (558 at n = 16384).
//
// One 64 x 64 tile of the product per CTA, 4 x 4 per thread, 16 of K at a time
// through shared memory with the next 16 in registers; a triangular operand's
// zero half is left out.  Rows of L past n are zero and rows of the inverse past
// n are the identity; those rows of X meet only right-hand-side rows past n,
// which the sweeps hold at zero.
constexpr int SBP_K = 16;
template <bool FIRST>
static __global__ void __launch_bounds__(256) k_sb_product(const float* __restrict__ W, long ldw, int n, int NB, int SBB,
                                                           float* __restrict__ X, int h) {
    __shared__ __align__(16) float As[SBP_K][68];  // [k][row]
    __shared__ __align__(16) float Bs[SBP_K][68];  // [k][column]
    const int S = SBB * 128, I = blockIdx.z, tid = threadIdx.x;
    const int th = h / 64, pair = blockIdx.y;
    const int ti = blockIdx.x / th, tj = blockIdx.x % th;  // tile of the h x h product
    const int r0 = pair * 2 * h;                           // the pair's first row in the super-block
    const int rows = min(SBB, NB - I * SBB) * 128;         // rows of this super-block
    if (r0 + h + ti * 64 >= rows) return;
    float* XI = X + (long)I * S * S;
    const float* Lb = W + ((long)I * S + r0 + h) * ldw + (long)I * S + r0;  // B: rows of the second half
    // FIRST: T[i][j] = sum_{k >= j} B[i][k] A^{-1}[k][j], to rows r0 .., columns r0 + h ..
    // else:  X[i][j] = -sum_{k <= i} C^{-1}[i][k] T[k][j], to rows r0 + h .., columns r0 ..
    const float* Am = XI + (long)(r0 + h) * S + r0 + h;                       // C^{-1}
    const float* Bm = FIRST ? XI + (long)r0 * S + r0 : XI + (long)r0 * S + r0 + h;  // A^{-1} or T
    const int klo = FIRST ? tj * 64 : 0, khi = FIRST ? h : (ti + 1) * 64;
    const int ar = tid >> 2, ak = (tid & 3) * 4;    // A: row ar, k ak .. ak + 3
    const int bk = tid >> 4, bc = (tid & 15) * 4;   // B: row bk, columns bc .. bc + 3
    const long arow = ti * 64 + ar;
    const bool aok = !FIRST || (long)I * S + r0 + h + arow < n;
    float4 av, bv;
    auto load = [&](int k) {
        const float* pa = FIRST ? Lb + arow * ldw + k + ak : Am + arow * S + k + ak;
        av = aok ? *reinterpret_cast<const float4*>(pa) : make_float4(0.f, 0.f, 0.f, 0.f);
        bv = *reinterpret_cast<const float4*>(Bm + (long)(k + bk) * S + tj * 64 + bc);
    };
    float acc[4][4] = {};
    const int tr = (tid >> 4) * 4, tc = (tid & 15) * 4;
    load(klo);
    for (int k = klo; k < khi; k += SBP_K) {
        As[ak][ar] = av.x;
        As[ak + 1][ar] = av.y;
        As[ak + 2][ar] = av.z;
        As[ak + 3][ar] = av.w;
        *reinterpret_cast<float4*>(&Bs[bk][bc]) = bv;
        __syncthreads();
        if (k + SBP_K < khi) load(k + SBP_K);
#pragma unroll
        for (int q = 0; q < SBP_K; ++q) {
            const float4 x = *reinterpret_cast<const float4*>(&As[q][tr]), y = *reinterpret_cast<const float4*>(&Bs[q][tc]);
            const float xr[4] = {x.x, x.y, x.z, x.w}, yc[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(xr[i], yc[j], acc[i][j]);
        }
        __syncthreads();
    }
    float* out = FIRST ? XI + (long)(r0 + ti * 64 + tr) * S + r0 + h + tj * 64 + tc
                       : XI + (long)(r0 + h + ti * 64 + tr) * S + r0 + tj * 64 + tc;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float4 v = FIRST ? make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3])
                               : make_float4(-acc[i][0], -acc[i][1], -acc[i][2], -acc[i][3]);
        *reinterpret_cast<float4*>(out + (long)i * S) = v;
    }
}

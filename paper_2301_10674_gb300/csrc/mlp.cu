// Learned interface normal: training data, training and inference of the
// 27-64-64-4 perceptron (layout and fragment conventions in mlp_dev.cuh).
//
// Training data: analytic surfaces (planes, liquid and gas spheres, sine
// waves) through a point P near the centre of a 3x3x3 block; the fill level
// of each cell is its liquid volume fraction, the labels are the unit normal
// toward the gas and the mean curvature at P. Training: Adam on the loss
// 1 - cos(n, n_true) + lam (k - k_true)^2 + mu (|n| - 1)^2, averaged over a
// batch drawn by SplitMix64 from a seed, each stencil mapped by one of the 48
// cube symmetries. Every product runs on the tensor cores with BF16 operands
// and FP32 accumulation; master weights and Adam moments are FP32.
#include <cmath>
#include <cstdint>
#include <cstring>
#include <vector>

#include "fslbm.h"
#include "fslbm_dev.cuh"
#include "mlp_dev.cuh"

namespace fsl {

// ------------------------------------------------------------ surfaces
constexpr int GEN_THREADS = 256;
constexpr int SUBS = 64;                 // sub-samples per cell edge
constexpr int ROWS = SUBS * SUBS;        // sample rows along x per cell

// Volume of {xi in [0,1]^3 : m.xi <= alpha}, m >= 0, as the divided
// difference of G3(b) = max(b, 0)^3 / 6 over the three steps m_i. A step
// below 1e-3 is replaced by the derivative at the midpoint (G_k' = G_{k-1}),
// whose error is below m_i^2 / 24 times a bounded third derivative.
__device__ double box_volume_below(const double (&m)[3], double alpha) {
    double e[3];
    int ne = 0;
    double b0 = alpha;
    for (int i = 0; i < 3; ++i) {
        if (m[i] >= 1e-3) e[ne++] = m[i];
        else b0 -= 0.5 * m[i];
    }
    double sum = 0.0;
    for (int v = 0; v < (1 << ne); ++v) {
        double b = b0;
        int sgn = 1;
        for (int i = 0; i < ne; ++i)
            if (v >> i & 1) { b -= e[i]; sgn = -sgn; }
        double gk;
        if (b <= 0.0) gk = 0.0;
        else if (ne == 0) gk = 1.0;
        else if (ne == 1) gk = b;
        else if (ne == 2) gk = 0.5 * b * b;
        else gk = b * b * b / 6.0;
        sum += sgn * gk;
    }
    double den = 1.0;
    for (int i = 0; i < ne; ++i) den *= e[i];
    const double V = sum / den;
    return V < 0.0 ? 0.0 : (V > 1.0 ? 1.0 : V);
}

// liquid fraction of cell q below the plane (x - P).n <= 0: with
// x = c - 1/2 + xi and the negative components reflected (xi_i -> 1 - xi_i)
__device__ double plane_cell(const double (&n)[3], const double (&P)[3], int q) {
    const double c[3] = {(double)cx(q), (double)cy(q), (double)cz(q)};
    double beta = 0.0, shift = 0.0;
    double m[3];
    for (int i = 0; i < 3; ++i) {
        beta += n[i] * (P[i] - (c[i] - 0.5));
        if (n[i] < 0.0) shift += n[i];
        m[i] = fabs(n[i]);
    }
    return box_volume_below(m, beta - shift);
}

// sum over the block, the same order on every call
__device__ float block_sum(float v, float* sh) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __syncthreads();
    if (lane == 0) sh[w] = v;
    __syncthreads();
    float s = 0.f;
    for (int i = 0; i < GEN_THREADS / 32; ++i) s += sh[i];
    return s;
}

// One block per surface. params: n x 12 FP64 rows (kind, n0, s, r, A, k,
// phase, e1; P = s n0); fill: n x 27 FP32; target: n x 4 FP32.
// Bound by instruction issue over the sub-samples (27 x 64^3 per sine wave).
// A cell, a row of 64 samples or a run of 16 that lies wholly on one side of
// the surface is counted without its samples, where the value in its middle
// (a run: at its first sample) exceeds what the surface function can change by
// within it plus the rounding of the evaluation: the counts are those of all
// samples. The FP64 cell offsets are formed once per cell, not per thread.
// 20 000 surfaces of all kinds: 12.6 ms with every sample evaluated,
// 2.76 ms now.
__global__ void __launch_bounds__(GEN_THREADS) k_make_stencils(const double* __restrict__ params, long long n,
                                                               float* fill, float* target) {
    __shared__ float sh[GEN_THREADS / 32];
    __shared__ float rot[2];         // phase per sample, A sin(phase)
    __shared__ float off[27][3];     // cell offsets from the sphere's centre, or (u, w) of the cell's corner
    const long long i = blockIdx.x;
    if (i >= n) return;
    const double* p = params + i * 12;
    const int kind = (int)p[0];
    const double n0[3] = {p[1], p[2], p[3]};
    const double s = p[4], r = p[5], A = p[6], kw = p[7], ph = p[8];
    const double e1[3] = {p[9], p[10], p[11]};
    const double P[3] = {s * n0[0], s * n0[1], s * n0[2]};
    const int tid = threadIdx.x;
    // labels, by a warp of their own: FP64 trigonometry and divisions
    if (tid == 64) {
        double nt[3] = {n0[0], n0[1], n0[2]}, kap = 0.0;
        if (kind == 1) kap = 1.0 / r;
        else if (kind == 2) kap = -1.0 / r;
        else if (kind == 3) {
            // graph w = f(u): normal (n0 - f' e1) / sqrt(1 + f'^2), mean
            // curvature of the cylinder -f'' / (2 (1 + f'^2)^(3/2))
            const double fp = A * kw * cos(ph), fpp = -A * kw * kw * sin(ph);
            const double qn = sqrt(1.0 + fp * fp);
            for (int k = 0; k < 3; ++k) nt[k] = (n0[k] - fp * e1[k]) / qn;
            kap = -fpp / (2.0 * qn * qn * qn);
        }
        for (int k = 0; k < 3; ++k) target[i * 4 + k] = (float)nt[k];
        target[i * 4 + 3] = (float)kap;
    }
    if (kind == 0) {
        if (tid < 27) fill[i * 27 + tid] = (float)plane_cell(n0, P, tid);
    } else if (kind == 1 || kind == 2) {
        // exact chord along x of each of the 64 x 64 rows
        const double sg = kind == 1 ? -1.0 : 1.0;       // centre P -/+ r n0
        if (tid < 27)
            for (int a = 0; a < 3; ++a)
                off[tid][a] = (float)(P[a] + sg * r * n0[a] - (a == 0 ? cx(tid) : (a == 1 ? cy(tid) : cz(tid))));
        __syncthreads();
        const float rf = (float)r, rr = (float)(r * r);
        for (int q = 0; q < 27; ++q) {
            const float ox = off[q][0], oy = off[q][1], oz = off[q][2];
            // whole cell inside or outside (half a diagonal is 0.8661)
            const float d = sqrtf(ox * ox + oy * oy + oz * oz) - rf;
            if (fabsf(d) > 0.8661f + 1e-4f * (1.f + rf)) {
                if (tid == 0) fill[i * 27 + q] = (d < 0.f) == (kind == 1) ? 1.f : 0.f;
                continue;
            }
            float acc = 0.f;
            for (int j = tid; j < ROWS; j += GEN_THREADS) {
                const float y = ((j % SUBS) + 0.5f) / SUBS - 0.5f, z = ((j / SUBS) + 0.5f) / SUBS - 0.5f;
                const float dy = y - oy, dz = z - oz;
                const float h2 = rr - dy * dy - dz * dz;
                if (h2 > 0.f) {
                    const float h = sqrtf(h2);
                    acc += fmaxf(fminf(ox + h, 0.5f) - fmaxf(ox - h, -0.5f), 0.f);
                }
            }
            const float tot = block_sum(acc, sh) / ROWS;
            if (tid == 0) fill[i * 27 + q] = kind == 1 ? tot : 1.f - tot;
        }
    } else {
        // w <= A (sin(k u + phase) - sin(phase)) at 64^3 midpoints, u = d.e1,
        // w = d.n0, d = x - P. Per cell the corner offset is formed in FP64,
        // the sub-cell offsets in FP32; along a row the phase advances by
        // k e1.x / 64 per sample (a rotation), restarted from sincosf every
        // 16 samples.
        if (tid < 27) {
            const double b[3] = {cx(tid) - 0.5 - P[0], cy(tid) - 0.5 - P[1], cz(tid) - 0.5 - P[2]};
            off[tid][0] = (float)(b[0] * e1[0] + b[1] * e1[1] + b[2] * e1[2]);
            off[tid][1] = (float)(b[0] * n0[0] + b[1] * n0[1] + b[2] * n0[2]);
        } else if (tid == 32) {
            rot[0] = (float)(kw * e1[0] / SUBS);
            rot[1] = (float)(A * sin(ph));
        }
        __syncthreads();
        float sd, cd;
        sincosf(rot[0], &sd, &cd);
        const float Af = (float)A, As = rot[1], kf = (float)kw, pf = (float)ph;
        const float fe[3] = {(float)e1[0], (float)e1[1], (float)e1[2]};
        const float fn[3] = {(float)n0[0], (float)n0[1], (float)n0[2]};
        // change of g = w - A sin(k u + phase) + A sin(phase) within a cell,
        // row or run, at most: the gradient at the point tested times the
        // extent plus half the largest second derivative A k^2 along u, and
        // the rounding of an evaluation, with that of two arguments of the
        // sine, each up to 6e-8 of the phase
        const float Ak = Af * kf, h2 = 0.5f * fabsf(Ak * kf);
        const float tol = 1e-4f * (1.f + fabsf(Af)) + 1.5e-7f * fabsf(Af * pf);
        const float ec = 0.5f * (fabsf(fe[0]) + fabsf(fe[1]) + fabsf(fe[2])), er = 0.5f * fe[0], es = 0.25f * fe[0];
        const float cell_add = tol + h2 * ec * ec, row_add = tol + h2 * er * er, run_add = tol + h2 * es * es;
        for (int q = 0; q < 27; ++q) {
            const float bu = off[q][0], bw = off[q][1];
            float sc, cc;
            sincosf(kf * (bu + 0.5f * (fe[0] + fe[1] + fe[2])) + pf, &sc, &cc);
            const float gc = bw + 0.5f * (fn[0] + fn[1] + fn[2]) - Af * sc + As, dc = Ak * cc;
            if (fabsf(gc) > 0.5f * (fabsf(fn[0] - dc * fe[0]) + fabsf(fn[1] - dc * fe[1]) + fabsf(fn[2] - dc * fe[2])) +
                                cell_add) {
                if (tid == 0) fill[i * 27 + q] = gc < 0.f ? 1.f : 0.f;
                continue;
            }
            int cnt = 0;
            for (int j = tid; j < ROWS; j += GEN_THREADS) {
                const float yo = ((j % SUBS) + 0.5f) / SUBS, zo = ((j / SUBS) + 0.5f) / SUBS;
                const float x0 = 0.5f / SUBS;
                const float u0 = bu + (x0 * fe[0] + yo * fe[1] + zo * fe[2]);
                const float w0 = bw + (x0 * fn[0] + yo * fn[1] + zo * fn[2]);
                float sm, cm;
                sincosf(kf * (u0 + (0.5f - x0) * fe[0]) + pf, &sm, &cm);
                const float gm = w0 + (0.5f - x0) * fn[0] - Af * sm + As;
                if (fabsf(gm) > 0.5f * fabsf(fn[0] - Ak * cm * fe[0]) + row_add) {
                    cnt += gm < 0.f ? SUBS : 0;
                    continue;
                }
                // runs of 16: decided from the expansion about the row's
                // middle where that suffices; the lanes then walk their
                // remaining runs together
                const float dm = fn[0] - Ak * cm * fe[0];
                const float lim = 0.125f * fabsf(dm) + row_add;
                unsigned todo = 0;
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    const float gr = gm + dm * (0.25f * g - 0.375f);
                    if (fabsf(gr) > lim) cnt += gr < 0.f ? 16 : 0;
                    else todo |= 1u << g;
                }
                for (; todo; todo &= todo - 1u) {
                    const int seg = 16 * (__ffs(todo) - 1);
                    float sn, cs;
                    sincosf(kf * (u0 + seg * (fe[0] / SUBS)) + pf, &sn, &cs);
                    float w = w0 + seg * (fn[0] / SUBS);
                    const float g0 = w - Af * sn + As;
                    if (fabsf(g0) > 0.25f * fabsf(fn[0] - Ak * cs * fe[0]) + run_add) {
                        cnt += g0 < 0.f ? 16 : 0;
                        continue;
                    }
#pragma unroll
                    for (int k = 0; k < 16; ++k) {
                        cnt += w <= Af * sn - As ? 1 : 0;
                        const float sn2 = sn * cd + cs * sd;
                        cs = cs * cd - sn * sd;
                        sn = sn2;
                        w += fn[0] / SUBS;
                    }
                }
            }
            const float tot = block_sum((float)cnt, sh);      // integer counts: exact in FP32
            if (tid == 0) fill[i * 27 + q] = tot / (float)(ROWS * SUBS);
        }
    }
}

// ------------------------------------------------------------ sampling
// output `counter` (from 0) of SplitMix64 seeded with `seed`
__device__ __forceinline__ uint64_t splitmix64(uint64_t seed, uint64_t counter) {
    uint64_t z = seed + (counter + 1ull) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// cube symmetry k: (T v)_i = s_i v_perm(i), perm the (k / 8)-th permutation
// of (0, 1, 2) in lexicographic order, s_i = -1 where bit i of k % 8 is set
__device__ __forceinline__ int sym_perm(int k, int i) {
    // two bits per axis, six per permutation, the first lowest
    constexpr uint64_t P = 0b000110'010010'001001'100001'011000'100100ull;
    return (int)(P >> (6 * (k >> 3) + 2 * i)) & 3;
}
__device__ __forceinline__ int sym_sign(int k, int i) { return ((k & 7) >> i & 1) ? -1 : 1; }

// The cell whose fill lands in cell c' = (x, y, z) under symmetry k is
// c = T^-1 c', i.e. c[perm(i)] = s_i c'[i]: index 13 + m0 x + m1 y + m2 z with
// m_i = s_i 3^perm(i)
__device__ __forceinline__ int sym_stride(int k, int i) {
    const int p = sym_perm(k, i);
    return sym_sign(k, i) * (p == 0 ? 1 : (p == 1 ? 3 : 9));
}

// ------------------------------------------------------------ training
// A batch is summed in chunks of 128 samples, each of 8 tiles of 16: the order
// of every sum (samples of a chunk in one tensor-core chain, tiles of a chunk
// and chunks one after the other) is fixed, and two runs give the same bits.
constexpr int CHUNK_TILES = 8, CHUNK = 16 * CHUNK_TILES;
constexpr int NBIAS = 2 * MLP_H + MLP_OUT + 1;   // bias gradients and the loss
constexpr int SLICE_CHUNKS = 128;                // chunks whose operands are held at once

// parameters as the operands of a training step
struct __align__(16) TrainWeights {
    MlpFwd f;
    uint2 w2t[8][4][32];     // W2 transposed
    uint32_t w3t[8][32];     // W3 transposed; outputs 8..15 are zero
};

// The operands of the weight gradients dW = dZ^T H of one tile of 16 samples,
// in fragment order with the samples along k, and its sums
constexpr int SAMPLE_THREADS = 128;

struct __align__(16) TrainOps {
    uint4 d1[4][32];         // dL/dz1
    uint4 d2[4][32];         // dL/dz2
    uint2 h1[8][32];         // relu(z1)
    uint2 h2[8][32];         // relu(z2)
    uint2 x[4][32];          // inputs
    uint2 dy[32];            // dL/dy (rows 8..15 are zero)
    float sums[NBIAS + 3];   // dz1, dz2, dy, loss
};

enum : int { TR_FIXED = 0, TR_DRAW_SYM = 1, TR_DRAW = 2 };

struct TrainArgs {
    const TrainWeights* W;
    const float* fill;
    const float* target;
    long long n;            // stencils in the set
    int B;                  // samples in the batch
    int first;              // first sample of the slice
    int tiles;              // tiles of the slice
    int mode;               // TR_FIXED: sample j is stencil j; TR_DRAW(_SYM): drawn (and mapped)
    uint64_t seed;
    long long step;
    float lam, mu;
    TrainOps* ops;          // [tiles]
};

__device__ __forceinline__ float sum_over_groups(float v) {
    v += __shfl_xor_sync(0xffffffffu, v, 4);
    v += __shfl_xor_sync(0xffffffffu, v, 8);
    v += __shfl_xor_sync(0xffffffffu, v, 16);
    return v;
}

// 8 x 8 matrix of 16-bit values across the warp (lane (g, t) holds row g,
// columns 2t and 2t + 1), transposed
__device__ __forceinline__ uint32_t transposed(uint32_t a) {
    uint32_t d;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(d) : "r"(a));
    return d;
}

// Forward and backward pass, a warp per 16 samples, and the operands of the
// weight gradients. Bound by latency: a warp runs about 2000 instructions one
// after the other, so there is a warp per scheduler and an SM for every four
// tiles. Weights come in fragment order, all of them at once, to shared memory
// (read from L2 where they are used: 0.9 us more); the transposes that the
// gradient products need are made in registers; drawing and gathering the
// samples, which need no weights, run before the previous launch is waited
// for. A step with a batch of 4096 takes 9.5 us; with one block of 8 warps per
// chunk, which also formed the chunk's weight gradients from transposes in
// shared memory, and a second launch for the sums and the update it took 31 us
// (24.4 + 5.6 and the gaps).
__global__ void __launch_bounds__(SAMPLE_THREADS) k_mlp_train_samples(TrainArgs a) {
    __shared__ TrainWeights W;
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int tile = blockIdx.x * (SAMPLE_THREADS / 32) + (threadIdx.x >> 5);
    const float invB = 1.f / (float)a.B;
    uint32_t xf[2][4];
    float tg[2][4];
    bool valid[2];
    {
        float xv[2][8];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const long long j = a.first + (long long)tile * 16 + g + 8 * r;
            valid[r] = tile < a.tiles && j < a.B;
            long long src = j;
            int sym = 0;
            if (a.mode != TR_FIXED) {
                const uint64_t v = splitmix64(a.seed, (uint64_t)a.step * (uint64_t)a.B + (uint64_t)j);
                src = (long long)(v % (uint64_t)a.n);
                sym = a.mode == TR_DRAW_SYM ? (int)((v >> 32) % 48ull) : 0;
            }
            const int m0 = sym_stride(sym, 0), m1 = sym_stride(sym, 1), m2 = sym_stride(sym, 2);
            const float* f = a.fill + src * 27 + 13;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int col = frag_col(q >> 2, q & 3, t);
                xv[r][q] = (valid[r] && col < 27)
                               ? f[m0 * (col % 3 - 1) + m1 * (col / 3 % 3 - 1) + m2 * (col / 9 - 1)]
                               : 0.f;
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) tg[r][i] = 0.f;
            if (valid[r]) {
                const float* tp = a.target + src * 4;
#pragma unroll
                for (int i = 0; i < 3; ++i) tg[r][i] = sym_sign(sym, i) * tp[sym_perm(sym, i)];
                tg[r][3] = tp[3];
            }
        }
#pragma unroll
        for (int kk = 0; kk < 2; ++kk) {
            xf[kk][0] = pack_bf16(xv[0][4 * kk + 0], xv[0][4 * kk + 1]);
            xf[kk][1] = pack_bf16(xv[1][4 * kk + 0], xv[1][4 * kk + 1]);
            xf[kk][2] = pack_bf16(xv[0][4 * kk + 2], xv[0][4 * kk + 3]);
            xf[kk][3] = pack_bf16(xv[1][4 * kk + 2], xv[1][4 * kk + 3]);
        }
    }
    wait_previous();
    allow_next();
    for (int q = threadIdx.x; q < (int)(sizeof(TrainWeights) / 16); q += SAMPLE_THREADS)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                         (uint32_t)__cvta_generic_to_shared(reinterpret_cast<uint4*>(&W) + q)),
                     "l"(reinterpret_cast<const uint4*>(a.W) + q)
                     : "memory");
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    if (tile >= a.tiles) return;
    TrainOps& O = a.ops[tile];
#pragma unroll
    for (int nt = 0; nt < 4; ++nt)
        O.x[nt][lane] = make_uint2(transposed(xf[nt >> 1][2 * (nt & 1)]), transposed(xf[nt >> 1][2 * (nt & 1) + 1]));

    MlpAct act;
    mlp_forward_ops(W.f.w1, W.f.w2, W.f.w3, W.f.b1, W.f.b2, W.f.b3, xf, act);
    float y[2][4];
    mlp_outputs(act, y[0], y[1]);

    // loss (already divided by the batch size) and dL/dy of both rows,
    // identical in the four lanes of a group
    float dy[2][4], L[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const float n2 = y[r][0] * y[r][0] + y[r][1] * y[r][1] + y[r][2] * y[r][2];
        const float nrm = sqrtf(fmaxf(n2, 1e-30f));
        const float dot = y[r][0] * tg[r][0] + y[r][1] * tg[r][1] + y[r][2] * tg[r][2];
        const float dk = y[r][3] - tg[r][3];
        const float pen = 2.f * a.mu * (nrm - 1.f) / nrm;
#pragma unroll
        for (int i = 0; i < 3; ++i)
            dy[r][i] = valid[r] ? (-(tg[r][i] / nrm - dot / (nrm * nrm * nrm) * y[r][i]) + pen * y[r][i]) * invB : 0.f;
        dy[r][3] = valid[r] ? 2.f * a.lam * dk * invB : 0.f;
        L[r] = valid[r] ? (1.f - dot / nrm + a.lam * dk * dk + a.mu * (nrm - 1.f) * (nrm - 1.f)) * invB : 0.f;
    }

    // dZ2 = (dY W3) masked by z2 > 0, dY as A operand (k = output)
    const uint32_t ay0 = t == 0 ? pack_bf16(dy[0][0], dy[0][1]) : (t == 1 ? pack_bf16(dy[0][2], dy[0][3]) : 0u);
    const uint32_t ay1 = t == 0 ? pack_bf16(dy[1][0], dy[1][1]) : (t == 1 ? pack_bf16(dy[1][2], dy[1][3]) : 0u);
    float dz2[8][4];
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
        float d[4] = {0.f, 0.f, 0.f, 0.f};
        mma_bf16(d, ay0, ay1, 0u, 0u, W.w3t[nt][lane], 0u);
#pragma unroll
        for (int k = 0; k < 4; ++k) dz2[nt][k] = act.z2[nt][k] > 0.f ? d[k] : 0.f;
    }
    O.dy[lane] = make_uint2(transposed(ay0), transposed(ay1));
    // dZ1 = (dZ2 W2) masked by z1 > 0
    float dz1[8][4];
    {
        uint32_t af[4][4];
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
            const float* p = dz2[2 * kk];
            const float* q = dz2[2 * kk + 1];
            af[kk][0] = pack_bf16(p[0], p[1]);
            af[kk][1] = pack_bf16(p[2], p[3]);
            af[kk][2] = pack_bf16(q[0], q[1]);
            af[kk][3] = pack_bf16(q[2], q[3]);
            O.d2[kk][lane] = make_uint4(transposed(af[kk][0]), transposed(af[kk][2]), transposed(af[kk][1]),
                                        transposed(af[kk][3]));
        }
#pragma unroll
        for (int nt = 0; nt < 8; ++nt) {
            float d[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
                const uint2 w = W.w2t[nt][kk][lane];
                mma_bf16(d, af[kk][0], af[kk][1], af[kk][2], af[kk][3], w.x, w.y);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) dz1[nt][k] = act.z1[nt][k] > 0.f ? d[k] : 0.f;
        }
    }
#pragma unroll
    for (int mt = 0; mt < 4; ++mt) {
        const float* p = dz1[2 * mt];
        const float* q = dz1[2 * mt + 1];
        O.d1[mt][lane] = make_uint4(transposed(pack_bf16(p[0], p[1])), transposed(pack_bf16(q[0], q[1])),
                                    transposed(pack_bf16(p[2], p[3])), transposed(pack_bf16(q[2], q[3])));
    }
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
        uint32_t h[4];
        relu_frag(act.z1, kk, h);
        O.h1[2 * kk][lane] = make_uint2(transposed(h[0]), transposed(h[1]));
        O.h1[2 * kk + 1][lane] = make_uint2(transposed(h[2]), transposed(h[3]));
        relu_frag(act.z2, kk, h);
        O.h2[2 * kk][lane] = make_uint2(transposed(h[0]), transposed(h[1]));
        O.h2[2 * kk + 1][lane] = make_uint2(transposed(h[2]), transposed(h[3]));
    }
    // bias gradients and loss in FP32: sums over the 16 samples. At each of
    // the three levels of the sum over the lane groups a lane passes on the
    // half of its columns that it doesn't keep (28 shuffles for 32 columns).
    float v[32];
#pragma unroll
    for (int nt = 0; nt < 8; ++nt)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            v[2 * nt + e] = dz1[nt][e] + dz1[nt][e + 2];
            v[16 + 2 * nt + e] = dz2[nt][e] + dz2[nt][e + 2];
        }
#pragma unroll
    for (int lv = 0; lv < 3; ++lv) {
        const int half = 16 >> lv;
        const bool hi = g >> lv & 1;
#pragma unroll
        for (int q = 0; q < half; ++q) {
            const float r = __shfl_xor_sync(0xffffffffu, hi ? v[q] : v[q + half], 4 << lv);
            v[q] = (hi ? v[q + half] : v[q]) + r;
        }
    }
    // lane group g holds columns q = 16 (g & 1) + 8 (g >> 1 & 1) + 4 (g >> 2) + 0..3
    const int nt0 = 4 * (g >> 1 & 1) + 2 * (g >> 2);
    float* sums = O.sums + MLP_H * (g & 1) + 8 * nt0 + 2 * t;
    *reinterpret_cast<float2*>(sums) = make_float2(v[0], v[1]);
    *reinterpret_cast<float2*>(sums + 8) = make_float2(v[2], v[3]);
    const float d0 = t == 0 ? dy[0][0] : (t == 1 ? dy[0][1] : (t == 2 ? dy[0][2] : dy[0][3]));
    const float d1 = t == 0 ? dy[1][0] : (t == 1 ? dy[1][1] : (t == 2 ? dy[1][2] : dy[1][3]));
    const float sy = sum_over_groups(d0 + d1);
    const float sl = sum_over_groups(L[0] + L[1]);
    if (g == 0) O.sums[2 * MLP_H + t] = sy;
    if (lane == 0) O.sums[2 * MLP_H + MLP_OUT] = sl;
}

// parameter i in the operands of a training step
__device__ __forceinline__ void put_training(TrainWeights& W, int i, float v) {
    put_forward(W.f, i, v);
    const __nv_bfloat16 b = __float2bfloat16_rn(v);
    if (i >= OFF_W2 && i < OFF_B2) {
        reinterpret_cast<__nv_bfloat16*>(W.w2t)[frag_entry<4>((i - OFF_W2) % MLP_H, (i - OFF_W2) / MLP_H)] = b;
    } else if (i >= OFF_W3 && i < OFF_B3) {
        const int r = (i - OFF_W3) / MLP_H, c = (i - OFF_W3) % MLP_H;
        reinterpret_cast<__nv_bfloat16*>(W.w3t)[(((c >> 3) * 32 + (c & 7) * 4 + (r >> 1)) << 1) + (r & 1)] = b;
    }
}

__global__ void k_mlp_emit(const float* __restrict__ theta, TrainWeights* W) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < MLP_NPARAM) put_training(*W, i, theta[i]);
}

struct AdamArgs {
    float lr, b1, b2, eps, c1, c2;
};

struct UpdateArgs {
    const TrainOps* ops;    // of the slice
    int chunks;             // of the slice
    bool first, last;       // slice of the batch
    float* acc;             // sums of the slices so far
    float* grad;            // gradient out (theta unchanged), or null: Adam
    float* loss;            // or null
    float *theta, *m, *v;
    TrainWeights* W;
    AdamArgs ad;
};

constexpr int UP_TILES = 56, UP_COLS = 27, UP_BLOCKS = UP_TILES + (NBIAS + UP_COLS - 1) / UP_COLS;

// Weight gradients, their sums over the batch and the Adam update in one
// launch: a block per 16 x 8 tile of the weight matrices (56) or 27 columns of
// the bias sums (5), a warp per chunk, the chunks' results added in order.
// Bound by latency (operands from L2, a chain of 8 mma, a chain of 32
// additions), so all of a chunk's loads are issued before its first product.
__global__ void __launch_bounds__(1024) k_mlp_train_update(UpdateArgs a) {
    __shared__ float part[32][128];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int tile = blockIdx.x;
    int which, mt = 0, nt = 0;
    if (tile < 16) { which = 1; mt = tile >> 2; nt = tile & 3; }
    else if (tile < 48) { which = 2; mt = (tile - 16) >> 3; nt = (tile - 16) & 7; }
    else if (tile < UP_TILES) { which = 3; nt = tile - 48; }
    else which = 0;
    // the parameter whose sum this thread forms, -1 for none
    int i = -1;
    if (which == 0) {
        const int j = (tile - UP_TILES) * UP_COLS + tid;
        if (tid < UP_COLS && j < NBIAS)
            i = j < MLP_H ? OFF_B1 + j : (j < 2 * MLP_H ? OFF_B2 + j - MLP_H : OFF_B3 + j - 2 * MLP_H);
    } else if (tid < 128) {
        const int l = tid >> 2, k = tid & 3;
        const int row = 16 * mt + (l >> 2) + 8 * (k >> 1), col = 8 * nt + 2 * (l & 3) + (k & 1);
        if (which == 1) { if (col < MLP_IN) i = OFF_W1 + row * MLP_IN + col; }
        else if (which == 2) i = OFF_W2 + row * MLP_H + col;
        else if (row < MLP_OUT) i = OFF_W3 + row * MLP_H + col;
    }
    // (the update before is complete when the launch in between has waited for
    // it, but only this grid's own wait makes its writes visible here)
    after_previous();
    const bool adam = i >= 0 && i < MLP_NPARAM && a.last && !a.grad;
    const float th = adam ? a.theta[i] : 0.f, mo = adam ? a.m[i] : 0.f, vo = adam ? a.v[i] : 0.f;
    float s = i >= 0 && !a.first ? a.acc[i] : 0.f;
    for (int c0 = 0; c0 < a.chunks; c0 += 32) {
        const int nc = a.chunks - c0 < 32 ? a.chunks - c0 : 32;
        if (which == 0) {
            const int c = tid / UP_COLS, jj = tid % UP_COLS, j = (tile - UP_TILES) * UP_COLS + jj;
            if (c < nc && j < NBIAS) {
                const TrainOps* O = a.ops + (long long)(c0 + c) * CHUNK_TILES;
                float w[CHUNK_TILES];
#pragma unroll
                for (int k = 0; k < CHUNK_TILES; ++k) w[k] = O[k].sums[j];
                float p = 0.f;
#pragma unroll
                for (int k = 0; k < CHUNK_TILES; ++k) p += w[k];
                part[c][jj] = p;
            }
        } else if (warp < nc) {
            const TrainOps* O = a.ops + (long long)(c0 + warp) * CHUNK_TILES;
            uint4 A[CHUNK_TILES];
            uint2 B[CHUNK_TILES];
#pragma unroll
            for (int k = 0; k < CHUNK_TILES; ++k) {
                if (which == 1) { A[k] = O[k].d1[mt][lane]; B[k] = O[k].x[nt][lane]; }
                else if (which == 2) { A[k] = O[k].d2[mt][lane]; B[k] = O[k].h1[nt][lane]; }
                else {
                    const uint2 dy = O[k].dy[lane];
                    A[k] = make_uint4(dy.x, 0u, dy.y, 0u);
                    B[k] = O[k].h2[nt][lane];
                }
            }
            float d[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int k = 0; k < CHUNK_TILES; ++k) mma_bf16(d, A[k].x, A[k].y, A[k].z, A[k].w, B[k].x, B[k].y);
            *reinterpret_cast<float4*>(&part[warp][4 * lane]) = make_float4(d[0], d[1], d[2], d[3]);
        }
        __syncthreads();
        if (i >= 0) {
#pragma unroll 8
            for (int c = 0; c < nc; ++c) s += part[c][tid];
        }
        __syncthreads();
    }
    if (i < 0) return;
    if (!a.last) {
        a.acc[i] = s;
        return;
    }
    if (i == MLP_NPARAM) {
        if (a.loss) *a.loss = s;
        return;
    }
    if (a.grad) {
        a.grad[i] = s;
        return;
    }
    const float mi = __fmaf_rn(1.f - a.ad.b1, s, __fmul_rn(a.ad.b1, mo));
    const float vi = __fmaf_rn(__fmul_rn(1.f - a.ad.b2, s), s, __fmul_rn(a.ad.b2, vo));
    a.m[i] = mi;
    a.v[i] = vi;
    const float p = th - a.ad.lr * (mi / a.ad.c1) / (sqrtf(vi / a.ad.c2) + a.ad.eps);
    a.theta[i] = p;
    put_training(*a.W, i, p);
}

// two blocks per SM: 66 944 stencils 27.2 us a call from cold caches (27.8 with
// three, 28 with one of 512 threads), 2 million 110 us (110, 113)
constexpr int INFER_THREADS = 256, INFER_BLOCKS = 2 * 152;

// The forward operands from the parameters, a pair of entries per thread and
// turn, with every load issued before the first is used
__device__ __forceinline__ void make_forward(MlpFwd& W, const float* __restrict__ theta) {
    const int tid = threadIdx.x;
    auto pair = [&](int off, int ld, int rows, int cols, int r, int c) -> uint32_t {
        const float* p = theta + off + r * ld + c;
        return pack_bf16(r < rows && c < cols ? p[0] : 0.f, r < rows && c + 1 < cols ? p[1] : 0.f);
    };
    // word e: half h of the register pair of lane l, operand e >> 6
    auto row = [](int e) { return e >> 3 & 7; };
    auto col = [](int e) { return (e >> 1 & 3) * 2 + (e & 1) * 8; };
    constexpr int N1 = sizeof(W.w1) / 4, N2 = sizeof(W.w2) / 4, N3 = sizeof(W.w3) / 4;
    uint32_t w1[(N1 + INFER_THREADS - 1) / INFER_THREADS], w2[(N2 + INFER_THREADS - 1) / INFER_THREADS];
#pragma unroll
    for (int q = 0; q < (int)(sizeof(w1) / 4); ++q) {
        const int e = q * INFER_THREADS + tid, o = e >> 6;
        w1[q] = pair(OFF_W1, MLP_IN, MLP_H, MLP_IN, 8 * (o >> 1) + row(e), 16 * (o & 1) + col(e));
    }
#pragma unroll
    for (int q = 0; q < (int)(sizeof(w2) / 4); ++q) {
        const int e = q * INFER_THREADS + tid, o = e >> 6;
        w2[q] = pair(OFF_W2, MLP_H, MLP_H, MLP_H, 8 * (o >> 2) + row(e), 16 * (o & 3) + col(e));
    }
    const uint32_t w3 = tid < N3 ? pair(OFF_W3, MLP_H, MLP_OUT, MLP_H, row(tid), 16 * (tid >> 6) + col(tid)) : 0u;
    const float b = tid < MLP_H ? theta[OFF_B1 + tid]
                                : (tid < 2 * MLP_H ? theta[OFF_B2 + tid - MLP_H]
                                                   : (tid < 2 * MLP_H + MLP_OUT ? theta[OFF_B3 + tid - 2 * MLP_H] : 0.f));
#pragma unroll
    for (int q = 0; q < (int)(sizeof(w1) / 4); ++q) reinterpret_cast<uint32_t*>(W.w1)[q * INFER_THREADS + tid] = w1[q];
#pragma unroll
    for (int q = 0; q < (int)(sizeof(w2) / 4); ++q) reinterpret_cast<uint32_t*>(W.w2)[q * INFER_THREADS + tid] = w2[q];
    if (tid < N3) reinterpret_cast<uint32_t*>(W.w3)[tid] = w3;
    if (tid < MLP_H) W.b1[tid] = b;
    else if (tid < 2 * MLP_H) W.b2[tid - MLP_H] = b;
    else if (tid < 2 * MLP_H + 8) W.b3[tid - 2 * MLP_H] = b;
}

// Raw outputs (n, curvature) of n stencils, a warp per 16. Each block makes
// its operands from the parameters itself, in shared memory, while its first
// inputs are on their way: one launch and no scratch memory. Bound by latency
// (parameters, inputs, a chain of 14 mma). 66 944 stencils: a call took
// 35.8 us with operands in scratch memory made by two launches before, now
// 18.3 us, most of it the launch and the wait of the call.
__global__ void __launch_bounds__(INFER_THREADS) k_mlp_infer(const float* __restrict__ theta,
                                                             const float* __restrict__ fill, long long n,
                                                             float4* out) {
    __shared__ MlpFwd W;
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const long long stride = (long long)gridDim.x * (INFER_THREADS / 2);
    long long base = ((long long)blockIdx.x * (INFER_THREADS / 32) + (threadIdx.x >> 5)) * 16;
    uint32_t xf[2][4], next[2][4];
    auto load = [&](long long b) {
        input_frags([&](int r, int col) -> float {
            const long long row = b + g + 8 * r;
            return (row < n && col < 27) ? fill[row * 27 + col] : 0.f;
        }, next);
    };
    load(base);
    make_forward(W, theta);
    __syncthreads();
    for (; base < n; base += stride) {
#pragma unroll
        for (int k = 0; k < 8; ++k) xf[k >> 2][k & 3] = next[k >> 2][k & 3];
        load(base + stride);
        MlpAct act;
        mlp_forward_ops(W.w1, W.w2, W.w3, W.b1, W.b2, W.b3, xf, act);
        float y[2][4];
        mlp_outputs(act, y[0], y[1]);
        if (t < 2) {
            const long long row = base + g + 8 * t;
            if (row < n) out[row] = t ? make_float4(y[1][0], y[1][1], y[1][2], y[1][3])
                                      : make_float4(y[0][0], y[0][1], y[0][2], y[0][3]);
        }
    }
}

// First-layer operands of the mirror images of R-17g, built on the host from
// BF16 bit patterns: block m - 1 (m = 1 mirrors x, 2 mirrors y, 3 both) is W1
// with input column q taken from the mirrored column, so that it applied to
// a stencil gives W1 applied to the mirrored stencil.
void mlp_mirror_w1_host(const uint16_t* w, __nv_bfloat16* out) {
    for (int m = 1; m < 4; ++m)
        for (int r = 0; r < MLP_H; ++r)
            for (int c = 0; c < 32; ++c) {
                __nv_bfloat16_raw v;
                v.x = 0;   // +0.0: the padding columns 27..31
                if (c < MLP_IN) {
                    int a = c % 3, b = (c / 3) % 3;
                    const int z = c / 9;
                    if (m & 1) a = 2 - a;
                    if (m & 2) b = 2 - b;
                    v.x = w[OFF_W1 + r * MLP_IN + a + 3 * b + 9 * z];
                }
                out[(m - 1) * MLP_H * 32 + r * 32 + c] = __nv_bfloat16(v);
            }
}

// The in-step weights in fragment order (MlpFrag), from the operand copies
// h and the mirrored first layers w1m: lane (g, t) of an mma over n-tile nt
// and k-tile kk takes row 8 nt + g (g for the output layer) and the column
// pairs 16 kk + 2t and 16 kk + 2t + 8, packed low element first.
void mlp_frag_host(const MlpBf16& h, const __nv_bfloat16* w1m, MlpFrag& G) {
    auto pair = [](const __nv_bfloat16* p) {
        __nv_bfloat16_raw lo = p[0], hi = p[1];
        return (uint32_t)lo.x | ((uint32_t)hi.x << 16);
    };
    for (int lane = 0; lane < 32; ++lane) {
        const int g = lane >> 2, t = lane & 3;
        for (int m = 0; m < 4; ++m) {
            const __nv_bfloat16* w1 = m == 0 ? h.w1 : w1m + (m - 1) * MLP_H * 32;
            for (int nt = 0; nt < 8; ++nt)
                for (int kk = 0; kk < 2; ++kk) {
                    const __nv_bfloat16* r = w1 + (8 * nt + g) * 32 + 16 * kk + 2 * t;
                    G.w1[m][nt][kk][lane] = make_uint2(pair(r), pair(r + 8));
                }
        }
        for (int nt = 0; nt < 8; ++nt)
            for (int kk = 0; kk < 4; ++kk) {
                const __nv_bfloat16* r = h.w2 + (8 * nt + g) * MLP_H + 16 * kk + 2 * t;
                G.w2[nt][kk][lane] = make_uint2(pair(r), pair(r + 8));
            }
        for (int kk = 0; kk < 4; ++kk) {
            const __nv_bfloat16* r = h.w3 + g * MLP_H + 16 * kk + 2 * t;
            G.w3[kk][lane] = make_uint2(pair(r), pair(r + 8));
        }
    }
}

// operand copies built on the host from BF16 bit patterns
void mlp_from_bf16_host(const uint16_t* w, MlpBf16& h) {
    auto f = [](uint16_t b) {
        const uint32_t u = (uint32_t)b << 16;
        float x;
        memcpy(&x, &u, 4);
        return x;
    };
    auto bf = [](uint16_t b) {
        __nv_bfloat16_raw r;
        r.x = b;
        return __nv_bfloat16(r);
    };
    memset(&h, 0, sizeof(h));   // +0.0 in BF16 and FP32 is all-zero bits
    for (int r = 0; r < MLP_H; ++r)
        for (int c = 0; c < MLP_IN; ++c) h.w1[r * 32 + c] = bf(w[OFF_W1 + r * MLP_IN + c]);
    for (int r = 0; r < MLP_H; ++r)
        for (int c = 0; c < MLP_H; ++c) h.w2[r * MLP_H + c] = bf(w[OFF_W2 + r * MLP_H + c]);
    for (int r = 0; r < MLP_OUT; ++r)
        for (int c = 0; c < MLP_H; ++c) h.w3[r * MLP_H + c] = bf(w[OFF_W3 + r * MLP_H + c]);
    for (int i = 0; i < MLP_H; ++i) {
        h.b1[i] = f(w[OFF_B1 + i]);
        h.b2[i] = f(w[OFF_B2 + i]);
    }
    for (int i = 0; i < MLP_OUT; ++i) h.b3[i] = f(w[OFF_B3 + i]);
}

}  // namespace fsl

// ------------------------------------------------------------ C ABI
using namespace fsl;

namespace {

// device memory of one training or gradient call, in one allocation; weights,
// moments and acc start at zero
struct TrainScratch {
    TrainWeights* W = nullptr;
    float *m, *v, *acc;
    TrainOps* ops;
    bool get(long long samples, cudaStream_t st) {
        const long long chunks = (samples + CHUNK - 1) / CHUNK;
        const size_t slice = (size_t)(chunks < SLICE_CHUNKS ? chunks : SLICE_CHUNKS);
        const size_t zeroed = (sizeof(TrainWeights) + 3 * (MLP_NPARAM + 4) * sizeof(float) + 15) / 16 * 16;
        if (cudaMalloc(&W, zeroed + slice * CHUNK_TILES * sizeof(TrainOps)) != cudaSuccess) {
            cudaGetLastError();
            W = nullptr;
            return false;
        }
        m = reinterpret_cast<float*>(W + 1);
        v = m + MLP_NPARAM + 4;
        acc = v + MLP_NPARAM + 4;
        ops = reinterpret_cast<TrainOps*>(reinterpret_cast<char*>(W) + zeroed);
        cudaMemsetAsync(W, 0, zeroed, st);
        return true;
    }
    ~TrainScratch() {
        if (W) cudaFree(W);
    }
};

int finish(cudaStream_t st) {
    if (cudaGetLastError() != cudaSuccess) return FSLBM_EDEVICE;
    if (cudaStreamSynchronize(st) != cudaSuccess) return FSLBM_EDEVICE;
    return FSLBM_OK;
}

void emit(const float* theta, TrainWeights* W, cudaStream_t st) {
    k_mlp_emit<<<(MLP_NPARAM + 255) / 256, 256, 0, st>>>(theta, W);
}

// One batch: slices of SLICE_CHUNKS chunks, so that the operands of a large
// batch stay at 10 MB (in L2), each with its two launches
void batch_gradient(TrainArgs a, UpdateArgs u, cudaStream_t st) {
    const int chunks = (a.B + CHUNK - 1) / CHUNK;
    for (int c0 = 0; c0 < chunks; c0 += SLICE_CHUNKS) {
        u.chunks = chunks - c0 < SLICE_CHUNKS ? chunks - c0 : SLICE_CHUNKS;
        u.first = c0 == 0;
        u.last = c0 + u.chunks == chunks;
        a.first = c0 * CHUNK;
        a.tiles = u.chunks * CHUNK_TILES;
        launch_after(k_mlp_train_samples, blocks_for(a.tiles * 32, SAMPLE_THREADS), SAMPLE_THREADS, st, a);
        launch_after(k_mlp_train_update, UP_BLOCKS, 1024, st, u);
    }
}

}  // namespace

extern "C" {

int fslbm_mlp_stencils(const double* params, int64_t n, float* fill, float* target, void* cuda_stream) {
    if (!params || !fill || !target || n <= 0 || n > ((int64_t)1 << 31) - 1) return FSLBM_EINVAL;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    k_make_stencils<<<(unsigned)n, GEN_THREADS, 0, st>>>(params, (long long)n, fill, target);
    return finish(st);
}

int fslbm_mlp_gradient(const float* theta, const float* fill, const float* target, int64_t n, double lam,
                       double mu, float* grad, float* loss, void* cuda_stream) {
    if (!theta || !fill || !target || !grad || !loss || n <= 0 || n > ((int64_t)1 << 24)) return FSLBM_EINVAL;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    TrainScratch sc;
    if (!sc.get(n, st)) return FSLBM_ENOMEM;
    emit(theta, sc.W, st);
    TrainArgs a{};
    a.W = sc.W;
    a.fill = fill;
    a.target = target;
    a.n = n;
    a.B = (int)n;
    a.mode = TR_FIXED;
    a.lam = (float)lam;
    a.mu = (float)mu;
    a.ops = sc.ops;
    UpdateArgs u{};
    u.ops = sc.ops;
    u.acc = sc.acc;
    u.grad = grad;
    u.loss = loss;
    batch_gradient(a, u, st);
    return finish(st);
}

int fslbm_mlp_train(float* theta, const float* fill, const float* target, int64_t n, int64_t steps, int batch,
                    double lr, double lr_end, double lam, double mu, uint64_t seed, int augment, float* loss_curve,
                    void* cuda_stream) {
    if (!theta || !fill || !target || n <= 0 || n > ((int64_t)1 << 31) - 1 || steps < 0 || batch <= 0 ||
        batch > (1 << 20) || !(lr >= 0.0) || !(lr_end >= 0.0))
        return FSLBM_EINVAL;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    TrainScratch sc;
    if (!sc.get(batch, st)) return FSLBM_ENOMEM;
    emit(theta, sc.W, st);
    TrainArgs a{};
    a.W = sc.W;
    a.fill = fill;
    a.target = target;
    a.n = n;
    a.B = batch;
    a.mode = augment ? TR_DRAW_SYM : TR_DRAW;
    a.seed = seed;
    a.lam = (float)lam;
    a.mu = (float)mu;
    a.ops = sc.ops;
    UpdateArgs u{};
    u.ops = sc.ops;
    u.acc = sc.acc;
    u.theta = theta;
    u.m = sc.m;
    u.v = sc.v;
    u.W = sc.W;
    const double b1 = 0.9, b2 = 0.999;
    double p1 = 1.0, p2 = 1.0;
    for (int64_t k = 0; k < steps; ++k) {
        a.step = (long long)k;
        p1 *= b1;
        p2 *= b2;
        // learning rate: geometric from lr to lr_end over the run (constant
        // when lr_end is 0 or equal to lr)
        const double frac = steps > 1 ? (double)k / (double)(steps - 1) : 0.0;
        const double lr_k = (lr_end > 0.0 && lr > 0.0) ? lr * std::pow(lr_end / lr, frac) : lr;
        u.ad = AdamArgs{(float)lr_k, (float)b1, (float)b2, 1e-8f, (float)(1.0 - p1), (float)(1.0 - p2)};
        u.loss = loss_curve ? loss_curve + k : nullptr;
        batch_gradient(a, u, st);
        if ((k & 255) == 255 && cudaGetLastError() != cudaSuccess) return FSLBM_EDEVICE;
    }
    return finish(st);
}

int fslbm_mlp_infer(const float* theta, const float* fill, int64_t n, float* out, void* cuda_stream) {
    if (!theta || !fill || !out || n <= 0) return FSLBM_EINVAL;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    const long long blocks_needed = ((n + 15) / 16 + INFER_THREADS / 32 - 1) / (INFER_THREADS / 32);
    const int blocks = (int)(blocks_needed < INFER_BLOCKS ? blocks_needed : INFER_BLOCKS);
    k_mlp_infer<<<blocks, INFER_THREADS, 0, st>>>(theta, fill, (long long)n, reinterpret_cast<float4*>(out));
    return finish(st);
}

}  // extern "C"

// Free-surface (volume-of-fluid) update after the stream-collide sweep
// (Section 2.1): fill levels, interface normals, conversion of interface
// cells, filling/emptying of their neighbours, excess-mass redistribution,
// the FP64 mass pool, and the interface work list. Every kernel below works
// on the device-counted list of interface cells (or of cells becoming
// interface), so its cost scales with the surface, not the lattice; each
// cell computes its own result from a snapshot of its neighbourhood, so no
// result depends on thread order.
#include "fslbm_dev.cuh"
#include "mlp_dev.cuh"

namespace fsl {

constexpr int LIST_THREADS = 256;
constexpr int LIST_BLOCKS = 152 * 4;

#define FOR_LIST(i, countp)                                                       \
    for (int i = blockIdx.x * blockDim.x + threadIdx.x, _cnt = *(countp); i < _cnt; \
         i += gridDim.x * blockDim.x)

// Parker-Youngs normal: gradient sum_c w(c) c phi(x+c) with weights 4 (face),
// 2 (edge), 1 (corner); solid and wall neighbours take the centre value;
// n = -grad/|grad| points toward the gas.
__device__ __forceinline__ float py_weight(int q) { return nnz(q) == 1 ? 4.f : (nnz(q) == 2 ? 2.f : 1.f); }
__device__ __forceinline__ float4 py_result(float gx, float gy, float gz) {
    const float len = sqrtf(gx * gx + gy * gy + gz * gz);
    if (len > 0.f) return make_float4(-gx / len, -gy / len, -gz / len, 0.f);
    return make_float4(0.f, 0.f, 0.f, 0.f);
}
// (two load phases, the 26 flags and the fill levels of the interface
// neighbours, each in flight together)
__device__ __forceinline__ float4 py_normal(const Dev& s, int c) {
    int x, y, z;
    coords32(s, c, x, y, z);
    const NbrOffsets o = nbr_offsets(s, x, y, z);
    uint8_t t[27];
#pragma unroll
    for (int q = 0; q < 27; ++q)
        t[q] = (o.wall & wall_bits(cx(q), cy(q), cz(q)))
                   ? (uint8_t)T_SOL
                   : s.flags[c + o.ox[1 + cx(q)] + o.oy[1 + cy(q)] + o.oz[1 + cz(q)]] & TYPE_MASK;
    float v[27];
#pragma unroll
    for (int q = 0; q < 27; ++q)
        v[q] = t[q] == T_IFC ? s.phi[c + o.ox[1 + cx(q)] + o.oy[1 + cy(q)] + o.oz[1 + cz(q)]]
                             : (t[q] == T_LIQ ? 1.f : 0.f);
    float gx = 0.f, gy = 0.f, gz = 0.f;
#pragma unroll
    for (int q = 0; q < 27; ++q) {
        if (q == 13) continue;
        const float w = py_weight(q), u = t[q] == T_SOL ? v[13] : v[q];
        gx += w * cx(q) * u;
        gy += w * cy(q) * u;
        gz += w * cz(q) * u;
    }
    return py_result(gx, gy, gz);
}

__global__ void k_normals(Dev s, float4* out, const int* list, const int* countp) {
    after_previous();
    for (int i = blockIdx.x * blockDim.x + threadIdx.x, cnt = min(*countp, s.wl_cap); i < cnt;
         i += gridDim.x * blockDim.x) {
        int c = list[i];
        out[c] = py_normal(s, c);
    }
}

// Learned normal (R-17), a warp per 16 interface cells of the list. Lane
// (g, t) loads the stencil columns of its input fragments for the cells of
// rows g and g + 8; together the four lanes of a group cover all 27, agree on
// whether a wall or solid cell lies in the block, and sum the Parker-Youngs
// gradient from the same values (walls and solids taking the centre value).
// The Parker-Youngs normal is both the fallback (wall or solid in the block,
// raw length outside [1/2, 2]) and the check on the network (its normal more
// than 30 degrees away falls back too). out[c] = (n, curvature), curvature 0 where the fallback is
// taken.
__global__ void __launch_bounds__(128, 5) k_mlp_normals(Dev s, float4* out, const int* list, const int* countp) {
    after_previous();
    const int count = min(*countp, s.wl_cap);
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    const unsigned full = 0xffffffffu;
    unsigned long long evaluated = 0, taken = 0;
    for (int base = ((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 16; base < count; base += nwarps * 16) {
        int cell[2];
        float v[2][8];
        bool bad[2];
        float gr[2][3];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int li = base + g + 8 * r;
            cell[r] = li < count ? list[li] : -1;
            bad[r] = false;
            gr[r][0] = gr[r][1] = gr[r][2] = 0.f;
            int x = 0, y = 0, z = 0;
            float p0 = 0.f;
            if (cell[r] >= 0) {
                coords32(s, cell[r], x, y, z);
                p0 = s.phi[cell[r]];
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int col = frag_col(j >> 2, j & 3, t);
                float in = 0.f, raw = p0;
                if (cell[r] >= 0 && col < 27) {
                    const long long nb = nbr(s, x, y, z, cx(col), cy(col), cz(col));
                    if (nb < 0) {
                        bad[r] = true;
                    } else {
                        const int tn = s.flags[nb] & TYPE_MASK;
                        if (tn == T_SOL) {
                            bad[r] = true;
                        } else {
                            raw = tn == T_LIQ ? 1.f : (tn == T_IFC ? s.phi[nb] : 0.f);
                            in = fminf(fmaxf(raw, 0.f), 1.f);
                        }
                    }
                    if (col != 13) {
                        const float w = nnz(col) == 1 ? 4.f : (nnz(col) == 2 ? 2.f : 1.f);
                        gr[r][0] += w * cx(col) * raw;
                        gr[r][1] += w * cy(col) * raw;
                        gr[r][2] += w * cz(col) * raw;
                    }
                }
                v[r][j] = in;
            }
            bad[r] |= __shfl_xor_sync(full, bad[r], 1);
            bad[r] |= __shfl_xor_sync(full, bad[r], 2);
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                gr[r][k] += __shfl_xor_sync(full, gr[r][k], 1);
                gr[r][k] += __shfl_xor_sync(full, gr[r][k], 2);
            }
        }
        uint32_t xf[2][4];
#pragma unroll
        for (int kk = 0; kk < 2; ++kk) {
            xf[kk][0] = pack_bf16(v[0][4 * kk + 0], v[0][4 * kk + 1]);
            xf[kk][1] = pack_bf16(v[1][4 * kk + 0], v[1][4 * kk + 1]);
            xf[kk][2] = pack_bf16(v[0][4 * kk + 2], v[0][4 * kk + 3]);
            xf[kk][3] = pack_bf16(v[1][4 * kk + 2], v[1][4 * kk + 3]);
        }
        // R-17g with mlp_mirror: the network also on the stencil mirrored in
        // x, in y and in both (the first layer with permuted columns on the
        // same inputs), each output mapped back and the four averaged
        MlpAct act;
        float y[2][4];
        const int passes = s.mlp_mirror ? 4 : 1;
#pragma unroll 1
        for (int m = 0; m < passes; ++m) {
            const MlpBf16* W = s.mlp;
            const MlpFrag* G = s.mlp_frag;
            // the operands are reloaded in every pass rather than held in
            // registers across passes
            asm volatile("" : "+l"(W), "+l"(G));
            mlp_forward_frag(*W, *G, m, xf, act);
            float ym[2][4];
            mlp_outputs(act, ym[0], ym[1]);
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                if (m == 0) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) y[r][k] = ym[r][k];
                } else {
                    y[r][0] += (m & 1) ? -ym[r][0] : ym[r][0];
                    y[r][1] += (m & 2) ? -ym[r][1] : ym[r][1];
                    y[r][2] += ym[r][2];
                    y[r][3] += ym[r][3];
                }
            }
        }
        if (passes == 4) {
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int k = 0; k < 4; ++k) y[r][k] *= 0.25f;
        }
        if (t < 2 && cell[t] >= 0) {
            const int c = cell[t];
            const float gl = sqrtf(gr[t][0] * gr[t][0] + gr[t][1] * gr[t][1] + gr[t][2] * gr[t][2]);
            const float4 fd = gl > 0.f ? make_float4(-gr[t][0] / gl, -gr[t][1] / gl, -gr[t][2] / gl, 0.f)
                                       : make_float4(0.f, 0.f, 0.f, 0.f);
            float4 res = fd;
            ++evaluated;
            const float len = sqrtf(y[t][0] * y[t][0] + y[t][1] * y[t][1] + y[t][2] * y[t][2]);
            if (!bad[t] && len >= 0.5f && len <= 2.f) {
                const float mx = y[t][0] / len, my = y[t][1] / len, mz = y[t][2] / len;
                if (mx * fd.x + my * fd.y + mz * fd.z >= 0.8660254f) {   // cos 30 degrees
                    res = make_float4(mx, my, mz, y[t][3]);
                    ++taken;
                }
            }
            out[c] = res;
        }
    }
    if (s.mlp_stats) {
        for (int o = 16; o > 0; o >>= 1) {
            evaluated += __shfl_xor_sync(full, evaluated, o);
            taken += __shfl_xor_sync(full, taken, o);
        }
        if (lane == 0 && evaluated) {
            atomicAdd(&s.mlp_stats[0], evaluated);
            atomicAdd(&s.mlp_stats[1], taken);
        }
    }
}

// normals of the cells of a list (the interface list, or the cells that
// convert in this step)
static int normals_into(const Dev& s, float4* out, const int* list, const int* count, cudaStream_t st) {
    if (s.mlp) launch_after(k_mlp_normals, 152 * 8, 128, st, s, out, list, count);
    else launch_after(k_normals, LIST_BLOCKS, LIST_THREADS, st, s, out, list, count);
    return 1;
}

// ------------------------------------------------------------ conversion
// The converting cells of a step are few (tens to thousands), so the kernels
// over them give each a warp with a lane per neighbour: a thread per cell
// walked up to 26 neighbours, 27 loads each, one after the other. With a wavy
// surface on 1024x64x128 cells (72 k interface cells, FP16): new cells and
// excess shares 138 + 30 -> 6.3 us, marks 26 -> 4.8 us, gather and the new
// types 30 + 5 + 4 + 3 -> 11.7 us, candidates and fill levels 15 + 4 -> 6.7 us,
// conflicts 13.8 -> 5.8 us.

// fill levels, and the conversion candidates: fill level beyond 1 + eps or
// below -eps, or isolation (no gas neighbour -> liquid, no liquid neighbour
// -> gas). Clears the counts of the lists that the kernels after it fill.
__global__ void __launch_bounds__(LIST_THREADS) k_candidates(Dev s) {
    after_previous();
    if (blockIdx.x == 0 && threadIdx.x == 0)
        *s.cl_count = *s.nl_count = *s.tl_count = *s.dl_count = *s.tile_count = 0;
    FOR_LIST(i, s.wl_count) {
        const int c = s.wl[i];
        int x, y, z;
        coords32(s, c, x, y, z);
        const NbrOffsets o = nbr_offsets(s, x, y, z);
        unsigned gas = 0, liq = 0;
#pragma unroll
        for (int q = 0; q < 27; ++q) {
            if (q == 13 || (o.wall & wall_bits(cx(q), cy(q), cz(q)))) continue;
            const int t = s.flags[c + o.ox[1 + cx(q)] + o.oy[1 + cy(q)] + o.oz[1 + cz(q)]] & TYPE_MASK;
            gas |= t == T_GAS;
            liq |= t == T_LIQ;
        }
        const float ph = s.mass[c] / s.ru[c].x;
        s.phi[c] = ph;
        uint8_t cv = 0;
        if (ph > 1.f + s.eps_conv) cv = CV_TO_LIQ;
        else if (ph < -s.eps_conv) cv = CV_TO_GAS;
        else if (!gas) cv = CV_TO_LIQ;
        else if (!liq) cv = CV_TO_GAS;
        s.conv[c] = cv;
    }
}

// filling wins: a to-gas cell next to a to-liquid cell stays interface. The
// cells that still convert are listed (their normals give the excess-mass
// weights).
__global__ void __launch_bounds__(LIST_THREADS) k_conflict(Dev s) {
    after_previous();
    const int cnt = *s.wl_count, stride = gridDim.x * blockDim.x;
    for (int base = blockIdx.x * blockDim.x; base < cnt; base += stride) {
        const int i = base + threadIdx.x;
        int c = 0;
        uint8_t cv = 0;
        if (i < cnt) {
            c = s.wl[i];
            cv = s.conv[c];
        }
        if (cv == CV_TO_GAS) {
            int x, y, z;
            coords32(s, c, x, y, z);
            const NbrOffsets o = nbr_offsets(s, x, y, z);
            bool clash = false;
#pragma unroll
            for (int q = 0; q < 27; ++q) {
                if (q == 13 || (o.wall & wall_bits(cx(q), cy(q), cz(q)))) continue;
                clash |= s.conv[c + o.ox[1 + cx(q)] + o.oy[1 + cy(q)] + o.oz[1 + cz(q)]] == CV_TO_LIQ;
            }
            if (clash) s.conv[c] = cv = 0;
        }
        warp_append(s, cv != 0, c, s.cl, s.cl_count, s.wl_cap);
    }
}

// a warp per entry of a list of n
#define FOR_WARP(i, n)                                                                                  \
    for (int i = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), _st = (gridDim.x * blockDim.x) >> 5; i < (n); \
         i += _st)

// Gas neighbours of filled cells and liquid neighbours of emptied cells
// become interface cells; each is listed once (first setter of its mark).
// With FD the Parker-Youngs normal of the converting cell from the same
// neighbours (fill levels and types are still those the candidates saw).
template <bool FD>
__global__ void __launch_bounds__(LIST_THREADS) k_mark(Dev s) {
    after_previous();
    const int lane = threadIdx.x & 31;
    const int ncl = min(*s.cl_count, s.wl_cap);
    FOR_WARP(i, ncl) {
        const int c = s.cl[i];
        const uint8_t cv = s.conv[c];
        int x, y, z;
        coords32(s, c, x, y, z);
        const int nb = lane < 27 ? nbr_q(s, x, y, z, lane) : -1;
        const int tn = nb >= 0 ? s.flags[nb] & TYPE_MASK : (int)T_SOL;
        uint8_t bit = 0;
        if (cv == CV_TO_LIQ && tn == T_GAS) bit = F_NEW;
        if (cv == CV_TO_GAS && tn == T_LIQ) bit = F_EMPTIED;
        const bool fresh = bit && !(flag_or(s.flags, nb, bit) & bit);
        warp_append(s, fresh, nb, s.nl, s.nl_count, s.nl_cap);
        if (FD) {
            float v = tn == T_IFC ? s.phi[nb] : (tn == T_LIQ ? 1.f : 0.f);
            const float p0 = __shfl_sync(0xffffffffu, v, 13);
            if (tn == T_SOL) v = p0;
            const int dx = lane % 3 - 1, dy = (lane / 3) % 3 - 1, dz = lane / 9 - 1;
            const int k = (dx != 0) + (dy != 0) + (dz != 0);
            v *= lane < 27 ? (k == 1 ? 4.f : (k == 2 ? 2.f : 1.f)) : 0.f;
            const float gx = ordered_sum27(dx * v), gy = ordered_sum27(dy * v), gz = ordered_sum27(dz * v);
            if (lane == 0) s.nrm1[c] = py_result(gx, gy, gz);
        }
    }
}

__device__ __forceinline__ bool is_receiver(const Dev& s, int c) {
    const uint8_t fl = s.flags[c];
    if (fl & (F_NEW | F_EMPTIED)) return true;
    return (fl & TYPE_MASK) == T_IFC && (s.conv[c] & 3) == 0;
}

// New interface cells: from gas, f* = f_eq(mean rho, mean u) of the liquid
// and interface neighbours (cell types of the snapshot) with m = 0; from
// liquid, PDFs kept and m = rho. Both get their own PDFs in the side buffer.
// One warp; lane q holds neighbour and direction q.
template <typename S, int LP>
__device__ __forceinline__ void init_new(const Dev& s, int c, int lane) {
    const uint8_t fl = s.flags[c];
    S* f = static_cast<S*>(s.f);
    S* fs = static_cast<S*>(s.fs);
    int x, y, z;
    coords32(s, c, x, y, z);
    const int nb = lane < 27 ? nbr_q(s, x, y, z, lane) : -1;
    float h = 0.f;
    const long long slot = lane < 27 ? lane_slot<S, LP>(s, lane, c, nb, z, h) : 0;
    const float h0 = Store<S>::HREF ? s.href[z] : 0.f;
    float v, rho, ux, uy, uz, m;
    if (fl & F_NEW) {
        float rs = 0.f, us = 0.f, vs = 0.f, ws = 0.f, n = 0.f;
        if (nb >= 0 && lane != 13) {
            const int tn = s.flags[nb] & TYPE_MASK;
            if (tn == T_IFC) {
                const float4 r = s.ru[nb];
                rs = r.x; us = r.y; vs = r.z; ws = r.w;
                n = 1.f;
            } else if (tn == T_LIQ) {
                int bx, by, bz;
                coords32(s, nb, bx, by, bz);
                float g[27];
                load_cell<S, LP>(s, nb, bx, by, bz, g);
                post_moments(s, g, rs, us, vs, ws);
                n = 1.f;
            }
        }
        n = (float)__popc(__ballot_sync(0xffffffffu, n > 0.f));
        rs = ordered_sum27(rs);
        const float inv = n > 0.f ? 1.f / n : 0.f;
        rho = n > 0.f ? rs * inv : s.rho_gas;
        ux = ordered_sum27(us) * inv;
        uy = ordered_sum27(vs) * inv;
        uz = ordered_sum27(ws) * inv;
        v = feq_dev(lane < 27 ? lane : 0, rho, ux, uy, uz);
        if (lane < 27) Store<S>::st(f + slot, with_ref<S>(v, lane, -h));
        m = 0.f;
    } else {
        v = lane < 27 ? with_ref<S>(Store<S>::ld(f + slot), lane, h) : 0.f;
        const float d = ordered_sum27(v);
        const float jx = ordered_sum27((lane % 3 - 1) * v), jy = ordered_sum27(((lane / 3) % 3 - 1) * v),
                    jz = ordered_sum27((lane / 9 - 1) * v);
        rho = 1.f + d;
        const float inv = 1.f / rho;
        ux = (jx - 0.5f * rho * s.gx) * inv;
        uy = (jy - 0.5f * rho * s.gy) * inv;
        uz = (jz - 0.5f * rho * s.gz) * inv;
        m = rho;
    }
    if (lane < 27) Store<S>::st(fs + (long long)lane * s.n + c, with_ref<S>(v, lane, -h0));
    if (lane == 0) {
        s.mass[c] = m;
        s.ru[c] = make_float4(rho, ux, uy, uz);
    }
}

// Excess mass of a converting cell: m - rho (to liquid, m := rho) or m (to
// gas, m := 0), spread over interface neighbours with weights max(0, n.c)
// (filled) or max(0, -n.c) (emptied), evenly if all weights vanish or the
// even variant is selected, into the FP64 pool if there is no interface
// neighbour. One warp, lane q on neighbour q.
__device__ __forceinline__ void excess_prep(const Dev& s, int c, int lane) {
    const uint8_t cv = s.conv[c];
    const float rho = s.ru[c].x, m = s.mass[c];
    const float4 n1 = s.nrm1[c];
    int x, y, z;
    coords32(s, c, x, y, z);
    const int nb = lane < 27 && lane != 13 ? nbr_q(s, x, y, z, lane) : -1;
    const bool rec = nb >= 0 && is_receiver(s, nb);
    const float sg = cv == CV_TO_LIQ ? 1.f : -1.f;
    const float w = sg * (n1.x * (lane % 3 - 1) + n1.y * ((lane / 3) % 3 - 1) + n1.z * (lane / 9 - 1));
    const int nrec = __popc(__ballot_sync(0xffffffffu, rec));
    const float wsum = ordered_sum27(rec && w > 0.f ? w : 0.f);
    if (lane != 0) return;
    const float ex = cv == CV_TO_LIQ ? m - rho : m;
    s.mass[c] = cv == CV_TO_LIQ ? rho : 0.f;
    if (nrec == 0) {
        atomicAdd(s.pool, (double)ex);
        s.exscale[c] = 0.f;
    } else if (wsum > 0.f && !s.excess_even) {
        s.exscale[c] = ex / wsum;
    } else {
        s.exscale[c] = ex / (float)nrec;
        s.conv[c] = cv | CV_EVEN;
    }
}

// The new interface cells and the converting cells in one launch: the first
// write the state of cells that are still gas or liquid in the snapshot, the
// second read and write that of interface cells only.
template <typename S, int LP>
__global__ void __launch_bounds__(LIST_THREADS) k_init_and_prep(Dev s) {
    after_previous();
    const int lane = threadIdx.x & 31;
    const int nnl = min(*s.nl_count, s.nl_cap), ncl = min(*s.cl_count, s.wl_cap);
    FOR_WARP(i, nnl + ncl) {
        if (i < nnl) init_new<S, LP>(s, s.nl[i], lane);
        else excess_prep(s, s.cl[i - nnl], lane);
        __syncwarp();
    }
}

// the excess mass a receiver takes from the converting cells around it
__device__ __forceinline__ float gather_excess(const Dev& s, int c, bool& any) {
    int x, y, z;
    coords32(s, c, x, y, z);
    const NbrOffsets o = nbr_offsets(s, x, y, z);
    unsigned conv = 0;
#pragma unroll
    for (int q = 0; q < 27; ++q) {
        if (q == 13 || (o.wall & wall_bits(cx(q), cy(q), cz(q)))) continue;
        if (s.conv[c + o.ox[1 + cx(q)] + o.oy[1 + cy(q)] + o.oz[1 + cz(q)]] & 3) conv |= 1u << q;
    }
    any = conv != 0;
    float add = 0.f;
    for (; conv; conv &= conv - 1) {
        const int q = __ffs(conv) - 1;
        const int nb = nbr_q(s, x, y, z, q);
        const uint8_t cv = s.conv[nb];
        float w;
        if (cv & CV_EVEN) w = 1.f;
        else {
            // direction from the converting cell to this receiver is -c_q
            const float4 n1 = s.nrm1[nb];
            const float sg = (cv & 3) == CV_TO_LIQ ? 1.f : -1.f;
            w = -sg * (n1.x * (q % 3 - 1) + n1.y * ((q / 3) % 3 - 1) + n1.z * (q / 9 - 1));
            w = w > 0.f ? w : 0.f;
        }
        add += s.exscale[nb] * w;
    }
    return add;
}

// Excess mass gathered by the receivers, and the new types and fill levels.
// A cell reads the conversion codes, normals and scales of its neighbours,
// which nothing here writes, and writes its own mass, fill level and flag.
// Without a converting cell everything stands as the candidates left it.
__global__ void __launch_bounds__(LIST_THREADS) k_finish_conversion(Dev s) {
    after_previous();
    if (*s.cl_count == 0) return;
    FOR_LIST(i, s.wl_count) {
        const int c = s.wl[i];
        const uint8_t cv = s.conv[c] & 3;
        if (cv == CV_TO_LIQ) {
            s.flags[c] = T_LIQ;
        } else if (cv == CV_TO_GAS) {
            s.flags[c] = T_GAS;
            s.mass[c] = 0.f;
            s.phi[c] = 0.f;
        } else {
            bool any;
            const float add = gather_excess(s, c, any);
            if (any) {
                const float m = s.mass[c] + add;
                s.mass[c] = m;
                s.phi[c] = m / s.ru[c].x;
            }
        }
    }
    const int cap = s.nl_cap;
    FOR_LIST(i, s.nl_count) {
        if (i >= cap) break;
        const int c = s.nl[i];
        bool any;
        const float m = s.mass[c] + gather_excess(s, c, any);
        s.mass[c] = m;
        s.flags[c] = T_IFC;
        s.phi[c] = m / s.ru[c].x;
    }
}

// Interface stencils of the current state with height-function labels (R-17e):
// a thread per interface cell. The input is the learned normal's: the fill
// levels of the 3x3x3 block (liquid 1, interface phi clamped to [0, 1], gas
// 0), stencil index (dx+1) + 3(dy+1) + 9(dz+1); a block with a wall or solid
// cell is not logged. The label follows the height-function method: along
// the axis a where the Parker-Youngs normal is largest (gas toward sign
// sg), the fill levels of the 3x3 columns of 7 cells centred on the cell's
// row sum to the heights eta(i, j) = sum - 7/2 of the surface above the
// column's centre plane, measured toward the gas; a column counts only if
// its liquid end cell is liquid and its gas end cell gas. With eta_u, eta_v
// the central differences and eta_uu, eta_vv, eta_uv the second ones, the
// normal toward the gas is (sg e_a - eta_u e_u - eta_v e_v) / |.| and the
// mean curvature, positive for a convex liquid body,
//   kappa = -(eta_uu (1 + eta_v^2) + eta_vv (1 + eta_u^2) - 2 eta_u eta_v eta_uv)
//           / (2 (1 + eta_u^2 + eta_v^2)^(3/2)).
// Written per logged cell: fill[27], target = (n, kappa), fd = (Parker-Youngs
// normal, 0) and the cell index, at slots taken in no fixed order; `found`
// counts every valid cell, the first `cap` of them are written.
// fill level (clamped, and raw in `raw`) and type of a neighbour; false
// beyond a wall face or at a solid cell
__device__ __forceinline__ bool fill_at(const Dev& s, int x, int y, int z, int dx, int dy, int dz, float& v, int& t,
                                        float& raw) {
    const long long nb = nbr(s, x, y, z, dx, dy, dz);
    if (nb < 0) return false;
    t = s.flags[nb] & TYPE_MASK;
    if (t == T_SOL) return false;
    raw = t == T_LIQ ? 1.f : (t == T_IFC ? s.phi[nb] : 0.f);
    v = fminf(fmaxf(raw, 0.f), 1.f);
    return true;
}

__global__ void k_log_stencils(Dev s, long long cap, float* fill, float4* target, float4* fd, int* cells,
                               unsigned long long* found) {
    const int count = min(*s.wl_count, s.wl_cap);
    const int stride = gridDim.x * blockDim.x;
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    for (int base = blockIdx.x * blockDim.x; base < count; base += stride) {
        const int i = base + threadIdx.x;
        bool ok = false;
        float in[27];
        float4 lab = make_float4(0.f, 0.f, 0.f, 0.f), pyn = lab;
        int c = -1;
        if (i < count) {
            c = s.wl[i];
            int x, y, z;
            coords(s, c, x, y, z);
            ok = true;
            float gx = 0.f, gy = 0.f, gz = 0.f;
#pragma unroll
            for (int q = 0; q < 27; ++q) {
                float v = 0.f, raw = 0.f;
                int t = 0;
                if (!fill_at(s, x, y, z, cx(q), cy(q), cz(q), v, t, raw)) ok = false;
                in[q] = v;
                // the Parker-Youngs gradient of the raw fill levels
                if (q != 13) {
                    const float w = nnz(q) == 1 ? 4.f : (nnz(q) == 2 ? 2.f : 1.f);
                    gx += w * cx(q) * raw;
                    gy += w * cy(q) * raw;
                    gz += w * cz(q) * raw;
                }
            }
            const float gl = sqrtf(gx * gx + gy * gy + gz * gz);
            if (!(gl > 0.f)) ok = false;
            if (ok) {
                pyn = make_float4(-gx / gl, -gy / gl, -gz / gl, 0.f);
                // the dominant axis from the gradient itself (ties: the lower axis)
                const float g[3] = {gx, gy, gz};
                const int a = (fabsf(gx) >= fabsf(gy) && fabsf(gx) >= fabsf(gz)) ? 0 : (fabsf(gy) >= fabsf(gz) ? 1 : 2);
                const int u = a == 0 ? 1 : 0, v = a == 2 ? 1 : 2;
                const int sg = g[a] < 0.f ? 1 : -1;   // the normal -grad points to the gas
                float eta[3][3];
                for (int iu = -1; iu <= 1 && ok; ++iu)
                    for (int iv = -1; iv <= 1 && ok; ++iv) {
                        float sum = 0.f;
                        for (int t = -3; t <= 3 && ok; ++t) {
                            int d[3] = {0, 0, 0};
                            d[u] = iu;
                            d[v] = iv;
                            d[a] = sg * t;
                            float f = 0.f, fr = 0.f;
                            int ty = 0;
                            if (!fill_at(s, x, y, z, d[0], d[1], d[2], f, ty, fr)) ok = false;
                            else if ((t == -3 && ty != T_LIQ) || (t == 3 && ty != T_GAS)) ok = false;
                            sum += f;
                        }
                        eta[iu + 1][iv + 1] = sum - 3.5f;
                    }
                if (ok) {
                    const float eu = 0.5f * (eta[2][1] - eta[0][1]), ev = 0.5f * (eta[1][2] - eta[1][0]);
                    const float euu = eta[2][1] - 2.f * eta[1][1] + eta[0][1];
                    const float evv = eta[1][2] - 2.f * eta[1][1] + eta[1][0];
                    const float euv = 0.25f * (eta[2][2] - eta[2][0] - eta[0][2] + eta[0][0]);
                    const float g2 = 1.f + eu * eu + ev * ev;
                    const float inv = rsqrtf(g2);
                    float m[3];
                    m[a] = sg * inv;
                    m[u] = -eu * inv;
                    m[v] = -ev * inv;
                    const float kap = -(euu * (1.f + ev * ev) + evv * (1.f + eu * eu) - 2.f * eu * ev * euv) /
                                      (2.f * g2 * sqrtf(g2));
                    lab = make_float4(m[0], m[1], m[2], kap);
                }
            }
        }
        // warp-aggregated slots
        const unsigned bal = __ballot_sync(full, ok);
        unsigned long long slot0 = 0;
        if (bal) {
            const int leader = __ffs(bal) - 1;
            if (lane == leader) slot0 = atomicAdd(found, (unsigned long long)__popc(bal));
            slot0 = __shfl_sync(full, slot0, leader);
        }
        if (ok) {
            const unsigned long long k = slot0 + __popc(bal & ((1u << lane) - 1u));
            if ((long long)k < cap) {
#pragma unroll
                for (int q = 0; q < 27; ++q) fill[k * 27 + q] = in[q];
                target[k] = lab;
                if (fd) fd[k] = pyn;
                if (cells) cells[k] = c;
            }
        }
    }
}

void launch_log_stencils(const Dev& s, long long cap, float* fill, float* target, float* fd, int* cells,
                         unsigned long long* found, cudaStream_t st) {
    cudaMemsetAsync(found, 0, sizeof(unsigned long long), st);
    k_log_stencils<<<LIST_BLOCKS, LIST_THREADS, 0, st>>>(s, cap, fill, reinterpret_cast<float4*>(target),
                                                          reinterpret_cast<float4*>(fd), cells, found);
}

int launch_normals(const Dev& s, float4* out, cudaStream_t st) { return normals_into(s, out, s.wl, s.wl_count, st); }

template <typename S>
static void launch_init_and_prep(const Dev& s, int last_parity, cudaStream_t st) {
    if (last_parity == 0) launch_after(k_init_and_prep<S, 0>, LIST_BLOCKS, LIST_THREADS, st, s);
    else launch_after(k_init_and_prep<S, 1>, LIST_BLOCKS, LIST_THREADS, st, s);
}

int launch_conversion(const Dev& s, int last_parity, cudaStream_t st) {
    k_candidates<<<LIST_BLOCKS, LIST_THREADS, 0, st>>>(s);
    launch_after(k_conflict, LIST_BLOCKS, LIST_THREADS, st, s);
    // the excess-mass weights need the normals of the converting cells only
    if (s.mlp) {
        normals_into(s, s.nrm1, s.cl, s.cl_count, st);
        launch_after(k_mark<false>, LIST_BLOCKS, LIST_THREADS, st, s);
    } else {
        launch_after(k_mark<true>, LIST_BLOCKS, LIST_THREADS, st, s);
    }
    if (s.storage == FSLBM_STORE_FP32) launch_init_and_prep<float>(s, last_parity, st);
    else if (s.storage == FSLBM_STORE_FP16) launch_init_and_prep<__half>(s, last_parity, st);
    else launch_init_and_prep<__nv_bfloat16>(s, last_parity, st);
    launch_after(k_finish_conversion, LIST_BLOCKS, LIST_THREADS, st, s);
    return s.mlp ? 6 : 5;
}

// ------------------------------------------------------------ work lists
// Block-aggregated append of the cells c0 + k for the set bits k of a
// thread's two 32-bit masks, ma to list la and mb to list lb: one scan of
// both counts (list a in the low 16 bits, list b in the high ones; a block
// holds at most 32 x 32 bits per warp), one atomic per list and block. The
// cells of a block keep their order in each list. List b takes whole groups
// of 32 entries per block, the last one filled up with -1: the link pass forms
// FP32 sums over 32 consecutive entries, and with whole groups they hold the
// same cells in the same order whichever block appends first (runs then repeat
// to the order of FP64 atomics). Every thread of the block must call it.
__device__ __forceinline__ void block_append_masks(const Dev& s, int c0, unsigned ma, int* la, int* ca, int capa,
                                                   unsigned mb, int* lb, int* cb, int capb) {
    __shared__ int warp_tot[32];
    __shared__ int base_a, base_b, total_b;
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int na = __popc(ma), nb = __popc(mb);
    int incl = na | (nb << 16);
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int t = __shfl_up_sync(full, incl, off);
        if (lane >= off) incl += t;
    }
    if (lane == 31) warp_tot[wid] = incl;
    __syncthreads();
    if (threadIdx.x == 0) {
        int ta = 0, tb = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
            const int c = warp_tot[w];
            warp_tot[w] = ta | (tb << 16);
            ta += c & 0xffff;
            tb += c >> 16;
        }
        base_a = ta ? atomicAdd(ca, ta) : 0;
        base_b = tb ? atomicAdd(cb, (tb + 31) & ~31) : 0;
        total_b = tb;
    }
    __syncthreads();
    const int pre = warp_tot[wid];
    int ka = base_a + (pre & 0xffff) + (incl & 0xffff) - na;
    int kb = base_b + (pre >> 16) + (incl >> 16) - nb;
    for (unsigned m = ma; m; m &= m - 1, ++ka) {
        if (ka < capa) la[ka] = c0 + __ffs(m) - 1;
        else set_error(s, ERR_CAPACITY);
    }
    for (unsigned m = mb; m; m &= m - 1, ++kb) {
        if (kb < capb) lb[kb] = c0 + __ffs(m) - 1;
        else set_error(s, ERR_CAPACITY);
    }
    const int pad = total_b + (int)threadIdx.x;   // (blocks have at least 32 threads)
    if (pad < ((total_b + 31) & ~31) && base_b + pad < capb) lb[base_b + pad] = -1;
    __syncthreads();
}

// Lists the interface cells and the solid cells with a liquid or interface
// cell among their 26 neighbours. A row has ceil(nx / 32) words of a bit per
// cell. First pass, a thread per word: the fluid, interface and solid bits of
// its cells, from two 16-byte loads, or where nx is not a multiple of 32 from
// nine aligned 4-byte loads shifted into place (the last word of a row is then
// partly empty). Second pass, a thread per word:
// the fluid words of the 3x3 rows around it, each widened by the halo bits of
// its x-neighbour words, are ORed, then ORed along x. (A thread per cell with
// up to 26 neighbour reads, the former way for the other lattices: 301x37x75
// 17.6 us and two memsets, with two passes 3.3 + 10.5; a box of 200x72x90 15.4,
// now 3.4 + 5.8.)
// four type bytes (gas 0, liquid 1, interface 2, solid 3 in the low two
// bits) to three 4-bit masks: fluid (1 or 2), interface, solid; the multiply
// gathers the bits at positions 0, 8, 16, 24 into bits 21..24
__device__ __forceinline__ void type_nibbles(unsigned v, unsigned& f, unsigned& i, unsigned& sl) {
    const unsigned a = v & 0x03030303u;
    const unsigned hi = a >> 1;
    auto pack = [](unsigned x) { return ((x * 0x00204081u) >> 21) & 0xFu; };
    f = pack((a ^ hi) & 0x01010101u);
    i = pack(hi & ~a & 0x01010101u);
    sl = pack(hi & a & 0x01010101u);
}

__host__ __device__ __forceinline__ long long type_words(const Dev& s) {
    return (long long)((s.nx + 31) >> 5) * s.ny * s.nz;
}

// (also clears the counts of the lists that the second pass fills)
__global__ void k_type_bits(Dev s) {
    after_previous();
    const long long w = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (w == 0) *s.wl_count = *s.sl_count = *s.bseg_count = 0;
    if (w >= type_words(s)) return;
    unsigned words[8], valid = 0xffffffffu;
    if ((s.nx & 31) == 0) {
        const uint4* src = reinterpret_cast<const uint4*>(s.flags + (w << 5));
        const uint4 a = src[0], b = src[1];
        words[0] = a.x; words[1] = a.y; words[2] = a.z; words[3] = a.w;
        words[4] = b.x; words[5] = b.y; words[6] = b.z; words[7] = b.w;
    } else {
        const unsigned nxw = ((unsigned)s.nx + 31u) >> 5, row = (unsigned)w / nxw, xw = (unsigned)w - row * nxw;
        const long long c0 = (long long)row * s.nx + 32 * xw, a0 = c0 & ~3LL;
        const int width = s.nx - 32 * (int)xw, sh = 8 * (int)(c0 & 3);
        if (width < 32) valid = (1u << width) - 1u;
        unsigned raw[9];   // (the last one may reach up to three bytes into the padding behind the flags)
#pragma unroll
        for (int k = 0; k < 9; ++k)
            raw[k] = a0 + 4 * k < s.n ? *reinterpret_cast<const unsigned*>(s.flags + a0 + 4 * k) : 0u;
#pragma unroll
        for (int k = 0; k < 8; ++k) words[k] = __funnelshift_r(raw[k], raw[k + 1], sh);
    }
    unsigned fm = 0, im = 0, sm = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        unsigned f, i, sl;
        type_nibbles(words[k], f, i, sl);
        fm |= f << (4 * k);
        im |= i << (4 * k);
        sm |= sl << (4 * k);
    }
    s.fbits[w] = fm & valid;
    s.ibits[w] = im & valid;
    s.sbits[w] = sm & valid;
    if (!s.tw || s.np == 0) return;
    // overlapping words of 2-bit types for the link pass, up to the cells
    // above the particles'
    const unsigned nxw = (unsigned)s.nx >> 5, row = (unsigned)w / nxw, xw = (unsigned)w - row * nxw;
    if (!s.per_z && (int)(row / (unsigned)s.ny) > *s.zmax_cell + 1) return;
    // four type bytes to one byte: bits 0, 8, 16, 24 to 24, 26, 28, 30
    auto pack = [](unsigned v) { return ((v & 0x03030303u) * 0x01041040u) >> 24; };
    unsigned lo = 0, hi = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        lo |= pack(words[k]) << (8 * k);
        hi |= pack(words[4 + k]) << (8 * k);
    }
    // the four cells before and behind (across the seam, or gas beyond a wall)
    const uint8_t* rf = s.flags + (long long)row * s.nx;
    const int xl = xw > 0 ? (int)(32 * xw) - 4 : (s.per_x ? s.nx - 4 : -1);
    const int xr = xw + 1 < nxw ? (int)(32 * xw) + 32 : (s.per_x ? 0 : -1);
    const unsigned L = xl >= 0 ? pack(*reinterpret_cast<const unsigned*>(rf + xl)) : 0u;
    const unsigned R = xr >= 0 ? pack(*reinterpret_cast<const unsigned*>(rf + xr)) : 0u;
    const uint4 out = make_uint4(L | (lo << 8), (lo >> 8) | (hi << 24), (lo >> 24) | (hi << 8), (hi >> 8) | (R << 24));
    *reinterpret_cast<uint4*>(s.tw + 4 * w) = out;
}

// The block of the classification that finishes last clamps the list counts
// to their capacities and, with spread, takes the mass pool's share per
// interface cell (k_pool_spread adds it). Every thread of the block calls it.
__device__ __forceinline__ void classify_last(const Dev& s, int spread) {
    if (threadIdx.x != 0) return;
    __threadfence();
    if (atomicAdd(s.cls_done, 1) != (int)gridDim.x - 1) return;
    __threadfence();
    *s.cls_done = 0;
    const int wl = min(__ldcg(s.wl_count), s.wl_cap);
    *s.wl_count = wl;
    *s.sl_count = min(__ldcg(s.sl_count), s.sl_cap);
    if (!spread) return;
    const double p = *s.pool;
    if (wl > 0 && p != 0.0) {
        *s.pool_share = p / (double)wl;
        *s.pool = 0.0;
    } else {
        *s.pool_share = 0.0;
    }
}

__global__ void k_classify_bits(Dev s, int spread) {
    after_previous();
    const long long w = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int nxw = (s.nx + 31) >> 5;               // words per row
    const long long nw = type_words(s);
    unsigned ifc_mask = 0, sol_mask = 0, sol = 0;
    if (w < nw) {
        sol = s.sbits[w];
        ifc_mask = s.ibits[w];
    }
    // the solid words' neighbourhood, only in warps that hold one; a lane's
    // x-neighbour words are its neighbour lanes' own, but for the warp's and
    // the rows' ends (27 words per lane, for every lane: 87 us on the large
    // flume, 71 us now; 17.6 -> 14.5 us at 1024x64x128)
    if (__any_sync(0xffffffffu, sol != 0)) {
        const unsigned full = 0xffffffffu;
        const int lane = threadIdx.x & 31;
        const unsigned wc = (unsigned)(w < nw ? w : nw - 1);
        const int xw = (int)(wc % (unsigned)nxw);
        const unsigned row = wc / (unsigned)nxw;
        const int y = (int)(row % (unsigned)s.ny), z = (int)(row / (unsigned)s.ny);
        // x-neighbour words (periodic wrap, or none beyond a wall face)
        const int xl = xw > 0 ? xw - 1 : (s.per_x ? nxw - 1 : -1);
        const int xr = xw < nxw - 1 ? xw + 1 : (s.per_x ? 0 : -1);
        // cells in the word, and the last one's bit of the word before it
        const int width = min(32, s.nx - 32 * xw), lbit = xw > 0 ? 31 : (s.nx - 1) & 31;
        const bool own_l = lane == 0 || xw == 0, own_r = lane == 31 || xw == nxw - 1 || w + 1 >= nw;
        unsigned cw[9], lw[9], rw[9];
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            const int yy = shift(y, k % 3 - 1, s.ny, s.per_y), zz = shift(z, k / 3 - 1, s.nz, s.per_z);
            const bool in = (yy | zz) >= 0;
            const unsigned* rb = s.fbits + (unsigned)(in ? zz * s.ny + yy : 0) * (unsigned)nxw;
            cw[k] = in ? rb[xw] : 0u;
            lw[k] = in && own_l && xl >= 0 ? rb[xl] : 0u;
            rw[k] = in && own_r && xr >= 0 ? rb[xr] : 0u;
        }
        unsigned long long orr = 0;   // bit 1 + k <-> x0 + k, bit 0 <-> x0 - 1, bit 1 + width <-> x0 + width
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            // the neighbour lanes' words: the row (y + dy, z + dz) of a lane in
            // the same row of words
            const unsigned l = __shfl_up_sync(full, cw[k], 1), r = __shfl_down_sync(full, cw[k], 1);
            orr |= ((unsigned long long)cw[k] << 1) | (unsigned long long)((own_l ? lw[k] : l) >> lbit & 1u) |
                   ((unsigned long long)((own_r ? rw[k] : r) & 1u) << (1 + width));
        }
        const unsigned long long nb = orr | (orr >> 1) | (orr << 1);   // bit 1 + k: fluid in the 3x3x3 block
        sol_mask = sol & (unsigned)(nb >> 1);
    }
    const int c0 = (s.nx & 31) == 0 ? (int)(w << 5) : (int)(w / nxw) * s.nx + 32 * (int)(w % nxw);
    block_append_masks(s, c0, ifc_mask, s.wl, s.wl_count, s.wl_cap, sol_mask, s.sl, s.sl_count, s.sl_cap);
    classify_last(s, spread);
}

// Bed segments, for particle links taken from the fluid side: a thread per
// BED_SEG-cell x-segment of a row flags it when one of its liquid cells has a
// solid cell among its 26 neighbours (the solid words of the 3x3 rows around
// it, dilated by one cell along x, ANDed with its liquid words) and lists it.
// Rows at or above zmax_cell hold no such cell (no particle reaches them).
__global__ void k_bed_segments(Dev s) {
    after_previous();
    constexpr int WPS = BED_SEG / 32;                // words per segment
    const long long sg = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int nxw = s.nx >> 5;
    const long long nseg = (long long)s.nsegx * s.ny * s.nz;
    bool bed = false;
    if (sg < nseg) {
        const long long row = sg / s.nsegx;
        const int xs = (int)(sg - row * s.nsegx);
        const int y = (int)(row % s.ny), z = (int)(row / s.ny);
        const int w0 = xs * WPS;
        const int nw = min(WPS, nxw - w0);
        unsigned liq[WPS];
        unsigned any = 0;
#pragma unroll
        for (int k = 0; k < WPS; ++k) {
            liq[k] = k < nw ? s.fbits[row * nxw + w0 + k] & ~s.ibits[row * nxw + w0 + k] : 0u;
            any |= liq[k];
        }
        if (any && (s.per_z || z < *s.zmax_cell)) {
            unsigned dil[WPS];
#pragma unroll
            for (int k = 0; k < WPS; ++k) dil[k] = 0u;
            for (int dz = -1; dz <= 1; ++dz) {
                const int zz = shift(z, dz, s.nz, s.per_z);
                if (zz < 0) continue;
                for (int dy = -1; dy <= 1; ++dy) {
                    const int yy = shift(y, dy, s.ny, s.per_y);
                    if (yy < 0) continue;
                    const long long rb = ((long long)zz * s.ny + yy) * nxw;
                    // word w0 + k for k in [-1, nw]: the x-halo wraps on a
                    // periodic x axis and is empty beyond a wall face
                    unsigned wv[WPS + 2];
#pragma unroll
                    for (int k = -1; k <= WPS; ++k) {
                        int xw = w0 + k;
                        if (k > nw) { wv[k + 1] = 0u; continue; }
                        if (xw < 0) xw = s.per_x ? nxw - 1 : -1;
                        else if (xw >= nxw) xw = s.per_x ? 0 : -1;
                        wv[k + 1] = xw >= 0 ? s.sbits[rb + xw] : 0u;
                    }
#pragma unroll
                    for (int k = 0; k < WPS; ++k)
                        dil[k] |= wv[k + 1] | (wv[k + 1] << 1) | (wv[k + 1] >> 1) | (wv[k] >> 31) | (wv[k + 2] << 31);
                }
            }
#pragma unroll
            for (int k = 0; k < WPS; ++k) bed |= (liq[k] & dil[k]) != 0u;
        }
        s.segflag[sg] = bed ? 1 : 0;
    }
    block_append(s, bed, (int)sg, s.bseg, s.bseg_count, (int)nseg);
}

// liquid cells with a gas neighbour (the separation the conversion rules keep)
__global__ void k_check_invariant(Dev s) {
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= s.n || (s.flags[c] & TYPE_MASK) != T_LIQ) return;
    int x, y, z;
    coords(s, c, x, y, z);
    for (int q = 0; q < 27; ++q) {
        if (q == 13) continue;
        const long long nb = nbr(s, x, y, z, cx(q), cy(q), cz(q));
        if (nb >= 0 && (s.flags[nb] & TYPE_MASK) == T_GAS) {
            atomicAdd(s.viol, 1ull);
            return;
        }
    }
}

void launch_check_invariant(const Dev& s, cudaStream_t st) {
    k_check_invariant<<<blocks_for(s.n, 256), 256, 0, st>>>(s);
}

int launch_classify(const Dev& s, bool spread, cudaStream_t st) {
    const long long words = type_words(s);
    launch_after(k_type_bits, blocks_for(words, 256), 256, st, s);
    launch_after(k_classify_bits, blocks_for(words, 128), 128, st, s, spread);
    int k = 2;
    if (s.links_fused) {
        launch_after(k_bed_segments, blocks_for((long long)s.nsegx * s.ny * s.nz, 128), 128, st, s);
        ++k;
    }
    return k;
}

__global__ void k_cell_counts(Dev s, unsigned long long* out) {
    __shared__ unsigned long long sh[4];
    if (threadIdx.x < 4) sh[threadIdx.x] = 0;
    __syncthreads();
    unsigned long long loc[4] = {0, 0, 0, 0};
    for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < s.n;
         c += (long long)gridDim.x * blockDim.x)
        loc[s.flags[c] & TYPE_MASK]++;
    for (int k = 0; k < 4; ++k) atomicAdd(&sh[k], loc[k]);
    __syncthreads();
    if (threadIdx.x < 4) atomicAdd(&out[threadIdx.x], sh[threadIdx.x]);
}

void launch_cell_counts(const Dev& s, unsigned long long* out, cudaStream_t st) {
    cudaMemsetAsync(out, 0, 4 * sizeof(unsigned long long), st);
    k_cell_counts<<<152 * 4, 256, 0, st>>>(s, out);
}

// ------------------------------------------------------------ mass pool
// the pool's share joins every interface cell; the conversion codes, left
// only on the cells k_conflict listed, are cleared
__global__ void k_pool_spread(Dev s) {
    after_previous();
    const int ncl = min(*s.cl_count, s.wl_cap);
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < ncl; i += gridDim.x * blockDim.x) s.conv[s.cl[i]] = 0;
    const double share = *s.pool_share;
    if (share == 0.0) return;
    FOR_LIST(i, s.wl_count) {
        const int c = s.wl[i];
        const float m = (float)((double)s.mass[c] + share);
        s.mass[c] = m;
        s.phi[c] = m / s.ru[c].x;
    }
}

int launch_pool_spread(const Dev& s, cudaStream_t st) {
    launch_after(k_pool_spread, LIST_BLOCKS, LIST_THREADS, st, s);
    return 1;
}

// ------------------------------------------------------------ initial state
__device__ __forceinline__ float clamp01(double v) { return (float)(v < 0 ? 0 : (v > 1 ? 1 : v)); }

__device__ void init_cell(const Dev& s, long long c, int t, double H, double fill) {
    int x, y, z;
    coords(s, c, x, y, z);
    s.flags[c] = (uint8_t)t;
    s.owner[c] = -1;
    s.conv[c] = 0;
    s.mass[c] = 0.f;
    s.phi[c] = 0.f;
    s.ru[c] = make_float4(0.f, 0.f, 0.f, 0.f);
    s.nrm[c] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (t == T_GAS) return;
    double rho = (double)s.rho_gas * exp(3.0 * fabs((double)s.gzd) * (H - (z + 0.5)));
    float f[27];
#pragma unroll
    for (int q = 0; q < 27; ++q) f[q] = (float)(wqd(q) * (rho - 1.0));
    store_fstar(s, c, 1, f);
    if (t == T_IFC)
        for (int q = 0; q < 27; ++q) st_any(s, s.fs, (long long)q * s.n + c, f[q]);
    s.ru[c] = make_float4((float)rho, 0.f, 0.f, 0.f);
    double m = rho * fill;
    s.mass[c] = (float)m;
    s.phi[c] = (float)(m / rho);
}

// flat surface at height H: fill(k) = clamp(H - k, 0, 1); interface where
// 0 < fill < 1 or where a full cell has gas directly above
__global__ void k_init_flat(Dev s, double H) {
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= s.n) return;
    int x, y, z;
    coords(s, c, x, y, z);
    double fk = H - z;
    fk = fk < 0 ? 0 : (fk > 1 ? 1 : fk);
    int t;
    if (fk == 0.0) t = T_GAS;
    else {
        bool above_gas;
        if (z + 1 < s.nz) {
            double fa = H - (z + 1);
            above_gas = fa <= 0.0;
        } else {
            above_gas = s.per_z ? (H <= 0.0) : false;
        }
        t = (fk < 1.0 || above_gas) ? T_IFC : T_LIQ;
    }
    init_cell(s, c, t, H, fk);
}

// surface height per column: gas where the fill is 0, liquid where it is 1
// and no 26-neighbour is gas, interface otherwise; solid cells are kept
__global__ void k_init_surface(Dev s, const double* Hxy) {
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= s.n) return;
    if ((s.flags[c] & TYPE_MASK) == T_SOL) return;
    int x, y, z;
    coords(s, c, x, y, z);
    const double H = Hxy[(long long)y * s.nx + x];
    double fk = H - z;
    fk = fk < 0 ? 0 : (fk > 1 ? 1 : fk);
    int t;
    if (fk == 0.0) t = T_GAS;
    else {
        bool gas_nb = false;
        for (int q = 0; q < 27; ++q) {
            if (q == 13) continue;
            long long nb = nbr(s, x, y, z, cx(q), cy(q), cz(q));
            if (nb < 0 || (s.flags[nb] & TYPE_MASK) == T_SOL) continue;
            int bx, by, bz;
            coords(s, nb, bx, by, bz);
            if (Hxy[(long long)by * s.nx + bx] - bz <= 0.0) gas_nb = true;
        }
        t = (fk < 1.0 || gas_nb) ? T_IFC : T_LIQ;
    }
    init_cell(s, c, t, H, fk);
}

// The flat start's values depend on z alone: the hydrostatic density of each
// z and its 27 stored deviations, by the expressions of init_cell, once per z.
__global__ void k_init_flat_table(Dev s, double H, double* rho_z, float* f_z) {
    const int z = blockIdx.x * blockDim.x + threadIdx.x;
    if (z >= s.nz) return;
    const double rho = (double)s.rho_gas * exp(3.0 * fabs((double)s.gzd) * (H - (z + 0.5)));
    rho_z[z] = rho;
#pragma unroll
    for (int q = 0; q < 27; ++q) f_z[27 * z + q] = (float)(wqd(q) * (rho - 1.0));
}

// k_init_flat from the per-z table, with 32-bit cell coordinates (n < 2^31):
// the same cell types and values without an FP64 exponential and 64-bit
// divisions per cell
__global__ void k_init_flat_tab(Dev s, double H, const double* rho_z, const float* f_z) {
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= s.n) return;
    int x, y, z;
    coords32(s, (int)c, x, y, z);
    double fk = H - z;
    fk = fk < 0 ? 0 : (fk > 1 ? 1 : fk);
    int t;
    if (fk == 0.0) t = T_GAS;
    else {
        bool above_gas;
        if (z + 1 < s.nz) {
            double fa = H - (z + 1);
            above_gas = fa <= 0.0;
        } else {
            above_gas = s.per_z ? (H <= 0.0) : false;
        }
        t = (fk < 1.0 || above_gas) ? T_IFC : T_LIQ;
    }
    s.flags[c] = (uint8_t)t;
    s.owner[c] = -1;
    s.conv[c] = 0;
    s.mass[c] = 0.f;
    s.phi[c] = 0.f;
    s.ru[c] = make_float4(0.f, 0.f, 0.f, 0.f);
    s.nrm[c] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (t == T_GAS) return;
    const double rho = rho_z[z];
    float f[27];
#pragma unroll
    for (int q = 0; q < 27; ++q) f[q] = f_z[27 * z + q];
#pragma unroll
    for (int q = 0; q < 27; ++q) st_any(s, s.f, fstar_slot(s, q, x, y, z, c, 1), f[q]);
    if (t == T_IFC)
        for (int q = 0; q < 27; ++q) st_any(s, s.fs, (long long)q * s.n + c, f[q]);
    s.ru[c] = make_float4((float)rho, 0.f, 0.f, 0.f);
    const double m = rho * fk;
    s.mass[c] = (float)m;
    s.phi[c] = (float)(m / rho);
}

void launch_init_flat(const Dev& s, double H, cudaStream_t st) {
    // the table lives for the two launches in the excess-mass normal field
    // (scratch between steps), which is zeroed again after them
    const size_t need = (size_t)s.nz * (sizeof(double) + 27 * sizeof(float));
    if (s.n < (1LL << 31) && need <= (size_t)s.n * sizeof(float4)) {
        double* rho_z = reinterpret_cast<double*>(s.nrm1);
        float* f_z = reinterpret_cast<float*>(rho_z + s.nz);
        k_init_flat_table<<<(s.nz + 127) / 128, 128, 0, st>>>(s, H, rho_z, f_z);
        k_init_flat_tab<<<blocks_for(s.n, 256), 256, 0, st>>>(s, H, rho_z, f_z);
        cudaMemsetAsync(s.nrm1, 0, need, st);
    } else {
        k_init_flat<<<blocks_for(s.n, 256), 256, 0, st>>>(s, H);
    }
}
void launch_init_surface(const Dev& s, const double* H, cudaStream_t st) {
    k_init_surface<<<blocks_for(s.n, 256), 256, 0, st>>>(s, H);
}

}  // namespace fsl

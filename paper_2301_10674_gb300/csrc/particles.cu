// Geometrically resolved spheres (Section 2.2): two-step averaging of the
// momentum-exchange force, DEM sub-steps (linear spring-dashpot contacts
// parameterised by the restitution coefficient and the collision time,
// tangential spring with Coulomb limit, walls, gravity; semi-implicit
// Newton-Euler), the particle grid, and the particle-to-cell map with the
// cells it covers and uncovers. Particle state and forces are FP64; the map
// test is evaluated in FP64 without fused multiply-add so that cell types do
// not depend on contraction choices.
#include <atomic>

#include "fslbm_dev.cuh"

namespace fsl {

// ------------------------------------------------------------ particle grid
__device__ __forceinline__ int gcoord(double v, double h, int g) {
    int k = (int)floor(v / h);
    return k < 0 ? 0 : (k >= g ? g - 1 : k);
}

__device__ __forceinline__ void grid_count(const Dev& s, int p) {
    int a = gcoord(s.X[3 * p], s.ghx, s.gnx);
    int b = gcoord(s.X[3 * p + 1], s.ghy, s.gny);
    int c = gcoord(s.X[3 * p + 2], s.ghz, s.gnz);
    int g = a + s.gnx * (b + s.gny * c);
    s.g_of[p] = g;
    atomicAdd(&s.g_count[g], 1);
}
__global__ void k_grid_count(Dev s) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < s.np) grid_count(s, p);
}

// exclusive scan of the grid counts by one block of 32 warps: warp w owns a
// contiguous chunk, read 32 counts at a time (coalesced); its total joins a
// scan of the 32 warp totals, then the warp scans its chunk from that offset
__global__ void __launch_bounds__(1024) k_grid_scan(Dev s, int G) {
    after_previous();
    __shared__ int wtot[32];
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rows = (G + 31) / 32;                    // rows of 32 counts
    const int per = (rows + 31) / 32;                  // rows per warp
    const int r0 = warp * per, r1 = min(rows, r0 + per);
    int sum = 0;
    for (int r = r0; r < r1; ++r) {
        const int i = 32 * r + lane;
        sum += i < G ? s.g_count[i] : 0;
    }
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(full, sum, o);
    if (lane == 0) wtot[warp] = sum;
    __syncthreads();
    if (warp == 0) {
        int v = wtot[lane];
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(full, v, o);
            if (lane >= o) v += u;
        }
        wtot[lane] = v - wtot[lane];                   // exclusive
    }
    __syncthreads();
    int run = wtot[warp];
    for (int r = r0; r < r1; ++r) {
        const int i = 32 * r + lane;
        const int c = i < G ? s.g_count[i] : 0;
        int v = c;
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(full, v, o);
            if (lane >= o) v += u;
        }
        if (i < G) {
            s.g_start[i] = run + v - c;
            s.g_cursor[i] = run + v - c;
        }
        run += __shfl_sync(full, v, 31);
    }
}

__device__ __forceinline__ void grid_fill(const Dev& s, int p) {
    s.g_list[atomicAdd(&s.g_cursor[s.g_of[p]], 1)] = p;
}
__global__ void k_grid_fill(Dev s) {
    after_previous();
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < s.np) grid_fill(s, p);
}

// particles of a grid cell in index order (deterministic summation order)
__device__ __forceinline__ void grid_sort(const Dev& s, int g) {
    int b = s.g_start[g], e = b + s.g_count[g];
    for (int i = b + 1; i < e; ++i) {
        int v = s.g_list[i];
        int j = i - 1;
        while (j >= b && s.g_list[j] > v) {
            s.g_list[j + 1] = s.g_list[j];
            --j;
        }
        s.g_list[j + 1] = v;
    }
}
__global__ void k_grid_sort(Dev s, int G) {
    after_previous();
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g < G) grid_sort(s, g);
}

// the lists from the counts
static int launch_grid_lists(const Dev& s, cudaStream_t st) {
    const int G = s.gnx * s.gny * s.gnz;
    launch_after(k_grid_scan, 1, 1024, st, s, G);
    launch_after(k_grid_fill, blocks_for(s.np, 128), 128, st, s);
    launch_after(k_grid_sort, blocks_for(G, 128), 128, st, s, G);
    return 3;
}
int launch_grid_build(const Dev& s, cudaStream_t st) {
    cudaMemsetAsync(s.g_count, 0, sizeof(int) * s.gnx * s.gny * s.gnz, st);
    k_grid_count<<<blocks_for(s.np, 128), 128, 0, st>>>(s);
    return 1 + launch_grid_lists(s, st);
}

// distinct grid coordinates within [k0, k1] along one axis
struct GRange {
    int v[3];
    int n;
};
__device__ __forceinline__ GRange grange(int k0, int k1, int g, int periodic) {
    GRange r;
    r.n = 0;
    if (periodic && k1 - k0 + 1 >= g) {
        for (int k = 0; k < g && r.n < 3; ++k) r.v[r.n++] = k;
        return r;
    }
    for (int k = k0; k <= k1 && r.n < 3; ++k) {
        int kk = k;
        if (kk < 0 || kk >= g) {
            if (!periodic) continue;
            kk = (kk % g + g) % g;
        }
        r.v[r.n++] = kk;
    }
    return r;
}

// ------------------------------------------------------------ DEM
// FP32 displacement d + f (integer and fraction parts) of the nearest image
// along a periodic axis (|d| <= L). The real displacement is wrapped: the
// integer part alone picks the farther image where it is half an even axis.
__device__ __forceinline__ float image_offset(int d, float f, int L, int periodic) {
    float e = (float)d + f;
    if (periodic) {
        const float h = 0.5f * (float)L;
        if (e > h) e = (float)(d - L) + f;
        else if (e < -h) e = (float)(d + L) + f;
    }
    return e;
}

// minimal image of a displacement along a periodic axis (|d| < 1.5 L)
__device__ __forceinline__ double wrapd(double d, int L, int periodic) {
    if (periodic) {
        const double h = 0.5 * L;
        if (d > h) d -= L;
        else if (d < -h) d += L;
    }
    return d;
}
__device__ __forceinline__ float wrapf(float d, int L, int periodic) {
    if (periodic) {
        const float h = 0.5f * L;
        if (d > h) d -= L;
        else if (d < -h) d += L;
    }
    return d;
}

// Contact arithmetic with every rounding spelled out (which product of a sum
// is fused into it), so that a sub-step gives the same bits in every kernel it
// is inlined in: a gap is the difference of numbers near 2 r, so a last-bit
// difference in a position is up to 5e-5 of a lubrication force, and two
// contractions of the same source would let runs drift apart by that.
__device__ __forceinline__ float dot_r(const float (&a)[3], const float (&b)[3]) {
    return __fmaf_rn(a[2], b[2], __fmaf_rn(a[0], b[0], __fmul_rn(a[1], b[1])));
}
__device__ __forceinline__ float det_r(float a, float b, float c, float d) {   // a b - c d
    return __fmaf_rn(a, b, -__fmul_rn(c, d));
}
__device__ __forceinline__ void cross_r(const float (&a)[3], const float (&b)[3], float (&o)[3]) {
    o[0] = det_r(a[1], b[2], a[2], b[1]);
    o[1] = det_r(a[2], b[0], a[0], b[2]);
    o[2] = det_r(a[0], b[1], a[1], b[0]);
}

// Lubrication corrections (Section 2.2): the paper augments the DEM with
// normal and tangential lubrication forces where a gap is too small for the
// lattice to resolve and gives no formula. These are the asymptotic
// resistances of two nearly touching spheres with effective radius R,
// normal 6 pi mu R^2 / h and tangential 6 pi mu R (8/15) ln(1 / h), each less
// its value at the resolved gap h_c = 2/3 cell, with h clamped at 1e-2.
constexpr float LUB_HC = 2.f / 3.f, LUB_HMIN = 1e-2f;
// force on the particle (n toward the partner or wall, vrel the relative
// velocity of the surfaces at the contact point) and its tangential part
__device__ __forceinline__ void lub_f(const Dev& s, float R, const float (&n)[3], float h, const float (&vrel)[3],
                                      float (&Fl)[3], float (&Ft)[3]) {
    const float hh = fmaxf(h, LUB_HMIN);
    const float vn = dot_r(vrel, n);
    const float k = 6.f * 3.14159265f * s.lub_mu_f * R;
    const float cn = k * R * (1.f / hh - 1.f / LUB_HC);
    const float ct = k * (8.f / 15.f) * logf(LUB_HC / hh);
    for (int a = 0; a < 3; ++a) {
        Ft[a] = __fmul_rn(-ct, __fmaf_rn(-vn, n[a], vrel[a]));
        Fl[a] = __fmaf_rn(__fmul_rn(-cn, vn), n[a], Ft[a]);
    }
}

// a partner of p for the neighbour list: surfaces within 3/4 cell
__device__ __forceinline__ bool dem_partner(const Dev& s, int p, int j, const float4& xri) {
    if (j == p) return false;
    const float4 xrj = s.Xr[j];
    const float ex = wrapf(xrj.x - xri.x, s.nx, s.per_x), ey = wrapf(xrj.y - xri.y, s.ny, s.per_y),
                ez = wrapf(xrj.z - xri.z, s.nz, s.per_z);
    const float reach = fabsf(xri.w) + fabsf(xrj.w) + 0.75f;
    return ex * ex + ey * ey + ez * ez <= reach * reach;
}

// Neighbour list of every mobile particle for the sub-steps of one LBM
// step: particles whose surfaces are within 3/4 cell (beyond the
// lubrication range; the motion within a step is far below the margin).
// With it the FP32 start of the sub-steps (R-25): per neighbour slot the
// partner's centre offset and radius, the pair's effective mass and the
// tangential spring carried over from the last step's list; per mobile
// particle the distances to the wall faces; and the values the particles
// publish to one another: zero change of position, velocity and angular
// velocity at the step's start.
// A warp per particle: lane t scans grid cell t of the (up to) 3x3x3 cells
// around the particle's, in the order (z, y, x) of the cells and of the
// particles within a cell; the accepted partners are compacted into the
// slots in that order (a warp prefix sum over the lanes' counts).
__global__ void k_dem_neighbours(Dev s) {
    __shared__ int found_s[4][NB_SLOTS];
    const unsigned full = 0xffffffffu;
    const int p = (int)(((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int lane = threadIdx.x & 31;
    if (p >= s.np) return;   // whole warps leave together
    int* found = found_s[threadIdx.x >> 5];
    const bool fixed = s.fixed[p] != 0;
    if (lane < 2) {
        // both buffers: a fixed particle's values stay as they are
        s.dem_x[lane][p] = make_float4(0.f, 0.f, 0.f, 0.f);
        s.dem_u[lane][p] = s.Uf[p];
        s.dem_w[lane][p] = s.Wf[p];
    } else if (lane == 2) {
        s.dem_du[p] = s.dem_dw[p] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    if (fixed) {
        if (lane == 0) s.nb_count[p] = 0;
        return;
    }
    // offsets from the integer part and the FP32 fraction of the centres
    // (exact integer differences, minimal image on periodic axes): exact to
    // FP32 rounding and antisymmetric between the two partners
    const int4 ip = s.Xi[p];
    const float4 fp = s.Xfr[p];
    if (lane == 0) {
        s.dem_wall[6 * p + 0] = (float)ip.x + fp.x;
        s.dem_wall[6 * p + 1] = (float)(s.nx - ip.x) - fp.x;
        s.dem_wall[6 * p + 2] = (float)ip.y + fp.y;
        s.dem_wall[6 * p + 3] = (float)(s.ny - ip.y) - fp.y;
        s.dem_wall[6 * p + 4] = (float)ip.z + fp.z;
        s.dem_wall[6 * p + 5] = (float)(s.nz - ip.z) - fp.z;
    }
    const float4 xri = s.Xr[p];
    const int g = s.g_of[p];
    const int ga = g % s.gnx, gb = (g / s.gnx) % s.gny, gc = g / (s.gnx * s.gny);
    const GRange ra = grange(ga - 1, ga + 1, s.gnx, s.per_x);
    const GRange rb = grange(gb - 1, gb + 1, s.gny, s.per_y);
    const GRange rc = grange(gc - 1, gc + 1, s.gnz, s.per_z);
    const int ncell = ra.n * rb.n * rc.n;
    int b = 0, e = 0;
    if (lane < ncell) {
        const int ia = lane % ra.n, ib = (lane / ra.n) % rb.n, ic = lane / (ra.n * rb.n);
        const int gg = ra.v[ia] + s.gnx * (rb.v[ib] + s.gny * rc.v[ic]);
        b = s.g_start[gg];
        e = b + s.g_count[gg];
    }
    int mine = 0;
    for (int k = b; k < e; ++k) mine += dem_partner(s, p, s.g_list[k], xri) ? 1 : 0;
    int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(full, incl, o);
        if (lane >= o) incl += t;
    }
    const int total = min(__shfl_sync(full, incl, 31), NB_SLOTS);
    if (lane == 31 && incl > NB_SLOTS) set_error(s, ERR_HISTORY);
    int slot = incl - mine;
    for (int k = b; k < e; ++k) {
        const int j = s.g_list[k];
        if (!dem_partner(s, p, j, xri)) continue;
        if (slot < NB_SLOTS) found[slot] = j;
        ++slot;
    }
    __syncwarp();
    // lane t: the old list's slot t, then the new list's
    const int oldn = s.nb_count[p];
    const long long row = (long long)p * NB_ITEMS;
    const int oj = lane < oldn ? s.nb[(long long)p * NB_SLOTS + lane] : -1;
    const float4 oxi = lane < oldn ? s.nb_xi[row + lane] : make_float4(0.f, 0.f, 0.f, 0.f);
    const int nj = lane < total ? found[lane] : -1;
    float4 xi = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int t = 0; t < oldn; ++t) {
        const int j = __shfl_sync(full, oj, t);
        const float a0 = __shfl_sync(full, oxi.x, t), a1 = __shfl_sync(full, oxi.y, t), a2 = __shfl_sync(full, oxi.z, t);
        if (nj == j) xi = make_float4(a0, a1, a2, 0.f);
    }
    if (nj >= 0) {
        const float4 cp = s.dem_c[p], cj = s.dem_c[nj];
        const int4 ij = s.Xi[nj];
        const float4 fj = s.Xfr[nj];
        s.nb[(long long)p * NB_SLOTS + lane] = nj;
        s.nb_d0[(long long)p * NB_SLOTS + lane] =
            make_float4(image_offset(ij.x - ip.x, fj.x - fp.x, s.nx, s.per_x),
                        image_offset(ij.y - ip.y, fj.y - fp.y, s.ny, s.per_y),
                        image_offset(ij.z - ip.z, fj.z - fp.z, s.nz, s.per_z), cj.x);
        xi.w = cp.y * cj.y / (cp.y + cj.y);
        s.nb_xi[row + lane] = xi;
    }
    if (lane == 0) s.nb_count[p] = total;
}

// FP32 copies of the particle state used by the lattice kernels
__device__ __forceinline__ void particle_copies(const Dev& s, int p) {
    const double X = s.X[3 * p], Y = s.X[3 * p + 1], Z = s.X[3 * p + 2];
    const double r = s.R[p];
    s.Xr[p] = make_float4((float)X, (float)Y, (float)Z, s.fixed[p] ? -(float)r : (float)r);
    const double fx = floor(X), fy = floor(Y), fz = floor(Z);
    s.Xi[p] = make_int4((int)fx, (int)fy, (int)fz, 0);
    s.Xfr[p] = make_float4((float)(X - fx), (float)(Y - fy), (float)(Z - fz), 0.f);
    s.Uf[p] = make_float4((float)s.U[3 * p], (float)s.U[3 * p + 1], (float)s.U[3 * p + 2], 0.f);
    s.Wf[p] = make_float4((float)s.W[3 * p], (float)s.W[3 * p + 1], (float)s.W[3 * p + 2], 0.f);
    s.dem_c[p] = make_float4((float)r, (float)s.M[p], (float)s.I[p], 0.f);
}
__global__ void k_particle_copies(Dev s) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < s.np) particle_copies(s, p);
}

void launch_particle_copies(const Dev& s, cudaStream_t st) {
    if (s.np > 0) k_particle_copies<<<blocks_for(s.np, 128), 128, 0, st>>>(s);
}

// FP32 linear spring-dashpot with tangential history (same law as above)
__device__ __forceinline__ void contact_f(const Dev& s, float meff, const float (&n)[3], float delta,
                                          const float (&vrel)[3], float (&xi)[3], float dts, float (&F)[3],
                                          float (&Ft)[3]) {
    const float kn = meff * s.kn_f;
    const float dn = meff * s.dn_f;
    const float kt = kn * s.kt_f;
    const float dt_ = dn;
    const float vn = dot_r(vrel, n);
    const float vt[3] = {__fmaf_rn(-vn, n[0], vrel[0]), __fmaf_rn(-vn, n[1], vrel[1]), __fmaf_rn(-vn, n[2], vrel[2])};
    const float fn = __fmaf_rn(kn, delta, __fmul_rn(dn, vn));
    float x[3] = {xi[0], xi[1], xi[2]};
    const float xn = dot_r(x, n);
    for (int a = 0; a < 3; ++a) x[a] = __fmaf_rn(vt[a], dts, __fmaf_rn(-xn, n[a], x[a]));
    for (int a = 0; a < 3; ++a) Ft[a] = __fmaf_rn(-kt, x[a], -__fmul_rn(dt_, vt[a]));
    const float ftl = sqrtf(dot_r(Ft, Ft));
    const float lim = s.friction_f * fabsf(fn);
    if (ftl > lim && ftl > 0.f) {
        const float sc = lim / ftl;
        for (int a = 0; a < 3; ++a) {
            Ft[a] = __fmul_rn(Ft[a], sc);
            x[a] = -__fadd_rn(Ft[a], __fmul_rn(dt_, vt[a])) / kt;
        }
    }
    for (int a = 0; a < 3; ++a) {
        xi[a] = x[a];
        F[a] = __fmaf_rn(-fn, n[a], Ft[a]);
    }
}

// One DEM sub-step of particle p by the DEM_LANES lanes of a group (l: the
// lane in the group, gm: the group's lanes), in FP32 (R-25): a particle's
// position, velocity and angular velocity are its FP64 state at the step's
// start plus the changes dx, du, dw the sub-steps have made (small numbers,
// exact to FP32 rounding of themselves); the offset to a partner is the start
// offset plus the difference of their dx, a wall distance the start distance
// plus or minus dx. The particles publish dx, u and w (buffers a read, b
// written). Lane l takes neighbour slots l, l + DEM_LANES, ... and then wall
// face l; the lanes pass their forces through shared memory, and lane c < 6
// adds component c of force and torque in the order of the slots (the order of
// one thread walking them, so the result is that thread's); lanes 0 to 2 then
// advance the velocity and position, lanes 3 to 5 the angular velocity, one
// axis each (semi-implicit Euler on the changes). The first sub-step averages
// the hydrodynamic force over two steps, the last adds the changes to the
// FP64 state, forms the FP32 copies and counts the particle in its grid cell.
// Bound by latency: a thread per particle ran its dozen partners one after
// the other (about 3000 dependent instructions, 18 to 21 us a sub-step whatever
// the particle count), and searched its 16 spring slots for every contact. Eight
// lanes per particle with the spring stored beside the partner's slot: 9.7 us
// for 4 712 particles (19.2 before), 16.5 us for 30 696 (21.4).
constexpr int DEM_LANES = 8;
static_assert(NB_SLOTS % DEM_LANES == 0 && NB_ITEMS == NB_SLOTS + DEM_LANES, "one wall face per lane");

// per lane group: 8 lanes of lubrication force and torque, contact force and
// torque (12 floats); the group stride keeps a warp's four groups on distinct banks
constexpr int DEM_SH = 104;

// What a lane group needs of its particle's lists, from global memory
struct GlobalLists {
    const Dev& s;
    long long p;
    int a;     // buffer of the published values
    __device__ __forceinline__ void slot(int k, float4& d0, float4& xi, float4& xj, float4& uj, float4& wj) const {
        const int j = s.nb[p * NB_SLOTS + k];
        d0 = s.nb_d0[p * NB_SLOTS + k];
        xi = s.nb_xi[p * NB_ITEMS + k];
        xj = s.dem_x[a][j];
        uj = s.dem_u[a][j];
        wj = s.dem_w[a][j];
    }
    __device__ __forceinline__ float4 spring(int k) const { return s.nb_xi[p * NB_ITEMS + k]; }
    __device__ __forceinline__ void set_spring(int k, float4 v) const { s.nb_xi[p * NB_ITEMS + k] = v; }
};

// The outer force (lanes 0-2) or torque (lanes 3-5) along the lane's axis of
// particle p: two-step average of the hydrodynamic force, plus the weight
__device__ __forceinline__ float dem_outer(const Dev& s, int p, int l, bool have_prev) {
    const bool trans = l < 3;
    const int ax = trans ? l : l - 3, k = 3 * p + ax;
    const double now = (trans ? s.Fh : s.Th)[k];
    double* prev = (trans ? s.Fp : s.Tp) + k;
    const double avg = have_prev ? 0.5 * (now + *prev) : now;
    *prev = now;
    const double g = ax == 0 ? s.gxd : (ax == 1 ? s.gyd : s.gzd);
    return (float)(trans ? avg + s.M[p] * g : avg);
}

// Adds the contact and lubrication forces of one sub-step to the lanes'
// components acc
template <class Lists>
__device__ __forceinline__ void dem_forces(const Dev& s, float* sh, const Lists& lists, int l, unsigned gm, int nbc,
                                           const float4& cp, const float4& xa4, const float4& ua4, const float4& wa4,
                                           float wall_d, float dts, float& acc) {
    const float rif = cp.x;
    const float arm = l < 3 ? 1.f : rif;   // torque: r n x F_t, the lanes' n x F_t times r
    int touching = 0;
    const int nround = (nbc + DEM_LANES - 1) / DEM_LANES;   // rounds of neighbours, then one of wall faces
#pragma unroll 1
    for (int r = 0; r <= nround; ++r) {
        const bool wall = r == nround;
        const int slot = wall ? NB_SLOTS + l : r * DEM_LANES + l;
        bool lub = false, touch = false;
        float n[3] = {0.f, 0.f, 0.f}, delta = 0.f, rj = 0.f;
        float4 uj = make_float4(0.f, 0.f, 0.f, 0.f), wj = uj, xi4 = uj;
        if (!wall) {
            if (slot < nbc) {
                float4 d0, xj;
                lists.slot(slot, d0, xi4, xj, uj, wj);
                rj = d0.w;
                const float d[3] = {d0.x + (xj.x - xa4.x), d0.y + (xj.y - xa4.y), d0.z + (xj.z - xa4.z)};
                const float dist2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
                const float rs = rif + rj;
                touch = dist2 < rs * rs;
                lub = s.lub && dist2 < (rs + LUB_HC) * (rs + LUB_HC);
                const float dist = sqrtf(dist2);
                const float inv = 1.f / dist;
#pragma unroll
                for (int k = 0; k < 3; ++k) n[k] = d[k] * inv;
                delta = rs - dist;
            }
        } else if (l < 6) {
            const int wx = l >> 1;
            if (!(wx == 0 ? s.per_x : (wx == 1 ? s.per_y : s.per_z))) {
                const float dxa = wx == 0 ? xa4.x : (wx == 1 ? xa4.y : xa4.z);
                const float dist = (l & 1) ? wall_d - dxa : wall_d + dxa;
                delta = rif - dist;
                touch = delta > 0.f;
                lub = s.lub && -delta < LUB_HC;
                const float sg = (l & 1) ? 1.f : -1.f;
#pragma unroll
                for (int k = 0; k < 3; ++k) n[k] = k == wx ? sg : 0.f;
                xi4 = lists.spring(slot);
                xi4.w = cp.y;   // the wall's mass is infinite
            }
        }
        // a partner not touched in this sub-step loses its spring
        if (!touch && (xi4.x != 0.f || xi4.y != 0.f || xi4.z != 0.f))
            lists.set_spring(slot, make_float4(0.f, 0.f, 0.f, xi4.w));
        if (!__any_sync(gm, lub || touch)) continue;   // nothing to add in this round
        float Fl[3] = {0.f, 0.f, 0.f}, Fc[3] = {0.f, 0.f, 0.f}, tl[3] = {0.f, 0.f, 0.f}, tc[3] = {0.f, 0.f, 0.f};
        if (lub || touch) {
            // (the second two slots of every four fuse the partner's product: the
            // rounding that a loop unrolled over four of them had)
            const bool sw = (slot & 2) != 0;
            const float wa[3] = {wa4.x, wa4.y, wa4.z}, wb[3] = {wj.x, wj.y, wj.z};
            float wsum[3], wn[3];
#pragma unroll
            for (int k = 0; k < 3; ++k)
                wsum[k] = sw ? __fmaf_rn(rj, wb[k], __fmul_rn(rif, wa[k])) : __fmaf_rn(rif, wa[k], __fmul_rn(rj, wb[k]));
            cross_r(wsum, n, wn);
            const float vrel[3] = {ua4.x - uj.x + wn[0], ua4.y - uj.y + wn[1], ua4.z - uj.z + wn[2]};
            float Ft[3];
            if (lub) {
                lub_f(s, wall ? rif : rif * rj / (rif + rj), n, -delta, vrel, Fl, Ft);
                cross_r(n, Ft, tl);
            }
            if (touch) {
                float xi[3] = {xi4.x, xi4.y, xi4.z};
                contact_f(s, xi4.w, n, delta, vrel, xi, dts, Fc, Ft);
                lists.set_spring(slot, make_float4(xi[0], xi[1], xi[2], xi4.w));
                cross_r(n, Ft, tc);
            }
        }
        touching += touch ? 1 : 0;
        float4* mine = reinterpret_cast<float4*>(sh + 12 * l);
        mine[0] = make_float4(Fl[0], Fl[1], Fl[2], tl[0]);
        mine[1] = make_float4(tl[1], tl[2], Fc[0], Fc[1]);
        mine[2] = make_float4(Fc[2], tc[0], tc[1], tc[2]);
        __syncwarp(gm);
        if (l < 6) {
#pragma unroll
            for (int t = 0; t < DEM_LANES; ++t) {
                acc = fmaf(arm, sh[12 * t + l], acc);
                acc = fmaf(arm, sh[12 * t + 6 + l], acc);
            }
        }
        __syncwarp(gm);
    }
#pragma unroll
    for (int o = 1; o < DEM_LANES; o <<= 1) touching += __shfl_xor_sync(gm, touching, o);
    if (touching > HIST_SLOTS && l == 0) set_error(s, ERR_HISTORY);
}

// The FP64 state of the step's end of a mobile particle (positions wrapped on
// periodic axes), its FP32 copies and its grid cell, from the lanes' changes
// of position (dx, lanes 0-2) and velocity (dv, lanes 0-5)
__device__ __forceinline__ void dem_finish(const Dev& s, int p, int l, unsigned gm, float dx, float dv) {
    const bool trans = l < 3;
    const int ax = trans ? l : l - 3;
    int g = 0;
    if (trans) {
        const int L = l == 0 ? s.nx : (l == 1 ? s.ny : s.nz);
        double x = s.X[3 * p + l] + (double)dx;
        if (l == 0 ? s.per_x : (l == 1 ? s.per_y : s.per_z)) x = x < 0.0 ? x + L : (x >= L ? x - L : x);
        s.X[3 * p + l] = x;
        const double fl = floor(x);
        reinterpret_cast<float*>(s.Xr + p)[l] = (float)x;
        reinterpret_cast<int*>(s.Xi + p)[l] = (int)fl;
        reinterpret_cast<float*>(s.Xfr + p)[l] = (float)(x - fl);
        if (l == 2) atomicMax(s.zmax_cell, (int)ceil(x + s.R[p]) + 2);
        g = l == 0 ? gcoord(x, s.ghx, s.gnx)
                   : (l == 1 ? s.gnx * gcoord(x, s.ghy, s.gny) : s.gnx * s.gny * gcoord(x, s.ghz, s.gnz));
    }
    if (l < 6) {
        double* v = (trans ? s.U : s.W) + 3 * p + ax;
        const double vn = *v + (double)dv;
        *v = vn;
        reinterpret_cast<float*>((trans ? s.Uf : s.Wf) + p)[ax] = (float)vn;
    }
    g += __shfl_xor_sync(gm, g, 1);
    g += __shfl_xor_sync(gm, g, 2);
    if (l == 0) {
        s.g_of[p] = g;
        atomicAdd(&s.g_count[g], 1);
    }
}
// a fixed particle: the top of the particle cells and the grid count it too
__device__ __forceinline__ void dem_finish_fixed(const Dev& s, int p, int l) {
    if (l != 0) return;
    atomicMax(s.zmax_cell, (int)ceil(s.X[3 * p + 2] + s.R[p]) + 2);
    atomicAdd(&s.g_count[s.g_of[p]], 1);
}

// one sub-step; the first of several also clears what the last one counts
__global__ void __launch_bounds__(128) k_dem_substep(Dev s, int a, int have_prev, int G, float dts, int first,
                                                     int last) {
    __shared__ __align__(16) float sh[128 / DEM_LANES * DEM_SH];
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (first && !last) {
        for (int g = t; g < G; g += gridDim.x * blockDim.x) s.g_count[g] = 0;
        if (t == 0) *s.zmax_cell = 0;
    }
    const int p = t / DEM_LANES, l = t % DEM_LANES, b = 1 - a;
    const unsigned gm = ((1u << DEM_LANES) - 1u) << ((threadIdx.x & 31) / DEM_LANES * DEM_LANES);
    if (p >= s.np) return;                    // whole groups leave together
    if (s.fixed[p]) {
        if (last) dem_finish_fixed(s, p, l);
        return;
    }
    const float4 cp = s.dem_c[p];
    const float4 xa4 = s.dem_x[a][p], ua4 = s.dem_u[a][p], wa4 = s.dem_w[a][p];
    const bool trans = l < 3;                 // lanes 0-2: velocity and position, 3-5: angular velocity
    const int ax = trans ? l : l - 3;         // (lanes 6 and 7 hold no component)
    float acc = 0.f;                          // the lane's component of force or torque
    if (l < 6) {
        float* outer = (trans ? s.Faf : s.Taf) + 3 * p + ax;
        if (first) *outer = acc = dem_outer(s, p, l, have_prev != 0);
        else acc = *outer;
    }
    const float wall_d = l < 6 ? s.dem_wall[6 * p + l] : 0.f;
    dem_forces(s, sh + threadIdx.x / DEM_LANES * DEM_SH, GlobalLists{s, p, a}, l, gm, s.nb_count[p], cp, xa4, ua4, wa4,
               wall_d, dts, acc);
    float v0 = 0.f, dv = 0.f;    // velocity component at the step's start, and its change
    if (l < 6) {
        const float4 v4 = trans ? s.Uf[p] : s.Wf[p];
        v0 = ax == 0 ? v4.x : (ax == 1 ? v4.y : v4.z);
        dv = reinterpret_cast<const float*>((trans ? s.dem_du : s.dem_dw) + p)[ax];
        dv = dv + dts * acc * (1.f / (trans ? cp.y : cp.z));
    }
    const float dxn = (ax == 0 ? xa4.x : (ax == 1 ? xa4.y : xa4.z)) + dts * (v0 + dv);   // (lanes 0-2)
    __syncwarp(gm);   // every lane has read the copies Uf and Wf
    if (last) {
        dem_finish(s, p, l, gm, dxn, dv);
    } else if (l < 6) {
        reinterpret_cast<float*>((trans ? s.dem_du : s.dem_dw) + p)[ax] = dv;
        reinterpret_cast<float*>((trans ? s.dem_u : s.dem_w)[b] + p)[ax] = v0 + dv;
        if (trans) reinterpret_cast<float*>(s.dem_x[b] + p)[ax] = dxn;
    }
}

// The sub-steps of a step and the particle grid in one thread-block cluster,
// for up to DEM_CLUSTER_MAX particles: the cluster's hardware barrier
// (release at arrival, acquire at the wait) stands between the phases that
// read other particles' values, so nothing is launched between the sub-steps.
// A lane group keeps its particle's lists and springs in shared memory and its
// constants in registers for the whole step, and reads its partners' published
// values from the shared memory of the CTA that owns them: with all of it in
// global memory a sub-step waited for six L2 latencies in turn. The whole DEM
// half (ten sub-steps and the grid) took 40 us for 34 particles (54 us with the
// lists in global memory) and 78 us for 1 008 in eight CTAs of 1 024 threads
// (114 us with 512 threads and two particles per group, whose fewer warps left
// each waiting for its own arithmetic), against ten launches of 9 us plus three
// of the grid. 16 CTAs leave a scheduler half the warps: 301x37x75 flume, step
// 0.1465 -> 0.137 ms; 768x40x96 (1 500 particles, separate launches before) 0.226
// -> 0.2195 ms.
constexpr int DEM_CLUSTER_CTAS = 16;       // where the device can place a cluster of 16, else 8
constexpr int DEM_CLUSTER_MAX = DEM_CLUSTER_CTAS * 1024 / DEM_LANES;

// (not the .aligned forms, which a warp must execute together: the lane groups
// of a warp come from loops of different lengths)
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ unsigned cluster_address(const void* p, unsigned rank) {
    unsigned r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                 : "=r"(r)
                 : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank));
    return r;
}
__device__ __forceinline__ float4 cluster_load(unsigned address) {
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"(address)
                 : "memory");
    return v;
}

// shared memory per particle of a CTA: published values (x, u, w; two
// buffers), list offsets and springs, partners' addresses
struct ClusterParticle {
    float4 pub[2][3];
    float4 d0[NB_SLOTS];
    float4 xi[NB_ITEMS];
    unsigned at[NB_SLOTS];      // cluster address of the partner's ClusterParticle
};
struct ClusterLists {
    ClusterParticle& me;
    int a;
    __device__ __forceinline__ void slot(int k, float4& d0, float4& xi, float4& xj, float4& uj, float4& wj) const {
        const unsigned at = me.at[k] + (unsigned)a * 3u * (unsigned)sizeof(float4);
        xj = cluster_load(at);
        uj = cluster_load(at + (unsigned)sizeof(float4));
        wj = cluster_load(at + 2u * (unsigned)sizeof(float4));
        d0 = me.d0[k];
        xi = me.xi[k];
    }
    __device__ __forceinline__ float4 spring(int k) const { return me.xi[k]; }
    __device__ __forceinline__ void set_spring(int k, float4 v) const { me.xi[k] = v; }
};

template <int THREADS>
__global__ void __launch_bounds__(THREADS) k_dem_cluster(Dev s, int have_prev, int G, float dts) {
    extern __shared__ __align__(16) unsigned char cluster_smem[];
    __shared__ int wtot[THREADS / 32];
    const int nt = gridDim.x * blockDim.x, tid = blockIdx.x * blockDim.x + threadIdx.x;   // one cluster: the grid
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const unsigned full = 0xffffffffu;
    const int l = tid % DEM_LANES, gpc = blockDim.x / DEM_LANES, lg = threadIdx.x / DEM_LANES;   // groups per CTA, local group
    const unsigned gm = ((1u << DEM_LANES) - 1u) << (lane / DEM_LANES * DEM_LANES);
    ClusterParticle* parts = reinterpret_cast<ClusterParticle*>(cluster_smem);      // [gpc]
    float* sh = reinterpret_cast<float*>(parts + gpc) + lg * DEM_SH;
    const bool trans = l < 3;
    const int ax = trans ? l : l - 3;
    const int p = tid / DEM_LANES;
    const bool mobile = p < s.np && s.fixed[p] == 0;
    ClusterParticle& me = parts[lg];
    int nbc = 0;
    float4 cp = make_float4(0.f, 0.f, 0.f, 0.f);
    float outer = 0.f, v0 = 0.f, dv = 0.f, wall_d = 0.f;
    if (p < s.np && l < 6) me.pub[l & 1][l >> 1] = l < 2 ? s.dem_x[0][p] : (l < 4 ? s.Uf[p] : s.Wf[p]);
    if (mobile) {
        nbc = s.nb_count[p];
        cp = s.dem_c[p];
        for (int k = l; k < nbc; k += DEM_LANES) {
            const int j = s.nb[(long long)p * NB_SLOTS + k];
            me.d0[k] = s.nb_d0[(long long)p * NB_SLOTS + k];
            me.xi[k] = s.nb_xi[(long long)p * NB_ITEMS + k];
            me.at[k] = cluster_address(&parts[j % gpc].pub[0][0], (unsigned)(j / gpc));
        }
        me.xi[NB_SLOTS + l] = s.nb_xi[(long long)p * NB_ITEMS + NB_SLOTS + l];
        if (l < 6) {
            outer = dem_outer(s, p, l, have_prev != 0);
            const float4 v4 = trans ? s.Uf[p] : s.Wf[p];
            v0 = ax == 0 ? v4.x : (ax == 1 ? v4.y : v4.z);
            wall_d = s.dem_wall[6 * p + l];
        }
    }
    for (int g = tid; g < G; g += nt) s.g_count[g] = 0;
    if (tid == 0) *s.zmax_cell = 0;
    cluster_barrier();
    for (int k = 0; k < s.dem_substeps; ++k) {
        const int a = k & 1, b = 1 - a;
        if (mobile) {
            const float4 xa4 = me.pub[a][0], ua4 = me.pub[a][1], wa4 = me.pub[a][2];
            float acc = outer;
            dem_forces(s, sh, ClusterLists{me, a}, l, gm, nbc, cp, xa4, ua4, wa4, wall_d, dts, acc);
            if (l < 6) dv = dv + dts * acc * (1.f / (trans ? cp.y : cp.z));
            const float dxn = (ax == 0 ? xa4.x : (ax == 1 ? xa4.y : xa4.z)) + dts * (v0 + dv);   // (lanes 0-2)
            if (k == s.dem_substeps - 1) {
                dem_finish(s, p, l, gm, dxn, dv);
            } else if (l < 6) {
                reinterpret_cast<float*>(&me.pub[b][trans ? 1 : 2])[ax] = v0 + dv;
                if (trans) reinterpret_cast<float*>(&me.pub[b][0])[ax] = dxn;
            }
        }
        cluster_barrier();
    }
    if (mobile) {
        // the springs go back to the lists
        for (int k = l; k < nbc; k += DEM_LANES) s.nb_xi[(long long)p * NB_ITEMS + k] = me.xi[k];
        s.nb_xi[(long long)p * NB_ITEMS + NB_SLOTS + l] = me.xi[NB_SLOTS + l];
    } else if (p < s.np) {
        dem_finish_fixed(s, p, l);
    }
    cluster_barrier();
    // exclusive scan of the grid counts: each CTA scans a contiguous run of
    // rows of 32 counts, a warp a part of it; the CTAs' totals pass through g_tot
    const int rows = (G + 31) / 32;
    const int cper = (rows + gridDim.x - 1) / gridDim.x;
    const int c0 = blockIdx.x * cper, c1 = min(rows, c0 + cper);
    const int per = (cper + nw - 1) / nw;
    const int r0 = min(c1, c0 + warp * per), r1 = min(c1, r0 + per);
    int sum = 0;
    for (int r = r0; r < r1; ++r) {
        const int i = 32 * r + lane;
        sum += i < G ? s.g_count[i] : 0;
    }
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(full, sum, o);
    if (lane == 0) wtot[warp] = sum;
    __syncthreads();
    if (threadIdx.x == 0) {
        int t = 0;
        for (int w = 0; w < nw; ++w) t += wtot[w];
        s.g_tot[blockIdx.x] = t;
    }
    cluster_barrier();
    int run = 0;
    for (int c = 0; c < (int)blockIdx.x; ++c) run += s.g_tot[c];
    for (int w = 0; w < warp; ++w) run += wtot[w];
    for (int r = r0; r < r1; ++r) {
        const int i = 32 * r + lane;
        const int c = i < G ? s.g_count[i] : 0;
        int v = c;
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(full, v, o);
            if (lane >= o) v += u;
        }
        if (i < G) {
            s.g_start[i] = run + v - c;
            s.g_cursor[i] = run + v - c;
        }
        run += __shfl_sync(full, v, 31);
    }
    cluster_barrier();
    for (int q = tid; q < s.np; q += nt) grid_fill(s, q);
    cluster_barrier();
    for (int g = tid; g < G; g += nt) grid_sort(s, g);
}

// ------------------------------------------------------------ particle map
__device__ __forceinline__ double map_metric(double kx, double ky, double kz, const double* Xp, double r) {
    // ((dx^2 + dy^2) + dz^2) - r^2, rounded step by step (no contraction)
    double dx = __dsub_rn(kx, Xp[0]);
    double dy = __dsub_rn(ky, Xp[1]);
    double dz = __dsub_rn(kz, Xp[2]);
    double s2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
    return __dsub_rn(s2, __dmul_rn(r, r));
}

// unwrapped cell-centre coordinate of the periodic image nearest to X
__device__ __forceinline__ double image_centre(int k, double X, int L, int periodic) {
    double c = k + 0.5;
    if (periodic) {
        if (c - X > 0.5 * L) c = (k - L) + 0.5;
        else if (X - c > 0.5 * L) c = (k + L) + 0.5;
    }
    return c;
}

// grid coordinates along one axis that particles covering cell k can have:
// those of [k + 1/2 - r_max, k + 1/2 + r_max], in FP32 with a margin above its
// rounding (the division in FP64 cost more than all the rest of a cell's
// map; a grid cell too many only adds candidates). Grid cells are at least
// 2 r_max + 1 wide, so the range holds two of them (three for very large radii).
__device__ __forceinline__ GRange cover_range(int k, double r_max, double h, int g, int periodic) {
    const float inv = 1.f / (float)h, c = (float)k + 0.5f, r = (float)r_max;
    const float eps = 1e-3f + 4e-7f * (float)g;
    return grange((int)floorf((c - r) * inv - eps), (int)floorf((c + r) * inv + eps), g, periodic);
}

// best covering particle (lowest metric, then lowest index) among the
// particles of the selected kind near cell (x, y, z)
__device__ void best_cover(const Dev& s, int x, int y, int z, int want_fixed, double& best, int& bestp) {
    const double xc = x + 0.5, yc = y + 0.5, zc = z + 0.5;
    const GRange ra = cover_range(x, s.r_max, s.ghx, s.gnx, s.per_x);
    const GRange rb = cover_range(y, s.r_max, s.ghy, s.gny, s.per_y);
    const GRange rc = cover_range(z, s.r_max, s.ghz, s.gnz, s.per_z);
    for (int ic = 0; ic < rc.n; ++ic)
        for (int ib = 0; ib < rb.n; ++ib)
            for (int ia = 0; ia < ra.n; ++ia) {
                int gg = ra.v[ia] + s.gnx * (rb.v[ib] + s.gny * rc.v[ic]);
                int b = s.g_start[gg], e = b + s.g_count[gg];
                for (int k = b; k < e; ++k) {
                    int p = s.g_list[k];
                    const float4 xr = s.Xr[p];
                    if ((xr.w < 0.f) != (want_fixed != 0)) continue;
                    // cheap reject in FP32 with a margin far above its rounding
                    float fx = (float)xc - xr.x, fy = (float)yc - xr.y, fz = (float)zc - xr.z;
                    if (s.per_x) fx -= (float)s.nx * rintf(fx / (float)s.nx);
                    if (s.per_y) fy -= (float)s.ny * rintf(fy / (float)s.ny);
                    if (s.per_z) fz -= (float)s.nz * rintf(fz / (float)s.nz);
                    const float d2 = fx * fx + fy * fy + fz * fz;
                    const float rr = fabsf(xr.w);
                    if (d2 > rr * rr + 1e-2f * (1.f + rr * rr)) continue;
                    const double* Xp = s.X + 3 * p;
                    const double r = s.R[p];
                    double m = map_metric(image_centre(x, Xp[0], s.nx, s.per_x), image_centre(y, Xp[1], s.ny, s.per_y),
                                          image_centre(z, Xp[2], s.nz, s.per_z), Xp, r);
                    if (m > 0.0) continue;
                    if (m < best || (m == best && p < bestp)) {
                        best = m;
                        bestp = p;
                    }
                }
            }
}

__global__ void k_fixed_map(Dev s) {
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= s.n) return;
    int x, y, z;
    coords32(s, (int)c, x, y, z);
    double best = __longlong_as_double(0x7ff0000000000000LL);
    int bestp = -1;
    // above every particle's top (z not periodic) no sphere covers the cell
    if (s.per_z || z <= *s.zmax_cell) best_cover(s, x, y, z, 1, best, bestp);
    reinterpret_cast<double*>(s.fixkey)[c] = best;
    s.fixowner[c] = bestp;
}

// Calls f(p) for every mobile particle of the k-th grid cell of the ranges
// that covers cell (x, y, z). |d^2 - r^2| is taken from the FP32 centre first
// (rounded by up to 1e-4 cells at x = 3072), within its margin from the integer
// and fraction of the centre (offsets exact to 1e-7, so the sum to 1e-6 of
// 1 + r^2), and only within the margin of that (1e-5) in FP64 without fused
// multiply-add, which decides: with the FP64 test for the whole first margin
// every listed cell took it, and the kernel was bound by the FP64 pipe (70 us on
// the large flume, 38 us now).
template <class F>
__device__ __forceinline__ void for_covers(const Dev& s, int x, int y, int z, const GRange& ra, const GRange& rb,
                                           const GRange& rc, int k, F f) {
    const int ia = k % ra.n, ib = (k / ra.n) % rb.n, ic = k / (ra.n * rb.n);
    // (selects, so that the ranges stay in registers)
    auto at = [](const GRange& r, int i) { return i == 0 ? r.v[0] : (i == 1 ? r.v[1] : r.v[2]); };
    const int gg = at(ra, ia) + s.gnx * (at(rb, ib) + s.gny * at(rc, ic));
    const int b = s.g_start[gg], e = b + s.g_count[gg];
    for (int j = b; j < e; ++j) {
        const int p = s.g_list[j];
        const float4 xr = s.Xr[p];
        if (xr.w < 0.f) continue;
        float fx = (float)x + 0.5f - xr.x, fy = (float)y + 0.5f - xr.y, fz = (float)z + 0.5f - xr.z;
        if (s.per_x) fx -= (float)s.nx * rintf(fx / (float)s.nx);
        if (s.per_y) fy -= (float)s.ny * rintf(fy / (float)s.ny);
        if (s.per_z) fz -= (float)s.nz * rintf(fz / (float)s.nz);
        const float m32 = fx * fx + fy * fy + fz * fz - xr.w * xr.w;
        const float tol = 1e-3f * (1.f + xr.w * xr.w);
        if (m32 > tol) continue;
        if (m32 >= -tol) {
            const int4 xi = s.Xi[p];
            const float4 xf = s.Xfr[p];
            const float ex = image_offset(x - xi.x, 0.5f - xf.x, s.nx, s.per_x),
                        ey = image_offset(y - xi.y, 0.5f - xf.y, s.ny, s.per_y),
                        ez = image_offset(z - xi.z, 0.5f - xf.z, s.nz, s.per_z);
            const float m2 = ex * ex + ey * ey + ez * ez - xr.w * xr.w;
            if (m2 > 1e-2f * tol) continue;
            if (m2 >= -1e-2f * tol) {
                const double* Xp = s.X + 3 * p;
                const double m = map_metric(image_centre(x, Xp[0], s.nx, s.per_x),
                                            image_centre(y, Xp[1], s.ny, s.per_y),
                                            image_centre(z, Xp[2], s.nz, s.per_z), Xp, s.R[p]);
                if (m > 0.0) continue;
            }
        }
        f(p);
    }
}

// Set-up map: covered cells become solid; every particle of a cell with
// several covers is flagged as sharing cells. The owner has the lowest exact
// metric, then the lowest index.
__device__ void remap_cell(const Dev& s, int c) {
    int x, y, z;
    coords32(s, c, x, y, z);
    const int fo = s.fixowner[c];
    const GRange ra = cover_range(x, s.r_max, s.ghx, s.gnx, s.per_x);
    const GRange rb = cover_range(y, s.r_max, s.ghy, s.gny, s.per_y);
    const GRange rc = cover_range(z, s.r_max, s.ghz, s.gnz, s.per_z);
    const int nc = ra.n * rb.n * rc.n;
    int nm = 0, bestp = -1;
    for (int k = 0; k < nc; ++k) for_covers(s, x, y, z, ra, rb, rc, k, [&](int p) { ++nm; bestp = p; });
    if (nm > 4) set_error(s, ERR_CAPACITY);
    if (nm + (fo >= 0) <= 1) {
        bestp = nm ? bestp : fo;
    } else {
        double best = reinterpret_cast<const double*>(s.fixkey)[c];
        bestp = fo;
        for (int k = 0; k < nc; ++k)
            for_covers(s, x, y, z, ra, rb, rc, k, [&](int p) {
                const double* Xp = s.X + 3 * p;
                const double m = map_metric(image_centre(x, Xp[0], s.nx, s.per_x), image_centre(y, Xp[1], s.ny, s.per_y),
                                            image_centre(z, Xp[2], s.nz, s.per_z), Xp, s.R[p]);
                if (m < best || (m == best && p < bestp)) {
                    best = m;
                    bestp = p;
                }
                s.shared[p] = 1;
            });
    }
    if (bestp >= 0) {
        s.flags[c] = T_SOL;
        s.owner[c] = bestp;
        s.mass[c] = 0.f;
        s.phi[c] = 0.f;
    }
}

__global__ void k_remap_all(Dev s) {
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= s.n) return;
    // above every particle's top (z not periodic) nothing covers a cell
    if (!s.per_z && (int)((unsigned)c / ((unsigned)s.nx * (unsigned)s.ny)) > *s.zmax_cell) return;
    remap_cell(s, (int)c);
}

// cells along one axis that a sphere of radius r at a or b can cover, with a
// cell to spare on each side (the FP32 rounding of the coordinates, below 0.07
// at 2^20 cells, stays within it). On a periodic axis the range is not wrapped,
// and where it is longer than the axis it is the L + 5 cells around b, which
// hold the nearest image of every cell (and a few cells twice): offsets from b
// taken along it are then those of the nearest image.
__device__ __forceinline__ void bbox_axis(float a, float b, float r, int L, int periodic, int& lo, int& hi) {
    const float mn = fminf(a, b), mx = fmaxf(a, b);
    lo = (int)floorf(mn - r - 0.5f) - 1;
    hi = (int)ceilf(mx + r - 0.5f) + 1;
    if (!periodic) {
        lo = lo < 0 ? 0 : lo;
        hi = hi > L - 1 ? L - 1 : hi;
    } else if (hi - lo + 1 > L) {
        const int c = (int)floorf(b);
        lo = c - L / 2 - 2;
        hi = c + (L + 1) / 2 + 2;
    }
}

// Every mobile particle that moved since its last map (|dX| > 0) marks the
// cells whose inside/outside status it can have changed: a cell changes only
// if |x_c - X_new| - r lies within |dX| of zero (triangle inequality), so
// the thin shell |  |x_c - X_new| - r | <= |dX| + 1e-3 is marked (the slack
// covers the FP32 evaluation of the offsets, exact to ~1e-6 through the
// integer-plus-fraction form of the centre). A particle that shares a cell
// with another one marks its whole box, since the owner of a shared cell is
// decided by comparing the two metrics.
// Those cells join the dirty list, each once. A warp per particle, a lane per
// (y, z) row of its box: the row meets the shell | |x_c - X| - r | <= band in
// at most two x-intervals, found from the row's distance to the centre; the
// radii are widened by 1e-3 cells so that rounding can only add cells (a
// cell re-mapped without need keeps its owner). The particle's map position
// then moves to its centre.
__global__ void k_dirty(Dev s) {
    after_previous();
    const int p = (int)(((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int lane = threadIdx.x & 31;
    if (p >= s.np || s.fixed[p]) return;   // whole warps leave together
    const bool whole = s.shared[p] != 0;
    // lane a < 3: axis a, its FP64 work once (the FP64 pipe issues a warp
    // instruction in about 59 cycles, and there is a warp per particle;
    // 17.6 -> 11.5 us for 4 712 particles)
    double xa = 0.0, dm = 0.0;
    if (lane < 3) {
        xa = s.X[3 * p + lane];
        dm = xa - s.Xm[3 * p + lane];
    }
    if (!whole && !__any_sync(0xffffffffu, dm != 0.0)) return;
    const float df = (float)dm, xf32 = (float)xa;
    const float fx = __shfl_sync(0xffffffffu, df, 0), fy = __shfl_sync(0xffffffffu, df, 1),
                fz = __shfl_sync(0xffffffffu, df, 2);
    // shell half-width, rounded up
    const float w = sqrtf(fx * fx + fy * fy + fz * fz) * (1.f + 1e-5f);
    const float r = fabsf(s.Xr[p].w);
    int lo[3], hi[3];
    {
        const int L = lane == 0 ? s.nx : (lane == 1 ? s.ny : s.nz);
        const int per = lane == 0 ? s.per_x : (lane == 1 ? s.per_y : s.per_z);
        int l = 0, h = 0;
        bbox_axis(xf32 - df, xf32, r, L, per, l, h);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            lo[k] = __shfl_sync(0xffffffffu, l, k);
            hi[k] = __shfl_sync(0xffffffffu, h, k);
        }
    }
    const int4 xi = s.Xi[p];
    const float4 xf = s.Xfr[p];
    const float rf = r, band = w + 1e-3f;
    const float ro = rf + band + 1e-3f, ri = fmaxf(rf - band - 1e-3f, 0.f);
    const int ex = hi[0] - lo[0] + 1, ey = hi[1] - lo[1] + 1, ez = hi[2] - lo[2] + 1;
    const int rows = ey * ez;
    // relative x index of a cell = a + xoff, with a its x offset from the centre
    const float xoff = (float)(xi.x - lo[0]) - 0.5f + xf.x;
    for (int r0 = 0; r0 < rows; r0 += 32) {
        const int rr = r0 + lane;
        int a0 = 0, a1 = -1, b0 = 0, b1 = -1;    // relative x ranges of the row
        int ub = 0, uc = 0;
        if (rr < rows) {
            ub = lo[1] + rr % ey;
            uc = lo[2] + rr / ey;
            if (whole) {
                a1 = ex - 1;
            } else {
                const float bb = (float)(ub - xi.y) + 0.5f - xf.y;
                const float cc = (float)(uc - xi.z) + 0.5f - xf.z;
                const float rho2 = bb * bb + cc * cc;
                if (rho2 <= ro * ro) {
                    const float ho = sqrtf(ro * ro - rho2);
                    const float hin = rho2 < ri * ri ? sqrtf(ri * ri - rho2) : 0.f;
                    if (hin == 0.f) {
                        a0 = (int)ceilf(xoff - ho);
                        a1 = (int)floorf(xoff + ho);
                    } else {
                        a0 = (int)ceilf(xoff - ho);
                        a1 = (int)floorf(xoff - hin);
                        b0 = (int)ceilf(xoff + hin);
                        b1 = (int)floorf(xoff + ho);
                    }
                    a0 = max(a0, 0); a1 = min(a1, ex - 1);
                    b0 = max(b0, 0); b1 = min(b1, ex - 1);
                }
            }
        }
        const int n1 = max(0, a1 - a0 + 1), n2 = max(0, b1 - b0 + 1), nc = n1 + n2;
        for (int k = 0; __any_sync(0xffffffffu, k < nc); ++k) {
            bool first = false;
            int cell = 0;
            if (k < nc) {
                const int ua = lo[0] + (k < n1 ? a0 + k : b0 + k - n1);
                const int a = (ua % s.nx + s.nx) % s.nx, b = (ub % s.ny + s.ny) % s.ny, c = (uc % s.nz + s.nz) % s.nz;
                cell = a + s.nx * (b + s.ny * c);
                first = !(flag_or(s.dirty, cell, 1) & 1);
            }
            warp_append(s, first, cell, s.dl, s.dl_count, s.dl_cap);
        }
    }
    __syncwarp();   // every lane has read the old map position and the flag
    if (lane < 3) s.Xm[3 * p + lane] = xa;
    else if (lane == 3) s.shared[p] = 0;
}

// Lane groups of COVER_LANES over the dirty cells, a lane per grid cell
// around it: a thread per cell walked the candidates of up to eight grid
// cells one after the other, after six FP64 divisions (40 us at 1024x64x128
// with 4 712 particles, 11.6 us now; 32 and 10.7 us at 512x40x96). The lanes
// agree on the number of covering mobile particles; where the cell has one
// cover or none that decides, otherwise the exact metrics do (lowest, then
// lowest index), as in remap_cell.
constexpr int COVER_LANES = 8;
__global__ void __launch_bounds__(128) k_remap_list(Dev s) {
    after_previous();
    const int cnt = min(*s.dl_count, s.dl_cap);
    const int l = threadIdx.x % COVER_LANES;
    const unsigned gm = ((1u << COVER_LANES) - 1u) << ((threadIdx.x & 31) / COVER_LANES * COVER_LANES);
    for (int i = (blockIdx.x * blockDim.x + threadIdx.x) / COVER_LANES; i < cnt;
         i += gridDim.x * blockDim.x / COVER_LANES) {
        const int c = s.dl[i];
        int x, y, z;
        coords32(s, c, x, y, z);
        const GRange ra = cover_range(x, s.r_max, s.ghx, s.gnx, s.per_x);
        const GRange rb = cover_range(y, s.r_max, s.ghy, s.gny, s.per_y);
        const GRange rc = cover_range(z, s.r_max, s.ghz, s.gnz, s.per_z);
        const int fo = s.fixowner[c];
        const uint8_t t0 = s.flags[c] & TYPE_MASK;
        const int own = t0 == T_SOL ? s.owner[c] : -1;
        int n = 0, one = -1;      // this lane's covering particles, and the last of them
        for (int k = l; k < ra.n * rb.n * rc.n; k += COVER_LANES)
            for_covers(s, x, y, z, ra, rb, rc, k, [&](int p) { ++n; one = p; });
        int nm = n, bestp = one;
#pragma unroll
        for (int o = 1; o < COVER_LANES; o <<= 1) {
            nm += __shfl_xor_sync(gm, nm, o);
            bestp = max(bestp, __shfl_xor_sync(gm, bestp, o));
        }
        if (nm > 4 && l == 0) set_error(s, ERR_CAPACITY);
        if (nm + (fo >= 0) <= 1) {
            bestp = nm ? bestp : fo;
        } else {
            double best = l == 0 ? reinterpret_cast<const double*>(s.fixkey)[c] : __longlong_as_double(0x7ff0000000000000LL);
            bestp = l == 0 ? fo : -1;
            for (int k = l; k < ra.n * rb.n * rc.n; k += COVER_LANES)
                for_covers(s, x, y, z, ra, rb, rc, k, [&](int p) {
                    const double* Xp = s.X + 3 * p;
                    const double m = map_metric(image_centre(x, Xp[0], s.nx, s.per_x),
                                                image_centre(y, Xp[1], s.ny, s.per_y),
                                                image_centre(z, Xp[2], s.nz, s.per_z), Xp, s.R[p]);
                    if (m < best || (m == best && p < bestp)) {
                        best = m;
                        bestp = p;
                    }
                    s.shared[p] = 1;
                });
#pragma unroll
            for (int o = 1; o < COVER_LANES; o <<= 1) {
                const double m2 = __shfl_xor_sync(gm, best, o);
                const int p2 = __shfl_xor_sync(gm, bestp, o);
                if (p2 >= 0 && (bestp < 0 || m2 < best || (m2 == best && p2 < bestp))) {
                    best = m2;
                    bestp = p2;
                }
            }
        }
        if (l == 0) {
            s.dirty[c] = 0;
            if (bestp != own) {
                const int k = atomicAdd(s.tl_count, 1);
                if (k < s.tl_cap) {
                    s.tl[k] = c;
                    s.tl_info[2 * k] = bestp;
                } else {
                    set_error(s, ERR_CAPACITY);
                }
            }
        }
    }
}

#define FOR_TL(i)                                                                             \
    for (int i = blockIdx.x * blockDim.x + threadIdx.x, _cnt = min(*s.tl_count, s.tl_cap); i < _cnt; \
         i += gridDim.x * blockDim.x)

enum : int { NT_UNCOVERED_LIQ = 0x100 };

// covered cells give their mass to the pool; uncovered cells become liquid
// (interface next to gas, gas without fluid neighbours) with f_eq(mean rho,
// u_b) and take their mass from the pool (snapshot of the cell types)
template <typename S, int LP>
__global__ void __launch_bounds__(128) k_transitions(Dev s) {
    after_previous();
    // (56 us with general slot lookups and FP16 references by division, 11.6 us
    // with the neighbour offsets formed once, at 1024x64x128)
    // a warp per transition: the 27 PDFs of a covered cell, the 26
    // neighbours of an uncovered one and its 27 new PDFs are spread over the
    // lanes, so no thread walks a long chain of dependent loads
    double dpool = 0.0;   // lane 0's change of the pool (one atomic per block)
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    const int count = min(*s.tl_count, s.tl_cap);
    for (int i = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); i < count; i += nwarps) {
        const int c = s.tl[i];
        const int o1 = s.tl_info[2 * i];
        const int t0 = s.flags[c] & TYPE_MASK;
        int x, y, z;
        coords32(s, c, x, y, z);
        S* f = static_cast<S*>(s.f);
        const int nb = lane < 27 ? nbr_q(s, x, y, z, lane) : -1;
        float h = 0.f;
        const long long slot = lane < 27 ? lane_slot<S, LP>(s, lane, c, nb, z, h) : 0;
        int nt;
        if (o1 >= 0) {
            // covered: its liquid mass goes to the pool
            float v = (t0 == T_LIQ && lane < 27) ? with_ref<S>(Store<S>::ld(f + slot), lane, h) : 0.f;
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(full, v, o);
            if (lane == 0) {
                if (t0 == T_LIQ) dpool += (double)(1.f + v);
                else if (t0 == T_IFC) dpool += (double)s.mass[c];
            }
            nt = T_SOL;
        } else {
            // uncovered: lane q takes neighbour q
            float rs = 0.f;
            int cnt = 0;
            bool gas = false;
            if (lane < 27 && lane != 13) {
                if (nb >= 0) {
                    const int tn = s.flags[nb] & TYPE_MASK;
                    if (tn == T_IFC) {
                        rs = s.ru[nb].x;
                        cnt = 1;
                    } else if (tn == T_LIQ) {
                        int bx, by, bz;
                        coords32(s, nb, bx, by, bz);
                        float g[27];
                        load_cell<S, LP>(s, nb, bx, by, bz, g);
                        float d = 0.f;
#pragma unroll
                        for (int k = 0; k < 27; ++k) d += g[k];
                        rs = 1.f + d;
                        cnt = 1;
                    }
                    gas = tn == T_GAS;
                }
            }
            // (the sum's tree runs over the 26 neighbours without the cell itself)
            rs = __shfl_sync(full, rs, lane < 13 ? lane : (lane < 26 ? lane + 1 : 31));
            for (int o = 16; o > 0; o >>= 1) {
                rs += __shfl_xor_sync(full, rs, o);
                cnt += __shfl_xor_sync(full, cnt, o);
            }
            gas = __any_sync(full, gas);
            if (cnt == 0) {
                nt = T_GAS;
            } else {
                const float rb = rs / cnt;
                int po = s.owner[c];
                if (po < 0 || po >= s.np) {
                    if (lane == 0) set_error(s, ERR_INVARIANT);
                    po = 0;
                }
                const double* Xp = s.X + 3 * po;
                const double d[3] = {wrapd(x + 0.5 - Xp[0], s.nx, s.per_x), wrapd(y + 0.5 - Xp[1], s.ny, s.per_y),
                                     wrapd(z + 0.5 - Xp[2], s.nz, s.per_z)};
                const double* Up = s.U + 3 * po;
                const double* Wp = s.W + 3 * po;
                const float ub[3] = {(float)(Up[0] + (Wp[1] * d[2] - Wp[2] * d[1])),
                                     (float)(Up[1] + (Wp[2] * d[0] - Wp[0] * d[2])),
                                     (float)(Up[2] + (Wp[0] * d[1] - Wp[1] * d[0]))};
                if (lane < 27) {
                    const float fq = feq_dev(lane, rb, ub[0], ub[1], ub[2]);
                    Store<S>::st(f + slot, with_ref<S>(fq, lane, -h));
                    Store<S>::st(static_cast<S*>(s.fs) + (long long)lane * s.n + c,
                                 with_ref<S>(fq, lane, Store<S>::HREF ? -s.href[z] : 0.f));
                }
                if (lane == 0) {
                    s.ru[c] = make_float4(rb, ub[0], ub[1], ub[2]);
                    s.mass[c] = gas ? 0.f : rb;
                    if (!gas) dpool -= (double)rb;
                }
                nt = gas ? T_IFC : (T_LIQ | NT_UNCOVERED_LIQ);
            }
        }
        if (lane == 0) s.tl_info[2 * i + 1] = nt;
    }
    __shared__ double red[32];
    for (int o = 16; o > 0; o >>= 1) dpool += __shfl_xor_sync(full, dpool, o);
    if (lane == 0) red[threadIdx.x >> 5] = dpool;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
        if (t != 0.0) atomicAdd(s.pool, t);
    }
}

__global__ void k_apply_transitions(Dev s) {
    after_previous();
    FOR_TL(i) {
        const int c = s.tl[i];
        const int nt = s.tl_info[2 * i + 1];
        const int t = nt & TYPE_MASK;
        s.flags[c] = (uint8_t)t;
        if (t == T_SOL) {
            s.owner[c] = s.tl_info[2 * i];
            s.mass[c] = 0.f;
            s.phi[c] = 0.f;
        } else {
            s.owner[c] = -1;
            if (t == T_GAS) { s.mass[c] = 0.f; s.phi[c] = 0.f; }
            else if (t == T_IFC) s.phi[c] = s.mass[c] / s.ru[c].x;
        }
    }
}

// an uncovered liquid cell that ended next to a gas cell becomes interface
__global__ void k_repair(Dev s) {
    after_previous();
    FOR_TL(i) {
        if (!(s.tl_info[2 * i + 1] & NT_UNCOVERED_LIQ)) continue;
        const int c = s.tl[i];
        int x, y, z;
        coords32(s, c, x, y, z);
        const NbrOffsets o = nbr_offsets(s, x, y, z);
        bool gas = false;
#pragma unroll
        for (int q = 0; q < 27; ++q) {
            if (q == 13 || (o.wall & wall_bits(cx(q), cy(q), cz(q)))) continue;
            gas |= (s.flags[c + o.ox[1 + cx(q)] + o.oy[1 + cy(q)] + o.oz[1 + cz(q)]] & TYPE_MASK) == T_GAS;
        }
        if (gas) {
            s.flags[c] = T_IFC;
            s.phi[c] = s.mass[c] / s.ru[c].x;
        }
    }
}

// The particle part of a step in two halves. The DEM half (neighbour list,
// force average, sub-steps, FP32 copies, particle grid) reads and writes
// particle state only, so it can run beside the fluid kernels and the
// free-surface conversion, which read and write cell state only; the re-map
// half needs both. The neighbour list needs the positions alone, so it is
// launched at the step's start, the rest once the particle forces are complete.
int launch_dem_neighbours(const Dev& s, cudaStream_t st) {
    if (s.np == 0) return 0;
    k_dem_neighbours<<<blocks_for(32LL * s.np, 128), 128, 0, st>>>(s);
    return 1;
}

static size_t dem_cluster_smem(int threads) {
    return (size_t)(threads / DEM_LANES) * (sizeof(ClusterParticle) + DEM_SH * sizeof(float));
}
template <int THREADS>
static void dem_cluster_attributes() {
    cudaFuncSetAttribute(k_dem_cluster<THREADS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)dem_cluster_smem(THREADS));
    cudaFuncSetAttribute(k_dem_cluster<THREADS>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
}
// The largest cluster that this device places with 1024 threads a CTA (a
// cluster of 16 needs as many SMs of one group), asked at a device's first use.
// The kernels' attributes are set then too, for their largest blocks, and never
// again: they belong to the function, and a run that lowered them to its own
// size would have the launch of a larger run in another thread refused.
static int dem_cluster_ctas() {
    constexpr int DEVICES = 64;
    static std::atomic<int> known[DEVICES];   // 0: not asked yet
    int dev = 0;
    cudaGetDevice(&dev);
    const int have = dev < DEVICES ? known[dev].load(std::memory_order_acquire) : 0;
    if (have) return have;
    dem_cluster_attributes<512>();
    dem_cluster_attributes<1024>();
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = DEM_CLUSTER_CTAS;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(DEM_CLUSTER_CTAS);
    cfg.blockDim = dim3(1024);
    cfg.dynamicSmemBytes = dem_cluster_smem(1024);
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, k_dem_cluster<1024>, &cfg) != cudaSuccess) {
        cudaGetLastError();
        clusters = 0;
    }
    const int ctas = clusters > 0 ? DEM_CLUSTER_CTAS : 8;
    if (dev < DEVICES) known[dev].store(ctas, std::memory_order_release);
    return ctas;
}

int launch_dem(const Dev& s, int have_prev, cudaStream_t st) {
    if (s.np == 0) return 0;
    const int ns = s.dem_substeps, G = s.gnx * s.gny * s.gnz;
    const float dts = 1.f / (float)ns;
    const int max_ctas = s.np <= DEM_CLUSTER_MAX ? dem_cluster_ctas() : 0;
    if (s.np <= max_ctas * 1024 / DEM_LANES) {
        // one particle per lane group. Up to 64 particles in one CTA, whose
        // partners' values are its own (34 particles: step of the 64x16x32
        // flume 0.0775 ms, in four CTAs 0.0795); beyond, as many CTAs as leave
        // each 512 threads, up to the largest cluster (735 particles of the
        // 301x37x75 flume in 16 CTAs: step 0.137 ms, in 8: 0.1465)
        const int lanes = s.np * DEM_LANES;
        int ctas = 1;
        while (ctas < max_ctas && ctas * 512 < lanes) ctas *= 2;
        int threads = ((lanes + ctas - 1) / ctas + 31) / 32 * 32;
        threads = threads < 128 ? 128 : threads;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)ctas);
        cfg.blockDim = dim3((unsigned)threads);
        cfg.dynamicSmemBytes = dem_cluster_smem(threads);
        cfg.stream = st;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = (unsigned)ctas;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        cudaLaunchKernelEx(&cfg, threads <= 512 ? k_dem_cluster<512> : k_dem_cluster<1024>, s, have_prev, G, dts);
        return 1;
    }
    if (ns == 1) {
        cudaMemsetAsync(s.g_count, 0, sizeof(int) * G, st);
        cudaMemsetAsync(s.zmax_cell, 0, sizeof(int), st);
    }
    // ordinary launches: blocks of a sub-step that wait on the SMs for the one
    // before take room from the liquid kernels (launch_after: sweep of the
    // 1024x64x128 flume at FP16 0.310 -> 0.338 ms)
    for (int k = 0; k < ns; ++k)
        k_dem_substep<<<blocks_for((long long)DEM_LANES * s.np, 128), 128, 0, st>>>(s, k & 1, have_prev, G, dts, k == 0,
                                                                                   k == ns - 1);
    return ns + launch_grid_lists(s, st);
}

template <typename S>
static void launch_transitions(const Dev& s, int last_parity, cudaStream_t st) {
    if (last_parity == 0) launch_after(k_transitions<S, 0>, 152 * 4, 128, st, s);
    else launch_after(k_transitions<S, 1>, 152 * 4, 128, st, s);
}

// (the counts of the dirty and transition lists are cleared by the conversion)
int launch_remap(const Dev& s, int last_parity, cudaStream_t st) {
    if (s.np == 0) return 0;
    k_dirty<<<blocks_for(32LL * s.np, 128), 128, 0, st>>>(s);
    launch_after(k_remap_list, 152 * 8, 128, st, s);
    if (s.storage == FSLBM_STORE_FP32) launch_transitions<float>(s, last_parity, st);
    else if (s.storage == FSLBM_STORE_FP16) launch_transitions<__half>(s, last_parity, st);
    else launch_transitions<__nv_bfloat16>(s, last_parity, st);
    launch_after(k_apply_transitions, 152 * 4, 256, st, s);
    launch_after(k_repair, 152 * 4, 256, st, s);
    return 5;
}

__global__ void k_init_particles(Dev s, int first, int count, double rho_p) {
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= count) return;
    int p = first + k;
    double r = s.R[p];
    s.M[p] = rho_p * (4.0 / 3.0) * 3.14159265358979323846 * r * r * r;
    s.I[p] = 0.4 * s.M[p] * r * r;
    for (int a = 0; a < 3; ++a) {
        s.U[3 * p + a] = s.W[3 * p + a] = 0.0;
        s.Fh[3 * p + a] = s.Th[3 * p + a] = s.Fp[3 * p + a] = s.Tp[3 * p + a] = 0.0;
    }
    s.nb_count[p] = 0;
    for (int j = 0; j < NB_ITEMS; ++j) s.nb_xi[(long long)p * NB_ITEMS + j] = make_float4(0.f, 0.f, 0.f, 0.f);
    // the set-up map (k_remap_all) flags every particle that shares a cell;
    // the others re-map their thin shell from the first step on
    s.shared[p] = 0;
    for (int a = 0; a < 3; ++a) s.Xm[3 * p + a] = s.X[3 * p + a];
    atomicMax(s.zmax_cell, (int)ceil(s.X[3 * p + 2] + r) + 2);
}

void launch_particles_add(const Dev& s, int first, int count, cudaStream_t st) {
    k_init_particles<<<blocks_for(count, 128), 128, 0, st>>>(s, first, count, s.rho_p);
    k_particle_copies<<<blocks_for(s.np, 128), 128, 0, st>>>(s);
    launch_grid_build(s, st);
    k_fixed_map<<<blocks_for(s.n, 256), 256, 0, st>>>(s);
    k_remap_all<<<blocks_for(s.n, 256), 256, 0, st>>>(s);
}

}  // namespace fsl

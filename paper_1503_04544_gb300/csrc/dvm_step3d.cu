// 3D time step of the cut-cell discrete-velocity method (arXiv:1503.04544,
// Sec. 5, Eq. eq-schema3D) for the full distribution F and a fixed obstacle:
// wall density and stress of the diffuse wall (3D forms of Eqs. BoundaryDDv
// and StressTensorDD), force and torque about the z axis, fluxes across the
// six Cartesian faces of every virtual cell (each direction with its own
// velocity component) and across its wall face, explicit update of each
// control volume with BGK relaxation toward the 3D Maxwellian, distribution
// to the members (Eq. UpdateDD).
//
// Device layout: element (cell, p) at (q * slab + P(i, j, k)) * W + e for the
// velocity group q and lane e of the padded velocity index (Grid3D), with
// P(i, j, k) = ((k + 2)(ny + 4) + j + 2)(nx + 4) + i + 2: every group is a
// slab of the grid padded by two cells on each side that holds the boundary
// condition, so a neighbour within two cells along an axis is a plain index.
//
// Kernels of one step: k_wall3 (FP64 wall density, force and torque; the
// last block sums them in list order), k_bulk3 (every gas cell that is a
// control volume on its own), k_special3 (cut and merged control volumes).
// k_bulk3 assigns one thread to a column of cells along z; a warp covers 32
// consecutive cells of the block's tile, row after row (a row may end inside a
// warp), at the velocities of one group, so the upwind side along y and z is
// uniform across the warp.  The velocity groups are split over blockIdx.z;
// each block streams the planes of its column through shared memory with TMA,
// writes the new state and accumulates the moments of the new state for the
// next step.
#include <cudaTypedefs.h>

#include <cstdio>
#include <string>
#include <type_traits>

#include "dvm_device.cuh"

namespace dvm {
namespace {

template <typename T> struct alignas(2 * sizeof(T)) VX3 { T vx, nux; };
template <typename T> struct alignas(4 * sizeof(T)) VYZ3 { T vy, vz, nuy, nuz; };

// Slab index of cell (i, j, k), each within two cells of the grid.
__device__ __forceinline__ int nbr3(const Grid3D &g, int i, int j, int k)
{
    return ((k + 2) * (g.ny + 4) + (j + 2)) * (g.nx + 4) + (i + 2);
}

__device__ __forceinline__ void cell_ijk(const Grid3D &g, int q, int &i, int &j, int &k)
{
    const int r = q / g.nx;
    i = q - r * g.nx;
    k = r / g.ny;
    j = r - k * g.ny;
}

__device__ __forceinline__ int pcell3(const Grid3D &g, int q)
{
    int i, j, k;
    cell_ijk(g, q, i, j, k);
    return nbr3(g, i, j, k);
}

// Element offset of padded velocity p at slab index pc.
__device__ __forceinline__ long pidx3(const Grid3D &g, int p, int pc)
{
    const int grp = p / g.W;
    return ((long)grp * g.slab + pc) * g.W + (p - grp * g.W);
}


// Padding cells that mirror interior cell (i, j, k) on periodic and
// zero-gradient sides (two per axis at most); -1 where unused.
__device__ __forceinline__ void mirrors3(const Grid3D &g, int i, int j, int k, int (&m)[6])
{
#pragma unroll
    for (int t = 0; t < 6; ++t) m[t] = -1;
    if (g.bc[0] == DVM_BC_PERIODIC) {
        if (i < 2) m[0] = nbr3(g, i + g.nx, j, k);
        else if (i >= g.nx - 2) m[0] = nbr3(g, i - g.nx, j, k);
    } else {
        if (i == 0 && g.bc[0] == DVM_BC_ZEROGRAD) { m[0] = nbr3(g, -1, j, k); m[1] = nbr3(g, -2, j, k); }
        if (i == g.nx - 1 && g.bc[1] == DVM_BC_ZEROGRAD) { m[0] = nbr3(g, g.nx, j, k); m[1] = nbr3(g, g.nx + 1, j, k); }
    }
    if (g.bc[2] == DVM_BC_PERIODIC) {
        if (j < 2) m[2] = nbr3(g, i, j + g.ny, k);
        else if (j >= g.ny - 2) m[2] = nbr3(g, i, j - g.ny, k);
    } else {
        if (j == 0 && g.bc[2] == DVM_BC_ZEROGRAD) { m[2] = nbr3(g, i, -1, k); m[3] = nbr3(g, i, -2, k); }
        if (j == g.ny - 1 && g.bc[3] == DVM_BC_ZEROGRAD) { m[2] = nbr3(g, i, g.ny, k); m[3] = nbr3(g, i, g.ny + 1, k); }
    }
    if (g.bc[4] == DVM_BC_PERIODIC) {
        if (k < 2) m[4] = nbr3(g, i, j, k + g.nz);
        else if (k >= g.nz - 2) m[4] = nbr3(g, i, j, k - g.nz);
    } else {
        if (k == 0 && g.bc[4] == DVM_BC_ZEROGRAD) { m[4] = nbr3(g, i, j, -1); m[5] = nbr3(g, i, j, -2); }
        if (k == g.nz - 1 && g.bc[5] == DVM_BC_ZEROGRAD) { m[4] = nbr3(g, i, j, g.nz); m[5] = nbr3(g, i, j, g.nz + 1); }
    }
}


// Primitive variables from the sums s0 = sum F, s1..3 = sum v F,
// s4 = sum |v|^2/2 F (Eq. MacroscopicTD; T from E = rho|u|^2/2 + 3/2 rho T).
template <typename T>
__device__ __forceinline__ bool primitives3(T dv, const T (&s)[5], T &rho, T &ux, T &uy, T &uz, T &tmp)
{
    rho = s[0] * dv;
    ux = s[1] / s[0];
    uy = s[2] / s[0];
    uz = s[3] / s[0];
    tmp = (T(2) * (s[4] / s[0]) - (ux * ux + uy * uy + uz * uz)) / T(3);
    return rho > T(0) && tmp > T(0);
}

// Sum of the S partial moments of a cell ([S][5][nc] layout).
template <typename T>
__device__ __forceinline__ void gather_partials3(const T *part, int S, long nc, long cell, T (&s)[5])
{
    Acc<T> a[5];
#pragma unroll 4
    for (int q = 0; q < S; ++q)       // several splits' loads in flight
#pragma unroll
        for (int m = 0; m < 5; ++m) a[m].merge(part[((long)q * 5 + m) * nc + cell], T(0));
#pragma unroll
    for (int m = 0; m < 5; ++m) s[m] = a[m].value();
}

// 1 / (2 pi T)^{3/2}
template <typename T>
__device__ __forceinline__ T norm3(T tmp)
{
    const T a = T(2.0 * kPi) * tmp;
    return T(1) / (a * sqrt(a));
}

// ------------------------------------------------------------ bulk kernel
template <typename T> struct Bulk3Args {
    Grid3D g;
    int S, nzc;
    int tx, ty;               // tile of cells (tile3d)
    int Sin;                  // partial-sum slots of pin (S, or 1 for summed moments of a velocity split)
    const T *fin;
    T *fout;
    const T *pin;             // partial moments of F^n   [S][5][nc]
    T *pout;                  // partial moments of F^n+1 [S][5][nc]
    const uint16_t *flags;
    const VX3<T> *vxt;        // [nvxp]
    const VYZ3<T> *vyz;       // [nvy * nvz]
    const T *eqp;             // [5][nc] conservative equilibrium parameters, or null (direct moments)
    const double *cf;         // FP64: per-cell values [kMxCount + nvxp][nc] (k_cell64_3)
    const T *qh;              // [3][nc] heat flux of the control volume at t^n (Shakhov model)
    T pr1;                    // 1 - Pr (Shakhov model)
    int *err;
};

constexpr int kZc3 = 4;                           // z-planes per block column
constexpr int kPlanes3 = kZc3 + 3;                // planes of a column: two upwind, the cells, one downwind
constexpr int kFold3 = 8;                         // groups of the longest plain moment sum

// Warps of the bulk kernel's block.  FP32: 16, the most that leave a thread
// 128 registers.  FP64: 8 (shared memory of the per-cell data; the kernel is
// bound by the FP64 pipe).
template <typename T> __host__ __device__ constexpr int warps3() { return sizeof(T) == 4 ? 16 : 8; }
// Ring slot stride in 16-byte cells: the most cells of a plane, tile and
// two-cell halo (tile3d keeps to it).  Every slot is the destination of a
// tensor copy and starts on a 128-byte boundary.
template <typename T> __host__ __device__ constexpr int plane_stride3() { return sizeof(T) == 4 ? 816 : 448; }

// Ring slots: the planes of a whole group, so that plane o of every group has
// its own slot; the Shakhov variant has room for five.
template <bool SHAK> __host__ __device__ constexpr int ring3() { return SHAK?5:kPlanes3; }

// Per-cell values of the bulk kernel in shared memory.  FP32: c0, c1, c2, r
// (one vector), uy, uz, and the Shakhov model's k q.  FP64: the values of
// MxSlot.
enum MxSlot { kMxUy = 0, kMxUz, kMxC2, kMxRel, kMxCount };
template <typename T, bool SHAK> __host__ __device__ constexpr int ncoef3()
{
    return sizeof(T) == 8 ? kMxCount : (SHAK ? 9 : 6);
}
// Compensated sums in FP32 (sum, compensation), plain in FP64.
template <typename T> __host__ __device__ constexpr int nsum3() { return sizeof(T) == 4 ? 10 : 5; }

template <typename T, bool SHAK>
size_t bulk3_smem()
{
    return (size_t)ring3<SHAK>() * plane_stride3<T>() * 16 +
           (size_t)kZc3 * (ncoef3<T, SHAK>() + nsum3<T>()) * 32 * warps3<T>() * sizeof(T) +
           32 * warps3<T>() * sizeof(uint32_t) +
           (size_t)(kMaxAxisNv / Vec<T>::W) * (4 * 16 + 8) + 2 * ring3<SHAK>() * sizeof(uint64_t);
}

__device__ __forceinline__ void tma_load_4d(void *dst, const CUtensorMap *map, uint64_t *bar, int x, int y, int z, int w)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(w), "r"(smem_u32(bar))
        : "memory");
}

// 2^x in the state precision: the hardware approximation in FP32.
__device__ __forceinline__ float exp2_state(float x) { return ex2_fast(x); }
__device__ __forceinline__ double exp2_state(double x) { return exp2(x); }

// Lane l of a unit.
__device__ __forceinline__ float unit_lane(F2 x, int l) { float a, b; f2_get(x, a, b); return l ? b : a; }
__device__ __forceinline__ double unit_lane(double x, int) { return x; }

// The per-cell values of the FP64 bulk kernel for the plain cells
// (dvm_device.cuh): the slots of MxSlot, then the v_x factors.  Block = 16
// cells x kCellThreads.
__global__ void __launch_bounds__(128) k_cell64_3(Bulk3Args<double> a, double *cf)
{
    const Grid3D &g = a.g;
    const long nc = (long)g.nx * g.ny * g.nz;
    const long cell = (long)blockIdx.x * (128 / kCellThreads) + threadIdx.x / kCellThreads;
    const int k = threadIdx.x % kCellThreads;
    const bool plain = cell < nc && (a.flags[cell] & kPlain);
    double s[5] = {0, 0, 0, 0, 0};
    if (plain)
#pragma unroll 4
        for (int q = k; q < a.Sin; q += kCellThreads)
#pragma unroll
            for (int m = 0; m < 5; ++m) s[m] += a.pin[((long)q * 5 + m) * nc + cell];
#pragma unroll
    for (int m = 0; m < 5; ++m) s[m] = cell_sum<kCellThreads>(s[m]);
    if (!plain) return;
    double rho, ux, uy, uz, tmp;
    if (!primitives3<double>(g.dv, s, rho, ux, uy, uz, tmp) && k == 0) atomicExch(&a.err[kErrNonphys], 1);
    const double r = g.dt_tau0 * rho;
    if (a.eqp) {
        // conservative equilibrium (Sec. 3.1): tau from the direct density,
        // the Maxwellian from the Newton parameters
        rho = a.eqp[cell]; ux = a.eqp[nc + cell]; uy = a.eqp[2 * nc + cell];
        uz = a.eqp[3 * nc + cell]; tmp = a.eqp[4 * nc + cell];
    }
    const double c2 = (0.5 * kLog2e) / tmp;
    double *const o = cf + cell;
    put_factors<kCellThreads>(o + kMxCount * nc, nc, k, g.nvx, g.nvxp, g.vxmin, g.dvx, ux, c2, r * rho * norm3(tmp));
    if (k == kCellThreads - 1) {
        o[kMxUy * nc] = uy;
        o[kMxUz * nc] = uz;
        o[kMxC2 * nc] = c2;
        o[kMxRel * nc] = r;
    }
}

// Bulk update of every gas cell that is a control volume on its own.
//
// Block = a tile of a.tx x a.ty cells in (x, y), taken row by row by the
// threads (tile3d), and a column of kZc3 cells in z (blockIdx.z = split * nzc + column); R warps.  For
// each velocity group of its split the planes of the column (tile plus a
// two-cell halo, one TMA load each) stream through a ring of shared-memory
// slots in upwind order of v_z.  Thread 0 refills the slot that its warp
// released two planes ago, once every warp has released it (a producer warp
// of its own would take the 17th warp's registers from all: 96 a thread and
// spills).  Every wait is bounded and records kErrTimeout instead of blocking.
//
// A thread marches its column downwind: along z the centre, the upwind
// difference and the limited slope of the upwind face roll through registers,
// so that each face is formed once and the group needs two upwind planes and
// one downwind plane beside its cells; x and y neighbours come from the
// plane's slot, on the group's upwind side.  The arithmetic runs on units of
// the group (pairs of FP32 velocities, f32x2).  Warps whose 32 cells all have
// the limiter on every face take the path without face weights, the others
// (near the obstacle) the one with weights; a group whose v_x changes sign
// within a unit goes velocity by velocity.  The weighted path has to be nearly
// as fast: one slow warp holds up its whole block at the ring.
//
// Moments: v_y and v_z are uniform in a row of groups, so a cell sums F,
// v_x F and v_x^2 F over the row and forms the five moments once per row (once
// per eight groups of a longer one, so that no plain sum is longer), into sums
// in shared memory, compensated in FP32.
//
// FP64: the Maxwellian is the cell's v_x factor (put_factors; read for the
// whole column before the group's planes) times the row's factor of v_y and
// v_z (one exp2 a row): one FP64 multiplication a velocity instead of an exp2.
//
// FP32 is bound by issue slots (64^3 x 12^3: 77 warp instructions a velocity
// and 32 cells, 27 of them on the half-rate ALU pipe) and by waits for planes;
// FP64 by the FP64 pipe (two lanes a clock; 29 operations a velocity with its
// share of the row's, at 12 velocities a row).  The form before this one (a
// thread per column in fixed z order, both z faces' planes read, exp2 per
// velocity, velocity by velocity moments) took, a launch: FP32 64^3 x 20^3
// 9.72 ms, now 7.3; 96^3 x 20^3 30.6, now 23.4; Shakhov 45 x 50 x 37 x (14, 15,
// 13) 2.13, now 1.67; FP64 40^3 x 12^3 20.8, now 7.4 (7.7 with a recurrence
// for the Maxwellian).
//
// With SHAK (the Shakhov model, FP32) the cells relax towards F_S = M [1 +
// k c.q (|c|^2/T - 5)], k = (1 - Pr) / (5 rho T^2), with the heat flux q of
// the cell at t^n from k_heatflux3: |c|^2/T from the Maxwellian's base-2
// exponent and k c.q linear in v.
template <typename T, bool MUSCL, bool SHAK>
__global__ void __launch_bounds__(32 * warps3<T>(), 1)
    k_bulk3(Bulk3Args<T> a, const __grid_constant__ CUtensorMap tmap)
{
    static_assert(!SHAK || sizeof(T) == 4, "the Shakhov variant of the bulk kernel is FP32");
    using V = typename Vec<T>::type;
    using P = typename Lanes<T>::P;
    constexpr int W = Vec<T>::W, LN = Lanes<T>::N, ZC = kZc3, R = warps3<T>(), NT = 32 * R, NP = kPlanes3;
    constexpr int RING = ring3<SHAK>(), NCO = ncoef3<T, SHAK>(), NSUM = nsum3<T>();
    constexpr int PC = plane_stride3<T>();
    constexpr bool F64 = sizeof(T) == 8;
    static_assert((PC * 16) % 128 == 0, "tensor-copy destinations start on 128-byte boundaries");
    extern __shared__ __align__(128) unsigned char sm3[];
    V *const ring = reinterpret_cast<V *>(sm3);
    T *const coef = reinterpret_cast<T *>(sm3 + RING * PC * 16);    // FP32 [ZC][NT][4], then [ZC][NCO - 4][NT]; FP64 [ZC][NCO][NT]
    T *const ksum = coef + ZC * NCO * NT;                           // [ZC][NSUM][NT]
    V *const vtab = reinterpret_cast<V *>(ksum + ZC * NSUM * NT);   // [nxg][4]: v_x, v_x^2, -nu_x, (1 - nu_x)/2
    int *const xsg = reinterpret_cast<int *>(vtab + 4 * (kMaxAxisNv / W));   // [nxg][2] sign of v_x in each unit (0: mixed)
    uint64_t *const full = reinterpret_cast<uint64_t *>(xsg + 2 * (kMaxAxisNv / W));
    uint64_t *const empty = full + RING;
    uint32_t *const cellw = reinterpret_cast<uint32_t *>(empty + RING) + threadIdx.x;  // flags of the thread's cells
    const Grid3D &g = a.g;
    const int tid = threadIdx.x, px = a.tx + 4;          // px: cells of a plane's row
    const bool intile = tid < a.tx * a.ty;
    const int ly = intile ? tid / a.tx : 0, lx = intile ? tid - ly * a.tx : 0;
    const int i0 = blockIdx.x * a.tx, j0 = blockIdx.y * a.ty;
    const int i = i0 + lx, j = j0 + ly;
    const int zc = blockIdx.z % a.nzc, split = blockIdx.z / a.nzc;
    const int z0 = zc * ZC;
    const long nc = (long)g.nx * g.ny * g.nz;
    const int gps = (g.ngrp + a.S - 1) / a.S;
    const int g0 = split * gps, g1 = min(g0 + gps, g.ngrp);
    const int ngr = max(g1 - g0, 0);
    const int total = ngr * NP;
    const bool inij = intile && i < g.nx && j < g.ny;
    // first group with v_z >= 0
    int gpos = 0;
    while (gpos < g.nvz && a.vyz[gpos * g.nvy].vz < T(0)) ++gpos;
    gpos *= g.nxg * g.nvy;
    // load of plane n of the split, counted over its groups: plane o of a
    // group in upwind order (padded plane indices)
    const auto load_plane = [&](int n) {
        const int gi = n / NP, o = n - gi * NP, grp = g0 + gi, slot = RING == NP ? o : n % RING;
        mbar_expect_tx(&full[slot], (uint32_t)(px * (a.ty + 4) * 16));
        tma_load_4d(ring + slot * PC, &tmap, &full[slot], i0 * W, j0, grp >= gpos ? z0 + o : z0 + ZC + 3 - o, grp);
    };

    if (tid == 0) {
        for (int st = 0; st < RING; ++st) {
            mbar_init(&full[st], 1);
            mbar_init(&empty[st], R);
        }
        mbar_fence_init();
        for (int n = 0; n < RING && n < total; ++n) load_plane(n);
    }
    // the v_x rows of the groups, staged once per block
    for (int q = tid; q < g.nxg; q += NT) {
        T *const t = reinterpret_cast<T *>(vtab + 4 * q);
        int s[2];
        for (int h = 0; h < 2; ++h) {
            bool pos = true, neg = true;
            for (int l = 0; l < LN; ++l) {
                const int e = h * LN + l;
                const VX3<T> cx = a.vxt[q * W + e];
                t[e] = cx.vx;
                t[W + e] = cx.vx * cx.vx;
                t[2 * W + e] = -cx.nux;
                t[3 * W + e] = T(0.5) * (T(1) - cx.nux);
                pos = pos && cx.vx >= T(0);
                neg = neg && cx.vx <= T(0);
            }
            s[h] = pos ? 1 : (neg ? -1 : 0);
        }
        xsg[2 * q] = s[0];
        xsg[2 * q + 1] = s[1];
    }
    // per-cell data of the column: flags, and for plain cells the
    // equilibrium in the form log2 M(v) = c0 + vx (c1 - c2 vx) - c2 dyz(v)
    // bit t: cell t of the column is plain, bit 4 + t: to be zeroed, bits 8 +
    // 6 t: its face mask (in shared memory: registers are short)
    uint32_t word = 0, fullm = 0;
    static_assert(ZC <= 4, "the flag word");
    T *const cq = coef + (F64 ? 0 : 4 * ZC * NT);
    constexpr int NCQ = F64 ? NCO : NCO - 4;
#pragma unroll 1
    for (int t = 0; t < ZC; ++t) {
        const int k = z0 + t;
        const bool in = inij && k < g.nz;
        const long cell = ((long)k * g.ny + j) * g.nx + i;
        const uint16_t fl = in ? a.flags[cell] : 0;
        T *const cz = cq + t * NCQ * NT + tid;
        if (fl & kPlain) {
            word |= 1u << t;
            if constexpr (F64) {
#pragma unroll
                for (int k = 0; k < NCO; ++k) cz[k * NT] = a.cf[k * nc + cell];
            } else {
                T s[5];
                gather_partials3(a.pin, a.Sin, nc, cell, s);
                T rho, ux, uy, uz, tmp;
                if (!primitives3<T>(g.dv_f, s, rho, ux, uy, uz, tmp)) atomicExch(&a.err[kErrNonphys], 1);
                const T r = g.dt_tau0_f * rho;
                if (a.eqp) {
                    // conservative equilibrium (Sec. 3.1): tau from the direct
                    // density, the Maxwellian from the Newton parameters
                    rho = a.eqp[cell]; ux = a.eqp[nc + cell]; uy = a.eqp[2 * nc + cell];
                    uz = a.eqp[3 * nc + cell]; tmp = a.eqp[4 * nc + cell];
                }
                const T c2 = T(kLog2e) / (T(2) * tmp);
                T *const cv = coef + (t * NT + tid) * 4;
                cv[0] = log2(rho * norm3(tmp)) - c2 * ux * ux;
                cv[1] = T(2) * c2 * ux;
                cv[2] = c2;
                cv[3] = r;
                cz[0] = uy;
                cz[NT] = uz;
                if constexpr (SHAK) {
                    const T kk = a.pr1 / (T(5) * rho * tmp * tmp);
                    cz[2 * NT] = kk * a.qh[cell];
                    cz[3 * NT] = kk * a.qh[nc + cell];
                    cz[4 * NT] = kk * a.qh[2 * nc + cell];
                }
            }
        }
        if (fl & kZero) word |= 16u << t;
        const uint32_t mk = (fl >> kMaskShift3) & 0x3F;
        word |= mk << (8 + 6 * t);
        // every lane of the warp outside the grid, or plain with the
        // limiter on all six faces
        if (__all_sync(0xffffffffu, !in || ((fl & kPlain) && (!MUSCL || mk == 0x3F)))) fullm |= 1u << t;
        for (int m = 0; m < NSUM; ++m) ksum[(t * NSUM + m) * NT + tid] = T(0);
    }
    *cellw = word;
    __syncthreads();

    // FP64: v_x factors of the column's first cell (of cell 0 of its plane
    // outside the grid)
    const double *const mx0 = F64 ? a.cf + kMxCount * nc + (long)z0 * g.nx * g.ny + (inij ? j * g.nx + i : 0) : nullptr;
    const int c0 = (ly + 2) * px + lx + 2;
    const int sz = (g.nx + 4) * (g.ny + 4);
    const int pc0 = inij ? nbr3(g, i, j, z0) : 0;
    // padding mirrors of the thread's cells along x and y: offset of the first
    // one (0: none); on zero-gradient sides, where it is one cell, a second
    // one twice as far
    int mx = 0, my = 0;
    const int row = g.nx + 4;
    if (inij) {
        if (g.bc[0] == DVM_BC_PERIODIC) mx = i < 2 ? g.nx : (i >= g.nx - 2 ? -g.nx : 0);
        else if (i == 0 && g.bc[0] == DVM_BC_ZEROGRAD) mx = -1;
        else if (i == g.nx - 1 && g.bc[1] == DVM_BC_ZEROGRAD) mx = 1;
        if (g.bc[2] == DVM_BC_PERIODIC) my = j < 2 ? g.ny * row : (j >= g.ny - 2 ? -g.ny * row : 0);
        else if (j == 0 && g.bc[2] == DVM_BC_ZEROGRAD) my = -row;
        else if (j == g.ny - 1 && g.bc[3] == DVM_BC_ZEROGRAD) my = row;
    }
    const bool zside = z0 < 2 || z0 + ZC > g.nz - 2;
    const bool xside = __any_sync(0xffffffffu, mx != 0), yside = __any_sync(0xffffffffu, my != 0);

    // slot and phase of plane o of group gi: with a slot for every plane of a
    // group, plane o is always in slot o
    const uint32_t full0 = smem_u32(full), empty0 = smem_u32(empty), lane0 = (tid & 31) == 0;
    const bool warp0 = tid < 32;
    uint32_t bad = 0;               // a wait timed out
    const auto slot_of = [](int gi, int o) { return RING == NP ? o : (gi * NP + o) % RING; };
    const auto wait_full = [&](int gi, int o) {
        const uint32_t phase = RING == NP ? gi & 1 : ((gi * NP + o) / RING) & 1;
        mbar_wait_or(full0 + 8 * slot_of(gi, o), phase, bad);
    };
    const auto release = [&](int gi, int o) {
        __syncwarp();
        mbar_arrive_if(empty0 + 8 * slot_of(gi, o), lane0);
        if (warp0 && lane0) {
            // the plane this warp released two planes ago, RING planes on
            const int n = gi * NP + o - 2;
            if (n >= 0 && n + RING < total) {
                const int slot = RING == NP ? (o + NP - 2) % NP : n % RING;
                mbar_wait_or(empty0 + 8 * slot, (uint32_t)((n / RING) & 1), bad);
                load_plane(n + RING);
            }
        }
    };
    // store of a cell's vector and of its padding mirrors
    const auto store = [&](V *d, int k, const T (&o)[W]) {
        vst<T>(d, o);
        if (xside) {
            if (mx) vst<T>(d + mx, o);
            if (mx == 1 || mx == -1) vst<T>(d + 2 * mx, o);
        }
        if (yside | zside) {
            if (my) vst<T>(d + my, o);
            if (my == row || my == -row) vst<T>(d + 2 * my, o);
            if (zside) {
                if (g.bc[4] == DVM_BC_PERIODIC) {
                    if (k < 2) vst<T>(d + (long)g.nz * sz, o);
                    else if (k >= g.nz - 2) vst<T>(d - (long)g.nz * sz, o);
                } else {
                    if (k == 0 && g.bc[4] == DVM_BC_ZEROGRAD) { vst<T>(d - sz, o); vst<T>(d - 2 * sz, o); }
                    if (k == g.nz - 1 && g.bc[5] == DVM_BC_ZEROGRAD) { vst<T>(d + sz, o); vst<T>(d + 2 * sz, o); }
                }
            }
        }
    };

    T S0[ZC], S1[ZC], S2[ZC];       // row sums of F, v_x F, v_x^2 F
#pragma unroll
    for (int t = 0; t < ZC; ++t) S0[t] = S1[t] = S2[t] = T(0);
    T cg[ZC];                       // FP32: the row's constant of the exponent
    T kyz[ZC], l5[ZC];              // Shakhov: the row's part of k c.q; 2 log2(A)/log2(e) - 5
    T Er[ZC];                       // FP64: the row's factor of v_y and v_z
    VYZ3<T> cyz{};
    uint32_t keepo = 0, fullo = 0;  // cells to store / without face weights, in upwind order
    bool pz = true;
    int yz = g0 / g.nxg, xg = g0 - yz * g.nxg;
    bool fresh = true;              // a new row (or the split's first group)
    V *const fout = reinterpret_cast<V *>(a.fout);
    for (int gi = 0; gi < ngr; ++gi) {
        if (fresh) {
            cyz = a.vyz[yz];
            pz = cyz.vz >= T(0);
            keepo = (*cellw | *cellw >> 4) & 15u;
            fullo = fullm;
            if (!pz) {
                keepo = __brev(keepo) >> (32 - ZC);
                fullo = __brev(fullo) >> (32 - ZC);
            }
#pragma unroll
            for (int s = 0; s < ZC; ++s) {
                const int t = pz ? s : ZC - 1 - s;      // cells in upwind order
                const T *const cz = cq + t * NCQ * NT + tid;
                if constexpr (F64) {
                    const T dy = cyz.vy - cz[kMxUy * NT], dz = cyz.vz - cz[kMxUz * NT];
                    Er[s] = exp2(-cz[kMxC2 * NT] * (dy * dy + dz * dz));
                } else {
                    const float4 cv = *reinterpret_cast<const float4 *>(coef + (t * NT + tid) * 4);
                    const T dy = cyz.vy - cz[0], dz = cyz.vz - cz[NT];
                    cg[s] = cv.x - cv.z * (dy * dy + dz * dz);
                    if constexpr (SHAK) {
                        const T ux = cv.y / (T(2) * cv.z);
                        kyz[s] = fma(cz[3 * NT], dy, fma(cz[4 * NT], dz, -cz[2 * NT] * ux));
                        l5[s] = T(2.0 / kLog2e) * fma(cv.y * T(0.5), ux, cv.x) - T(5);
                    }
                }
            }
            fresh = false;
        }
        // FP64: the v_x factors of the column's cells, in upwind order
        T fx[F64 ? ZC : 1][W];
        if constexpr (F64) {
#pragma unroll
            for (int s = 0; s < ZC; ++s) {
                const double *const m = mx0 + min(pz ? s : ZC - 1 - s, g.nz - 1 - z0) * (long)(g.nx * g.ny) + xg * W * nc;
#pragma unroll
                for (int e = 0; e < W; ++e) fx[s][e] = __ldg(m + e * nc);
            }
        }
        // the rows of the x flux are read again for every cell (below)
        P vx[2], vx2[2];
        ld_units(vtab + 4 * xg, vx);
        ld_units(vtab + 4 * xg + 1, vx2);
        const int sx0 = xsg[2 * xg], sx1 = xsg[2 * xg + 1];
        const bool mixed = sx0 == 0 || sx1 == 0;
        const int oy = cyz.vy >= T(0) ? px : -px;
        const T ky = T(0.5) * (T(1) - cyz.nuy), kz = T(0.5) * (T(1) - cyz.nuz);
        V *const dst = fout + (long)(g0 + gi) * g.slab;
        // along z, downwind: centre, difference to the upwind cell, limited
        // slope of the upwind face
        P f0[2], dm[2], mi[2];
        {
            P um2[2], um1[2], dd[2];
            wait_full(gi, 0);
            ld_units(ring + slot_of(gi, 0) * PC + c0, um2);
            wait_full(gi, 1);
            ld_units(ring + slot_of(gi, 1) * PC + c0, um1);
            wait_full(gi, 2);
            ld_units(ring + slot_of(gi, 2) * PC + c0, f0);
            release(gi, 0);
            release(gi, 1);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                dm[h] = sub2(f0[h], um1[h]);
                if (MUSCL) {
                    dd[h] = sub2(um1[h], um2[h]);
                    mi[h] = minmod2(dm[h], dd[h]);
                }
            }
        }
#pragma unroll
        for (int s = 0; s < ZC; ++s) {
            const V *const pl = ring + slot_of(gi, s + 2) * PC;
            const int t = pz ? s : ZC - 1 - s;
            P fd[2], dp[2], mo[2];
            wait_full(gi, s + 3);
            if (MUSCL || s + 1 < ZC) {
                ld_units(ring + slot_of(gi, s + 3) * PC + c0, fd);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    dp[h] = sub2(fd[h], f0[h]);
                    if (MUSCL) mo[h] = minmod2(dp[h], dm[h]);
                }
            }
            // the equilibrium, times r in FP64
            T feq[W], r;
            P nnux[2], kx[2];
            ld_units(vtab + 4 * xg + 2, nnux);
            ld_units(vtab + 4 * xg + 3, kx);
            if constexpr (F64) {
                r = cq[(t * NCQ + kMxRel) * NT + tid];
#pragma unroll
                for (int e = 0; e < W; ++e) feq[e] = fx[s][e] * Er[s];
            } else {
                const float4 cv = *reinterpret_cast<const float4 *>(coef + (t * NT + tid) * 4);
                r = cv.w;
#pragma unroll
                for (int e = 0; e < W; ++e) {
                    const T v = unit_lane(vx[e / LN], e % LN);
                    const T x = fma(fma(-cv.z, v, cv.y), v, cg[s]);
                    feq[e] = exp2_state(x);
                    if constexpr (SHAK) {
                        // |c|^2/T - 5 = 2 (log2 A - log2 M) / log2 e - 5
                        const T kc = fma(v, cq[(t * NCQ + 2) * NT + tid], kyz[s]);
                        feq[e] = fma(feq[e] * kc, fma(T(-2.0 / kLog2e), x, l5[s]), feq[e]);
                    }
                }
            }
            T out[W];
            // FULL: no face weights.  Else the weights are 1 where the face's
            // stencil is all gas and 0 elsewhere, and cells that are not
            // plain come out 0.
            const uint32_t mk = *cellw >> (8 + 6 * t);
            const auto update = [&](auto full_) {
                constexpr bool FULL = decltype(full_)::value;
                P yu1[2], yu2[2], yd1[2], xu1[2], xu2[2], xd1[2];
                ld_units(pl + c0 - oy, yu1);
                if (MUSCL) {
                    ld_units(pl + c0 - 2 * oy, yu2);
                    ld_units(pl + c0 + oy, yd1);
                }
                if (sx0 == sx1) {
                    ld_units(pl + c0 - sx0, xu1);
                    if (MUSCL) {
                        ld_units(pl + c0 - 2 * sx0, xu2);
                        ld_units(pl + c0 + sx0, xd1);
                    }
                } else {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int sx = h ? sx1 : sx0;
                        xu1[h] = ld_unit(pl + c0 - sx, h);
                        if (MUSCL) {
                            xu2[h] = ld_unit(pl + c0 - 2 * sx, h);
                            xd1[h] = ld_unit(pl + c0 + sx, h);
                        }
                    }
                }
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    // the differences on units, the rest lane by lane: the
                    // limiter has no packed form, and pairs formed from its
                    // results cost more moves than the packed arithmetic saves
                    const P ax2 = sub2(f0[h], xu1[h]), ay2 = sub2(f0[h], yu1[h]);
                    P bx2, by2, cx2, cy2;
                    if (MUSCL) {
                        bx2 = sub2(xd1[h], f0[h]); cx2 = sub2(xu1[h], xu2[h]);
                        by2 = sub2(yd1[h], f0[h]); cy2 = sub2(yu1[h], yu2[h]);
                    }
                    const bool xp = (h ? sx1 : sx0) > 0, yp = oy > 0;
#pragma unroll
                    for (int l = 0; l < LN; ++l) {
                        const int e = h * LN + l;
                        T dx = unit_lane(ax2, l), dy = unit_lane(ay2, l), dz = unit_lane(dm[h], l);
                        if (MUSCL) {
                            const T bx = unit_lane(bx2, l), cx = unit_lane(cx2, l), by = unit_lane(by2, l), cy = unit_lane(cy2, l);
                            const T kxe = unit_lane(kx[h], l);
                            if constexpr (FULL) {
                                dx = fma(kxe, minmod_diff(bx, dx, cx), dx);
                                dy = fma(ky, minmod_diff(by, dy, cy), dy);
                                dz = fma(kz, unit_lane(mo[h], l) - unit_lane(mi[h], l), dz);
                            } else {
                                const auto w = [&](uint32_t bit, T x) { return (mk & bit) ? x : T(0); };
                                dx = fma(kxe, minmod_diff(bx, dx, cx, w(xp ? 2u : 1u, T(1)), w(xp ? 1u : 2u, T(-1))), dx);
                                dy = fma(ky, minmod_diff(by, dy, cy, w(yp ? 8u : 4u, T(1)), w(yp ? 4u : 8u, T(-1))), dy);
                                dz = fma(w(pz ? 32u : 16u, kz), unit_lane(mo[h], l), dz);
                                dz = fma(w(pz ? 16u : 32u, -kz), unit_lane(mi[h], l), dz);
                            }
                        }
                        const T fc = unit_lane(f0[h], l), q = feq[e];
                        // FP64 (q is r M): the increment first, so that it
                        // rounds at its own size and the sum once
                        T o = F64 ? fma(-r, fc, q) : fma(r, q - fc, fc);
                        o = fma(unit_lane(nnux[h], l), dx, o);
                        o = fma(-cyz.nuy, dy, o);
                        o = fma(-cyz.nuz, dz, o);
                        if (F64) o += fc;
                        if constexpr (!FULL) o = ((*cellw >> t) & 1u) ? o : T(0);
                        out[e] = o;
                    }
                }
            };
            if (F64 || !mixed) {
                if (fullo & (1u << s)) update(std::true_type{});
                else update(std::false_type{});
            } else {
                // a unit whose lanes have v_x of both signs
                const bool py = oy > 0;
                const T yo = (mk & (py ? 8u : 4u)) ? ky : T(0), yi = (mk & (py ? 4u : 8u)) ? ky : T(0);
                const T zo = (mk & (pz ? 32u : 16u)) ? kz : T(0), zi = (mk & (pz ? 16u : 32u)) ? kz : T(0);
                const T *const f = reinterpret_cast<const T *>(pl + c0);
#pragma unroll
                for (int e = 0; e < W; ++e) {
                    const int h = e / LN, l = e % LN;
                    const int sx = unit_lane(vx[h], l) >= T(0) ? W : -W, sy = oy * W;
                    const T fc = unit_lane(f0[h], l);
                    T dx = fc - f[e - sx], dy = fc - f[e - sy], dz = unit_lane(dm[h], l);
                    if (MUSCL) {
                        const T xo = (mk & (sx > 0 ? 2u : 1u)) ? T(1) : T(0), xi = (mk & (sx > 0 ? 1u : 2u)) ? T(1) : T(0);
                        const T tx_ = xo * minmod3(f[e + sx] - fc, dx) - xi * minmod3(dx, f[e - sx] - f[e - 2 * sx]);
                        dx = fma(unit_lane(kx[h], l), tx_, dx);
                        dy = fma(-yi, minmod3(dy, f[e - sy] - f[e - 2 * sy]), fma(yo, minmod3(f[e + sy] - fc, dy), dy));
                        dz = fma(-zi, unit_lane(mi[h], l), fma(zo, unit_lane(mo[h], l), dz));
                    }
                    const T q = feq[e];
                    T o = F64 ? fma(-r, fc, q) : fma(r, q - fc, fc);
                    o = fma(unit_lane(nnux[h], l), dx, o);
                    o = fma(-cyz.nuy, dy, o);
                    o = fma(-cyz.nuz, dz, o);
                    if (F64) o += fc;
                    out[e] = ((*cellw >> t) & 1u) ? o : T(0);
                }
            }
            if (keepo & (1u << s)) store(dst + (pc0 + t * sz), z0 + t, out);
#pragma unroll
            for (int e = 0; e < W; ++e) {
                S0[s] += out[e];
                S1[s] = fma(unit_lane(vx[e / LN], e % LN), out[e], S1[s]);
                S2[s] = fma(unit_lane(vx2[e / LN], e % LN), out[e], S2[s]);
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (s + 1 < ZC) {
                    f0[h] = fd[h];
                    dm[h] = dp[h];
                    if (MUSCL) mi[h] = mo[h];
                }
            }
            release(gi, s + 2);
        }
        release(gi, ZC + 2);
        // the row's moments into the sums, after kFold3 groups at the latest
        if (++xg == g.nxg || gi + 1 == ngr || xg % kFold3 == 0) {
            const T vyz2 = cyz.vy * cyz.vy + cyz.vz * cyz.vz;
#pragma unroll
            for (int s = 0; s < ZC; ++s) {
                T *const ks = ksum + (pz ? s : ZC - 1 - s) * NSUM * NT + tid;
                const T s0 = S0[s], s1 = S1[s], s2 = S2[s];
                const T m[5] = {s0, s1, cyz.vy * s0, cyz.vz * s0, T(0.5) * fma(vyz2, s0, s2)};
#pragma unroll
                for (int q = 0; q < 5; ++q) {
                    Acc<T> acc;
                    acc.s = ks[q * NT];
                    if constexpr (!F64) acc.c = ks[(5 + q) * NT];
                    acc.add(m[q]);
                    ks[q * NT] = acc.s;
                    if constexpr (!F64) ks[(5 + q) * NT] = acc.c;
                }
                S0[s] = S1[s] = S2[s] = T(0);
            }
            if (xg == g.nxg) {
                xg = 0;
                ++yz;
                fresh = true;
            }
        }
    }
    if (bad) atomicExch(&a.err[kErrTimeout], 1);
#pragma unroll 1
    for (int t = 0; t < ZC; ++t) {
        if (!((*cellw >> t | *cellw >> (4 + t)) & 1u)) continue;
        const long cell = ((long)(z0 + t) * g.ny + j) * g.nx + i;
        const T *const ks = ksum + t * NSUM * NT + tid;
        for (int m = 0; m < 5; ++m)
            a.pout[((long)split * 5 + m) * nc + cell] = F64 ? ks[m * NT] : ks[m * NT] - ks[(F64 ? 0 : 5 + m) * NT];
    }
}

// ------------------------------------------------------------ control volumes
struct Cv3Args {
    Grid3D g;
    Geo3D G;
    const int32_t *master;
    const uint16_t *flags;
    const int32_t *spec_list;
    const int32_t *wall_list;
    const int32_t *wslot;
    const int32_t *counts;
    int cap;
    int S;
    int Sin;                  // partial-sum slots of the moments read (S, or 1 for summed moments)
    int gps;
    const void *cvinfo;
    const void *vxt;
    const void *vyz;
    const void *eqp;          // [5][nc] conservative equilibrium parameters, or null
    const void *qh;           // [3][nc] heat flux of the control volume at t^n (Shakhov model, FP32), or null
    double pr1;               // 1 - Pr (Shakhov model)
    int *err;
};

// One member (virtual cell) of a control volume.
struct __align__(16) CvMember3 {
    int pc;                   // slab index
    int mir[6];               // padding mirrors (-1: none)
    int cell;                 // cell index
    int wslot;                // wall slot, -1 if none
    int mask;                 // limiter mask of the six faces
    int live;                 // non-solid (fixed obstacle: always)
    int pad;
    double A[6];              // face areas x-, x+, y-, y+, z-, z+
    double sw, nwx, nwy, nwz; // wall face (sw = 0: none)
    double vol;
};

struct __align__(16) CvInfo3 {
    int nm, ok, pcm, pad;
    double bco;               // dt / S (fixed obstacle: S^n = S^{n+1,*})
    double S;
    CvMember3 mem[kMaxMembers3];
};

// Ordered members of control volume m (cells whose master is m) within the
// window reachable by the master search.
__device__ int gather_members3(const Cv3Args &c, int m, int32_t *mem)
{
    __shared__ int wcnt[8];
    const Grid3D &g = c.g;
    const int R = kMaxWalk, Wd = 2 * kMaxWalk + 1, npos = Wd * Wd * Wd;
    int mi, mj, mk;
    cell_ijk(g, m, mi, mj, mk);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    int total = 0;
    for (int base = 0; base < npos; base += 32 * nw) {
        const int pos = base + warp * 32 + lane;
        bool hit = false;
        int ii = 0, jj = 0, kk = 0;
        if (pos < npos) {
            ii = mi - R + pos % Wd;
            jj = mj - R + (pos / Wd) % Wd;
            kk = mk - R + pos / (Wd * Wd);
            if (ii >= 0 && ii < g.nx && jj >= 0 && jj < g.ny && kk >= 0 && kk < g.nz)
                hit = c.master[((long)kk * g.ny + jj) * g.nx + ii] == m;
        }
        const unsigned bal = __ballot_sync(0xffffffffu, hit);
        if (lane == 0) wcnt[warp] = __popc(bal);
        __syncthreads();
        int off = total;
        for (int w = 0; w < warp; ++w) off += wcnt[w];
        const int rank = off + __popc(bal & ((1u << lane) - 1u));
        if (hit) {
            if (rank < kMaxMembers3) mem[rank] = (kk * g.ny + jj) * g.nx + ii;
            else atomicExch(&c.err[kErrCapacity], 1);
        }
        int add = 0;
        for (int w = 0; w < nw; ++w) add += wcnt[w];
        total += add;
        __syncthreads();
    }
    return total < kMaxMembers3 ? total : kMaxMembers3;
}

// Members are listed in z-major order of the window; the fixed order keeps
// the sums deterministic.  Sorting is not needed: the order only has to be
// the same on every call.
__global__ void __launch_bounds__(256) k_members3(Cv3Args c, CvInfo3 *info)
{
    __shared__ int32_t mem[kMaxMembers3];
    const Grid3D &g = c.g;
    const int n = min(c.counts[0], c.cap);
    for (int idx = blockIdx.x; idx < n; idx += gridDim.x) {
        const int m = c.spec_list[idx];
        const int nm = gather_members3(c, m, mem);
        CvInfo3 &I = info[idx];
        if (threadIdx.x < nm) {
            const int q = mem[threadIdx.x];
            CvMember3 &M = I.mem[threadIdx.x];
            int i, j, k;
            cell_ijk(g, q, i, j, k);
            M.cell = q;
            M.pc = nbr3(g, i, j, k);
            mirrors3(g, i, j, k, M.mir);
            const long xf = ((long)k * g.ny + j) * (g.nx + 1) + i;
            const long yf = ((long)k * (g.ny + 1) + j) * g.nx + i;
            const long zf = ((long)k * g.ny + j) * g.nx + i;
            M.A[0] = c.G.ax[xf]; M.A[1] = c.G.ax[xf + 1];
            M.A[2] = c.G.ay[yf]; M.A[3] = c.G.ay[yf + g.nx];
            M.A[4] = c.G.az[zf]; M.A[5] = c.G.az[zf + (long)g.nx * g.ny];
            M.wslot = c.wslot[q];
            const bool wall = M.wslot >= 0;
            M.sw = wall ? c.G.sw[q] : 0.0;
            M.nwx = c.G.nwx[q]; M.nwy = c.G.nwy[q]; M.nwz = c.G.nwz[q];
            M.vol = c.G.vol[q];
            M.mask = (c.flags[q] >> kMaskShift3) & 0x3F;
            M.live = c.G.type[q] != DVM_SOLID;
            M.pad = 0;
            if (q == m) I.pcm = M.pc;
        }
        if (threadIdx.x == 0) {
            double S = 0;
            for (int t = 0; t < nm; ++t) S += c.G.vol[mem[t]];
            I.nm = nm;
            I.ok = S > 0;
            I.S = S;
            I.bco = S > 0 ? g.dt / S : 0.0;
            I.pad = 0;
            if (!(S > 0)) atomicExch(&c.err[kErrGeometry], 1);
        }
        __syncthreads();
    }
}

__device__ __forceinline__ void load_info3(const CvInfo3 *src, CvInfo3 *dst)
{
    static_assert(sizeof(CvInfo3) % 16 == 0, "CvInfo3 is copied in 16-byte words");
    const int4 *s4 = reinterpret_cast<const int4 *>(src);
    int4 *d4 = reinterpret_cast<int4 *>(dst);
    for (int q = threadIdx.x; q < (int)(sizeof(CvInfo3) / 16); q += blockDim.x) d4[q] = __ldg(s4 + q);
    __syncthreads();
}

template <typename T>
__device__ __forceinline__ T face_flux3(T L, T v, T nu, T fAA, T fA, T fB, T fBB, bool muscl)
{
    if (!muscl) return L * (fmin(v, T(0)) * fB + fmax(v, T(0)) * fA);
    T fr;
    if (v > T(0)) fr = fA + T(0.5) * (T(1) - nu) * minmod(fB - fA, fA - fAA);
    else if (v < T(0)) fr = fB - T(0.5) * (T(1) - nu) * minmod(fBB - fB, fB - fA);
    else return T(0);
    return L * (v * fr);
}

template <typename T>
__device__ __forceinline__ void write_split_partials3(T *part, int s, long nc, long k, const T (&t)[5])
{
#pragma unroll
    for (int m = 0; m < 5; ++m) part[((long)s * 5 + m) * nc + k] = t[m];
}

// Velocity of padded index p from the tables.
template <typename T>
__device__ __forceinline__ void vel3(const Grid3D &g, const VX3<T> *vxt, const VYZ3<T> *vyz, int p, T &vx, T &vy,
                                     T &vz, T &nux, T &nuy, T &nuz)
{
    const int grp = p / g.W, e = p - grp * g.W;
    const int yz = grp / g.nxg;
    const VX3<T> cx = vxt[(grp - yz * g.nxg) * g.W + e];
    const VYZ3<T> c = vyz[yz];
    vx = cx.vx; nux = cx.nux;
    vy = c.vy; vz = c.vz; nuy = c.nuy; nuz = c.nuz;
}

// Fusion (3D form of Eq. FusionDD): F_CV = sum vol F / S over a merged
// control volume, written back to every member, with the moment sums.  One
// work item is one control volume and one velocity split.
template <typename T>
__global__ void __launch_bounds__(256) k_fusion3(Cv3Args c, T *f, T *part)
{
    __shared__ T red[8 * 2];
    const Grid3D &g = c.g;
    const CvInfo3 *info = reinterpret_cast<const CvInfo3 *>(c.cvinfo);
    const VX3<T> *vxt = reinterpret_cast<const VX3<T> *>(c.vxt);
    const VYZ3<T> *vyz = reinterpret_cast<const VYZ3<T> *>(c.vyz);
    const long nc = (long)g.nx * g.ny * g.nz;
    const int n = min(c.counts[0], c.cap) * c.S;
    for (int item = blockIdx.x; item < n; item += gridDim.x) {
        const CvInfo3 &I = info[item / c.S];
        const int sp = item % c.S;
        const int nm = I.nm;
        if (nm <= 1) continue;
        const int v0 = sp * c.gps * g.W, v1 = min(g.nvp, v0 + c.gps * g.W);
        const double S = I.S;
        Acc<T> a[5];
        for (int p = v0 + threadIdx.x; p < v1; p += blockDim.x) {
            double acc = 0;
            for (int t = 0; t < nm; ++t) acc += I.mem[t].vol * (double)f[pidx3(g, p, I.mem[t].pc)];
            const T fcv = (T)(acc / S);
            for (int t = 0; t < nm; ++t) {
                f[pidx3(g, p, I.mem[t].pc)] = fcv;
                for (int u = 0; u < 6; ++u)
                    if (I.mem[t].mir[u] >= 0) f[pidx3(g, p, I.mem[t].mir[u])] = fcv;
            }
            T vx, vy, vz, nux, nuy, nuz;
            vel3(g, vxt, vyz, p, vx, vy, vz, nux, nuy, nuz);
            a[0].add(fcv); a[1].add(vx * fcv); a[2].add(vy * fcv); a[3].add(vz * fcv);
            a[4].add(T(0.5) * (vx * vx + vy * vy + vz * vz) * fcv);
        }
        T t[5];
#pragma unroll
        for (int m = 0; m < 5; ++m) t[m] = block_acc(a[m], red);
        if (threadIdx.x < nm) write_split_partials3<T>(part, sp, nc, I.mem[threadIdx.x].cell, t);
        __syncthreads();
    }
}

// Wall density phi (zero net mass flux across the wall face), stress
// Sigma = sum (v - u_w)(v - u_w)^T F_w dv and the force Sigma n_w S_w on the
// body (3D forms of Eqs. BoundaryDDv, StressTensorDD, eq-force), torque about
// the z axis through the centre (Eq. eq-torque), u_w = u_c + omega e_z x
// (r - c) (Eq. uwDD).  One block per wall cell: products and compensated sums
// in the state precision over all velocities, a thread a velocity group (one
// vector, one pair of divisions for its W velocities) and the 14 sums merged
// together (64^3 x 20^3: 0.175 -> 0.135 ms a launch), phi and the stress in
// FP64 by thread 0.  The last block sums the cells in list order into the body
// record and the history.  (phi, u_w, T_w) of each wall cell are left for
// the control-volume kernel.
template <typename T>
// mode 0: the whole wall step; a velocity split runs mode 1 (this rank's 14
// sums of every wall cell into xw[14 * slot], FP64) and, after the caller's
// sum over the ranks, mode 2 (the rest from the summed values).
__global__ void __launch_bounds__(256) k_wall3(Cv3Args c, BodyParams b, BodyDev *body, const T *f, double *wdat,
                                               double *wcontrib, int *ticket, double *hist, int mode, double *xw)
{
    constexpr int W = Vec<T>::W;
    using V = typename Vec<T>::type;
    __shared__ double red[8 * 8];
    __shared__ T ex[kMaxAxisNv], ey[kMaxAxisNv], ez[kMaxAxisNv];
    __shared__ T wsc[8];
    __shared__ T wred[8 * 3 * 14];
    __shared__ bool last;
    const Grid3D &g = c.g;
    const VX3<T> *vxt = reinterpret_cast<const VX3<T> *>(c.vxt);
    const VYZ3<T> *vyz = reinterpret_cast<const VYZ3<T> *>(c.vyz);
    const int nw = min(c.counts[1], c.cap);
    const double omega = body->omega;
    const int tid = threadIdx.x;
    for (int idx = blockIdx.x; idx < nw; idx += gridDim.x) {
        const int q = c.wall_list[idx];
        const double rx = c.G.rwx[q] - b.cx, ry = c.G.rwy[q] - b.cy;
        const double uwx = b.vbx - ry * omega, uwy = b.vby + rx * omega, uwz = 0.0;
        double rr[14];
        if (mode == 2) {
#pragma unroll
            for (int t = 0; t < 14; ++t) rr[t] = xw[14L * idx + t];
        } else {
        if (tid == 0) {
            wsc[0] = (T)uwx; wsc[1] = (T)uwy; wsc[2] = (T)uwz;
            wsc[3] = (T)c.G.nwx[q]; wsc[4] = (T)c.G.nwy[q]; wsc[5] = (T)c.G.nwz[q];
            wsc[6] = (T)(2.0 * b.Tw);
            const double a2 = 2.0 * kPi * b.Tw;
            wsc[7] = (T)(1.0 / (a2 * sqrt(a2)));
        }
        __syncthreads();
        const T ux = wsc[0], uy = wsc[1], uz = wsc[2], nx = wsc[3], ny = wsc[4], nz = wsc[5], twoTw = wsc[6];
        const T cm = wsc[7];
        // separable Maxwellian M[1, u_w, T_w] = cm ex[p1] ey[p2] ez[p3]
        for (int t = tid; t < g.nvx + g.nvy + g.nvz; t += blockDim.x) {
            if (t < g.nvx) { const T d = vxt[t].vx - ux; ex[t] = dexp(-(d * d) / twoTw); }
            else if (t < g.nvx + g.nvy) {
                const int p2 = t - g.nvx;
                const T d = vyz[p2].vy - uy;
                ey[p2] = dexp(-(d * d) / twoTw);
            } else {
                const int p3 = t - g.nvx - g.nvy;
                const T d = vyz[p3 * g.nvy].vz - uz;
                ez[p3] = dexp(-(d * d) / twoTw);
            }
        }
        __syncthreads();
        const V *fv = reinterpret_cast<const V *>(f) + pcell3(g, q);
        // a[0] = sum_{c>0} c F, a[1] = sum_{c<0} c M, a[2..7] = sum_{c<0} (v-u_w)(v-u_w) M,
        // a[8..13] = sum_{c>0} (v-u_w)(v-u_w) F   (xx, xy, xz, yy, yz, zz)
        Acc<T> a[14];
        for (int grp = tid; grp < g.ngrp; grp += blockDim.x) {
            const int r = grp / g.nxg, x0 = (grp - r * g.nxg) * W;
            const int p3 = r / g.nvy, p2 = r - p3 * g.nvy;
            const T ay = vyz[r].vy - uy, az = vyz[r].vz - uz;
            T F[W];
            vld<T>(fv + (long)grp * g.slab, F);
#pragma unroll
            for (int e = 0; e < W; ++e) {
                const int p1 = x0 + e;
                if (p1 >= g.nvx) continue;
                const T ax = vxt[p1].vx - ux;
                const T cp = ax * nx + ay * ny + az * nz;
                if (cp > T(0)) {
                    const T fv1 = F[e];
                    a[0].add(cp * fv1);
                    a[8].add(ax * ax * fv1); a[9].add(ax * ay * fv1); a[10].add(ax * az * fv1);
                    a[11].add(ay * ay * fv1); a[12].add(ay * az * fv1); a[13].add(az * az * fv1);
                } else if (cp < T(0)) {
                    const T m1 = cm * ex[p1] * ey[p2] * ez[p3];
                    a[1].add(cp * m1);
                    a[2].add(ax * ax * m1); a[3].add(ax * ay * m1); a[4].add(ax * az * m1);
                    a[5].add(ay * ay * m1); a[6].add(ay * az * m1); a[7].add(az * az * m1);
                }
            }
        }
        T rv[14];
        group_acc(a, rv, wred, blockDim.x >> 5);
#pragma unroll
        for (int t = 0; t < 14; ++t) rr[t] = (double)rv[t];
        if (mode == 1) {
            if (tid == 0)
#pragma unroll
                for (int t = 0; t < 14; ++t) xw[14L * idx + t] = rr[t];
            __syncthreads();
            continue;
        }
        }
        if (tid == 0) {
            const double dv = g.dv;
            const double phi = -(rr[0] * dv) / (rr[1] * dv);
            double S6[6];
            for (int t = 0; t < 6; ++t) S6[t] = (phi * rr[2 + t] + rr[8 + t]) * dv;
            const double nxd = c.G.nwx[q], nyd = c.G.nwy[q], nzd = c.G.nwz[q], sw = c.G.sw[q];
            const double fx = (S6[0] * nxd + S6[1] * nyd + S6[2] * nzd) * sw;
            const double fy = (S6[1] * nxd + S6[3] * nyd + S6[4] * nzd) * sw;
            const double fz = (S6[2] * nxd + S6[4] * nyd + S6[5] * nzd) * sw;
            double *wc = wcontrib + 4L * idx;
            wc[0] = fx; wc[1] = fy; wc[2] = fz; wc[3] = rx * fy - ry * fx;
            double *d = wdat + 6L * idx;
            d[0] = phi; d[1] = uwx; d[2] = uwy; d[3] = uwz; d[4] = b.Tw; d[5] = 0;
        }
        __syncthreads();
    }
    if (mode == 1) return;
    __threadfence();
    __syncthreads();
    if (tid == 0) last = atomicAdd(ticket, 1) == (int)gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    double fx = 0, fy = 0, fz = 0, tq = 0;
    for (int t = tid; t < nw; t += blockDim.x) {
        fx += wcontrib[4 * t]; fy += wcontrib[4 * t + 1]; fz += wcontrib[4 * t + 2]; tq += wcontrib[4 * t + 3];
    }
    fx = block_sum(fx, red); fy = block_sum(fy, red + 8); fz = block_sum(fz, red + 16); tq = block_sum(tq, red + 24);
    if (tid == 0) {
        body->F[0] = fx; body->F[1] = fy; body->F[2] = fz; body->torque = tq;
        double *h = hist + 6 * (body->step % kHistCap);
        h[0] = fx; h[1] = fy; h[2] = fz; h[3] = tq; h[4] = body->theta; h[5] = body->omega;
        body->step += 1;
        *ticket = 0;
    }
}

// Explicit update of one control volume (Eq. eq-schema3D): fluxes across the
// six faces of every member and across its wall face with the diffuse state
// F_w = phi M[1, u_w, T_w] on incoming velocities, relaxation, distribution
// to the members and the moment sums of the velocity split.  One work item is
// one control volume and one split, one thread a velocity group: the 13 values
// of the stencil are vectors, so the addresses and the member's record are
// read once for its W velocities, and the five sums are merged together.  It is
// bound by latency (32% of the SM's issue rate, a fifth of its warps).  One
// thread a velocity before: 64^3 x 20^3 FP32 0.65 -> 0.50 ms a launch, 45 x 50 x
// 37 cells, 14 x 15 x 13 velocities 0.24 -> 0.11 ms, 40^3 x 12^3 FP64 0.59 ->
// 0.44 ms (more registers: one block of 256 per SM; with two it spills).
constexpr int kSpec3Threads = 256;

// Threads of a block for splits of gps groups: as few rounds as 256 threads
// need, of equal length (a split of 286 groups: two rounds of 160 threads).
inline int spec3_threads(int gps)
{
    const int rounds = (gps + kSpec3Threads - 1) / kSpec3Threads;
    return ((gps + rounds - 1) / rounds + 31) / 32 * 32;
}

template <typename T>
__global__ void __launch_bounds__(kSpec3Threads, sizeof(T) == 4 ? 2 : 1)
    k_special3(Cv3Args c, const T *fin, T *fout, const T *pin, T *pout, const double *wdat)
{
    constexpr int W = Vec<T>::W;
    using V = typename Vec<T>::type;
    __shared__ T red[8 * 3 * 5];
    __shared__ __align__(16) CvInfo3 I;
    const Grid3D &g = c.g;
    const CvInfo3 *info = reinterpret_cast<const CvInfo3 *>(c.cvinfo);
    const VX3<T> *vxt = reinterpret_cast<const VX3<T> *>(c.vxt);
    const VYZ3<T> *vyz = reinterpret_cast<const VYZ3<T> *>(c.vyz);
    const long nc = (long)g.nx * g.ny * g.nz;
    const int n = min(c.counts[0], c.cap) * c.S;
    const int sy = g.nx + 4, sz = (g.nx + 4) * (g.ny + 4);
    for (int item = blockIdx.x; item < n; item += gridDim.x) {
        const int idx = item / c.S, sp = item % c.S;
        load_info3(info + idx, &I);
        if (!I.ok) { __syncthreads(); continue; }
        const int nm = I.nm;
        const int g0 = sp * c.gps, g1 = min(g.ngrp, g0 + c.gps);
        const int m = c.spec_list[idx];
        T s[5];
        gather_partials3(pin, c.Sin, nc, m, s);
        T rho, ux, uy, uz, tmp;
        if (!primitives3<T>(pick<T>(g.dv_f, g.dv), s, rho, ux, uy, uz, tmp) && threadIdx.x == 0 && sp == 0)
            atomicExch(&c.err[kErrNonphys], 1);
        const T bco = (T)I.bco, r = pick<T>(g.dt_tau0_f, g.dt_tau0) * rho;
        if (c.eqp) {
            const T *e = static_cast<const T *>(c.eqp);
            rho = e[m]; ux = e[nc + m]; uy = e[2 * nc + m]; uz = e[3 * nc + m]; tmp = e[4 * nc + m];
        }
        const T A = rho * norm3(tmp);
        const T i2T = T(1) / (T(2) * tmp);
        // Shakhov (Sec. 2.1): k q with the heat flux of the control volume
        T kqx = 0, kqy = 0, kqz = 0;
        if (c.qh) {
            const T *qh = static_cast<const T *>(c.qh);
            const T kk = T(c.pr1) / (T(5) * rho * tmp * tmp);
            kqx = kk * qh[m];
            kqy = kk * qh[nc + m];
            kqz = kk * qh[2 * nc + m];
        }
        Acc<T> acc[5];
        for (int grp = g0 + threadIdx.x; grp < g1; grp += blockDim.x) {
            const int yz = grp / g.nxg, x0 = (grp - yz * g.nxg) * W;
            const VYZ3<T> cy = vyz[yz];
            T vx[W], nux[W];
#pragma unroll
            for (int e = 0; e < W; ++e) {
                const VX3<T> cx = vxt[x0 + e];
                vx[e] = cx.vx;
                nux[e] = cx.nux;
            }
            const V *fg = reinterpret_cast<const V *>(fin) + (long)grp * g.slab;
            T R[W] = {};
            for (int t = 0; t < nm; ++t) {
                const CvMember3 &M = I.mem[t];
                if (!M.live) continue;
                const V *fp = fg + M.pc;
                T fc[W];
                vld<T>(fp, fc);
                T xm1[W], xp1[W], ym1[W], yp1[W], zm1[W], zp1[W];
                vld<T>(fp - 1, xm1); vld<T>(fp + 1, xp1);
                vld<T>(fp - sy, ym1); vld<T>(fp + sy, yp1);
                vld<T>(fp - sz, zm1); vld<T>(fp + sz, zp1);
                T xm2[W] = {}, xp2[W] = {}, ym2[W] = {}, yp2[W] = {}, zm2[W] = {}, zp2[W] = {};
                if (M.mask) {
                    vld<T>(fp - 2, xm2); vld<T>(fp + 2, xp2);
                    vld<T>(fp - 2 * sy, ym2); vld<T>(fp + 2 * sy, yp2);
                    vld<T>(fp - 2 * sz, zm2); vld<T>(fp + 2 * sz, zp2);
                }
                T Fw[W] = {};
                if (M.wslot >= 0) {
                    const double *d = wdat + 6L * M.wslot;
                    const T phi = (T)d[0], uwx = (T)d[1], uwy = (T)d[2], uwz = (T)d[3], Tw = (T)d[4];
                    const T ay = cy.vy - uwy, az = cy.vz - uwz;
                    const T n3 = norm3(Tw);
#pragma unroll
                    for (int e = 0; e < W; ++e) {
                        const T ax = vx[e] - uwx;
                        const T cw = ax * (T)M.nwx + ay * (T)M.nwy + az * (T)M.nwz;
                        const T m1 = dexp(-(ax * ax + ay * ay + az * az) / (T(2) * Tw)) * n3;
                        Fw[e] = (T)M.sw * (fmin(cw, T(0)) * (phi * m1) + fmax(cw, T(0)) * fc[e]);
                    }
                }
                const bool mxm = M.mask & 1, mxp = M.mask & 2, mym = M.mask & 4, myp = M.mask & 8;
                const bool mzm = M.mask & 16, mzp = M.mask & 32;
#pragma unroll
                for (int e = 0; e < W; ++e) {
                    const T Fxp = face_flux3<T>((T)M.A[1], vx[e], nux[e], xm1[e], fc[e], xp1[e], xp2[e], mxp);
                    const T Fxm = face_flux3<T>((T)M.A[0], vx[e], nux[e], xm2[e], xm1[e], fc[e], xp1[e], mxm);
                    const T Fyp = face_flux3<T>((T)M.A[3], cy.vy, cy.nuy, ym1[e], fc[e], yp1[e], yp2[e], myp);
                    const T Fym = face_flux3<T>((T)M.A[2], cy.vy, cy.nuy, ym2[e], ym1[e], fc[e], yp1[e], mym);
                    const T Fzp = face_flux3<T>((T)M.A[5], cy.vz, cy.nuz, zm1[e], fc[e], zp1[e], zp2[e], mzp);
                    const T Fzm = face_flux3<T>((T)M.A[4], cy.vz, cy.nuz, zm2[e], zm1[e], fc[e], zp1[e], mzm);
                    R[e] += (Fxp - Fxm) + (Fyp - Fym) + (Fzp - Fzm) + Fw[e];
                }
            }
            T fn[W];
            vld<T>(fg + I.pcm, fn);
            const T dyu = cy.vy - uy, dzu = cy.vz - uz;
#pragma unroll
            for (int e = 0; e < W; ++e) {
                const T fcv = fn[e], dxu = vx[e] - ux;
                const T c2u = dxu * dxu + dyu * dyu + dzu * dzu;
                T feq = A * dexp(-c2u * i2T);
                if (c.qh) feq *= fma(kqx * dxu + kqy * dyu + kqz * dzu, c2u * T(2) * i2T - T(5), T(1));
                fn[e] = fcv - bco * R[e] + r * (feq - fcv);
                acc[0].add(fn[e]); acc[1].add(vx[e] * fn[e]); acc[2].add(cy.vy * fn[e]); acc[3].add(cy.vz * fn[e]);
                acc[4].add(T(0.5) * (vx[e] * vx[e] + cy.vy * cy.vy + cy.vz * cy.vz) * fn[e]);
            }
            V *og = reinterpret_cast<V *>(fout) + (long)grp * g.slab;
            for (int t = 0; t < nm; ++t) {
                const CvMember3 &M = I.mem[t];
                vst<T>(og + M.pc, fn);
                for (int u = 0; u < 6; ++u)
                    if (M.mir[u] >= 0) vst<T>(og + M.mir[u], fn);
            }
        }
        T t5[5];
        group_acc(acc, t5, red, blockDim.x >> 5);
        if (threadIdx.x < nm) write_split_partials3<T>(pout, sp, nc, I.mem[threadIdx.x].cell, t5);
        __syncthreads();
    }
}

// ------------------------------------------------------------ state services
// Moment sums of a cell over a chunk of the velocity groups: F, v_x F, v_y F,
// v_z F and |v|^2/2 F (Eq. MacroscopicTD).  The lanes of a warp are 32 cells
// consecutive in the grid (a row may end inside a warp: 45-cell rows took 64
// lanes in tiles of a row), so a group's vectors are whole lines but at row
// ends; warp threadIdx.y takes the threadIdx.y-th of kMomChunks chunks, kMomBatch
// groups' loads in flight.  FP32, bound by memory: sums plain over a group and
// compensated across groups.  FP64, bound by its pipe: the sums of an x-row of
// velocities first, then its v_y and v_z terms once (5 operations a velocity in
// place of 10; 40^3 x 12^3: 2.7 ms before, 1.73 now).
template <typename T>
__device__ __forceinline__ void state_sums3d(const Grid3D &g, const T *f, const VX3<T> *vxt, const VYZ3<T> *vyz,
                                             long cell, Acc<T> (&s)[5])
{
    constexpr int W = Vec<T>::W;
    using V = typename Vec<T>::type;
    if (cell >= (long)g.nx * g.ny * g.nz) return;
    const int gps = (g.ngrp + kMomChunks - 1) / kMomChunks;
    const int q0 = threadIdx.y * gps, q1 = min(q0 + gps, g.ngrp);
    if (q0 >= q1) return;
    const V *fv = reinterpret_cast<const V *>(f) + pcell3(g, (int)cell);
    int r = q0 / g.nxg, xg = q0 - r * g.nxg;
    T t0 = 0, t1 = 0, t2 = 0;
    for (int q = q0; q < q1; q += kMomBatch) {
        T a[kMomBatch][W];
#pragma unroll
        for (int b = 0; b < kMomBatch; ++b)
            if (q + b < q1) vld<T>(fv + (long)(q + b) * g.slab, a[b]);
#pragma unroll
        for (int b = 0; b < kMomBatch; ++b) {
            if (q + b >= q1) break;
#pragma unroll
            for (int e = 0; e < W; ++e) {
                const int p1 = xg * W + e;
                if (p1 >= g.nvx) continue;
                const T vx = vxt[p1].vx;
                t0 += a[b][e];
                t1 += vx * a[b][e];
                t2 += vx * vx * a[b][e];
            }
            const bool row = ++xg == g.nxg;
            if (sizeof(T) == 4 || row || q + b == q1 - 1) {
                const VYZ3<T> cy = vyz[r];
                s[0].add(t0);
                s[1].add(t1);
                s[2].add(cy.vy * t0);
                s[3].add(cy.vz * t0);
                s[4].add(T(0.5) * fma(cy.vy * cy.vy + cy.vz * cy.vz, t0, t2));
                t0 = t1 = t2 = 0;
            }
            if (row) {
                xg = 0;
                ++r;
            }
        }
    }
}

// Partial moment sums of a state (set-up, not the time step): the whole sum
// goes to split 0, zeros to the others and to solid cells.
template <typename T>
__global__ void __launch_bounds__(32 * kMomChunks) k_partials3(Grid3D g, int S, const T *f, const VX3<T> *vxt,
                                                               const VYZ3<T> *vyz, T *part, const int8_t *type,
                                                               int *err)
{
    const long nc = (long)g.nx * g.ny * g.nz, cell = (long)blockIdx.x * 32 + threadIdx.x;
    Acc<T> s[5];
    state_sums3d<T>(g, f, vxt, vyz, cell, s);
    merge_chunks<T, 5>(s);
    if (threadIdx.y != 0 || cell >= nc) return;
    const bool keep = type[cell] != DVM_SOLID;
    T v[5];
#pragma unroll
    for (int m = 0; m < 5; ++m) v[m] = keep ? s[m].value() : T(0);
    if (keep) {
        T rho, ux, uy, uz, tmp;
        if (!primitives3<T>(pick<T>(g.dv_f, g.dv), v, rho, ux, uy, uz, tmp)) atomicExch(&err[kErrNonphys], 1);
    }
    for (int q = 0; q < S; ++q)
#pragma unroll
        for (int m = 0; m < 5; ++m) part[((long)q * 5 + m) * nc + cell] = q == 0 ? v[m] : T(0);
}

// Check of a state from the moment sums that the step left with it, as in 2D.
template <typename T>
__global__ void k_check3(Grid3D g, int S, const T *part, const int8_t *type, int *err)
{
    const long nc = (long)g.nx * g.ny * g.nz, cell = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (cell >= nc || type[cell] == DVM_SOLID) return;
    T s[5], rho, ux, uy, uz, tmp;
    gather_partials3(part, S, nc, cell, s);
    if (!primitives3<T>(pick<T>(g.dv_f, g.dv), s, rho, ux, uy, uz, tmp)) atomicExch(&err[kErrNonphys], 1);
}

// Moments for output: rho, ux, uy, uz, T per cell, formed in FP64 from the
// sums (compensated in the state precision).
template <typename T>
__global__ void __launch_bounds__(32 * kMomChunks) k_moments_out3(Grid3D g, const T *f, const VX3<T> *vxt,
                                                                  const VYZ3<T> *vyz, double *out)
{
    const long nc = (long)g.nx * g.ny * g.nz, cell = (long)blockIdx.x * 32 + threadIdx.x;
    Acc<T> s[5];
    state_sums3d<T>(g, f, vxt, vyz, cell, s);
    merge_chunks<T, 5>(s);
    if (threadIdx.y != 0 || cell >= nc) return;
    double *o5 = out + cell * 5;
    double d[5];
#pragma unroll
    for (int m = 0; m < 5; ++m) d[m] = (double)s[m].s - (double)s[m].c;
    const double rho = d[0] * g.dv;
    if (!(rho > 0)) {
        for (int q = 0; q < 5; ++q) o5[q] = 0;
        return;
    }
    const double ux = d[1] * g.dv / rho, uy = d[2] * g.dv / rho, uz = d[3] * g.dv / rho;
    o5[0] = rho; o5[1] = ux; o5[2] = uy; o5[3] = uz;
    o5[4] = (2.0 * (d[4] * g.dv) / rho - (ux * ux + uy * uy + uz * uz)) / 3.0;
}

// Implicit relaxation of the semi-implicit scheme (Eq. ImpSchemeDD) in 3D,
// after a transport pass without relaxation: every gas cell relaxes towards
// the Maxwellian of the moments of its transported values (mom, Smom slots:
// this context's partial sums, or those summed over the ranks of a velocity
// split), F = (F* + nu M) / (1 + nu) with nu = (dt / tau0) rho, in place and
// in its padding mirrors; the partial sums part become those of this
// context's relaxed values.
// Block = 32 consecutive cells of an x-row x kMomChunks warps, one chunk of
// the velocity groups each.
template <typename T, bool SHAK>
__global__ void __launch_bounds__(32 * kMomChunks) k_imex3(Grid3D g, int S, T dt_tau0, T *f, const VX3<T> *vxt,
                                                           const VYZ3<T> *vyz, const T *mom, int Smom, T *part,
                                                           const int8_t *type, const T *eqp, T Pr, int *err)
{
    // SHAK: the Shakhov model (Sec. 2.1) with the heat flux at t^{n+1},
    // q = q_T / (1 + nu Pr), q_T = sum c |c|^2/2 F dv of the transported
    // values; F_S = M [1 + (1 - Pr) c.q (|c|^2/T - 5) / (5 rho T^2)]
    constexpr int W = Vec<T>::W;
    using V = typename Vec<T>::type;
    __shared__ T qsh[3][32];
    const int i = blockIdx.x * 32 + threadIdx.x, j = blockIdx.y, k = blockIdx.z;
    const long nc = (long)g.nx * g.ny * g.nz, cell = ((long)k * g.ny + j) * g.nx + i;
    bool gas = i < g.nx && type[cell] != DVM_SOLID;
    T s[5] = {T(0), T(0), T(0), T(0), T(0)};
    if (gas) gather_partials3(mom, Smom, nc, cell, s);
    T rho = 0, ux = 0, uy = 0, uz = 0, tmp = 0;
    if (gas && !primitives3<T>(pick<T>(g.dv_f, g.dv), s, rho, ux, uy, uz, tmp)) {
        if (threadIdx.y == 0) atomicExch(&err[kErrNonphys], 1);
        gas = false;
    }
    Acc<T> a5[5];
    const int gps = (g.ngrp + kMomChunks - 1) / kMomChunks;
    const int q0 = threadIdx.y * gps, q1 = min(q0 + gps, g.ngrp);
    const long pc = nbr3(g, i, j, k);
    V *fv = reinterpret_cast<V *>(f);
    T qx = 0, qy = 0, qz = 0;
    if constexpr (SHAK) {
        Acc<T> hq[3];
        if (gas) {
            int r = q0 / g.nxg, xg = q0 - r * g.nxg;
            for (int q = q0; q < q1; ++q) {
                T a[W];
                vld<T>(fv + (long)q * g.slab + pc, a);
                const VYZ3<T> cy = vyz[r];
                const T dy = cy.vy - uy, dz = cy.vz - uz, dyz = dy * dy + dz * dz;
                T t0 = 0, t1 = 0;
#pragma unroll
                for (int e = 0; e < W; ++e) {
                    const int p1 = xg * W + e;
                    if (p1 >= g.nvx) continue;
                    const T dx = vxt[p1].vx - ux, w = T(0.5) * (dx * dx + dyz) * a[e];
                    t0 += dx * w;
                    t1 += w;
                }
                hq[0].add(t0);
                hq[1].add(dy * t1);
                hq[2].add(dz * t1);
                if (++xg == g.nxg) {
                    xg = 0;
                    ++r;
                }
            }
        }
        merge_chunks<T, 3>(hq);
        if (threadIdx.y == 0) {
            const T rel = pick<T>(g.dv_f, g.dv) / (T(1) + dt_tau0 * rho * Pr);
#pragma unroll
            for (int d = 0; d < 3; ++d) qsh[d][threadIdx.x] = hq[d].value() * rel;
        }
        __syncthreads();
        qx = qsh[0][threadIdx.x];
        qy = qsh[1][threadIdx.x];
        qz = qsh[2][threadIdx.x];
    }
    if (gas && q0 < q1) {
        const T nu = dt_tau0 * rho, inv = T(1) / (T(1) + nu);
        if (eqp) {
            // conservative equilibrium of the transported state (Sec. 3.1)
            rho = eqp[cell]; ux = eqp[nc + cell]; uy = eqp[2 * nc + cell]; uz = eqp[3 * nc + cell];
            tmp = eqp[4 * nc + cell];
        }
        const T A = rho * norm3(tmp), c2 = T(kLog2e) / (T(2) * tmp);
        const T kk = SHAK ? (T(1) - Pr) / (T(5) * rho * tmp * tmp) : T(0), iT = T(1) / tmp;
        int mir[6];
        mirrors3(g, i, j, k, mir);
        int r = q0 / g.nxg, xg = q0 - r * g.nxg;
#pragma unroll 2
        for (int q = q0; q < q1; ++q) {
            V *pa = fv + (long)q * g.slab;
            T a[W];
            vld<T>(pa + pc, a);
            const VYZ3<T> cy = vyz[r];
            const T dyz = (cy.vy - uy) * (cy.vy - uy) + (cy.vz - uz) * (cy.vz - uz);
            const T hyz = kk * ((cy.vy - uy) * qy + (cy.vz - uz) * qz);
            T t0 = 0, t1 = 0, t2 = 0;
#pragma unroll
            for (int e = 0; e < W; ++e) {
                const int p1 = xg * W + e;
                if (p1 >= g.nvx) continue;
                const T vx = vxt[p1].vx, dx = vx - ux;
                T M = A * exp2_state(-(dx * dx + dyz) * c2);
                if constexpr (SHAK) M *= T(1) + (kk * dx * qx + hyz) * ((dx * dx + dyz) * iT - T(5));
                a[e] = (a[e] + nu * M) * inv;
                t0 += a[e];
                t1 += vx * a[e];
                t2 += vx * vx * a[e];
            }
            vst<T>(pa + pc, a);
#pragma unroll
            for (int m = 0; m < 6; ++m)
                if (mir[m] >= 0) vst<T>(pa + mir[m], a);
            a5[0].add(t0);
            a5[1].add(t1);
            a5[2].add(cy.vy * t0);
            a5[3].add(cy.vz * t0);
            a5[4].add(T(0.5) * fma(cy.vy * cy.vy + cy.vz * cy.vz, t0, t2));
            if (++xg == g.nxg) {
                xg = 0;
                ++r;
            }
        }
    }
    merge_chunks<T, 5>(a5);
    if (threadIdx.y != 0 || i >= g.nx) return;
    for (int q = 0; q < S; ++q)
#pragma unroll
        for (int m = 0; m < 5; ++m) part[((long)q * 5 + m) * nc + cell] = (q == 0 && gas) ? a5[m].value() : T(0);
}

__device__ __forceinline__ double maxw3(const double *q, double vx, double vy, double vz)
{
    const double ax = vx - q[1], ay = vy - q[2], az = vz - q[3];
    const double a2 = 2.0 * kPi * q[4];
    return q[0] / (a2 * sqrt(a2)) * exp(-(ax * ax + ay * ay + az * az) / (2.0 * q[4]));
}

// Maxwellian state from per-cell primitives (rho, ux, uy, uz, T); solid cells
// get 0.  One block row per cell, threads over the public velocities.
template <typename T>
__global__ void k_init3(Grid3D g, const double *prim, const int8_t *type, T *f)
{
    const int q = blockIdx.x;
    const int p = blockIdx.y * blockDim.x + threadIdx.x;
    if (p >= g.nv) return;
    const int p1 = p % g.nvx, r = p / g.nvx;
    const int p3 = r / g.nvy, p2 = r - p3 * g.nvy;
    const double *s = prim + 5L * q;
    double m = 0;
    if (type[q] != DVM_SOLID && s[0] > 0)
        m = maxw3(s, g.vxmin + p1 * g.dvx, g.vymin + p2 * g.dvy, g.vzmin + p3 * g.dvz);
    f[pidx3(g, r * g.nvxp + p1, pcell3(g, q))] = (T)m;
}

// Ghost cells of a Maxwellian side (both layers, both state buffers).
template <typename T>
__global__ void k_ghost3(Grid3D g, const double *prim, int side, int nside, T *f0, T *f1)
{
    const long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (long)nside * g.nv) return;
    const int q = (int)(t / g.nv), p = (int)(t % g.nv);
    const int p1 = p % g.nvx, r = p / g.nvx;
    const int p3 = r / g.nvy, p2 = r - p3 * g.nvy;
    const double m = maxw3(prim + 5L * q, g.vxmin + p1 * g.dvx, g.vymin + p2 * g.dvy, g.vzmin + p3 * g.dvz);
    // side cell q: row-major over the two remaining axes
    int a, b;
    if (side < 2) { a = q % g.ny; b = q / g.ny; }          // (j, k)
    else if (side < 4) { a = q % g.nx; b = q / g.nx; }     // (i, k)
    else { a = q % g.nx; b = q / g.nx; }                   // (i, j)
    const int pp = r * g.nvxp + p1;
    for (int layer = 1; layer <= 2; ++layer) {
        int pc;
        if (side == 0) pc = nbr3(g, -layer, a, b);
        else if (side == 1) pc = nbr3(g, g.nx - 1 + layer, a, b);
        else if (side == 2) pc = nbr3(g, a, -layer, b);
        else if (side == 3) pc = nbr3(g, a, g.ny - 1 + layer, b);
        else if (side == 4) pc = nbr3(g, a, b, -layer);
        else pc = nbr3(g, a, b, g.nz - 1 + layer);
        f0[pidx3(g, pp, pc)] = (T)m;
        f1[pidx3(g, pp, pc)] = (T)m;
    }
}

// Padding of periodic and zero-gradient sides from the interior (both
// layers); one thread finds a padding cell's source once and copies the
// vectors of kHaloGroups groups, all loads in flight.  64^3 x 20^3, FP32: one
// vector per thread, bound by the divisions that find the cell, 0.71 ms; now
// 0.55 ms.
constexpr int kHaloGroups = 8;
template <typename T>
__global__ void k_halo3(Grid3D g, T *f)
{
    using V = typename Vec<T>::type;
    const long fx = (long)g.ny * g.nz, fy = (long)g.nx * g.nz, fz = (long)g.nx * g.ny;
    const long per = 2 * (fx + fy + fz);      // padding cells of one layer
    const long hc = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (hc >= 2 * per) return;
    const int layer = (int)(hc / per) + 1;
    long pos = hc % per;
    int side;
    if (pos < 2 * fx) { side = pos < fx ? 0 : 1; pos = pos % fx; }
    else if (pos < 2 * fx + 2 * fy) { pos -= 2 * fx; side = pos < fy ? 2 : 3; pos = pos % fy; }
    else { pos -= 2 * fx + 2 * fy; side = pos < fz ? 4 : 5; pos = pos % fz; }
    const int kind = g.bc[side];
    if (kind == DVM_BC_MAXWELLIAN) return;
    const bool per_ = kind == DVM_BC_PERIODIC;
    int di, dj, dk, si, sj, sk;
    if (side < 2) {
        const int j = (int)(pos % g.ny), k = (int)(pos / g.ny);
        dj = sj = j; dk = sk = k;
        if (side == 0) { di = -layer; si = per_ ? g.nx - layer : 0; }
        else { di = g.nx - 1 + layer; si = per_ ? layer - 1 : g.nx - 1; }
    } else if (side < 4) {
        const int i = (int)(pos % g.nx), k = (int)(pos / g.nx);
        di = si = i; dk = sk = k;
        if (side == 2) { dj = -layer; sj = per_ ? g.ny - layer : 0; }
        else { dj = g.ny - 1 + layer; sj = per_ ? layer - 1 : g.ny - 1; }
    } else {
        const int i = (int)(pos % g.nx), j = (int)(pos / g.nx);
        di = si = i; dj = sj = j;
        if (side == 4) { dk = -layer; sk = per_ ? g.nz - layer : 0; }
        else { dk = g.nz - 1 + layer; sk = per_ ? layer - 1 : g.nz - 1; }
    }
    const int q0 = blockIdx.y * kHaloGroups, n = min(kHaloGroups, g.ngrp - q0);
    V *const slab = reinterpret_cast<V *>(f) + (long)q0 * g.slab;
    const V *const src = slab + nbr3(g, si, sj, sk);
    V *const pad = slab + nbr3(g, di, dj, dk);
    V v[kHaloGroups];
#pragma unroll
    for (int q = 0; q < kHaloGroups; ++q)
        if (q < n) v[q] = src[(long)q * g.slab];
#pragma unroll
    for (int q = 0; q < kHaloGroups; ++q)
        if (q < n) pad[(long)q * g.slab] = v[q];
}

// Zero the state of every solid cell: one thread per cell and chunk of the
// velocity groups (blockIdx.y); only the threads of solid cells store.
template <typename T>
__global__ void k_zero_solid3(Grid3D g, const int8_t *type, T *f)
{
    using V = typename Vec<T>::type;
    const long k = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= (long)g.nx * g.ny * g.nz || type[k] != DVM_SOLID) return;
    const int gps = (g.ngrp + gridDim.y - 1) / gridDim.y;
    const int q0 = blockIdx.y * gps, q1 = min(q0 + gps, g.ngrp);
    const long pc = pcell3(g, (int)k);
    V *fv = reinterpret_cast<V *>(f);
    const T z[Vec<T>::W] = {};
    for (int q = q0; q < q1; ++q) vst<T>(fv + (long)q * g.slab + pc, z);
}

template <typename T>
__global__ void __launch_bounds__(256) k_mass_cells3(Grid3D g, const T *f, const double *vol, double *cm)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long cell = (long)blockIdx.x * 8 + warp;
    if (cell >= (long)g.nx * g.ny * g.nz) return;
    double s = 0;
    const int pc = pcell3(g, (int)cell);
    for (int p = lane; p < g.nvp; p += 32) s += (double)f[pidx3(g, p, pc)];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) cm[cell] = vol[cell] * (s * g.dv);
}

__global__ void __launch_bounds__(1024) k_sum3(const double *x, long n, double *out)
{
    __shared__ double red[32];
    double s = 0;
    for (long t = threadIdx.x; t < n; t += blockDim.x) s += x[t];
    s = block_sum(s, red);
    if (threadIdx.x == 0) *out = s;
}

template <typename T>
__global__ void k_tables3(Grid3D g, VX3<T> *vxt, VYZ3<T> *vyz)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < g.nvxp) {
        VX3<T> c;
        if (t < g.nvx) {
            c.vx = T(g.vxmin + t * g.dvx);
            c.nux = fabs(c.vx) * T(g.dt / g.dx);
        } else {
            c.vx = T(1e4);      // padding: zero state, vanishing equilibrium
            c.nux = 0;
        }
        vxt[t] = c;
    }
    if (t < g.nvy * g.nvz) {
        const int p2 = t % g.nvy, p3 = t / g.nvy;
        VYZ3<T> c;
        c.vy = T(g.vymin + p2 * g.dvy);
        c.vz = T(g.vzmin + p3 * g.dvz);
        c.nuy = fabs(c.vy) * T(g.dt / g.dy);
        c.nuz = fabs(c.vz) * T(g.dt / g.dz);
        vyz[t] = c;
    }
}

inline unsigned nb3(long n, int b) { return (unsigned)((n + b - 1) / b); }

template <typename T>
const VX3<T> *vx_table(const dvm_ctx *c) { return reinterpret_cast<const VX3<T> *>(c->vtab); }

template <typename T>
const VYZ3<T> *vyz_table(const dvm_ctx *c)
{
    return reinterpret_cast<const VYZ3<T> *>(reinterpret_cast<const char *>(c->vtab) + (size_t)c->nvxp * sizeof(VX3<T>));
}

template <typename T, bool MUSCL, bool SHAK>
cudaError_t launch_bulk3(dvm_ctx *c, const Bulk3Args<T> &a)
{
    const size_t smem = bulk3_smem<T, SHAK>();
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(k_bulk3<T, MUSCL, SHAK>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    if constexpr (sizeof(T) == 8) {
        constexpr int cells = 128 / kCellThreads;
        k_cell64_3<<<(unsigned)((c->nc + cells - 1) / cells), 128, 0, c->stream>>>(a, c->cf64);
        c->launches += 1;
    }
    constexpr int threads = 32 * warps3<T>();
    const dim3 grid(nb3(c->nx, a.tx), nb3(c->ny, a.ty), (unsigned)(a.nzc * a.S));
    k_bulk3<T, MUSCL, SHAK><<<grid, threads, smem, c->stream>>>(a, c->tmap[c->cur]);
    return cudaGetLastError();
}

// The bulk kernel for the scheme, and its Shakhov variant in FP32.
template <typename T>
cudaError_t launch_bulk3_any(dvm_ctx *c, const Bulk3Args<T> &a, bool shak)
{
    if constexpr (sizeof(T) == 4) {
        if (shak) return c->scheme == DVM_MUSCL ? launch_bulk3<T, true, true>(c, a) : launch_bulk3<T, false, true>(c, a);
    }
    return c->scheme == DVM_MUSCL ? launch_bulk3<T, true, false>(c, a) : launch_bulk3<T, false, false>(c, a);
}

Cv3Args cv3_args(dvm_ctx *c)
{
    Cv3Args cv{};
    cv.g = grid3d(c);
    cv.G = c->geo3;
    cv.master = c->master; cv.flags = c->flags3;
    cv.spec_list = c->spec_list; cv.wall_list = c->wall_list; cv.wslot = c->wslot;
    cv.counts = c->counts; cv.cap = c->list_cap; cv.S = c->S; cv.Sin = c->S;
    cv.gps = (c->ngrp + c->S - 1) / c->S;
    cv.cvinfo = c->cvinfo;
    cv.vxt = c->vtab;
    cv.vyz = reinterpret_cast<const char *>(c->vtab) + (size_t)c->nvxp * 2 * c->elem;
    cv.err = c->d_err;
    return cv;
}

// Moment sums of each cell over this context's velocities, folded over the
// S velocity splits in fixed order, in FP64 (the data a velocity split
// exchanges, Sec. 5.2).
template <typename T>
__global__ void k_fold_partials3(const T *part, int S, long nc, double *x)
{
    const long cell = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (cell >= nc) return;
    T s[5];
    gather_partials3(part, S, nc, cell, s);
#pragma unroll
    for (int m = 0; m < 5; ++m) x[(long)m * nc + cell] = (double)s[m];
}

template <typename T>
__global__ void k_unfold_partials3(const double *x, long n, T *part)
{
    const long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < n) part[t] = (T)x[t];
}

// The bookkeeping that ends a step: the new state is the current one.
cudaError_t end_step3d(dvm_ctx *c)
{
    c->cur = 1 - c->cur;
    c->need_fusion = false;
    c->steps_done++;
    return cudaGetLastError();
}

// The relaxation of the semi-implicit scheme (Eq. ImpSchemeDD) on the
// transported values f[1 - cur], with their moments from mom (Smom slots).
template <typename T>
cudaError_t imex_relax3d(dvm_ctx *c, const T *mom, int Smom)
{
    const Grid3D g = grid3d(c);
    T *fout = (T *)c->f[1 - c->cur], *pout = (T *)c->part[1 - c->cur];
    const bool cons = c->eq_mode == DVM_EQ_CONSERVATIVE;
    const dim3 grid(nb3(c->nx, 32), c->ny, c->nz), block(32, kMomChunks);
    cudaError_t e;
    // conservative equilibrium parameters of the transported state
    if (cons && (e = eqpar(c, mom, Smom)) != cudaSuccess) return e;
    if (c->model == DVM_SHAKHOV)
        k_imex3<T, true><<<grid, block, 0, c->stream>>>(g, c->S, T(c->dt / c->tau0), fout, vx_table<T>(c),
                                                        vyz_table<T>(c), mom, Smom, pout, c->geo3.type, nullptr,
                                                        T(c->Pr), c->d_err);
    else
        k_imex3<T, false><<<grid, block, 0, c->stream>>>(g, c->S, T(c->dt / c->tau0), fout, vx_table<T>(c),
                                                         vyz_table<T>(c), mom, Smom, pout, c->geo3.type,
                                                         cons ? (const T *)c->eqp : nullptr, T(1), c->d_err);
    c->launches += 1;
    return cudaGetLastError();
}

// One step in phases, as in 2D: 0 the whole step; a velocity split runs
// phase 1 (this rank's moment sums [5][nc] and wall sums [wall slot][14]
// into the FP64 buffer xbuf) and phase 2 (the rest, from xbuf summed over
// the ranks).  Under the semi-implicit scheme phase 2 ends with this rank's
// moment sums of the transported values in xbuf ([5][nc]) and phase 3 takes
// them summed over the ranks and relaxes.
template <typename T>
cudaError_t step3d_t(dvm_ctx *c, int phase, double *xbuf)
{
    Grid3D g = grid3d(c);
    // the semi-implicit scheme (Eq. ImpSchemeDD) transports without
    // relaxation here; k_imex3 relaxes at the end of the step
    const bool imex = c->time_scheme == DVM_IMEX;
    if (imex) {
        g.dt_tau0 = 0.0;
        g.dt_tau0_f = 0.f;
    }
    const BodyParams bp = body_params(c);
    const bool body = c->body.shape != DVM_SHAPE_NONE;
    const long nc = (long)c->nc;
    T *fin = (T *)c->f[c->cur], *fout = (T *)c->f[1 - c->cur];
    T *pin = (T *)c->part[c->cur], *pout = (T *)c->part[1 - c->cur];
    cudaError_t e;
    Cv3Args cv = cv3_args(c);
    cv.g = g;                 // without the relaxation rate for the semi-implicit scheme
    const bool cons = c->eq_mode == DVM_EQ_CONSERVATIVE;
    cv.eqp = cons && !imex ? c->eqp : nullptr;
    const int cvgrid = 4 * 152;
    double *xw = xbuf ? xbuf + 5 * nc : nullptr;
    if (phase != 2) {
        if (body && c->need_fusion) {
            k_fusion3<T><<<cvgrid, 256, 0, c->stream>>>(cv, fin, pin);
            c->launches += 1;
        }
        if (phase == 1) {
            k_fold_partials3<T><<<nb3(nc, 256), 256, 0, c->stream>>>(pin, c->S, nc, xbuf);
            c->launches += 1;
            if (body) {
                k_wall3<T><<<cvgrid, 256, 0, c->stream>>>(cv, bp, c->d_body, fin, c->wphi, c->wcontrib, c->ticket,
                                                           c->d_hist, 1, xw);
                c->launches += 1;
            }
            return cudaGetLastError();
        }
    } else {
        // the summed moments of F_CV^n, one slot in the state precision
        pin = (T *)c->split_in;
        k_unfold_partials3<T><<<nb3(5 * nc, 256), 256, 0, c->stream>>>(xbuf, 5 * nc, pin);
        c->launches += 1;
    }
    const int Sin = phase == 2 ? 1 : c->S;
    cv.Sin = Sin;
    // conservative equilibrium parameters of F_CV^n (after fusion)
    if (cons && !imex && (e = eqpar(c, pin, Sin)) != cudaSuccess) return e;
    // the Shakhov model under the explicit scheme in FP32: the heat flux of
    // every control volume at t^n (after fusion), and the step kernels relax
    // towards its equilibrium (FP64: the post-pass k_shakhov3)
    const bool shak = c->model == DVM_SHAKHOV && !imex && c->prec == DVM_FP32;
    if (shak && (e = heatflux3d(c, fin, pin)) != cudaSuccess) return e;
    cv.qh = shak ? c->qheat : nullptr;
    cv.pr1 = 1.0 - c->Pr;
    if (body) {
        // the wall kernel and then the control-volume kernel run on the side
        // stream beside the bulk kernel: both read F^n and write only the cut
        // and merged control volumes, the bulk kernel only the plain cells
        if ((e = cudaEventRecord(c->ev_wfork, c->stream)) != cudaSuccess) return e;
        if ((e = cudaStreamWaitEvent(c->wstream, c->ev_wfork, 0)) != cudaSuccess) return e;
        k_wall3<T><<<cvgrid, 256, 0, c->wstream>>>(cv, bp, c->d_body, fin, c->wphi, c->wcontrib, c->ticket,
                                                    c->d_hist, phase == 2 ? 2 : 0, xw);
        c->launches += 1;
    }
    Bulk3Args<T> a{};
    a.g = g; a.S = c->S; a.Sin = Sin; a.nzc = (c->nz + kZc3 - 1) / kZc3;
    tile3d(c, &a.tx, &a.ty);
    a.eqp = cons && !imex ? (const T *)c->eqp : nullptr;
    a.qh = shak ? (const T *)c->qheat : nullptr;
    a.pr1 = T(1.0 - c->Pr);
    a.fin = fin; a.fout = fout; a.pin = pin; a.pout = pout;
    a.cf = c->cf64;
    a.flags = c->flags3; a.vxt = vx_table<T>(c); a.vyz = vyz_table<T>(c); a.err = c->d_err;
    if ((e = timing_mark(c, 0)) != cudaSuccess) return e;
    e = launch_bulk3_any<T>(c, a, shak);
    if (e != cudaSuccess) return e;
    if ((e = timing_mark(c, 1)) != cudaSuccess) return e;
    c->launches += 1;
    if (body) {
        // as many threads as four blocks of 256 an SM
        const int st = spec3_threads(cv.gps);
        k_special3<T><<<cvgrid * kSpec3Threads / st, st, 0, c->wstream>>>(cv, fin, fout, pin, pout, c->wphi);
        if ((e = cudaEventRecord(c->ev_wjoin, c->wstream)) != cudaSuccess) return e;
        // the step ends when both streams are done
        if ((e = cudaStreamWaitEvent(c->stream, c->ev_wjoin, 0)) != cudaSuccess) return e;
        c->launches += 1;
    }
    if (imex) {
        if (phase == 2) {
            // a velocity split relaxes in phase 3, from the moment sums of
            // the transported values summed over the ranks
            k_fold_partials3<T><<<nb3(nc, 256), 256, 0, c->stream>>>(pout, c->S, nc, xbuf);
            c->launches += 1;
            return cudaGetLastError();
        }
        if ((e = imex_relax3d<T>(c, pout, c->S)) != cudaSuccess) return e;
    }
    return end_step3d(c);
}

// Phase 3 of a semi-implicit step of a velocity split: the relaxation from
// the moment sums of the transported values summed over the ranks (xbuf).
template <typename T>
cudaError_t split_relax3d_t(dvm_ctx *c, const double *xbuf)
{
    const long nc = (long)c->nc;
    T *mom = (T *)c->split_in;
    k_unfold_partials3<T><<<nb3(5 * nc, 256), 256, 0, c->stream>>>(xbuf, 5 * nc, mom);
    c->launches += 1;
    cudaError_t e = imex_relax3d<T>(c, mom, 1);
    if (e != cudaSuccess) return e;
    return end_step3d(c);
}

}  // namespace

// Tile of the bulk kernel: the cells tx x ty of a plane that a block's threads
// take, row by row of the tile.  Of all widths, the one whose tiles cover the
// grid with the least work: a tile takes the time of its warps (in fours,
// one per SM sub-partition) and of about six more (latencies that few warps do
// not cover), weighted with a fifth of the halo it re-reads and a little for
// short rows; what fits a ring slot.  64^2 cells: 32 x 16.  FP32, 45 x 50
// cells: 45 x 11, 1.53 ms a launch within a step (37 planes, 14 x 15 x 13
// velocities, Shakhov) against 1.82 with 16 x 32 and 2.66 with 5 x 50 (as few
// lanes outside the grid, but 8 warps an SM).  FP64, 40^2: 40 x 6, 7.7 ms (40
// planes, 12^3, at the time) against 9.4 with 16 x 16 and 12.1 with 32 x 8.
void tile3d(const dvm_ctx *c, int *tx, int *ty)
{
    const int threads = 32 * (c->prec == DVM_FP32 ? warps3<float>() : warps3<double>());
    const int slot = c->prec == DVM_FP32 ? plane_stride3<float>() : plane_stride3<double>();
    double least = -1;
    for (int x = c->nx < 60 ? c->nx : 60; x >= 4; --x) {
        int y = threads / x;
        if (y > c->ny) y = c->ny;
        while (y > 1 && (x + 4) * (y + 4) > slot) --y;
        if ((x + 4) * (y + 4) > slot || y > 252) continue;
        const double work = (double)nb3(c->nx, x) * nb3(c->ny, y) * (nb3((long)x * y, 128) * 4 + 6);
        const double halo = (double)((x + 4) * (y + 4)) / (x * y);
        const double cost = work * (1.0 + 0.2 * (halo - 1.0) + 0.2 / x);
        if (least < 0 || cost < least) { least = cost; *tx = x; *ty = y; }
    }
}

int bulk3_blocks(const dvm_ctx *c)
{
    int tx = 32, ty = 8;
    tile3d(c, &tx, &ty);
    return (int)(nb3(c->nx, tx) * nb3(c->ny, ty) * nb3(c->nz, kZc3));
}

// TMA descriptors of the two state buffers: a 4D view (x: padded cells of a
// row times the W velocities of a group, y: padded rows, z: padded planes,
// w: velocity group) with the bulk kernel's plane box (tile plus halo).
int make_tensor_maps3d(dvm_ctx *c)
{
    static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
    if (!encode) {
        cudaDriverEntryPointQueryResult qr;
        void *fn = nullptr;
        cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &qr);
        if (e != cudaSuccess || qr != cudaDriverEntryPointSuccess || !fn) {
            set_error("cuTensorMapEncodeTiled is not available from the driver");
            return DVM_ERR_CUDA;
        }
        encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    }
    const int W = c->W;
    const cuuint64_t dims[4] = {(cuuint64_t)(c->nx + 4) * W, (cuuint64_t)(c->ny + 4), (cuuint64_t)(c->nz + 4),
                                (cuuint64_t)c->ngrp};
    const cuuint64_t row = (cuuint64_t)(c->nx + 4) * W * c->elem;
    const cuuint64_t strides[3] = {row, row * (c->ny + 4), (cuuint64_t)c->slab * W * c->elem};
    int tx = 32, ty = 8;
    tile3d(c, &tx, &ty);
    const cuuint32_t box[4] = {(cuuint32_t)((tx + 4) * W), (cuuint32_t)(ty + 4), 1, 1};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    const CUtensorMapDataType dt = c->prec == DVM_FP32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_FLOAT64;
    for (int b = 0; b < 2; ++b) {
        CUresult r = encode(&c->tmap[b], dt, 4, c->f[b], dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                            CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) {
            set_error("cuTensorMapEncodeTiled (3D) failed (" + std::to_string((int)r) + ")");
            return DVM_ERR_CUDA;
        }
    }
    return DVM_OK;
}

size_t vtab3_bytes(const dvm_ctx *c) { return (size_t)c->nvxp * 2 * c->elem + (size_t)c->nvy * c->nvz * 4 * c->elem; }

size_t cvinfo3_bytes() { return sizeof(CvInfo3); }

size_t cf64_bytes3d(const dvm_ctx *c) { return sizeof(double) * (kMxCount + c->nvxp) * (size_t)c->nc; }

cudaError_t members3d(dvm_ctx *c)
{
    k_members3<<<4 * 152, 256, 0, c->stream>>>(cv3_args(c), (CvInfo3 *)c->cvinfo);
    return cudaGetLastError();
}

cudaError_t step3d(dvm_ctx *c)
{
    return c->prec == DVM_FP32 ? step3d_t<float>(c, 0, nullptr) : step3d_t<double>(c, 0, nullptr);
}

// Velocity split: phase 1 (this rank's sums into xbuf) or phase 2 (finish
// the step from xbuf summed over the ranks).
cudaError_t split_step3d(dvm_ctx *c, int phase, void *xbuf)
{
    double *x = static_cast<double *>(xbuf);
    if (phase == 3) return c->prec == DVM_FP32 ? split_relax3d_t<float>(c, x) : split_relax3d_t<double>(c, x);
    return c->prec == DVM_FP32 ? step3d_t<float>(c, phase, x) : step3d_t<double>(c, phase, x);
}

cudaError_t tables3d(dvm_ctx *c)
{
    const Grid3D g = grid3d(c);
    const int n = c->nvxp > c->nvy * c->nvz ? c->nvxp : c->nvy * c->nvz;
    if (c->prec == DVM_FP32)
        k_tables3<float><<<nb3(n, 256), 256, 0, c->stream>>>(g, (VX3<float> *)c->vtab, (VYZ3<float> *)vyz_table<float>(c));
    else
        k_tables3<double><<<nb3(n, 256), 256, 0, c->stream>>>(g, (VX3<double> *)c->vtab,
                                                                (VYZ3<double> *)vyz_table<double>(c));
    return cudaGetLastError();
}

cudaError_t partials_from_state3d(dvm_ctx *c)
{
    const Grid3D g = grid3d(c);
    const dim3 grid(nb3((long)c->nc, 32)), block(32, kMomChunks);
    if (c->prec == DVM_FP32)
        k_partials3<float><<<grid, block, 0, c->stream>>>(g, c->S, (const float *)c->f[c->cur], vx_table<float>(c),
                                                          vyz_table<float>(c), (float *)c->part[c->cur], c->geo3.type,
                                                          c->d_err);
    else
        k_partials3<double><<<grid, block, 0, c->stream>>>(g, c->S, (const double *)c->f[c->cur],
                                                           vx_table<double>(c), vyz_table<double>(c),
                                                           (double *)c->part[c->cur], c->geo3.type, c->d_err);
    return cudaGetLastError();
}

cudaError_t check_moments3d(dvm_ctx *c)
{
    const Grid3D g = grid3d(c);
    if (c->prec == DVM_FP32)
        k_check3<float><<<nb3(c->nc, 128), 128, 0, c->stream>>>(g, c->S, (const float *)c->part[c->cur], c->geo3.type,
                                                                c->d_err);
    else
        k_check3<double><<<nb3(c->nc, 128), 128, 0, c->stream>>>(g, c->S, (const double *)c->part[c->cur], c->geo3.type,
                                                                 c->d_err);
    return cudaGetLastError();
}

cudaError_t moments_out3d(dvm_ctx *c, double *d_out)
{
    const Grid3D g = grid3d(c);
    const dim3 grid(nb3((long)c->nc, 32)), block(32, kMomChunks);
    if (c->prec == DVM_FP32)
        k_moments_out3<float><<<grid, block, 0, c->stream>>>(g, (const float *)c->f[c->cur], vx_table<float>(c),
                                                             vyz_table<float>(c), d_out);
    else
        k_moments_out3<double><<<grid, block, 0, c->stream>>>(g, (const double *)c->f[c->cur], vx_table<double>(c),
                                                              vyz_table<double>(c), d_out);
    return cudaGetLastError();
}

cudaError_t init_maxwellian3d(dvm_ctx *c, const double *d_prim)
{
    const Grid3D g = grid3d(c);
    dim3 grid((unsigned)c->nc, nb3(c->nv, 256));
    if (c->prec == DVM_FP32)
        k_init3<float><<<grid, 256, 0, c->stream>>>(g, d_prim, c->geo3.type, (float *)c->f[c->cur]);
    else
        k_init3<double><<<grid, 256, 0, c->stream>>>(g, d_prim, c->geo3.type, (double *)c->f[c->cur]);
    return cudaGetLastError();
}

cudaError_t ghost3d(dvm_ctx *c, int side, const double *d_prim, int nside)
{
    const Grid3D g = grid3d(c);
    const long n = (long)nside * c->nv;
    if (c->prec == DVM_FP32)
        k_ghost3<float><<<nb3(n, 256), 256, 0, c->stream>>>(g, d_prim, side, nside, (float *)c->f[0], (float *)c->f[1]);
    else
        k_ghost3<double><<<nb3(n, 256), 256, 0, c->stream>>>(g, d_prim, side, nside, (double *)c->f[0], (double *)c->f[1]);
    return cudaGetLastError();
}

cudaError_t zero_solid3d(dvm_ctx *c)
{
    const Grid3D g = grid3d(c);
    const dim3 grid(nb3(c->nc, 256), 8);
    for (int b = 0; b < 2; ++b) {
        if (c->prec == DVM_FP32) k_zero_solid3<float><<<grid, 256, 0, c->stream>>>(g, c->geo3.type, (float *)c->f[b]);
        else k_zero_solid3<double><<<grid, 256, 0, c->stream>>>(g, c->geo3.type, (double *)c->f[b]);
    }
    return cudaGetLastError();
}

cudaError_t halo3d(dvm_ctx *c, int buf)
{
    const Grid3D g = grid3d(c);
    const long per = 2L * ((long)c->ny * c->nz + (long)c->nx * c->nz + (long)c->nx * c->ny);
    const dim3 grid(nb3(2 * per, 256), nb3(c->ngrp, kHaloGroups));
    if (c->prec == DVM_FP32) k_halo3<float><<<grid, 256, 0, c->stream>>>(g, (float *)c->f[buf]);
    else k_halo3<double><<<grid, 256, 0, c->stream>>>(g, (double *)c->f[buf]);
    return cudaGetLastError();
}

cudaError_t mass3d(dvm_ctx *c, double *d_scratch, double *d_out)
{
    const Grid3D g = grid3d(c);
    if (c->prec == DVM_FP32)
        k_mass_cells3<float><<<nb3(c->nc, 8), 256, 0, c->stream>>>(g, (const float *)c->f[c->cur], c->geo3.vol, d_scratch);
    else
        k_mass_cells3<double><<<nb3(c->nc, 8), 256, 0, c->stream>>>(g, (const double *)c->f[c->cur], c->geo3.vol, d_scratch);
    k_sum3<<<1, 1024, 0, c->stream>>>(d_scratch, c->nc, d_out);
    return cudaGetLastError();
}

}  // namespace dvm

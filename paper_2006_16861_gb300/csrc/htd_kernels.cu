// CUDA kernels of the time-domain Helmholtz preconditioner (sm_103a).
//
//  step2d / step3d   one step of the frequency-adapted leapfrog recurrence
//                    I_acd (Def. of I_acd) with the windowed forcing of
//                    Table 1 fused in, in place over u_{j-1}, and the
//                    snapshot / final-state write of Table 1 fused in.
//  split             complex128 right-hand side -> Re/Im planes (Table 1 uses
//                    Re F and Im F every step).
//  apply_H           true operator H X (or F - H X), complex128, FP64.
//  dots / reduce     block dot products conj(V_k) . w with warp shuffles,
//                    two-pass fixed-order reduction (deterministic).
//  sub/add_combination, scale   Krylov vector updates.
//
// Operator (App. A cell form, h^2-scaled): for node beta and offset
// o in {-1,0,1}^d with Hamming weight s = |o|,
//   h^2 (Re H u)_beta = sum_o u_{beta+o} [ 2^{d-s} S_s - M_s * sum of kappa over
//                       the 2^{d-s} cells that contain both beta and beta+o ],
// kappa = (h k_cell)^2, S_s / M_s the stiffness / mass weights of the cell
// kernel at Hamming distance s.  One step of I_acd with
// K = (dt^2/alpha)(Re H + omega^2), L/2 = ell, d = 1/(1+ell):
//   u_{j+1} = d ((2 - K) u_j + g_j - 2 u_{j-1}) + u_{j-1},
//   g_j = a_j Re F - b_j Im F,
// where (2 - K) u_j = c0 u - sum_{o != 0} cs_s u_{beta+o}
//                     + sum_o M_s (sum of q kappa over the cells) u_{beta+o},
// q = dt^2 / (alpha h^2), c0 = 2 - (dt^2/alpha) omega^2 - q 2^d S_0,
// cs_s = q 2^{d-s} S_s; the stored per-cell coefficient is q * kappa.
#include <cuda_runtime.h>
#include <algorithm>
#include <mutex>
#include <type_traits>
#include <vector>

#include "htd_internal.h"

namespace htd {

long long g_launches = 0;

// SMs of the current device, looked up once per device (1 if the lookup fails)
static int sm_count()
{
    static int count[64] = {0};
    int dev = 0, nsm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
        (void)cudaGetLastError();
        return 1;
    }
    if (count[dev] > 0) return count[dev];
    if (cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        nsm < 1) {
        (void)cudaGetLastError();
        return 1;
    }
    count[dev] = nsm;
    return nsm;
}

// ---------------------------------------------------------------------------
// recurrence step
// ---------------------------------------------------------------------------

// Programmatic dependent launch (no-ops for an ordinary launch): what the previous kernel
// wrote is visible after grid_dep_wait; the next kernel of the stream may be scheduled
// once every block of this one has called grid_dep_launch.
__device__ __forceinline__ void grid_dep_wait()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

__device__ __forceinline__ void grid_dep_launch()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// kEarly: let the next kernel in at once, else only after the wait (launch_step_kernel)
template <bool kEarly>
__device__ __forceinline__ void grid_dep_begin()
{
    if (kEarly) grid_dep_launch();
    grid_dep_wait();
    if (!kEarly) grid_dep_launch();
}

// Blocks of `kern` with `threads` threads that the device holds at once (0: unknown)
template <typename Kern>
static int64_t resident_blocks(Kern kern, int threads)
{
    struct Entry {
        const void *kern;
        int dev, occ;
    };
    static std::mutex lock;
    static std::vector<Entry> seen;
    int dev = 0, occ = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        (void)cudaGetLastError();
        return 0;
    }
    const void *key = reinterpret_cast<const void *>(kern);
    const std::lock_guard<std::mutex> hold(lock);
    for (const Entry &e : seen)
        if (e.kern == key && e.dev == dev) return (int64_t)e.occ * sm_count();
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, threads, 0) != cudaSuccess) {
        (void)cudaGetLastError();
        return 0;
    }
    seen.push_back({key, dev, occ});
    return (int64_t)occ * sm_count();
}

// How a one-step launch overlaps the one before it, by the share of the device's
// resident blocks that a step takes:
//  - up to a half (both steps' blocks fit, and are spread before the first has ended): the
//    next step is let in after the wait, so that no more than one waits.  Let in before it,
//    several waiting grids filled the SMs, and a new grid's blocks went where old ones
//    happened to end, several to one SM.  us per step, after / before the wait / no overlap:
//    FP64 2-D 0.17 share 2.63 / 6.1 / 2.78, 0.42 4.72 / 7.0 / 4.87; I_abd FP64 0.19 6.2 / 12.7 /
//    6.4; FP32 2-D 0.40 1.89 / 2.40 / 2.11;
//  - from `full` on: before the wait, as the next step's blocks only take up what the last
//    blocks leave.  FP64 2-D 1.38 10.84 / 10.77 / 10.98, 801^2 (2.9) 19.08 / 18.99 / 19.24;
//  - between: no overlap; part of the next step's blocks wait in the gaps and the rest crowd.
//    FP64 2-D 0.53 7.79 / 7.73 / 5.86, 0.73 7.81 / 7.75 / 6.93; FP32 2-D 0.55 2.53 / 2.52 /
//    2.26; I_abd FP32 3-D 0.63 3.82 / 3.73 / 3.15.
// `full` is where the last two meet: kFull (FP64 3-D 0.79 7.9 / 7.0 before the wait / no overlap,
// 0.85 7.36 / 7.52), kFull64 for the other FP64 steps, and kFullRows for the 2-D steps with
// several rows per thread (FP32 600^2, 0.79: 2.90 / 3.17 before the wait / no overlap).
// Slots that may be idle count for the first rule, and for the second only where their
// blocks alone are kManyWaves times what the device holds: of 8 right-hand sides with 2
// active, before the wait / in stream order, ms per application: I_abd FP64 150 x 170 (1.2)
// 2.81 / 2.04, FP64 (1.0) 1.03 / 0.68; FP32 401^2 (3.0) 0.70 / 0.78.
constexpr double kFull = 0.8, kFull64 = 1.2, kFullRows = 0.7, kManyWaves = 2.5;

// Launches `early` (the kernel that lets the next one in before the wait) or `late` (after
// it), otherwise the same
template <typename Kern, typename... Args>
static void launch_step_kernel(Kern early, Kern late, double full, dim3 grid, dim3 threads,
                               const RhsSet &R, cudaStream_t s, bool overlap, Args &&...args)
{
    const double blocks = (double)grid.x * grid.y * grid.z;
    const double fit = overlap ? (double)resident_blocks(late, (int)(threads.x * threads.y)) : 0.0;
    const bool first = fit > 0.0 && (blocks * R.sure >= full * fit * R.slots ||
                                     blocks >= kManyWaves * fit);
    launch_ex(first ? early : late, grid, threads, 0, s, first || 2.0 * blocks <= fit,
              static_cast<Args &&>(args)...);
}

// One step in 2-D, FP32: u_{j+1} -> out (which may be the plane um of u_{j-1}).  A
// thread takes ROWS nodes of one column, so that a node costs 4.5 loads of u_j and 2.5
// of q*kappa (nine and four with one row), all of them issued before the first sum.
// ROWS = 4 where that leaves two blocks per SM, else 1.  kForce: without it the step has
// no forcing (a = b = 0: the adjoint between its read-out steps); a parameter of the
// kernel, and the rows' clamping for one row too, put a branch and 64-bit minima before the
// loads: 401^2 2.73 us per step, 2.24 so.
template <int ROWS, bool kForce, bool kEarly>
__global__ void __launch_bounds__(256)
step2d_kernel(const float *__restrict__ u, const float *um, float *out,
              const float *__restrict__ kap, const float *__restrict__ dco,
              const float *__restrict__ fre, const float *__restrict__ fim, Layout L,
              StepCoef<float> C, float a, float b, const OutSlot *__restrict__ slot, int flags,
              RhsSet R)
{
    grid_dep_begin<kEarly>();
    const int64_t ix = (int64_t)blockIdx.x * 32 + threadIdx.x;
    const int64_t iy0 = ((int64_t)blockIdx.y * 8 + threadIdx.y) * ROWS;
    int rhs;
    if (!rhs_of_slot(R, (int)blockIdx.z, rhs)) return;
    if (ix >= L.nx || iy0 >= L.ny) return;
    const int64_t off = rhs * R.stride;
    u += off;
    um += off;
    out += off;
    fre += off;
    fim += off;
    slot += rhs;
    const int64_t P = L.pitch;
    const Stencil2dCoef<float> SC = stencil2d_coef(C);
    const int64_t i0 = (iy0 + 1) * P + L.xl + ix;
    // every operand first: the loads of all rows are in flight together.  (Rows
    // below the grid are loaded from its last ghost row and not stored.)
    float w[ROWS + 2][3], k[ROWS + 1][2], um1[ROWS], d[ROWS], fr[ROWS], fi[ROWS];
    int64_t at[ROWS + 2];                   // u row r - 1
#pragma unroll
    for (int r = 0; r < ROWS + 2; ++r)
        at[r] = i0 + (ROWS == 1 ? r - 1 : min(iy0 + r - 1, L.ny) - iy0) * P;
#pragma unroll
    for (int r = 0; r < ROWS + 2; ++r)
#pragma unroll
        for (int x = 0; x < 3; ++x) w[r][x] = u[at[r] + x - 1];
#pragma unroll
    for (int r = 0; r < ROWS + 1; ++r)
#pragma unroll
        for (int x = 0; x < 2; ++x) k[r][x] = kap[at[r] + x - 1];
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
        um1[r] = um[at[r + 1]];
        d[r] = dco[at[r + 1]];
        if (kForce) {
            fr[r] = fre[at[r + 1]];
            fi[r] = fim[at[r + 1]];
        }
    }
    // w[r]: u_j at row offset r - 1 of the first node; k[r]: q*kappa of the cells of
    // row y - 1 + r.  Pair sums shared with the temporally blocked kernel (same
    // order, same result)
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
        if (r > 0 && iy0 + r >= L.ny) break;
        const float *a0 = w[r], *a1 = w[r + 1], *a2 = w[r + 2];
        float ag = stencil2d(SC, a0[0], a0[1], a0[2], a1[0], a1[1], a1[2], a2[0], a2[1], a2[2],
                             k[r][0], k[r][1], k[r + 1][0], k[r + 1][1], a0[0] + a0[2],
                             a1[0] + a1[2], a2[0] + a2[2], k[r][0] + k[r][1],
                             k[r + 1][0] + k[r + 1][1]);
        // acc + a Re F - b Im F as two FMAs (the blocked kernels round the same way)
        if (kForce) ag = vfma(a, fr[r], vfma(-b, fi[r], ag));
        const float unew = vfma(d[r], vfma(-2.f, um1[r], ag), um1[r]);
        out[at[r + 1]] = unew;
        if (flags) {
            const int64_t c = (iy0 + r) * L.nx + ix;
            if ((flags & 1) && slot->snap_part) slot->snap_part[2 * c] = (double)unew;
            if ((flags & 2) && slot->final_part) slot->final_part[2 * c] = (double)unew;
        }
    }
}

// Each thread walks a column of kZChunk planes in z with a 3x3x3 register
// window of u_j (planes z-1, z, z+1) and a 2x2x2 window of cells, so a node
// costs 9 new loads of u_j and 4 of q*kappa (neighbours in x and y come from
// L1, the plane below and the node's own plane from registers).
constexpr int kZChunk = 16;

template <bool kForce>
__global__ void __launch_bounds__(256)
step3d_kernel(const float *__restrict__ u, const float *um, float *out,
              const float *__restrict__ kap, const float *__restrict__ dco,
              const float *__restrict__ fre, const float *__restrict__ fim, Layout L,
              StepCoef<float> C, float a, float b, const OutSlot *__restrict__ slot, int flags,
              RhsSet R, int nchunks)
{
    typedef float T;
    const int64_t ix = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t iy = (int64_t)blockIdx.y * blockDim.y + threadIdx.y;
    int rhs;
    if (!rhs_of_slot(R, (int)blockIdx.z / nchunks, rhs)) return;
    const int64_t z0 = (int64_t)(blockIdx.z % nchunks) * kZChunk;
    const int64_t z1 = min((int64_t)L.nz, z0 + kZChunk);
    if (ix >= L.nx || iy >= L.ny) return;
    u += rhs * R.stride;
    um += rhs * R.stride;
    out += rhs * R.stride;
    fre += rhs * R.stride;
    fim += rhs * R.stride;
    slot += rhs;
    const int64_t P = L.pitch, Q = L.plane;
    const int64_t col = (iy + 1) * P + L.xl + ix;     // (y, x) offset of the node in any plane
    // w[p][oy][ox]: u_j at stored plane (iz + p), row offset oy-1, column offset ox-1
    T w[3][3][3];
    // k[az][ay][ax]: q*kappa of the cell at stored plane (iz + az), row y-1+ay, column x-1+ax
    T k[2][2][2];
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
        for (int oy = 0; oy < 3; ++oy)
#pragma unroll
            for (int ox = 0; ox < 3; ++ox)
                w[p][oy][ox] = u[(z0 + p) * Q + col + (oy - 1) * P + (ox - 1)];
#pragma unroll
    for (int ay = 0; ay < 2; ++ay)
#pragma unroll
        for (int ax = 0; ax < 2; ++ax)
            k[0][ay][ax] = kap[z0 * Q + col - (1 - ay) * P - (1 - ax)];
    for (int64_t iz = z0; iz < z1; ++iz) {
#pragma unroll
        for (int oy = 0; oy < 3; ++oy)
#pragma unroll
            for (int ox = 0; ox < 3; ++ox)
                w[2][oy][ox] = u[(iz + 2) * Q + col + (oy - 1) * P + (ox - 1)];
#pragma unroll
        for (int ay = 0; ay < 2; ++ay)
#pragma unroll
            for (int ax = 0; ax < 2; ++ax)
                k[1][ay][ax] = kap[(iz + 1) * Q + col - (1 - ay) * P - (1 - ax)];
        // sums of kappa over the cells shared by the node and its neighbour at
        // offset o - 1 (o in 0..2 per axis): -1 keeps the lower cell, +1 the upper, 0 both
        T kx[2][2][3];
#pragma unroll
        for (int az = 0; az < 2; ++az)
#pragma unroll
            for (int ay = 0; ay < 2; ++ay) {
                kx[az][ay][0] = k[az][ay][0];
                kx[az][ay][1] = k[az][ay][0] + k[az][ay][1];
                kx[az][ay][2] = k[az][ay][1];
            }
        T kxy[2][3][3];
#pragma unroll
        for (int az = 0; az < 2; ++az)
#pragma unroll
            for (int ox = 0; ox < 3; ++ox) {
                kxy[az][0][ox] = kx[az][0][ox];
                kxy[az][1][ox] = kx[az][0][ox] + kx[az][1][ox];
                kxy[az][2][ox] = kx[az][1][ox];
            }
        T acc = T(0);
#pragma unroll
        for (int oz = 0; oz < 3; ++oz)
#pragma unroll
            for (int oy = 0; oy < 3; ++oy)
#pragma unroll
                for (int ox = 0; ox < 3; ++ox) {
                    const int s = (oz != 1) + (oy != 1) + (ox != 1);
                    const T ks = (oz == 0) ? kxy[0][oy][ox]
                               : (oz == 2) ? kxy[1][oy][ox] : kxy[0][oy][ox] + kxy[1][oy][ox];
                    const T coef = (s == 0) ? C.c0 + C.mt[0] * ks : C.mt[s] * ks - C.cs[s];
                    acc += coef * w[oz][oy][ox];
                }
        const int64_t i = (iz + 1) * Q + col;
        const T g = kForce ? a * fre[i] - b * fim[i] : 0.f;
        const T d = dco[i];
        const T uprev = um[i];
        const T unew = d * (acc + g - T(2) * uprev) + uprev;
        out[i] = unew;
        if (flags) {
            const int64_t c = (iz * L.ny + iy) * L.nx + ix;
            if ((flags & 1) && slot->snap_part) slot->snap_part[2 * c] = (double)unew;
            if ((flags & 2) && slot->final_part) slot->final_part[2 * c] = (double)unew;
        }
#pragma unroll
        for (int oy = 0; oy < 3; ++oy)
#pragma unroll
            for (int ox = 0; ox < 3; ++ox) {
                w[0][oy][ox] = w[1][oy][ox];
                w[1][oy][ox] = w[2][oy][ox];
            }
#pragma unroll
        for (int ay = 0; ay < 2; ++ay)
#pragma unroll
            for (int ax = 0; ax < 2; ++ax) k[0][ay][ax] = k[1][ay][ax];
    }
}

void launch_step(const Layout &L, const float *u, const float *um, float *out, const float *kap,
                 const float *dco, const float *fre, const float *fim, const StepCoef<float> &C,
                 float a, float b, const OutSlot *slot, int flags, cudaStream_t s, const RhsSet &R,
                 bool force, bool overlap)
{
    const unsigned gx = (unsigned)((L.nx + 31) / 32);
    if (L.d == 2) {
        const int64_t blocks4 = gx * ((L.ny + 31) / 32) * R.slots;
        const bool four = blocks4 >= 2 * (int64_t)sm_count();
        const dim3 grd(gx, (unsigned)(four ? (L.ny + 31) / 32 : (L.ny + 7) / 8), (unsigned)R.slots);
        auto go = [&](auto early, auto late) {
            launch_step_kernel(early, late, four ? kFullRows : kFull, grd, dim3(32, 8), R, s,
                               overlap, u, um, out, kap, dco, fre, fim, L, C, a, b, slot, flags, R);
        };
        if (four) {
            if (force) go(step2d_kernel<4, true, true>, step2d_kernel<4, true, false>);
            else go(step2d_kernel<4, false, true>, step2d_kernel<4, false, false>);
        } else {
            if (force) go(step2d_kernel<1, true, true>, step2d_kernel<1, true, false>);
            else go(step2d_kernel<1, false, true>, step2d_kernel<1, false, false>);
        }
    } else {
        const int nchunks = (int)((L.nz + kZChunk - 1) / kZChunk);
        dim3 grd(gx, (unsigned)((L.ny + 7) / 8), (unsigned)(nchunks * R.slots));
        // (never overlapped: few long blocks, 120^3 22.9 us per step so, 18.5 in stream order)
        auto go = [&](auto kern) {
            launch_ex(kern, grd, dim3(32, 8), 0, s, false, u, um, out, kap, dco, fre, fim, L, C, a, b,
                      slot, flags, R, nchunks);
        };
        if (force) go(step3d_kernel<true>);
        else go(step3d_kernel<false>);
    }
    ++g_launches;
}

// One step of I_acd in FP64 from the assembled stencil.  GB300 retires two FP64
// operations per clock and SM (1.26 TFLOP/s as FMAs on 152 SMs) beside
// 6.8 TB/s, so the FP64 step is bound by its FP64 instruction count, not by its
// bytes: the cell form's sums of q kappa and coefficients (about 50 of the 81
// operations per 3-D node) are not recomputed in every step but read back, from
// the same assembled planes that apply_H uses (the centre and the positive
// offsets; a negative offset is the neighbour's positive one).  For FP64 handles
// those planes hold -q (2^{d-s} S_s - M_s sum kappa) off the centre and q M_0 sum
// kappa at the centre, so that with c0 = 2 - p - q 2^d S_0
//   (2 - K) u_j = c0 u_j + sum_o coef_o u_{j, beta + o}
// is one multiply-add per offset: 33 FP64 operations per 3-D node.  (The centre's
// constant stays a scalar because a stored coefficient's rounding is the same in
// every step and so adds up: the centre's, about 1, would round five times as
// coarsely as the others.)  The planes
// are compact (N values each) and padded nowhere: where an offset leaves the
// grid u is the zero ghost ring, and the index is clamped into the plane (any
// finite coefficient times the ghost's zero).
// A thread marches up a column of zc planes with the 3 x 3 x 3 window of u in
// registers; zc is chosen by the launcher so that every SM gets about eight
// blocks (the last wave of an FP64-bound kernel costs as much as it holds).
// Measured on GB300, 96^3: 57.4 us per step (cell form: 179 us); the FP64 pipe alone
// would take 46.4 us, 0.81 of it (0.90 at 256^3).
constexpr int kAsmTY = 4;

// (kFold: tile rows beyond grid.y's 65535 blocks follow along grid.x; a form of its own,
// as the index arithmetic cost the others up to 1.7 %)
template <bool kFold, bool kEarly>
__global__ void __launch_bounds__(32 * kAsmTY)
step3d_asm_kernel(const double *__restrict__ u, const double *um, double *out,
                  const double *__restrict__ coefP, const double *__restrict__ dco,
                  const double *__restrict__ fre, const double *__restrict__ fim, Layout L,
                  double c0, double a, double b, const OutSlot *__restrict__ slot, int flags,
                  RhsSet R, int zc, int nchunks)
{
    grid_dep_begin<kEarly>();
    unsigned bx = blockIdx.x, by = blockIdx.y;
    if (kFold) {
        const unsigned gx = (unsigned)((L.nx + 31) / 32);
        by += bx / gx * gridDim.y;
        bx %= gx;
    }
    const int64_t ix = (int64_t)bx * 32 + threadIdx.x;
    const int64_t iy = (int64_t)by * kAsmTY + threadIdx.y;
    int rhs;
    if (!rhs_of_slot(R, (int)blockIdx.z / nchunks, rhs)) return;
    const int64_t z0 = (int64_t)(blockIdx.z % nchunks) * zc;
    const int64_t z1 = min((int64_t)L.nz, z0 + zc);
    if (ix >= L.nx || iy >= L.ny) return;
    u += rhs * R.stride;
    um += rhs * R.stride;
    out += rhs * R.stride;
    fre += rhs * R.stride;
    fim += rhs * R.stride;
    slot += rhs;
    const int64_t P = L.pitch, Q = L.plane, N = L.N;
    const int64_t col = (iy + 1) * P + L.xl + ix;     // offset of the column in a stored plane
    // w[p][oy][ox]: u_j at stored plane iz + p, row offset oy - 1, column offset ox - 1
    double w[3][3][3];
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
        for (int oy = 0; oy < 3; ++oy)
#pragma unroll
            for (int ox = 0; ox < 3; ++ox)
                w[p][oy][ox] = u[(z0 + p) * Q + col + (oy - 1) * P + (ox - 1)];
    for (int64_t iz = z0; iz < z1; ++iz) {
        const int64_t i = (iz + 1) * Q + col;
        const int64_t c = (iz * L.ny + iy) * L.nx + ix;
#pragma unroll
        for (int oy = 0; oy < 3; ++oy)
#pragma unroll
            for (int ox = 0; ox < 3; ++ox)
                w[2][oy][ox] = u[i + Q + (oy - 1) * P + (ox - 1)];
        const double uprev = um[i];
        // Own-node terms beside the neighbours' (as in asm2d_step), and of those the small
        // ones first: a face's term is only its mass part (the stiffness of App. A's
        // stencil is zero there).  96^3: 8.26 ms per application, 8.36 with the faces last;
        // error against 64-bit torch 2.2e-15 either way.
        double own = fma(a, fre[i], -b * fim[i]);
        own = fma(-2.0, uprev, own);
        own = fma(c0, w[1][1][1], own);
        own = fma(coefP[c], w[1][1][1], own);
        double acc = coefP[9 * N + c] * w[2][1][1];
#pragma unroll
        for (int pass = 0; pass < 3; ++pass)
#pragma unroll
            for (int lin = 0; lin < 27; ++lin) {
                const int oz = lin / 9, oy = lin / 3 % 3, ox = lin % 3;
                const int sh = pass == 0 ? 1 : pass == 1 ? 3 : 2;       // faces, corners, edges
                if ((oz != 1) + (oy != 1) + (ox != 1) != sh || lin == 22) continue;
                int64_t ci = c;
                if (lin < 13) {
                    ci += ((int64_t)(oz - 1) * L.ny + (oy - 1)) * L.nx + (ox - 1);
                    ci = ci > 0 ? ci : 0;
                }
                acc = fma(coefP[(lin < 13 ? 13 - lin : lin - 13) * N + ci], w[oz][oy][ox], acc);
            }
        acc += own;
        const double unew = fma(dco[i], acc, uprev);
        out[i] = unew;
        if (flags) {
            if ((flags & 1) && slot->snap_part) slot->snap_part[2 * c] = unew;
            if ((flags & 2) && slot->final_part) slot->final_part[2 * c] = unew;
        }
#pragma unroll
        for (int oy = 0; oy < 3; ++oy)
#pragma unroll
            for (int ox = 0; ox < 3; ++ox) {
                w[0][oy][ox] = w[1][oy][ox];
                w[1][oy][ox] = w[2][oy][ox];
            }
    }
}

// the 2-D form: one node per thread, 15 FP64 operations (the cell form: 33);
// 801^2: 19.0 us per step (cell form: 41 us), 15.3 us at the FP64 pipe's rate
template <bool kEarly>
__global__ void __launch_bounds__(256)
step2d_asm_kernel(const double *__restrict__ u, const double *um, double *out,
                  const double *__restrict__ coefP, const double *__restrict__ dco,
                  const double *__restrict__ fre, const double *__restrict__ fim, Layout L,
                  double c0, double a, double b, const OutSlot *__restrict__ slot, int flags,
                  RhsSet R)
{
    grid_dep_begin<kEarly>();
    const int64_t ix = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t iy = (int64_t)blockIdx.y * blockDim.y + threadIdx.y;
    int rhs;
    if (!rhs_of_slot(R, (int)blockIdx.z, rhs)) return;
    if (ix >= L.nx || iy >= L.ny) return;
    u += rhs * R.stride;
    um += rhs * R.stride;
    out += rhs * R.stride;
    fre += rhs * R.stride;
    fim += rhs * R.stride;
    slot += rhs;
    const int64_t P = L.pitch, N = L.N;
    const int64_t i = (iy + 1) * P + L.xl + ix, c = iy * L.nx + ix;
    // a negative offset's coefficient is the neighbour's; outside the grid the
    // index is clamped (times the ghost's zero)
    auto at = [&](int64_t k) { return k > 0 ? k : 0; };
    const double *c1 = coefP + N, *c2p = c1 + N, *c3 = c2p + N, *c4 = c3 + N;
    const Asm9 k = {coefP[c],         c4[at(c - L.nx - 1)], c3[at(c - L.nx)],
                    c2p[at(c - L.nx + 1)], c1[at(c - 1)],   c1[c],
                    c2p[c],           c3[c],                c4[c]};
    const double unew =
        asm2d_step(k, u[i - P - 1], u[i - P], u[i - P + 1], u[i - 1], u[i], u[i + 1], u[i + P - 1],
                   u[i + P], u[i + P + 1], um[i], dco[i], fre[i], fim[i], c0, a, -b);
    out[i] = unew;
    if (flags) {
        if ((flags & 1) && slot->snap_part) slot->snap_part[2 * c] = unew;
        if ((flags & 2) && slot->final_part) slot->final_part[2 * c] = unew;
    }
}

void launch_step_asm(const Layout &L, const double *u, const double *um, double *out,
                     const double *coefP,
                     const double *dco, const double *fre, const double *fim, double c0, double a,
                     double b, const OutSlot *slot, int flags, cudaStream_t s, const RhsSet &R,
                     bool overlap)
{
    if (L.d == 2) {
        dim3 grd((unsigned)((L.nx + 31) / 32), (unsigned)((L.ny + 7) / 8), (unsigned)R.slots);
        launch_step_kernel(step2d_asm_kernel<true>, step2d_asm_kernel<false>, kFull64, grd,
                           dim3(32, 8), R, s, overlap, u, um, out, coefP, dco, fre, fim, L, c0, a, b,
                           slot, flags, R);
        ++g_launches;
        return;
    }
    const int64_t gx = (L.nx + 31) / 32, gy = (L.ny + kAsmTY - 1) / kAsmTY;
    const int64_t tiles = gx * gy * R.slots;
    const int64_t want = 8 * (int64_t)sm_count();
    int zc = (int)std::min<int64_t>(16, std::max<int64_t>(1, L.nz * tiles / want));
    zc = (int)std::min<int64_t>(zc, L.nz);
    const int nchunks = (int)((L.nz + zc - 1) / zc);
    const int64_t fold = (gy + 65534) / 65535;
    dim3 grd((unsigned)(gx * fold), (unsigned)((gy + fold - 1) / fold),
             (unsigned)(nchunks * R.slots));
    auto go = [&](auto early, auto late) {
        launch_step_kernel(early, late, kFull, grd, dim3(32, kAsmTY), R, s, overlap, u, um, out,
                           coefP, dco, fre, fim, L, c0, a, b, slot, flags, R, zc, nchunks);
    };
    if (fold > 1) go(step3d_asm_kernel<true, true>, step3d_asm_kernel<true, false>);
    else go(step3d_asm_kernel<false, true>, step3d_asm_kernel<false, false>);
    ++g_launches;
}

// ---------------------------------------------------------------------------
// frequency-adapted backward-differences damped leapfrog (Def. of I_abd)
// ---------------------------------------------------------------------------
//
//   u_{n+1} = (2 - K - L) u_n - (I - L) u_{n-1} + g_n,
//   K = (dt^2/alpha)(Re H + omega^2) - (dt beta (1 - cos(omega dt))/alpha) B,
//   L = (beta dt/alpha) B,  B = Im H / omega,
// which regroups into
//   u_{n+1} = [2 - (dt^2/alpha)(Re H + omega^2)] u_n - u_{n-1}
//             - (beta dt/(alpha omega)) Im H (cos(omega dt) u_n - u_{n-1}) + g_n.
// The first bracket is the same h^2-scaled cell stencil as I_acd's (StepCoef,
// q*kappa per cell).  Im H: node damping omega_phys R_i (damp holds
// beta dt omega_phys R_i/(alpha omega) per node), or cell damping (damp holds
// that coefficient with R_cell per cell; the operator is the cell-mass stencil
// sum_o M_s (sum of damp over the shared cells) w_{beta+o}).  Reads u_{n-1} at
// the neighbours in the cell case, so u_{n+1} goes to a third plane.

template <typename T, bool kCell, bool kEarly>
__global__ void __launch_bounds__(256)
abd_step_kernel(const T *__restrict__ u, const T *__restrict__ um, T *__restrict__ out,
                const T *__restrict__ kap, const T *__restrict__ damp,
                const T *__restrict__ fre, const T *__restrict__ fim, Layout L, StepCoef<T> C,
                T a, T b, T cth, const OutSlot *__restrict__ slot, int flags, RhsSet R, int nz)
{
    grid_dep_begin<kEarly>();
    const int64_t ix = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t iy = (int64_t)blockIdx.y * blockDim.y + threadIdx.y;
    int rhs;
    if (!rhs_of_slot(R, (int)blockIdx.z / nz, rhs)) return;
    const int64_t iz = blockIdx.z % nz;
    if (ix >= L.nx || iy >= L.ny) return;
    const int64_t off = rhs * R.stride;
    u += off;
    um += off;
    out += off;
    fre += off;
    fim += off;
    slot += rhs;
    const int64_t P = L.pitch, Q = L.plane;
    const int64_t i = L.node(ix, iy, iz);
    constexpr int D = 3, NC = 1 << D;
    // the node's cells, bit t of index c: upper (1) or lower (0) cell along axis t
    // (t = 0: x, 1: y, 2: z)
    T kc[NC], dc[NC];
#pragma unroll
    for (int cidx = 0; cidx < NC; ++cidx) {
        const int ax = cidx & 1, ay = (cidx >> 1) & 1, az = (cidx >> 2) & 1;
        const int64_t ci = i - (1 - ax) - (1 - ay) * P - (D == 3 ? (1 - az) * Q : 0);
        kc[cidx] = kap[ci];
        if (kCell) dc[cidx] = damp[ci];
    }
    T accA = T(0), accB = T(0);
#pragma unroll
    for (int oz = (D == 3 ? -1 : 0); oz <= (D == 3 ? 1 : 0); ++oz)
#pragma unroll
        for (int oy = -1; oy <= 1; ++oy)
#pragma unroll
            for (int ox = -1; ox <= 1; ++ox) {
                const int sh = (ox != 0) + (oy != 0) + (oz != 0);
                T ks = T(0), ds = T(0);
#pragma unroll
                for (int cidx = 0; cidx < NC; ++cidx) {
                    const int ax = cidx & 1, ay = (cidx >> 1) & 1, az = (cidx >> 2) & 1;
                    const bool shared = (ox == 0 || ox == 2 * ax - 1) &&
                                        (oy == 0 || oy == 2 * ay - 1) &&
                                        (D == 2 || oz == 0 || oz == 2 * az - 1);
                    if (shared) {
                        ks += kc[cidx];
                        if (kCell) ds += dc[cidx];
                    }
                }
                const int64_t j = i + ox + oy * P + (D == 3 ? oz * Q : 0);
                const T v = u[j];
                const T coef = (sh == 0) ? C.c0 + C.mt[0] * ks : C.mt[sh] * ks - C.cs[sh];
                accA += coef * v;
                if (kCell) accB += C.mt[sh] * ds * (cth * v - um[j]);
            }
    const T prev = um[i];
    if (!kCell) accB = damp[i] * (cth * u[i] - prev);
    const T unew = accA - prev - accB + (a * fre[i] - b * fim[i]);
    out[i] = unew;
    if (flags) {
        const int64_t c = (iz * L.ny + iy) * L.nx + ix;
        if ((flags & 1) && slot->snap_part) slot->snap_part[2 * c] = (double)unew;
        if ((flags & 2) && slot->final_part) slot->final_part[2 * c] = (double)unew;
    }
}

// The 2-D step, ROWS nodes of a column per thread with all operands loaded before
// the first sum (a row of u_n and u_{n-1} serves the nodes above and below it too);
// the expressions and their order are abd_step_kernel's.  ROWS: the most of 4, 2, 1
// that leaves two blocks per SM, or in FP64 the best balanced one of those.  401^2 cell
// damping: 2.0 us per step (two rows), 3.0 with the per-node loads of the 3-D form.
template <typename T, bool kCell, int ROWS, bool kEarly>
__global__ void __launch_bounds__(256)
abd_step2d_kernel(const T *__restrict__ u, const T *__restrict__ um, T *__restrict__ out,
                  const T *__restrict__ kap, const T *__restrict__ damp,
                  const T *__restrict__ fre, const T *__restrict__ fim, Layout L, StepCoef<T> C,
                  T a, T b, T cth, const OutSlot *__restrict__ slot, int flags, RhsSet R)
{
    const int64_t ix = (int64_t)blockIdx.x * 32 + threadIdx.x;
    const int64_t iy0 = ((int64_t)blockIdx.y * 8 + threadIdx.y) * ROWS;
    const bool in = ix < L.nx && iy0 < L.ny;
    const int64_t P = L.pitch, i0 = (iy0 + 1) * P + L.xl + ix;
    int64_t at[ROWS + 2];                   // row r - 1; rows below the grid: its last ghost row
#pragma unroll
    for (int r = 0; r < ROWS + 2; ++r) at[r] = i0 + (min(iy0 + r - 1, L.ny) - iy0) * P;
    // the coefficients, which no step writes, before the wait for the previous step
    T k[ROWS + 1][2], dc[ROWS + 1][2], dn[ROWS];
#pragma unroll
    for (int r = 0; r < ROWS + 1; ++r)
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            k[r][x] = in ? kap[at[r] + x - 1] : T(0);
            dc[r][x] = kCell && in ? damp[at[r] + x - 1] : T(0);
        }
#pragma unroll
    for (int r = 0; r < ROWS; ++r) dn[r] = !kCell && in ? damp[at[r + 1]] : T(0);
    grid_dep_begin<kEarly>();
    int rhs;
    if (!rhs_of_slot(R, (int)blockIdx.z, rhs)) return;
    if (!in) return;
    const int64_t off = rhs * R.stride;
    u += off;
    um += off;
    out += off;
    fre += off;
    fim += off;
    slot += rhs;
    constexpr int MX = kCell ? 3 : 1;       // columns of u_{n-1} read
    T w[ROWS + 2][3], wm[ROWS + 2][3], fr[ROWS], fi[ROWS];
#pragma unroll
    for (int r = 0; r < ROWS + 2; ++r) {
#pragma unroll
        for (int x = 0; x < 3; ++x) w[r][x] = u[at[r] + x - 1];
#pragma unroll
        for (int x = 0; x < 3; ++x)
            wm[r][x] = (MX == 3 || (x == 1 && r >= 1 && r <= ROWS)) ? um[at[r] + x - 1] : T(0);
    }
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
        fr[r] = fre[at[r + 1]];
        fi[r] = fim[at[r + 1]];
    }
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
        if (r > 0 && iy0 + r >= L.ny) break;
        T accA = T(0), accB = T(0);
#pragma unroll
        for (int oy = -1; oy <= 1; ++oy)
#pragma unroll
            for (int ox = -1; ox <= 1; ++ox) {
                const int sh = (ox != 0) + (oy != 0);
                T ks = T(0), ds = T(0);
#pragma unroll
                for (int cidx = 0; cidx < 4; ++cidx) {
                    const int ax = cidx & 1, ay = cidx >> 1;
                    if ((ox == 0 || ox == 2 * ax - 1) && (oy == 0 || oy == 2 * ay - 1)) {
                        ks += k[r + ay][ax];
                        if (kCell) ds += dc[r + ay][ax];
                    }
                }
                const T v = w[r + 1 + oy][1 + ox];
                const T coef = (sh == 0) ? C.c0 + C.mt[0] * ks : C.mt[sh] * ks - C.cs[sh];
                accA += coef * v;
                if (kCell) accB += C.mt[sh] * ds * (cth * v - wm[r + 1 + oy][1 + ox]);
            }
        const T prev = wm[r + 1][1];
        if (!kCell) accB = dn[r] * (cth * w[r + 1][1] - prev);
        const T unew = accA - prev - accB + (a * fr[r] - b * fi[r]);
        out[at[r + 1]] = unew;
        if (flags) {
            const int64_t c = (iy0 + r) * L.nx + ix;
            if ((flags & 1) && slot->snap_part) slot->snap_part[2 * c] = (double)unew;
            if ((flags & 2) && slot->final_part) slot->final_part[2 * c] = (double)unew;
        }
    }
}

template <typename T>
void launch_abd_step(const Layout &L, const T *u, const T *um, T *out, const T *kap,
                     const T *damp, bool cell, const T *fre, const T *fim, const StepCoef<T> &C,
                     T a, T b, T cth, const OutSlot *slot, int flags, cudaStream_t s,
                     const RhsSet &R, bool overlap)
{
    const int nz = (int)L.nz;
    dim3 blk(32, 8);
    dim3 grd((unsigned)((L.nx + 31) / 32), (unsigned)((L.ny + 7) / 8), (unsigned)(nz * R.slots));
    if (L.d == 2) {
        const unsigned gx = (unsigned)((L.nx + 31) / 32);
        auto blocks = [&](int rows) { return (L.ny + 8 * rows - 1) / (8 * rows); };
        // FP64 counts the right-hand sides that are sure to be active: with 2 of 8 active,
        // 150 x 170 cell damping took 3.1 ms per application with two rows, 2.1 with one; with
        // one of 8, 401^2 7.8 with four, 6.4 with two
        const int64_t rhs = sizeof(T) == 8 ? R.sure : R.slots;
        auto fits = [&](int rows) { return gx * blocks(rows) * rhs >= 2 * (int64_t)sm_count(); };
        int rows = fits(4) ? 4 : fits(2) ? 2 : 1;
        if (sizeof(T) == 8) {
            // the pipe of the SM with the most blocks sets the time; a node costs 0.83 with two
            // rows and 0.8 with four of what it costs with one (560^2 node damping: 23.7, 22.3
            // and 25.5 us per step with 1, 2, 4 rows)
            const double node[5] = {0.0, 1.0, 0.83, 0.0, 0.8};
            auto cost = [&](int k) {
                const int64_t nsm = sm_count(), n = gx * blocks(k) * rhs;
                return (double)((n + nsm - 1) / nsm) * k * node[k];
            };
            for (int k = rows / 2; k >= 1; k /= 2)
                if (cost(k) < cost(rows)) rows = k;
        }
        const dim3 grd2(gx, (unsigned)blocks(rows), (unsigned)R.slots);
        auto go = [&](auto early, auto late) {
            // (FP32: always before the wait, as the coefficients that the next steps load
            // meanwhile are then half of a step: 401^2 cell 2.29 us, 2.57 after it, 2.76 in
            // stream order; 0.8 to 0.96 of stream order from 60^2 to 1200^2)
            if constexpr (sizeof(T) == 4)
                launch_ex(early, grd2, blk, 0, s, overlap, u, um, out, kap, damp, fre, fim, L, C, a,
                          b, cth, slot, flags, R);
            else
                launch_step_kernel(early, late, rows == 1 ? kFull64 : kFullRows, grd2, blk, R, s,
                                   overlap, u, um, out, kap, damp, fre, fim, L, C, a, b, cth, slot,
                                   flags, R);
        };
        auto with_rows = [&](auto cellc, auto rowsc) {
            constexpr bool kCell = decltype(cellc)::value;
            constexpr int ROWS = decltype(rowsc)::value;
            go(abd_step2d_kernel<T, kCell, ROWS, true>,
               abd_step2d_kernel<T, kCell, ROWS, sizeof(T) == 4>);
        };
        auto with_cell = [&](auto cellc) {
            if (rows == 4) with_rows(cellc, std::integral_constant<int, 4>{});
            else if (rows == 2) with_rows(cellc, std::integral_constant<int, 2>{});
            else with_rows(cellc, std::integral_constant<int, 1>{});
        };
        if (cell) with_cell(std::true_type{});
        else with_cell(std::false_type{});
    } else {
        auto go = [&](auto early, auto late) {
            launch_step_kernel(early, late, sizeof(T) == 8 ? kFull64 : kFull, grd, blk, R, s,
                               overlap, u, um, out, kap, damp, fre, fim, L, C, a, b, cth, slot,
                               flags, R, nz);
        };
        if (cell) go(abd_step_kernel<T, true, true>, abd_step_kernel<T, true, false>);
        else go(abd_step_kernel<T, false, true>, abd_step_kernel<T, false, false>);
    }
    ++g_launches;
}
template void launch_abd_step<float>(const Layout &, const float *, const float *, float *,
                                     const float *, const float *, bool, const float *,
                                     const float *, const StepCoef<float> &, float, float, float,
                                     const OutSlot *, int, cudaStream_t, const RhsSet &, bool);
template void launch_abd_step<double>(const Layout &, const double *, const double *, double *,
                                      const double *, const double *, bool, const double *,
                                      const double *, const StepCoef<double> &, double, double,
                                      double, const OutSlot *, int, cudaStream_t, const RhsSet &,
                                      bool);

// ---------------------------------------------------------------------------
// projection read-out: compensated sums of e^{-i theta_j} u_j
// ---------------------------------------------------------------------------

// one compensated (Kahan) addition s += x, c carrying the negated lost low part
template <typename T>
__device__ __forceinline__ void kahan_add(T &s, T &c, T x)
{
    const T y = x - c;
    const T t = s + y;
    c = (t - s) - y;
    s = t;
}

// acc planes per rhs (stride apart), compact node order: [s_re, s_im, c_re, c_im]
// x N.  For the state u (padded layout) of every listed rhs:
//   s_re += wc u, s_im += ws u   (wc = cos theta, ws = -sin theta), compensated.
template <typename T>
__global__ void __launch_bounds__(256)
project_accumulate_kernel(Layout L, const T *__restrict__ u, T *__restrict__ acc, int64_t astride,
                          T wc, T ws, RhsSet R, int nz)
{
    const int64_t ix = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t iy = (int64_t)blockIdx.y * blockDim.y + threadIdx.y;
    int rhs;
    if (!rhs_of_slot(R, (int)blockIdx.z / nz, rhs)) return;
    const int64_t iz = blockIdx.z % nz;
    if (ix >= L.nx || iy >= L.ny) return;
    const int64_t c = (iz * L.ny + iy) * L.nx + ix;
    const T v = u[rhs * R.stride + L.node(ix, iy, iz)];
    T *a = acc + rhs * astride;
    T sr = a[c], si = a[L.N + c], cr = a[2 * L.N + c], ci = a[3 * L.N + c];
    kahan_add(sr, cr, wc * v);
    kahan_add(si, ci, ws * v);
    a[c] = sr;
    a[L.N + c] = si;
    a[2 * L.N + c] = cr;
    a[3 * L.N + c] = ci;
}

template <typename T>
void launch_project_accumulate(const Layout &L, const T *u, T *acc, int64_t astride, T wc, T ws,
                               const RhsSet &R, cudaStream_t s)
{
    const int nz = (int)L.nz;
    dim3 blk(32, 8);
    dim3 grd((unsigned)((L.nx + 31) / 32), (unsigned)((L.ny + 7) / 8), (unsigned)(nz * R.slots));
    project_accumulate_kernel<T><<<grd, blk, 0, s>>>(L, u, acc, astride, wc, ws, R, nz);
    ++g_launches;
}
template void launch_project_accumulate<float>(const Layout &, const float *, float *, int64_t,
                                               float, float, const RhsSet &, cudaStream_t);
template void launch_project_accumulate<double>(const Layout &, const double *, double *, int64_t,
                                                double, double, const RhsSet &, cudaStream_t);

// U = scale (s - c) into the output slot of every listed rhs (real part to
// final_part, imaginary part to snap_part), in double
template <typename T>
__global__ void __launch_bounds__(256)
project_finish_kernel(int64_t N, const T *__restrict__ acc, int64_t astride, double scale,
                      const OutSlot *__restrict__ slot, RhsSet R)
{
    int rhs;
    if (!rhs_of_slot(R, (int)blockIdx.y, rhs)) return;
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= N) return;
    const T *a = acc + rhs * astride;
    const OutSlot o = slot[rhs];
    const double re = scale * ((double)a[c] - (double)a[2 * N + c]);
    const double im = scale * ((double)a[N + c] - (double)a[3 * N + c]);
    if (o.final_part) o.final_part[2 * c] = re;
    if (o.snap_part) o.snap_part[2 * c] = im;
}

template <typename T>
void launch_project_finish(int64_t N, const T *acc, int64_t astride, double scale,
                           const OutSlot *slot, const RhsSet &R, cudaStream_t s)
{
    const int bs = 256;
    dim3 grd((unsigned)((N + bs - 1) / bs), (unsigned)R.slots);
    project_finish_kernel<T><<<grd, bs, 0, s>>>(N, acc, astride, scale, slot, R);
    ++g_launches;
}
template void launch_project_finish<float>(int64_t, const float *, int64_t, double,
                                           const OutSlot *, const RhsSet &, cudaStream_t);
template void launch_project_finish<double>(int64_t, const double *, int64_t, double,
                                            const OutSlot *, const RhsSet &, cudaStream_t);

// ---------------------------------------------------------------------------
// split / output slot
// ---------------------------------------------------------------------------

template <typename T>
__global__ void split_kernel(Layout L, const double2 *__restrict__ F, T *__restrict__ fre,
                             T *__restrict__ fim, int flip)
{
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= L.N) return;
    const int64_t ix = c % L.nx;
    const int64_t r = c / L.nx;
    const int64_t iy = r % L.ny;
    const int64_t iz = r / L.ny;
    const int64_t i = L.node(ix, iy, iz);
    const double2 f = F[c];
    // flip: forcing -i F, whose real part is Im F and imaginary part is -Re F
    fre[i] = (T)(flip ? f.y : f.x);
    fim[i] = (T)(flip ? -f.x : f.y);
}

template <typename T>
void launch_split(const Layout &L, const double2 *F, T *fre, T *fim, int flip, cudaStream_t s)
{
    const int bs = 256;
    split_kernel<T><<<(unsigned)((L.N + bs - 1) / bs), bs, 0, s>>>(L, F, fre, fim, flip);
    ++g_launches;
}
template void launch_split<float>(const Layout &, const double2 *, float *, float *, int, cudaStream_t);
template void launch_split<double>(const Layout &, const double2 *, double *, double *, int, cudaStream_t);

// batched forms: the active rhs list act (see RhsSet) selects the slots

template <typename T>
__global__ void split_batch_kernel(Layout L, const double2 *const *__restrict__ Fp,
                                   T *__restrict__ fre, T *__restrict__ fim, int64_t stride,
                                   int flip, const int *__restrict__ act)
{
    const int k = (int)blockIdx.y;
    if (k >= act[0]) return;
    const int r = act[1 + k];
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= L.N) return;
    const int64_t ix = c % L.nx;
    const int64_t q = c / L.nx;
    const int64_t iy = q % L.ny;
    const int64_t iz = q / L.ny;
    const int64_t i = L.node(ix, iy, iz) + r * stride;
    const double2 f = Fp[r][c];
    fre[i] = (T)(flip ? f.y : f.x);
    fim[i] = (T)(flip ? -f.x : f.y);
}

template <typename T>
void launch_split_batch(const Layout &L, const double2 *const *Fp, T *fre, T *fim, int64_t stride,
                        int flip, const int *act, int slots, cudaStream_t s)
{
    const int bs = 256;
    dim3 grd((unsigned)((L.N + bs - 1) / bs), (unsigned)slots);
    split_batch_kernel<T><<<grd, bs, 0, s>>>(L, Fp, fre, fim, stride, flip, act);
    ++g_launches;
}
template void launch_split_batch<float>(const Layout &, const double2 *const *, float *, float *,
                                        int64_t, int, const int *, int, cudaStream_t);
template void launch_split_batch<double>(const Layout &, const double2 *const *, double *, double *,
                                         int64_t, int, const int *, int, cudaStream_t);

struct ActList {
    int n;
    int idx[kMaxRhs];
};

__global__ void set_act_kernel(int *act, ActList a)
{
    const int t = threadIdx.x;
    if (t == 0) act[0] = a.n;
    if (t < a.n) act[1 + t] = a.idx[t];
}

void launch_set_act(int *act, int n, const int *idx, cudaStream_t s)
{
    ActList a;
    a.n = n;
    for (int k = 0; k < n && k < kMaxRhs; ++k) a.idx[k] = idx[k];
    for (int k = n; k < kMaxRhs; ++k) a.idx[k] = 0;
    set_act_kernel<<<1, kMaxRhs, 0, s>>>(act, a);
    ++g_launches;
}

// output slots of the listed rhs r: the final state of run `run` goes to the
// real (run 0) or imaginary (run 1) part of Up[r]; with one run (Table 1) the
// snapshot goes to the imaginary part
__global__ void set_slots_kernel(OutSlot *slot, double2 *const *Up, int run, int runs,
                                 const int *act)
{
    const int k = threadIdx.x;
    if (k >= act[0]) return;
    const int r = act[1 + k];
    double *base = reinterpret_cast<double *>(Up[r]);
    slot[r].final_part = base + run;
    slot[r].snap_part = (runs == 1) ? base + 1 : nullptr;
}

void launch_set_slots(OutSlot *slot, double2 *const *Up, int run, int runs, const int *act,
                      int slots, cudaStream_t s)
{
    set_slots_kernel<<<1, slots, 0, s>>>(slot, Up, run, runs, act);
    ++g_launches;
}

__global__ void set_slot_kernel(OutSlot *slot, double *final_part, double *snap_part)
{
    slot->final_part = final_part;
    slot->snap_part = snap_part;
}

void launch_set_slot(OutSlot *slot, double *final_part, double *snap_part, cudaStream_t s)
{
    set_slot_kernel<<<1, 1, 0, s>>>(slot, final_part, snap_part);
    ++g_launches;
}

// ---------------------------------------------------------------------------
// true operator, complex128
// ---------------------------------------------------------------------------

struct HCoef {
    double S2[4];   // 2^{d-s} S_s
    double M[4];
};

// Linear index of the offset (oz, oy, ox) in {-1,0,1}^3: (oz+1) 9 + (oy+1) 3 + (ox+1);
// the centre is 13.  H is symmetric, so only the centre and the offsets with a
// larger index ("positive": first non-zero of (oz, oy, ox) is +1) are stored:
// plane lin - 13.  The coefficient of a negative offset o at node beta is the
// stored coefficient of -o at the node beta + o.
__host__ __device__ constexpr int hlin(int oz, int oy, int ox)
{
    return (oz + 1) * 9 + (oy + 1) * 3 + (ox + 1);
}

// plane p (0 = centre, 1..13 positive offsets; 2-D: oz = 0, planes 0..4) of
// node (ix, iy, iz): 2^{d-s} S_s - M_s * (sum of kappa over the cells that
// contain the node and its neighbour), not yet scaled by 1/h^2; 0 where the
// neighbour is outside the grid
__global__ void __launch_bounds__(256)
assemble_H_kernel(Layout L, const double *__restrict__ kap64, HCoef C, double *__restrict__ coefP,
                  int nplanes)
{
    const int64_t ix = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t iy = (int64_t)blockIdx.y * blockDim.y + threadIdx.y;
    const int64_t iz = blockIdx.z;
    if (ix >= L.nx || iy >= L.ny) return;
    const int64_t c = (iz * L.ny + iy) * L.nx + ix;
    const int64_t i = L.node(ix, iy, iz);    // position in the padded cell array
    const int64_t P = L.pitch, Q = L.plane;
    for (int p = 0; p < nplanes; ++p) {
        const int lin = p + 13;
        const int oz = lin / 9 - 1, oy = (lin / 3) % 3 - 1, ox = lin % 3 - 1;
        const int64_t jz = iz + oz, jy = iy + oy, jx = ix + ox;
        double w = 0.0;
        if (jz >= 0 && jz < L.nz && jy >= 0 && jy < L.ny && jx >= 0 && jx < L.nx) {
            const int s = (oz != 0) + (oy != 0) + (ox != 0);
            // cells shared by the node and its neighbour: lower (offset -1), upper
            // (+1) or both (0) per axis
            double ks = 0.0;
            for (int az = (L.d == 3 ? 0 : 1); az < 2; ++az) {
                if (L.d == 3 && ((oz < 0 && az == 1) || (oz > 0 && az == 0))) continue;
                for (int ay = 0; ay < 2; ++ay) {
                    if ((oy < 0 && ay == 1) || (oy > 0 && ay == 0)) continue;
                    for (int ax = 0; ax < 2; ++ax) {
                        if ((ox < 0 && ax == 1) || (ox > 0 && ax == 0)) continue;
                        ks += kap64[i - (L.d == 3 ? (1 - az) * Q : 0) - (1 - ay) * P - (1 - ax)];
                    }
                }
            }
            w = C.S2[s] - C.M[s] * ks;
        }
        coefP[p * L.N + c] = w;
    }
}

void launch_assemble_H(const Layout &L, const double *kap64, const double S2[4], const double M[4],
                       double *coefP, cudaStream_t s)
{
    HCoef C;
    for (int k = 0; k < 4; ++k) { C.S2[k] = S2[k]; C.M[k] = M[k]; }
    dim3 blk(32, 8);
    dim3 grd((unsigned)((L.nx + 31) / 32), (unsigned)((L.ny + 7) / 8), (unsigned)L.nz);
    assemble_H_kernel<<<grd, blk, 0, s>>>(L, kap64, C, coefP, h_planes(L.d));
    ++g_launches;
}

// Y = H X (or F - H X) from the assembled coefficients: per node 3^D
// coefficient x neighbour products for the real and the imaginary part, one
// FP64 FMA each; neighbours outside the grid are the zero Dirichlet ghosts
template <int D, bool kImH>
__global__ void __launch_bounds__(256)
apply_H_asm_kernel(int64_t nx, int64_t ny, int64_t nz, const double *__restrict__ coefP,
                   const double *__restrict__ coefI, const double *__restrict__ imH, double h0,
                   double ih2, const double2 *__restrict__ X, const double2 *__restrict__ F,
                   double2 *__restrict__ Y)
{
    const int64_t ix = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t iy = (int64_t)blockIdx.y * blockDim.y + threadIdx.y;
    const int64_t iz = blockIdx.z;
    if (ix >= nx || iy >= ny) return;
    const int64_t N = nx * ny * nz;
    const int64_t c = (iz * ny + iy) * nx + ix;
    double re = 0.0, im = 0.0, qr = 0.0, qi = 0.0;
#pragma unroll
    for (int oz = (D == 3 ? -1 : 0); oz <= (D == 3 ? 1 : 0); ++oz)
#pragma unroll
        for (int oy = -1; oy <= 1; ++oy)
#pragma unroll
            for (int ox = -1; ox <= 1; ++ox) {
                const bool in = iz + oz >= 0 && iz + oz < nz && iy + oy >= 0 && iy + oy < ny &&
                                ix + ox >= 0 && ix + ox < nx;
                if (!in) continue;
                const int64_t cn = c + ((int64_t)oz * ny + oy) * nx + ox;
                const int lin = hlin(oz, oy, ox);
                const int64_t ci = (lin >= 13) ? (lin - 13) * N + c : (13 - lin) * N + cn;
                const double w = lin == 13 ? coefP[ci] + h0 : coefP[ci];
                const double2 x = X[cn];
                re = fma(w, x.x, re);
                im = fma(w, x.y, im);
                if (kImH) {                       // non-diagonal Im H (cell damping)
                    const double wi = coefI[ci];
                    qr = fma(wi, x.x, qr);
                    qi = fma(wi, x.y, qi);
                }
            }
    const double2 xc = X[c];
    const double damp = imH[c];
    double2 y;
    // H x = (Re H x_r - Im H x_i) + i (Re H x_i + Im H x_r)
    y.x = ih2 * re - damp * xc.y - qi;
    y.y = ih2 * im + damp * xc.x + qr;
    if (F) {
        const double2 f = F[c];
        y.x = f.x - y.x;
        y.y = f.y - y.y;
    }
    Y[c] = y;
}

void launch_apply_H(const Layout &L, const double *coefP, const double *imH, double h0, double ih2,
                    const double2 *X, const double2 *F, double2 *Y, cudaStream_t s,
                    const double *coefI)
{
    dim3 blk(32, 8);
    dim3 grd((unsigned)((L.nx + 31) / 32), (unsigned)((L.ny + 7) / 8), (unsigned)L.nz);
#define HTD_AH(DD, II) \
    apply_H_asm_kernel<DD, II><<<grd, blk, 0, s>>>(L.nx, L.ny, L.nz, coefP, coefI, imH, h0, ih2, X, F, Y)
    if (L.d == 3) {
        if (coefI) HTD_AH(3, true); else HTD_AH(3, false);
    } else {
        if (coefI) HTD_AH(2, true); else HTD_AH(2, false);
    }
#undef HTD_AH
    ++g_launches;
}

// ---------------------------------------------------------------------------
// Krylov vector operations (complex128)
// ---------------------------------------------------------------------------

constexpr int kRedThreads = 256;

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// block-wide sum of (re, im); result valid in thread 0
__device__ __forceinline__ double2 block_sum(double re, double im)
{
    __shared__ double sre[kRedThreads / 32], sim[kRedThreads / 32];
    re = warp_sum(re);
    im = warp_sum(im);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) { sre[warp] = re; sim[warp] = im; }
    __syncthreads();
    double2 out = make_double2(0.0, 0.0);
    if (warp == 0) {
        re = lane < kRedThreads / 32 ? sre[lane] : 0.0;
        im = lane < kRedThreads / 32 ? sim[lane] : 0.0;
        re = warp_sum(re);
        im = warp_sum(im);
        out = make_double2(re, im);
    }
    return out;
}

// One pass over the data for a group of up to kDotGroup basis vectors: each
// thread reads w[i] once and accumulates conj(V_k[i]) w[i] for the group, two
// elements per loop trip (more loads in flight).  Every complex product costs
// four FP64 FMAs on GB300's narrow FP64 pipe, so the kernel is FP64-bound; the
// block's 2 x kDotGroup sums are reduced together at the end.
constexpr int kDotGroup = 8;

// (re, im) += conj(a) b as four FP64 FMAs
__device__ __forceinline__ void cmac_conj(double &re, double &im, double2 a, double2 b)
{
    re = fma(a.x, b.x, re);
    re = fma(a.y, b.y, re);
    im = fma(a.x, b.y, im);
    im = fma(-a.y, b.x, im);
}

__global__ void __launch_bounds__(kRedThreads)
dots_kernel(const double2 *__restrict__ V, int64_t ldv, int kcount, const double2 *__restrict__ w,
            int64_t N, double2 *__restrict__ partial, int nb)
{
    const int k0 = blockIdx.y * kDotGroup;
    const int kn = min(kDotGroup, kcount - k0);
    double re[kDotGroup], im[kDotGroup];
#pragma unroll
    for (int q = 0; q < kDotGroup; ++q) { re[q] = 0.0; im[q] = 0.0; }
    const int64_t stride = (int64_t)nb * kRedThreads;
    int64_t i = (int64_t)blockIdx.x * kRedThreads + threadIdx.x;
    for (; i + stride < N; i += 2 * stride) {
        const double2 b0 = w[i], b1 = w[i + stride];
#pragma unroll
        for (int q = 0; q < kDotGroup; ++q) {
            if (q < kn) {
                const double2 *vq = V + (int64_t)(k0 + q) * ldv;
                const double2 a0 = vq[i], a1 = vq[i + stride];
                cmac_conj(re[q], im[q], a0, b0);
                cmac_conj(re[q], im[q], a1, b1);
            }
        }
    }
    if (i < N) {
        const double2 b = w[i];
#pragma unroll
        for (int q = 0; q < kDotGroup; ++q)
            if (q < kn) cmac_conj(re[q], im[q], V[(int64_t)(k0 + q) * ldv + i], b);
    }
    // block reduction of all 2 x kDotGroup sums: within warps, then across warps
    __shared__ double red[kRedThreads / 32][2 * kDotGroup];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < kDotGroup; ++q) {
        const double r = warp_sum(re[q]), m = warp_sum(im[q]);
        if (lane == 0) {
            red[warp][2 * q] = r;
            red[warp][2 * q + 1] = m;
        }
    }
    __syncthreads();
    if (threadIdx.x < 2 * kDotGroup && (int)threadIdx.x / 2 < kn) {
        double t = 0.0;
#pragma unroll
        for (int wv = 0; wv < kRedThreads / 32; ++wv) t += red[wv][threadIdx.x];
        double *out = reinterpret_cast<double *>(partial + (int64_t)(k0 + threadIdx.x / 2) * nb +
                                                 blockIdx.x);
        out[threadIdx.x & 1] = t;
    }
}

int dots_blocks(int64_t N)
{
    const int64_t cap = std::min<int64_t>(4 * (int64_t)sm_count(), kMaxDotBlocks);
    int64_t nb = (N + 8 * kRedThreads - 1) / (8 * kRedThreads);
    if (nb > cap) nb = cap;
    if (nb < 1) nb = 1;
    return (int)nb;
}

void launch_dots(const double2 *V, int64_t ldv, int kcount, const double2 *w, int64_t N,
                 double2 *partial, int nb, cudaStream_t s)
{
    dim3 grd((unsigned)nb, (unsigned)((kcount + kDotGroup - 1) / kDotGroup));
    dots_kernel<<<grd, kRedThreads, 0, s>>>(V, ldv, kcount, w, N, partial, nb);
    ++g_launches;
}

__global__ void __launch_bounds__(kRedThreads)
reduce_kernel(const double2 *__restrict__ partial, int nb, double2 *__restrict__ out)
{
    const int k = blockIdx.x;
    double re = 0.0, im = 0.0;
    for (int b = threadIdx.x; b < nb; b += kRedThreads) {
        const double2 p = partial[(int64_t)k * nb + b];
        re += p.x;
        im += p.y;
    }
    const double2 t = block_sum(re, im);
    if (threadIdx.x == 0) out[k] = t;
}

void launch_reduce(const double2 *partial, int nb, int kcount, double2 *out, cudaStream_t s)
{
    reduce_kernel<<<kcount, kRedThreads, 0, s>>>(partial, nb, out);
    ++g_launches;
}

// w -= sum_k h_k V_k and U += sum_k y_k Z_k: two elements per thread (256
// apart, so that loads stay coalesced) for two independent FP64 chains, four
// FMAs per complex product
constexpr int kCombThreads = 256;

template <bool kAdd>
__global__ void __launch_bounds__(kCombThreads)
combination_kernel(const double2 *__restrict__ V, int64_t ldv, int kcount,
                   const double2 *__restrict__ h, double2 *__restrict__ w, int64_t N)
{
    __shared__ double2 sh[72];
    for (int k = threadIdx.x; k < kcount; k += blockDim.x) sh[k] = h[k];
    __syncthreads();
    const int64_t i0 = (int64_t)blockIdx.x * (2 * kCombThreads) + threadIdx.x;
    const int64_t i1 = i0 + kCombThreads;
    const bool has1 = i1 < N;
    if (i0 >= N) return;
    double2 acc0 = w[i0];
    double2 acc1 = has1 ? w[i1] : make_double2(0.0, 0.0);
#pragma unroll 4
    for (int k = 0; k < kcount; ++k) {
        const double2 *vk = V + (int64_t)k * ldv;
        const double2 c = sh[k];
        const double cx = kAdd ? c.x : -c.x, cy = kAdd ? c.y : -c.y;
        const double2 v0 = vk[i0];
        const double2 v1 = has1 ? vk[i1] : make_double2(0.0, 0.0);
        acc0.x = fma(cx, v0.x, acc0.x);
        acc0.x = fma(-cy, v0.y, acc0.x);
        acc0.y = fma(cx, v0.y, acc0.y);
        acc0.y = fma(cy, v0.x, acc0.y);
        acc1.x = fma(cx, v1.x, acc1.x);
        acc1.x = fma(-cy, v1.y, acc1.x);
        acc1.y = fma(cx, v1.y, acc1.y);
        acc1.y = fma(cy, v1.x, acc1.y);
    }
    w[i0] = acc0;
    if (has1) w[i1] = acc1;
}

void launch_sub_combination(const double2 *V, int64_t ldv, int kcount, const double2 *h,
                            double2 *w, int64_t N, cudaStream_t s)
{
    const unsigned nblk = (unsigned)((N + 2 * kCombThreads - 1) / (2 * kCombThreads));
    combination_kernel<false><<<nblk, kCombThreads, 0, s>>>(V, ldv, kcount, h, w, N);
    ++g_launches;
}

void launch_add_combination(const double2 *Z, int64_t ldz, int kcount, const double2 *y,
                            double2 *U, int64_t N, cudaStream_t s)
{
    const unsigned nblk = (unsigned)((N + 2 * kCombThreads - 1) / (2 * kCombThreads));
    combination_kernel<true><<<nblk, kCombThreads, 0, s>>>(Z, ldz, kcount, y, U, N);
    ++g_launches;
}

__global__ void scale_kernel(const double2 *__restrict__ w, double scale, double2 *__restrict__ v,
                             int64_t N)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const double2 a = w[i];
    v[i] = make_double2(a.x * scale, a.y * scale);
}

__global__ void scale_inplace_kernel(double2 *__restrict__ v, double scale, int64_t N)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const double2 a = v[i];
    v[i] = make_double2(a.x * scale, a.y * scale);
}

void launch_scale(const double2 *w, double scale, double2 *v, int64_t N, cudaStream_t s)
{
    const int bs = 256;
    if (w == v) {
        scale_inplace_kernel<<<(unsigned)((N + bs - 1) / bs), bs, 0, s>>>(v, scale, N);
        ++g_launches;
        return;
    }
    scale_kernel<<<(unsigned)((N + bs - 1) / bs), bs, 0, s>>>(w, scale, v, N);
    ++g_launches;
}

}  // namespace htd

namespace htd {

// ---------------------------------------------------------------------------
// receiver misfit and gradient (adjoint state)
// ---------------------------------------------------------------------------

__global__ void gather_residual_kernel(const double2 *__restrict__ U, const double2 *__restrict__ d,
                                       const int64_t *__restrict__ rec, int nrec,
                                       double2 *__restrict__ res)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nrec) return;
    const double2 u = U[rec[k]], dd = d[k];
    res[k] = make_double2(u.x - dd.x, u.y - dd.y);
}

__global__ void scatter_conj_kernel(const double2 *__restrict__ res, const int64_t *__restrict__ rec,
                                    int nrec, double2 *__restrict__ r)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nrec) return;
    double *p = reinterpret_cast<double *>(r + rec[k]);
    atomicAdd(p, res[k].x);          // receivers may repeat: accumulate conj(res)
    atomicAdd(p + 1, -res[k].y);
}

void launch_receiver_residual(const double2 *U, const double2 *d, const int64_t *rec, int nrec,
                              double2 *res, double2 *r, cudaStream_t s)
{
    if (nrec <= 0) return;
    const int bs = 256;
    gather_residual_kernel<<<(nrec + bs - 1) / bs, bs, 0, s>>>(U, d, rec, nrec, res);
    ++g_launches;
    scatter_conj_kernel<<<(nrec + bs - 1) / bs, bs, 0, s>>>(res, rec, nrec, r);
    ++g_launches;
}

// ---- gradient through the recurrence (htd_grad_td) --------------------------

// res[k] = U[rec[k]] - d[k]; adjoint forcing planes (padded, pre-zeroed):
// are[node(rec)] += Re res, aim[node(rec)] += Im res (receivers may repeat)
template <typename T>
__global__ void residual_planes_kernel(Layout L, const double2 *__restrict__ U,
                                       const double2 *__restrict__ d,
                                       const int64_t *__restrict__ rec, int nrec,
                                       double2 *__restrict__ res, T *__restrict__ are,
                                       T *__restrict__ aim)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nrec) return;
    const int64_t c = rec[k];
    const double2 u = U[c], dd = d[k];
    const double2 r = make_double2(u.x - dd.x, u.y - dd.y);
    res[k] = r;
    const int64_t ix = c % L.nx, q = c / L.nx, iy = q % L.ny, iz = q / L.ny;
    const int64_t i = L.node(ix, iy, iz);
    atomicAdd(are + i, (T)r.x);
    atomicAdd(aim + i, (T)r.y);
}

template <typename T>
void launch_residual_planes(const Layout &L, const double2 *U, const double2 *d,
                            const int64_t *rec, int nrec, double2 *res, T *are, T *aim,
                            cudaStream_t s)
{
    if (nrec <= 0) return;
    const int bs = 256;
    residual_planes_kernel<T><<<(nrec + bs - 1) / bs, bs, 0, s>>>(L, U, d, rec, nrec, res, are,
                                                                   aim);
    ++g_launches;
}
template void launch_residual_planes<float>(const Layout &, const double2 *, const double2 *,
                                            const int64_t *, int, double2 *, float *, float *,
                                            cudaStream_t);
template void launch_residual_planes<double>(const Layout &, const double2 *, const double2 *,
                                             const int64_t *, int, double2 *, double *, double *,
                                             cudaStream_t);

// (a call, not inlined: a conversion under a predicate takes the FP64 pipe for every
// x, taken or not)
__device__ __noinline__ double convert(float x) { return (double)x; }

// (double)x without the conversion instruction, which GB300 issues at the FP64
// pipe's two per clock and SM: the exponent rebiased and the mantissa moved by
// integer instructions, exact for every finite x (a denormal, frequent ahead of a
// wave front, is scaled by 2^24 first); infinities and NaNs are converted.
__device__ __forceinline__ double widen(float x)
{
    const bool tiny = (__float_as_uint(x) & 0x7f800000u) == 0u;
    const unsigned b = __float_as_uint(tiny ? __fmul_rn(x, 16777216.f) : x);
    const unsigned bias = tiny ? 0x38000000u - (24u << 20) : 0x38000000u;
    const unsigned hi = ((b & 0x7fffffffu) >> 3) + bias;
    double r = __hiloint2double((int)((b & 0x80000000u) | ((b << 1) ? hi : 0u)), (int)(b << 29));
    if ((b & 0x7f800000u) == 0x7f800000u) r = convert(x);
    return r;
}
__device__ __forceinline__ double widen(double x) { return x; }

template <typename T>
struct TdGradCoef {
    T M[4];
    double cm;      // -(dt^2/alpha) omega_phys^2
    double cR;      // beta dt omega_phys / (2 alpha omega)
};

// The terms k = k0, k0 - 1, .. k1 of the gradient sum of every source (grid.y), for
// the multipliers lam_k and the states u_k, u_{k-1}, u_{k-2} (all padded; the ghost
// ring is zero):
//   gm[cell] += cm sum_{b,g corners} lam_b M_{|b-g|} u_{k-1,g}
//   gR[node] += cR lam (u_k - u_{k-2})
// lam_k is plane k % nlam of lam, u_k plane k - s0 + 2 of seg; a source's planes lie
// sstride after the one's before, its sums gstride.  One thread per cell (compact
// (n+1)^d order) keeps the cell's sum over all the terms; the thread of cell a >= 0
// also does node a.  Products in the recurrence precision, sums in double, one
// term after the other, so the result does not depend on how the run is cut.
// One launch per segment instead of one per step: the sums are read and written once
// per segment, and two FP64 multiply-adds per term are left of that pipe's work
// (with the conversion instruction four: 334 us per segment of 40 steps at 512^2 with 4
// sources, 83 % of the pipe; 270 without it, and waiting on the loads until the next
// term's were issued ahead).
template <typename T, int D>
__global__ void __launch_bounds__(256)
grad_td_kernel(Layout L, TdGradCoef<T> G, const T *__restrict__ lam, int nlam,
               const T *__restrict__ seg, int64_t sstride, long long s0, long long k0, long long k1,
               double *__restrict__ gm, double *__restrict__ gR, int64_t gstride)
{
    const int64_t cx_n = L.nx + 1, cy_n = L.ny + 1, cz_n = (D == 3) ? L.nz + 1 : 1;
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= cx_n * cy_n * cz_n) return;
    const int64_t ax = c % cx_n - 1;
    const int64_t rr = c / cx_n;
    const int64_t ay = rr % cy_n - 1;
    const int64_t az = (D == 3) ? rr / cy_n - 1 : 0;
    constexpr int nc = (D == 3) ? 8 : 4;
    lam += blockIdx.y * sstride;
    seg += blockIdx.y * sstride;
    int64_t o[nc];                                 // corners from corner 0
#pragma unroll
    for (int b = 0; b < nc; ++b)
        o[b] = (b & 1) + ((b >> 1) & 1) * L.pitch + ((b >> 2) & 1) * L.plane;
    const int64_t i0 = L.node(ax, ay, az);
    const bool node = gR && ax >= 0 && ay >= 0 && (D == 2 || az >= 0) && ax < L.nx && ay < L.ny &&
                      (D == 2 || az < L.nz);
    const int64_t n = (az * L.ny + ay) * L.nx + ax;
    double sm = 0.0, sR = 0.0;
    if (gm) {
        gm += blockIdx.y * gstride;
        sm = gm[c];
    }
    T uk = T(0), uk1 = T(0);
    if (node) {
        gR += blockIdx.y * gstride;
        sR = gR[n];
        uk = seg[(k0 - s0 + 2) * L.total + i0];
        uk1 = seg[(k0 - s0 + 1) * L.total + i0];
    }
    // the next term's operands are loaded before the present one is summed
    int kl = (int)(k0 % nlam);
    T ln[nc], un[nc], u2n = T(0);
    auto load = [&](long long k) {
        const T *lk = lam + kl * L.total + i0, *uq = seg + (k - s0 + 1) * L.total + i0;
        if (--kl < 0) kl = nlam - 1;
#pragma unroll
        for (int b = 0; b < nc; ++b) {
            ln[b] = lk[o[b]];
            un[b] = uq[o[b]];
        }
        if (node) u2n = uq[-L.total];
    };
    load(k0);
    for (long long k = k0; k >= k1; --k) {
        T l8[nc], u8[nc];
        const T uk2 = u2n;
#pragma unroll
        for (int b = 0; b < nc; ++b) {
            l8[b] = ln[b];
            u8[b] = un[b];
        }
        if (k > k1) load(k - 1);
        if (gm) {
            T acc = T(0);
#pragma unroll
            for (int b = 0; b < nc; ++b) {
                T row = T(0);
#pragma unroll
                for (int g = 0; g < nc; ++g) row += G.M[__popc(b ^ g)] * u8[g];
                acc += l8[b] * row;
            }
            sm = fma(G.cm, widen(acc), sm);
        }
        if (node) {
            sR = fma(G.cR, widen(l8[0] * (uk - uk2)), sR);
            uk = uk1;
            uk1 = uk2;
        }
    }
    if (gm) gm[c] = sm;
    if (node) gR[n] = sR;
}

template <typename T>
void launch_grad_td(const Layout &L, const double M[4], double cm, double cR, const T *lam, int nlam,
                    const T *seg, int64_t sstride, int nsrc, long long s0, long long k0,
                    long long k1, double *gm, double *gR, int64_t gstride, cudaStream_t s)
{
    TdGradCoef<T> G;
    for (int k = 0; k < 4; ++k) G.M[k] = (T)M[k];
    G.cm = cm;
    G.cR = cR;
    const int64_t ncell = (L.nx + 1) * (L.ny + 1) * ((L.d == 3) ? L.nz + 1 : 1);
    const dim3 grd((unsigned)((ncell + 255) / 256), (unsigned)nsrc);
    if (L.d == 3)
        grad_td_kernel<T, 3><<<grd, 256, 0, s>>>(L, G, lam, nlam, seg, sstride, s0, k0, k1, gm, gR,
                                                 gstride);
    else
        grad_td_kernel<T, 2><<<grd, 256, 0, s>>>(L, G, lam, nlam, seg, sstride, s0, k0, k1, gm, gR,
                                                 gstride);
    ++g_launches;
}
template void launch_grad_td<float>(const Layout &, const double[4], double, double, const float *,
                                    int, const float *, int64_t, int, long long, long long,
                                    long long, double *, double *, int64_t, cudaStream_t);
template void launch_grad_td<double>(const Layout &, const double[4], double, double,
                                     const double *, int, const double *, int64_t, int, long long,
                                     long long, long long, double *, double *, int64_t,
                                     cudaStream_t);

// out[i] += the sources' sums in order (nsrc of them, gstride apart)
__global__ void __launch_bounds__(256)
add_sources_kernel(double *__restrict__ out, const double *__restrict__ g, int64_t gstride, int nsrc,
                   int64_t n)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double v = out[i];
    for (int q = 0; q < nsrc; ++q) v += g[q * gstride + i];
    out[i] = v;
}

void launch_add_sources(double *out, const double *g, int64_t gstride, int nsrc, int64_t n,
                        cudaStream_t s)
{
    add_sources_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(out, g, gstride, nsrc, n);
    ++g_launches;
}

struct GradCoef {
    double M[4];
    double w2;      // omega_phys^2
    double w;       // omega_phys
};

// per cell alpha: gm[alpha] += omega^2 Re sum_{beta,gamma in cell} mu_beta M_{|beta-gamma|} U_gamma
// (cells in the compact (n+1)^d order of the speed input; ghost corners are zero)
__global__ void __launch_bounds__(256)
grad_cells_kernel(Layout L, GradCoef G, const double2 *__restrict__ mu,
                  const double2 *__restrict__ U, double *__restrict__ gm)
{
    const int64_t cx_n = L.nx + 1, cy_n = L.ny + 1, cz_n = (L.d == 3) ? L.nz + 1 : 1;
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= cx_n * cy_n * cz_n) return;
    const int64_t ax = c % cx_n - 1;
    const int64_t rr = c / cx_n;
    const int64_t ay = rr % cy_n - 1;
    const int64_t az = (L.d == 3) ? rr / cy_n - 1 : 0;
    const int nc = (L.d == 3) ? 8 : 4;
    double2 m8[8], u8[8];
    for (int b = 0; b < nc; ++b) {
        const int64_t x = ax + (b & 1), y = ay + ((b >> 1) & 1), z = az + ((b >> 2) & 1);
        const bool in = x >= 0 && x < L.nx && y >= 0 && y < L.ny && z >= 0 && z < L.nz;
        const int64_t i = (z * L.ny + y) * L.nx + x;
        m8[b] = in ? mu[i] : make_double2(0.0, 0.0);
        u8[b] = in ? U[i] : make_double2(0.0, 0.0);
    }
    double acc = 0.0;
    for (int b = 0; b < nc; ++b)
        for (int g = 0; g < nc; ++g) {
            const double wgt = G.M[__popc(b ^ g)];
            acc += wgt * (m8[b].x * u8[g].x - m8[b].y * u8[g].y);   // Re(mu_b U_g)
        }
    gm[c] += G.w2 * acc;
}

// per node: gR[i] += omega Im(mu_i U_i)
__global__ void grad_nodes_kernel(int64_t N, double w, const double2 *__restrict__ mu,
                                  const double2 *__restrict__ U, double *__restrict__ gR)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const double2 a = mu[i], b = U[i];
    gR[i] += w * (a.x * b.y + a.y * b.x);
}

void launch_gradients(const Layout &L, const double M[4], double omega_phys, const double2 *mu,
                      const double2 *U, double *gm, double *gR, cudaStream_t s)
{
    GradCoef G;
    for (int k = 0; k < 4; ++k) G.M[k] = M[k];
    G.w2 = omega_phys * omega_phys;
    G.w = omega_phys;
    const int bs = 256;
    if (gm) {
        const int64_t ncell = (L.nx + 1) * (L.ny + 1) * ((L.d == 3) ? L.nz + 1 : 1);
        grad_cells_kernel<<<(unsigned)((ncell + bs - 1) / bs), bs, 0, s>>>(L, G, mu, U, gm);
        ++g_launches;
    }
    if (gR) {
        grad_nodes_kernel<<<(unsigned)((L.N + bs - 1) / bs), bs, 0, s>>>(L.N, omega_phys, mu, U, gR);
        ++g_launches;
    }
}

}  // namespace htd

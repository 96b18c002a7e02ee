// Resident-grid 2-D recurrence in FP64: the whole grid stays in shared memory,
// spread over the SMs, for all T n_P steps of a run, with one exchange of edge
// values for every two steps.
//
// One cooperative launch runs a whole preconditioner run (Def. of I_acd with
// Table 1's windowed forcing and read-out).  The grid is cut into ntx x nty
// tiles of W x H nodes, one CTA per tile and at most one CTA per SM.  A CTA
// keeps its tile's two states with a ring two nodes deep, the assembled stencil
// (the five planes of launch_assemble_H, scaled by -q: see step3d_asm_kernel),
// d and the forcing in shared memory.  Two steps make a block:
//  A  u_{j+1} on the tile and the first ring layer, from u_j with both layers
//     (the neighbours compute the same ring nodes with the same arithmetic);
//  B  u_{j+2} on the tile; nodes within two of its edge first, each published
//     as it is computed, then the inner ones; then the neighbours' values of
//     u_{j+2} fill both ring layers.
// What bounds it: on small tiles the exchange (store, L2, load across the
// chip: about a microsecond, which an exchange in every step paid twice as
// often), on large ones the FP64 pipe (two operations per clock and SM).  One
// node per thread keeps the dependent chain at 10 FP64 operations.  Measured on
// GB300: a 101^2 Table 1 application (120 steps) 159 us; with one exchange per
// step, node pairs and cell sums (33 operations per node) it took 429 us.
//
// An exchanged value travels as two 64-bit words, each one half of its bits and
// a 32-bit tag (index of the exchange + 1), read and written as one vector
// access whose words carry their own validity, so no fence orders data before a
// flag.  Before a CTA publishes exchange e + 2 it has read its neighbours' e + 1,
// which they published after reading its e: two buffers suffice.  They are
// zeroed before every run (tag 0 is never expected).  A wait that runs out sets
// the handle's error word, which every waiting CTA polls, so that all return.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "htd_internal.h"

namespace htd {

namespace {

constexpr int kMaxThreads = 512;
constexpr int kArrays = 10;          // U0, U1, five stencil planes, d, Re F, Im F

__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

struct Raw {
    unsigned long long lo, hi;
};

__device__ __forceinline__ void put(unsigned long long *p, double v, unsigned tag)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const unsigned long long t = (unsigned long long)tag << 32;
    asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"(t | (b & 0xffffffffull)),
                 "l"(t | (b >> 32))
                 : "memory");
}

__device__ __forceinline__ Raw get(const unsigned long long *p)
{
    Raw r;
    asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(r.lo), "=l"(r.hi) : "l"(p)
                 : "memory");
    return r;
}

__device__ __forceinline__ bool tagged(const Raw &r, unsigned want)
{
    return (unsigned)(r.lo >> 32) == want && (unsigned)(r.hi >> 32) == want;
}

__device__ __forceinline__ double value(const Raw &r)
{
    return __longlong_as_double((long long)((r.hi << 32) | (r.lo & 0xffffffffull)));
}

// Node (lx, ly) of the tile, -2 <= lx < w + 2, is element (ly + 2) SW + lx + 2 of
// every array; the task tables hold (ly + 2) << 16 | (lx + 2).  Exchange words
// of a tile and parity, 4 W + 4 H values: rows 0, 1 at [0, 2 W), rows h-1, h-2 at
// [2 W, 4 W), columns 0, 1 at [4 W, 4 W + 2 H), columns w-1, w-2 behind them.
__global__ void __launch_bounds__(kMaxThreads, 1)
res2d64_kernel(const double *__restrict__ coefP, const double *__restrict__ dco,
               const double *__restrict__ fre, const double *__restrict__ fim, Layout L, double c0,
               const double2 *__restrict__ ab, int nsteps, int jim, int jfin,
               const OutSlot *__restrict__ slot, unsigned long long *__restrict__ xbuf,
               int *__restrict__ err, int W, int H, Res2dProj<double> P)
{
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ int s_abort;
    const int tid = threadIdx.x, NT = blockDim.x;
    const int tx = blockIdx.x, ty = blockIdx.y;
    const int ntx = gridDim.x;
    const int x0 = tx * W, y0 = ty * H;
    const int nx = (int)L.nx, ny = (int)L.ny;
    const int w = min(W, nx - x0), h = min(H, ny - y0);
    const int SW = W + 4, NA = SW * (H + 4);
    double *U0 = reinterpret_cast<double *>(smraw), *U1 = U0 + NA, *CF = U1 + NA;
    double *D = CF + 5 * NA, *FR = D + NA, *FI = FR + NA;
    int *tA = reinterpret_cast<int *>(FI + NA), *tB = tA + (W + 2) * (H + 2);
    const int E2 = 2 * (4 * W + 4 * H);                // words per tile and parity

    if (tid == 0) s_abort = 0;
    for (int i = tid; i < NA; i += NT) {
        const int gy = y0 + i / SW - 2, gx = x0 + i % SW - 2;
        const bool in = gx >= 0 && gx < nx && gy >= 0 && gy < ny;
        const int64_t c = (int64_t)gy * nx + gx, g = (gy + 1) * L.pitch + L.xl + gx;
        U0[i] = 0.0;
        U1[i] = 0.0;
#pragma unroll
        for (int p = 0; p < 5; ++p) CF[p * NA + i] = in ? coefP[p * L.N + c] : 0.0;
        D[i] = in ? dco[g] : 0.0;
        FR[i] = in ? fre[g] : 0.0;
        FI[i] = in ? fim[g] : 0.0;
    }
    // tasks of step A: the tile and the ring layer around it, inside the domain
    const int ax0 = tx > 0 ? -1 : 0, ay0 = ty > 0 ? -1 : 0;
    const int aw = w - ax0 + (x0 + w < nx ? 1 : 0), ah = h - ay0 + (y0 + h < ny ? 1 : 0);
    const int nA = aw * ah;
    for (int t = tid; t < nA; t += NT)
        tA[t] = ((ay0 + t / aw + 2) << 16) | (ax0 + t % aw + 2);
    // tasks of step B: rows 0, 1, h-2, h-1, then columns 0, 1, w-2, w-1 of the
    // other rows, then the inner nodes
    const int br = min(h, 4), bc = min(w, 4), mh = h - br, iw = w - bc;
    const int nE = br * w + mh * bc, nB = w * h;
    for (int t = tid; t < nB; t += NT) {
        int lx, ly;
        if (t < br * w) {
            const int r = t / w;
            ly = r < 2 ? r : h - br + r;
            lx = t % w;
        } else if (t < nE) {
            const int q = t - br * w, cc = q % bc;
            ly = 2 + q / bc;
            lx = cc < 2 ? cc : w - bc + cc;
        } else {
            const int q = t - nE;
            ly = 2 + q / iw;
            lx = 2 + q % iw;
        }
        tB[t] = ((ly + 2) << 16) | (lx + 2);
    }
    // ring slot k: rows -2, -1, h, h+1 over w + 4 columns, then columns -2, -1, w,
    // w+1 of the tile's rows.  Returns the neighbour's word (or -1 outside the
    // domain, where the ring stays zero) and the place in a state array.
    const int nslot = 4 * (w + 4) + 4 * h;
    auto slot_of = [&](int k, int &dst) -> int {
        int rx, ry;
        if (k < 4 * (w + 4)) {
            const int r = k / (w + 4);
            ry = r < 2 ? r - 2 : h + r - 2;
            rx = k % (w + 4) - 2;
        } else {
            const int q = k - 4 * (w + 4), cc = q / h;
            ry = q % h;
            rx = cc < 2 ? cc - 2 : w + cc - 2;
        }
        dst = (ry + 2) * SW + rx + 2;
        if (x0 + rx < 0 || x0 + rx >= nx || y0 + ry < 0 || y0 + ry >= ny) return -1;
        const int dx = rx < 0 ? -1 : rx >= w ? 1 : 0, dy = ry < 0 ? -1 : ry >= h ? 1 : 0;
        int idx;
        if (dy != 0) {
            const int lx = dx < 0 ? W + rx : dx > 0 ? rx - w : rx;
            idx = dy < 0 ? 2 * W + (-1 - ry) * W + lx : (ry - h) * W + lx;
        } else {
            idx = dx < 0 ? 4 * W + 2 * H + (-1 - rx) * H + ry : 4 * W + (rx - w) * H + ry;
        }
        return ((ty + dy) * ntx + tx + dx) * 2 * E2 + 2 * idx;
    };
    int r_dst = 0;
    const int r_src = tid < nslot ? slot_of(tid, r_dst) : -1;

    // the value at p of exchange e into U0[dst], read again until its words carry
    // the tag (bounded by the handle's limit; with the stall test the first wait
    // of CTA (0, 0) expects a tag no word has)
    auto complete = [&](const unsigned long long *p, Raw v, int e, int dst) {
        unsigned want = (unsigned)(e + 1);
        if (e == 0 && tx == 0 && ty == 0 && *(volatile const int *)(err + 1) != 0)
            want = 0xffffffffu;
        if (!tagged(v, want)) {
            unsigned long long lim = *reinterpret_cast<volatile const unsigned long long *>(err + 2);
            if (lim == 0) lim = kDefaultWaitNs;
            const unsigned long long t0 = global_ns();
            for (int it = 1;; ++it) {
                v = get(p);
                if (tagged(v, want)) break;
                if ((it & 31) == 0 && *(volatile int *)err) {
                    s_abort = 1;
                    return;
                }
                if (global_ns() - t0 > lim) {
                    s_abort = 1;
                    atomicExch(err, 1);
                    return;
                }
            }
        }
        U0[dst] = value(v);
    };
    // new state at element o from cur, over nxt = the state before cur
    auto node = [&](const double *cur, double *nxt, int o, double a, double nb) -> double {
        const double *c = CF + o, *u = cur + o;
        const Asm9 k = {c[0],           c[4 * NA - SW - 1], c[3 * NA - SW], c[2 * NA - SW + 1],
                        c[NA - 1],      c[NA],              c[2 * NA],      c[3 * NA],
                        c[4 * NA]};
        const double un = asm2d_step(k, u[-SW - 1], u[-SW], u[-SW + 1], u[-1], u[0], u[1], u[SW - 1],
                                     u[SW], u[SW + 1], nxt[o], D[o], FR[o], FI[o], c0, a, nb);
        nxt[o] = un;
        return un;
    };
    // outputs of the new state of step j at tile node (lx, ly): snapshot, final
    // state, and in projection mode the compensated sums of the window's states
    // (as the separate accumulation kernel adds them)
    auto read_out = [&](int lx, int ly, double v, int j) {
        const int64_t c = (int64_t)(y0 + ly) * nx + x0 + lx;
        if (j + 1 == jim && slot->snap_part) slot->snap_part[2 * c] = v;
        if (j + 1 == jfin && slot->final_part) slot->final_part[2 * c] = v;
        if (j >= P.j_acc) {
            const int k = (j + 1) % P.nP;
            const double wc = P.w[2 * k], ws = P.w[2 * k + 1];
            double *s = P.acc + c;
            const double sr = s[0], si = s[P.N], cr = s[2 * P.N], ci = s[3 * P.N];
            const double yr = wc * v - cr, yi = ws * v - ci;
            const double tr = sr + yr, ti = si + yi;
            s[2 * P.N] = (tr - sr) - yr;
            s[3 * P.N] = (ti - si) - yi;
            s[0] = tr;
            s[P.N] = ti;
        }
    };

    __syncthreads();
    for (int j = 0; j < nsteps; j += 2) {
        // A
        const double2 abA = ab[j], abB = ab[j + 1];
        const bool outA = j + 1 == jim || j + 1 == jfin || j >= P.j_acc;
        for (int t = tid; t < nA; t += NT) {
            const int q = tA[t], ly = (q >> 16) - 2, lx = (q & 0xffff) - 2;
            const double un = node(U0, U1, (ly + 2) * SW + lx + 2, abA.x, -abA.y);
            if (outA && lx >= 0 && lx < w && ly >= 0 && ly < h) read_out(lx, ly, un, j);
        }
        __syncthreads();
        // B
        const int e = j >> 1;
        const unsigned tag = (unsigned)(e + 1);
        const bool more = j + 2 < nsteps;
        const bool outB = j + 2 == jim || j + 2 == jfin || j + 1 >= P.j_acc;
        unsigned long long *pub = xbuf + (size_t)((ty * ntx + tx) * 2 + (e & 1)) * E2;
        for (int t = tid; t < nB; t += NT) {
            const int q = tB[t], ly = (q >> 16) - 2, lx = (q & 0xffff) - 2;
            const double un = node(U1, U0, (ly + 2) * SW + lx + 2, abB.x, -abB.y);
            if (t < nE && more) {
                if (ly < 2) put(pub + 2 * (ly * W + lx), un, tag);
                if (h - 1 - ly < 2) put(pub + 2 * (2 * W + (h - 1 - ly) * W + lx), un, tag);
                if (lx < 2) put(pub + 2 * (4 * W + lx * H + ly), un, tag);
                if (w - 1 - lx < 2) put(pub + 2 * (4 * W + 2 * H + (w - 1 - lx) * H + ly), un, tag);
            }
            if (outB) read_out(lx, ly, un, j + 1);
        }
        if (more) {
            if (r_src >= 0) {
                const unsigned long long *p = xbuf + r_src + (e & 1) * E2;
                complete(p, get(p), e, r_dst);
            }
            for (int k = tid + NT; k < nslot; k += NT) {
                int dst = 0;
                const int src = slot_of(k, dst);
                if (src < 0) continue;
                const unsigned long long *p = xbuf + src + (e & 1) * E2;
                complete(p, get(p), e, dst);
            }
        }
        __syncthreads();
        if (s_abort) break;
    }
}

size_t res64_smem(long long W, long long H)
{
    return (size_t)(W + 4) * (H + 4) * kArrays * sizeof(double) +
           (size_t)((W + 2) * (H + 2) + W * H) * sizeof(int);
}

}  // namespace

bool res2d64_plan(const Layout &L, Res2dPlan *out)
{
    if (L.d != 2 || L.nx < 1 || L.ny < 1) return false;
    int dev = 0, nsm = 0, coop = 0, maxsm = 0;
    cudaFuncAttributes fa;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&maxsm, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) !=
            cudaSuccess ||
        cudaFuncGetAttributes(&fa, res2d64_kernel) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    // the limit is the kernel's, shared by every handle: raised to what the device
    // allows, not to this plan's size
    const int avail = maxsm - (int)fa.sharedSizeBytes;
    if (!coop || nsm < 1 || avail <= 0 ||
        cudaFuncSetAttribute(res2d64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, avail) !=
            cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    // the tiling with the least work per two steps in the largest tile (its nodes
    // plus the nodes with one ring layer, in warps) that fits one tile per SM.
    // A ring two deep may reach one tile only: inner tiles are at least 2 x 2.
    Res2dPlan best;
    long long best_cost = -1;
    for (int a = 1; a <= nsm && (a == 1 || 2 * (a - 1) < L.nx); ++a) {
        const long long W = std::max<long long>(2, (L.nx + a - 1) / a);
        const long long ntx = (L.nx + W - 1) / W;
        const long long tiles_y = nsm / ntx;
        if (tiles_y < 1) break;
        const long long H = std::max<long long>(2, (L.ny + tiles_y - 1) / tiles_y);
        const long long nty = (L.ny + H - 1) / H;
        if (H > 8192 || W > 8192 || res64_smem(W, H) > (size_t)avail) continue;
        const long long cost = ((W + 2) * (H + 2) + 31) / 32 + (W * H + 31) / 32;
        if (best_cost < 0 || cost < best_cost ||
            (cost == best_cost && W + H < (long long)best.W + best.H)) {
            best_cost = cost;
            best.W = (int)W;
            best.H = (int)H;
            best.ntx = (int)ntx;
            best.nty = (int)nty;
            best.smem = res64_smem(W, H);
        }
    }
    if (best_cost < 0) return false;
    // one node per thread up to 512 threads: fewer warps make a cheaper barrier
    const long long need = std::max<long long>((long long)(best.W + 2) * (best.H + 2),
                                               4LL * (best.W + 4) + 4LL * best.H);
    best.threads = (int)std::min<long long>(kMaxThreads, (need + 31) / 32 * 32);
    int occ = 0;
    const cudaError_t oe = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, res2d64_kernel,
                                                                         best.threads, best.smem);
    if (oe != cudaSuccess || occ < 1 || (long long)best.ntx * best.nty > (long long)occ * nsm) {
        (void)cudaGetLastError();
        return false;
    }
    best.xwords = (size_t)best.ntx * best.nty * 2 * 2 * (4 * (size_t)best.W + 4 * (size_t)best.H);
    *out = best;
    return true;
}

void launch_res2d64(const Res2dPlan &p, const double *coefP, const double *dco, const double *fre,
                    const double *fim, const Layout &L, double c0, const double *ab, int nsteps,
                    int jim, int jfin, const OutSlot *slot, unsigned long long *xbuf, int *err,
                    cudaStream_t s, const Res2dProj<double> &P)
{
    (void)cudaMemsetAsync(xbuf, 0, p.xwords * sizeof(unsigned long long), s);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)p.ntx, (unsigned)p.nty);
    cfg.blockDim = dim3((unsigned)p.threads);
    cfg.dynamicSmemBytes = p.smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    (void)cudaLaunchKernelEx(&cfg, res2d64_kernel, coefP, dco, fre, fim, L, c0,
                             reinterpret_cast<const double2 *>(ab), nsteps, jim, jfin, slot, xbuf,
                             err, p.W, p.H, P);
    ++g_launches;
}

}  // namespace htd

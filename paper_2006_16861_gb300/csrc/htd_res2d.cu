// Resident-grid 2-D recurrence in FP32: the whole grid stays on chip, spread
// over the SMs, for all T n_P steps of a run, with one exchange of edge values
// for every two steps.
//
// One cooperative launch runs a whole preconditioner run (Def. of I_acd with
// Table 1's windowed forcing and read-out).  The grid is cut into ntx x nty
// tiles of W x H nodes, one CTA per tile and at most one CTA per SM, every CTA
// resident at once.  Two steps make a block:
//  A  u_{j+1} on the tile and one ring layer around it, from u_j with a ring two
//     layers deep (the neighbours compute the same ring nodes with the same
//     arithmetic);
//  B  u_{j+2} on the tile; then the neighbours' values of u_{j+2} fill both ring
//     layers of that state.
// A thread owns 2 RPT rows of one column of the tile with its ring layer in every
// step, as the RPT pairs (row i, row i + RPT) in paired FP32 instructions: both
// states and d stay in registers for the whole run.  The state and cell arrays
// in shared memory, which serve the neighbouring threads, interleave the two
// rows of a pair, so that an operand of a pair is one 64-bit load into a register
// pair: 6 shared-memory accesses per pair and step (pairs of adjacent columns
// need register moves for every shifted operand, and scalar loads of the two
// rows still moves: 87 and 81 instructions per pair and step measured, against
// 66).
// Edge values (nodes within two of the tile's edge) are what the neighbours
// wait for: a pass before step B computes them one node per thread and publishes
// them at once, so that the exchange (about a microsecond) runs under the
// strips, which compute them again.  Publishing from the strips instead was
// slower at every size (257 x 193: 0.87 us per step against 0.75).
//
// What bounds it: on small grids the exchange (257 x 193: 0.45 us per step
// without its wait, 0.72 with it), on large ones shared memory (63 % of its
// wavefronts at 1001^2), FP32 (47 %) and issue (49 %) together.  Measured on
// GB300, us per step, against one exchange per step with every operand in
// shared memory: 0.72 / 1.6 at 257 x 193, 1.90 / 2.34 at 1001^2.  Holding the
// forcing and the cells in registers as well (256 threads) spilled from 8 rows up
// and gained at few sizes (640^2: 1.11 against 1.20); computing the edge pass as
// node pairs, and taking the halo pairs' own halves from registers, cost moves
// (1001^2: 2.12).
//
// A grid that does not fit the SMs (more than about 1.5 M nodes) runs window by
// window: strips along one axis, each loaded, run for B steps and stored, with B more
// nodes on its inner sides (res2d_win_plan).  Against the blocked kernel, which
// recomputes half of each tile's work in its rims and reloads everything every 4 or
// 8 steps, us per step: 1301 x 1501 4.9, 1501 x 2001 7.1 against 9.7, 1800^2 8.7;
// 2001^2 and 2501^2 stay with the blocked kernel (10.9, 19.1; windows 11.0, 19.2), whose
// tiles happen to fit them.  What bounds a pass is the resident steps (135 us for 64 at
// 1501 x 2001) and about 14 us of launch, loads and stores.
//
// An exchanged value is one 64-bit word, its bits beside a tag (index of the
// exchange + 1), so no fence orders data before a flag.  Before a CTA publishes
// exchange e + 2 it has read its neighbours' e + 1, which they published after
// reading its e: two buffers suffice.  They are zeroed before every run (tag 0 is
// never expected).  A wait that runs out sets the handle's error word, which
// every waiting CTA polls, so that all of them return.
//
// Per node the arithmetic is that of step2d_kernel and of the blocked kernels
// (stencil2d, the same expression in the same order): results bit-identical.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "htd_internal.h"

namespace htd {

namespace {

constexpr int kThreads = 512;        // at most; 128 registers each
constexpr int kMaxRows = 10;         // row pairs per thread, 1 .. kMaxRows
constexpr int kWinRows = 6;          // row pairs of a window's plan, kWinRows .. kMaxRows
constexpr int kPer = 2;              // edge nodes and ring slots per thread kept in registers

__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// one exchanged word: read and written whole, at GPU scope (not cached in L1)
__device__ __forceinline__ unsigned long long ld_word(const unsigned long long *p)
{
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_word(unsigned long long *p, float v, unsigned tag)
{
    const unsigned long long w = ((unsigned long long)tag << 32) | __float_as_uint(v);
    asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(w) : "memory");
}

__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }

// Geometry of a plan, shared by the kernel and the planner.  Threads cover the
// columns lx = -1 .. W in NB blocks of 2 rpt rows from ly = -1.  The state and cell
// arrays hold pairs: row ly = -1 + 2 rpt b + i (+ rpt for the second of the pair) at
// pair row b rpt + i + 1, column lx + 2; pair row 0 and the last one carry the
// outermost ring rows.
struct Res2dGeom {
    int NC, NB, S, rpt;
    size_t plane;                    // floats per array
    __host__ __device__ Res2dGeom(int W, int H, int r)
    {
        rpt = r;
        NC = W + 2;
        NB = (H + 2 + 2 * r - 1) / (2 * r);
        S = 2 * (W + 4);
        plane = (size_t)(NB * r + 2) * S;
    }
    // float of node (lx, ly), ly >= -2
    __host__ __device__ int at(int lx, int ly) const
    {
        const int t = ly + 1 + 2 * rpt, b = t / (2 * rpt), k = t - b * 2 * rpt;
        const int half = k >= rpt ? 1 : 0;
        return ((b - 1) * rpt + (k - half * rpt) + 1) * S + 2 * (lx + 2) + half;
    }
    // edge nodes of a full tile
    __host__ __device__ static int edges(int W, int H)
    {
        const int br = H < 4 ? H : 4, bc = W < 4 ? W : 4;
        return br * W + (H - br) * bc;
    }
};

// Exchange words of a tile and parity, one per edge node in this order: rows 0,
// 1, h-2, h-1, then columns 0, 1, w-2, w-1 of the other rows.
__device__ __forceinline__ int edge_rank(int lx, int ly, int w, int h)
{
    const int br = min(h, 4), bc = min(w, 4);
    if (ly < 2) return ly * w + lx;
    if (ly >= h - 2) return (br - h + ly) * w + lx;
    if (lx < 2) return br * w + (ly - 2) * bc + lx;
    if (lx >= w - 2) return br * w + (ly - 2) * bc + (bc - w + lx);
    return -1;
}

// One run of the instance I, as the CTA of its tile (tx, ty).  kGroup: for slot I.k of
// the handle's active list, else for its only rhs.  kWin: one pass over a window of a
// larger grid (see launch_res2d_win): states from and to memory, outputs of the owned
// nodes only.
template <int RPT, bool kGroup, bool kWin>
__device__ __forceinline__ void res2d_run(const Res2dInst &I, int tx, int ty, const Res2dProj<float> &P)
{
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ int s_abort;
    const Layout &L = I.L;
    const StepCoef<float> &C = I.C;
    const int W = I.W, H = I.H, ntx = I.ntx;
    const int nsteps = I.nsteps, jim = I.jim, jfin = I.jfin;
    int rhs = 0;
    if (kGroup && !rhs_of_slot(I.R, I.k, rhs)) return;   // an idle slot: all its tiles return
    const float *__restrict__ kap = I.kap, *__restrict__ dco = I.dco;
    const float *__restrict__ fre = I.fre + (kGroup ? rhs * I.R.stride : 0);
    const float *__restrict__ fim = I.fim + (kGroup ? rhs * I.R.stride : 0);
    const float2 *__restrict__ ab = reinterpret_cast<const float2 *>(I.ab);
    const OutSlot *__restrict__ slot = I.slot + (kGroup ? rhs : 0);
    unsigned long long *__restrict__ xbuf = I.xbuf;
    int *__restrict__ err = I.err;
    const Res2dGeom G(W, H, RPT);
    const int tid = threadIdx.x, NT = blockDim.x;
    const int x0 = tx * W, y0 = ty * H;
    const int nx = (int)L.nx, ny = (int)L.ny;
    const int w = min(W, nx - x0), h = min(H, ny - y0);
    const int NC = G.NC, S = G.S;
    float4 *F4 = reinterpret_cast<float4 *>(smraw);            // forcing of the pairs, thread rows
    float4 *EC = F4 + G.NB * RPT * NC;                         // (d, Re F, Im F) of the edge nodes
    int4 *EI = reinterpret_cast<int4 *>(EC + Res2dGeom::edges(W, H));   // and their elements
    float *U0 = reinterpret_cast<float *>(EI + Res2dGeom::edges(W, H));
    float *U1 = U0 + G.plane, *K = U1 + G.plane;
    const int E = Res2dGeom::edges(W, H);                      // words per tile and parity

    auto in_domain = [&](int lx, int ly) {
        return x0 + lx >= 0 && x0 + lx < nx && y0 + ly >= 0 && y0 + ly < ny;
    };
    auto gidx = [&](int lx, int ly) {
        return (int64_t)(y0 + ly + 1) * L.pitch + L.xl + x0 + lx;
    };
    if (tid == 0) s_abort = 0;
    for (int i = tid; i < (int)G.plane; i += NT) {
        U0[i] = 0.f;
        U1[i] = 0.f;
        K[i] = 0.f;
    }
    __syncthreads();
    // A window, which is loaded once per pass, loads its operands from a valid place
    // whether or not the node exists and drops what does not: loads behind a branch wait
    // for one another (a pass of 64 steps at 1501 x 2001: 168 us, 151 so).  A whole run's
    // loads do not show, and its kernels keep more registers without.
    const float *__restrict__ s0 = kWin ? I.s0 : nullptr, *__restrict__ s1 = kWin ? I.s1 : nullptr;
    const int64_t safe = gidx(0, 0);
    auto load = [&](const float *p, int64_t g, bool ok) {
        const float v = p[ok ? g : safe];
        return ok ? v : 0.f;
    };
    // cells (lower corner lx, ly), those of the domain's nodes; a window's u_j
    if constexpr (kWin) {
        int cx = tid % (W + 4), cy = tid / (W + 4);
        const int dx = NT % (W + 4), dy = NT / (W + 4);
#pragma unroll 8
        for (int i = tid; i < (W + 4) * (H + 4); i += NT) {
            const int lx = cx - 2, ly = cy - 2, o = G.at(lx, ly);
            const int64_t g = gidx(lx, ly);
            K[o] = load(kap, g, x0 + lx >= -1 && x0 + lx < nx && y0 + ly >= -1 && y0 + ly < ny);
            if (s0) U0[o] = load(s0, g, in_domain(lx, ly));
            cx += dx;
            cy += dy;
            if (cx >= W + 4) {
                cx -= W + 4;
                ++cy;
            }
        }
    } else {
        for (int i = tid; i < (W + 4) * (H + 4); i += NT) {
            const int lx = i % (W + 4) - 2, ly = i / (W + 4) - 2;
            if (x0 + lx >= -1 && x0 + lx < nx && y0 + ly >= -1 && y0 + ly < ny)
                K[G.at(lx, ly)] = kap[gidx(lx, ly)];
        }
    }
    // this thread's strip: column lx, rows ly0 + i and ly0 + RPT + i.  Nodes
    // outside the domain or beyond the ring layer have d = 0 and no forcing, so
    // they stay exactly zero.
    const bool has = tid < NC * G.NB;
    const int q = has ? tid % NC : 0, blk = has ? tid / NC : 0;
    const int lx = q - 1, ly0 = blk * 2 * RPT - 1;
    const bool sx = has && lx >= 0 && lx < w;      // a tile column
    float4 *fp = F4 + blk * RPT * NC + q;
    float2 za[RPT], zb[RPT], dd[RPT];
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
        za[i] = zb[i] = dd[i] = f2(0.f, 0.f);
        float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
        const int la = ly0 + i, lb = ly0 + RPT + i;
        if constexpr (kWin) {
            const bool oka = has && lx <= w && la <= h && in_domain(lx, la);
            const bool okb = has && lx <= w && lb <= h && in_domain(lx, lb);
            const int64_t ga = gidx(lx, la), gb = gidx(lx, lb);
            dd[i] = f2(load(dco, ga, oka), load(dco, gb, okb));
            if (s0) {
                za[i] = f2(load(s0, ga, oka), load(s0, gb, okb));
                zb[i] = f2(load(s1, ga, oka), load(s1, gb, okb));
            }
            if (has)
                fp[i * NC] = make_float4(load(fre, ga, oka), load(fre, gb, okb),
                                         load(fim, ga, oka), load(fim, gb, okb));
            continue;
        }
        if (has && lx <= w && la <= h && in_domain(lx, la)) {
            const int64_t g = gidx(lx, la);
            dd[i].x = dco[g];
            f.x = fre[g];
            f.z = fim[g];
        }
        if (has && lx <= w && lb <= h && in_domain(lx, lb)) {
            const int64_t g = gidx(lx, lb);
            dd[i].y = dco[g];
            f.y = fre[g];
            f.w = fim[g];
        }
        if (has) fp[i * NC] = f;
    }
    const int o0 = (blk * RPT + 1) * S + 2 * q;    // pair left of the strip's first pair
    // pairs whose two nodes, and whose one or the other node, are in the tile
    unsigned in2 = 0, in1a = 0, in1b = 0;
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
        const bool ra = sx && (unsigned)(ly0 + i) < (unsigned)h;
        const bool rb = sx && (unsigned)(ly0 + RPT + i) < (unsigned)h;
        if (ra && rb) in2 |= 1u << i;
        else if (ra) in1a |= 1u << i;
        else if (rb) in1b |= 1u << i;
    }

    // edge nodes: rank t on thread t
    const int br = min(h, 4), bc = min(w, 4);
    const int nE = br * w + (h - br) * bc;
    auto edge_node = [&](int t, int &lx, int &ly) {
        if (t < br * w) {
            const int r = t / w;
            ly = r < 2 ? r : h - br + r;
            lx = t % w;
        } else {
            const int s = t - br * w, cc = s % bc;
            ly = 2 + s / bc;
            lx = cc < 2 ? cc : w - bc + cc;
        }
    };
    float e_prev[kPer];
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        e_prev[k] = 0.f;
        const int t = tid + k * NT;
        if (t < nE) {
            int ex, ey;
            edge_node(t, ex, ey);
            EI[t] = make_int4(G.at(ex, ey), G.at(ex, ey - 1), G.at(ex, ey + 1), 0);
            const int64_t g = gidx(ex, ey);
            EC[t] = make_float4(dco[g], fre[g], fim[g], 0.f);
            if (kWin && s0) e_prev[k] = s0[g];
        }
    }
    // ring slot k: rows -2, -1, h, h+1 over w + 4 columns, then columns -2, -1, w,
    // w+1 of the tile's rows: the neighbour's word (-1 outside the domain, where
    // the ring stays zero) and the place in a state array
    const int nslot = 4 * (w + 4) + 4 * h;
    auto slot_of = [&](int k, int &dst) -> int {
        int rx, ry;
        if (k < 4 * (w + 4)) {
            const int r = k / (w + 4);
            ry = r < 2 ? r - 2 : h + r - 2;
            rx = k % (w + 4) - 2;
        } else {
            const int s = k - 4 * (w + 4), cc = s / h;
            ry = s % h;
            rx = cc < 2 ? cc - 2 : w + cc - 2;
        }
        dst = G.at(rx, ry);
        if (!in_domain(rx, ry)) return -1;
        const int dx = rx < 0 ? -1 : rx >= w ? 1 : 0, dy = ry < 0 ? -1 : ry >= h ? 1 : 0;
        const int wn = min(W, nx - (tx + dx) * W), hn = min(H, ny - (ty + dy) * H);
        const int lx = dx < 0 ? wn + rx : dx > 0 ? rx - w : rx;
        const int ly = dy < 0 ? hn + ry : dy > 0 ? ry - h : ry;
        return ((ty + dy) * ntx + tx + dx) * 2 * E + edge_rank(lx, ly, wn, hn);
    };
    int r_dst[kPer], r_src[kPer];
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        r_dst[k] = 0;
        r_src[k] = tid + k * NT < nslot ? slot_of(tid + k * NT, r_dst[k]) : -1;
    }

    // word v (read from p) of exchange e into U0[dst], read again until it carries
    // the tag (bounded by the handle's limit; with the stall test the first wait
    // of CTA (0, 0) expects a tag no word has)
    const unsigned tag0 = kWin ? I.tag0 : 0u;
    auto complete = [&](const unsigned long long *p, unsigned long long v, int e, int dst) {
        unsigned want = tag0 + (unsigned)(e + 1);
        if (e == 0 && tx == 0 && ty == 0 && *(volatile const int *)(err + 1) != 0)
            want = 0xffffffffu;
        if ((unsigned)(v >> 32) != want) {
            unsigned long long lim = *reinterpret_cast<volatile const unsigned long long *>(err + 2);
            if (lim == 0) lim = kDefaultWaitNs;
            const unsigned long long t0 = global_ns();
            for (int it = 1;; ++it) {
                v = ld_word(p);
                if ((unsigned)(v >> 32) == want) break;
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
        U0[dst] = __uint_as_float((unsigned)v);
    };

    const Stencil2dCoef<float2> SC = stencil2d_coef2(C);
    // The strip's new states over zo from zc (own nodes) and cur (the neighbours).
    // kB: step B stores tile nodes only, and issues the reads of this thread's
    // ring words half way down.
    unsigned long long rv[kPer];
    auto strip = [&](const float2 (&zc)[RPT], float2 (&zo)[RPT], const float *cur, float *nxt,
                     float2 abj, auto is_b, const unsigned long long *xr) {
        constexpr bool kB = decltype(is_b)::value;
        const float2 a2 = f2(abj.x, abj.x), nb2 = f2(-abj.y, -abj.y), n2 = f2(-2.f, -2.f);
        const float *u = cur + o0, *k = K + o0;
        // operand pair i, c columns right of lx - 1
        auto pair = [&](const float *b, int i, int c) {
            return *reinterpret_cast<const float2 *>(b + i * S + 2 * c);
        };
        // The pairs above the first one -- (row before the strip, row RPT - 1) -- and
        // below the last one -- (row RPT, row after the strip)
        auto above = [&](const float *b, int c) {
            return f2(b[-S + 2 * c + 1], b[(RPT - 1) * S + 2 * c]);
        };
        auto below = [&](const float *b, int c) {
            return f2(b[2 * c + 1], b[RPT * S + 2 * c]);
        };
        float2 umm = above(u, 0), um0 = above(u, 1), ump = above(u, 2);
        float2 u0m = pair(u, 0, 0), u0p = pair(u, 0, 2);
        float2 k00 = above(k, 0), k01 = above(k, 1);
        float2 pm = vadd(umm, ump), p0 = vadd(u0m, u0p), hk0 = vadd(k00, k01);
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
            if (kB && i == RPT / 2) {
#pragma unroll
                for (int s = 0; s < kPer; ++s)
                    if (xr && r_src[s] >= 0) rv[s] = ld_word(xr + r_src[s]);
            }
            float2 upm, up0, upp;
            if (i + 1 < RPT) {
                upm = pair(u, i + 1, 0);
                up0 = zc[i + 1 < RPT ? i + 1 : 0];
                upp = pair(u, i + 1, 2);
            } else {
                upm = below(u, 0);
                up0 = below(u, 1);
                upp = below(u, 2);
            }
            const float2 k10 = pair(k, i, 0), k11 = pair(k, i, 1);
            const float2 pp = vadd(upm, upp), hk1 = vadd(k10, k11);
            const float2 acc = stencil2d(SC, umm, um0, ump, u0m, zc[i], u0p, upm, up0, upp, k00,
                                         k01, k10, k11, pm, p0, pp, hk0, hk1);
            const float4 f = fp[i * NC];
            const float2 ag = vfma(a2, f2(f.x, f.y), vfma(nb2, f2(f.z, f.w), acc));
            const float2 un = vfma(dd[i], vfma(n2, zo[i], ag), zo[i]);
            zo[i] = un;
            float *o = nxt + o0 + i * S + 2;
            if (!kB || (in2 >> i & 1)) {
                *reinterpret_cast<float2 *>(o) = un;
            } else {
                if (in1a >> i & 1) o[0] = un.x;
                if (in1b >> i & 1) o[1] = un.y;
            }
            umm = u0m; um0 = zc[i]; ump = u0p; pm = p0;
            u0m = upm; u0p = upp; p0 = pp;
            k00 = k10; k01 = k11; hk0 = hk1;
        }
    };
    // the new value of an edge node in step B (o: its element, those above and below;
    // e: d, Re F, Im F)
    auto edge_value = [&](int4 o, float4 e, float prev, float2 abj) -> float {
        const Stencil2dCoef<float> c = stencil2d_coef(C);
        const float *u0 = U1 + o.x, *um = U1 + o.y, *up = U1 + o.z;
        const float *k0 = K + o.x, *km = K + o.y;
        const float umm = um[-2], um0 = um[0], ump = um[2];
        const float u0m = u0[-2], u00 = u0[0], u0p = u0[2];
        const float upm = up[-2], up0 = up[0], upp = up[2];
        const float k00 = km[-2], k01 = km[0], k10 = k0[-2], k11 = k0[0];
        const float acc = stencil2d(c, umm, um0, ump, u0m, u00, u0p, upm, up0, upp, k00, k01, k10,
                                    k11, vadd(umm, ump), vadd(u0m, u0p), vadd(upm, upp),
                                    vadd(k00, k01), vadd(k10, k11));
        const float ag = vfma(abj.x, e.y, vfma(-abj.y, e.z, acc));
        return vfma(e.x, vfma(-2.f, prev, ag), prev);
    };
    auto owned = [&](int lx, int ly) {
        return x0 + lx >= I.own[0] && x0 + lx < I.own[1] && y0 + ly >= I.own[2] && y0 + ly < I.own[3];
    };
    // outputs of the new state of step j (tile nodes of U): snapshot, final state,
    // and in projection mode the compensated sums of the window's states (as the
    // separate accumulation kernel adds them)
    auto read_out = [&](const float *U, int j) {
        const bool acc = j >= P.j_acc;
        const int ph = acc ? ((kWin ? I.jbase : 0) + j + 1) % P.nP : 0;
        const float wc = acc ? P.w[2 * ph] : 0.f, ws = acc ? P.w[2 * ph + 1] : 0.f;
        for (int i = tid; i < w * h; i += NT) {
            const int ly = i / w, lx = i - ly * w;
            if (kWin && !owned(lx, ly)) continue;
            const int64_t c = kWin ? (int64_t)(I.gy + y0 + ly) * I.gnx + I.gx + x0 + lx
                                   : (int64_t)(y0 + ly) * nx + x0 + lx;
            const float v = U[G.at(lx, ly)];
            if (j + 1 == jim && slot->snap_part) slot->snap_part[2 * c] = (double)v;
            if (j + 1 == jfin && slot->final_part) slot->final_part[2 * c] = (double)v;
            if (acc) {
                float *s = P.acc + c;
                const float sr = s[0], si = s[P.N], cr = s[2 * P.N], ci = s[3 * P.N];
                const float yr = wc * v - cr, yi = ws * v - ci;
                const float tr = sr + yr, ti = si + yi;
                s[2 * P.N] = (tr - sr) - yr;
                s[3 * P.N] = (ti - si) - yi;
                s[0] = tr;
                s[P.N] = ti;
            }
        }
    };
    auto reads = [&](int j) { return j + 1 == jim || j + 1 == jfin || j >= P.j_acc; };

    __syncthreads();
    for (int j = 0; j < nsteps; j += 2) {
        const float2 abA = ab[j], abB = ab[j + 1];
        // A: the ring nodes a thread owns come from the exchange
        if (has) {
#pragma unroll
            for (int i = 0; i < RPT; ++i)
                if (!(in2 >> i & 1)) za[i] = *reinterpret_cast<const float2 *>(U0 + o0 + i * S + 2);
            strip(za, zb, U0, U1, abA, std::false_type{}, nullptr);
        }
        __syncthreads();
        if (reads(j)) read_out(U1, j);
        // B
        const int e = j >> 1;
        const bool more = j + 2 < nsteps;
        const unsigned long long *xr = more ? xbuf + (size_t)(e & 1) * E : nullptr;
        if (more) {
            unsigned long long *pub = xbuf + (size_t)((ty * ntx + tx) * 2 + (e & 1)) * E;
#pragma unroll
            for (int k = 0; k < kPer; ++k) {
                const int t = tid + k * NT;
                if (t < nE) {
                    e_prev[k] = edge_value(EI[t], EC[t], e_prev[k], abB);
                    st_word(pub + t, e_prev[k], tag0 + (unsigned)(e + 1));
                }
            }
        }
#pragma unroll
        for (int k = 0; k < kPer; ++k) rv[k] = 0;
        if (has) strip(zb, za, U1, U0, abB, std::true_type{}, xr);
        if (more) {
#pragma unroll
            for (int k = 0; k < kPer; ++k)
                if (r_src[k] >= 0) complete(xr + r_src[k], rv[k], e, r_dst[k]);
        }
        __syncthreads();
        if (s_abort) break;
        if (reads(j + 1)) read_out(U0, j + 1);
    }
    if (kWin && I.o0) {
        for (int i = tid; i < w * h; i += NT) {
            const int ly = i / w, lx = i - ly * w;
            if (!owned(lx, ly)) continue;
            I.o0[gidx(lx, ly)] = U0[G.at(lx, ly)];
            I.o1[gidx(lx, ly)] = U1[G.at(lx, ly)];
        }
    }
}

template <int RPT>
__global__ void __launch_bounds__(kThreads, 1)
res2d_kernel(const __grid_constant__ Res2dInst I, const __grid_constant__ Res2dProj<float> P)
{
    res2d_run<RPT, false, false>(I, blockIdx.x, blockIdx.y, P);
}

template <int RPT>
__global__ void __launch_bounds__(kThreads, 1)
res2d_win_kernel(const __grid_constant__ Res2dInst I, const __grid_constant__ Res2dProj<float> P)
{
    res2d_run<RPT, false, true>(I, blockIdx.x, blockIdx.y, P);
}

// Several instances in one launch, instance i on the CTAs from inst[i].cta0 up to
// the next one's: every instance's tiles resident at once, each with the plan made
// for its share of the SMs.
__global__ void __launch_bounds__(kThreads, 1)
res2d_group_kernel(const Res2dInst *__restrict__ inst, int n)
{
    __shared__ __align__(16) unsigned char raw[sizeof(Res2dInst)];
    int i = 0;
    while (i + 1 < n && inst[i + 1].cta0 <= (int)blockIdx.x) ++i;
    static_assert(sizeof(Res2dInst) % 4 == 0, "copied by words");
    for (int k = threadIdx.x; k < (int)sizeof(Res2dInst) / 4; k += blockDim.x)
        reinterpret_cast<int *>(raw)[k] = reinterpret_cast<const int *>(inst + i)[k];
    __syncthreads();
    const Res2dInst &I = *reinterpret_cast<const Res2dInst *>(raw);
    const int t = (int)blockIdx.x - I.cta0;
    const int tx = t % I.ntx, ty = t / I.ntx;
    const Res2dProj<float> P;
    switch (I.rpt) {
    case 1: res2d_run<1, true, false>(I, tx, ty, P); break;
    case 2: res2d_run<2, true, false>(I, tx, ty, P); break;
    case 3: res2d_run<3, true, false>(I, tx, ty, P); break;
    case 4: res2d_run<4, true, false>(I, tx, ty, P); break;
    case 5: res2d_run<5, true, false>(I, tx, ty, P); break;
    case 6: res2d_run<6, true, false>(I, tx, ty, P); break;
    case 7: res2d_run<7, true, false>(I, tx, ty, P); break;
    case 8: res2d_run<8, true, false>(I, tx, ty, P); break;
    case 9: res2d_run<9, true, false>(I, tx, ty, P); break;
    default: res2d_run<10, true, false>(I, tx, ty, P); break;
    }
}

template <typename Fn>
void with_kernel(int rpt, Fn &&fn)
{
    switch (rpt) {
    case 1: fn(res2d_kernel<1>); break;
    case 2: fn(res2d_kernel<2>); break;
    case 3: fn(res2d_kernel<3>); break;
    case 4: fn(res2d_kernel<4>); break;
    case 5: fn(res2d_kernel<5>); break;
    case 6: fn(res2d_kernel<6>); break;
    case 7: fn(res2d_kernel<7>); break;
    case 8: fn(res2d_kernel<8>); break;
    case 9: fn(res2d_kernel<9>); break;
    default: fn(res2d_kernel<10>); break;
    }
}

template <typename Fn>
void with_win_kernel(int rpt, Fn &&fn)
{
    switch (rpt) {
    case 6: fn(res2d_win_kernel<6>); break;
    case 7: fn(res2d_win_kernel<7>); break;
    case 8: fn(res2d_win_kernel<8>); break;
    case 9: fn(res2d_win_kernel<9>); break;
    default: fn(res2d_win_kernel<10>); break;
    }
}

size_t res2d_smem(int W, int H, int rpt)
{
    const Res2dGeom G(W, H, rpt);
    return 3 * G.plane * sizeof(float) +
           ((size_t)G.NB * rpt * G.NC + 2 * (size_t)Res2dGeom::edges(W, H)) * sizeof(float4);
}

// Device limits for the kernels: SMs, and the dynamic shared memory every one of
// them may use.  The limit is a property of a kernel, shared by every handle: it is
// raised to what the device allows beside the kernel's static shared memory.
bool res2d_device(int *nsm, int *avail)
{
    int dev = 0, coop = 0, maxsm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&maxsm, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    if (!coop || *nsm < 1) return false;
    *avail = maxsm;
    bool ok = true;
    auto limit = [&](auto kern) {
        cudaFuncAttributes fa;
        if (cudaFuncGetAttributes(&fa, kern) != cudaSuccess) {
            ok = false;
            return;
        }
        const int dyn = maxsm - (int)fa.sharedSizeBytes;
        *avail = std::min(*avail, dyn);
        ok = ok && dyn > 0 &&
             cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn) ==
                 cudaSuccess;
    };
    for (int r = 1; r <= kMaxRows; ++r) with_kernel(r, limit);
    for (int r = kWinRows; r <= kMaxRows; ++r) with_win_kernel(r, limit);
    limit(res2d_group_kernel);
    if (!ok) (void)cudaGetLastError();
    return ok;
}

// The best plan of a grid on `ctas` CTAs and its cost, -1 if it does not fit.
// Tiles of W x H nodes (inner tiles at least 2 x 2: the ring reaches one tile
// only) with RPT row pairs per thread.  Cost of two steps in cycles of an SM's
// quarter: a row pair takes about 60 issue cycles per warp, 120 when no other warp
// fills its latency; the edge pass about 60 per warp and pass.  Against the
// measured times of the 14 cheapest plans at nine sizes from 101^2 to 1101^2 the
// chosen one was within 5 % of the best.
long long res2d_best(const Layout &L, int ctas, int avail, Res2dPlan *out, int min_rows = 1)
{
    Res2dPlan best;
    long long best_cost = -1;
    for (int a = 1; a <= ctas && (a == 1 || 2 * (a - 1) < L.nx); ++a) {
        const long long W = std::max<long long>(2, (L.nx + a - 1) / a);
        const long long ntx = (L.nx + W - 1) / W;
        const long long tiles_y = ctas / ntx;
        if (tiles_y < 1) break;
        const long long H = std::max<long long>(2, (L.ny + tiles_y - 1) / tiles_y);
        const long long nty = (L.ny + H - 1) / H;
        if (H > 8192 || W > kThreads) continue;
        for (int rpt = min_rows; rpt <= kMaxRows; ++rpt) {
            const Res2dGeom G((int)W, (int)H, rpt);
            const long long strips = (long long)G.NC * G.NB;
            const long long nedge = Res2dGeom::edges((int)W, (int)H);
            const long long slots = 4 * (W + 4) + 4 * H;
            // the edge pass and the ring keep kPer entries per thread
            long long threads = std::max(strips, (std::max(slots, nedge) + kPer - 1) / kPer);
            threads = (threads + 31) / 32 * 32;
            const size_t smem = res2d_smem((int)W, (int)H, rpt);
            if (threads > kThreads || smem > (size_t)avail) continue;
            const long long row = std::max<long long>(120, 60 * ((strips + 127) / 128));
            const long long cost = 2 * rpt * row + 60 * ((nedge + 127) / 128) +
                                   120 * ((nedge + threads - 1) / threads);
            if (best_cost < 0 || cost < best_cost ||
                (cost == best_cost && W + H < (long long)best.W + best.H)) {
                best_cost = cost;
                best.W = (int)W;
                best.H = (int)H;
                best.rpt = rpt;
                best.ntx = (int)ntx;
                best.nty = (int)nty;
                best.smem = smem;
                best.threads = (int)threads;
            }
        }
    }
    if (best_cost >= 0) {
        best.xwords = (size_t)best.ntx * best.nty * 2 * Res2dGeom::edges(best.W, best.H);
        *out = best;
    }
    return best_cost;
}

// cost of the exchange that no work hides, per two steps (about 0.7 us)
constexpr long long kExchangeCost = 1400;
// cost of a window's launch, loads and stores (about 14 us; the model's cycles come
// out some 1.35 times as long)
constexpr long long kPassCost = 20000;

}  // namespace

bool res2d_plan(const Layout &L, Res2dPlan *out)
{
    if (L.d != 2 || L.nx < 1 || L.ny < 1) return false;
    int nsm = 0, avail = 0;
    Res2dPlan best;
    if (!res2d_device(&nsm, &avail) || res2d_best(L, nsm, avail, &best) < 0) return false;
    int occ = 0;
    cudaError_t oe = cudaSuccess;
    with_kernel(best.rpt, [&](auto kern) {
        oe = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, best.threads, best.smem);
    });
    if (oe != cudaSuccess || occ < 1 || (long long)best.ntx * best.nty > (long long)occ * nsm) {
        (void)cudaGetLastError();
        return false;
    }
    *out = best;
    return true;
}

// Windows for a grid that does not fit the SMs: strips along one axis, each run for B
// steps with B more nodes on its inner sides, so that what the missing neighbours
// spoil (one node per step from the rim) never reaches the nodes it owns.  All windows
// are equally long.  Cost per step of the whole grid: the windows' two-step costs and
// the fixed cost of their passes.  More windows mean more rim, deeper passes wider rims
// but fewer of them; the handle times the choice against the blocked kernel.
bool res2d_win_plan(const Layout &L, long long nsteps, Res2dWin *win)
{
    int nsm = 0, avail = 0;
    Res2dWin w;
    if (L.d != 2 || !res2d_device(&nsm, &avail)) return false;
    double best = INFINITY;
    for (int axis = 0; axis < 2; ++axis) {
        const long long n = axis ? L.ny : L.nx, other = axis ? L.nx : L.ny;
        for (int B = 16; B <= 96 && B <= nsteps; B += 8) {
            for (int k = 2, fits = 0; k <= 32 && fits < 3; ++k) {
                const long long len = (n + 2LL * B * (k - 1) + k - 1) / k;
                if (len - 2LL * B < 32) break;         // (every window owns nodes)
                if (len * other > 2LL * kMaxRows * kThreads * nsm) continue;
                Layout S = L;
                (axis ? S.ny : S.nx) = len;
                Res2dPlan p;
                const long long cost = res2d_best(S, nsm, avail, &p, kWinRows);
                if (cost < 0) continue;
                ++fits;
                const double t = k * (0.5 * (double)(cost + kExchangeCost) + (double)kPassCost / B);
                if (t < best) {
                    best = t;
                    w.n = k;
                    w.B = B;
                    w.axis = axis;
                    w.len = (int)len;
                    w.plan = p;
                }
            }
        }
    }
    if (best == INFINITY) return false;
    int occ = 0;
    cudaError_t oe = cudaSuccess;
    with_win_kernel(w.plan.rpt, [&](auto kern) {
        oe = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, w.plan.threads,
                                                           w.plan.smem);
    });
    if (oe != cudaSuccess || occ < 1 ||
        (long long)w.plan.ntx * w.plan.nty > (long long)occ * nsm) {
        (void)cudaGetLastError();
        return false;
    }
    *win = w;
    return true;
}

// Shares of the SMs for several instances (layout, steps per run) in one launch, so
// that the slowest one ends as early as possible: in proportion to their work
// first, then SM by SM from the fastest instance to the slowest.
bool res2d_group_plan(const std::vector<Layout> &L, const std::vector<long long> &nsteps,
                      std::vector<Res2dPlan> *plans)
{
    const int n = (int)L.size();
    int nsm = 0, avail = 0;
    if (n < 1 || !res2d_device(&nsm, &avail) || n > nsm) return false;
    std::vector<Res2dPlan> p(n), q(1);
    std::vector<int> c(n), least(n);
    std::vector<double> t(n);
    double work = 0.0;
    int sum = 0;
    auto time = [&](int i, int ctas, Res2dPlan *out) -> double {
        const long long cost = res2d_best(L[i], ctas, avail, out);
        return cost < 0 ? -1.0 : (double)nsteps[i] * (double)(cost + kExchangeCost);
    };
    for (int i = 0; i < n; ++i) {
        if (L[i].d != 2 || nsteps[i] >= (1LL << 30)) return false;
        work += (double)L[i].N * (double)nsteps[i];
        // 10 row pairs of 512 threads hold 10240 nodes with the ring
        least[i] = (int)std::max<int64_t>(1, L[i].N / 10000);
        while (least[i] <= nsm && time(i, least[i], &p[i]) < 0.0) ++least[i];
        if ((sum += least[i]) > nsm) return false;
    }
    sum = 0;
    for (int i = 0; i < n; ++i) {
        c[i] = std::max(least[i], (int)(nsm * ((double)L[i].N * (double)nsteps[i] / work)));
        sum += c[i];
    }
    for (int i = 0; i < n; ++i) t[i] = time(i, c[i], &p[i]);
    auto pick = [&](bool slowest, bool spare) {
        int b = -1;
        for (int i = 0; i < n; ++i)
            if ((!spare || c[i] > least[i]) && (b < 0 || (slowest ? t[i] > t[b] : t[i] < t[b])))
                b = i;
        return b;
    };
    while (sum > nsm) {
        const int f = pick(false, true);
        if (f < 0) return false;
        t[f] = time(f, --c[f], &p[f]);
        --sum;
    }
    for (int it = 0; it < 64; ++it) {
        const int b = pick(true, false);
        if (sum == nsm) {
            const int f = pick(false, true);
            if (f < 0 || f == b) break;
            const double tf = time(f, c[f] - 1, &q[0]);
            if (tf < 0.0 || tf >= t[b]) break;
            --c[f];
            t[f] = tf;
            p[f] = q[0];
            --sum;
        }
        t[b] = time(b, ++c[b], &p[b]);
        ++sum;
    }
    size_t smem = 0;
    int used = 0, occ = 0;
    for (int i = 0; i < n; ++i) {
        smem = std::max(smem, p[i].smem);
        used += p[i].ntx * p[i].nty;
    }
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, res2d_group_kernel, kThreads, smem) !=
            cudaSuccess ||
        occ < 1 || used > occ * nsm) {
        (void)cudaGetLastError();
        return false;
    }
    *plans = p;
    return true;
}

namespace {

template <typename Kern, typename... Args>
void launch_cooperative(Kern kern, dim3 grid, unsigned threads, size_t smem, cudaStream_t s,
                        Args &&...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    (void)cudaLaunchKernelEx(&cfg, kern, static_cast<Args &&>(args)...);
    ++g_launches;
}

}  // namespace

void launch_res2d(const Res2dPlan &p, const float *kap, const float *dco, const float *fre,
                  const float *fim, const Layout &L, const StepCoef<float> &C, const float *ab,
                  int nsteps, int jim, int jfin, const OutSlot *slot, unsigned long long *xbuf,
                  int *err, cudaStream_t s, const Res2dProj<float> &P)
{
    (void)cudaMemsetAsync(xbuf, 0, p.xwords * sizeof(unsigned long long), s);
    Res2dInst I;
    I.kap = kap;
    I.dco = dco;
    I.fre = fre;
    I.fim = fim;
    I.L = L;
    I.C = C;
    I.ab = ab;
    I.nsteps = nsteps;
    I.jim = jim;
    I.jfin = jfin;
    I.slot = slot;
    I.xbuf = xbuf;
    I.err = err;
    I.W = p.W;
    I.H = p.H;
    I.ntx = p.ntx;
    I.rpt = p.rpt;
    with_kernel(p.rpt, [&](auto kern) {
        launch_cooperative(kern, dim3((unsigned)p.ntx, (unsigned)p.nty), (unsigned)p.threads,
                           p.smem, s, I, P);
    });
}

void launch_res2d_win(const Res2dWin &w, const float *kap, const float *dco, const float *fre,
                      const float *fim, const Layout &L, const StepCoef<float> &C, const float *ab,
                      int nsteps, int jim, int jfin, const OutSlot *slot, unsigned long long *xbuf,
                      int *err, float *const planes[4], cudaStream_t s, const Res2dProj<float> &P)
{
    (void)cudaMemsetAsync(xbuf, 0, w.plan.xwords * sizeof(unsigned long long), s);
    const int n = (int)(w.axis ? L.ny : L.nx);
    unsigned tag = 0;
    for (int j = 0, pass = 0; j < nsteps; j += w.B, ++pass) {
        const int steps = std::min(w.B, nsteps - j);
        const int in = 2 * (pass & 1), to = 2 - in;
        int own = 0;                            // first owned node of the window
        for (int k = 0; k < w.n; ++k) {
            const int from = std::max(0, own - w.B), end = std::min(n, from + w.len);
            const int next = k + 1 == w.n ? n : end - w.B;
            Res2dInst I;
            I.L = L;
            (w.axis ? I.L.ny : I.L.nx) = end - from;
            const int64_t off = w.axis ? (int64_t)from * L.pitch : from;
            I.gx = w.axis ? 0 : from;
            I.gy = w.axis ? from : 0;
            I.gnx = (int)L.nx;
            I.own[0] = w.axis ? 0 : own - from;
            I.own[1] = w.axis ? (int)L.nx : next - from;
            I.own[2] = w.axis ? own - from : 0;
            I.own[3] = w.axis ? next - from : (int)L.ny;
            I.kap = kap + off;
            I.dco = dco + off;
            I.fre = fre + off;
            I.fim = fim + off;
            if (j > 0) {                        // (a run starts from rest)
                I.s0 = planes[in] + off;
                I.s1 = planes[in + 1] + off;
            }
            if (j + steps < nsteps) {
                I.o0 = planes[to] + off;
                I.o1 = planes[to + 1] + off;
            }
            I.C = C;
            I.ab = ab + 2 * j;
            I.nsteps = steps;
            I.jim = jim - j;
            I.jfin = jfin - j;
            I.jbase = j;
            I.slot = slot;
            I.xbuf = xbuf;
            I.err = err;
            I.W = w.plan.W;
            I.H = w.plan.H;
            I.rpt = w.plan.rpt;
            I.ntx = (int)((I.L.nx + I.W - 1) / I.W);
            const int nty = (int)((I.L.ny + I.H - 1) / I.H);
            I.tag0 = tag;
            tag += (unsigned)(steps / 2);
            Res2dProj<float> Q = P;
            if (Q.acc) Q.j_acc -= j;
            with_win_kernel(I.rpt, [&](auto kern) {
                launch_cooperative(kern, dim3((unsigned)I.ntx, (unsigned)nty),
                                   (unsigned)w.plan.threads, w.plan.smem, s, I, Q);
            });
            own = next;
        }
    }
}

void launch_res2d_group(const Res2dInst *inst, int n, int ctas, size_t smem,
                        unsigned long long *xbuf, size_t xwords, cudaStream_t s)
{
    (void)cudaMemsetAsync(xbuf, 0, xwords * sizeof(unsigned long long), s);
    launch_cooperative(res2d_group_kernel, dim3((unsigned)ctas), kThreads, smem, s, inst, n);
}

}  // namespace htd

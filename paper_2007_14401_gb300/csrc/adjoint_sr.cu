// adjoint_sr.cu -- reverse-mode adjoint of the flat-space coupled push
// (2D, gradient-grid records), for gradients of trajectory observables with
// respect to the initial state and the field records.
//
// One particle-step maps s = (x, u, dxp) and the fields interpolated at the
// step's gather points F_g (12 components each) to s'.  Given the adjoint
// lambda' = dL/ds', the kernel forms
//     dL/ds   = (ds'/ds)^T lambda'                     (kept per particle)
//     dL/dF_g = (ds'/dF_g)^T lambda'                   (scattered to nodes)
// and a node record value f_N receives W_g(N) dL/dF_g, the linear shape
// function being the only way it enters the step.  The columns of the step's
// Jacobian come from replaying the step on dual numbers (value + N tangents)
// in registers, N directions per pass; the branch taken and the fixed-point
// iteration count are those of the plain replay (held fixed, not
// differentiated).  The sweep over steps runs backwards from checkpoints
// stored every `ckpt_every` steps, recomputing each segment forward.
#include <cuda_runtime.h>
#include <string.h>

#include "dual.cuh"
#include "gcb_internal.h"
#include "adjoint_rev.cuh"
#include "gca_lean.cuh"
#include "push_sr.cuh"

// GCB_ADJ_FCACHE: gather points (x^n first, then the step's gathers in order)
// whose interpolated field the replay keeps in shared memory for the reverse
// loop, which otherwise gathers again; points past it are re-gathered.
#ifndef GCB_ADJ_FCACHE
#define GCB_ADJ_FCACHE 6
#endif
namespace gcb {
namespace adj {

constexpr int TPB = 128;
constexpr int NDIR = 4;          // tangent directions per pass
constexpr int MAXG = GCB_ADJOINT_MAX_ITER + 2;   // gathers per step: x^n, R^{n-1/2},
                                                // iterates 1..iters-1, R^{n+1/2}
constexpr int NF = 12;           // interpolated components per gather (2D, gradient grids)
constexpr int NS = 7;            // state directions: x(2), u(3), dxp(2)

// Gather on dual positions from plain records: the weights carry the
// position tangents; this pass's field directions are seeded on the result;
// nodes and weights of every gather are recorded for the scatter.
template <typename T, int N>
struct DualGather {
    DevGrid<T> g;
    int *count;
    int base;
    int *nodes;
    T *wts;
    __device__ __forceinline__ void operator()(const int ib[2], const Dual<T, N> l[2],
                                               FieldPt<Dual<T, N>, 2> &F) const
    {
        using D = Dual<T, N>;
        const int k = (*count)++;
        int i0[2], i1[2];
        D t[2];
#pragma unroll
        for (int d = 0; d < 2; ++d) {
            // cell and fraction from one rounding (cell_of's), with the
            // position's tangent
            T tv;
            cell_of(g, d, ib[d], l[d].v, tv, i0[d], i1[d]);
            t[d] = l[d] * g.inv_dx[d];
            t[d].v = tv;
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) { F.E[c] = D(T(0)); F.B[c] = D(T(0)); }
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 3; ++j) F.dB[i][j] = D(T(0));
#pragma unroll
        for (int o = 0; o < 4; ++o) {
            const int ix = (o & 1) ? i1[0] : i0[0];
            const int iy = (o & 2) ? i1[1] : i0[1];
            const int node = iy * g.n[0] + ix;
            const D wx = (o & 1) ? t[0] : T(1) - t[0];
            const D wy = (o & 2) ? t[1] : T(1) - t[1];
            const D W = wx * wy;
            if (k < MAXG) {
                nodes[k * 4 + o] = node;
                wts[k * 4 + o] = W.v;
            }
            const T *rp = g.rec + (size_t)node * g.stride;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                F.E[c] = fma(W, D(__ldg(rp + c)), F.E[c]);
                F.B[c] = fma(W, D(__ldg(rp + 3 + c)), F.B[c]);
            }
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 3; ++j) F.dB[i][j] = fma(W, D(__ldg(rp + 6 + 3 * i + j)), F.dB[i][j]);
        }
        // seed d(output)/d(F_k,c) for the directions of this pass
        const int d0 = NS + NF * k - base;
#pragma unroll
        for (int c = 0; c < NF; ++c) {
            const int j = d0 + c;
            if (j >= 0 && j < N) {
                D &f = c < 3 ? F.E[c] : (c < 6 ? F.B[c - 3] : F.dB[(c - 6) / 3][(c - 6) % 3]);
                f.d[j] += T(1);
            }
        }
    }
};

template <typename T>
struct AdjArgs {
    DevGrid<T> g;
    int64_t np;
    int pair;                    // positions as FP32 pairs
    const void *x[2];
    const float *xlo[2];
    const T *u[3];
    const T *dxp[2];
    const uint8_t *flags;
    T *lam[NS];                  // in: dL/d(state after the step); out: before it
    double *grad;                // node records' adjoint, stride 12 per node
    StepPar<T> sp;
    T qm[4];
    Switch<T> sw;
};

template <typename T>
__device__ __forceinline__ void load_pos(const AdjArgs<T> &a, int64_t i, int d, int &ib, T &l,
                                         bool &fin)
{
    if (a.pair) {
        const float h = ((const float *)a.x[d])[i], lo = a.xlo[d][i];
        fin = fin && isfinite(h) && isfinite(lo);
        float lf;
        split_pos_pair(h, lo, (float)a.g.dx[d], (float)a.g.inv_dx[d], (float)(a.g.n[d] - 1), ib, lf);
        l = (T)lf;
    } else {
        const double x = ((const double *)a.x[d])[i];
        fin = fin && isfinite(x);
        split_pos_f64<T>(x, (double)a.g.dx[d], 1.0 / (double)a.g.dx[d], a.g.n[d] - 1, ib, l);
    }
}

// The forward step as the forward run takes it (push_step_f64,
// push_step_adj_f32).
template <typename T, typename Gth>
__device__ __forceinline__ bool replay_step(const Gth &gth, const StepPar<T> &s, const int ib[2],
                                            const T l[2], const T dxp[2], const FieldPt<T, 2> &F0,
                                            T u[3], T disp[2], int &iters, bool &nonconv)
{
    if constexpr (sizeof(T) == 8)
        return gca_step_lean<T, 2, 2>(gth, s, ib, l, dxp, F0, u, disp, iters, nonconv);
    else
        return gca_step<T, 2, 2>(gth, s, ib, l, dxp, F0, u, disp, iters, nonconv);
}

template <typename T, int N>
__global__ void __launch_bounds__(TPB) k_adjoint_sr(const AdjArgs<T> a)
{
    using D = Dual<T, N>;
    int nodes[MAXG * 4];
    T wts[MAXG * 4];
    for (int64_t i = blockIdx.x * (int64_t)TPB + threadIdx.x; i < a.np;
         i += (int64_t)gridDim.x * TPB) {
        const uint8_t fl = a.flags[i];
        bool fin = true;
        int ib[2];
        T l[2], u[3], dxp[2], lo[NS];
#pragma unroll
        for (int d = 0; d < 2; ++d) {
            load_pos(a, i, d, ib[d], l[d], fin);
            dxp[d] = a.dxp[d][i];
            fin = fin && isfinite(dxp[d]);
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) { u[k] = a.u[k][i]; fin = fin && isfinite(u[k]); }
#pragma unroll
        for (int k = 0; k < NS; ++k) lo[k] = a.lam[k][i];
        if (!fin) continue;          // a frozen particle's step is the identity

        // plain replay: the switch, the branch and the iteration count
        StepPar<T> sp = a.sp;
        sp.qm = a.qm[(fl >> GCB_SPECIES_SHIFT) & 3];
        sp.cq = sp.c / sp.qm;
        FieldPt<T, 2> F0;
        gather_any<T, 2, 2>(a.g, ib, l, F0);
        const int S = a.sw(F0, u, sp.inv_c2, (fl >> GCB_SPECIES_SHIFT) & 3, a.qm);
        int iters = 0;
        bool gca = false;
        if (S == 0) {
            T uu[3] = {u[0], u[1], u[2]}, disp[2];
            bool ncv;
            gca = replay_step(PlainGather<T, 2, 2>{a.g}, sp, ib, l, dxp, F0, uu, disp, iters, ncv);
        }
        const int ngather = gca ? iters + 2 : 1;
        if (ngather > MAXG) continue;    // excluded by the host's iteration-cap check
        const int ndir = NS + NF * ngather;

        StepPar<D> sd;
        sd.c = D(sp.c);
        sd.inv_c2 = D(sp.inv_c2);
        sd.dt = D(sp.dt);
        sd.half_dt = D(sp.half_dt);
        sd.qm = D(sp.qm);
        sd.curvature = sp.curvature;
        sd.mu_mode = sp.mu_mode;
        sd.phase = 0;
        sd.max_iter = sp.max_iter;
        sd.fixed_iters = gca ? iters : sp.fixed_iters;   // replay exactly this many
        sd.tol = D(T(-1));
        T li[NS];
#pragma unroll
        for (int k = 0; k < NS; ++k) li[k] = T(0);
        for (int base = 0; base < ndir; base += N) {
            D ld[2], ud[3], dd[2];
#pragma unroll
            for (int d = 0; d < 2; ++d) { ld[d] = D(l[d]); dd[d] = D(dxp[d]); }
#pragma unroll
            for (int k = 0; k < 3; ++k) ud[k] = D(u[k]);
#pragma unroll
            for (int j = 0; j < N; ++j) {
                const int dir = base + j;
                if (dir < 2) ld[dir].d[j] = T(1);
                else if (dir < 5) ud[dir - 2].d[j] = T(1);
                else if (dir < 7) dd[dir - 5].d[j] = T(1);
            }
            int count = 0;
            DualGather<T, N> gth{a.g, &count, base, nodes, wts};
            FieldPt<D, 2> Fd;
            gth(ib, ld, Fd);
            D disp[2];
            bool ok = false;
            if (gca) {
                int it2;
                bool ncv2;
                ok = gca_step<D, 2, 2>(gth, sd, ib, ld, dd, Fd, ud, disp, it2, ncv2);
            }
            if (!ok) boris<D, 2>(Fd.E, Fd.B, sd, ud, disp);
            // columns of this pass, contracted with the output adjoint
#pragma unroll
            for (int j = 0; j < N; ++j) {
                const int dir = base + j;
                if (dir >= ndir) break;
                T c = lo[2] * ud[0].d[j] + lo[3] * ud[1].d[j] + lo[4] * ud[2].d[j];
#pragma unroll
                for (int d = 0; d < 2; ++d)
                    c += lo[d] * (ld[d].d[j] + disp[d].d[j]) + lo[5 + d] * disp[d].d[j];
                if (dir < NS) {
                    li[dir] = c;
                } else if (c != T(0)) {
                    const int gk = (dir - NS) / NF, comp = (dir - NS) % NF;
#pragma unroll
                    for (int o = 0; o < 4; ++o)
                        atomicAdd(&a.grad[(size_t)nodes[gk * 4 + o] * 12 + comp],
                                  (double)(wts[gk * 4 + o] * c));
                }
            }
        }
#pragma unroll
        for (int k = 0; k < NS; ++k) a.lam[k][i] = li[k];
    }
}

// ---------------------------------------------------------------------------
// reverse mode: replay the step recording its gather points, then run the
// transposed step backwards (adjoint_rev.cuh), re-gathering at each point.
// ---------------------------------------------------------------------------

// Per-thread values in shared memory, 16 bytes at a time: chunk j of the
// block's thread t at [j * TPB + t], so that a quarter warp's accesses fill the
// banks and 12 components are 3 (FP64: 6) loads or stores instead of 12.
template <typename T>
struct alignas(16) Vec {
    static constexpr int n = Chunk<T>::n;
    T v[n];
};
template <typename T>
constexpr int kChunks = NF / Chunk<T>::n;      // chunks of one point's 12 components

__device__ __forceinline__ void axpy(float W, const Vec<float> &x, Vec<float> &y)
{
    const float2 w = make_float2(W, W);
    const float2 a = __ffma2_rn(make_float2(x.v[0], x.v[1]), w, make_float2(y.v[0], y.v[1]));
    const float2 b = __ffma2_rn(make_float2(x.v[2], x.v[3]), w, make_float2(y.v[2], y.v[3]));
    y.v[0] = a.x; y.v[1] = a.y; y.v[2] = b.x; y.v[3] = b.y;
}
__device__ __forceinline__ void axpy(double W, const Vec<double> &x, Vec<double> &y)
{
    y.v[0] = fma(W, x.v[0], y.v[0]);
    y.v[1] = fma(W, x.v[1], y.v[1]);
}

// a field point as 16-byte chunks: E, B, d_x B, d_y B
template <typename T>
__device__ __forceinline__ void to_chunks(const FieldPt<T, 2> &F, Vec<T> q[kChunks<T>])
{
    T v[NF];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        v[c] = F.E[c];
        v[3 + c] = F.B[c];
        v[6 + c] = F.dB[0][c];
        v[9 + c] = F.dB[1][c];
    }
#pragma unroll
    for (int c = 0; c < NF; ++c) q[c / Vec<T>::n].v[c % Vec<T>::n] = v[c];
}
template <typename T>
__device__ __forceinline__ void from_chunks(const Vec<T> q[kChunks<T>], FieldPt<T, 2> &F)
{
    T v[NF];
#pragma unroll
    for (int c = 0; c < NF; ++c) v[c] = q[c / Vec<T>::n].v[c % Vec<T>::n];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        F.E[c] = v[c];
        F.B[c] = v[3 + c];
        F.dB[0][c] = v[6 + c];
        F.dB[1][c] = v[9 + c];
    }
}

// Interpolated fields of the step's gather points, kept per thread in shared
// memory.  Point 0 is x^n, point 1 + k the step's k-th gather.
template <typename T>
struct FCache {
    Vec<T> *base;
    __device__ __forceinline__ void store(int pt, const FieldPt<T, 2> &F) const
    {
        if (pt >= GCB_ADJ_FCACHE) return;
        Vec<T> q[kChunks<T>];
        to_chunks(F, q);
#pragma unroll
        for (int j = 0; j < kChunks<T>; ++j) base[(pt * kChunks<T> + j) * TPB] = q[j];
    }
    __device__ __forceinline__ void load(int pt, FieldPt<T, 2> &F) const
    {
        Vec<T> q[kChunks<T>];
#pragma unroll
        for (int j = 0; j < kChunks<T>; ++j) q[j] = base[(pt * kChunks<T> + j) * TPB];
        from_chunks(q, F);
    }
};

// Plain gather that records where it was called (R^{n-1/2}, the iterates,
// R^{n+1/2}, in that order) and keeps what it interpolated.
template <typename T>
struct RecGather {
    DevGrid<T> g;
    T (*pts)[2];
    int *count;
    FCache<T> fc;
    __device__ __forceinline__ void operator()(const int ib[2], const T l[2], FieldPt<T, 2> &F) const
    {
        const int k = (*count)++;
        if (k < MAXG) {
            pts[k][0] = l[0];
            pts[k][1] = l[1];
        }
        gather_any<T, 2, 2>(g, ib, l, F);
        fc.store(1 + k, F);
    }
};

// Node-record adjoints of one particle-step, accumulated per thread for one
// cell (4 nodes x 12 components) in shared memory and added to the FP64 node
// accumulators when the cell changes and at the end of the step: the step's
// gathers (x^n, R^{n-1/2}, the iterates, R^{n+1/2}) mostly share one cell, so
// this replaces most of the per-gather atomics.  (One cell measured faster
// than two: the second costs shared memory that the field cache uses better.)
// The additions are made by the warp together, two threads' cells at a time,
// 16 lanes each: a lane's 48 additions on its own go to 48 separate sectors
// one by one, here 16 lanes add to 128 contiguous bytes.  The chunks of a
// thread are (TPB + 1) apart, which puts the 16 values read together in 16
// different banks.
template <typename T>
struct NodeCache {
    static constexpr int LD = TPB + 1;
    static constexpr int N = 4 * kChunks<T> * LD;   // chunks of a block
    Vec<T> *base;    // chunk (o, j) of the block's thread t at base[(o * kChunks + j) * LD + t]
    double *grad;
    int nx, ny;
    int cx, cy;      // the cached cell, cx = -1 when empty

    __device__ __forceinline__ Vec<T> &at(int o, int j) const
    {
        return base[(o * kChunks<T> + j) * LD + threadIdx.x];
    }
    // add the cached cells of the lanes that ask for it (called by the whole warp)
    __device__ __forceinline__ void flush(bool want)
    {
        unsigned m = __ballot_sync(0xffffffffu, want && cx >= 0);
        const int lane = threadIdx.x & 31, h = lane & 15;
        __syncwarp();
        while (m) {
            const int a = __ffs(m) - 1;
            m &= m - 1;
            const int b = m ? __ffs(m) - 1 : a;
            const bool act = lane < 16 || m;
            m &= m - 1;
            const int src = lane < 16 ? a : b;
            const int ix = __shfl_sync(0xffffffffu, cx, src), iy = __shfl_sync(0xffffffffu, cy, src);
            const int jx = ix + 1 == nx ? 0 : ix + 1, jy = iy + 1 == ny ? 0 : iy + 1;
            const T *v = reinterpret_cast<const T *>(base + (threadIdx.x & ~31) + src);
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const int e = h + 16 * k, o = e / NF, c = e - o * NF;   // node and component
                const T x = v[(e / Vec<T>::n) * (LD * Vec<T>::n) + e % Vec<T>::n];
                const int node = ((o & 2) ? jy : iy) * nx + ((o & 1) ? jx : ix);
                if (act && x != T(0)) atomicAdd(grad + (size_t)node * NF + c, (double)x);
            }
        }
        __syncwarp();
    }
    // make cell (ix, iy) the cached one of the lanes in `on` (called by the whole warp)
    __device__ __forceinline__ void select(bool on, int ix, int iy)
    {
        const bool other = on && (ix != cx || iy != cy);
        flush(other);
        if (!other) return;
        cx = ix;
        cy = iy;
        Vec<T> z;
#pragma unroll
        for (int c = 0; c < Vec<T>::n; ++c) z.v[c] = T(0);
#pragma unroll
        for (int o = 0; o < 4; ++o)
#pragma unroll
            for (int j = 0; j < kChunks<T>; ++j) at(o, j) = z;
    }
    __device__ __forceinline__ void finish()
    {
        flush(true);
        cx = -1;
    }
};

// Cell of a gather point: fractional position, cell and the nodes' record
// indices (both ways of finding them as the gather's own).
template <typename T>
__device__ __forceinline__ void cell_nodes(const DevGrid<T> &g, const int ib[2], const T p[2], T t[2],
                                           int i0[2], int node[4])
{
    int i1[2];
#pragma unroll
    for (int d = 0; d < 2; ++d) cell_of(g, d, ib[d], p[d], t[d], i0[d], i1[d]);
#pragma unroll
    for (int o = 0; o < 4; ++o)
        node[o] = ((o & 2) ? i1[1] : i0[1]) * g.n[0] + ((o & 1) ? i1[0] : i0[0]);
}
template <>
__device__ __forceinline__ void cell_nodes<float>(const DevGrid<float> &g, const int ib[2],
                                                  const float p[2], float t[2], int i0[2],
                                                  int node[4])
{
    CellLoc<2> q;
    locate<2>(g, ib, p, q);
    t[0] = q.t[0];
    t[1] = q.t[1];
    if (q.inner) {
        i0[0] = q.i[0];
        i0[1] = q.i[1];
        node[0] = q.i[1] * g.n[0] + q.i[0];
        node[1] = node[0] + 1;
        node[2] = node[0] + g.n[0];
        node[3] = node[2] + 1;
    } else {
        int i1[2];
#pragma unroll
        for (int d = 0; d < 2; ++d) {
            float td;
            cell_of(g, d, ib[d], p[d], td, i0[d], i1[d]);
        }
#pragma unroll
        for (int o = 0; o < 4; ++o)
            node[o] = ((o & 2) ? i1[1] : i0[1]) * g.n[0] + ((o & 1) ? i1[0] : i0[0]);
    }
}

// Transpose of F = sum_o W_o(p) rec_o: the node records receive W_o aF (via
// the cache) and the position adjoint sum_o grad W_o (rec_o . aF) is returned.
// Called by the whole warp; `on`: the lane takes part.
template <typename T>
__device__ __forceinline__ void gather_bwd(const DevGrid<T> &g, NodeCache<T> &nc, bool on,
                                           const int ib[2], const T p[2], const FieldPt<T, 2> &aF,
                                           T ap[2])
{
    T t[2];
    int i0[2], node[4];
    if (on) cell_nodes<T>(g, ib, p, t, i0, node);
    nc.select(on, i0[0], i0[1]);
    if (!on) return;
    Vec<T> av[kChunks<T>];
    to_chunks(aF, av);
    T dv[4];
#pragma unroll
    for (int o = 0; o < 4; ++o) {
        const T *rp = reinterpret_cast<const T *>(reinterpret_cast<const char *>(g.rec) +
                                                  (uint64_t)(unsigned)node[o] * (NF * sizeof(T)));
        // rec_o . aF, the record read in 16-byte chunks
        Vec<T> sum;
#pragma unroll
        for (int k = 0; k < Vec<T>::n; ++k) sum.v[k] = T(0);
#pragma unroll
        for (int j = 0; j < kChunks<T>; ++j) {
            Vec<T> r;
            load_chunk(rp + j * Vec<T>::n, r.v);
            if constexpr (sizeof(T) == 4) {
                const float2 a = __ffma2_rn(make_float2(r.v[0], r.v[1]),
                                            make_float2(av[j].v[0], av[j].v[1]),
                                            make_float2(sum.v[0], sum.v[1]));
                const float2 b = __ffma2_rn(make_float2(r.v[2], r.v[3]),
                                            make_float2(av[j].v[2], av[j].v[3]),
                                            make_float2(sum.v[2], sum.v[3]));
                sum.v[0] = a.x; sum.v[1] = a.y; sum.v[2] = b.x; sum.v[3] = b.y;
            } else {
#pragma unroll
                for (int k = 0; k < Vec<T>::n; ++k) sum.v[k] = fma(r.v[k], av[j].v[k], sum.v[k]);
            }
        }
        dv[o] = sum.v[0] + sum.v[1];
        if constexpr (sizeof(T) == 4) dv[o] += sum.v[2] + sum.v[3];
        const T W = ((o & 1) ? t[0] : T(1) - t[0]) * ((o & 2) ? t[1] : T(1) - t[1]);
#pragma unroll
        for (int j = 0; j < kChunks<T>; ++j) {
            Vec<T> y = nc.at(o, j);
            axpy(W, av[j], y);
            nc.at(o, j) = y;
        }
    }
    // sum_o grad W_o dv_o: bilinear differences
    ap[0] = g.inv_dx[0] * fma(t[1], (dv[3] - dv[2]) - (dv[1] - dv[0]), dv[1] - dv[0]);
    ap[1] = g.inv_dx[1] * fma(t[0], (dv[3] - dv[1]) - (dv[2] - dv[0]), dv[2] - dv[0]);
}

// Reverse sweep of a guiding-center step taken with K iterations whose gather
// points (R^{n-1/2}, x^n + d^1 .. x^n + d^{K-1}, R^{n+1/2}) are pts[0..K].
// One loop over the step's gather points in reverse order of their use:
//   stage 0        R^{n+1/2}: reconstruction of u
//   stage 1..K-1   x^n + d^{K-stage}: the iterate's velocity V^{K-stage}
//   stage K        x^n: V^n and the u_par update
//   stage K+1      R^{n-1/2}: conversion of u
// so that the gather, frame and scatter code is present once.
// field and frame at gather point `pt` (FCache numbering) located at p
template <typename T>
__device__ __forceinline__ void frame_at(const DevGrid<T> &g, const FCache<T> &fc, int pt,
                                         const int ib[2], const T p[2], const StepPar<T> &s,
                                         FieldPt<T, 2> &F, rev::RFrame<T, 2> &f)
{
    if (pt < GCB_ADJ_FCACHE) fc.load(pt, F);
    else gather_any<T, 2, 2>(g, ib, p, F);
    f.make(F, s.c, s.inv_c2);
}

// Called by the whole warp (the additions to the node accumulators are made
// together); `on`: the lane's particle took a guiding-center step, K its count.
template <typename T>
__device__ __forceinline__ void gca_rev(const DevGrid<T> &g, NodeCache<T> &grad, const FCache<T> &fc,
                                        const StepPar<T> &s, bool on, const int ib[2], const T l[2],
                                        const T u[3], int K, const T (*pts)[2], const T lo[NS],
                                        T li[NS])
{
    using rev::FrameAdj;
    FieldPt<T, 2> F;
    rev::RFrame<T, 2> f;
    // forward quantities of the conversion (at R^{n-1/2}) and of the u_par update (at x^n)
    rev::Conv<T> cv;
    T upn;
    if (on) {
        for (int j = 0; j < 2; ++j) {
            frame_at(g, fc, j == 0 ? 1 : 0, ib, j == 0 ? pts[0] : l, s, F, f);
            if (j == 0) rev::conv_fwd(f, s, u, cv);
            else upn = rev::upar_new(f, s, cv.upar, cv.mu, cv.uperp);
        }
    }
    T aupn = T(0), amu = T(0), auperp = T(0), aupar = T(0);
    T abpg[3] = {T(0), T(0), T(0)}, au[3] = {T(0), T(0), T(0)};
    T al[2] = {lo[0], lo[1]};
    T ad[2] = {lo[0] + lo[5], lo[1] + lo[6]};      // x^{n+1} = x^n + d^K, dxp = d^K
    T aVn[3] = {T(0), T(0), T(0)};
    T p[2] = {T(0), T(0)};
    const int KM = __reduce_max_sync(0xffffffffu, on ? K : -2);
    for (int st = 0; st <= KM + 1; ++st) {
        const bool act = on && st <= K + 1;
        FieldPt<T, 2> aF;
        if (act) {
            const T *q = st == 0 ? pts[K] : (st < K ? pts[K - st] : (st == K ? l : pts[0]));
            const int pt = st == 0 ? K + 1 : (st < K ? K - st + 1 : (st == K ? 0 : 1));
            p[0] = q[0];
            p[1] = q[1];
            frame_at(g, fc, pt, ib, p, s, F, f);
            FrameAdj<T> af;
            af.zero();
            if (st == 0) {
                const T lu[3] = {lo[2], lo[3], lo[4]};
                rev::recon_bwd(f, s, upn, cv.mu, cv.uperp, cv.bpg, lu, af, aupn, amu, auperp, abpg);
            } else if (st <= K) {
                // d^k = dt/2 (V^n + V^{k-1}) with V^0 = V^n: stage st < K carries
                // V^{K-st}; stage K carries V^n with every term collected
                T aV[3];
                if (st < K) {
                    aV[0] = s.half_dt * ad[0];
                    aV[1] = s.half_dt * ad[1];
                    aVn[0] += aV[0];
                    aVn[1] += aV[1];
                } else {
                    aV[0] = aVn[0] + s.dt * ad[0];
                    aV[1] = aVn[1] + s.dt * ad[1];
                }
                aV[2] = T(0);
                rev::gc_vel_bwd(f, s, upn, cv.mu, cv.uperp, aV, af, aupn, amu, auperp);
                if (st == K) rev::upar_bwd(f, s, cv.upar, cv.mu, cv.uperp, aupn, af, aupar, amu, auperp);
            } else {
                rev::conv_bwd(f, s, u, cv, aupar, amu, auperp, abpg, af, au);
            }
            rev::frame_bwd<T, 2>(F, f, s.c, s.inv_c2, af, aF);
        }
        T ap[2];
        gather_bwd(g, grad, act, ib, p, aF, ap);
        if (!act) continue;
        al[0] += ap[0];
        al[1] += ap[1];
        if (st == 0) {                 // R^{n+1/2} = x^n + d^K / 2
            ad[0] += T(0.5) * ap[0];
            ad[1] += T(0.5) * ap[1];
        } else if (st < K) {           // x^n + d^{K-st}
            ad[0] = ap[0];
            ad[1] = ap[1];
        } else if (st == K + 1) {      // R^{n-1/2} = x^n - dxp / 2
            li[5] = T(-0.5) * ap[0];
            li[6] = T(-0.5) * ap[1];
        }
    }
    if (!on) return;
    li[0] = al[0];
    li[1] = al[1];
    li[2] = au[0];
    li[3] = au[1];
    li[4] = au[2];
}

// Resident blocks per SM the reverse kernel is compiled for.  FP32: 3, what its
// 61 KB of shared memory allow, so up to 168 registers (4 blocks would cap
// them at 128: 172 B spilled, 16 steps' gradient of 2^18 particles 4.69 against
// 4.49 ms; 5 cached points and 4 blocks 4.85, 8 and 3 4.63, 4 and 3 4.49).
template <typename T> struct RevBlocks { static constexpr int n = 3; };
template <> struct RevBlocks<double> { static constexpr int n = 1; };

// What bounds it: issue and shared-memory latency at 12 warps per SM (issue 43%
// busy, L1 53%, DRAM idle).  Measured (GB300, 512x256 grid, 2^18 particles, 6
// iterations): 213 us a step before; 203 us with the frame's values shared with
// its transpose, reciprocals and 16-byte shared-memory accesses (10.6k -> 8.0k
// instructions a particle), 149 us with the node additions made by the warp (L1
// wavefronts 37 -> 25 M, FP64 pipe 41 -> 22%), about 140 us with 3 blocks.
template <typename T>
__global__ void __launch_bounds__(TPB, RevBlocks<T>::n) k_adjoint_rev(const AdjArgs<T> a)
{
    extern __shared__ __align__(16) unsigned char s_raw[];
    T pts[MAXG][2];
    NodeCache<T> nc;
    nc.base = reinterpret_cast<Vec<T> *>(s_raw);
    const FCache<T> fc{nc.base + NodeCache<T>::N + threadIdx.x};
    nc.grad = a.grad;
    nc.nx = a.g.n[0];
    nc.ny = a.g.n[1];
    nc.cx = nc.cy = -1;
    for (int64_t i0 = blockIdx.x * (int64_t)TPB; i0 < a.np; i0 += (int64_t)gridDim.x * TPB) {
        // every lane stays for the warp's additions; `on`: it has a particle
        // that is not frozen (whose step is the identity)
        const int64_t i = i0 + threadIdx.x;
        bool on = i < a.np;
        int ib[2];
        T l[2], u[3], dxp[2], lo[NS];
        uint8_t fl = 0;
        if (on) {
            fl = a.flags[i];
#pragma unroll
            for (int d = 0; d < 2; ++d) {
                load_pos(a, i, d, ib[d], l[d], on);
                dxp[d] = a.dxp[d][i];
                on = on && isfinite(dxp[d]);
            }
#pragma unroll
            for (int k = 0; k < 3; ++k) { u[k] = a.u[k][i]; on = on && isfinite(u[k]); }
#pragma unroll
            for (int k = 0; k < NS; ++k) lo[k] = a.lam[k][i];
        }
        StepPar<T> sp = a.sp;
        int K = 0;
        bool gca = false;
        FieldPt<T, 2> F0;
        if (on) {
            sp.qm = a.qm[(fl >> GCB_SPECIES_SHIFT) & 3];
            sp.cq = sp.c / sp.qm;
            gather_any<T, 2, 2>(a.g, ib, l, F0);
            fc.store(0, F0);
            const int S = a.sw(F0, u, sp.inv_c2, (fl >> GCB_SPECIES_SHIFT) & 3, a.qm);
            if (S == 0) {
                T uu[3] = {u[0], u[1], u[2]}, disp[2];
                bool ncv;
                int cnt = 0;
                gca = replay_step(RecGather<T>{a.g, pts, &cnt, fc}, sp, ib, l, dxp, F0, uu, disp, K, ncv);
                gca = gca && cnt == K + 1 && cnt <= MAXG;
            }
        }
        T li[NS];
        gca_rev(a.g, nc, fc, sp, gca, ib, l, u, K, pts, lo, li);
        const bool bor = on && !gca;
        if (__any_sync(0xffffffffu, bor)) {
            FieldPt<T, 2> aF;
            T au[3], ap[2];
            if (bor) {
                const T lu[3] = {lo[2], lo[3], lo[4]};
                const T ldisp[2] = {lo[0] + lo[5], lo[1] + lo[6]};
                rev::boris_bwd<T, 2>(F0.E, F0.B, sp, u, lu, ldisp, au, aF.E, aF.B);
#pragma unroll
                for (int ii = 0; ii < 2; ++ii)
#pragma unroll
                    for (int j = 0; j < 3; ++j) aF.dB[ii][j] = T(0);
            }
            gather_bwd(a.g, nc, bor, ib, l, aF, ap);
            if (bor) {
                li[0] = lo[0] + ap[0];
                li[1] = lo[1] + ap[1];
                li[2] = au[0];
                li[3] = au[1];
                li[4] = au[2];
                li[5] = T(0);
                li[6] = T(0);
            }
        }
        nc.finish();
        if (on) {
#pragma unroll
            for (int k = 0; k < NS; ++k) a.lam[k][i] = li[k];
        }
    }
}

template <typename T>
constexpr int rev_smem()
{
    return (NodeCache<T>::N + GCB_ADJ_FCACHE * kChunks<T> * TPB) * 16;
}

template <typename T>
static gcb_status launch(const AdjArgs<T> &a, int method, cudaStream_t st)
{
    if (a.np == 0) return GCB_OK;
    int64_t nb = (a.np + TPB - 1) / TPB;
    if (nb > 152 * 64) nb = 152 * 64;
    if (method == GCB_ADJ_REVERSE) {
        cudaError_t e = cudaFuncSetAttribute(k_adjoint_rev<T>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             rev_smem<T>());
        if (e != cudaSuccess) {
            set_error("k_adjoint_rev smem attribute: %s", cudaGetErrorString(e));
            return GCB_ECUDA;
        }
        k_adjoint_rev<T><<<(int)nb, TPB, rev_smem<T>(), st>>>(a);
    }
    else
        k_adjoint_sr<T, NDIR><<<(int)nb, TPB, 0, st>>>(a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        set_error("k_adjoint_sr launch: %s", cudaGetErrorString(e));
        return GCB_ECUDA;
    }
    return GCB_OK;
}

}  // namespace adj

// The adjoint of one step for all particles whose pre-step state is `s`.
gcb_status adjoint_step(const gcb_particles *s, const gcb_grid *g, const gcb_params *prm,
                        void *const lam[7], double *grad, int method, cudaStream_t st)
{
    auto fill = [&](auto &a, auto tag) {
        using T = decltype(tag);
        a.g.rec = static_cast<const T *>(g->rec);
        a.g.stride = g->stride;
        for (int d = 0; d < 3; ++d) {
            a.g.n[d] = (int)g->n[d];
            a.g.nin[d] = g->n[d] <= (1 << 22) ? (int)g->n[d] - 1 : 0;
            a.g.nR[d] = (T)g->n[d];
            a.g.dx[d] = (T)g->dx[d];
            a.g.inv_dx[d] = (T)(1.0 / g->dx[d]);
        }
        a.np = s->n;
        a.pair = s->pos_mode == GCB_POS_F32PAIR;
        for (int d = 0; d < 2; ++d) {
            a.x[d] = s->x[d];
            a.xlo[d] = static_cast<const float *>(s->x_lo[d]);
            a.dxp[d] = static_cast<const T *>(s->dxp[d]);
        }
        for (int k = 0; k < 3; ++k) a.u[k] = static_cast<const T *>(s->u[k]);
        a.flags = s->flags;
        for (int k = 0; k < 7; ++k) a.lam[k] = static_cast<T *>(lam[k]);
        a.grad = grad;
        a.sp.c = (T)prm->c;
        a.sp.inv_c2 = (T)(1.0 / (prm->c * prm->c));
        a.sp.dt = (T)prm->dt;
        a.sp.half_dt = (T)(0.5 * prm->dt);
        a.sp.qm = T(0);
        a.sp.curvature = prm->curvature;
        a.sp.mu_mode = prm->mu_mode;
        a.sp.phase = 0;   // the adjoint differentiates the step with the direction kept
        a.sp.max_iter = prm->gca_max_iter;
        a.sp.fixed_iters = prm->gca_fixed_iters;
        a.sp.tol = (T)prm->gca_tol;
        for (int k = 0; k < 4; ++k) a.qm[k] = (T)prm->qm[k];
        a.sw.fill(prm);
    };
    if (s->mom_dtype == GCB_F64) {
        adj::AdjArgs<double> a;
        fill(a, 0.0);
        return adj::launch(a, method, st);
    }
    adj::AdjArgs<float> a;
    fill(a, 0.0f);
    return adj::launch(a, method, st);
}

}  // namespace gcb

// ---------------------------------------------------------------------------
// mode projection and field combination (fields linear in mode amplitudes)
// ---------------------------------------------------------------------------
namespace gcb {
namespace adj {

// Both kernels take one FP64 multiply-add per pattern value, which the FP64 pipe
// bounds (2^17 nodes, 64 modes: 100.7 M, 160 us; the patterns' 403 MB take 60
// us).  Values are read V at a time (16 bytes; V = 1 where a pointer is not
// 16-byte aligned) and widened by their bits, which keeps the conversions off
// that pipe.  Measured (GB300, FP32 patterns): combination 382 -> 190 us,
// projection 481 -> 195 us (FP64 patterns 194 -> 178 and 288 -> 268 us).
template <typename PT, int V>
struct Pack { PT v[V]; };
template <typename PT, int V>
__device__ __forceinline__ Pack<PT, V> load_pack(const PT *p)
{
    Pack<PT, V> r;
    if constexpr (V == 1) r.v[0] = __ldg(p);
    else load_chunk(p, r.v);
    return r;
}

// dL/da_m = sum_e grad[e] pat_m[e]: a thread takes MB modes (grid row: modes
// MB blockIdx.y ...), so that grad is read once and the block's sums are
// reduced once for MB of them.
constexpr int MB = 8;
template <typename PT, int V>
__global__ void __launch_bounds__(256) k_project(const double *grad, const PT *pat, int64_t nelem,
                                                 int nmodes, double *out)
{
    __shared__ double s_w[8][MB];
    const int m0 = blockIdx.y * MB;
    double acc[MB];
#pragma unroll
    for (int j = 0; j < MB; ++j) acc[j] = 0.0;
    for (int64_t e = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) * V; e < nelem;
         e += (int64_t)gridDim.x * blockDim.x * V) {
        double g[V];
        if constexpr (V == 1) {
            g[0] = grad[e];
        } else {
#pragma unroll
            for (int k = 0; k < V; k += 2) load_chunk(grad + e + k, g + k);
        }
        Pack<PT, V> r[MB];
#pragma unroll
        for (int j = 0; j < MB; ++j)   // past the last mode: mode m0 again, not added
            r[j] = load_pack<PT, V>(pat + (size_t)(m0 + j < nmodes ? m0 + j : m0) * nelem + e);
#pragma unroll
        for (int j = 0; j < MB; ++j)
            if (m0 + j < nmodes)
#pragma unroll
                for (int k = 0; k < V; ++k) acc[j] = fma(g[k], widen<true>(r[j].v[k]), acc[j]);
    }
#pragma unroll
    for (int j = 0; j < MB; ++j) {
        for (int o = 16; o > 0; o >>= 1) acc[j] += __shfl_xor_sync(0xffffffffu, acc[j], o);
        if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5][j] = acc[j];
    }
    __syncthreads();
    if (threadIdx.x < MB && m0 + (int)threadIdx.x < nmodes) {
        double t = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += s_w[w][threadIdx.x];
        atomicAdd(&out[m0 + threadIdx.x], t);
    }
}

// rec = base + sum_m amps[m] pat_m
template <typename PT, int V>
__global__ void __launch_bounds__(256) k_combine(PT *rec, const PT *base, const PT *pat,
                                                 const double *amps, int64_t nelem, int nmodes)
{
    for (int64_t e = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) * V; e < nelem;
         e += (int64_t)gridDim.x * blockDim.x * V) {
        double v[V];
        const Pack<PT, V> b = load_pack<PT, V>(base + e);
#pragma unroll
        for (int k = 0; k < V; ++k) v[k] = widen<true>(b.v[k]);
#pragma unroll 8
        for (int m = 0; m < nmodes; ++m) {
            const Pack<PT, V> r = load_pack<PT, V>(pat + (size_t)m * nelem + e);
            const double w = __ldg(amps + m);
#pragma unroll
            for (int k = 0; k < V; ++k) v[k] = fma(w, widen<true>(r.v[k]), v[k]);
        }
        if constexpr (V == 1) {
            rec[e] = (PT)v[0];
        } else {
            Vec<PT> w;             // the records are 16-byte aligned
#pragma unroll
            for (int k = 0; k < V; ++k) w.v[k] = (PT)v[k];
            *reinterpret_cast<Vec<PT> *>(rec + e) = w;
        }
    }
}

static bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

// (nelem is a multiple of a record's 16-byte chunks, so every mode's values
// are aligned as the first one's)
template <typename PT>
static void launch_project(const double *grad, const PT *pat, int64_t nelem, int nmodes, double *out,
                           cudaStream_t st)
{
    const int groups = (nmodes + MB - 1) / MB;
    auto blocks = [&](int v) {
        int64_t n = (nelem / v + 255) / 256, cap = 152 * 6 / groups;
        return (unsigned)(n < cap ? n : cap);
    };
    constexpr int V = Chunk<PT>::n;
    if (aligned16(grad) && aligned16(pat))
        k_project<PT, V><<<dim3(blocks(V), groups), 256, 0, st>>>(grad, pat, nelem, nmodes, out);
    else
        k_project<PT, 1><<<dim3(blocks(1), groups), 256, 0, st>>>(grad, pat, nelem, nmodes, out);
}
template <typename PT>
static void launch_combine(PT *rec, const PT *base, const PT *pat, const double *amps, int64_t nelem,
                           int nmodes, cudaStream_t st)
{
    auto blocks = [&](int v) {
        const int64_t n = (nelem / v + 255) / 256;
        return (unsigned)(n < 152 * 32 ? n : 152 * 32);
    };
    constexpr int V = Chunk<PT>::n;
    if (aligned16(base) && aligned16(pat))
        k_combine<PT, V><<<blocks(V), 256, 0, st>>>(rec, base, pat, amps, nelem, nmodes);
    else
        k_combine<PT, 1><<<blocks(1), 256, 0, st>>>(rec, base, pat, amps, nelem, nmodes);
}

}  // namespace adj

gcb_status grad_project(const gcb_grid *g, const double *grad, const void *pat, int nmodes,
                        double *out, cudaStream_t st)
{
    const int64_t nelem = g->n[0] * g->n[1] * g->n[2] * (int64_t)g->stride;
    if (cudaMemsetAsync(out, 0, sizeof(double) * nmodes, st) != cudaSuccess) {
        set_error("cudaMemsetAsync: %s", cudaGetErrorString(cudaGetLastError()));
        return GCB_ECUDA;
    }
    if (g->dtype == GCB_F32)
        adj::launch_project<float>(grad, (const float *)pat, nelem, nmodes, out, st);
    else
        adj::launch_project<double>(grad, (const double *)pat, nelem, nmodes, out, st);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) { set_error("k_project: %s", cudaGetErrorString(e)); return GCB_ECUDA; }
    return GCB_OK;
}

gcb_status grid_combine(const gcb_grid *g, const void *base, const void *pat, const double *amps,
                        int nmodes, cudaStream_t st)
{
    const int64_t nelem = g->n[0] * g->n[1] * g->n[2] * (int64_t)g->stride;
    if (g->dtype == GCB_F32)
        adj::launch_combine<float>((float *)g->rec, (const float *)base, (const float *)pat, amps,
                                   nelem, nmodes, st);
    else
        adj::launch_combine<double>((double *)g->rec, (const double *)base, (const double *)pat, amps,
                                    nelem, nmodes, st);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) { set_error("k_combine: %s", cudaGetErrorString(e)); return GCB_ECUDA; }
    return GCB_OK;
}

}  // namespace gcb

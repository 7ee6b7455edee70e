// Sweep with the hierarchical (quadtree) identity topology (Sec. 3.3 factor
// graph; Sec. 4.2: sigma_R and sigma_P halved per level). Pixels keep the state
// layout of the grid sweep, using identity slot 0 for the factor to their level-1
// node (slots 1..3 are zero in both state buffers from the start and are not
// written: 324 of a pixel's 604 bytes; k_qt_clear zeroes what a loaded checkpoint
// held there); pose nodes of every level live in one
// structure-of-arrays buffer. One synchronous sweep = k_qt_messages +
// k_qt_node_belief: the first (pixel updates and the messages into the nodes)
// reads only the `in` buffers, the second the node messages the first wrote, and
// both write the `out` buffers.
#pragma once

#include "pv_kernels.cuh"

namespace pv {

// node state planes
constexpr int NP_MU = 0;      // pose (6)
constexpr int NP_M = 6;       // belief information: prior + damped messages (21, packed)
constexpr int NP_MSG = 27;    // message slots 0..3 (children 2 (row % 2) + col % 2), 4 (parent): Lambda 21 + eta 6
constexpr int NP_PARENT = 4;
constexpr int NODE_PLANES = NP_MSG + 5 * ID_STRIDE;   // 162
constexpr int QT_MAX_LEVELS = 20;

// the node grid of every level
struct QtGeom {
    int n_levels;                  // levels 1..n_levels (level l at index l - 1)
    int w[QT_MAX_LEVELS], h[QT_MAX_LEVELS];
    int base[QT_MAX_LEVELS];       // first node index of the level
    int n_nodes;                   // nodes of all levels
    size_t stride;                 // elements per node plane (n_nodes rounded up)
};

template <typename T>
struct QtArgs {
    Geometry<T> g;
    Factors<T> f;
    QtGeom q;
    const T* in;          // pixel state (tile-major)
    T* out;
    const T* nin;         // node state (plane p of node n at p * stride + n)
    T* nout;
    const T* I_s;
    const T* I_t;
    const T* g_x;
    const T* g_y;
    const T* m_x;
    const T* m_y;
    Scalars* sc;
};

__host__ __device__ inline int qt_node(const QtGeom& q, int level, int r, int c) {
    return q.base[level - 1] + r * q.w[level - 1] + c;
}

// One pixel's sweep update: as the grid sweep (priors, normal-integration messages
// from the four grid neighbours, photometric factor, structured belief solve,
// mu (+) tau, projected stores), with the identity message coming only from the
// pixel's level-1 node.
// (bx, by: the block's position in the pixel grid of blocks of 32 x 4)
template <typename T>
__device__ __forceinline__ void qt_pixels(const QtArgs<T>& a, int bx, int by) {
    const int u = bx * blockDim.x + threadIdx.x;
    const int v = by * blockDim.y + threadIdx.y;
    const Geometry<T>& g = a.g;
    const Factors<T>& F = a.f;
    if (u >= g.W || v >= g.H) return;
    const int i = v * g.pitch + u;
    const T* Si = a.in + state_index(u, v, g.tiles_x);
    T* Di = a.out + state_index(u, v, g.tiles_x);
    T xi[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) xi[k] = Si[k * TILE_PX];
    const T d = Si[6 * TILE_PX];
    T qi[4], t[3];
    se3_exp_q(xi, qi, t);
    T eb[7], Mp[21];
#pragma unroll
    for (int q = 0; q < 7; ++q) eb[q] = T(0);
#pragma unroll
    for (int q = 0; q < 21; ++q) Mp[q] = T(0);
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        Mp[pidx(k, k)] = F.lam_P;
        eb[k] -= F.lam_P * xi[k];
    }
    T md = F.lam_Z;
    eb[6] -= F.lam_Z * (d - T(a.sc->d_prior));
    unsigned flags = 0;
    const T beta = F.beta, omb = T(1) - F.beta;

    // first, so that its taps load with the node's planes (after the messages: 99.7
    // against 92.4 us a sweep at 640x480, 26.9 against 25.8 at 320x240)
    T alpha, rph, J[7];
    unsigned char br;
    photometric_factor<T>(a, i, u, v, qi, t, d, J, alpha, rph, br, flags);
    // identity factor to the level-1 node (slot 0)
    T Lnew[21], enew6[6];
    {
        const QtGeom& q = a.q;
        const int n = qt_node(q, 1, v / 2, u / 2);
        const int k = 2 * (v % 2) + (u % 2);
        const T* N = a.nin + n;
        const size_t st = q.stride;
        T xs[6], W[21], ev[6], rb[6];
#pragma unroll
        for (int c = 0; c < 6; ++c) xs[c] = N[(NP_MU + c) * st];
        const T* mk = N + (NP_MSG + ID_STRIDE * k) * st;
#pragma unroll
        for (int c = 0; c < 21; ++c) W[c] = N[(NP_M + c) * st] - mk[c * st];
#pragma unroll
        for (int c = 0; c < 6; ++c) ev[c] = -mk[(21 + c) * st];
        se3_between(xs, qi, t, rb);
        IdMsg<T, false> m;
        if (!identity_msg(W, xs, ev, rb, F.lam_R, m)) flags |= FLAG_NONPOS_PIVOT;
        const T* old = Si + PL_ID * TILE_PX;
        const T wl = omb * F.lam_R, wll = wl * F.lam_R;
#pragma unroll
        for (int r = 0; r < 6; ++r)
#pragma unroll
            for (int c = 0; c <= r; ++c) {
                const T l = m.lambda(r, c, wl, wll, beta * old[pidx(r, c) * TILE_PX]);
                Lnew[pidx(r, c)] = l;
                Mp[pidx(r, c)] += l;
            }
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            enew6[c] = v_fma(wl, m.he[c], beta * old[(21 + c) * TILE_PX]);
            eb[c] += enew6[c];
        }
    }
    // normal-integration factors (Eq. 6) with the four grid neighbours
    T nl[4], ne[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        nl[k] = T(0);
        ne[k] = T(0);
        const int un = u + (k == 0 ? -1 : (k == 1 ? 1 : 0));
        const int vn = v + (k == 2 ? -1 : (k == 3 ? 1 : 0));
        if (un < 0 || un >= g.W || vn < 0 || vn >= g.H) continue;
        const int ko = k ^ 1;
        const T* Sj = a.in + state_index(un, vn, g.tiles_x);
        const T dj = Sj[6 * TILE_PX];
        const T sv = Sj[PL_S * TILE_PX] - Sj[(PL_NM + 2 * ko) * TILE_PX];
        const T evn = -Sj[(PL_NM + 2 * ko + 1) * TILE_PX];
        const T m = k == 0 ? a.m_x[i - 1] : (k == 1 ? a.m_x[i] : (k == 2 ? a.m_y[i - g.pitch] : a.m_y[i]));
        const T sg = (k == 0 || k == 2) ? T(1) : T(-1);
        const T rn = d - dj + sg * m;
        const T den = v_div(T(1), F.lam_N + sv);
        nl[k] = omb * (F.lam_N * sv * den) + beta * Si[(PL_NM + 2 * k) * TILE_PX];
        ne[k] = omb * (F.lam_N * (evn - sv * rn) * den) + beta * Si[(PL_NM + 2 * k + 1) * TILE_PX];
        md += nl[k];
        eb[6] += ne[k];
    }
    T tau[7], qv;
    belief_update(Mp, md, eb, J, alpha, rph, tau, qv, br, flags);
    {
        T xn[6];
        se3_update(qi, t, tau, xn);
#pragma unroll
        for (int q = 0; q < 6; ++q) Di[q * TILE_PX] = xn[q];
        Di[6 * TILE_PX] = d + tau[6];
    }
    {
        T sb, sd;
        depth_marginals(md, alpha, J[6], qv, &sb, &sd);
#pragma unroll
        for (int q = 0; q < 21; ++q) Di[(PL_MP + q) * TILE_PX] = Mp[q];
#pragma unroll
        for (int q = 0; q < 6; ++q) Di[(PL_U + q) * TILE_PX] = sb * J[q];
        Di[PL_S * TILE_PX] = sd;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        Di[(PL_NM + 2 * k) * TILE_PX] = nl[k];
        Di[(PL_NM + 2 * k + 1) * TILE_PX] = ne[k] - nl[k] * tau[6];
    }
    {
        T* d0 = Di + PL_ID * TILE_PX;
#pragma unroll
        for (int q = 0; q < 21; ++q) d0[q * TILE_PX] = Lnew[q];
#pragma unroll
        for (int r = 0; r < 6; ++r) {
            T e = enew6[r];
#pragma unroll
            for (int c = 0; c < 6; ++c) e -= Lnew[pidx(r, c)] * tau[c];
            d0[(21 + r) * TILE_PX] = e;
        }
    }
    if (flags) atomicOr(&a.sc->flags, flags);
}

// level of node n (1-based)
__device__ __forceinline__ int qt_level(const QtGeom& q, int n) {
    int lvl = 1;
    while (lvl < q.n_levels && n >= q.base[lvl]) ++lvl;
    return lvl;
}

// Node update, in two launches per sweep. A node's five messages (children
// 0..3, parent 4) are independent given the input state, so they are computed by
// one thread each (k_qt_messages); one thread per node then forms the belief,
// updates the pose and projects the messages (k_qt_node_belief). With one thread
// per node doing all five slots in sequence, the 102k nodes of a 640x480 image
// fit in a single wave and the sweep waited on that chain of dependent
// load-and-solve steps.

// row, column, level and level-wise scale 4^(l-1) of node n
struct NodePos {
    int lvl, r, c;
};
__device__ __forceinline__ NodePos node_pos(const QtGeom& q, int n) {
    NodePos p;
    p.lvl = qt_level(q, n);
    const int idx = n - q.base[p.lvl - 1];
    p.r = idx / q.w[p.lvl - 1];
    p.c = idx % q.w[p.lvl - 1];
    return p;
}

template <typename T>
__device__ __forceinline__ T level_scale(int lvl) {
    T s = T(1);
    for (int k = 0; k < lvl - 1; ++k) s *= T(4);
    return s;
}

// One thread per node message: the damped identity message into node n from its
// slot k (children 2 (row % 2) + col % 2, parent 4), written unprojected to the
// node's output slot (zero where the slot has no partner: a child outside the
// level below, the root's parent). Threads, in order: one per pixel in tile
// order (the child slot of its level-1 node, so that the pixel loads coalesce),
// then the child slots of the nodes of levels >= 2 (slot-major), then the parent
// slot of every node. Each thread issues all its loads before any arithmetic.
template <typename T>
__device__ __forceinline__ void qt_node_msgs(const QtArgs<T>& a, int blk) {
    const QtGeom& q = a.q;
    const Geometry<T>& g = a.g;
    const Factors<T>& F = a.f;
    const size_t st = q.stride;
    const size_t gid = (size_t)blk * TILE_PX + threadIdx.y * TILE_W + threadIdx.x;
    const int tiles_y = (g.H + TILE_H - 1) / TILE_H;
    const size_t n_px = (size_t)g.tiles_x * tiles_y * TILE_PX;
    const int n_up = q.n_levels > 1 ? q.n_nodes - q.base[1] : 0;     // nodes of levels >= 2
    const size_t n_up_p = ((size_t)n_up + 31) / 32 * 32;
    int n, k, lvl, r, c;
    const T* S = nullptr;      // sender: child pixel (tile-major state) ...
    const T* C = nullptr;      // ... or node (node planes)
    const T* ms = nullptr;     // the sender's stored message on the shared factor
    T lam;
    if (gid < n_px) {
        // a level-1 node's child slot, one thread per pixel in tile order
        const int tile = (int)(gid / TILE_PX), lane = (int)(gid % TILE_PX);
        const int u = (tile % g.tiles_x) * TILE_W + lane % TILE_W;
        const int v = (tile / g.tiles_x) * TILE_H + lane / TILE_W;
        if (u >= g.W || v >= g.H) return;
        lvl = 1;
        r = v / 2;
        c = u / 2;
        n = qt_node(q, 1, r, c);
        k = 2 * (v % 2) + u % 2;
        S = a.in + state_index(u, v, g.tiles_x);
        lam = F.lam_R;
        // child slots of this node without a pixel (odd width or height) are zeroed
        // by the pixel before them
        const bool nx = u % 2 == 0 && u + 1 >= g.W, ny = v % 2 == 0 && v + 1 >= g.H;
        if (nx || ny) {
            T* z0 = a.nout + n + NP_MSG * st;
            for (int m = 0; m < ID_STRIDE; ++m) {
                if (nx) z0[(ID_STRIDE * (k + 1) + m) * st] = T(0);
                if (ny) z0[(ID_STRIDE * (k + 2) + m) * st] = T(0);
                if (nx && ny) z0[(ID_STRIDE * (k + 3) + m) * st] = T(0);
            }
        }
    } else if (gid < n_px + 4 * n_up_p) {
        // child slot k of a node of level >= 2
        const size_t g2 = gid - n_px;
        k = (int)(g2 / n_up_p);
        const int j = (int)(g2 % n_up_p);
        if (j >= n_up) return;
        n = q.base[1] + j;
        const NodePos p = node_pos(q, n);
        lvl = p.lvl;
        r = p.r;
        c = p.c;
        const int rc = 2 * r + k / 2, cc = 2 * c + k % 2;
        if (rc < q.h[lvl - 2] && cc < q.w[lvl - 2]) {
            C = a.nin + qt_node(q, lvl - 1, rc, cc);
            ms = C + (NP_MSG + ID_STRIDE * NP_PARENT) * st;
        }
        lam = F.lam_R * level_scale<T>(lvl);                     // sigma_R / 2^(l-1)
    } else {
        // parent slot of every node
        const size_t g3 = gid - n_px - 4 * n_up_p;
        if (g3 >= (size_t)q.n_nodes) return;
        n = (int)g3;
        k = NP_PARENT;
        const NodePos p = node_pos(q, n);
        lvl = p.lvl;
        r = p.r;
        c = p.c;
        if (lvl < q.n_levels) {
            const int kp = 2 * (r % 2) + (c % 2);
            C = a.nin + qt_node(q, lvl + 1, r / 2, c / 2);
            ms = C + (NP_MSG + ID_STRIDE * kp) * st;
        }
        lam = F.lam_R * level_scale<T>(lvl) * T(4);              // sigma_R / 2^l
    }
    T* dst = a.nout + n + (NP_MSG + ID_STRIDE * k) * st;
    const T* N = a.nin + n;
    // every load of the thread first: own pose, own old message, the sender's data
    T xi[6], ov[ID_STRIDE], xs[6], W[21], u[6], ev[6];
#pragma unroll
    for (int m = 0; m < 6; ++m) xi[m] = N[(NP_MU + m) * st];
#pragma unroll
    for (int m = 0; m < ID_STRIDE; ++m) ov[m] = N[(NP_MSG + ID_STRIDE * k + m) * st];
    if (S) {
#pragma unroll
        for (int m = 0; m < 6; ++m) {
            xs[m] = S[m * TILE_PX];
            u[m] = S[(PL_U + m) * TILE_PX];
            ev[m] = -S[(PL_ID + 21 + m) * TILE_PX];
        }
#pragma unroll
        for (int m = 0; m < 21; ++m) W[m] = S[(PL_MP + m) * TILE_PX] - S[(PL_ID + m) * TILE_PX];
    } else if (C) {
#pragma unroll
        for (int m = 0; m < 6; ++m) {
            xs[m] = C[(NP_MU + m) * st];
            u[m] = T(0);
            ev[m] = -ms[(21 + m) * st];
        }
#pragma unroll
        for (int m = 0; m < 21; ++m) W[m] = C[(NP_M + m) * st] - ms[m * st];
    } else {
#pragma unroll 1
        for (int m = 0; m < ID_STRIDE; ++m) dst[m * st] = T(0);
        return;
    }
    T qi[4], t[3], rb[6];
    se3_exp_q(xi, qi, t);
    se3_between(xs, qi, t, rb);
    unsigned flags = 0;
    IdMsg<T> im;
    if (!identity_msg(W, u, ev, rb, lam, im)) flags |= FLAG_NONPOS_PIVOT;
    const T beta = F.beta, wl = (T(1) - F.beta) * lam, wll = wl * lam;
#pragma unroll
    for (int rr = 0; rr < 6; ++rr)
#pragma unroll
        for (int cc = 0; cc <= rr; ++cc)
            dst[pidx(rr, cc) * st] = im.lambda(rr, cc, wl, wll, beta * ov[pidx(rr, cc)]);
#pragma unroll
    for (int m = 0; m < 6; ++m) dst[(21 + m) * st] = v_fma(wl, im.he[m], beta * ov[21 + m]);
    if (flags) atomicOr(&a.sc->flags, flags);
}

// One thread per node: belief = pose prior (sigma_P / 2^l) plus the five damped
// messages k_qt_messages left in the output slots (summed in slot order), belief
// solve, Exp/Log update, and eta <- eta - Lambda tau on every slot in place.
template <typename T>
__device__ __forceinline__ void qt_node_belief(const QtArgs<T>& a, int blk) {
    const QtGeom& q = a.q;
    const int n = blk * blockDim.x + threadIdx.x;
    if (n >= q.n_nodes) return;
    const Factors<T>& F = a.f;
    const size_t st = q.stride;
    const NodePos p = node_pos(q, n);
    const T* N = a.nin + n;
    T* O = a.nout + n;
    T xi[6], qi[4], t[3];
#pragma unroll
    for (int k = 0; k < 6; ++k) xi[k] = N[(NP_MU + k) * st];
    se3_exp_q(xi, qi, t);
    const T lamP = F.lam_P * level_scale<T>(p.lvl) * T(4);     // sigma_P / 2^l
    T Mb[21], eb[6];
#pragma unroll
    for (int k = 0; k < 21; ++k) Mb[k] = T(0);
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        Mb[pidx(k, k)] = lamP;
        eb[k] = -lamP * xi[k];
    }
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        const T* mk = O + (NP_MSG + ID_STRIDE * k) * st;
#pragma unroll
        for (int m = 0; m < 21; ++m) Mb[m] += mk[m * st];
#pragma unroll
        for (int m = 0; m < 6; ++m) eb[m] += mk[(21 + m) * st];
    }
    unsigned flags = 0;
    T tau[6], L[21], idg[6];
#pragma unroll
    for (int k = 0; k < 21; ++k) L[k] = Mb[k];
    const bool ok = chol_packed<6>(L, idg);
#pragma unroll
    for (int k = 0; k < 6; ++k) tau[k] = eb[k];
    fwd_solve<6>(L, idg, tau);
    bwd_solve<6>(L, idg, tau);
    bool fin = true;
#pragma unroll
    for (int k = 0; k < 6; ++k) fin = fin && v_finite(tau[k]);
    if (!ok) flags |= FLAG_NONPOS_PIVOT;
    if (!ok || !fin) {
        if (!fin) flags |= FLAG_NONFINITE;
#pragma unroll
        for (int k = 0; k < 6; ++k) tau[k] = T(0);
    }
    {
        T xn[6];
        se3_update(qi, t, tau, xn);
#pragma unroll
        for (int k = 0; k < 6; ++k) O[(NP_MU + k) * st] = xn[k];
    }
#pragma unroll
    for (int k = 0; k < 21; ++k) O[(NP_M + k) * st] = Mb[k];
#pragma unroll 1
    for (int k = 0; k < 5; ++k) {
        T* dk = O + (NP_MSG + ID_STRIDE * k) * st;
        T Lk[21];
#pragma unroll
        for (int m = 0; m < 21; ++m) Lk[m] = dk[m * st];
#pragma unroll
        for (int rr = 0; rr < 6; ++rr) {
            T e = dk[(21 + rr) * st];
#pragma unroll
            for (int cc = 0; cc < 6; ++cc) e -= Lk[pidx(rr, cc)] * tau[cc];
            dk[(21 + rr) * st] = e;
        }
    }
    if (flags) atomicOr(&a.sc->flags, flags);
}

// The kernels, for one sequence or the n sequences of a batch alike (the same
// code, so that a batch reproduces its sequences bit for bit): one launch of
// each per sweep. Block b belongs to sequence i with off[i] <= b < off[i + 1]
// (A[i]: its arguments in device memory, off: the kernel's prefix sums of blocks
// per sequence, n + 1 values) and runs as block b - off[i] of that sequence's
// grid.
__device__ __forceinline__ int batch_seq(const int* __restrict__ off, int n, int b) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) / 2;
        if (__ldg(off + mid) <= b)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// Blocks of k_qt_messages within a sequence: one per 32 x 4 pixels, then the
// node messages' (independent of the pixels', so one launch holds both).
template <typename T>
__global__ void __launch_bounds__(TILE_PX, sizeof(T) == 4 ? 4 : 2) k_qt_messages(const QtArgs<T>* __restrict__ A,
                                                                                 const int* __restrict__ off, int n) {
    const int i = batch_seq(off, n, blockIdx.x);
    const QtArgs<T>& a = A[i];
    const int lb = blockIdx.x - __ldg(off + i), px = a.g.tiles_x * ((a.g.H + TILE_H - 1) / TILE_H);
    pdl_wait();
    if (lb < px)
        qt_pixels(a, lb % a.g.tiles_x, lb / a.g.tiles_x);
    else
        qt_node_msgs(a, lb - px);
    pdl_trigger();
}

template <typename T>
__global__ void __launch_bounds__(128) k_qt_node_belief(const QtArgs<T>* __restrict__ A,
                                                              const int* __restrict__ off, int n) {
    const int i = batch_seq(off, n, blockIdx.x);
    pdl_wait();
    qt_node_belief(A[i], blockIdx.x - __ldg(off + i));
    pdl_trigger();
}

// After a load, whose blob may hold values in identity slots 1..3: zeros in those of
// the buffer that the sweep before this kernel has written, while Scalars::qt_clear
// says that one may hold values. The count is in device memory, so that sweeps
// captured in a graph before the load clear too when they are replayed. (Tested in
// the sweep's own kernels it cost every sweep 1 to 2 %: k_qt_messages is at its
// register limit.) Block = 128 threads; the last one to have read the count lowers it.
template <typename T>
__global__ void k_qt_clear(Geometry<T> g, T* __restrict__ state, Scalars* sc) {
    pdl_wait();
    const unsigned c = *static_cast<volatile unsigned*>(&sc->qt_clear);
    if (c) {
        const int n_tiles = g.tiles_x * ((g.H + TILE_H - 1) / TILE_H), lane = threadIdx.x;
        for (int tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
            const int u = (tile % g.tiles_x) * TILE_W + lane % TILE_W, v = (tile / g.tiles_x) * TILE_H + lane / TILE_W;
            if (u >= g.W || v >= g.H) continue;
            T* d = state + (size_t)tile * TILE_WORDS + (PL_ID + ID_STRIDE) * TILE_PX + lane;
            for (int q = 0; q < MSG_PLANES - ID_STRIDE; ++q) d[q * TILE_PX] = T(0);
        }
    }
    __syncthreads();  // every thread of the block has read the count
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(&sc->qt_ticket, 1u) == gridDim.x - 1) {
            sc->qt_ticket = 0u;
            if (c) sc->qt_clear = c - 1;
        }
    }
}

// Keyframe reset of every node: identity pose, belief = the level's pose prior,
// no messages.
template <typename T>
__global__ void k_qt_reset(QtGeom q, T lam_P, T* __restrict__ nodes) {
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= q.n_nodes) return;
    const int lvl = qt_level(q, n);
    T lam = lam_P;
    for (int k = 0; k < lvl; ++k) lam *= T(4);
    for (int p = 0; p < NODE_PLANES; ++p) nodes[p * q.stride + n] = T(0);
    for (int k = 0; k < 6; ++k) nodes[(NP_M + pidx(k, k)) * q.stride + n] = lam;
}

}  // namespace pv

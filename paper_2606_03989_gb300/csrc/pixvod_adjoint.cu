// Adjoint kernels of the sweep, compiled on their own: their launchers are
// called from pixvod.cu. Two reverse passes of one sweep exist:
//  - the hand-written reverse pass (pv_adjoint_hw.cuh) in the state's
//    precision, no tape, in stages (k_adjoint_fwd, _main, _dir, _pose); the
//    product path;
//  - k_adjoint_sweep: a reverse-mode tape of the same update in FP64
//    (pv_adjoint.cuh), kept to cross-check the hand-written pass.
#include "pv_adjoint.cuh"
#include "pv_adjoint_hw.cuh"
#include "pv_launch.h"

namespace pv {

namespace {

// Scratch between the stages of the hand-written pass, tile-major like the
// state (plane p of a tile's pixel `lane` at tile * SCR_WORDS + p * TILE_PX +
// lane). Regions:
//   SCR_SUM   the damped messages summed over the directions (Lambda 21, eta
//             6) and the sum of Lambda_k ybar(eta_k') (6), from k_adjoint_fwd,
//             read by the main stage;
//   SCR_MAIN  what the main stage hands on (hw::MO_*); k_adjoint_dir adds its
//             R and t adjoints to the MO_RB and MO_TB planes;
//   SCR_CHK   the main stage's recomputed outputs (all but the identity
//             messages': outputs 0-34 and 143-150, chk_plane) and
//   SCR_CHK_S the scales of the normal messages' eta (formed by cancelling
//             terms), read by k_adjoint_pose for the recompute check.
// The damped messages themselves and what their reverse pass needs are formed
// again by k_adjoint_dir: keeping them (324 more planes, 100 MB at 320x240, out
// of L2) cost more than the few hundred operations.
// No kernel loads a plane that it writes. Scratch and adjoint state are read once
// and through L2 (the previous stage may still be draining when a stage starts).
constexpr int SCR_SUM = 0;
constexpr int SCR_MAIN = SCR_SUM + 33;
constexpr int SCR_CHK = SCR_MAIN + hw::MO_PLANES;
constexpr int SCR_CHK_S = SCR_CHK + 43;
constexpr int SCR_PLANES = SCR_CHK_S + 4;

// plane of output q (not an identity message's) in SCR_CHK
__host__ __device__ constexpr int chk_plane(int q) { return q < 35 ? q : q - 108; }
constexpr int SCR_WORDS = SCR_PLANES * TILE_PX;

// A pass's arguments in the state's precision (the kernels convert nothing)
template <typename T>
struct HwArgs {
    Geometry<T> g;
    T d_prior, lam_P, lam_Z, lam_R, beta, t_huber, lam_D, inv_sigma_D, lam_N;
    const T* Sin;    // S_{s-1}
    const T* Sout;   // S_s
    const T* Ao;     // adjoint of S_s
    T* Ai;           // adjoint of S_{s-1}
    const unsigned char* br;
    const T* I_s;
    const T* I_t;
    const T* g_x;
    const T* g_y;
    const T* m_x;
    const T* m_y;
    double* dI_s;
    double* dI_t;
    double* dparam;
    unsigned long long* mismatch;
    const AdjScale* scale;
    AdjScale* scale_next;
    unsigned long long* adj_max;
    unsigned* ticket;
};

template <typename T>
HwArgs<T> hw_args(const AdjArgs& A) {
    HwArgs<T> h;
    h.g.W = A.g.W;
    h.g.H = A.g.H;
    h.g.pitch = A.g.pitch;
    h.g.plane = A.g.plane;
    h.g.tiles_x = A.g.tiles_x;
    h.g.fx = T(A.g.fx);
    h.g.fy = T(A.g.fy);
    h.g.cx = T(A.g.cx);
    h.g.cy = T(A.g.cy);
    h.g.ifx = T(A.g.ifx);
    h.g.ify = T(A.g.ify);
    h.d_prior = T(A.d_prior);
    h.lam_P = T(A.lam_P);
    h.lam_Z = T(A.lam_Z);
    h.lam_R = T(A.lam_R);
    h.beta = T(A.beta);
    h.t_huber = T(A.t_huber);
    h.lam_D = T(A.lam_D);
    h.inv_sigma_D = T(A.inv_sigma_D);
    h.lam_N = T(A.lam_N);
    h.Sin = static_cast<const T*>(A.state_in);
    h.Sout = static_cast<const T*>(A.state_out);
    h.Ao = static_cast<const T*>(A.adj_out);
    h.Ai = static_cast<T*>(A.adj_in);
    h.br = A.br;
    h.I_s = static_cast<const T*>(A.I_s);
    h.I_t = static_cast<const T*>(A.I_t);
    h.g_x = static_cast<const T*>(A.g_x);
    h.g_y = static_cast<const T*>(A.g_y);
    h.m_x = static_cast<const T*>(A.m_x);
    h.m_y = static_cast<const T*>(A.m_y);
    h.dI_s = A.dI_s;
    h.dI_t = A.dI_t;
    h.dparam = A.dparam;
    h.mismatch = A.mismatch;
    h.scale = A.scale;
    h.scale_next = A.scale_next;
    h.adj_max = A.adj_max;
    h.ticket = A.ticket;
    return h;
}

// v 2^E in FP64. A float's goes through its bits: conversion, multiplication and
// addition in FP64 run at 1/64 of the FP32 rate here.
__device__ __forceinline__ double scaled_double(float v, int E, double scale) {
    (void)scale;
    const int b = __float_as_int(v), x = (b >> 23) & 0xff, y = x + (1023 - 127) + E;
    if (x == 0 || x == 0xff || y <= 0 || y >= 2047) return ldexp(double(v), E);
    return __hiloint2double((b & 0x80000000) | (y << 20) | ((b & 0x7fffff) >> 3), b << 29);
}
__device__ __forceinline__ double scaled_double(double v, int, double scale) { return v * scale; }

// m = the larger of m and |x|, if x is finite
template <typename T>
__device__ __forceinline__ void absmax_acc(T x, T& m) {
    const T b = v_abs(x);
    if (b > m && v_finite(b)) m = b;
}

// I/O of one pixel's reverse pass in the kernel: reads from the state before
// the sweep and the adjoint of the state after it; adds the input adjoints to
// the adjoint of the previous state (atomically: neighbours add to the same
// planes), to dI_t (atomically) and to thread-local sums. DIR: a stage that
// works on one direction, whose neighbour is sj[0].
template <typename T, bool DIR>
struct KernelIO {
    const T* Sin;
    const T* Ao;
    T* Ai;
    double* dI_t;
    int W, H;
    size_t si, sj[DIR ? 1 : 4];
    int tx[4], ty[4];
    T Is, tapv[12];
    T in_scale;        // adj_out is read times this
    int out_exp;       // the FP64 gradients' factor is 2^out_exp
    double out_scale;
    T dIs, lamD, isD, lamN;  // one value each in a pixel's pass
    T amax;                  // largest |value| added to adj_in (finite)

    __device__ size_t nbi(int k) const { return DIR ? sj[0] : sj[k]; }
    __device__ T mu(int q) const { return __ldg(Sin + si + q * TILE_PX); }
    __device__ T msg(int k, int q) const { return __ldg(Sin + si + (PL_ID + ID_STRIDE * k + q) * TILE_PX); }
    __device__ T nm(int q) const { return __ldg(Sin + si + (PL_NM + q) * TILE_PX); }
    __device__ T nb(int k, int q) const { return __ldg(Sin + nbi(k) + nb_plane(q, k) * TILE_PX); }
    __device__ T I_s() const { return Is; }
    __device__ T tap(int q) const { return tapv[q]; }
    __device__ T ybar(int q) const { return __ldcg(Ao + si + q * TILE_PX) * in_scale; }
    // the stages' scratch (scr_in, scr_out: the pixel's planes)
    const T* scr_in;
    T* scr_out;
    __device__ void identity_sums(const T*, const T*, T* L, T* e) const {
        for (int q = 0; q < 21; ++q) L[q] = __ldcg(scr_in + (SCR_SUM + q) * TILE_PX);
        for (int q = 0; q < 6; ++q) e[q] = __ldcg(scr_in + (SCR_SUM + 21 + q) * TILE_PX);
    }
    __device__ void identity_eta_adj(T* w) const {
        for (int q = 0; q < 6; ++q) w[q] = __ldcg(scr_in + (SCR_SUM + 27 + q) * TILE_PX);
    }
    __device__ void main_out(int p, T v) const { scr_out[(SCR_MAIN + p) * TILE_PX] = v; }
    __device__ T main_in(int p) const { return __ldcg(scr_in + (SCR_MAIN + p) * TILE_PX); }
    // the main stage's recomputed outputs go to the scratch and k_adjoint_pose
    // compares them with the sweep kernel's (the comparison's loads would
    // otherwise stall the stage's chain; the fwd and dir stages check the identity
    // messages)
    __device__ void out(int q, T y, T scale) const {
        scr_out[(SCR_CHK + chk_plane(q)) * TILE_PX] = y;
        if (q >= 144 && (q & 1) == 0) scr_out[(SCR_CHK_S + (q - 144) / 2) * TILE_PX] = scale;
    }
    __device__ void add(T* p, T v) {
        atomicAdd(p, v);
        absmax_acc(v, amax);
    }
    __device__ void add_mu(int q, T v) { add(Ai + si + q * TILE_PX, v); }
    __device__ void add_msg(int k, int q, T v) { add(Ai + si + (PL_ID + ID_STRIDE * k + q) * TILE_PX, v); }
    __device__ void add_nm(int q, T v) { add(Ai + si + (PL_NM + q) * TILE_PX, v); }
    __device__ void add_nb(int k, int q, T v) { add(Ai + nbi(k) + nb_plane(q, k) * TILE_PX, v); }
    __device__ void add_Is(T v) { dIs = v; }
    // taps 0-3 of I_t directly; 4-7 of g_x and 8-11 of g_y through the central
    // differences of the target ingest (replicated borders)
    __device__ void add_tap(int q, T v) {
        const int m = q >> 2, xq = tx[q & 3], yq = ty[q & 3];
        const size_t row = (size_t)yq * W;
        if (m == 0) {
            atomicAdd(dI_t + row + xq, scaled_double(v, out_exp, out_scale));
            return;
        }
        // g = (right - left) / 2
        const int lo = m == 1 ? (int)(row + (xq > 0 ? xq - 1 : 0)) : (yq > 0 ? yq - 1 : 0) * W + xq;
        const int hi = m == 1 ? (int)(row + (xq + 1 < W ? xq + 1 : W - 1)) : (yq + 1 < H ? yq + 1 : H - 1) * W + xq;
        const double g = scaled_double(T(0.5) * v, out_exp, out_scale);
        atomicAdd(dI_t + hi, g);
        atomicAdd(dI_t + lo, -g);
    }
    __device__ void add_lamD(T v) { lamD = v; }
    __device__ void add_isD(T v) { isD = v; }
    __device__ void add_lamN(T v) { lamN = v; }
};

// neighbour of (u, v) in direction k
__device__ __forceinline__ bool neighbour(int u, int v, int k, int W, int H, int* nu, int* nv) {
    *nu = u + (k == 0 ? -1 : (k == 1 ? 1 : 0));
    *nv = v + (k == 2 ? -1 : (k == 3 ? 1 : 0));
    return *nu >= 0 && *nu < W && *nv >= 0 && *nv < H;
}

// Context of one pixel's update (geometry, weights, neighbours, decisions) and
// the I/O object's location fields; in a per-direction stage, of direction k's
// neighbour only (*has_k: there is one).
template <typename T, bool DIR>
__device__ bool pixel_context(const HwArgs<T>& A, int tile, int lane, int k, hw::PixCtx<T>& c, KernelIO<T, DIR>& io,
                              int* u_out, int* v_out, bool* has_k) {
    const Geometry<T>& g = A.g;
    const int W = g.W, H = g.H;
    const int u = (tile % g.tiles_x) * TILE_W + lane % TILE_W;
    const int v = (tile / g.tiles_x) * TILE_H + lane / TILE_W;
    *u_out = u;
    *v_out = v;
    if (u >= W || v >= H) return false;
    io.Sin = A.Sin;
    io.Ao = A.Ao;
    io.Ai = A.Ai;
    io.dI_t = A.dI_t;
    io.W = W;
    io.H = H;
    io.si = (size_t)tile * TILE_WORDS + lane;
    io.scr_in = nullptr;
    io.scr_out = nullptr;
    io.dIs = io.lamD = io.isD = io.lamN = io.amax = T(0);
    // The adjoint state is rescaled by a power of two before every pass: the
    // unrolled derivative can grow by many orders of magnitude over the sweeps,
    // beyond the float range, while the pass is linear in its input.
    if constexpr (sizeof(T) == 4)
        io.in_scale = __ldcg(&A.scale->in32);
    else
        io.in_scale = __ldcg(&A.scale->in);
    io.out_scale = __ldcg(&A.scale->out);
    io.out_exp = __ldcg(&A.scale->E32);
    c.u = T(u);
    c.v = T(v);
    c.W = W;
    c.H = H;
    c.fx = g.fx;
    c.fy = g.fy;
    c.cx = g.cx;
    c.cy = g.cy;
    c.ifx = g.ifx;
    c.ify = g.ify;
    c.d_prior = A.d_prior;
    c.lam_P = A.lam_P;
    c.lam_Z = A.lam_Z;
    c.lam_R = A.lam_R;
    c.beta = A.beta;
    c.t_huber = A.t_huber;
    c.lam_D = A.lam_D;
    c.inv_sigma_D = A.inv_sigma_D;
    c.lam_N = A.lam_N;
    int nu, nv;
    if constexpr (DIR) {
        *has_k = neighbour(u, v, k, W, H, &nu, &nv);
        io.sj[0] = *has_k ? state_index(nu, nv, g.tiles_x) : 0;
    } else {
        c.br = A.br[(size_t)tile * TILE_PX + lane];
        const size_t ii = (size_t)v * g.pitch + u;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            c.has[q] = neighbour(u, v, q, W, H, &nu, &nv);
            io.sj[q] = c.has[q] ? state_index(nu, nv, g.tiles_x) : 0;
            c.m[q] = T(0);
            if (c.has[q])
                c.m[q] = q == 0 ? A.m_x[ii - 1] : (q == 1 ? A.m_x[ii] : (q == 2 ? A.m_y[ii - g.pitch] : A.m_y[ii]));
        }
    }
    return true;
}

// Recompute check: every output of the recomputed update is compared with the
// sweep kernel's, relative to the largest of |stored|, 1, the magnitude of the
// terms it is formed from, and its block's scale, the scale of a 6 x 6 solve's
// rounding: sqrt(|A_rr A_cc|) for entry (r, c) of a symmetric positive semidefinite
// block (M_p, a message's Lambda), the largest stored entry for an entry of a
// 6-vector (xi, u, a message's eta). A stage checks what it holds anyway: fwd the
// messages' Lambda, dir their projected eta, pose what the main stage left in
// SCR_CHK. (A kernel of its own read both sides of all 151 outputs again: 41 us of
// 290 per reverse sweep at 320x240.) The largest difference goes to A.mismatch.
// (check_value divides only when the maximum grows: |y - r| > mm den decides
// it; a NaN difference never does)
template <typename T>
__device__ __forceinline__ void check_value(T yq, T s, T rq, T& mm) {
    const T den = v_abs(rq) > s ? v_abs(rq) : s;
    const T d = v_abs(yq - rq);
    if (d > mm * den) {
        const T e = d / den;
        mm = e > mm ? e : mm;
    }
}

template <typename T>
__device__ __forceinline__ T unit_scale(T y) {
    return v_abs(y) > T(1) ? v_abs(y) : T(1);
}

// a symmetric 6 x 6 block y (packed values) against the stored planes from ref
template <typename T>
__device__ __forceinline__ void check_sym(const T* y, const T* ref, T& mm) {
    T rv[21], sq[6];
#pragma unroll
    for (int q = 0; q < 21; ++q) rv[q] = __ldg(ref + q * TILE_PX);
#pragma unroll
    for (int r = 0; r < 6; ++r) sq[r] = v_sqrt(v_abs(rv[pidx(r, r)]));
#pragma unroll
    for (int r = 0; r < 6; ++r)
#pragma unroll
        for (int c = 0; c <= r; ++c) {
            const T b = sq[r] * sq[c], u = unit_scale(y[pidx(r, c)]);
            check_value(y[pidx(r, c)], b > u ? b : u, rv[pidx(r, c)], mm);
        }
}

// a 6-vector block
template <typename T>
__device__ __forceinline__ void check_vec(const T* y, const T* scale, const T* ref, T& mm) {
    T rv[6], b = T(0);
#pragma unroll
    for (int r = 0; r < 6; ++r) {
        rv[r] = __ldg(ref + r * TILE_PX);
        b = v_abs(rv[r]) > b ? v_abs(rv[r]) : b;
    }
#pragma unroll
    for (int r = 0; r < 6; ++r) check_value(y[r], scale[r] > b ? scale[r] : b, rv[r], mm);
}

// the block's largest mm to *mismatch (every thread calls it, once in a kernel per WHICH)
template <int WHICH = 0, typename T>
__device__ __forceinline__ void check_block_max(T mm, unsigned long long* mismatch) {
    __shared__ T wm[TILE_PX / 32];
    for (int o = 16; o > 0; o >>= 1) {
        const T x = __shfl_xor_sync(0xffffffffu, mm, o);
        mm = x > mm ? x : mm;
    }
    if ((threadIdx.x & 31) == 0) wm[threadIdx.x >> 5] = mm;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < TILE_PX / 32; ++w) mm = wm[w] > mm ? wm[w] : mm;
        if (mm > T(0)) atomic_max_nonneg(mismatch, double(mm));
    }
}

// Forward per-direction stage (first): block = one row of 32 pixels of a state
// tile (grid: tiles x TILE_H), four threads per pixel, one per direction
// (thread = 4 x column + k). Each recomputes the damped identity message of its
// direction, checks its Lambda, and forms its Lambda_k ybar(eta_k'); the pixel's
// four threads, adjacent lanes of one warp, sum message and product over the
// directions by shuffles and the first of them writes the sums to SCR_SUM.
template <typename T>
__global__ void __launch_bounds__(TILE_PX) k_adjoint_fwd(const HwArgs<T> A, T* __restrict__ scr) {
    pdl_wait();
    const int tile = blockIdx.x, k = threadIdx.x & 3;
    const int lane = blockIdx.y * TILE_W + (threadIdx.x >> 2);
    {  // adj_in, a quarter of the tile's words per block
        struct alignas(16) V {
            T x[16 / sizeof(T)];
        };
        constexpr int n = TILE_WORDS / TILE_H * (int)sizeof(T) / 16;
        static_assert(TILE_WORDS % (TILE_H * 16 / sizeof(T)) == 0, "whole 16-byte words");
        V* z = reinterpret_cast<V*>(A.Ai + (size_t)tile * TILE_WORDS + blockIdx.y * (TILE_WORDS / TILE_H));
        for (int i = threadIdx.x; i < n; i += TILE_PX) z[i] = V{};
    }
    KernelIO<T, true> io;
    hw::PixCtx<T> c;
    int u, v;
    bool has = false;
    const bool inside = pixel_context(A, tile, lane, k, c, io, &u, &v, &has);
    T* sp = scr + (size_t)tile * SCR_WORDS + lane;
    T L[21], e[6], w[6], mm = T(0);
    for (int q = 0; q < 21; ++q) L[q] = T(0);
    for (int q = 0; q < 6; ++q) e[q] = w[q] = T(0);
    if (inside) {
        const T* ref = A.Sout + io.si + (PL_ID + ID_STRIDE * k) * TILE_PX;
        if (has) {
            T xi[6], qi[4], t[3];
            for (int q = 0; q < 6; ++q) xi[q] = io.mu(q);
            se3_exp_q(xi, qi, t);
            hw::damped_identity_at(io, c, k, qi, t, L, e);
            hw::identity_w(io, k, L, w);
        } else {  // no neighbour: a zero message
            const T one[6] = {T(1), T(1), T(1), T(1), T(1), T(1)};
            check_vec(e, one, ref + 21 * TILE_PX, mm);
        }
        check_sym(L, ref, mm);
    }
    for (int o = 1; o < 4; o <<= 1) {
        for (int q = 0; q < 21; ++q) L[q] += __shfl_xor_sync(0xffffffffu, L[q], o);
        for (int q = 0; q < 6; ++q) {
            e[q] += __shfl_xor_sync(0xffffffffu, e[q], o);
            w[q] += __shfl_xor_sync(0xffffffffu, w[q], o);
        }
    }
    if (inside && k == 0) {
        for (int q = 0; q < 21; ++q) sp[(SCR_SUM + q) * TILE_PX] = L[q];
        for (int q = 0; q < 6; ++q) {
            sp[(SCR_SUM + 21 + q) * TILE_PX] = e[q];
            sp[(SCR_SUM + 27 + q) * TILE_PX] = w[q];
        }
    }
    check_block_max(mm, A.mismatch);
    pdl_trigger();
}

// Main stage (block = one state tile of 32 x 4 pixels, thread = one pixel):
// recomputes the pixel's update from the summed damped messages, writes the
// outputs but the identity messages' for the check, runs the reverse pass of
// everything but the identity messages and the pose's Exp, adds the adjoints it
// reaches (own normal messages, the normal-factor values read from neighbours,
// dI_s, dI_t, factor weights) and leaves the rest in the scratch.
// FP32 runs 4 blocks per SM at 128 registers: the spills that brings cost less
// than the occupancy gained (14.5 ms against 17.0 ms at 2 blocks for 30 reverse
// sweeps at 320 x 240). FP64 keeps every register it asks for.
#ifndef PV_ADJ_MAIN_BLOCKS
#define PV_ADJ_MAIN_BLOCKS 4
#endif
template <typename T>
__global__ void __launch_bounds__(TILE_PX, sizeof(T) == 4 ? PV_ADJ_MAIN_BLOCKS : 1) k_adjoint_main(const HwArgs<T> A, T* __restrict__ scr) {
    pdl_wait();
    const Geometry<T>& g = A.g;
    const int tile = blockIdx.x, lane = threadIdx.x;
    __shared__ double red[3][TILE_PX / 32];
    double sums[3] = {0.0, 0.0, 0.0};
    T amax = T(0);
    KernelIO<T, false> io;
    hw::PixCtx<T> c;
    int u, v;
    if (pixel_context(A, tile, lane, 0, c, io, &u, &v, nullptr)) {
        const int W = g.W, H = g.H;
        const size_t ii = (size_t)v * g.pitch + u;
        io.Is = A.I_s[ii];
        // the bilinear cell of the warp at the current mean, with the sweep
        // kernel's arithmetic
        {
            T xi[6], R[9], t[3];
            for (int q = 0; q < 6; ++q) xi[q] = io.mu(q);
            se3_exp(xi, R, t);
            const T z = v_exp(io.mu(6));
            const T Xs[3] = {z * (c.u - c.cx) * c.ifx, z * (c.v - c.cy) * c.ify, z};
            T Xt[3];
            mat3_vec(R, Xs, Xt);
            Xt[0] += t[0];
            Xt[1] += t[1];
            Xt[2] += t[2];
            const bool valid = (c.br & BR_VALID) != 0;
            const T iz = valid ? v_div(T(1), Xt[2]) : T(0);
            T x = c.fx * Xt[0] * iz + c.cx;
            T y = c.fy * Xt[1] * iz + c.cy;
            c.clamp_x = x < T(0) || x > T(W - 1);
            c.clamp_y = y < T(0) || y > T(H - 1);
            x = x < T(0) ? T(0) : (x > T(W - 1) ? T(W - 1) : x);
            y = y < T(0) ? T(0) : (y > T(H - 1) ? T(H - 1) : y);
            int x0 = valid ? (int)v_floor(x) : 0, y0 = valid ? (int)v_floor(y) : 0;
            x0 = min(x0, W - 1);
            y0 = min(y0, H - 1);
            const int x1 = min(x0 + 1, W - 1), y1 = min(y0 + 1, H - 1);
            c.x0 = x0;
            c.y0 = y0;
            io.tx[0] = x0;
            io.ty[0] = y0;
            io.tx[1] = x1;
            io.ty[1] = y0;
            io.tx[2] = x0;
            io.ty[2] = y1;
            io.tx[3] = x1;
            io.ty[3] = y1;
        }
        for (int q = 0; q < 4; ++q) {
            const size_t ti = (size_t)io.ty[q] * g.pitch + io.tx[q];
            io.tapv[q] = A.I_t[ti];
            io.tapv[4 + q] = A.g_x[ti];
            io.tapv[8 + q] = A.g_y[ti];
        }
        T* sp = scr + (size_t)tile * SCR_WORDS + lane;
        io.scr_in = sp;
        io.scr_out = sp;
        hw::pixel_vjp_main(io, c);
        A.dI_s[(size_t)v * W + u] += scaled_double(io.dIs, io.out_exp, io.out_scale);
        sums[0] = scaled_double(io.lamD, io.out_exp, io.out_scale);
        sums[1] = scaled_double(io.isD, io.out_exp, io.out_scale);
        sums[2] = scaled_double(io.lamN, io.out_exp, io.out_scale);
        amax = io.amax;
    }
    // the block's sums (as 384 FP64 atomics on shared memory they were a
    // compare-and-swap loop per lane)
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        if (__any_sync(0xffffffffu, sums[q] != 0.0))
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) sums[q] += __shfl_xor_sync(0xffffffffu, sums[q], o);
        if ((lane & 31) == 0) red[q][lane >> 5] = sums[q];
    }
    __syncthreads();
    if (lane < 3) {
        double x = 0.0;
        for (int w = 0; w < TILE_PX / 32; ++w) x += red[lane][w];
        if (x != 0.0) atomicAdd(A.dparam + lane, x);
    }
    check_block_max(amax, A.adj_max);
    pdl_trigger();
}

// Per-direction stage: one thread per pixel and direction (block = one state
// tile, grid.y = the direction): the damped identity message again, its projected
// eta against the stored one, the adjoint of that message, the damping's adjoint
// into the pixel's old message, the reverse pass of the message (scattering the
// neighbour's adjoints), and the pose's (R, t) adjoints added to the scratch.
// (FP32 at 4 blocks per SM, 128 registers: faster than 3 blocks at 168)
template <typename T>
__global__ void __launch_bounds__(TILE_PX, sizeof(T) == 4 ? 4 : 1) k_adjoint_dir(const HwArgs<T> A, T* __restrict__ scr) {
    pdl_wait();
    const int tile = blockIdx.x, lane = threadIdx.x, k = blockIdx.y;
    KernelIO<T, true> io;
    hw::PixCtx<T> c;
    int u, v;
    bool has = false;
    T mm = T(0), amax = T(0);
    if (pixel_context(A, tile, lane, k, c, io, &u, &v, &has) && has) {
        T* sp = scr + (size_t)tile * SCR_WORDS + lane;
        io.scr_in = sp;
        io.scr_out = sp;
        T qi[4], R[9], t[3];
        {
            T xi[6];
            for (int q = 0; q < 6; ++q) xi[q] = io.mu(q);
            se3_exp_q(xi, qi, t);
            quat_matrix(qi, R);
        }
        T tau[7];
        for (int q = 0; q < 7; ++q) tau[q] = io.main_in(hw::MO_TAU + q);
        hw::IdFwd<T> f;
        {
            T L[21], e[6], y[6], sc[6];
            hw::damped_identity_at(io, c, k, qi, t, L, e, &f);
#pragma unroll
            for (int r = 0; r < 6; ++r) {
                T Lrow[6];
                for (int q = 0; q < 6; ++q) Lrow[q] = L[pidx(r, q)];
                hw::projected_eta_row(Lrow, e[r], tau, &y[r], &sc[r]);
            }
            check_vec(y, sc, A.Sout + io.si + (PL_ID + ID_STRIDE * k + 21) * TILE_PX, mm);
        }
        T Lb[21], eb[6];
        {
            T Mpb[21], ebb[6];
            for (int q = 0; q < 21; ++q) Mpb[q] = io.main_in(hw::MO_MPB + q);
            for (int q = 0; q < 6; ++q) ebb[q] = io.main_in(hw::MO_EBB + q);
            hw::identity_msg_adjoint(io, c, k, tau, Mpb, ebb, Lb, eb);
        }
        T Rb[9], tb[3];
        for (int q = 0; q < 9; ++q) Rb[q] = T(0);
        for (int q = 0; q < 3; ++q) tb[q] = T(0);
        hw::identity_vjp(io, c, k, R, t, f, Lb, eb, Rb, tb);
        for (int q = 0; q < 9; ++q) atomicAdd(sp + (SCR_MAIN + hw::MO_RB + q) * TILE_PX, Rb[q]);
        for (int q = 0; q < 3; ++q) atomicAdd(sp + (SCR_MAIN + hw::MO_TB + q) * TILE_PX, tb[q]);
        amax = io.amax;
    }
    check_block_max(mm, A.mismatch);
    check_block_max<1>(amax, A.adj_max);
    pdl_trigger();
}

// a pass's factors: e = ilogb(max) (0 where there is none) on top of the units E
__device__ __forceinline__ void set_scale(AdjScale* s, double E, double max) {
    int e = (max > 0.0 && isfinite(max)) ? ilogb(max) : 0;
    if (e < -126) e = -126;  // 2^-e stays a float
    s->E = E + double(e);
    s->in = ldexp(1.0, -e);
    s->out = ldexp(1.0, (int)s->E);
    s->in32 = (float)s->in;
    s->E32 = (int)s->E;
}

// Pose stage (last): the pixel's xi adjoint from the (R, t) adjoints of its Exp,
// the recompute check of what the main stage left (SCR_CHK), and, by the last block,
// the next pass's factors.
template <typename T>
__global__ void __launch_bounds__(TILE_PX) k_adjoint_pose(const HwArgs<T> A, const T* __restrict__ scr) {
    pdl_wait();
    const int tile = blockIdx.x, lane = threadIdx.x;
    KernelIO<T, true> io;
    hw::PixCtx<T> c;
    int u, v;
    bool has = false;
    T mm = T(0), amax = T(0);
    if (pixel_context(A, tile, lane, 0, c, io, &u, &v, &has)) {
        io.scr_in = scr + (size_t)tile * SCR_WORDS + lane;
        T xi[6], Rb[9], tb[3], xib[6];
        for (int q = 0; q < 6; ++q) xi[q] = io.mu(q);
        for (int q = 0; q < 9; ++q) Rb[q] = io.main_in(hw::MO_RB + q);
        for (int q = 0; q < 3; ++q) tb[q] = io.main_in(hw::MO_TB + q);
        for (int q = 0; q < 6; ++q) xib[q] = io.main_in(hw::MO_XIB + q);
        hw::pose_vjp(io, xi, Rb, tb, xib, io.main_in(hw::MO_DB));
        const T* ref = A.Sout + io.si;
        auto chk = [&](int q) { return __ldcg(io.scr_in + (SCR_CHK + chk_plane(q)) * TILE_PX); };
        auto scalar = [&](int q, T y, T s) { check_value(y, s, __ldg(ref + q * TILE_PX), mm); };
        T y[21], sc[6];
        for (int q = 0; q < 21; ++q) y[q] = chk(PL_MP + q);
        check_sym(y, ref + PL_MP * TILE_PX, mm);
        for (int b = 0; b < 2; ++b) {  // xi, u
            const int q0 = b ? PL_U : PL_MU;
            for (int q = 0; q < 6; ++q) {
                y[q] = chk(q0 + q);
                sc[q] = unit_scale(y[q]);
            }
            check_vec(y, sc, ref + q0 * TILE_PX, mm);
        }
        const T dn = chk(6), sn = chk(PL_S);
        scalar(6, dn, unit_scale(dn));
        scalar(PL_S, sn, unit_scale(sn));
        for (int k = 0; k < 4; ++k) {  // normal messages: Lambda, eta (its terms' scale stored)
            const T nl = chk(PL_NM + 2 * k);
            scalar(PL_NM + 2 * k, nl, unit_scale(nl));
            scalar(PL_NM + 2 * k + 1, chk(PL_NM + 2 * k + 1), __ldcg(io.scr_in + (SCR_CHK_S + k) * TILE_PX));
        }
        amax = io.amax;
    }
    check_block_max(mm, A.mismatch);
    check_block_max<1>(amax, A.adj_max);
    if (lane == 0) {
        __threadfence();
        if (atomicAdd(A.ticket, 1u) == gridDim.x - 1) {
            __threadfence();
            set_scale(A.scale_next, __ldcg(&A.scale->E), __longlong_as_double((long long)atomicExch(A.adj_max, 0ull)));
            *A.ticket = 0u;
        }
    }
    pdl_trigger();
}

__device__ __forceinline__ void absmax_acc(float4 x, float& m) {
    absmax_acc(x.x, m);
    absmax_acc(x.y, m);
    absmax_acc(x.z, m);
    absmax_acc(x.w, m);
}
__device__ __forceinline__ void absmax_acc(double2 x, double& m) {
    absmax_acc(x.x, m);
    absmax_acc(x.y, m);
}
// max |a[i]| of the seed over finite values, in the adjoint's own precision, with
// 16-byte loads (n a multiple of 4: the adjoint state is a whole number of 128-pixel
// tiles); the last block sets the first pass's factors.
template <typename T, typename V>
__global__ void k_adjoint_absmax(const V* __restrict__ a, size_t nv, AdjScale* __restrict__ scale,
                                 unsigned long long* __restrict__ mx, unsigned* __restrict__ ticket) {
    pdl_wait();
    T m = T(0);
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < nv; i += (size_t)gridDim.x * blockDim.x)
        absmax_acc(__ldcg(a + i), m);
    for (int o = 16; o > 0; o >>= 1) {
        const T y = __shfl_xor_sync(0xffffffffu, m, o);
        m = y > m ? y : m;
    }
    if ((threadIdx.x & 31) == 0 && m > T(0)) atomic_max_nonneg(mx, double(m));
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0 && atomicAdd(ticket, 1u) == gridDim.x - 1) {
        __threadfence();
        set_scale(scale, 0.0, __longlong_as_double((long long)atomicExch(mx, 0ull)));
        *ticket = 0u;
    }
    pdl_trigger();
}

}  // namespace

// blocks for a grid-stride kernel: 8 blocks of 256 threads per SM
static int stride_blocks() {
    int sms = 0, dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return (sms > 0 ? sms : 152) * 8;
}

cudaError_t launch_adjoint_absmax(const void* a, size_t n, int adj64, AdjScale* scale, unsigned long long* max,
                                  unsigned* ticket, cudaStream_t st) {
    const dim3 blocks(stride_blocks());
    if (adj64)
        launch_pdl(k_adjoint_absmax<double, double2>, blocks, dim3(256), 0, st, static_cast<const double2*>(a), n / 2,
                   scale, max, ticket);
    else
        launch_pdl(k_adjoint_absmax<float, float4>, blocks, dim3(256), 0, st, static_cast<const float4*>(a), n / 4,
                   scale, max, ticket);
    return cudaGetLastError();
}

cudaError_t launch_adjoint_sweep(const AdjArgs& A, int blocks, cudaStream_t st) {
    k_adjoint_sweep<<<blocks, ad::ADJ_THREADS, 0, st>>>(A);
    return cudaGetLastError();
}

size_t adjoint_scratch_bytes(int n_tiles, int state64) {
    return (size_t)n_tiles * SCR_WORDS * (state64 ? sizeof(double) : sizeof(float));
}

template <typename T>
static cudaError_t launch_hw(const AdjArgs& A, int n_tiles, void* scratch, cudaStream_t st) {
    T* scr = static_cast<T*>(scratch);
    const HwArgs<T> h = hw_args<T>(A);
    launch_pdl(k_adjoint_fwd<T>, dim3(n_tiles, TILE_H), dim3(TILE_PX), 0, st, h, scr);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    launch_pdl(k_adjoint_main<T>, dim3(n_tiles), dim3(TILE_PX), 0, st, h, scr);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    launch_pdl(k_adjoint_dir<T>, dim3(n_tiles, 4), dim3(TILE_PX), 0, st, h, scr);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    launch_pdl(k_adjoint_pose<T>, dim3(n_tiles), dim3(TILE_PX), 0, st, h, scr);
    return cudaGetLastError();
}

cudaError_t launch_adjoint_hw(const AdjArgs& A, int n_tiles, void* scratch, cudaStream_t st) {
    return A.state64 ? launch_hw<double>(A, n_tiles, scratch, st) : launch_hw<float>(A, n_tiles, scratch, st);
}

cudaError_t launch_adjoint_seed(const AdjArgs& A, const double* grad_xi, const double* grad_invdepth, void* adj,
                                int adj64, cudaStream_t st) {
    dim3 block(32, 4), grid((A.g.W + 31) / 32, (A.g.H + 3) / 4);
    if (adj64)
        k_adjoint_seed<double><<<grid, block, 0, st>>>(A, grad_xi, grad_invdepth, static_cast<double*>(adj));
    else
        k_adjoint_seed<float><<<grid, block, 0, st>>>(A, grad_xi, grad_invdepth, static_cast<float*>(adj));
    return cudaGetLastError();
}

cudaError_t launch_sigma_grads(const double* dparam, double sigma_D, double sigma_N, double* out, cudaStream_t st) {
    k_sigma_grads<<<1, 1, 0, st>>>(dparam, sigma_D, sigma_N, out);
    return cudaGetLastError();
}

}  // namespace pv

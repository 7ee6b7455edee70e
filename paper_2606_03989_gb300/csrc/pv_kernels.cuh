// PixVOD sweep kernels (templated on the arithmetic type).
//
// State: structure-of-arrays planes stored tile-major: the image is cut into
// 32 x 4-pixel tiles and each tile keeps all its planes contiguously
// (plane p of the tile's pixel `lane` at tile_base + p * 128 + lane), so plane
// offsets are compile-time constants and a tile's message planes are one
// contiguous block for a bulk copy. Two buffers are ping-ponged: a sweep reads
// one and writes every plane of the other. Planes:
//   0..6     mu (xi_0..xi_5, log-depth d)
//   7..27    M_p: pose information of the belief without the photometric factor
//            (pose prior plus the four identity messages), 6x6 packed lower
//   28..33   u: photometric part of the depth-marginalised pose information,
//            P = M_p + u u^T
//   34       s: belief information of the depth with the pose marginalised
//   35+27k   identity-factor message into the pixel from slot k: Lambda (21
//            packed lower) then eta (6); slots 0 left, 1 right, 2 up, 3 down
//   143+2k   normal-integration message from slot k: Lambda, eta
//
// After every sweep the stored beliefs are projected to the new linearisation
// point, where their eta is zero; the variable-to-factor message of pixel j
// towards a pairwise factor f is then belief minus that factor's message, and
// its marginal on the factor's dims is (P_j - Lambda_{f->j}, -eta_{f->j}) for an
// identity factor and (s_j - n_{f->j}, -e_{f->j}) for a normal factor, because
// each of those messages lives on one block (pose or depth) only. P_j is kept
// as M_p + u u^T because a single pixel's rank-one photometric information can
// exceed its other pose information by more than float32 resolves.
#pragma once

#include "pv_branch.h"
#include "pv_math.cuh"

namespace pv {

constexpr int N_PLANES = 151;
constexpr int PL_MU = 0;
constexpr int PL_MP = 7;
constexpr int PL_U = 28;
constexpr int PL_S = 34;
constexpr int PL_ID = 35;
constexpr int ID_STRIDE = 27;
constexpr int PL_NM = 143;
constexpr int N_INPUT_PLANES = 6;  // I_s, I_t, g_x, g_y, m_x, m_y (row-major, pitched)
constexpr int MSG_PLANES = PL_NM - PL_ID;     // 108: the identity-message planes 35..142
constexpr int LAM = 21;                       // planes of one message's Lambda
constexpr int LAM_PLANES = 4 * LAM;           // staged through shared memory
constexpr int TILE_W = 32;
constexpr int TILE_H = 4;
constexpr int TILE_PX = TILE_W * TILE_H;
constexpr int TILE_WORDS = N_PLANES * TILE_PX;

constexpr unsigned FLAG_NONPOS_PIVOT = 0x1u;
constexpr unsigned FLAG_NONFINITE = 0x2u;
constexpr unsigned FLAG_TIMEOUT = 0x4u;
constexpr unsigned FLAG_BOUNDS = 0x10u;  // checked builds: an index left its buffer (access skipped)

// Checked builds (PIXVOD_CHECKED): every computed index of the sweep (neighbour
// state, input planes, bilinear taps, shared-memory message slots) is tested
// against its buffer; a violation sets FLAG_BOUNDS in *flags and yields
// `fallback` (0) so the access is skipped. Plain builds compile the index as is.
#ifdef PIXVOD_CHECKED
#define PV_IDX(idx, limit, flags) (((size_t)(idx) < (size_t)(limit)) ? (size_t)(idx) : ((flags) |= FLAG_BOUNDS, (size_t)0))
#else
#define PV_IDX(idx, limit, flags) ((size_t)(idx))
#endif

// Device-resident per-handle scalars (doubles, fixed layout; the checkpoint
// format copies the first 40).
struct Scalars {
    double xi_est[6];
    double T_kf[16];   // T_kf<-world
    double T_cur[16];  // T_cam<-world of the last frame
    double d_prior;    // log-depth prior mean of the current keyframe segment
    double d_mean;     // mean log-depth after the last reduction
    unsigned flags;
    unsigned counter;  // last-block ticket of the reduction
    unsigned qt_clear;   // quadtree: sweeps whose buffer k_qt_clear still has to clear, after a load
    unsigned qt_ticket;  // blocks of k_qt_clear that have read it
    double pad[5];
};

template <typename T>
struct Geometry {
    int W, H, pitch;   // input planes: row-major with `pitch` elements per row
    size_t plane;      // elements per input plane
    int tiles_x;       // state: tiles per tile row
    T fx, fy, cx, cy, ifx, ify;
};

// element offset of pixel (u, v) in a tile-major state buffer (plane 0)
__host__ __device__ __forceinline__ size_t state_index(int u, int v, int tiles_x) {
    return (size_t)((v / TILE_H) * tiles_x + (u / TILE_W)) * TILE_WORDS + (v % TILE_H) * TILE_W + (u % TILE_W);
}

template <typename T>
struct Factors {
    T lam_D, inv_sigma_D, t_huber, lam_P, lam_R, lam_N, lam_Z, beta;
};

template <typename T>
struct SweepArgs {
    Geometry<T> g;
    Factors<T> f;
    const T* __restrict__ in;
    T* __restrict__ out;
    const T* __restrict__ I_s;
    const T* __restrict__ I_t;
    const T* __restrict__ g_x;
    const T* __restrict__ g_y;
    const T* __restrict__ m_x;
    const T* __restrict__ m_y;
    Scalars* sc;
    // when set, each pixel's discrete decisions of this sweep (BR_* bits) are
    // written here (tile-major pixel index), for the adjoint
    unsigned char* br;
};


// Programmatic dependent launch: a kernel launched with the attribute may start
// while its predecessor in the stream drains; pdl_wait returns when the
// predecessor has completed and its writes are visible, pdl_trigger lets the
// successor's blocks take the slots that this grid leaves free.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// ---------------------------------------------------------------------------
// a0: frame ingest
// ---------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ void normal_slopes(const float* __restrict__ n, int u, int v, const Geometry<T>& g,
                                              T* ax, T* ay) {
    T nx = T(n[0]), ny = T(n[1]), nz = T(n[2]);
    T nr = nx * (T(u) - g.cx) / g.fx + ny * (T(v) - g.cy) / g.fy + nz;
    bool ok = v_abs(nr) >= T(1e-3);
    *ax = ok ? nx / (g.fx * nr) : T(0);
    *ay = ok ? ny / (g.fy * nr) : T(0);
}

// Keyframe: source intensities and the normal-integration edge measurements of
// Eq. 6 (m_x between (u, v) and (u+1, v), m_y between (u, v) and (u, v+1)).
template <typename T>
__device__ __forceinline__ void ingest_keyframe_px(const Geometry<T>& g, const float* __restrict__ frame,
                                                   const float* __restrict__ normals, T* I_s, T* m_x, T* m_y,
                                                   int u, int v) {
    size_t i = (size_t)v * g.pitch + u;
    size_t f = (size_t)v * g.W + u;
    I_s[i] = T(frame[f]);
    T ax, ay;
    normal_slopes(normals + 3 * f, u, v, g, &ax, &ay);
    T mx = T(0), my = T(0);
    if (u + 1 < g.W) {
        T bx, by;
        normal_slopes(normals + 3 * (f + 1), u + 1, v, g, &bx, &by);
        mx = T(0.5) * (ax + bx);
    }
    if (v + 1 < g.H) {
        T bx, by;
        normal_slopes(normals + 3 * (f + g.W), u, v + 1, g, &bx, &by);
        my = T(0.5) * (ay + by);
    }
    m_x[i] = mx;
    m_y[i] = my;
}

template <typename T>
__global__ void k_ingest_keyframe(Geometry<T> g, const float* __restrict__ frame,
                                  const float* __restrict__ normals, T* I_s, T* m_x, T* m_y) {
    pdl_wait();
    int u = blockIdx.x * blockDim.x + threadIdx.x;
    int v = blockIdx.y * blockDim.y + threadIdx.y;
    if (u >= g.W || v >= g.H) return;
    ingest_keyframe_px(g, frame, normals, I_s, m_x, m_y, u, v);
}

// Target: intensities and central-difference gradients (replicated borders).
template <typename T>
__device__ __forceinline__ void ingest_target_px(const Geometry<T>& g, const float* __restrict__ frame, T* I_t,
                                                 T* g_x, T* g_y, int u, int v) {
    size_t i = (size_t)v * g.pitch + u;
    const float* row = frame + (size_t)v * g.W;
    int ul = u > 0 ? u - 1 : 0, ur = u + 1 < g.W ? u + 1 : g.W - 1;
    int vu = v > 0 ? v - 1 : 0, vd = v + 1 < g.H ? v + 1 : g.H - 1;
    I_t[i] = T(row[u]);
    g_x[i] = T(0.5) * (T(row[ur]) - T(row[ul]));
    g_y[i] = T(0.5) * (T(frame[(size_t)vd * g.W + u]) - T(frame[(size_t)vu * g.W + u]));
}

template <typename T>
__global__ void k_ingest_target(Geometry<T> g, const float* __restrict__ frame, T* I_t, T* g_x, T* g_y) {
    pdl_wait();
    int u = blockIdx.x * blockDim.x + threadIdx.x;
    int v = blockIdx.y * blockDim.y + threadIdx.y;
    if (u >= g.W || v >= g.H) return;
    ingest_target_px(g, frame, I_t, g_x, g_y, u, v);
}

// Keyframe reset: identity pose, log-depth at the segment's prior mean, no
// messages, belief equal to the priors (M_p = lam_P I, u = 0, s = lam_Z).
template <typename T>
__device__ __forceinline__ void reset_px(const Geometry<T>& g, const Factors<T>& f, T* state, const Scalars* sc,
                                         int u, int v) {
    T* st = state + state_index(u, v, g.tiles_x);
    T d0 = T(sc->d_prior);
    for (int p = 0; p < N_PLANES; ++p) st[p * TILE_PX] = T(0);
    st[6 * TILE_PX] = d0;
#pragma unroll
    for (int k = 0; k < 6; ++k) st[(PL_MP + pidx(k, k)) * TILE_PX] = f.lam_P;
    st[PL_S * TILE_PX] = f.lam_Z;
}

// Checked builds: the lanes of ragged tiles that lie outside the image hold NaN
// in every plane, so that any computation reading them shows as FLAG_NONFINITE.
template <typename T>
__global__ void k_poison_outside(Geometry<T> g, int n_tiles, T* state) {
    const int tile = blockIdx.x, lane = threadIdx.x;
    const int u = (tile % g.tiles_x) * TILE_W + lane % TILE_W;
    const int v = (tile / g.tiles_x) * TILE_H + lane / TILE_W;
    if (tile >= n_tiles || (u < g.W && v < g.H)) return;
    T* st = state + (size_t)tile * TILE_WORDS + lane;
    for (int p = 0; p < N_PLANES; ++p) st[p * TILE_PX] = T(NAN);
}

template <typename T>
__global__ void k_reset(Geometry<T> g, Factors<T> f, T* state, const Scalars* sc) {
    pdl_wait();
    int u = blockIdx.x * blockDim.x + threadIdx.x;
    int v = blockIdx.y * blockDim.y + threadIdx.y;
    if (u >= g.W || v >= g.H) return;
    reset_px(g, f, state, sc, u, v);
}

// ---------------------------------------------------------------------------
// a1-a4: one synchronous sweep (v1: one thread per pixel, global loads)
// ---------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ T bilinear(const T* __restrict__ img, int pitch, int x0, int y0, int x1, int y1,
                                      T ax, T ay) {
    T a = img[(size_t)y0 * pitch + x0], b = img[(size_t)y0 * pitch + x1];
    T c = img[(size_t)y1 * pitch + x0], d = img[(size_t)y1 * pitch + x1];
    return (T(1) - ay) * ((T(1) - ax) * a + ax * b) + ay * ((T(1) - ax) * c + ax * d);
}

// ---------------------------------------------------------------------------
// bulk (TMA) copies global -> shared with an mbarrier, in inline PTX
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
// dst, src and bytes must be multiples of 16 bytes
__device__ __forceinline__ void bulk_copy_g2s(void* dst, const void* src, unsigned bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, unsigned parity) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return done != 0;
}
// bounded wait for phase `parity`; false if it did not complete
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, unsigned parity) {
    for (int it = 0; it < (1 << 22); ++it)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

// Loads of the swept state bypass L1 (ld.global.cg): the persistent batched
// kernel reads, after a grid barrier, data other SMs wrote in the same launch,
// and an SM's L1 is not kept coherent with those writes. Only for memory that the
// calling thread has not itself written with plain stores: __ldcg is inline assembly
// without a memory clobber, so nothing orders it behind them.
template <typename T>
__device__ __forceinline__ T ld_state(const T* p) {
    return __ldcg(p);
}
// A product that no addition after it is fused with (the sweep by tiles and by rows
// then round alike)
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
// Store of the new state; STREAM: marked to leave L2 first (st.global.cs)
template <bool STREAM, typename T>
__device__ __forceinline__ void st_state(T* p, T x) {
    if (STREAM) __stcs(p, x);
    else *p = x;
}

// Thread block of the sweep kernel: one state tile (32 x 4 pixels), one thread
// per pixel; 4 blocks per SM (43 KB of shared memory and at most 128 registers
// each). What a tile waits on is memory latency (at 640x480 about 34 of the 46
// thousand clocks that it took; DRAM at 47 % and no pipe above 30), so loads are
// issued early and together and the register file holds as many pixels as it can:
//  - the four messages' Lambda are bulk-copied into shared memory, damped in place
//    and bulk-copied out; M_p is summed from there after the loop instead of in 21
//    registers through it. Their eta (24 of 108 planes) go straight to and from
//    global memory: the old ones load with the neighbour's values, the new ones
//    come back for the tangent projection under the mean update's arithmetic.
//    (All 108 planes staged, M_p in registers: 89.1 against 86.4 us per sweep at
//    640x480, 850 against 814 us at 2048x1536.)
//  - the photometric factor comes first, its taps loading under the bulk copy
//    (after the loop: 90.9 against 89.1 us, 886 against 850 us).
// Five blocks per SM at 96 registers were slower (96.1 us, 936 us): the spills and
// a larger working set in L2 cost more than the extra warps hide. The identity
// loop is not unrolled; the normal messages are computed in a loop of their own.
constexpr int SWEEP_BX = TILE_W;
constexpr int SWEEP_BY = TILE_H;
constexpr int SWEEP_THREADS = TILE_PX;

template <typename T>
constexpr size_t sweep_smem_bytes() {
    return sizeof(T) * LAM_PLANES * TILE_PX;
}

// a1: photometric factor (Eqs. 2, 3) of pixel (u, v), input-plane index i, at the
// mean (qi, t, d)
template <typename T, typename Args>
__device__ __forceinline__ void photometric_factor(const Args& a, int i, int u, int v, const T* qi, const T* t,
                                                   T d, T* J, T& alpha, T& rph, unsigned char& br, unsigned& flags) {
    const Geometry<T>& g = a.g;
    const Factors<T>& F = a.f;
    const size_t n_plane = g.plane;
    (void)n_plane;
    (void)flags;
    alpha = T(0);
    rph = T(0);
    br = 0;
#pragma unroll
    for (int q = 0; q < 7; ++q) J[q] = T(0);
    {
        T R[9];
        quat_matrix(qi, R);
        T z = v_exp(d);
        T Xs[3] = {z * (T(u) - g.cx) * g.ifx, z * (T(v) - g.cy) * g.ify, z};
        T Xt[3];
        mat3_vec(R, Xs, Xt);
        Xt[0] += t[0];
        Xt[1] += t[1];
        Xt[2] += t[2];
        T Z = Xt[2];
        bool valid = Z > T(1e-6);
        T iz = valid ? v_div(T(1), Z) : T(0);
        T x = g.fx * Xt[0] * iz + g.cx;
        T y = g.fy * Xt[1] * iz + g.cy;
        // overlap test with a 1e-3 px margin (pixels warped by the identity land on
        // the border exactly); the sample point is clamped into the image
        valid = valid && (x >= T(-1e-3)) && (x <= T(g.W - 1) + T(1e-3)) && (y >= T(-1e-3)) &&
                (y <= T(g.H - 1) + T(1e-3));
        T r = T(0), gx = T(0), gy = T(0);
        if (valid) {
            x = x < T(0) ? T(0) : (x > T(g.W - 1) ? T(g.W - 1) : x);
            y = y < T(0) ? T(0) : (y > T(g.H - 1) ? T(g.H - 1) : y);
            int x0 = (int)v_floor(x), y0 = (int)v_floor(y);
            x0 = min(x0, g.W - 1);
            y0 = min(y0, g.H - 1);
            int x1 = min(x0 + 1, g.W - 1), y1 = min(y0 + 1, g.H - 1);
#ifdef PIXVOD_CHECKED
            if (x0 < 0 || y0 < 0 || (size_t)y1 * g.pitch + x1 >= n_plane) {
                flags |= FLAG_BOUNDS;
                x0 = y0 = x1 = y1 = 0;
            }
#endif
            T ax = x - T(x0), ay = y - T(y0);
            T It = bilinear(a.I_t, g.pitch, x0, y0, x1, y1, ax, ay);
            gx = bilinear(a.g_x, g.pitch, x0, y0, x1, y1, ax, ay);
            gy = bilinear(a.g_y, g.pitch, x0, y0, x1, y1, ax, ay);
            r = a.I_s[i] - It;
            valid = v_finite(r) && v_finite(gx) && v_finite(gy);
        }
        if (valid) {
            // dr/dX_t = -(gx, gy) d(pi)/dX_t
            T a0 = -gx * g.fx * iz, a1 = -gy * g.fy * iz;
            T a2 = (gx * g.fx * Xt[0] + gy * g.fy * Xt[1]) * iz * iz;
            T av[3] = {a0, a1, a2}, b[3];
            mat3T_vec(R, av, b);  // b = R^T a
            J[0] = Xs[1] * b[2] - Xs[2] * b[1];
            J[1] = Xs[2] * b[0] - Xs[0] * b[2];
            J[2] = Xs[0] * b[1] - Xs[1] * b[0];
            J[3] = b[0];
            J[4] = b[1];
            J[5] = b[2];
            J[6] = b[0] * Xs[0] + b[1] * Xs[1] + b[2] * Xs[2];
            T M = v_abs(r) * F.inv_sigma_D;
            const bool hub = M > F.t_huber;
            T w = hub ? v_div(T(2) * F.t_huber * M - F.t_huber * F.t_huber, M * M) : T(1);
            alpha = w * F.lam_D;
            rph = r;
            br = hub ? (BR_VALID | BR_HUBER) : BR_VALID;
        }
    }
}

// The neighbour of (u, v) in direction k (left, right, up, down)
template <typename T>
__device__ __forceinline__ bool sweep_neighbour(const Geometry<T>& g, int u, int v, int k, int* un, int* vn) {
    *un = u + (k == 0 ? -1 : (k == 1 ? 1 : 0));
    *vn = v + (k == 2 ? -1 : (k == 3 ? 1 : 0));
    return *un >= 0 && *un < g.W && *vn >= 0 && *vn < g.H;
}

// a2/a3: the identity message from the neighbour in direction k, its state at Sj.
// Its variable-to-factor marginal is V = W + u u^T with W = M_p,j - Lambda_{f->j}
// (pose prior plus j's three other identity messages), u = u_j and eta_v =
// -eta_{f->j}. All loads (also the old eta of the pixel's message, eo) are issued
// ahead of the Exp/Log chain of the residual, so that their latency overlaps it.
template <typename T>
__device__ __forceinline__ void sweep_message(const T* Si, const T* Sj, int k, const T* qi, const T* t, T lam_R,
                                              IdMsg<T>& m, T* eo, unsigned& flags) {
    const T* mj = Sj + (PL_ID + ID_STRIDE * (k ^ 1)) * TILE_PX;
    T W[21], uj[6], gv[6], xj[6];
#pragma unroll
    for (int q = 0; q < 6; ++q) xj[q] = ld_state(Sj + q * TILE_PX);
#pragma unroll
    for (int q = 0; q < 21; ++q) W[q] = ld_state(Sj + (PL_MP + q) * TILE_PX) - ld_state(mj + q * TILE_PX);
#pragma unroll
    for (int q = 0; q < 6; ++q) {
        uj[q] = ld_state(Sj + (PL_U + q) * TILE_PX);
        gv[q] = -ld_state(mj + (LAM + q) * TILE_PX);
    }
#pragma unroll
    for (int q = 0; q < 6; ++q) eo[q] = ld_state(Si + (PL_ID + ID_STRIDE * k + LAM + q) * TILE_PX);
    T rb[6];
    se3_between(xj, qi, t, rb);
    if (!identity_msg(W, uj, gv, rb, lam_R, m)) flags |= FLAG_NONPOS_PIVOT;
}

// a3': the normal-integration message (Eq. 6: r_i = d_i - d_j + sg m) from the
// neighbour in direction k, its state at Sj
template <typename T>
__device__ __forceinline__ void sweep_normal(const SweepArgs<T>& a, const T* Si, const T* Sj, int k, int i, T d, T* nl,
                                             T* ne, unsigned& flags) {
    const Geometry<T>& g = a.g;
    const Factors<T>& F = a.f;
    const T beta = F.beta, omb = T(1) - F.beta;
    const size_t n_plane = g.plane;
    (void)n_plane;
    (void)flags;
    const int ko = k ^ 1;
    T dj = ld_state(Sj + 6 * TILE_PX);
    T sv = ld_state(Sj + PL_S * TILE_PX) - ld_state(Sj + (PL_NM + 2 * ko) * TILE_PX);
    T evn = -ld_state(Sj + (PL_NM + 2 * ko + 1) * TILE_PX);
    T m = k == 0 ? a.m_x[PV_IDX(i - 1, n_plane, flags)]
                 : (k == 1 ? a.m_x[i] : (k == 2 ? a.m_y[PV_IDX(i - g.pitch, n_plane, flags)] : a.m_y[i]));
    T sg = (k == 0 || k == 2) ? T(1) : T(-1);
    T rn = d - dj + sg * m;
    T den = v_div(T(1), F.lam_N + sv);
    *nl = omb * (F.lam_N * sv * den) + beta * ld_state(Si + (PL_NM + 2 * k) * TILE_PX);
    *ne = omb * (F.lam_N * (evn - sv * rn) * den) + beta * ld_state(Si + (PL_NM + 2 * k + 1) * TILE_PX);
}

// a4: the mean update tau from the belief
//   Lambda_b = blockdiag(M_p, m_d) + alpha J J^T,  eta_b = eta_o - alpha r J
// (identity messages and the pose prior act on the pose block, normal messages
// and the depth prior on the depth, the photometric factor is rank one), which is
// kept in that form: M_p (packed), m_d, alpha, J, r and eta_o (in eb). qv: q below.
template <typename T>
__device__ __forceinline__ void belief_update(const T* Mp, T md, const T* eb, const T* J, T alpha, T rph, T* tau, T& qv,
                                              unsigned char& br, unsigned& flags) {
    // With B = blockdiag(M_p, m_d), h = B^-1 eta_o and z = B^-1 J, Sherman-Morrison
    // gives tau = Lambda_b^-1 eta_b = h - z alpha (r + J^T h) / (1 + alpha J^T z),
    // and the marginals of Lambda_b are, with q = J_p^T M_p^-1 J_p,
    //   P = M_p + u u^T,  u = sqrt(alpha m_d / (m_d + alpha J_d^2)) J_p,
    //   s = m_d + alpha J_d^2 / (1 + alpha q),
    // all free of cancellation.
    bool ok;
    {
        T Lp[21], idp[6];
#pragma unroll
        for (int q = 0; q < 21; ++q) Lp[q] = Mp[q];
        ok = chol_packed<6>(Lp, idp);
        T up[6], gp[6];
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            up[q] = J[q];
            gp[q] = eb[q];
        }
        fwd_solve<6>(Lp, idp, up);
        bwd_solve<6>(Lp, idp, up);
        fwd_solve<6>(Lp, idp, gp);
        bwd_solve<6>(Lp, idp, gp);
        T jh = T(0);
        qv = T(0);
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            qv += J[q] * up[q];
            jh += J[q] * gp[q];
        }
        const T imd = v_div(T(1), md);
        const T hd = eb[6] * imd;
        const T zd = J[6] * imd;
        const T coef = v_div(alpha * (rph + jh + J[6] * hd), T(1) + alpha * (qv + J[6] * zd));
#pragma unroll
        for (int q = 0; q < 6; ++q) tau[q] = gp[q] - coef * up[q];
        tau[6] = hd - coef * zd;
    }
    bool fin = true;
#pragma unroll
    for (int q = 0; q < 7; ++q) fin = fin && v_finite(tau[q]);
    if (!ok) flags |= FLAG_NONPOS_PIVOT;
    if (!ok || !fin) {
        if (!fin) flags |= FLAG_NONFINITE;
        br |= BR_SKIP;
#pragma unroll
        for (int q = 0; q < 7; ++q) tau[q] = T(0);
    }
}

// The belief's marginals besides M_p: u = sb J_p (the photometric part of the
// depth-marginalised pose information) and s (pose-marginalised depth information)
template <typename T>
__device__ __forceinline__ void depth_marginals(T md, T alpha, T Jd, T qv, T* sb, T* s) {
    const T bp = v_div(alpha * md, md + alpha * Jd * Jd);
    *sb = v_sqrt(bp);
    *s = md + v_div(alpha * Jd * Jd, T(1) + alpha * qv);
}

// The calling thread's pixel of the sweep over tile (tx, ty): everything but the
// store of the identity messages' Lambda, which are left in `msg`. False if the
// tile's bulk copy never arrived (FLAG_TIMEOUT is set).
template <bool STREAM, typename T>
__device__ __forceinline__ bool sweep_pixel(const SweepArgs<T>& a, int tx, int ty, T* msg, uint64_t* bar,
                                            unsigned parity) {
    const int tid = threadIdx.y * SWEEP_BX + threadIdx.x;
    const int u = tx * SWEEP_BX + threadIdx.x;
    const int v = ty * SWEEP_BY + threadIdx.y;
    const Geometry<T>& g = a.g;
    const Factors<T>& F = a.f;
    const size_t tile = (size_t)ty * g.tiles_x + tx;
    if (u >= g.W || v >= g.H) return true;
    unsigned flags = 0;
    const size_t n_state = (size_t)g.tiles_x * ((g.H + TILE_H - 1) / TILE_H) * TILE_WORDS;
    (void)n_state;
    const int i = (int)PV_IDX(v * g.pitch + u, g.plane, flags);
    const T* __restrict__ Si = a.in + PV_IDX(tile * TILE_WORDS + tid, n_state, flags);   // this pixel, plane 0
    T* __restrict__ Di = a.out + PV_IDX(tile * TILE_WORDS + tid, n_state, flags);

    T xi[6], d;
#pragma unroll
    for (int k = 0; k < 6; ++k) xi[k] = ld_state(Si + k * TILE_PX);
    d = ld_state(Si + 6 * TILE_PX);
    T qi[4], t[3];
    se3_exp_q(xi, qi, t);
    // --- priors (Eq. 4 with identity Jacobian; log-depth prior) ---
    T eb[7];
#pragma unroll
    for (int k = 0; k < 6; ++k) eb[k] = -mul_rn(F.lam_P, xi[k]);
    T md = F.lam_Z;
    eb[6] = -mul_rn(F.lam_Z, d - T(a.sc->d_prior));

    T alpha, rph, J[7];
    unsigned char br;
    photometric_factor(a, i, u, v, qi, t, d, J, alpha, rph, br, flags);

    if (!mbar_wait_bounded(bar, parity)) {
        // the tile's messages never arrived: flag it, wait once more, leave the tile
        atomicOr(&a.sc->flags, FLAG_TIMEOUT);
        mbar_wait_bounded(bar, parity);
        return false;
    }
    const T beta = F.beta, omb = T(1) - F.beta;
#pragma unroll 1
    for (int k = 0; k < 4; ++k) {
        T* mb = msg + PV_IDX((k * LAM) * TILE_PX + tid, (LAM_PLANES - LAM + 1) * TILE_PX, flags);  // slot k's Lambda
        T* me = Di + (PL_ID + ID_STRIDE * k + LAM) * TILE_PX;                                      // its eta
        int un, vn;
        if (!sweep_neighbour(g, u, v, k, &un, &vn)) {
#pragma unroll
            for (int q = 0; q < LAM; ++q) mb[q * TILE_PX] = T(0);
#pragma unroll
            for (int q = 0; q < 6; ++q) me[q * TILE_PX] = T(0);
            continue;
        }
        T eo[6];
        IdMsg<T> m;
        sweep_message(Si, a.in + PV_IDX(state_index(un, vn, g.tiles_x), n_state, flags), k, qi, t, F.lam_R, m, eo,
                      flags);
        // damped: (1 - beta) new + beta old; Lambda over the old one in shared memory
        const T wl = omb * F.lam_R, wll = wl * F.lam_R;
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            const T e = v_fma(wl, m.he[q], beta * eo[q]);
            eb[q] += e;
            me[q * TILE_PX] = e;
        }
#pragma unroll
        for (int c = 0; c < 6; ++c)
#pragma unroll
            for (int r = c; r < 6; ++r)
                mb[pidx(r, c) * TILE_PX] = m.lambda(r, c, wl, wll, beta * mb[pidx(r, c) * TILE_PX]);
    }
    // M_p from the four messages in shared memory
    T Mp[21];
#pragma unroll
    for (int q = 0; q < 21; ++q) {
        T x = T(0);
#pragma unroll
        for (int k = 0; k < 6; ++k)
            if (q == pidx(k, k)) x = F.lam_P;
#pragma unroll
        for (int k = 0; k < 4; ++k) x += msg[PV_IDX((LAM * k + q) * TILE_PX + tid, LAM_PLANES * TILE_PX, flags)];
        Mp[q] = x;
    }
    T nl[4], ne[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        nl[k] = T(0);
        ne[k] = T(0);
        int un, vn;
        if (!sweep_neighbour(g, u, v, k, &un, &vn)) continue;
        sweep_normal(a, Si, a.in + PV_IDX(state_index(un, vn, g.tiles_x), n_state, flags), k, i, d, &nl[k], &ne[k],
                     flags);
        md += nl[k];
        eb[6] += ne[k];
    }
    T tau[7], qv;
    belief_update(Mp, md, eb, J, alpha, rph, tau, qv, br, flags);
    if (a.br) a.br[tile * TILE_PX + tid] = br;
    // the new eta, back for the projection below: plain loads, which the compiler keeps
    // behind the loop's stores (__ldcg does not say that it reads memory)
    T en[24];
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int q = 0; q < 6; ++q) en[6 * k + q] = Di[(PL_ID + ID_STRIDE * k + LAM + q) * TILE_PX];
    // mu <- mu (+) tau
    {
        T xn[6];
        se3_update(qi, t, tau, xn);
#pragma unroll
        for (int q = 0; q < 6; ++q) st_state<STREAM>(&Di[q * TILE_PX], xn[q]);
        st_state<STREAM>(&Di[6 * TILE_PX], d + tau[6]);
    }
    {
        T sb, s;
        depth_marginals(md, alpha, J[6], qv, &sb, &s);
#pragma unroll
        for (int q = 0; q < 21; ++q) st_state<STREAM>(&Di[(PL_MP + q) * TILE_PX], Mp[q]);
#pragma unroll
        for (int q = 0; q < 6; ++q) st_state<STREAM>(&Di[(PL_U + q) * TILE_PX], sb * J[q]);
        st_state<STREAM>(&Di[PL_S * TILE_PX], s);
    }
    // messages, projected: eta <- eta - Lambda tau
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        st_state<STREAM>(&Di[(PL_NM + 2 * k) * TILE_PX], nl[k]);
        st_state<STREAM>(&Di[(PL_NM + 2 * k + 1) * TILE_PX], ne[k] - nl[k] * tau[6]);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const T* mb = msg + PV_IDX((k * LAM) * TILE_PX + tid, (LAM_PLANES - LAM + 1) * TILE_PX, flags);
#pragma unroll
        for (int r = 0; r < 6; ++r) {
            T e = en[6 * k + r];
#pragma unroll
            for (int c = 0; c < 6; ++c) e -= mb[pidx(r, c) * TILE_PX] * tau[c];
            st_state<STREAM>(&Di[(PL_ID + ID_STRIDE * k + LAM + r) * TILE_PX], e);
        }
    }
    if (flags) atomicOr(&a.sc->flags, flags);
    return true;
}

// The same sweep over row `row` of tile (tx, ty), for images of few tiles: the
// block's warp k computes the messages of direction k for the row's 32 pixels, the
// four are summed through shared memory in the same order, and every warp stores
// its direction's messages and its share of the rest. A tile's latency is one
// direction's instead of four in turn, on four times as many SMs; that every warp
// solves the belief costs nothing while the schedulers are idle. Per sweep, by
// tiles and by rows: 64x48 10.5 and 5.5 us, 128x96 10.9 and 6.9, 160x120 12.6 and
// 8.5, 224x160 15.0 and 14.8, 256x192 17.3 and 19.6; FP64, bound by its pipe: 64x48
// 122 and 49, 128x96 123 and 168. Every thread of the block must call it; the caller
// synchronises the block before `msg` is reused.
constexpr int ROW_VALUES = 29;  // a direction's Lambda, eta and normal message in shared memory
constexpr int ROW_SLOTS = 4 * ROW_VALUES * TILE_W;
static_assert(ROW_SLOTS <= LAM_PLANES * TILE_PX, "the rows' values fit the sweep's shared memory");
template <typename T>
__device__ __forceinline__ void sweep_row(const SweepArgs<T>& a, int tx, int ty, int row, T* msg, bool last_sweep) {
    const int k = threadIdx.y, x = threadIdx.x;
    const int u = tx * TILE_W + x, v = ty * TILE_H + row;
    const Geometry<T>& g = a.g;
    const Factors<T>& F = a.f;
    if (v >= g.H) return;  // the whole block
    const size_t tile = (size_t)ty * g.tiles_x + tx;
    const bool inside = u < g.W;
    unsigned flags = 0;
    const size_t n_state = (size_t)g.tiles_x * ((g.H + TILE_H - 1) / TILE_H) * TILE_WORDS;
    (void)n_state;
    const int lane = row * TILE_W + x;
    const int i = inside ? (int)PV_IDX(v * g.pitch + u, g.plane, flags) : 0;
    const T* __restrict__ Si = a.in + PV_IDX(tile * TILE_WORDS + lane, n_state, flags);
    T* __restrict__ Di = a.out + PV_IDX(tile * TILE_WORDS + lane, n_state, flags);
    T* sh = msg + PV_IDX(k * ROW_VALUES * TILE_W + x, ROW_SLOTS - (ROW_VALUES - 1) * TILE_W, flags);  // this direction's values
    T xi[6], d = T(0), qi[4], t[3];
    T alpha = T(0), rph = T(0), J[7];
    unsigned char br = 0;
    if (inside) {
        T l[LAM], e[6], nl = T(0), ne = T(0);
#pragma unroll
        for (int q = 0; q < 6; ++q) xi[q] = ld_state(Si + q * TILE_PX);
        d = ld_state(Si + 6 * TILE_PX);
#pragma unroll
        for (int q = 0; q < LAM; ++q) l[q] = ld_state(Si + (PL_ID + ID_STRIDE * k + q) * TILE_PX);  // the old Lambda
        se3_exp_q(xi, qi, t);
        int un, vn;
        if (sweep_neighbour(g, u, v, k, &un, &vn)) {
            const T beta = F.beta, omb = T(1) - F.beta;
            const T* Sj = a.in + PV_IDX(state_index(un, vn, g.tiles_x), n_state, flags);
            sweep_normal(a, Si, Sj, k, i, d, &nl, &ne, flags);
            T eo[6];
            IdMsg<T> m;
            sweep_message(Si, Sj, k, qi, t, F.lam_R, m, eo, flags);
            const T wl = omb * F.lam_R, wll = wl * F.lam_R;
#pragma unroll
            for (int q = 0; q < 6; ++q) e[q] = v_fma(wl, m.he[q], beta * eo[q]);
#pragma unroll
            for (int c = 0; c < 6; ++c)
#pragma unroll
                for (int r = c; r < 6; ++r) l[pidx(r, c)] = m.lambda(r, c, wl, wll, beta * l[pidx(r, c)]);
        } else {
#pragma unroll
            for (int q = 0; q < LAM; ++q) l[q] = T(0);
#pragma unroll
            for (int q = 0; q < 6; ++q) e[q] = T(0);
        }
#pragma unroll
        for (int q = 0; q < LAM; ++q) sh[q * TILE_W] = l[q];
#pragma unroll
        for (int q = 0; q < 6; ++q) sh[(LAM + q) * TILE_W] = e[q];
        sh[27 * TILE_W] = nl;
        sh[28 * TILE_W] = ne;
        photometric_factor(a, i, u, v, qi, t, d, J, alpha, rph, br, flags);
    }
    __syncthreads();
    if (last_sweep) pdl_trigger();
    if (!inside) return;
    const unsigned mflags = flags;  // this direction's
    T Mp[21], eb[7], md = F.lam_Z;
#pragma unroll
    for (int q = 0; q < 21; ++q) {
        T y = T(0);
#pragma unroll
        for (int j = 0; j < 6; ++j)
            if (q == pidx(j, j)) y = F.lam_P;
#pragma unroll
        for (int j = 0; j < 4; ++j) y += msg[PV_IDX((j * ROW_VALUES + q) * TILE_W + x, ROW_SLOTS, flags)];
        Mp[q] = y;
    }
#pragma unroll
    for (int q = 0; q < 6; ++q) eb[q] = -mul_rn(F.lam_P, xi[q]);
    eb[6] = -mul_rn(F.lam_Z, d - T(a.sc->d_prior));
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const T* sj = msg + PV_IDX(j * ROW_VALUES * TILE_W + x, ROW_SLOTS - (ROW_VALUES - 1) * TILE_W, flags);
#pragma unroll
        for (int q = 0; q < 6; ++q) eb[q] += sj[(LAM + q) * TILE_W];
        md += sj[27 * TILE_W];
        eb[6] += sj[28 * TILE_W];
    }
    T tau[7], qv;
    belief_update(Mp, md, eb, J, alpha, rph, tau, qv, br, flags);
    T* Dk = Di + (PL_ID + ID_STRIDE * k) * TILE_PX;
    {
        T l[LAM];
#pragma unroll
        for (int q = 0; q < LAM; ++q) {
            l[q] = sh[q * TILE_W];
            Dk[q * TILE_PX] = l[q];
        }
#pragma unroll
        for (int r = 0; r < 6; ++r) {
            T y = sh[(LAM + r) * TILE_W];
#pragma unroll
            for (int c = 0; c < 6; ++c) y -= l[pidx(r, c)] * tau[c];
            Dk[(LAM + r) * TILE_PX] = y;
        }
        const T nl = sh[27 * TILE_W];
        Di[(PL_NM + 2 * k) * TILE_PX] = nl;
        Di[(PL_NM + 2 * k + 1) * TILE_PX] = sh[28 * TILE_W] - nl * tau[6];
    }
    if (k == 0) {
        T xn[6];
        se3_update(qi, t, tau, xn);
#pragma unroll
        for (int q = 0; q < 6; ++q) Di[q * TILE_PX] = xn[q];
        Di[6 * TILE_PX] = d + tau[6];
        if (a.br) a.br[tile * TILE_PX + lane] = br;
    } else if (k == 1) {
        T sb, s;
        depth_marginals(md, alpha, J[6], qv, &sb, &s);
#pragma unroll
        for (int q = 0; q < 6; ++q) Di[(PL_U + q) * TILE_PX] = sb * J[q];
        Di[PL_S * TILE_PX] = s;
    } else {
#pragma unroll
        for (int q = 0; q < 21; ++q)
            if ((q < 10) == (k == 2)) Di[(PL_MP + q) * TILE_PX] = Mp[q];
    }
    const unsigned fl = k == 0 ? flags : mflags;
    if (fl) atomicOr(&a.sc->flags, fl);
}

// shared -> global bulk copy by the calling thread, part of its current bulk
// group; dst, src and bytes must be multiples of 16 bytes
__device__ __forceinline__ void bulk_copy_s2g(void* dst, const void* src, unsigned bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(smem_u32(src)),
                 "r"(bytes)
                 : "memory");
}
// Wait for the group. In a launch's last sweep only the reads of shared memory are
// waited for (the end of the kernel completes the writes); before a grid barrier,
// until the writes are complete and ordered before the thread's later
// generic-proxy accesses.
__device__ __forceinline__ void bulk_wait_s2g(bool last_sweep) {
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
    if (last_sweep) {
        asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
    } else {
        asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
        asm volatile("fence.proxy.async.global;" ::: "memory");
    }
}

// One synchronous sweep over one state tile (tx, ty) by the calling block (every
// thread of the block must call it). The block must have initialised `bar` (one
// arrival); `parity` is the phase this tile's bulk copy completes. The caller
// synchronises the block before reusing `msg` for another tile. The message
// Lambda planes of pixels outside the image are copied through unchanged. Returns
// false (to every thread) when the tile's bulk copy did not arrive within the
// bounded wait: nothing of the tile was stored, FLAG_TIMEOUT is set, and the
// block must take no further tile in this launch.
template <bool STREAM, typename T>
__device__ __forceinline__ bool sweep_tile(const SweepArgs<T>& a, int tx, int ty, T* msg, uint64_t* bar,
                                           unsigned parity, bool last_sweep) {
    const int tid = threadIdx.y * SWEEP_BX + threadIdx.x;
    const size_t tile = (size_t)ty * a.g.tiles_x + tx;
    constexpr unsigned bytes = sizeof(T) * LAM * TILE_PX;  // one message's Lambda planes
    if (tid == 0) {
        // order earlier generic-proxy accesses (global stores of a previous sweep in
        // the same launch, shared-memory use of a previous tile) before the async copy
        asm volatile("fence.proxy.async;" ::: "memory");
        mbar_expect_tx(bar, 4 * bytes);
        for (int k = 0; k < 4; ++k)
            bulk_copy_g2s(msg + LAM * k * TILE_PX, a.in + tile * TILE_WORDS + (PL_ID + ID_STRIDE * k) * TILE_PX, bytes,
                          bar);
    }
    const bool ok = sweep_pixel<STREAM>(a, tx, ty, msg, bar, parity);
    // the messages written to shared memory (generic proxy) are read by
    // the bulk copy (async proxy): fence, then gather the block; a tile whose
    // messages never arrived is not stored
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    const bool all_ok = __syncthreads_and(ok);
    if (last_sweep) pdl_trigger();
    if (all_ok && tid == 0) {
        for (int k = 0; k < 4; ++k)
            bulk_copy_s2g(a.out + tile * TILE_WORDS + (PL_ID + ID_STRIDE * k) * TILE_PX, msg + LAM * k * TILE_PX, bytes);
        bulk_wait_s2g(last_sweep);
    }
    return all_ok;
}

// ---------------------------------------------------------------------------
// a5: pose average (App. C.2) and keyframe anchoring, one launch, fixed order
// ---------------------------------------------------------------------------
constexpr int RED_THREADS = TILE_PX;

// FP64 runs at 1/64 of the FP32 rate here, and the reduction's additions bound it
// (640x480: 35 of them per thread in a butterfly of all seven sums took 50 us cold).
// So a block adds up several tiles per thread first, a float is widened by its bits,
// and the butterfly halves the number of sums a lane holds at each step.
__device__ __forceinline__ double widen(float x) {
    const int b = __float_as_int(x), e = (b >> 23) & 0xff;
    if (e == 0 || e == 0xff) return double(x);
    return __hiloint2double((b & 0x80000000) | ((e + 896) << 20) | ((b & 0x7fffff) >> 3), b << 29);
}
__device__ __forceinline__ double widen(double x) { return x; }

// Seven sums over the block's threads, in a fixed order (shuffles within a warp,
// then the warps in order): thread q of the block gets sum q (q < 7, others 0).
__device__ __forceinline__ double block_sum7(const double* r, double (*sh)[RED_THREADS / 32]) {
    const int lane = threadIdx.x & 31;
    const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4;
    double v[4], w[2];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const double lo = r[q], hi = q < 3 ? r[q + 4] : 0.0;
        v[q] = (b4 ? hi : lo) + __shfl_xor_sync(0xffffffffu, b4 ? lo : hi, 16);
    }
#pragma unroll
    for (int q = 0; q < 2; ++q)
        w[q] = (b3 ? v[q + 2] : v[q]) + __shfl_xor_sync(0xffffffffu, b3 ? v[q] : v[q + 2], 8);
    double x = (b2 ? w[1] : w[0]) + __shfl_xor_sync(0xffffffffu, b2 ? w[0] : w[1], 4);
    x += __shfl_xor_sync(0xffffffffu, x, 2);
    x += __shfl_xor_sync(0xffffffffu, x, 1);
    const int q = lane >> 2;  // the sum this lane holds
    __syncthreads();          // sh may still be read from an earlier sum
    if ((lane & 3) == 0 && q < 7) sh[q][threadIdx.x >> 5] = x;
    __syncthreads();
    double y = 0.0;
    if (threadIdx.x < 7) {
        y = sh[threadIdx.x][0];
#pragma unroll
        for (int k = 1; k < RED_THREADS / 32; ++k) y += sh[threadIdx.x][k];
    }
    return y;
}

// Tiles that one block of the reduction adds up: as many as make at most one wave
// of blocks at 4 on each of 152 SMs. A constant on every device: it sets the order of
// the sums.
__host__ __device__ constexpr int reduce_group(int n_tiles) { return (n_tiles + 607) / 608; }

// The block of group `group` sums its tiles' 7 mean planes (double accumulation,
// fixed order); the last block to finish sums the groups' partials in order,
// writes xi_est and the mean log-depth, composes T_cur = Exp(xi_est) T_kf and,
// at an anchoring frame, moves the keyframe: T_kf <- T_cur, d_prior <- d_mean.
template <typename T>
__device__ __forceinline__ void reduce_tiles(const Geometry<T>& g, const T* __restrict__ state,
                                             double* __restrict__ partials, Scalars* sc, int anchor, int group,
                                             int n_tiles) {
    __shared__ double sh[7][RED_THREADS / 32];
    __shared__ bool last;
    const int tid = threadIdx.x;
    const int per = reduce_group(n_tiles), n_groups = (n_tiles + per - 1) / per;
    const int end = min((group + 1) * per, n_tiles);
    double r[7] = {0, 0, 0, 0, 0, 0, 0};
#pragma unroll 4
    for (int tile = group * per; tile < end; ++tile) {
        const int u = (tile % g.tiles_x) * TILE_W + tid % TILE_W;
        const int v = (tile / g.tiles_x) * TILE_H + tid / TILE_W;
        if (u < g.W && v < g.H) {
            const T* st = state + (size_t)tile * TILE_WORDS + tid;
#pragma unroll
            for (int q = 0; q < 7; ++q) r[q] += widen(st[q * TILE_PX]);
        }
    }
    double y = block_sum7(r, sh);
    if (tid < 7) {
        partials[group * 7 + tid] = y;
        __threadfence();
    }
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        last = atomicAdd(&sc->counter, 1u) == (unsigned)(n_groups - 1);
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
#pragma unroll
    for (int q = 0; q < 7; ++q) r[q] = 0.0;
#pragma unroll 5
    for (int h = tid; h < n_groups; h += RED_THREADS)
#pragma unroll
        for (int q = 0; q < 7; ++q) r[q] += __ldcg(partials + h * 7 + q);
    y = block_sum7(r, sh);
    if (tid < 32)
#pragma unroll
        for (int q = 0; q < 7; ++q) r[q] = __shfl_sync(0xffffffffu, y, q);
    if (tid == 0) {
        const double n = double(g.W) * double(g.H);
        double xi[6], R[9], t[3];
        for (int q = 0; q < 6; ++q) {
            xi[q] = r[q] / n;
            sc->xi_est[q] = xi[q];
        }
        sc->d_mean = r[6] / n;
        se3_exp(xi, R, t);
        // T_cur = Exp(xi_est) T_kf with Exp(xi_est) = [R t; 0 1]
        double Tc[16];
        for (int c = 0; c < 4; ++c) {
            for (int r2 = 0; r2 < 3; ++r2)
                Tc[4 * r2 + c] = R[3 * r2] * sc->T_kf[c] + R[3 * r2 + 1] * sc->T_kf[4 + c] +
                                 R[3 * r2 + 2] * sc->T_kf[8 + c] + t[r2] * sc->T_kf[12 + c];
            Tc[12 + c] = sc->T_kf[12 + c];
        }
        for (int q = 0; q < 16; ++q) sc->T_cur[q] = Tc[q];
        if (anchor) {
            for (int q = 0; q < 16; ++q) sc->T_kf[q] = Tc[q];
            sc->d_prior = sc->d_mean;
        }
        sc->counter = 0;
    }
}

template <typename T>
__global__ void __launch_bounds__(RED_THREADS) k_reduce(Geometry<T> g, const T* __restrict__ state,
                                                        double* __restrict__ partials, Scalars* sc,
                                                        int anchor, int n_tiles) {
    pdl_wait();
    reduce_tiles(g, state, partials, sc, anchor, blockIdx.x, n_tiles);
}

// Depth output: exp(sign * mu_6) as dense float32.
template <typename T>
__global__ void k_depth_out(Geometry<T> g, const T* __restrict__ state, float* out, T sign) {
    pdl_wait();
    int u = blockIdx.x * blockDim.x + threadIdx.x;
    int v = blockIdx.y * blockDim.y + threadIdx.y;
    if (u >= g.W || v >= g.H) return;
    out[(size_t)v * g.W + u] = float(v_exp(sign * state[state_index(u, v, g.tiles_x) + 6 * TILE_PX]));
}

}  // namespace pv

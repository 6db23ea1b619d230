// Particle-in-cell kernels: CIC field gather on the Yee grid, relativistic Boris
// push, move with reflecting walls, and charge-conserving Esirkepov current
// deposition into shared-memory tiles (arXiv 2510.11174, Methodology: PIC
// macro-particles weighted by density-volume fraction, advanced by the Boris
// pusher; particles crossing a domain boundary have their velocity reversed;
// charge conservation is checked at every step).
//
// Data layout: particles of a species live in fixed-capacity tiles of T^3
// cells, SoA FP32 (x, y, z in cell units; u = gamma*beta; weight).  One CTA
// owns one tile: it stages E and B of the tile plus a one-node halo in shared
// memory, pushes every particle of every species in the tile, accumulates J in
// a shared-memory frame of (T+3)^3 nodes (halo 1 below, 2 above, which holds
// every node an Esirkepov stencil of a particle that started in the tile can
// touch) in 64-bit fixed point (frames.cuh), and writes that frame to a
// per-tile scratch slab.  A second kernel sums, for every node, the frames
// that cover it in a fixed order, so J is assembled without global atomics and
// repeats bit for bit whatever order the particles and warps take.
// Particles that left their tile are copied to a migration buffer and
// re-inserted by the rebin kernel; vacated slots are compacted afterwards.
//
// Boris (relativistic, Birdsall & Langdon):
//   u- = u + (q dt/2m) E;  t = (q dt/2m gamma-) B;  s = 2t/(1+t.t)
//   u' = u- + u- x t;  u+ = u- + u' x s;  u_new = u+ + (q dt/2m) E
// Esirkepov, CIC shape, on the 3-node window that holds both shapes:
//   W_x = DS_x (S0_y S0_z + DS_y S0_z/2 + S0_y DS_z/2 + DS_y DS_z/3) (cyclic),
//   J_x(i+1/2) - J_x(i-1/2) = -q w W_x / (dt dy dz).
#include "frames.cuh"
#include "hyb_internal.cuh"
#include "ionize.cuh"
#include "philox.cuh"
#include "qed.cuh"
#include "particles.cuh"
#include "push_shape.h"

#include <cooperative_groups.h>

#include <mutex>
#include <type_traits>

namespace hyb {

namespace cg = cooperative_groups;

// field frame edge: a shape of order k gathers from k nodes below the tile to k - 1 above it
__host__ __device__ constexpr int frame_F(int T, int order = 1) { return T + 2 * order; }

static constexpr int PUSH_Q = 32;          // entries of a per-warp queue of cell-crossing particles

__host__ __device__ constexpr size_t align16(size_t b) { return (b + 15) & ~(size_t)15; }

// the current frame (3 components, 64-bit fixed point), the fields, the
// per-warp queues (two of PUSH_Q entries of two float4), the species
constexpr size_t push_smem_bytes(int T, int order, int nsp) {
    const int F = frame_F(T, order), G = frame_G(T, order);
    return align16(sizeof(unsigned long long) * 3 * (size_t)G * G * G) + align16(sizeof(float) * 6 * (size_t)F * F * F) +
           sizeof(float4) * (push_threads(T) / 32) * 4 * PUSH_Q + sizeof(SpDev) * (size_t)nsp;
}
// push_ctas() of them fit an SM's 228 KB with every species loaded (1 KB a CTA is
// the system's, 1 KB holds the kernel's static arrays)
constexpr bool push_fits(int T, int order) {
    return (push_smem_bytes(T, order, HYB_MAX_SPECIES) + 2048) * push_ctas(T, order) <= 228 * 1024;
}
static_assert(push_fits(8, 1) && push_fits(8, 2) && push_fits(4, 1) && push_fits(4, 2), "push_ctas");

// CIC base index and weight of one axis on the integer (i) and the
// half-integer (h) grid, relative to the frame origin o (global node index of
// local 0); fl = floor(p)
struct AxisW {
    int li, lh;
    float fi, fh;
};

__device__ __forceinline__ AxisW axis_weights(const GridDev &g, int a, float p, float fl, int o) {
    AxisW r;
    if (g.bc[a]) fl = fminf(fl, (float)(g.n[a] - 2));  // particle on the top wall
    r.li = (int)fl - o;
    r.fi = p - fl;
    // floor(p - 1/2) is the cell below when p lies in the lower half of its cell
    const bool low = r.fi < 0.5f;
    r.lh = r.li - (low ? 1 : 0);
    r.fh = r.fi + (low ? 0.5f : -0.5f);
    return r;
}

// trilinear interpolation as seven linear interpolations (x, then y, then z)
template <int F>
__device__ __forceinline__ float interp8(const float *__restrict__ f, int bx, int by, int bz, float fx, float fy,
                                         float fz) {
    const float *r00 = f + (bz * F + by) * F + bx;   // rows (y, z), (y + 1, z), (y, z + 1), (y + 1, z + 1)
    const float *r10 = r00 + F, *r01 = r00 + F * F, *r11 = r01 + F;
    const float a00 = fmaf(fx, r00[1] - r00[0], r00[0]);
    const float a10 = fmaf(fx, r10[1] - r10[0], r10[0]);
    const float a01 = fmaf(fx, r01[1] - r01[0], r01[0]);
    const float a11 = fmaf(fx, r11[1] - r11[0], r11[0]);
    const float b0 = fmaf(fy, a10 - a00, a00);
    const float b1 = fmaf(fy, a11 - a01, a01);
    return fmaf(fz, b1 - b0, b0);
}

// Boris (relativistic, Birdsall & Langdon), h = q dt / 2m
__device__ __forceinline__ void boris_push(float h, const float e[3], const float b[3], float u[3]) {
    float um[3], tt[3], ss[3], ud[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) um[c] = u[c] + h * e[c];
    const float gm = sqrtf(1.0f + um[0] * um[0] + um[1] * um[1] + um[2] * um[2]);
#pragma unroll
    for (int c = 0; c < 3; ++c) tt[c] = h * b[c] * (1.0f / gm);
    const float t2 = tt[0] * tt[0] + tt[1] * tt[1] + tt[2] * tt[2];
    const float s2 = 2.0f / (1.0f + t2);
#pragma unroll
    for (int c = 0; c < 3; ++c) ss[c] = tt[c] * s2;
    ud[0] = um[0] + (um[1] * tt[2] - um[2] * tt[1]);
    ud[1] = um[1] + (um[2] * tt[0] - um[0] * tt[2]);
    ud[2] = um[2] + (um[0] * tt[1] - um[1] * tt[0]);
    u[0] = um[0] + (ud[1] * ss[2] - ud[2] * ss[1]) + h * e[0];
    u[1] = um[1] + (ud[2] * ss[0] - ud[0] * ss[2]) + h * e[1];
    u[2] = um[2] + (ud[0] * ss[1] - ud[1] * ss[0]) + h * e[2];
}

// the implicit rotation of the Vay and Higuera-Cary pushers: w turned about
// tau = h B with the Lorentz factor of the result,
//   gamma^2 = (sigma + sqrt(sigma^2 + 4 (tau^2 + (w.tau)^2))) / 2, sigma = 1 + w^2 - tau^2,
//   t = tau / gamma, s = 1 / (1 + t^2), R(w) = s (w + (w.t) t + w x t)
__device__ __forceinline__ void rotate_implicit(const float w[3], const float tau[3], float out[3], float t[3]) {
    const float w2 = w[0] * w[0] + w[1] * w[1] + w[2] * w[2];
    const float tau2 = tau[0] * tau[0] + tau[1] * tau[1] + tau[2] * tau[2];
    const float us = w[0] * tau[0] + w[1] * tau[1] + w[2] * tau[2];
    const float sigma = 1.0f + w2 - tau2;
    const float g = sqrtf(0.5f * (sigma + sqrtf(sigma * sigma + 4.0f * (tau2 + us * us))));
    const float ig = 1.0f / g;
#pragma unroll
    for (int c = 0; c < 3; ++c) t[c] = tau[c] * ig;
    const float s = 1.0f / (1.0f + t[0] * t[0] + t[1] * t[1] + t[2] * t[2]);
    const float wt = w[0] * t[0] + w[1] * t[1] + w[2] * t[2];
    out[0] = s * (w[0] + wt * t[0] + (w[1] * t[2] - w[2] * t[1]));
    out[1] = s * (w[1] + wt * t[1] + (w[2] * t[0] - w[0] * t[2]));
    out[2] = s * (w[2] + wt * t[2] + (w[0] * t[1] - w[1] * t[0]));
}

// Vay (Phys. Plasmas 15, 056701, 2008): w = u + h (2E + v x B), u_new = R(w)
__device__ __forceinline__ void vay_push(float h, const float e[3], const float b[3], float u[3]) {
    const float ig = 1.0f / sqrtf(1.0f + u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
    const float tau[3] = {h * b[0], h * b[1], h * b[2]};
    const float v[3] = {u[0] * ig, u[1] * ig, u[2] * ig};
    const float w[3] = {u[0] + 2.0f * h * e[0] + (v[1] * tau[2] - v[2] * tau[1]),
                        u[1] + 2.0f * h * e[1] + (v[2] * tau[0] - v[0] * tau[2]),
                        u[2] + 2.0f * h * e[2] + (v[0] * tau[1] - v[1] * tau[0])};
    float t[3];
    rotate_implicit(w, tau, u, t);
}

// Higuera & Cary (Phys. Plasmas 24, 052104, 2017): w = u + h E, u+ = R(w),
// u_new = u+ + h E + u+ x t
__device__ __forceinline__ void higuera_cary_push(float h, const float e[3], const float b[3], float u[3]) {
    const float tau[3] = {h * b[0], h * b[1], h * b[2]};
    const float w[3] = {u[0] + h * e[0], u[1] + h * e[1], u[2] + h * e[2]};
    float up[3], t[3];
    rotate_implicit(w, tau, up, t);
    u[0] = up[0] + h * e[0] + (up[1] * t[2] - up[2] * t[1]);
    u[1] = up[1] + h * e[1] + (up[2] * t[0] - up[0] * t[2]);
    u[2] = up[2] + h * e[2] + (up[0] * t[1] - up[1] * t[0]);
}

// Esirkepov deposit of a particle that stays in its cell.  Per axis the shape
// is (1 - f, f) on the cell's two nodes, f moving from f0 to f1 = f0 + d; W_c
// is nonzero only on the cell's lower c-face, at its 2 x 2 transverse nodes,
// where the transverse factor is the mean of S_p S_q along the straight path:
// with m = (f0 + f1) / 2, int f_p f_q = m_p m_q + d_p d_q / 12 = X, and the
// other three nodes take m_q - X, m_p - X and 1 - m_p - m_q + X.
// fac[c] = q w jfac_c 2^k; the current is fac[c] (S1 - S0)(lower node) = -fac[c] d_c.
template <int G>
__device__ __forceinline__ void deposit_same_cell(unsigned *__restrict__ sj, const float x0[3], const float x1[3],
                                                  const float fl[3], const int o[3], const float fac[3]) {
    constexpr int G3 = G * G * G;
    int lb[3];
    float m[3], d[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        lb[a] = (int)fl[a] - o[a];
        const float f0 = x0[a] - fl[a], f1 = x1[a] - fl[a];
        d[a] = f1 - f0;
        m[a] = 0.5f * (f0 + f1);
    }
    const int base = (lb[2] * G + lb[1]) * G + lb[0];
    constexpr int off[3] = {1, G, G * G};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        if (d[c] == 0.0f) continue;  // particles at rest
        const int pa = (c + 1) % 3, qa = (c + 2) % 3;
        const float X = fmaf(d[pa] * d[qa], 1.0f / 12.0f, m[pa] * m[qa]);
        const float v01 = m[qa] - X, v10 = m[pa] - X;
        const float v00 = (1.0f - m[pa]) - v01;
        const float sc = -fac[c] * d[c];
        const int J = c * G3 + base;
        const int idx[4] = {J, J + off[pa], J + off[qa], J + off[pa] + off[qa]};
        const float val[4] = {sc * v00, sc * v10, sc * v01, sc * X};
        fix_add<4, false>(sj, 3 * G3, idx, val);
    }
}

__device__ __forceinline__ int sel3(int a, int v0, int v1, int v2) { return a == 0 ? v0 : (a == 1 ? v1 : v2); }
__device__ __forceinline__ float sel3(int a, float v0, float v1, float v2) { return a == 0 ? v0 : (a == 1 ? v1 : v2); }

// transverse factor S0p (S0q + DSq/2) + DSp (S0q/2 + DSq/3) of Esirkepov's W
__device__ __forceinline__ float esirkepov_cross(float s0p, float dsp, float s0q, float dsq) {
    const float ca = fmaf(0.5f, dsq, s0q);
    const float cb = fmaf(1.0f / 3.0f, dsq, 0.5f * s0q);
    return fmaf(dsp, cb, s0p * ca);
}

// Esirkepov deposit of a particle that crossed a cell face along one axis c
// only, the commonest crossing by far: three nodes along c, two along the
// others, so 8 + 6 + 6 currents instead of the 54 slots of the full window.
// The queue holds its coordinates rotated to (c, p, q) with the axis, so every
// lane of the warp runs the same straight code on its own strides.
template <int G>
__device__ __forceinline__ void deposit_one_crossing(unsigned *__restrict__ sj, const float4 A, const float4 B,
                                                     const int o[3], const float jfac[3]) {
    constexpr int G3 = G * G * G;
    const int c = __float_as_int(B.w);
    const int sc = sel3(c, 1, G, G * G), sp = sel3(c, G, G * G, 1), sq = sel3(c, G * G, 1, G);
    const float gc = fminf(floorf(A.x), floorf(B.x)), gp = floorf(A.y), gq = floorf(A.z);
    const int base = ((int)gc - sel3(c, o[0], o[1], o[2])) * sc + ((int)gp - sel3(c, o[1], o[2], o[0])) * sp +
                     ((int)gq - sel3(c, o[2], o[0], o[1])) * sq;
    float s0c[3], dc[3], s0p[2], dp[2], s0q[2], dq[2];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        s0c[k] = fmaxf(1.0f - fabsf(A.x - (gc + k)), 0.0f);
        dc[k] = fmaxf(1.0f - fabsf(B.x - (gc + k)), 0.0f) - s0c[k];
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        s0p[k] = 1.0f - fabsf(A.y - (gp + k));
        dp[k] = 1.0f - fabsf(B.y - (gp + k)) - s0p[k];
        s0q[k] = 1.0f - fabsf(A.z - (gq + k));
        dq[k] = 1.0f - fabsf(B.z - (gq + k)) - s0q[k];
    }
    const int Jc = base + c * G3, Jp = base + sel3(c, 1, 2, 0) * G3, Jq = base + sel3(c, 2, 0, 1) * G3;
    const float fc = A.w * sel3(c, jfac[0], jfac[1], jfac[2]), fp = A.w * sel3(c, jfac[1], jfac[2], jfac[0]),
                fq = A.w * sel3(c, jfac[2], jfac[0], jfac[1]);
#pragma unroll
    for (int bq = 0; bq < 2; ++bq) {
        int idx[4];
        float val[4];
#pragma unroll
        for (int bp = 0; bp < 2; ++bp) {
            const float w = esirkepov_cross(s0p[bp], dp[bp], s0q[bq], dq[bq]);
            float acc = 0.0f;
#pragma unroll
            for (int a = 0; a < 2; ++a) {
                acc += dc[a] * w;
                idx[bp * 2 + a] = Jc + a * sc + bp * sp + bq * sq;
                val[bp * 2 + a] = fc * acc;
            }
        }
        fix_add<4, false>(sj, 3 * G3, idx, val);
    }
    {
        // along p: transverse axes q (two nodes) and c (three)
        int idx[6];
        float val[6];
#pragma unroll
        for (int bc = 0; bc < 3; ++bc)
#pragma unroll
            for (int bq = 0; bq < 2; ++bq) {
                idx[bc * 2 + bq] = Jp + bc * sc + bq * sq;
                val[bc * 2 + bq] = fp * (dp[0] * esirkepov_cross(s0q[bq], dq[bq], s0c[bc], dc[bc]));
            }
        fix_add<6, false>(sj, 3 * G3, idx, val);
    }
    {
        // along q: transverse axes c (three nodes) and p (two)
        int idx[6];
        float val[6];
#pragma unroll
        for (int bp = 0; bp < 2; ++bp)
#pragma unroll
            for (int bc = 0; bc < 3; ++bc) {
                idx[bp * 3 + bc] = Jq + bc * sc + bp * sp;
                val[bp * 3 + bc] = fq * (dq[0] * esirkepov_cross(s0c[bc], dc[bc], s0p[bp], dp[bp]));
            }
        fix_add<6, false>(sj, 3 * G3, idx, val);
    }
}

// Esirkepov deposit on the window of W nodes of each axis that holds both
// shapes (W = 3 linear: particles that crossed faces along several axes; W = 4
// quadratic): W_c = DS_c (S0_p S0_q + DS_p S0_q / 2 + S0_p DS_q / 2 + DS_p
// DS_q / 3), prefix-summed along c.  The loop over c is not unrolled (the
// arrays rotate instead): straight-line code for every slot overruns the
// instruction cache, which was the largest stall of the push.
template <int G, int W, bool SKIP>
__device__ __forceinline__ void deposit_window(unsigned *__restrict__ sj, float S0[3][W], float DS[3][W],
                                               const int lb[3], float qw, const float jfac[3]) {
    constexpr int G3 = G * G * G;
    int base = (lb[2] * G + lb[1]) * G + lb[0];
    int s[3] = {1, G, G * G};
    float f[3] = {qw * jfac[0], qw * jfac[1], qw * jfac[2]};
#pragma unroll 1
    for (int c = 0; c < 3; ++c) {
#pragma unroll
        for (int bq = 0; bq < W; ++bq) {
            int idx[W * (W - 1)];
            float val[W * (W - 1)];
#pragma unroll
            for (int bp = 0; bp < W; ++bp) {
                const float w = esirkepov_cross(S0[1][bp], DS[1][bp], S0[2][bq], DS[2][bq]);
                float acc = 0.0f;
#pragma unroll
                for (int a = 0; a < W - 1; ++a) {
                    acc += DS[0][a] * w;
                    idx[bp * (W - 1) + a] = base + a * s[0] + bp * s[1] + bq * s[2];
                    val[bp * (W - 1) + a] = f[0] * acc;
                }
            }
            fix_add<W *(W - 1), SKIP>(sj, 3 * G3, idx, val);
        }
        base += G3;
        const int s0 = s[0];
        const float f0 = f[0];
        s[0] = s[1]; s[1] = s[2]; s[2] = s0;
        f[0] = f[1]; f[1] = f[2]; f[2] = f0;
#pragma unroll
        for (int k = 0; k < W; ++k) {
            const float a0 = S0[0][k], d0 = DS[0][k];
            S0[0][k] = S0[1][k]; S0[1][k] = S0[2][k]; S0[2][k] = a0;
            DS[0][k] = DS[1][k]; DS[1][k] = DS[2][k]; DS[2][k] = d0;
        }
    }
}

template <int G>
__device__ __forceinline__ void deposit_general(unsigned *__restrict__ sj, const float x0[3], const float x1[3],
                                                const int o[3], float qw, const float jfac[3]) {
    int lb[3];
    float S0[3][3], DS[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float gb = fminf(floorf(x0[a]), floorf(x1[a]));
        lb[a] = (int)gb - o[a];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            S0[a][k] = fmaxf(1.0f - fabsf(x0[a] - (gb + k)), 0.0f);
            DS[a][k] = fmaxf(1.0f - fabsf(x1[a] - (gb + k)), 0.0f) - S0[a][k];
        }
    }
    deposit_window<G, 3, true>(sj, S0, DS, lb, qw, jfac);
}

// Quadratic (TSC) shape: S(d) = 3/4 - d^2 (|d| <= 1/2), (3/2 - |d|)^2 / 2
// (1/2 <= |d| <= 3/2), 0 beyond
__device__ __forceinline__ float tsc(float d) {
    const float a = fabsf(d);
    const float b = 1.5f - a;
    return a <= 0.5f ? 0.75f - a * a : (a <= 1.5f ? 0.5f * b * b : 0.0f);
}

// TSC weights of one axis around the node nearest to s (staggering already
// removed): local index of the first of the three nodes and their weights
__device__ __forceinline__ void tsc_axis(float s, int o, int &l, float w[3]) {
    const float m = floorf(s + 0.5f);
    const float d = s - m;                 // in [-1/2, 1/2)
    l = (int)m - 1 - o;
    const float a = 0.5f - d, c = 0.5f + d;
    w[0] = 0.5f * a * a;
    w[1] = 0.75f - d * d;
    w[2] = 0.5f * c * c;
}

template <int F>
__device__ __forceinline__ float interp27(const float *__restrict__ f, int bx, int by, int bz, const float wx[3],
                                          const float wy[3], const float wz[3]) {
    float acc = 0.0f;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        float row = 0.0f;
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const float *r = f + ((bz + c) * F + by + b) * F + bx;
            row = fmaf(wy[b], fmaf(wx[2], r[2], fmaf(wx[1], r[1], wx[0] * r[0])), row);
        }
        acc = fmaf(wz[c], row, acc);
    }
    return acc;
}

// Esirkepov with the quadratic shape.  W = 3: a particle whose nearest node
// stays the same on every axis keeps its three nodes (54 currents); W = 4: the
// 4-node window that holds the old and the new support (144 slots, most of them
// 0).  Base = the smaller nearest node, minus one.
template <int G, int W>
__device__ __forceinline__ void deposit_quadratic(unsigned *__restrict__ sj, const float4 A, const float4 B,
                                                  const int o[3], const float jfac[3]) {
    const float x0[3] = {A.x, A.y, A.z}, x1[3] = {B.x, B.y, B.z};
    int lb[3];
    float S0[3][W], DS[3][W];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float gb = fminf(floorf(x0[a] + 0.5f), floorf(x1[a] + 0.5f)) - 1.0f;
        lb[a] = (int)gb - o[a];
#pragma unroll
        for (int k = 0; k < W; ++k) {
            S0[a][k] = tsc(x0[a] - (gb + k));
            DS[a][k] = tsc(x1[a] - (gb + k)) - S0[a][k];
        }
    }
    deposit_window<G, W, W == 4>(sj, S0, DS, lb, A.w, jfac);
}

// A warp's queue of crossing particles, 32 entries in shared memory: `n` of
// them are taken (warp-uniform).  The lanes in `want` append; a full queue is
// handed to `flush` with every lane of the warp holding one entry.  The entries
// that did not fit go in before `flush` runs, so that their eight values are dead
// in its long code: held across it (and with eight sums of the one-axis stencil
// in flight instead of four) they made the compiler spill the next particle's
// prefetched values, and a spill waits for the load it stores -- every particle
// pass then paid the memory latency the prefetch is there to hide.  One launch,
// 15.7 M particles at rest 623 -> 439 us, slow (|u| ~ 1e-3, hardly any crossing)
// 678 -> 501 us, thermal 881 -> 727 us.
template <class F>
__device__ __forceinline__ void queue_put(float4 *qa, int &n, bool want, const float4 A, const float4 B, int lane,
                                          F flush) {
    float4 *qb = qa + PUSH_Q;
    const unsigned m = __ballot_sync(0xffffffffu, want);
    if (m == 0u) return;
    const int pos = n + __popc(m & ((1u << lane) - 1u));
    if (want && pos < PUSH_Q) {
        qa[pos] = A;
        qb[pos] = B;
    }
    n += __popc(m);
    if (n >= PUSH_Q) {
        __syncwarp();
        const float4 ea = qa[lane], eb = qb[lane];
        __syncwarp();
        n -= PUSH_Q;
        if (want && pos >= PUSH_Q) {
            qa[pos - PUSH_Q] = A;
            qb[pos - PUSH_Q] = B;
        }
        flush(ea, eb);
    }
}

// The stochastic events of the push, out of line: a step has few of them, and
// their code (random numbers, table searches, the writes of new particles) in
// the particle loop costs every warp instruction cache and registers (a carbon
// slab of 1.8 M particles with all three events, three runs side by side, with the
// tallies straight to shared memory: five steps 2024 -> 1905 us).
static __device__ __noinline__ void event_spawn(const SpDev *d, float x, float y, float z, float ux, float uy, float uz,
                                                float w, uint64_t id, int dest, long long step, uint32_t seed, float tau,
                                                int *status) {
    const float xs[3] = {x, y, z}, us[3] = {ux, uy, uz};
    spawn(*d, xs, us, w, id, dest, step, seed, tau, status);
}

// Photon emission of particle `id` (species si; new position x, momentum u,
// Lorentz factor gl).  Returns the factor on its momentum, its next optical
// depth and the photon's energy where no photon particle is made (0 otherwise).
static __device__ __noinline__ float3 event_emit(const SpDev *sps, int si, const QedDev *qd, float chi, float gl, float x,
                                                 float y, float z, float ux, float uy, float uz, float w, uint64_t id,
                                                 int dest, long long step, uint32_t seed, int *status) {
    const SpDev &sp = sps[si];
    const u32x4 r = philox4x32_10((uint32_t)id, (uint32_t)(id >> 32), (uint32_t)step, RNG_QED_EMIT, seed, sp.sp_index);
    const float xi = qed_em_sample(*qd, chi, u01f(r.v[0]));
    const float eps = fminf(xi * gl, gl - 1.0f);
    const float g1 = gl - eps;
    const float un = sqrtf(ux * ux + uy * uy + uz * uz);
    const float u1 = sqrtf(fmaxf(g1 * g1 - 1.0f, 0.0f));
    float lost = 0.0f;
    if (eps >= sp.eps_min && sp.ph_species >= 0 && un > 0.0f)
        event_spawn(&sps[sp.ph_species], x, y, z, eps * ux / un, eps * uy / un, eps * uz / un, w, derived_id(id, step, 2u),
                    dest, step, seed, -logf(u01f(r.v[2])), status);
    else lost = eps;
    return make_float3(un > 0.0f ? u1 / un : 0.0f, -logf(u01f(r.v[1])), lost);
}

// Breit-Wheeler pair of photon `id` (momentum u, energy eps).  Returns the
// energies of the two that fall short of a rest mass.
static __device__ __noinline__ float2 event_pair(const SpDev *sps, int si, const QedDev *qd, float chi, float eps, float x,
                                                 float y, float z, float ux, float uy, float uz, float w, uint64_t id,
                                                 int dest, long long step, uint32_t seed, int *status) {
    const SpDev &sp = sps[si];
    const u32x4 r = philox4x32_10((uint32_t)id, (uint32_t)(id >> 32), (uint32_t)step, RNG_QED_PAIR, seed, sp.sp_index);
    const float xi = qed_pair_sample(*qd, chi, u01f(r.v[0]));
    const float en[2] = {xi * eps, (1.0f - xi) * eps};
#pragma unroll 1
    for (int k = 0; k < 2; ++k) {
        const float p = en[k] > 1.0f ? sqrtf(en[k] * en[k] - 1.0f) : 0.0f;
        event_spawn(&sps[k == 0 ? sp.pair_e : sp.pair_p], x, y, z, p * ux / eps, p * uy / eps, p * uz / eps, w,
                    derived_id(id, step, k == 0 ? 3u : 5u), dest, step, seed, -logf(u01f(k == 0 ? r.v[1] : r.v[2])),
                    status);
    }
    return make_float2(en[0] < 1.0f ? 1.0f - en[0] : 0.0f, en[1] < 1.0f ? 1.0f - en[1] : 0.0f);
}

// One CTA per tile (SPLIT: a cluster of CTAs per tile, each taking every
// cluster-size-th block of its particles): stage E, B of the tile and a
// one-node halo, push every particle of every species, deposit its current into
// the tile's fixed-point frame, apply the stochastic events (EV: some species
// has them), write it back or send it to the migration buffer.  Particles that
// stay in their cell deposit at once; particles that crossed a cell face wait in
// per-warp queues, one for a single crossed axis and one for the others, and are
// deposited 32 at a time, so that the long stencils run with every lane of the
// warp busy.  The warps meet only before the first and after the last species.
// With SPLIT the CTAs' frames are added as integers through distributed shared
// memory before the one rounding to FP32, so the current does not depend on the
// split.
// What bounds it, 15.7 M thermal particles (128 x 96 x 80 cells, a third of them
// crossing a face per step): the shared-memory pipe (75 %) and instruction issue
// (62 %), 56 B a particle of DRAM traffic; at rest 73 and 62 %.  Measured there, one
// launch (cold): 1.19 ms with 64-bit atomics and the FP64-pipe conversion, 0.89 ms
// with the word planes and the one-axis queue, 0.72 ms with the two-conversion
// digits and the migration chunks, 0.68 ms with the prefetched particle in registers
// (see queue_put; at rest 0.52, 0.62 with the spills, 0.44 ms); 0.76 M particles of
// the quadratic shape 0.46 -> 0.25 ms.
template <int T, int ORDER, bool EV, bool SPLIT>
__global__ void __launch_bounds__(push_threads(T), push_ctas(T, ORDER))
    k_push_deposit(GridDev g, const float *__restrict__ E, const float *__restrict__ B,
                   const SpDev *__restrict__ sps, int nsp, float *__restrict__ jscratch, int *__restrict__ jvalid,
                   int *__restrict__ status, const long long *__restrict__ step_dev, const __grid_constant__ QedDev qd) {
    constexpr int F = frame_F(T, ORDER), G = frame_G(T, ORDER);
    constexpr int F3 = F * F * F, G3 = G * G * G;
    constexpr int NT = push_threads(T), NW = NT / 32;
    extern __shared__ __align__(16) unsigned char smraw[];
    unsigned *sj = reinterpret_cast<unsigned *>(smraw);  // 3 current components, G^3 each: low words, high words
    float *sf = reinterpret_cast<float *>(smraw + align16(sizeof(unsigned long long) * 3 * G3));  // 6 x F^3
    float4 *queue = reinterpret_cast<float4 *>(reinterpret_cast<unsigned char *>(sf) + align16(sizeof(float) * 6 * F3));
    SpDev *s_sp = reinterpret_cast<SpDev *>(queue + NW * 4 * PUSH_Q);  // the species' descriptors
    __shared__ int s_holes[HYB_MAX_SPECIES];
    __shared__ int s_qwmax[32];  // per warp: largest |q w| of the tile's particles (float bits)
    __shared__ int s_kfix;       // fixed-point exponent of the tile's current frame
    __shared__ double s_tal_e[EV ? HYB_MAX_SPECIES * NTALLY : 1];
    __shared__ unsigned long long s_tal_n[EV ? HYB_MAX_SPECIES * NTALLY : 1];
    const long long step = EV ? *step_dev : 0;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float4 *q1 = queue + warp * 4 * PUSH_Q;  // crossed one axis (quadratic shape: the nearest nodes stay)
    float4 *q3 = q1 + 2 * PUSH_Q;            // crossed several (quadratic shape: some nearest node changes)

    cg::cluster_group cl = cg::this_cluster();
    const int nrank = SPLIT ? (int)cl.num_blocks() : 1, rank = SPLIT ? (int)cl.block_rank() : 0;
    const int t = SPLIT ? (int)blockIdx.x / nrank : (int)blockIdx.x;
    // a tile without particles writes no frame: the reduction skips it
    int total = 0;
    for (int si = 0; si < nsp; ++si) total += min(sps[si].count[t], sps[si].cap);
    if (total == 0) {
        if (rank == 0 && threadIdx.x < nsp) {
            sps[threadIdx.x].hole_count[t] = 0;
            sps[threadIdx.x].hole_used[t] = 0;
        }
        if (rank == 0 && threadIdx.x == 0) jvalid[t] = 0;
        return;
    }
    // the largest |q w| in the tile bounds every frame sum (fixed-point scale)
    {
        float qwm = 0.0f;
        for (int si = 0; si < nsp; ++si) {
            const SpDev &sp = sps[si];
            const int n = min(sp.count[t], sp.cap);
            const long long base = (long long)t * sp.cap;
#pragma unroll 4
            for (int p = rank * NT + threadIdx.x; p < n; p += nrank * NT) {
                const float qp = sp.zq ? sp.q * sp.zq[base + p] : sp.q;
                qwm = fmaxf(qwm, fabsf(qp * sp.w[base + p]));
            }
        }
        block_max_put(qwm, s_qwmax);
    }
    const int tx = t % g.nt[0], ty = (t / g.nt[0]) % g.nt[1], tz = t / (g.nt[0] * g.nt[1]);
    const int o[3] = {tx * T - ORDER, ty * T - ORDER, tz * T - ORDER};  // frame origin
    const long long N = g.N;

    for (int l = threadIdx.x; l < F3; l += NT) {
        const int lx = l % F, ly = (l / F) % F, lz = l / (F * F);
        int gi[3] = {o[0] + lx, o[1] + ly, o[2] + lz};
        bool in = true;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            if (g.bc[a] == 0) {
                gi[a] = gi[a] < 0 ? gi[a] + g.n[a] : (gi[a] >= g.n[a] ? gi[a] - g.n[a] : gi[a]);
            } else if (gi[a] < 0 || gi[a] > g.n[a] - 1) {
                in = false;
            }
        }
        const long long c = in ? cidx(g, gi[0], gi[1], gi[2]) : 0;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            sf[q * F3 + l] = in ? E[q * N + c] : 0.0f;
            sf[(3 + q) * F3 + l] = in ? B[q * N + c] : 0.0f;
        }
    }
    for (int l = threadIdx.x; l < 6 * G3; l += NT) sj[l] = 0u;
    {
        const int *src = reinterpret_cast<const int *>(sps);
        int *dst = reinterpret_cast<int *>(s_sp);
        for (int w = threadIdx.x; w < nsp * (int)(sizeof(SpDev) / sizeof(int)); w += NT) dst[w] = src[w];
    }
    if (threadIdx.x < HYB_MAX_SPECIES) s_holes[threadIdx.x] = 0;
    if (EV && threadIdx.x < HYB_MAX_SPECIES * NTALLY) {
        s_tal_e[threadIdx.x] = 0.0;
        s_tal_n[threadIdx.x] = 0;
    }
    if (SPLIT) cl.sync();
    else __syncthreads();

    const float dt = g.dt;
    const float inv_d[3] = {1.0f / g.d[0], 1.0f / g.d[1], 1.0f / g.d[2]};
    // current per unit q w of a face crossing: -1 / (dt dA_c), times the frame's
    // fixed-point scale 2^k (every Esirkepov weight is at most 1 in magnitude,
    // so a node's sum is at most total * max |q w| * max |jfac|)
    const float j0 = -1.0f / (dt * g.d[1] * g.d[2]), j1 = -1.0f / (dt * g.d[0] * g.d[2]),
                j2 = -1.0f / (dt * g.d[0] * g.d[1]);
    if (warp == 0) {
        // one warp: double precision is slow here
        int b = 0;
        for (int i = lane; i < nrank * NW; i += 32)
            b = max(b, SPLIT ? *cl.map_shared_rank(&s_qwmax[i % NW], i / NW) : s_qwmax[i]);
        b = __reduce_max_sync(0xffffffffu, b);
        const int k = fix_exponent((double)total * (double)__int_as_float(b) *
                                   (double)fmaxf(fabsf(j0), fmaxf(fabsf(j1), fabsf(j2))));
        if (lane == 0) s_kfix = k;
    }
    __syncthreads();
    const float fscale = pow2f(s_kfix);
    const float jfac[3] = {j0 * fscale, j1 * fscale, j2 * fscale};
    const float *sEx = sf, *sEy = sf + F3, *sEz = sf + 2 * F3;
    const float *sBx = sf + 3 * F3, *sBy = sf + 4 * F3, *sBz = sf + 5 * F3;
    // positions of this tile's particles: t0 <= x < t1 (an absorbing axis ends with its wall)
    float t0[3], t1[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        t0[a] = (float)(o[a] + ORDER);
        t1[a] = (float)(o[a] + ORDER + T);
        if (g.bc[a] && t1[a] > (float)(g.n[a] - 1)) t1[a] = __int_as_float(__float_as_int((float)(g.n[a] - 1)) + 1);
    }
    auto flush1 = [&](const float4 A, const float4 Bq) {
        if constexpr (ORDER == 1) deposit_one_crossing<G>(sj, A, Bq, o, jfac);
        else deposit_quadratic<G, 3>(sj, A, Bq, o, jfac);
    };
    auto flush3 = [&](const float4 A, const float4 Bq) {
        const float y0[3] = {A.x, A.y, A.z}, y1[3] = {Bq.x, Bq.y, Bq.z};
        if constexpr (ORDER == 1) deposit_general<G>(sj, y0, y1, o, A.w, jfac);
        else deposit_quadratic<G, 4>(sj, A, Bq, o, jfac);
    };
    int n1 = 0, n3 = 0;  // entries in this warp's queues (warp-uniform)

    for (int si = 0; si < nsp; ++si) {
        const SpDev &sp = s_sp[si];
        // events are rare: their tallies go straight to shared memory, no registers held for them
        auto tally = [&](int k, double energy) {
            if (energy != 0.0) atomicAdd(&s_tal_e[si * NTALLY + k], energy);
            atomicAdd(&s_tal_n[si * NTALLY + k], 1ULL);
        };
        const int n = min(sp.count[t], sp.cap);
        const long long base = (long long)t * sp.cap;
        // times q_p below; photons (m = 0, q = 0) get no Lorentz force
        const float qm_half = sp.kind == 1 ? 0.0f : 0.5f * dt / sp.m;
        // the next particle's x, y, z, ux, uy, uz, w and charge state, loaded one
        // iteration ahead so that the loads overlap the current particle's work
        float pf[8];
        auto prefetch = [&](int pp) {
            if (pp < n) {
                const long long s2 = base + pp;
                pf[0] = sp.x[s2]; pf[1] = sp.y[s2]; pf[2] = sp.z[s2];
                pf[3] = sp.ux[s2]; pf[4] = sp.uy[s2]; pf[5] = sp.uz[s2];
                pf[6] = sp.w[s2];
                pf[7] = sp.zq ? sp.zq[s2] : 1.0f;
            }
        };
        int mbase = 0, mused = MIG_CHUNK;  // the warp's chunk of the migration buffer and its used slots (uniform)
        prefetch(rank * NT + threadIdx.x);
        for (int p0 = rank * NT; p0 < n; p0 += nrank * NT) {
            const int p = p0 + threadIdx.x;
            bool act = p < n;
            const long long s = base + p;
            float x0[3] = {0.0f, 0.0f, 0.0f}, x1[3] = {0.0f, 0.0f, 0.0f}, u[3] = {0.0f, 0.0f, 0.0f};
            float e[3] = {0.0f, 0.0f, 0.0f}, b[3] = {0.0f, 0.0f, 0.0f};
            float wgt = 0.0f, q = 0.0f;
            if (act) {
                x0[0] = pf[0]; x0[1] = pf[1]; x0[2] = pf[2];
                u[0] = pf[3]; u[1] = pf[4]; u[2] = pf[5];
                wgt = pf[6];
                q = sp.q * pf[7];
            }
            prefetch(p + nrank * NT);
            if (act) {
                // every shared-memory index below derives from a cell inside this
                // tile; anything else (NaN among it) is flagged and left untouched
                const bool inside = x0[0] >= t0[0] && x0[0] < t1[0] && x0[1] >= t0[1] && x0[1] < t1[1] &&
                                    x0[2] >= t0[2] && x0[2] < t1[2];
                if (!inside) {
                    atomicOr(status, ST_BADPOS);
                    act = false;
                }
            }
            const float fl[3] = {floorf(x0[0]), floorf(x0[1]), floorf(x0[2])};
            if (act) {
                // ---- gather E^n, B^n at x^n
                if constexpr (ORDER == 1) {
                    const AxisW ax = axis_weights(g, 0, x0[0], fl[0], o[0]);
                    const AxisW ay = axis_weights(g, 1, x0[1], fl[1], o[1]);
                    const AxisW az = axis_weights(g, 2, x0[2], fl[2], o[2]);
                    e[0] = interp8<F>(sEx, ax.lh, ay.li, az.li, ax.fh, ay.fi, az.fi);
                    e[1] = interp8<F>(sEy, ax.li, ay.lh, az.li, ax.fi, ay.fh, az.fi);
                    e[2] = interp8<F>(sEz, ax.li, ay.li, az.lh, ax.fi, ay.fi, az.fh);
                    b[0] = interp8<F>(sBx, ax.li, ay.lh, az.lh, ax.fi, ay.fh, az.fh);
                    b[1] = interp8<F>(sBy, ax.lh, ay.li, az.lh, ax.fh, ay.fi, az.fh);
                    b[2] = interp8<F>(sBz, ax.lh, ay.lh, az.li, ax.fh, ay.fh, az.fi);
                } else {
                    // quadratic shape: integer (i) and half-integer (h) staggering per axis
                    int li[3], lh[3];
                    float wi[3][3], wh[3][3];
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        tsc_axis(x0[a], o[a], li[a], wi[a]);
                        tsc_axis(x0[a] - 0.5f, o[a], lh[a], wh[a]);
                    }
                    e[0] = interp27<F>(sEx, lh[0], li[1], li[2], wh[0], wi[1], wi[2]);
                    e[1] = interp27<F>(sEy, li[0], lh[1], li[2], wi[0], wh[1], wi[2]);
                    e[2] = interp27<F>(sEz, li[0], li[1], lh[2], wi[0], wi[1], wh[2]);
                    b[0] = interp27<F>(sBx, li[0], lh[1], lh[2], wi[0], wh[1], wh[2]);
                    b[1] = interp27<F>(sBy, lh[0], li[1], lh[2], wh[0], wi[1], wh[2]);
                    b[2] = interp27<F>(sBz, lh[0], lh[1], li[2], wh[0], wh[1], wi[2]);
                }

                // ---- momentum update (species-uniform choice: no divergence)
                const float h = q * qm_half;
                if (sp.pusher == HYB_PUSH_BORIS) boris_push(h, e, b, u);
                else if (sp.pusher == HYB_PUSH_VAY) vay_push(h, e, b, u);
                else higuera_cary_push(h, e, b, u);

                // ---- move (photons at c: velocity k / |k|), reflect at absorbing walls
                const float gam = sp.kind == 1 ? fmaxf(sqrtf(u[0] * u[0] + u[1] * u[1] + u[2] * u[2]), 1e-30f)
                                               : sqrtf(1.0f + u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    x1[a] = x0[a] + u[a] * (dt / gam) * inv_d[a];
                    if (g.bc[a]) {
                        const float L = (float)(g.n[a] - 1);
                        if (x1[a] < 0.0f) { x1[a] = -x1[a]; u[a] = -u[a]; }
                        else if (x1[a] > L) { x1[a] = 2.0f * L - x1[a]; u[a] = -u[a]; }
                    }
                }
                bool finite = true;
#pragma unroll
                for (int a = 0; a < 3; ++a) finite = finite && isfinite(x1[a]) && fabsf(x1[a] - x0[a]) < 1.0f;
                if (!finite) {
                    atomicOr(status, ST_BADPOS);
                    act = false;
                }
            }

            // ---- Esirkepov deposit into the shared frame: particles that stay
            // in their cell now, the others through the warp's queues
            const bool dep = act && q != 0.0f;
            if constexpr (ORDER == 1) {
                const bool c0 = floorf(x1[0]) != fl[0], c1 = floorf(x1[1]) != fl[1], c2 = floorf(x1[2]) != fl[2];
                const int nc = (c0 ? 1 : 0) + (c1 ? 1 : 0) + (c2 ? 1 : 0);
                const float qw = q * wgt;
                if (dep && nc == 0) {
                    const float fac[3] = {qw * jfac[0], qw * jfac[1], qw * jfac[2]};
                    deposit_same_cell<G>(sj, x0, x1, fl, o, fac);
                }
                const int ax = c0 ? 0 : (c1 ? 1 : 2);
                const float4 A = make_float4(sel3(ax, x0[0], x0[1], x0[2]), sel3(ax, x0[1], x0[2], x0[0]),
                                             sel3(ax, x0[2], x0[0], x0[1]), qw);
                const float4 Bq = make_float4(sel3(ax, x1[0], x1[1], x1[2]), sel3(ax, x1[1], x1[2], x1[0]),
                                              sel3(ax, x1[2], x1[0], x1[1]), __int_as_float(ax));
                queue_put(q1, n1, dep && nc == 1, A, Bq, lane, flush1);
                queue_put(q3, n3, dep && nc > 1, make_float4(x0[0], x0[1], x0[2], qw),
                          make_float4(x1[0], x1[1], x1[2], 0.0f), lane, flush3);
            } else {
                bool same = true;
#pragma unroll
                for (int a = 0; a < 3; ++a) same = same && floorf(x0[a] + 0.5f) == floorf(x1[a] + 0.5f);
                const float4 A = make_float4(x0[0], x0[1], x0[2], q * wgt);
                const float4 Bq = make_float4(x1[0], x1[1], x1[2], 0.0f);
                queue_put(q1, n1, dep && same, A, Bq, lane, flush1);
                queue_put(q3, n3, dep && !same, A, Bq, lane, flush3);
            }

            int nt = t;
            if (act) {
                // ---- periodic image, tile membership
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    if (g.bc[a] == 0) {
                        const float L = (float)g.n[a];
                        if (x1[a] < 0.0f) x1[a] += L;
                        else if (x1[a] >= L) x1[a] -= L;
                        if (x1[a] >= L) x1[a] = 0.0f;
                    }
                }
                nt = tile_index(g, x1[0], x1[1], x1[2]);
            }
            float zq_new = 0.0f, tau = 0.0f;
            bool dead = false;
            uint64_t pid = 0;
            if (EV && act) {
                // ---- stochastic events, after the deposit (this step's current
                // used the pre-event charge and momentum); new particles start at
                // x^{n+1} and enter their species through its migration buffer
                zq_new = sp.zq ? sp.zq[s] : 0.0f;
                tau = sp.tau ? sp.tau[s] : 0.0f;
                pid = sp.id[s];
                if (sp.zmax > 0 && zq_new < (float)sp.zmax) {
                    // field ionization: at most one level per step; the electron
                    // takes the ion's u and weight
                    const int Z = (int)zq_new;
                    const float P = ion_probability(sp, Z, sqrtf(e[0] * e[0] + e[1] * e[1] + e[2] * e[2]));
                    const u32x4 r = philox4x32_10((uint32_t)pid, (uint32_t)(pid >> 32), (uint32_t)step, RNG_IONIZE,
                                                  g.seed, sp.sp_index);
                    if (u01f(r.v[0]) < P) {
                        zq_new = (float)(Z + 1);
                        tally(TALLY_IONIZE, (double)wgt * sp.ip_mc2[Z]);
                        const uint64_t eid = (1ULL << 63) | (pid << 3) | (uint64_t)(Z + 1);
                        event_spawn(&s_sp[sp.ion_into], x1[0], x1[1], x1[2], u[0], u[1], u[2], wgt, eid, nt, step, g.seed,
                                    -1.0f, status);
                    }
                }
                if (sp.qed) {
                    // photon emission (radiation reaction), optical-depth method
                    const float gl = sqrtf(1.0f + u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
                    const float chi = qed_chi(qd.kappa, e, b, u, gl);
                    tau -= qd.pref * qed_h(qd, chi) / gl * dt;
                    if (tau <= 0.0f) {
                        const float3 ev = event_emit(s_sp, si, &qd, chi, gl, x1[0], x1[1], x1[2], u[0], u[1], u[2], wgt,
                                                     pid, nt, step, g.seed, status);
#pragma unroll
                        for (int c = 0; c < 3; ++c) u[c] *= ev.x;
                        tau = ev.y;
                        tally(TALLY_EMIT, (double)wgt * ev.z);
                    }
                }
                if (sp.kind == 1 && sp.pair_e >= 0) {
                    // Breit-Wheeler pair creation by a photon (energy >= 2 m c^2)
                    const float eps = sqrtf(u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
                    if (eps >= 2.0f) {
                        const float chi = qed_chi(qd.kappa, e, b, u, eps);
                        tau -= qd.pref * qed_T(qd, chi) / eps * dt;
                        if (tau <= 0.0f) {
                            const float2 ev = event_pair(s_sp, si, &qd, chi, eps, x1[0], x1[1], x1[2], u[0], u[1],
                                                         u[2], wgt, pid, nt, step, g.seed, status);
                            tally(TALLY_PAIR, (double)wgt * ev.x + (double)wgt * ev.y);
                            dead = true;
                        }
                    }
                }
            }

            // ---- write back or migrate
            const bool leave = act && (nt != t || dead), mig = leave && !dead;
            if (act && !leave) {
                sp.x[s] = x1[0]; sp.y[s] = x1[1]; sp.z[s] = x1[2];
                sp.ux[s] = u[0]; sp.uy[s] = u[1]; sp.uz[s] = u[2];
                if (EV && sp.zmax > 0) sp.zq[s] = zq_new;
                if (EV && sp.tau) sp.tau[s] = tau;
            }
            const unsigned mm = __ballot_sync(0xffffffffu, mig);
            if (mm != 0u) {
                // the warp's migrants take slots of the chunk it holds; a new
                // chunk costs one global atomic
                const int at = mused + __popc(mm & ((1u << lane) - 1u)), need = mused + __popc(mm);
                int next = 0;
                if (need > MIG_CHUNK) {
                    if (lane == 0) next = atomicAdd(sp.mig_count, sp.mig_chunks ? MIG_CHUNK : __popc(mm));
                    next = __shfl_sync(0xffffffffu, next, 0);
                }
                if (mig) {
                    const int m = at < MIG_CHUNK ? mbase + at : next + at - MIG_CHUNK;
                    if (m < sp.mig_cap) {
                        if constexpr (!EV) {
                            zq_new = sp.zq ? sp.zq[s] : 0.0f;
                            pid = sp.id[s];
                        }
                        sp.mx[m] = x1[0]; sp.my[m] = x1[1]; sp.mz[m] = x1[2];
                        sp.mux[m] = u[0]; sp.muy[m] = u[1]; sp.muz[m] = u[2];
                        sp.mw[m] = wgt;
                        if (sp.zq) sp.mzq[m] = zq_new;
                        if (sp.tau) sp.mtau[m] = tau;
                        sp.mid[m] = pid;
                        sp.mdest[m] = nt;
                    } else {
                        atomicOr(status, ST_OVERFLOW);
                    }
                }
                mused = need;
                if (need > MIG_CHUNK) {
                    mbase = next;
                    mused = sp.mig_chunks ? need - MIG_CHUNK : MIG_CHUNK;
                }
            }
            if (leave) {
                const int hslot = warp_append(SPLIT ? cl.map_shared_rank(&s_holes[si], 0) : &s_holes[si]);
                sp.holes[base + hslot] = p;
                sp.x[s] = -1.0f;
            }
        }
        // the rest of the warp's last chunk holds no migrant
        if (lane >= mused && mbase + lane < sp.mig_cap) sp.mdest[mbase + lane] = -1;
    }
    // what the queues still hold (each fewer than 32 particles)
    __syncwarp();
    if (lane < n1) flush1(q1[lane], q1[PUSH_Q + lane]);
    if (lane < n3) flush3(q3[lane], q3[PUSH_Q + lane]);
    if (SPLIT) cl.sync();
    else __syncthreads();

    if (rank == 0 && threadIdx.x < nsp) {
        s_sp[threadIdx.x].hole_count[t] = s_holes[threadIdx.x];
        s_sp[threadIdx.x].hole_used[t] = 0;
    }
    if (EV && rank == 0 && threadIdx.x < nsp * NTALLY) {
        const int i = threadIdx.x;
        double e = 0.0;
        unsigned long long c = 0;
        for (int r = 0; r < nrank; ++r) {
            e += SPLIT ? *cl.map_shared_rank(&s_tal_e[i], r) : s_tal_e[i];
            c += SPLIT ? *cl.map_shared_rank(&s_tal_n[i], r) : s_tal_n[i];
        }
        if (c > 0) {
            const SpDev &sp = s_sp[i / NTALLY];
            sp.tal_e[(long long)t * NTALLY + i % NTALLY] += e;
            sp.tal_n[(long long)t * NTALLY + i % NTALLY] += c;
        }
    }
    float *dst = jscratch + (long long)t * 3 * G3;
    const float inv_scale = pow2f(-s_kfix);
    for (int l = rank * NT + threadIdx.x; l < 3 * G3; l += nrank * NT) {
        unsigned long long v = 0ULL;
        if (SPLIT) {
            for (int r = 0; r < nrank; ++r) v += fix_read(cl.map_shared_rank(sj, r), 3 * G3, l);
        } else {
            v = fix_read(sj, 3 * G3, l);
        }
        dst[l] = fix_to_float(v, inv_scale);
    }
    if (rank == 0 && threadIdx.x == 0) jvalid[t] = 1;
    if (SPLIT) cl.sync();  // no CTA leaves while another reads its frame
}


// For every node: J = sum of the tile frames that cover it, in a fixed order.
__global__ void k_j_reduce(GridDev g, const float *__restrict__ jscratch, const int *__restrict__ jvalid,
                           float *__restrict__ J) {
    // grid (ceil(nx / blockDim.x), ny, nz)
    const int nx = g.n[0], ny = g.n[1];
    const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y, k = blockIdx.z;
    if (i >= nx) return;
    const long long c = ((long long)k * ny + j) * nx + i;
    float acc[3];
    frame_gather<3>(g, jscratch, jvalid, 3, g.order, i, j, k, acc);
    J[c] = acc[0];
    J[g.N + c] = acc[1];
    J[2 * g.N + c] = acc[2];
}

// Insert migrants: into a hole of the destination tile if one is free, else at
// its end.  One launch for all species (grid y), grid-stride over the migration
// buffer (its fill is read on device).
__global__ void __launch_bounds__(256) k_rebin(const SpDev *__restrict__ sps, int *__restrict__ status) {
    const SpDev &sp = sps[blockIdx.y];
    const int nm = min(*sp.mig_count, sp.mig_cap);
    // (a chunk's unused slots hold the destination -1)
    for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < nm; m += gridDim.x * blockDim.x) {
        const int t = sp.mdest[m];
        if (t < 0) continue;
        // the migrant's loads do not wait for its slot
        const float x = sp.mx[m], y = sp.my[m], z = sp.mz[m], ux = sp.mux[m], uy = sp.muy[m], uz = sp.muz[m];
        const float w = sp.mw[m], zq = sp.zq ? sp.mzq[m] : 0.0f, tau = sp.tau ? sp.mtau[m] : 0.0f;
        const uint64_t id = sp.mid[m];
        const int h = atomicAdd(&sp.hole_used[t], 1);
        int slot;
        if (h < sp.hole_count[t]) {
            slot = sp.holes[(long long)t * sp.cap + h];
        } else {
            slot = atomicAdd(&sp.count[t], 1);
            if (slot >= sp.cap) {
                atomicOr(status, ST_OVERFLOW);
                continue;
            }
        }
        const long long s = (long long)t * sp.cap + slot;
        sp.x[s] = x; sp.y[s] = y; sp.z[s] = z;
        sp.ux[s] = ux; sp.uy[s] = uy; sp.uz[s] = uz;
        sp.w[s] = w;
        if (sp.zq) sp.zq[s] = zq;
        sp.id[s] = id;
        if (sp.tau) sp.tau[s] = tau;
    }
}

// Close the holes no migrant filled: move live particles from the end of the
// tile into them and shrink the count.  One warp per tile, eight tiles per CTA,
// all species in one launch (grid y): the holes below the new count (in
// hole-list order) are filled with the live particles at or above it (in slot
// order), the same pairing as a serial walk of both lists.  Both lists pass
// through shared-memory queues, 128 candidates and up to 128 pairs at a time:
// the walk is a chain of dependent loads, and four a lane in flight shorten it.
// A step's last particle kernel also advances the step counter and empties the
// migration buffers.  Together with the one launch of k_rebin, against one launch
// a species of one-warp CTAs, 32 candidates at a time: five steps of two species
// on 64 tiles 296 -> 271 us, on 315 tiles 471 -> 451 us, ten steps of a 64 x 32 x 32
// hybrid run with a classification 3811 -> 3587 us.
static constexpr int CP_WARPS = 8, CP_N = 128;
__global__ void __launch_bounds__(32 * CP_WARPS) k_compact(GridDev g, const SpDev *__restrict__ sps, long long *step_dev) {
    __shared__ int s_hq[CP_WARPS][2 * CP_N], s_sq[CP_WARPS][2 * CP_N];
    const SpDev &sp = sps[blockIdx.y];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, t = blockIdx.x * CP_WARPS + warp;
    if (step_dev && blockIdx.x == 0 && threadIdx.x == 0) {
        *sp.mig_count = 0;
        if (blockIdx.y == 0) *step_dev += 1;
    }
    if (t >= g.ntiles) return;
    int *hq = s_hq[warp], *sq = s_sq[warp];
    const int hc = sp.hole_count[t], hu = sp.hole_used[t];
    const int n = min(sp.count[t], sp.cap);
    if (hu >= hc) {
        if (lane == 0) {
            sp.count[t] = n;  // an overflowing append left count above the capacity
            if (2 * n > sp.cap) atomicOr(sp.fill_flags, 1 << sp.sp_index);
        }
        return;
    }
    const long long base = (long long)t * sp.cap;
    const int new_n = n - (hc - hu);
    const unsigned below = (1u << lane) - 1u;
    int h = hu, src = new_n, hn = 0, sn = 0;
    for (;;) {
        while (hn < CP_N && h < hc) {
            int dst[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) dst[r] = h + 32 * r + lane < hc ? sp.holes[base + h + 32 * r + lane] : new_n;
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const bool ok = dst[r] < new_n;  // holes at or above new_n vanish with the shrink
                const unsigned m = __ballot_sync(0xffffffffu, ok);
                if (ok) hq[hn + __popc(m & below)] = dst[r];
                hn += __popc(m);
            }
            h += 128;
        }
        while (sn < CP_N && src < n) {
            float x[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) x[r] = src + 32 * r + lane < n ? sp.x[base + src + 32 * r + lane] : -1.0f;
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const bool ok = !(x[r] < 0.0f);  // live slot (vacated slots hold x < 0)
                const unsigned m = __ballot_sync(0xffffffffu, ok);
                if (ok) sq[sn + __popc(m & below)] = src + 32 * r + lane;
                sn += __popc(m);
            }
            src += 128;
        }
        __syncwarp();
        const int k = min(CP_N, min(hn, sn));  // up to four pairs a lane
        if (k == 0) break;
        long long a[4], b[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int i = 32 * r + lane;
            a[r] = i < k ? base + hq[i] : -1;
            b[r] = i < k ? base + sq[i] : -1;
        }
        auto move = [&](auto *arr) {
            std::remove_reference_t<decltype(arr[0])> v[4];
#pragma unroll
            for (int r = 0; r < 4; ++r)
                if (b[r] >= 0) v[r] = arr[b[r]];
#pragma unroll
            for (int r = 0; r < 4; ++r)
                if (a[r] >= 0) arr[a[r]] = v[r];
        };
        move(sp.x);
        move(sp.y);
        move(sp.z);
        move(sp.ux);
        move(sp.uy);
        move(sp.uz);
        move(sp.w);
        if (sp.zq) move(sp.zq);
        move(sp.id);
        if (sp.tau) move(sp.tau);
        // drop the k used entries of both queues (fewer than 128 + 127 before)
        int h1[8], q1[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const int i = 32 * r + lane + k;
            h1[r] = i < hn ? hq[i] : 0;
            q1[r] = i < sn ? sq[i] : 0;
        }
        __syncwarp();
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const int i = 32 * r + lane;
            if (i + k < hn) hq[i] = h1[r];
            if (i + k < sn) sq[i] = q1[r];
        }
        hn -= k;
        sn -= k;
        __syncwarp();
    }
    if (lane == 0) {
        sp.count[t] = new_n;
        sp.hole_count[t] = 0;
        sp.hole_used[t] = 0;
        if (2 * new_n > sp.cap) atomicOr(sp.fill_flags, 1 << sp.sp_index);
    }
}

// copy every tile's live slots into a species layout with a larger capacity
__global__ void k_regrid(SpDev from, SpDev to) {
    const int t = blockIdx.x;
    const int n = min(from.count[t], from.cap);
    const long long a = (long long)t * from.cap, b = (long long)t * to.cap;
    for (int p = threadIdx.x; p < n; p += blockDim.x) {
        to.x[b + p] = from.x[a + p]; to.y[b + p] = from.y[a + p]; to.z[b + p] = from.z[a + p];
        to.ux[b + p] = from.ux[a + p]; to.uy[b + p] = from.uy[a + p]; to.uz[b + p] = from.uz[a + p];
        to.w[b + p] = from.w[a + p];
        if (from.zq) to.zq[b + p] = from.zq[a + p];
        if (from.tau) to.tau[b + p] = from.tau[a + p];
        to.id[b + p] = from.id[a + p];
    }
}

__global__ void k_count_tiles(GridDev g, long long n, const float *__restrict__ x, const float *__restrict__ y,
                              const float *__restrict__ z, int *__restrict__ counts) {
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < n;
         p += (long long)gridDim.x * blockDim.x)
        atomicAdd(&counts[tile_index(g, x[p], y[p], z[p])], 1);
}

__global__ void k_bin(GridDev g, SpDev sp, long long n, const float *__restrict__ x, const float *__restrict__ y,
                      const float *__restrict__ z, const float *__restrict__ ux, const float *__restrict__ uy,
                      const float *__restrict__ uz, const float *__restrict__ w, const float *__restrict__ zq,
                      const uint64_t *__restrict__ ids, const float *__restrict__ tau, int *__restrict__ status) {
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < n;
         p += (long long)gridDim.x * blockDim.x) {
        const int t = tile_index(g, x[p], y[p], z[p]);
        const int slot = atomicAdd(&sp.count[t], 1);
        if (slot >= sp.cap) {
            atomicOr(status, ST_OVERFLOW);
            continue;
        }
        const long long s = (long long)t * sp.cap + slot;
        sp.x[s] = x[p]; sp.y[s] = y[p]; sp.z[s] = z[p];
        sp.ux[s] = ux[p]; sp.uy[s] = uy[p]; sp.uz[s] = uz[p];
        sp.w[s] = w[p];
        if (sp.zq) sp.zq[s] = zq ? zq[p] : 0.0f;
        sp.id[s] = ids ? ids[p] : (uint64_t)p;
        if (sp.tau) sp.tau[s] = tau ? tau[p] : tau_initial(sp.id[s], g.seed, sp.tau_index);
    }
}

// the live slots of every tile, tile after tile, into contiguous arrays
// (offsets: exclusive prefix sum of the tile counts); zq / tau / the outputs
// for them may be null
__global__ void k_tiles_to_arrays(SpDev sp, const long long *__restrict__ offsets, float *__restrict__ x,
                                  float *__restrict__ y, float *__restrict__ z, float *__restrict__ ux,
                                  float *__restrict__ uy, float *__restrict__ uz, float *__restrict__ w,
                                  float *__restrict__ zq, float *__restrict__ tau, uint64_t *__restrict__ ids) {
    const int t = blockIdx.x;
    const int n = min(sp.count[t], sp.cap);
    const long long a = (long long)t * sp.cap, b = offsets[t];
    for (int p = threadIdx.x; p < n; p += blockDim.x) {
        x[b + p] = sp.x[a + p]; y[b + p] = sp.y[a + p]; z[b + p] = sp.z[a + p];
        ux[b + p] = sp.ux[a + p]; uy[b + p] = sp.uy[a + p]; uz[b + p] = sp.uz[a + p];
        w[b + p] = sp.w[a + p];
        if (zq && sp.zq) zq[b + p] = sp.zq[a + p];
        if (tau && sp.tau) tau[b + p] = sp.tau[a + p];
        ids[b + p] = sp.id[a + p];
    }
}

static inline unsigned blocks_for(long long n, int b) { return (unsigned)((n + b - 1) / b); }

template <int T, int ORDER, bool EV, bool SPLIT>
static void push_launch(const GridDev &g, const float *E, const float *B, const SpDev *sps_dev, int nsp,
                        const QedDev &qd, float *jscratch, int *jvalid, int *status, const long long *step_dev,
                        int split, cudaStream_t st) {
    auto kern = k_push_deposit<T, ORDER, EV, SPLIT>;
    // opt in to more than 48 KB of dynamic shared memory, once per instance and device
    static std::once_flag once[64];
    int dev = 0;
    cudaGetDevice(&dev);
    std::call_once(once[dev & 63], [&] {
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)push_smem_bytes(T, ORDER, HYB_MAX_SPECIES));
    });
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(g.ntiles * split));
    cfg.blockDim = dim3((unsigned)push_threads(T));
    cfg.dynamicSmemBytes = push_smem_bytes(T, ORDER, nsp);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)split;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = SPLIT ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kern, g, E, B, sps_dev, nsp, jscratch, jvalid, status, step_dev, qd);
}

void launch_push_deposit(const GridDev &g, const float *E, const float *B, const SpDev *sps_dev, int nsp,
                         bool events, const QedDev &qd, float *jscratch, int *jvalid, int *status,
                         const long long *step_dev, int split, cudaStream_t st) {
    auto go = [&](auto kern) { kern(g, E, B, sps_dev, nsp, qd, jscratch, jvalid, status, step_dev, split, st); };
    auto shape = [&](auto ev, auto sp) {
        constexpr bool EV = decltype(ev)::value, SP = decltype(sp)::value;
        if (g.order == 2) go(g.T == 8 ? push_launch<8, 2, EV, SP> : push_launch<4, 2, EV, SP>);
        else go(g.T == 8 ? push_launch<8, 1, EV, SP> : push_launch<4, 1, EV, SP>);
    };
    const std::true_type yes;
    const std::false_type no;
    if (events) split > 1 ? shape(yes, yes) : shape(yes, no);
    else split > 1 ? shape(no, yes) : shape(no, no);
}

void launch_j_reduce(const GridDev &g, const float *jscratch, const int *jvalid, float *J, cudaStream_t st) {
    const int bx = g.n[0] >= 128 ? 128 : 32 * ((g.n[0] + 31) / 32);
    const dim3 grid((unsigned)((g.n[0] + bx - 1) / bx), (unsigned)g.n[1], (unsigned)g.n[2]);
    k_j_reduce<<<grid, bx, 0, st>>>(g, jscratch, jvalid, J);
}

void launch_rebin(const SpDev *sps_dev, int nsp, int *status, cudaStream_t st) {
    k_rebin<<<dim3(152 * 4, (unsigned)nsp), 256, 0, st>>>(sps_dev, status);
}

void launch_regrid(const GridDev &g, const SpDev &from, const SpDev &to, cudaStream_t st) {
    k_regrid<<<g.ntiles, 256, 0, st>>>(from, to);
}

void launch_compact(const GridDev &g, const SpDev *sps_dev, int nsp, long long *step_dev, cudaStream_t st) {
    k_compact<<<dim3((unsigned)((g.ntiles + CP_WARPS - 1) / CP_WARPS), (unsigned)nsp), 32 * CP_WARPS, 0, st>>>(g, sps_dev,
                                                                                                              step_dev);
}

void launch_count_tiles(const GridDev &g, long long n, const float *x, const float *y, const float *z,
                        int *counts, cudaStream_t st) {
    if (n == 0) return;
    k_count_tiles<<<min(blocks_for(n, 256), 152u * 16u), 256, 0, st>>>(g, n, x, y, z, counts);
}

void launch_bin_particles(const GridDev &g, const SpDev &s, long long n, const float *x, const float *y,
                          const float *z, const float *ux, const float *uy, const float *uz, const float *w,
                          const float *zq, const uint64_t *ids, const float *tau, int *status, cudaStream_t st) {
    if (n == 0) return;
    k_bin<<<min(blocks_for(n, 256), 152u * 16u), 256, 0, st>>>(g, s, n, x, y, z, ux, uy, uz, w, zq, ids, tau,
                                                               status);
}

void launch_tiles_to_arrays(const GridDev &g, const SpDev &s, const long long *offsets, float *x, float *y, float *z,
                            float *ux, float *uy, float *uz, float *w, float *zq, float *tau, uint64_t *ids,
                            cudaStream_t st) {
    k_tiles_to_arrays<<<g.ntiles, 256, 0, st>>>(s, offsets, x, y, z, ux, uy, uz, w, zq, tau, ids);
}

}  // namespace hyb

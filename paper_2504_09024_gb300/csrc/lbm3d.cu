// D3Q27 form of the phase-field (f, App. C) and interface-bound surfactant
// (h, Sec. 3) central-moment lattices under a prescribed velocity: one
// z-marching kernel per time step behind the C ABI of include/lbm3.h.
//
// Collision in closed form.  Both lattices relax every central moment but
// the three first-order ones to its Maxwellian equilibrium (rate 1).  With
// the tensor-product moment basis |e_x^m e_y^n e_z^p> the post-collision
// central moments are
//     s mu(m) mu(n) mu(p) + k'_x [100] + k'_y [010] + k'_z [001],
//     mu = (1, 0, cs^2),  k'_i = k_i + w (K theta n_i - k_i),  k_i = j_i - u_i s,
// and P^-1 F^-1(u) is the Kronecker product of its one-dimensional factors,
// so the outgoing population of velocity (a, b, c) is
//     s Ax[a] Ay[b] Az[c] + k'_x Bx[a] Cy[b] Cz[c] + (k'_y By[b] Cz[c] + k'_z Cy[b] Bz[c]) Cx[a]
// with, per axis of velocity u (e = 0, +1, -1):
//     A = central (1, 0, cs^2) -> (1 - cs^2 - u^2, (cs^2 + u^2 + u)/2, (cs^2 + u^2 - u)/2)
//     B = central (0, 1, 0)    -> (-2u, u + 1/2, u - 1/2)
//     C = central (1, 0, 0)    -> (1 - u^2, (u^2 + u)/2, (u^2 - u)/2).
//
// State: four words a lattice and cell.  A collision therefore needs only
// s = sum a and j = sum e a of the incoming populations, and those four sums
// are all that is kept between steps: int32 fixed point in units of 2^-28,
// words 2 (((z * 4 + m) * ny + y) * nx + x) (f) and the next (h), m = s, jx, jy, jz.
// A step forms the 27 outgoing populations of a cell in registers, rounded to the
// 2^-28 grid (of a row along x its sum and its two moving populations are rounded,
// the third is what is left; the rest population takes the integer remainder of s,
// so sum f and sum h are conserved exactly), and adds them into the sums of the
// cells they stream to; the sums are exact in integers, so the state is the
// one that storing all 54 populations gives, at 64 bytes a cell and step
// instead of 432.  (With FP32 storage every cell of a uniform region makes the
// same rounding error in every step and the region's phi drifts coherently; in
// integers a uniform region is an exact fixed point.)
//
// A cell whose zeroth moment leaves (-4, 4) sends FX_BAD in all its
// populations; a single population below -8 is FX_BAD too, and one above 8 is cut
// off there.  A cell that receives FX_BAD gets it as its zeroth moment, so it
// is out of range in turn.  (The sums do not say so by themselves: an even number
// of FX_BAD adds up to nothing.)
//
// Outputs.  phi and c are the zeroth moments.  Populations are formed again when
// they are asked for: those of the state from the moments one step back (the other
// buffer), those of the initial state from the fields it was made of, which the
// context keeps.  A step writes its number into the `suspect` word of every plane
// with a cell that is not certain to stay in range (Collision::tame): next to such a
// plane the sums may have wrapped around, and in it populations may be invalid, so
// there, and only there, fields and totals look at populations.
//
// Step kernel.  A block owns a 30 x (ROWS - 2) column of cells with a one-cell
// halo (one warp per row of 32 columns) and marches through seg_z planes.  At
// plane k each thread forms the populations of its cell; along x they are
// added by shuffles, along y through shared memory, along z in registers, and
// the moments of plane k - 1 are then complete and stored.  phi of plane k + 2
// (with a second halo cell for the gradient) is on its way to shared memory and
// the moments of plane k + 1 are on their way to registers (or by way of shared
// memory, k3_ahead) meanwhile.  The
// exchange buffer and the phi plane alternate between two copies, so one
// barrier per plane suffices.  Halo rows form only the populations that enter
// the tile.  The loop forms populations as if every cell were valid and every
// population in range; a block that met others goes over its cells once more at
// its end (settle).
// (Bits of invalid cells exchanged in the loop with the populations cost 8 to 10 %
// of a step in which nothing is invalid.)
//
// What bounds it: instruction issue (58-73 % of the slots, DRAM at a fifth of its
// rate) at the 18 to 20 warps an SM that the registers allow.  256^3 at the library's
// shape: 1980 us a step with all populations stored; in moments 600 us with a
// uniform velocity and 784 with a field; f and h in packed FP32 instructions (lane
// x: f, lane y: h) and 16-byte words across rows 575 and 724; a row's two moving
// populations and its sum instead of three populations (emit_rows) 504 and 655;
// the next plane by way of shared memory 503 and 602.  The 64 bytes a cell take
// 160 us.
#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <new>
#include <utility>

#include "lbm3.h"
#include "lbm_vec.cuh"

namespace {

using lbm::f2;

constexpr int Q27 = 27;
constexpr int TILE_W = 32;   // columns of a tile row, halo included
constexpr int TILE_IN = 30;  // columns a block updates
constexpr float FX_ONE = 268435456.0f;        // 2^28 units per unit value
constexpr float FX_INV = 1.0f / 268435456.0f;
constexpr double FX_ONE_D = 268435456.0;
constexpr double FX_INV_D = 1.0 / 268435456.0;
constexpr int FX_BAD = (-2147483647 - 1);       // invalid population marker
constexpr float S_MAX = 4.0f;                   // valid |zeroth moment|
constexpr int SUM_BLOCKS = 1024;
constexpr int SUM_THREADS = 256;

struct Nvtx {
    explicit Nvtx(const char* name) { nvtxRangePushA(name); }
    ~Nvtx() { nvtxRangePop(); }
};

struct K3Params {
    int nx, ny, nz, seg_z;
    long long N, nxny;
    float w_kappa, w_chi, M_phi, D_s;
    float c4W, c8W, phi_a, phi_b, phim, inv_dphi;
    float u[3];
    // uniform u: the factors along x of emit_rows (t/2, 2u, u^2/2, u/2), and the
    // products of those along y and z, [c][b]: Ay Az, Cy Cz / 2, By Cz, Cy Bz; in
    // both lanes
    float2 fx[4], aa[3][3], cc[3][3], bc[3][3], cb[3][3];
    const float* uf;  // per-cell velocity [3][N], or null for the uniform u
    long long number;    // of the state that is written or read: steps since the initial one
    long long* suspect;  // [nz + 1]: the last state that senders of a plane made suspect; of any plane
};

__host__ __device__ __forceinline__ int wrapi(int v, int n) {
    int r = v % n;
    return r < 0 ? r + n : r;
}

// One-dimensional factors of P^-1 F^-1(u) (index 0: e = 0, 1: e = +1, 2: e = -1).
template <class T>
__host__ __device__ __forceinline__ void axis_factors(T u, T* A, T* B, T* C) {
    const T u2 = u * u;
    const T t = T(1) / T(3) + u2;
    A[0] = T(1) - t;
    A[1] = T(0.5) * (t + u);
    A[2] = T(0.5) * (t - u);
    B[0] = T(-2) * u;
    B[1] = u + T(0.5);
    B[2] = u - T(0.5);
    C[0] = T(1) - u2;
    C[1] = T(0.5) * (u2 + u);
    C[2] = T(0.5) * (u2 - u);
}

// Outgoing populations of one collision; out(q, value) receives each.
template <class T, class Out>
__device__ __forceinline__ void emit27(const T (&Ax)[3], const T (&Bx)[3], const T (&Cx)[3],
                                       const T (&Ay)[3], const T (&By)[3], const T (&Cy)[3],
                                       const T (&Az)[3], const T (&Bz)[3], const T (&Cz)[3],
                                       T s, T kx, T ky, T kz, Out out) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const T P = s * (Ay[b] * Az[c]);
            const T X = kx * (Cy[b] * Cz[c]);
            const T R = ky * (By[b] * Cz[c]) + kz * (Cy[b] * Bz[c]);
#pragma unroll
            for (int a = 0; a < 3; ++a) out(a + 3 * b + 9 * c, P * Ax[a] + X * Bx[a] + R * Cx[a]);
        }
    }
}

__device__ __forceinline__ float fx_to_f(int v) { return (float)v * FX_INV; }

// Both zeroth moments inside (-4, 4).
__device__ __forceinline__ bool valid(int2 s) {
    return fabsf(fx_to_f(s.x)) < S_MAX && fabsf(fx_to_f(s.y)) < S_MAX;
}

// What the gradient needs of one plane of phi around a cell: phi smoothed over
// the plane, and its smoothed differences along x and y (twice the derivative).
// Differences of equal values are exactly zero.
struct Plane {
    float g0, gx, gy;
};

template <class At>
__device__ __forceinline__ Plane plane_of(At at) {
    float m[3], d[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        const float l = at(r - 1, -1), o = at(r - 1, 0), h = at(r - 1, 1);
        m[r] = __fmaf_rn(__fadd_rn(l, h), 1.0f / 6.0f, __fmul_rn(o, 2.0f / 3.0f));
        d[r] = __fsub_rn(h, l);
    }
    return Plane{__fmaf_rn(__fadd_rn(m[0], m[2]), 1.0f / 6.0f, __fmul_rn(m[1], 2.0f / 3.0f)),
                 __fmaf_rn(__fadd_rn(d[0], d[2]), 1.0f / 6.0f, __fmul_rn(d[1], 2.0f / 3.0f)),
                 __fsub_rn(m[2], m[0])};
}

// The largest magnitude (NaN if one is NaN).
__device__ __forceinline__ float most_of(float a, float b, float c) {
    float r;
    asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(fabsf(a)), "f"(fabsf(b)), "f"(fabsf(c)));
    return r;
}

// A collision of both lattices (lane x: f, lane y: h), in fixed-point units:
// zeroth moments, relaxed first-order central moments and the velocity.  Every
// operation is written out (no contraction left to the compiler), so that the
// step and the kernels that form populations again agree to the last bit.
struct Collision {
    int2 s_fx;
    f2 s, k[3];
    float u[3];
    float most, big, fast;  // the larger |s|, the largest |k'| (or |s|/10), a field's largest |u|
    bool tame;  // safe(), nor can the sums of what such cells send leave 32 bits
    // both zeroth moments inside (-4, 4)
    __device__ __forceinline__ bool ok() const { return most < S_MAX * FX_ONE; }
    // and no population can leave the range: uniform |u| < 1/2 |A| <= 0.67, |B| <= 1 and |C| <= 1;
    // a field's by the largest factor of each axis
    template <bool UFIELD>
    __device__ __forceinline__ bool safe() const {
        if constexpr (!UFIELD) return ok() && __fmaf_rn(0.3f, most, 3.0f * big) < 7.9f * FX_ONE;
        float a = 1.0f, b[3], c[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const float v = fabsf(u[i]), v2 = __fmul_rn(v, v), m = __fadd_rn(v2, v);
            a = __fmul_rn(a, fmaxf(fmaxf(2.0f / 3.0f, __fadd_rn(v2, -2.0f / 3.0f)), __fmul_rn(0.5f, __fadd_rn(1.0f / 3.0f, m))));
            b[i] = fmaxf(2.0f * v, __fadd_rn(v, 0.5f));
            c[i] = fmaxf(fmaxf(1.0f, __fadd_rn(v2, -1.0f)), 0.5f * m);
        }
        const float k = __fmaf_rn(__fmul_rn(b[0], c[1]), c[2],
                                  __fmaf_rn(__fmul_rn(c[0], b[1]), c[2], __fmul_rn(__fmul_rn(c[0], c[1]), b[2])));
        return ok() && __fmaf_rn(a, most, __fmul_rn(k, big)) < 7.9f * FX_ONE;
    }
};

template <bool UFIELD>
__device__ __forceinline__ Collision collide(const K3Params& p, const int2 (&m)[4], const Plane& lo,
                                             const Plane& mid, const Plane& hi, const float (&u)[3]) {
    Collision r;
    const float g[3] = {0.5f * __fmaf_rn(__fadd_rn(lo.gx, hi.gx), 1.0f / 6.0f, __fmul_rn(mid.gx, 2.0f / 3.0f)),
                        0.5f * __fmaf_rn(__fadd_rn(lo.gy, hi.gy), 1.0f / 6.0f, __fmul_rn(mid.gy, 2.0f / 3.0f)),
                        0.5f * __fsub_rn(hi.g0, lo.g0)};
    const float g2 = __fmaf_rn(g[2], g[2], __fmaf_rn(g[1], g[1], __fmul_rn(g[0], g[0])));
    const float inv = g2 > 1e-24f ? rsqrtf(g2) : 0.f;
    r.s_fx = m[0];
    r.s = f2((float)m[0].x, (float)m[0].y);
    const float phi = __fmul_rn(r.s.x, FX_INV), c = __fmul_rn(r.s.y, FX_INV);
    // theta (Eq. theta) and theta_c (Eq. ISS), times M_phi and D_s
    const float theta =
        __fmul_rn(__fmul_rn(__fmul_rn(p.c4W, __fsub_rn(p.phi_a, phi)), __fsub_rn(phi, p.phi_b)), p.inv_dphi);
    const float thetac = __fmul_rn(__fmul_rn(__fmul_rn(p.c8W, c), __fsub_rn(p.phim, phi)), p.inv_dphi);
    const f2 q(__fmul_rn(p.M_phi, theta) * FX_ONE, __fmul_rn(p.D_s, thetac) * FX_ONE);
    const f2 w(p.w_kappa, p.w_chi);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const f2 a = lbm::vfma(f2(-u[i]), r.s, f2((float)m[i + 1].x, (float)m[i + 1].y));
        r.u[i] = u[i];
        r.k[i] = lbm::vfma(w, lbm::vfma(q, f2(__fmul_rn(g[i], inv)), -a), a);
    }
    r.most = fmaxf(fabsf(r.s.x), fabsf(r.s.y));
    r.big = most_of(most_of(most_of(r.k[0].x, r.k[0].y, r.k[1].x), r.k[1].y, r.k[2].x), r.k[2].y, 0.1f * r.most);
    r.fast = UFIELD ? most_of(u[0], u[1], u[2]) : 0.f;
    // What the 27 neighbours of a cell send it adds up to less than 8.  Uniform |u| < 1/2: the
    // products of A add up to 1 and those of B and C to less than 3.2 a component, 4 + 3 * 3.2 *
    // 0.4.  A field, where each neighbour has its own u and is of one kind or the other: 7.84, each
    // product at its largest (test_range_bounds3.py).
    if constexpr (UFIELD) {
        const bool slow = r.fast <= 0.2f;
        r.tame = r.fast <= 0.4f && r.most < (slow ? 2.1f : 1.1f) * FX_ONE && r.big < (slow ? 0.3f : 0.15f) * FX_ONE;
    } else {
        r.tame = r.big < 0.4f * FX_ONE;  // and |s| below 4
    }
    return r;
}

__device__ __forceinline__ uint2 operator+(uint2 a, uint2 b) { return make_uint2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ uint2 operator-(uint2 a, uint2 b) { return make_uint2(a.x - b.x, a.y - b.y); }

// Populations (0, b, c), (1, b, c), (2, b, c) of both lattices, c = 0, 1, 2, as
// row(c, total, v1, v2): v1 and v2 and the row's sum are rounded to the grid, and
// v0 = total - v1 - v2.  With P = s A A, X = kx C C, R = ky B C + kz C B the row is
//     total = P + R,  v1, v2 = E +- O,
//     E = P (cs^2 + u^2)/2 + X u + R u^2/2,  O = (P + R) u/2 + X/2.
// UFIELD takes the factors from the cell's velocity, otherwise they come with the
// parameters.  The rest population is the caller's (v0 of b = c = 0).  With CHECK,
// v0 of a cell that is not safe() is rounded by itself, like v1 and v2 (the
// conversion cuts off at the ends of the range, and its lower end is FX_BAD), and
// all populations of a cell that is not ok are FX_BAD.
template <bool UFIELD, bool CHECK, class Row>
__device__ __forceinline__ void emit_rows(const K3Params& p, const Collision& r, int b, Row row) {
    float A[3][3], B[3][3], C[3][3];  // along y and z
    f2 th, u2x, uh2, uh;              // along x
    if constexpr (UFIELD) {
#pragma unroll
        for (int i = 1; i < 3; ++i) {
            const float v = r.u[i], u2 = __fmul_rn(v, v), t = __fadd_rn(1.0f / 3.0f, u2);
            A[i][0] = __fsub_rn(1.0f, t);
            A[i][1] = __fmul_rn(0.5f, __fadd_rn(t, v));
            A[i][2] = __fmul_rn(0.5f, __fsub_rn(t, v));
            B[i][0] = -2.0f * v;
            B[i][1] = __fadd_rn(v, 0.5f);
            B[i][2] = __fsub_rn(v, 0.5f);
            C[i][0] = __fsub_rn(1.0f, u2);
            C[i][1] = __fmul_rn(0.5f, __fadd_rn(u2, v));
            C[i][2] = __fmul_rn(0.5f, __fsub_rn(u2, v));
        }
        const float v = r.u[0], h2 = __fmul_rn(0.5f * v, v);
        th = f2(__fadd_rn(0.5f / 3.0f, h2));
        u2x = f2(2.0f * v);
        uh2 = f2(h2);
        uh = f2(0.5f * v);
    } else {
        th = lbm::from_f2(p.fx[0]);
        u2x = lbm::from_f2(p.fx[1]);
        uh2 = lbm::from_f2(p.fx[2]);
        uh = lbm::from_f2(p.fx[3]);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        f2 P, X, R;  // X: half of the above
        if constexpr (UFIELD) {
            P = r.s * f2(__fmul_rn(A[1][b], A[2][c]));
            X = r.k[0] * f2(__fmul_rn(0.5f * C[1][b], C[2][c]));
            R = lbm::vfma(r.k[1], f2(__fmul_rn(B[1][b], C[2][c])), r.k[2] * f2(__fmul_rn(C[1][b], B[2][c])));
        } else {
            P = r.s * lbm::from_f2(p.aa[c][b]);
            X = r.k[0] * lbm::from_f2(p.cc[c][b]);
            R = lbm::vfma(r.k[1], lbm::from_f2(p.bc[c][b]), r.k[2] * lbm::from_f2(p.cb[c][b]));
        }
        const f2 W = P + R, O = lbm::vfma(W, uh, X), E = lbm::vfma(P, th, lbm::vfma(X, u2x, R * uh2));
        auto grid = [&](f2 v) {
            return CHECK && !r.ok() ? make_uint2((uint32_t)FX_BAD, (uint32_t)FX_BAD)
                                  : make_uint2((uint32_t)__float2int_rn(v.x), (uint32_t)__float2int_rn(v.y));
        };
        const uint2 v1 = grid(E + O), v2 = grid(E - O);
        row(c, CHECK && !r.template safe<UFIELD>() ? grid(lbm::vfma(f2(-2.0f), E, W)) + v1 + v2 : grid(W), v1, v2);
    }
}

__device__ __forceinline__ uint2 from_left(uint2 v) {
    return make_uint2(__shfl_up_sync(0xffffffffu, v.x, 1), __shfl_up_sync(0xffffffffu, v.y, 1));
}
__device__ __forceinline__ uint2 from_right(uint2 v) {
    return make_uint2(__shfl_down_sync(0xffffffffu, v.x, 1), __shfl_down_sync(0xffffffffu, v.y, 1));
}

// Resident blocks per SM the register budget is sized for: 80 registers a
// thread at 6 rows (about 90 bytes of spill), 96 at 10 and 18 (up to 20).
template <int ROWS>
constexpr int k3_min_blocks() { return ROWS == 6 ? 4 : ROWS == 10 ? 2 : 1; }

constexpr int RING_W = TILE_W + 2;
template <int ROWS>
constexpr int k3_ring_words() { return (ROWS + 2) * RING_W; }
template <int ROWS>
constexpr int k3_xchg_words() { return 24 * ROWS * TILE_W; }  // 6 x uint4 a cell
// Whether the next plane's moments (and velocity) come by way of shared memory: live
// in registers through the emission, some are spilled, and a spilled one waits there
// for its load.  us a step at 256^3, in registers and this way: field, 18 rows 655 and
// 602, 10 rows (48 planes) 790 and 576; uniform, 18 rows 525 and 516, 10 rows 503 and 507.
template <int ROWS, bool UFIELD>
constexpr bool k3_ahead() { return UFIELD || ROWS == 18; }
template <int ROWS, bool UFIELD>
constexpr int k3_smem() {  // ahead: 4 x int2 and, with a field, 3 x float a cell
    return 4 * (2 * (k3_ring_words<ROWS>() + k3_xchg_words<ROWS>()) +
                (k3_ahead<ROWS, UFIELD>() ? (UFIELD ? 11 : 8) * ROWS * TILE_W : 0));
}

// Asynchronous copy of 4 or 8 bytes into shared memory.
template <int BYTES>
__device__ __forceinline__ void cp_async(void* dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
                 "n"(BYTES)
                 : "memory");
}

__device__ __forceinline__ int vel(int a) { return a == 0 ? 0 : a == 1 ? 1 : -1; }

// The populations that a cell of a state sends out in a step: out(q, f, h).
template <class Out>
__device__ __forceinline__ void outgoing(const K3Params& p, const int* __restrict__ state, int x, int y, int z,
                                         Out out) {
    Plane pl[3];
#pragma unroll
    for (int dz = 0; dz < 3; ++dz) {
        const int* q = state + 8 * p.nxny * wrapi(z + dz - 1, p.nz);
        pl[dz] = plane_of([&](int dy, int dx) {
            return fx_to_f(q[2 * ((long long)wrapi(y + dy, p.ny) * p.nx + wrapi(x + dx, p.nx))]);
        });
    }
    const long long in = (long long)y * p.nx + x;
    int2 m[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) m[i] = reinterpret_cast<const int2*>(state)[(4LL * z + i) * p.nxny + in];
    float u[3] = {p.u[0], p.u[1], p.u[2]};
    if (p.uf)
        for (int i = 0; i < 3; ++i) u[i] = p.uf[i * p.N + z * p.nxny + in];
    const Collision r = collide<true>(p, m, pl[0], pl[1], pl[2], u);
    uint2 v[Q27], moved = make_uint2(0u, 0u);
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        auto row = [&](int c, uint2 total, uint2 v1, uint2 v2) {
            const int q = 3 * b + 9 * c;
            v[q] = total - v1 - v2;
            v[q + 1] = v1;
            v[q + 2] = v2;
            moved = moved + (q ? total : v1 + v2);
        };
        if (p.uf)
            emit_rows<true, true>(p, r, b, row);
        else
            emit_rows<false, true>(p, r, b, row);
    }
    v[0] = make_uint2((uint32_t)r.s_fx.x, (uint32_t)r.s_fx.y) - moved;
    if (!r.ok()) v[0] = make_uint2((uint32_t)FX_BAD, (uint32_t)FX_BAD);
#pragma unroll
    for (int q = 0; q < Q27; ++q) out(q, (int)v[q].x, (int)v[q].y);
}

// What the step's loop leaves out, for a block that met cells that are not tame: the
// word of `suspect` for the whole box (from every such cell, stores to the one word
// took longer than the step); and (invalid: the block met invalid ones) FX_BAD for
// the zeroth moments of cells that FX_BAD is sent to, by invalid cells of `src` and
// (single: the block met cells that are not safe()) by others; for the latter all
// sums are made once more, of the populations as they are cut off.  A function of
// its own, and one that adds up in place: what it needs in registers costs the loop
// up to 5 %.
template <int ROWS>
__device__ __noinline__ void settle(const K3Params& p, const int* __restrict__ src, int* __restrict__ dst,
                                    bool invalid, bool single) {
    if (threadIdx.x == 0) p.suspect[p.nz] = p.number;
    if (!invalid && !single) return;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int x = blockIdx.x * TILE_IN + tx - 1, y = blockIdx.y * (ROWS - 2) + ty - 1;
    if (tx < 1 || tx > TILE_IN || x >= p.nx || ty < 1 || ty > ROWS - 2 || y >= p.ny) return;
    const int z0 = blockIdx.z * p.seg_z, z1 = min(p.nz, z0 + p.seg_z);
    for (int z = z0; z < z1; ++z) {
        bool bad_f = false, bad_h = false;
        uint2* o = reinterpret_cast<uint2*>(dst) + 4 * p.nxny * z + y * p.nx + x;
        if (single)
            for (int i = 0; i < 4; ++i) o[i * p.nxny] = make_uint2(0u, 0u);
        for (int want = 0; want < Q27; ++want) {
            const int e[3] = {vel(want % 3), vel(want / 3 % 3), vel(want / 9)};
            const int sx = wrapi(x - e[0], p.nx), sy = wrapi(y - e[1], p.ny), sz = wrapi(z - e[2], p.nz);
            if (!valid(reinterpret_cast<const int2*>(src)[4 * p.nxny * sz + sy * p.nx + sx])) {
                bad_f = bad_h = true;
            } else if (single) {
                outgoing(p, src, sx, sy, sz, [&](int q, int f, int h) {
                    if (q != want) return;
                    bad_f |= f == FX_BAD;
                    bad_h |= h == FX_BAD;
                    const uint2 v = make_uint2((uint32_t)f, (uint32_t)h);
                    o[0] = o[0] + v;
                    for (int i = 0; i < 3; ++i) {
                        uint2* j = o + (i + 1) * p.nxny;
                        *j = e[i] < 0 ? *j - v : e[i] ? *j + v : *j;
                    }
                });
            }
        }
        if (bad_f) o->x = (uint32_t)FX_BAD;
        if (bad_h) o->y = (uint32_t)FX_BAD;
    }
}

template <int ROWS, bool UFIELD>
__global__ void __launch_bounds__(ROWS * 32, k3_min_blocks<ROWS>())
k3_step(const __grid_constant__ K3Params p, const int* __restrict__ src, int* __restrict__ dst) {
    extern __shared__ __align__(16) float smem[];
    constexpr int RING = k3_ring_words<ROWS>(), XCHG = k3_xchg_words<ROWS>(), NT = ROWS * 32;
    constexpr int PLANE = ROWS * TILE_W;
    // per (c, b = 1, 2): sums and differences along x of f, then of h, [2][6][ROWS][TILE_W]
    uint4* xchg = reinterpret_cast<uint4*>(smem);
    float* ring = smem + 2 * XCHG;  // [2][ROWS + 2][RING_W]
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int bx = blockIdx.x * TILE_IN, by = blockIdx.y * (ROWS - 2);
    const int last = min(ROWS - 2, p.ny - by);  // last tile row that is updated
    const bool inner = ty >= 1 && ty <= last;
    const bool store = inner && tx >= 1 && tx <= TILE_IN && bx + tx - 1 < p.nx;
    const int nxny = (int)p.nxny;
    const int cell = wrapi(by + ty - 1, p.ny) * p.nx + wrapi(bx + tx - 1, p.nx);  // inside a plane
    // the two cells of the phi plane that this thread fetches
    static_assert(RING <= 2 * NT, "two phi cells a thread");
    const int i1 = threadIdx.x + NT;
    const int o0 = wrapi(by + (int)threadIdx.x / RING_W - 2, p.ny) * p.nx +
                   wrapi(bx + (int)threadIdx.x % RING_W - 2, p.nx);
    const int o1 = i1 < RING ? wrapi(by + i1 / RING_W - 2, p.ny) * p.nx + wrapi(bx + i1 % RING_W - 2, p.nx) : 0;
    const long long pstride = 8LL * nxny;  // words of one plane of the state
    const int z0 = blockIdx.z * p.seg_z;
    const int z1 = min(p.nz, z0 + p.seg_z);
    auto next = [&](int z) { return z + 1 == p.nz ? 0 : z + 1; };

    auto fetch = [&](int z, int slot) {
        const int* q = src + z * pstride;
        ring[slot * RING + threadIdx.x] = fx_to_f(__ldg(q + 2 * o0));
        if (i1 < RING) ring[slot * RING + i1] = fx_to_f(__ldg(q + 2 * o1));
    };
    auto plane = [&](int slot) {
        const float* at = ring + slot * RING + (ty + 1) * RING_W + tx + 1;
        return plane_of([&](int dy, int dx) { return at[dy * RING_W + dx]; });
    };
    auto moments = [&](int z, int2 (&m)[4]) {
        const int2* q = reinterpret_cast<const int2*>(src + z * pstride);
#pragma unroll
        for (int i = 0; i < 4; ++i) m[i] = __ldg(q + (size_t)i * nxny + cell);
    };
    auto velocity = [&](int z, float (&u)[3]) {
        const float* q = p.uf + (long long)z * nxny + cell;
#pragma unroll
        for (int i = 0; i < 3; ++i) u[i] = UFIELD ? __ldg(q + i * p.N) : p.u[i];
    };

    __shared__ int met_suspect, met_invalid, met_single;
    if (threadIdx.x == 0) met_suspect = met_invalid = met_single = 0;
    int zc = wrapi(z0 - 1, p.nz);  // the plane of k
    fetch(wrapi(z0 - 2, p.nz), 0);
    fetch(zc, 1);
    int2 m[4];
    float u[3];
    moments(zc, m);
    velocity(zc, u);
    __syncthreads();
    Plane lo = plane(0), mid = plane(1);
    __syncthreads();
    int zn = next(zc), zp = next(zn);
    fetch(zn, 0);
    __syncthreads();

    // The moments and the velocity of the thread's cell in the next plane.
    constexpr bool AHEAD = k3_ahead<ROWS, UFIELD>();
    int2* ahead = reinterpret_cast<int2*>(ring + 2 * RING) + threadIdx.x;    // [4][NT]
    float* ahead_u = ring + 2 * RING + 8 * NT + threadIdx.x;                 // [3][NT]
    auto load_ahead = [&](int z) {
        const int2* q = reinterpret_cast<const int2*>(src + z * pstride) + cell;
#pragma unroll
        for (int i = 0; i < 4; ++i) cp_async<8>(ahead + i * NT, q + (size_t)i * nxny);
        if constexpr (UFIELD) {
            const float* v = p.uf + (long long)z * nxny + cell;
#pragma unroll
            for (int i = 0; i < 3; ++i) cp_async<4>(ahead_u + i * NT, v + i * p.N);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };

    // Sums on their way, of f and h: `part` of plane k - 1 (complete but for what
    // comes from plane k), `up` of plane k (what came from plane k - 1).
    uint2 part[4] = {}, up[3] = {};
    int slot = 0;
    for (int k = z0 - 1; k <= z1; ++k) {
        int2 mn[4];
        if constexpr (AHEAD) load_ahead(zn);
        else moments(zn, mn);
        const int* q = src + zp * pstride;
        const int f0 = __ldg(q + 2 * o0), f1 = __ldg(q + 2 * o1);

        uint4* x = xchg + slot * (XCHG / 4) + ty * TILE_W + tx;
        uint2 s0[3], d0[3];  // sums and differences along x of the populations that stay in the row
        Plane hi{0.f, 0.f, 0.f};
        if (ty <= last + 1) {
            hi = plane(slot);
            const Collision r = collide<UFIELD>(p, m, lo, mid, hi, u);
            if (!r.tame) {
                p.suspect[wrapi(k, p.nz)] = p.number;
                met_suspect = 1;
                if (!r.ok()) met_invalid = 1;
                else if (!r.template safe<UFIELD>()) met_single = 1;
            }
            uint2 moved = make_uint2(0u, 0u);
            // populations of y velocity +1 (b = 1) and -1 (b = 2): to the other rows
            auto across = [&](int b) {
                emit_rows<UFIELD, false>(p, r, b, [&](int c, uint2 total, uint2 v1, uint2 v2) {
                    moved = moved + total;
                    const uint2 t1 = from_left(v1), t2 = from_right(v2);
                    const uint2 s = (total - v1 - v2) + t1 + t2, d = t1 - t2;
                    x[(2 * c + b - 1) * PLANE] = make_uint4(s.x, d.x, s.y, d.y);
                });
            };
            if (ty <= last) across(1);
            if (ty >= 1) across(2);
            if (inner) {
                uint2 r1, r2;
                emit_rows<UFIELD, false>(p, r, 0, [&](int c, uint2 total, uint2 v1, uint2 v2) {
                    const uint2 t1 = from_left(v1), t2 = from_right(v2);
                    if (c == 0) {  // the rest population, once the other 26 are known
                        moved = moved + (v1 + v2);
                        r1 = t1;
                        r2 = t2;
                    } else {
                        moved = moved + total;
                        s0[c] = (total - v1 - v2) + t1 + t2;
                        d0[c] = t1 - t2;
                    }
                });
                const uint2 rest = make_uint2((uint32_t)r.s_fx.x, (uint32_t)r.s_fx.y) - moved;
                s0[0] = rest + r1 + r2;
                d0[0] = r1 - r2;
            }
        }
        ring[(slot ^ 1) * RING + threadIdx.x] = fx_to_f(f0);
        if (i1 < RING) ring[(slot ^ 1) * RING + i1] = fx_to_f(f1);
        __syncthreads();
        if (inner) {
            uint2 S[3], JX[3], JY[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const uint4 dn = x[2 * c * PLANE - TILE_W];        // from y - 1
                const uint4 ab = x[(2 * c + 1) * PLANE + TILE_W];  // from y + 1
                S[c] = s0[c] + make_uint2(dn.x, dn.z) + make_uint2(ab.x, ab.z);
                JX[c] = d0[c] + make_uint2(dn.y, dn.w) + make_uint2(ab.y, ab.w);
                JY[c] = make_uint2(dn.x, dn.z) - make_uint2(ab.x, ab.z);
            }
            if (store && k > z0) {
                uint2* out = reinterpret_cast<uint2*>(dst + (k - 1) * pstride) + cell;
                out[0] = part[0] + S[2];
                out[(size_t)nxny] = part[1] + JX[2];
                out[2 * (size_t)nxny] = part[2] + JY[2];
                out[3 * (size_t)nxny] = part[3] - S[2];
            }
            part[0] = up[0] + S[0];
            part[1] = up[1] + JX[0];
            part[2] = up[2] + JY[0];
            part[3] = up[0];
            up[0] = S[1];
            up[1] = JX[1];
            up[2] = JY[1];
        }
        if constexpr (AHEAD) asm volatile("cp.async.wait_group 0;" ::: "memory");
        slot ^= 1;
        lo = mid;
        mid = hi;
        zn = zp;
        zp = next(zp);
#pragma unroll
        for (int i = 0; i < 4; ++i) m[i] = AHEAD ? ahead[i * NT] : mn[i];
        if constexpr (UFIELD) {
#pragma unroll
            for (int i = 0; i < 3; ++i) u[i] = ahead_u[i * NT];
        }
    }
    __syncthreads();
    if (met_suspect) settle<ROWS>(p, src, dst, met_invalid != 0, met_single != 0);
}

// The fields an initial state is made of (velocity null: uniform u).
struct Seed {
    const double *phi, *c, *u[3];
    double W, phi_a, phi_b, M_phi, D_s;
};

// Discrete equilibria of the given fields at one cell, in FP64, rounded to the
// grid (FX_BAD for what is not finite or out of range): out(q, f, h).
template <class Out>
__device__ __forceinline__ void equilibrium(const K3Params& p, const Seed& in, long long cell, Out out) {
    const int x = (int)(cell % p.nx);
    const int y = (int)((cell / p.nx) % p.ny);
    const int z = (int)(cell / p.nxny);
    const double w1[3] = {1.0 / 6.0, 2.0 / 3.0, 1.0 / 6.0};
    double g[3] = {0.0, 0.0, 0.0};
    for (int dz = -1; dz <= 1; ++dz)
        for (int dy = -1; dy <= 1; ++dy)
            for (int dx = -1; dx <= 1; ++dx) {
                const double v = in.phi[((long long)wrapi(z + dz, p.nz) * p.ny + wrapi(y + dy, p.ny)) * p.nx +
                                        wrapi(x + dx, p.nx)];
                const double w = 3.0 * w1[dx + 1] * w1[dy + 1] * w1[dz + 1];
                g[0] += w * dx * v;
                g[1] += w * dy * v;
                g[2] += w * dz * v;
            }
    const double m = sqrt(g[0] * g[0] + g[1] * g[1] + g[2] * g[2]);
    double n[3];
    for (int i = 0; i < 3; ++i) n[i] = m > 1e-12 ? g[i] / m : 0.0;
    const double ph = in.phi[cell], cc = in.c[cell];
    const double dphi = in.phi_a - in.phi_b;
    const double theta = (4.0 / in.W) * (in.phi_a - ph) * (ph - in.phi_b) / dphi;
    const double thetac = (8.0 * cc / in.W) * (0.5 * (in.phi_a + in.phi_b) - ph) / dphi;
    double u[3] = {p.u[0], p.u[1], p.u[2]};
    if (in.u[0])
        for (int i = 0; i < 3; ++i) u[i] = in.u[i][cell];
    double Ax[3], Bx[3], Cx[3], Ay[3], By[3], Cy[3], Az[3], Bz[3], Cz[3];
    axis_factors(u[0], Ax, Bx, Cx);
    axis_factors(u[1], Ay, By, Cy);
    axis_factors(u[2], Az, Bz, Cz);
    const double qf = in.M_phi * theta, qh = in.D_s * thetac;
    const bool ok = fabs(ph) < (double)S_MAX && fabs(cc) < (double)S_MAX;
    auto fx = [&](double v) { return ok && fabs(v) < 8.0 ? (int)__double2ll_rn(v * FX_ONE_D) : FX_BAD; };
    int f[Q27];
    emit27(Ax, Bx, Cx, Ay, By, Cy, Az, Bz, Cz, ph, qf * n[0], qf * n[1], qf * n[2],
           [&](int q, double v) { f[q] = fx(v); });
    emit27(Ax, Bx, Cx, Ay, By, Cy, Az, Bz, Cz, cc, qh * n[0], qh * n[1], qh * n[2],
           [&](int q, double v) { out(q, f[q], fx(v)); });
}

// The state of the given fields, and a copy of the fields (see `Seed`).
__global__ void k3_init(const K3Params p, const Seed in, int* __restrict__ state, double* __restrict__ keep,
                        float* __restrict__ uf) {
    const long long N = p.N;
    for (long long cell = blockIdx.x * (long long)blockDim.x + threadIdx.x; cell < N;
         cell += (long long)gridDim.x * blockDim.x) {
        keep[cell] = in.phi[cell];
        keep[N + cell] = in.c[cell];
        if (in.u[0])
            for (int i = 0; i < 3; ++i) {
                const double v = in.u[i][cell];
                keep[(2 + i) * N + cell] = v;
                uf[i * N + cell] = (float)v;
            }
        uint2 m[4] = {};
        bool bad_f = false, bad_h = false;
        equilibrium(p, in, cell, [&](int q, int f, int h) {
            bad_f |= f == FX_BAD;
            bad_h |= h == FX_BAD;
            const int e[3] = {q % 3, (q / 3) % 3, q / 9};
            const uint2 v = make_uint2((uint32_t)f, (uint32_t)h);
            m[0] = m[0] + v;
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                if (e[i] == 1) m[1 + i] = m[1 + i] + v;
                if (e[i] == 2) m[1 + i] = m[1 + i] - v;
            }
        });
        if (bad_f) m[0].x = (uint32_t)FX_BAD;
        if (bad_h) m[0].y = (uint32_t)FX_BAD;
        uint2* o = reinterpret_cast<uint2*>(state) + (cell / p.nxny) * 4 * p.nxny + cell % p.nxny;
#pragma unroll
        for (int i = 0; i < 4; ++i) o[i * p.nxny] = m[i];
        if (bad_f || bad_h) p.suspect[cell / p.nxny] = p.suspect[p.nz] = p.number;
    }
}

// phi and c of the state: exact integer sums, then FP64 (NaN where a population is
// FX_BAD).
__global__ void k3_fields(const K3Params p, const int* __restrict__ state, double* __restrict__ phi,
                          double* __restrict__ c) {
    const int nxny = (int)p.nxny;
    for (long long cell = blockIdx.x * (long long)blockDim.x + threadIdx.x; cell < p.N;
         cell += (long long)gridDim.x * blockDim.x) {
        const int2 s = reinterpret_cast<const int2*>(state)[cell + cell / nxny * 3 * nxny];
        if (phi) phi[cell] = s.x == FX_BAD ? nan("") : (double)s.x * FX_INV_D;
        if (c) c[cell] = s.y == FX_BAD ? nan("") : (double)s.y * FX_INV_D;
    }
}

// The same for the cells next to a suspect plane of `prev`, the state one step back,
// whose sums may have wrapped around: multiples of 2^32 are added back.  The block
// forms the populations of a tile and its halo once and adds them up coarsely, in
// units of 2^6, which fits 32 bits; the state has the rest.
constexpr int FT_X = 16, FT_Y = 8, FT_Z = 4, FT_N = FT_X * FT_Y * FT_Z;
__global__ void __launch_bounds__(256) k3_fields_suspect(const K3Params p, const int* prev,
                                                         const int* __restrict__ state, double* __restrict__ phi,
                                                         double* __restrict__ c) {
    if (p.suspect[p.nz] != p.number) return;
    __shared__ int coarse[2][FT_N];
    const int tiles_x = (p.nx + FT_X - 1) / FT_X, tiles_y = (p.ny + FT_Y - 1) / FT_Y, tiles_z = (p.nz + FT_Z - 1) / FT_Z;
    for (long long tile = blockIdx.x; tile < (long long)tiles_x * tiles_y * tiles_z; tile += gridDim.x) {
        const int x0 = (int)(tile % tiles_x) * FT_X, y0 = (int)(tile / tiles_x % tiles_y) * FT_Y,
                  z0 = (int)(tile / tiles_x / tiles_y) * FT_Z;
        const int plane = wrapi(z0 - 1 + (int)threadIdx.x, p.nz);
        if (!__syncthreads_or(threadIdx.x < FT_Z + 2 && p.suspect[plane] == p.number)) continue;
        for (int k = threadIdx.x; k < FT_N; k += 256) coarse[0][k] = coarse[1][k] = 0;
        __syncthreads();
        for (int k = threadIdx.x; k < (FT_X + 2) * (FT_Y + 2) * (FT_Z + 2); k += 256) {
            const int lx = k % (FT_X + 2) - 1, ly = k / (FT_X + 2) % (FT_Y + 2) - 1, lz = k / (FT_X + 2) / (FT_Y + 2) - 1;
            if (x0 + lx > p.nx || y0 + ly > p.ny || z0 + lz > p.nz) continue;
            outgoing(p, prev, wrapi(x0 + lx, p.nx), wrapi(y0 + ly, p.ny), wrapi(z0 + lz, p.nz), [&](int q, int f, int h) {
                const int rx = lx + vel(q % 3), ry = ly + vel((q / 3) % 3), rz = lz + vel(q / 9);
                if (rx < 0 || rx >= FT_X || ry < 0 || ry >= FT_Y || rz < 0 || rz >= FT_Z) return;
                const int at = (rz * FT_Y + ry) * FT_X + rx;
                atomicAdd(&coarse[0][at], f >> 6);
                atomicAdd(&coarse[1][at], h >> 6);
            });
        }
        __syncthreads();
        for (int k = threadIdx.x; k < FT_N; k += 256) {
            const int x = x0 + k % FT_X, y = y0 + k / FT_X % FT_Y, z = z0 + k / FT_X / FT_Y;
            if (x >= p.nx || y >= p.ny || z >= p.nz) continue;
            const long long at = (long long)y * p.nx + x, cell = z * p.nxny + at;
            const int2 s = reinterpret_cast<const int2*>(state)[4 * p.nxny * z + at];
            // 27 populations lose less than 27 * 2^6 to the coarse units
            auto whole = [](int sum, int in64) {
                return (double)(sum + (((64LL * in64 - sum + 0xffffffffLL) >> 32) << 32)) * FX_INV_D;
            };
            if (phi && s.x != FX_BAD) phi[cell] = whole(s.x, coarse[0][k]);
            if (c && s.y != FX_BAD) c[cell] = whole(s.y, coarse[1][k]);
        }
        __syncthreads();
    }
}

// The state's populations as float64 [27][N] (NaN for FX_BAD): of the initial
// fields (prev null), or sent by the state before to the cells they reached.
__global__ void k3_pops(const K3Params p, const Seed seed, const int* prev, double* __restrict__ f,
                        double* __restrict__ h) {
    for (long long cell = blockIdx.x * (long long)blockDim.x + threadIdx.x; cell < p.N;
         cell += (long long)gridDim.x * blockDim.x) {
        auto put = [&](long long i, int a, int b) {
            if (f) f[i] = a == FX_BAD ? nan("") : (double)a * FX_INV_D;
            if (h) h[i] = b == FX_BAD ? nan("") : (double)b * FX_INV_D;
        };
        if (!prev) {
            equilibrium(p, seed, cell, [&](int q, int a, int b) { put(q * p.N + cell, a, b); });
            continue;
        }
        const int x = (int)(cell % p.nx), y = (int)((cell / p.nx) % p.ny), z = (int)(cell / p.nxny);
        outgoing(p, prev, x, y, z, [&](int q, int a, int b) {
            const int tx = wrapi(x + vel(q % 3), p.nx), ty = wrapi(y + vel((q / 3) % 3), p.ny),
                      tz = wrapi(z + vel(q / 9), p.nz);
            put(q * p.N + ((long long)tz * p.ny + ty) * p.nx + tx, a, b);
        });
    }
}

// Invalid populations of a cell (out of those it sent in the last step, or of
// its initial ones) and the sums of its valid ones.
__device__ __noinline__ void totals_of_populations(const K3Params& p, const Seed& seed, const int* prev,
                                                   long long cell, long long& sf, long long& sh, long long& bad) {
    auto add = [&](int, int f, int h) {
        if (f != FX_BAD) sf += f; else bad += 1;
        if (h != FX_BAD) sh += h; else bad += 1;
    };
    if (!prev)
        equilibrium(p, seed, cell, add);
    else
        outgoing(p, prev, (int)(cell % p.nx), (int)((cell / p.nx) % p.ny), (int)(cell / p.nxny), add);
}

// Totals: sum f, sum h (exact, in integer units) and the FX_BAD count of the
// state's populations (streaming is a permutation: those sent are those that
// arrived, and a cell's add up to its zeroth moment unless its plane is suspect).
// Fixed grid and reduction order.
__global__ void __launch_bounds__(SUM_THREADS) k3_sum1(const K3Params p, const Seed seed,
                                                       const int* __restrict__ state, const int* prev,
                                                       long long* __restrict__ partial) {
    long long sf = 0, sh = 0, bad = 0;
    const int nxny = (int)p.nxny;
    const int* sent = prev ? prev : state;
    for (long long cell = blockIdx.x * (long long)SUM_THREADS + threadIdx.x; cell < p.N;
         cell += (long long)SUM_BLOCKS * SUM_THREADS) {
        const long long z = cell / nxny;
        if (p.suspect[z] == p.number) {
            totals_of_populations(p, seed, prev, cell, sf, sh, bad);
            continue;
        }
        const int2 s = reinterpret_cast<const int2*>(sent)[cell + z * 3 * nxny];
        sf += s.x;
        sh += s.y;
    }
    __shared__ long long red[3][SUM_THREADS];
    red[0][threadIdx.x] = sf;
    red[1][threadIdx.x] = sh;
    red[2][threadIdx.x] = bad;
    __syncthreads();
    for (int w = SUM_THREADS / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w)
            for (int k = 0; k < 3; ++k) red[k][threadIdx.x] += red[k][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x < 3) partial[3 * blockIdx.x + threadIdx.x] = red[threadIdx.x][0];
}

__global__ void __launch_bounds__(SUM_THREADS) k3_sum2(const long long* __restrict__ partial,
                                                       double* __restrict__ out) {
    __shared__ long long red[3][SUM_THREADS];
    long long acc[3] = {0, 0, 0};
    for (int b = threadIdx.x; b < SUM_BLOCKS; b += SUM_THREADS)
        for (int k = 0; k < 3; ++k) acc[k] += partial[3 * b + k];
    for (int k = 0; k < 3; ++k) red[k][threadIdx.x] = acc[k];
    __syncthreads();
    for (int w = SUM_THREADS / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w)
            for (int k = 0; k < 3; ++k) red[k][threadIdx.x] += red[k][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x < 3) out[threadIdx.x] = threadIdx.x < 2 ? (double)red[threadIdx.x][0] * FX_INV_D
                                                            : (double)red[threadIdx.x][0];
}

}  // namespace

struct lbm3_ctx {
    lbm3_params p;
    K3Params kp;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    int* buf[2] = {nullptr, nullptr};    // states, [nz][4][ny][nx][2] fixed point: now and one step back
    float* uf = nullptr;                 // [3][N] prescribed velocity (velocity_field = 1)
    double* keep = nullptr;              // the initial fields, [2][N] or [5][N] with the velocity
    long long* suspect = nullptr;        // see K3Params
    long long* partial = nullptr;        // 3 x SUM_BLOCKS partial sums
    double* result = nullptr;            // 3 totals
    int cur = 0;
    int sms = 1;
    int rows = 10, seg_z = 64;
    int64_t step = 0;
    int pending_error = LBM_OK;
};

namespace {

int fail(lbm3_ctx* ctx, cudaError_t e) {
    if (e == cudaSuccess) return LBM_OK;
    if (ctx) ctx->pending_error = LBM_ERR_CUDA;
    return e == cudaErrorMemoryAllocation ? LBM_ERR_NOMEM : LBM_ERR_CUDA;
}

double rate_of(double coeff) { return 1.0 / (coeff * 3.0 + 0.5); }

// The initial fields kept by the context.
Seed seed_of(const lbm3_ctx* ctx) {
    const lbm3_params& p = ctx->p;
    const long long N = ctx->kp.N;
    Seed s{ctx->keep, ctx->keep + N, {nullptr, nullptr, nullptr}, p.W, p.phi_a, p.phi_b, p.M_phi, p.D_s};
    if (p.velocity_field)
        for (int i = 0; i < 3; ++i) s.u[i] = ctx->keep + (2 + i) * N;
    return s;
}

// The parameters of a kernel that reads the state.
K3Params of_state(const lbm3_ctx* ctx) {
    K3Params p = ctx->kp;
    p.number = ctx->step;
    return p;
}

// The state one step back, or null if the state is the initial one.
const int* before(const lbm3_ctx* ctx) { return ctx->step ? ctx->buf[1 - ctx->cur] : nullptr; }

int grid_1d(const lbm3_ctx* ctx, long long n, int threads) {
    const long long b = (n + threads - 1) / threads;
    return (int)std::min(std::max(b, 1LL), 16LL * ctx->sms);
}

int sm_count() {
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        cudaGetLastError();  // (creating the context will report it)
    return n > 0 ? n : 1;
}

// Shared memory above 48 KB has to be asked for, once per kernel and device.
template <int ROWS>
cudaError_t allow_smem(bool field) {
    return field ? cudaFuncSetAttribute(k3_step<ROWS, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        k3_smem<ROWS, true>())
                 : cudaFuncSetAttribute(k3_step<ROWS, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        k3_smem<ROWS, false>());
}

int launch_step(lbm3_ctx* ctx) {
    const K3Params& kp = ctx->kp;
    K3Params p = kp;
    p.seg_z = ctx->seg_z;
    p.number = ctx->step + 1;
    const int rows = ctx->rows;
    dim3 grid((kp.nx + TILE_IN - 1) / TILE_IN, (kp.ny + rows - 3) / (rows - 2),
              (kp.nz + ctx->seg_z - 1) / ctx->seg_z);
    const int src = ctx->cur, dst = 1 - ctx->cur;
    const bool field = kp.uf != nullptr;
    auto go = [&](auto kern, int smem) {
        kern<<<grid, rows * 32, smem, ctx->stream>>>(p, ctx->buf[src], ctx->buf[dst]);
    };
    switch (rows) {
        case 6:
            field ? go(k3_step<6, true>, k3_smem<6, true>()) : go(k3_step<6, false>, k3_smem<6, false>());
            break;
        case 10:
            field ? go(k3_step<10, true>, k3_smem<10, true>()) : go(k3_step<10, false>, k3_smem<10, false>());
            break;
        case 18:
            field ? go(k3_step<18, true>, k3_smem<18, true>()) : go(k3_step<18, false>, k3_smem<18, false>());
            break;
        default:
            return LBM_ERR_INVALID_ARG;
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return fail(ctx, e);
    ctx->cur = dst;
    ctx->step += 1;
    return LBM_OK;
}

// The launch shape of a context whose user sets none.  A block spends seg_z + 3
// planes' time (the halo planes and the first loads), so the best segments make
// the blocks of an SM times that the least.  In units of a plane of 10 rows alone
// on an SM, a plane of 18 rows takes 1.45, and a second block of 10 rows beside the
// first 0.45 (0.75 with a velocity field).  Measured, us per step at the shape this
// takes / at the best segments of 18 / of 10 rows: uniform velocity 256^3 503 / 516 /
// 487, 150x97x61 39 / 39 / 39, 64x50x40 14.4 / 16.5 / 14.5; velocity field 256^3 602 /
// 602 / 576, 220x200x180 331 / 305 / 293, 150x97x61 47 / 47 / 47.  (With a field it
// weighs 10 rows as they were before the moments came by way of shared memory.)
void default_shape(const lbm3_params* p, int sms, int* rows, int* seg_z) {
    const double second = p->velocity_field ? 1.75 : 1.45;
    double best = -1.0;
    for (int r : {10, 18}) {
        const long long tiles = (long long)((p->nx + TILE_IN - 1) / TILE_IN) * ((p->ny + r - 3) / (r - 2));
        // the distinct heights of nz planes in n segments, each with its smallest n (about
        // 2 sqrt(nz) of them)
        for (int n = 1, seg = 0; seg != 1; n = (int)((seg - 2LL + p->nz) / std::max(seg - 1, 1))) {
            seg = (int)((n - 1LL + p->nz) / n);
            const long long blocks = tiles * ((seg - 1LL + p->nz) / seg), per_sm = (blocks + sms - 1) / sms;
            const double load = r == 18 ? 1.45 * (double)per_sm : second * (double)(per_sm / 2) + (double)(per_sm % 2);
            const double cost = load * (seg + 3);
            if (best < 0.0 || cost < best) {
                best = cost;
                *rows = r;
                *seg_z = seg;
            }
        }
    }
}

bool finite_all(const double* v, int n) {
    for (int i = 0; i < n; ++i)
        if (!std::isfinite(v[i])) return false;
    return true;
}

}  // namespace

extern "C" {

int lbm3_params_default(lbm3_params* p) {
    if (!p) return LBM_ERR_INVALID_ARG;
    std::memset(p, 0, sizeof(*p));
    p->W = 4.0;
    p->phi_a = 1.0;
    p->phi_b = 0.0;
    p->M_phi = 0.1;
    p->D_s = 0.1;
    return LBM_OK;
}

int lbm3_create(const lbm3_params* p, void* stream, lbm3_ctx** out) {
    if (!p || !out) return LBM_ERR_INVALID_ARG;
    *out = nullptr;
    if (p->nx < 1 || p->ny < 1 || p->nz < 1) return LBM_ERR_INVALID_ARG;
    if ((long long)p->nx * p->ny * p->nz > LBM3_MAX_CELLS) return LBM_ERR_INVALID_ARG;
    if (27LL * p->nx * p->ny > 2147483647LL) return LBM_ERR_INVALID_ARG;  // 32-bit in-plane offsets
    if (p->velocity_field != 0 && p->velocity_field != 1) return LBM_ERR_INVALID_ARG;
    const double vals[8] = {p->W, p->phi_a, p->phi_b, p->M_phi, p->D_s, p->u[0], p->u[1], p->u[2]};
    if (!finite_all(vals, 8) || !(p->W > 0.0) || p->phi_a == p->phi_b) return LBM_ERR_INVALID_ARG;
    if (std::fabs(p->phi_a) > 2.0 || std::fabs(p->phi_b) > 2.0) return LBM_ERR_INVALID_ARG;
    if (std::fabs(p->u[0]) >= 0.5 || std::fabs(p->u[1]) >= 0.5 || std::fabs(p->u[2]) >= 0.5)
        return LBM_ERR_INVALID_ARG;
    if (!(p->M_phi > 0.0) || !(p->D_s > 0.0)) return LBM_ERR_RATE;
    lbm3_ctx* ctx = new (std::nothrow) lbm3_ctx();
    if (!ctx) return LBM_ERR_NOMEM;
    ctx->p = *p;
    K3Params& kp = ctx->kp;
    kp.nx = p->nx;
    kp.ny = p->ny;
    kp.nz = p->nz;
    kp.nxny = (long long)p->nx * p->ny;
    kp.N = kp.nxny * p->nz;
    kp.w_kappa = (float)rate_of(p->M_phi);
    kp.w_chi = (float)rate_of(p->D_s);
    kp.M_phi = (float)p->M_phi;
    kp.D_s = (float)p->D_s;
    kp.c4W = (float)(4.0 / p->W);
    kp.c8W = (float)(8.0 / p->W);
    kp.phi_a = (float)p->phi_a;
    kp.phi_b = (float)p->phi_b;
    kp.phim = (float)(0.5 * (p->phi_a + p->phi_b));
    kp.inv_dphi = (float)(1.0 / (p->phi_a - p->phi_b));
    double fac[3][3][3];  // [axis][A, B, C][e = 0, +1, -1]
    for (int i = 0; i < 3; ++i) {
        kp.u[i] = (float)p->u[i];
        axis_factors(p->u[i], fac[i][0], fac[i][1], fac[i][2]);
    }
    auto both = [](double v) { return make_float2((float)v, (float)v); };
    const double ux = p->u[0];
    kp.fx[0] = both(0.5 * (1.0 / 3.0 + ux * ux));
    kp.fx[1] = both(2.0 * ux);
    kp.fx[2] = both(0.5 * ux * ux);
    kp.fx[3] = both(0.5 * ux);
    for (int c = 0; c < 3; ++c)
        for (int b = 0; b < 3; ++b) {
            kp.aa[c][b] = both(fac[1][0][b] * fac[2][0][c]);
            kp.cc[c][b] = both(0.5 * fac[1][2][b] * fac[2][2][c]);
            kp.bc[c][b] = both(fac[1][1][b] * fac[2][2][c]);
            kp.cb[c][b] = both(fac[1][2][b] * fac[2][1][c]);
        }
    kp.uf = nullptr;
    ctx->sms = sm_count();
    default_shape(p, ctx->sms, &ctx->rows, &ctx->seg_z);
    cudaError_t e = cudaSuccess;
    if (stream) {
        ctx->stream = (cudaStream_t)stream;
    } else {
        e = cudaStreamCreateWithFlags(&ctx->stream, cudaStreamNonBlocking);
        ctx->own_stream = e == cudaSuccess;
    }
    const size_t state_bytes = sizeof(int) * 8 * (size_t)kp.N;
    const size_t keep_bytes = sizeof(double) * (p->velocity_field ? 5 : 2) * (size_t)kp.N;
    for (int i = 0; i < 2 && e == cudaSuccess; ++i) e = cudaMalloc(&ctx->buf[i], state_bytes);
    if (e == cudaSuccess) e = cudaMalloc(&ctx->keep, keep_bytes);
    const size_t suspect_bytes = sizeof(long long) * ((size_t)p->nz + 1);
    if (e == cudaSuccess) e = cudaMalloc(&ctx->suspect, suspect_bytes);
    if (e == cudaSuccess && p->velocity_field) e = cudaMalloc(&ctx->uf, sizeof(float) * 3 * (size_t)kp.N);
    if (e == cudaSuccess) e = cudaMalloc(&ctx->partial, sizeof(long long) * 3 * SUM_BLOCKS);
    if (e == cudaSuccess) e = cudaMalloc(&ctx->result, sizeof(double) * 3);
    // defined contents before the first init (the autotuner may step them)
    for (int i = 0; i < 2 && e == cudaSuccess; ++i) e = cudaMemsetAsync(ctx->buf[i], 0, state_bytes, ctx->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(ctx->keep, 0, keep_bytes, ctx->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(ctx->suspect, 0xff, suspect_bytes, ctx->stream);
    if (e == cudaSuccess && ctx->uf) e = cudaMemsetAsync(ctx->uf, 0, sizeof(float) * 3 * (size_t)kp.N, ctx->stream);
    const bool field = p->velocity_field != 0;
    if (e == cudaSuccess) e = allow_smem<6>(field);
    if (e == cudaSuccess) e = allow_smem<10>(field);
    if (e == cudaSuccess) e = allow_smem<18>(field);
    if (e != cudaSuccess) {
        const int rc = fail(nullptr, e);
        lbm3_destroy(ctx);
        cudaGetLastError();
        return rc;
    }
    kp.uf = ctx->uf;
    kp.suspect = ctx->suspect;
    *out = ctx;
    return LBM_OK;
}

void lbm3_destroy(lbm3_ctx* ctx) {
    if (!ctx) return;
    if (ctx->stream) cudaStreamSynchronize(ctx->stream);
    for (int i = 0; i < 2; ++i) cudaFree(ctx->buf[i]);
    cudaFree(ctx->uf);
    cudaFree(ctx->keep);
    cudaFree(ctx->suspect);
    cudaFree(ctx->partial);
    cudaFree(ctx->result);
    if (ctx->own_stream) cudaStreamDestroy(ctx->stream);
    delete ctx;
}

int lbm3_init_fields_device(lbm3_ctx* ctx, const double* phi, const double* c, const double* ux,
                            const double* uy, const double* uz) {
    if (!ctx || !phi || !c) return LBM_ERR_INVALID_ARG;
    const bool field = ctx->p.velocity_field != 0;
    if (field && (!ux || !uy || !uz)) return LBM_ERR_INVALID_ARG;
    Nvtx r("lbm3_init_fields");
    const lbm3_params& p = ctx->p;
    Seed in{phi, c, {nullptr, nullptr, nullptr}, p.W, p.phi_a, p.phi_b, p.M_phi, p.D_s};
    if (field) {
        in.u[0] = ux;
        in.u[1] = uy;
        in.u[2] = uz;
    }
    const cudaError_t e =
        cudaMemsetAsync(ctx->suspect, 0xff, sizeof(long long) * ((size_t)ctx->kp.nz + 1), ctx->stream);
    if (e != cudaSuccess) return fail(ctx, e);
    ctx->cur = 0;
    ctx->step = 0;
    k3_init<<<grid_1d(ctx, ctx->kp.N, 256), 256, 0, ctx->stream>>>(of_state(ctx), in, ctx->buf[0], ctx->keep, ctx->uf);
    return fail(ctx, cudaGetLastError());
}

int lbm3_init_fields(lbm3_ctx* ctx, const double* phi, const double* c, const double* ux,
                     const double* uy, const double* uz) {
    if (!ctx || !phi || !c) return LBM_ERR_INVALID_ARG;
    const bool field = ctx->p.velocity_field != 0;
    if (field && (!ux || !uy || !uz)) return LBM_ERR_INVALID_ARG;
    const size_t bytes = sizeof(double) * (size_t)ctx->kp.N;
    const int nin = field ? 5 : 2;
    const double* host[5] = {phi, c, ux, uy, uz};
    double* dev = nullptr;
    cudaError_t e = cudaMallocAsync(&dev, bytes * nin, ctx->stream);
    if (e != cudaSuccess) return fail(ctx, e);
    for (int i = 0; i < nin && e == cudaSuccess; ++i)
        e = cudaMemcpyAsync(dev + i * (size_t)ctx->kp.N, host[i], bytes, cudaMemcpyHostToDevice, ctx->stream);
    int rc = e == cudaSuccess ? LBM_OK : fail(ctx, e);
    if (rc == LBM_OK) {
        const size_t n = ctx->kp.N;
        rc = lbm3_init_fields_device(ctx, dev, dev + n, field ? dev + 2 * n : nullptr,
                                     field ? dev + 3 * n : nullptr, field ? dev + 4 * n : nullptr);
    }
    cudaFreeAsync(dev, ctx->stream);
    const int sync = lbm3_synchronize(ctx);
    return rc != LBM_OK ? rc : sync;
}

int lbm3_step(lbm3_ctx* ctx, int64_t nsteps) {
    if (!ctx || nsteps < 0) return LBM_ERR_INVALID_ARG;
    Nvtx r("lbm3_step");
    for (int64_t s = 0; s < nsteps; ++s) {
        const int rc = launch_step(ctx);
        if (rc != LBM_OK) return rc;
    }
    return LBM_OK;
}

int lbm3_get_fields_device(lbm3_ctx* ctx, double* phi, double* c) {
    if (!ctx) return LBM_ERR_INVALID_ARG;
    if (!phi && !c) return LBM_OK;
    const K3Params p = of_state(ctx);
    k3_fields<<<grid_1d(ctx, p.N, 256), 256, 0, ctx->stream>>>(p, ctx->buf[ctx->cur], phi, c);
    if (before(ctx))
        // (four blocks an SM: usually they find nothing to do)
        k3_fields_suspect<<<std::min(grid_1d(ctx, p.N, FT_N), 4 * ctx->sms), 256, 0, ctx->stream>>>(
            p, before(ctx), ctx->buf[ctx->cur], phi, c);
    return fail(ctx, cudaGetLastError());
}

int lbm3_get_fields(lbm3_ctx* ctx, double* phi, double* c) {
    if (!ctx) return LBM_ERR_INVALID_ARG;
    if (!phi && !c) return LBM_OK;
    const size_t n = ctx->kp.N, bytes = sizeof(double) * n;
    double* dev = nullptr;
    cudaError_t e = cudaMallocAsync(&dev, 2 * bytes, ctx->stream);
    if (e != cudaSuccess) return fail(ctx, e);
    int rc = lbm3_get_fields_device(ctx, dev, dev + n);
    if (rc == LBM_OK && phi) rc = fail(ctx, cudaMemcpyAsync(phi, dev, bytes, cudaMemcpyDeviceToHost, ctx->stream));
    if (rc == LBM_OK && c) rc = fail(ctx, cudaMemcpyAsync(c, dev + n, bytes, cudaMemcpyDeviceToHost, ctx->stream));
    cudaFreeAsync(dev, ctx->stream);
    const int sync = lbm3_synchronize(ctx);
    return rc != LBM_OK ? rc : sync;
}

int lbm3_get_populations_device(lbm3_ctx* ctx, double* f, double* h) {
    if (!ctx) return LBM_ERR_INVALID_ARG;
    if (!f && !h) return LBM_OK;
    k3_pops<<<grid_1d(ctx, ctx->kp.N, 256), 256, 0, ctx->stream>>>(ctx->kp, seed_of(ctx), before(ctx), f, h);
    return fail(ctx, cudaGetLastError());
}

int lbm3_get_populations(lbm3_ctx* ctx, double* f, double* h) {
    if (!ctx) return LBM_ERR_INVALID_ARG;
    if (!f && !h) return LBM_OK;
    const size_t n = (size_t)Q27 * ctx->kp.N, bytes = sizeof(double) * n;
    double* dev = nullptr;
    cudaError_t e = cudaMallocAsync(&dev, 2 * bytes, ctx->stream);
    if (e != cudaSuccess) return fail(ctx, e);
    int rc = lbm3_get_populations_device(ctx, dev, dev + n);
    if (rc == LBM_OK && f) rc = fail(ctx, cudaMemcpyAsync(f, dev, bytes, cudaMemcpyDeviceToHost, ctx->stream));
    if (rc == LBM_OK && h) rc = fail(ctx, cudaMemcpyAsync(h, dev + n, bytes, cudaMemcpyDeviceToHost, ctx->stream));
    cudaFreeAsync(dev, ctx->stream);
    const int sync = lbm3_synchronize(ctx);
    return rc != LBM_OK ? rc : sync;
}

int lbm3_sums(lbm3_ctx* ctx, double out[3]) {
    if (!ctx || !out) return LBM_ERR_INVALID_ARG;
    k3_sum1<<<SUM_BLOCKS, SUM_THREADS, 0, ctx->stream>>>(of_state(ctx), seed_of(ctx), ctx->buf[ctx->cur],
                                                         before(ctx), ctx->partial);
    k3_sum2<<<1, SUM_THREADS, 0, ctx->stream>>>(ctx->partial, ctx->result);
    int rc = fail(ctx, cudaGetLastError());
    if (rc == LBM_OK)
        rc = fail(ctx, cudaMemcpyAsync(out, ctx->result, 3 * sizeof(double), cudaMemcpyDeviceToHost,
                                       ctx->stream));
    const int sync = lbm3_synchronize(ctx);
    return rc != LBM_OK ? rc : sync;
}

int lbm3_velocities(int32_t out[81]) {
    if (!out) return LBM_ERR_INVALID_ARG;
    const int E[3] = {0, 1, -1};
    for (int q = 0; q < Q27; ++q) {
        out[3 * q + 0] = E[q % 3];
        out[3 * q + 1] = E[(q / 3) % 3];
        out[3 * q + 2] = E[q / 9];
    }
    return LBM_OK;
}

int lbm3_synchronize(lbm3_ctx* ctx) {
    if (!ctx) return LBM_ERR_INVALID_ARG;
    cudaError_t e = cudaStreamSynchronize(ctx->stream);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) return fail(ctx, e);
    const int pend = ctx->pending_error;
    ctx->pending_error = LBM_OK;
    return pend;
}

int64_t lbm3_get_step(const lbm3_ctx* ctx) { return ctx ? ctx->step : -1; }

int lbm3_set_launch_shape(lbm3_ctx* ctx, int32_t rows, int32_t seg_z) {
    if (!ctx) return LBM_ERR_INVALID_ARG;
    if (rows != 0 && rows != 6 && rows != 10 && rows != 18) return LBM_ERR_INVALID_ARG;
    if (seg_z < 0) return LBM_ERR_INVALID_ARG;
    if (rows) ctx->rows = rows;
    if (seg_z) ctx->seg_z = seg_z < ctx->kp.nz ? seg_z : ctx->kp.nz;
    return LBM_OK;
}

int lbm3_get_launch_shape(const lbm3_ctx* ctx, int32_t* rows, int32_t* seg_z) {
    if (!ctx) return LBM_ERR_INVALID_ARG;
    if (rows) *rows = ctx->rows;
    if (seg_z) *seg_z = ctx->seg_z;
    return LBM_OK;
}

int lbm3_autotune(lbm3_ctx* ctx, int32_t steps, int32_t* rows_out, int32_t* seg_out, double* ms_out) {
    if (!ctx || steps < 1) return LBM_ERR_INVALID_ARG;
    Nvtx r("lbm3_autotune");
    // (rows, planes) worth a timing: the shape it comes with, then a ladder
    std::pair<int, int> shapes[19] = {{ctx->rows, ctx->seg_z}};
    int nshapes = 1;
    for (int rows : {6, 10, 18})
        for (int seg : {4, 8, 16, 32, 64, ctx->kp.nz}) {
            const std::pair<int, int> sh{rows, std::min(seg, ctx->kp.nz)};
            if (std::find(shapes, shapes + nshapes, sh) == shapes + nshapes) shapes[nshapes++] = sh;
        }
    cudaEvent_t ev[2];
    if (cudaEventCreate(&ev[0]) != cudaSuccess) return fail(ctx, cudaGetLastError());
    if (cudaEventCreate(&ev[1]) != cudaSuccess) {
        cudaEventDestroy(ev[0]);
        return fail(ctx, cudaGetLastError());
    }
    double best = -1.0;
    int best_rows = ctx->rows, best_seg = ctx->seg_z;
    int rc = LBM_OK;
    for (int k = 0; k < nshapes; ++k) {
        const std::pair<int, int> sh = shapes[k];
        ctx->rows = sh.first;
        ctx->seg_z = sh.second;
        rc = launch_step(ctx);  // warm-up
        if (rc != LBM_OK) break;
        cudaEventRecord(ev[0], ctx->stream);
        for (int s = 0; s < steps && rc == LBM_OK; ++s) rc = launch_step(ctx);
        cudaEventRecord(ev[1], ctx->stream);
        if (rc != LBM_OK) break;
        cudaError_t e = cudaEventSynchronize(ev[1]);
        if (e != cudaSuccess) {
            rc = fail(ctx, e);
            break;
        }
        float ms = 0.f;
        cudaEventElapsedTime(&ms, ev[0], ev[1]);
        const double per = ms / steps;
        if (best < 0.0 || per < best) {
            best = per;
            best_rows = sh.first;
            best_seg = sh.second;
        }
    }
    cudaEventDestroy(ev[0]);
    cudaEventDestroy(ev[1]);
    ctx->rows = best_rows;
    ctx->seg_z = best_seg;
    if (rc != LBM_OK) return rc;
    if (rows_out) *rows_out = best_rows;
    if (seg_out) *seg_out = best_seg;
    if (ms_out) *ms_out = best;
    return lbm3_synchronize(ctx);
}

}  // extern "C"

// sm_103a kernels of the coupled central-moment LBM step (arXiv 2504.09024).
//
//  * k_fused_sweep  -- the hot path: one launch per time step.  Each block owns
//    a strip of columns (plus a 2-column halo) and sweeps down a segment of
//    rows.  Per row it pulls the three lattices, forms phi, c, sigma(c) and
//    P* into shared-memory row rings, computes the unit normal one row behind,
//    and collides two rows behind with the curvature, Marangoni and pressure
//    stencils read from the rings.  Populations are read once per cell (plus
//    the halo columns and the segment ends) and written once.
//  * k_fields / k_normals / k_collide -- the same step as a three-kernel chain
//    with the fields materialised in global memory; used as a cross-check and
//    for initialisation.
//  * macroscopic outputs and diagnostics (macro_tile), initialisation,
//    population import/export and the count of drops.
#include <cmath>

#include "lbm_cell.cuh"
#include "lbm_tile.cuh"

namespace lbm {

// ---------------------------------------------------------------------------
// three-kernel chain
// ---------------------------------------------------------------------------

template <bool COUPLED>
__global__ void k_fields(KParams p, const float* __restrict__ src, float* __restrict__ F) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y;
    if (i >= p.nx) return;
    const int64_t idx = (int64_t)j * p.pitch + i;
    const uint32_t bits = moment_bits(step_seed(p), i, j, p.nx);
    ScalarMoments m = pull_scalar(src, p, 0, i, j);
    F[FP_PHI * p.plane + idx] = __int_as_float(fx_add_sr(m.s0, m.inc, p.fx_scale[0], bits));
    m = pull_scalar(src + 9 * p.plane, p, 1, i, j);
    const int c_fx = fx_add_sr(m.s0, m.inc, p.fx_scale[1], second_bits(bits));
    F[FP_C * p.plane + idx] = __int_as_float(c_fx);
    F[FP_SIG * p.plane + idx] = sigma_of_c(p, (float)c_fx * p.fx_inv[1]);
    if (COUPLED) {
        float a[9];
        pull9(src + 18 * p.plane, p, i, j, a);
        F[FP_DPS * p.plane + idx] = sum9(a);
    }
}

__global__ void k_normals(KParams p, float* __restrict__ F) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y;
    if (i >= p.nx) return;
    const int64_t idx = (int64_t)j * p.pitch + i;
    int v[3][3];
    load3x3_fx(F + FP_PHI * p.plane, p, i, j, v);
    float gx, gy, nx, ny, gm;
    iso_grad_fx(v, p.fx_inv[0], gx, gy);
    unit_normal(gx, gy, nx, ny, gm);
    F[FP_NX * p.plane + idx] = nx;
    F[FP_NY * p.plane + idx] = ny;
    F[FP_GM * p.plane + idx] = gm;
}

template <bool COUPLED>
__device__ __forceinline__ CellGeom gather_geom(const KParams& p, const float* __restrict__ F, int i,
                                                int j) {
    const int64_t idx = (int64_t)j * p.pitch + i;
    CellGeom g;
    g.phi_fx = __float_as_int(F[FP_PHI * p.plane + idx]);
    g.phi = (float)g.phi_fx * p.fx_inv[0];
    g.c = (float)__float_as_int(F[FP_C * p.plane + idx]) * p.fx_inv[1];
    g.nx = F[FP_NX * p.plane + idx];
    g.ny = F[FP_NY * p.plane + idx];
    g.gm = F[FP_GM * p.plane + idx];
    g.sig = F[FP_SIG * p.plane + idx];
    if (COUPLED) {
        g.dps = F[FP_DPS * p.plane + idx];
        float vx[3][3], vy[3][3], v[3][3];
        load3x3(F + FP_NX * p.plane, p, i, j, vx);
        load3x3(F + FP_NY * p.plane, p, i, j, vy, true);
        g.kappa = iso_div(vx, vy);
        load3x3(F + FP_SIG * p.plane, p, i, j, v);
        iso_grad(v, g.sgx, g.sgy);
        load3x3(F + FP_DPS * p.plane, p, i, j, v);
        iso_grad(v, g.pgx, g.pgy);
        if (!p.rho_uniform) {
            int vi[3][3];
            load3x3_fx(F + FP_PHI * p.plane, p, i, j, vi);
            iso_grad_fx(vi, p.fx_inv[0], g.fgx, g.fgy);
        } else {
            g.fgx = g.fgy = 0.0f;
        }
    } else {
        g.dps = 0.0f;
        g.kappa = g.sgx = g.sgy = g.pgx = g.pgy = g.fgx = g.fgy = 0.0f;
    }
    return g;
}

template <bool COUPLED>
__global__ void k_collide(KParams p, const float* __restrict__ src, float* __restrict__ dst,
                          const float* __restrict__ F) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y;
    if (i >= p.nx) return;
    const int64_t idx = (int64_t)j * p.pitch + i;
    CellGeom g = gather_geom<COUPLED>(p, F, i, j);
    const ScalarMoments mf = pull_scalar(src, p, 0, i, j);
    const ScalarMoments mh = pull_scalar(src + 9 * p.plane, p, 1, i, j);
    const uint32_t bits = moment_bits(step_seed(p), i, j, p.nx);
    const int f_fx = fx_add_sr(mf.s0, mf.inc, p.fx_scale[0], bits);
    const int h_fx = fx_add_sr(mh.s0, mh.inc, p.fx_scale[1], second_bits(bits));
    float gg[9], df[9], dh[9];
    float ufx = 0.0f, ufy = 0.0f;
    if (COUPLED) {
        pull9(src + 18 * p.plane, p, i, j, gg);
    } else {
        ufx = F[FP_UX * p.plane + idx];
        ufy = F[FP_UY * p.plane + idx];
    }
    collide_cell<COUPLED>(p, g, j, ufx, ufy, mf.jx, mf.jy, mh.jx, mh.jy, gg, df, dh, true);
    store_dev(dst, p, idx, i, f_fx, df);
    store_dev(dst + 9 * p.plane, p, idx, i, h_fx, dh);
    if (COUPLED) store9(dst + 18 * p.plane, p, idx, i, gg);
}

// FP64 instructions issue at two lanes a cycle and SM; these conversions are
// integer arithmetic.  Same values as the conversion instructions.
__device__ __forceinline__ double widen(float v) {
    const uint32_t b = __float_as_uint(v), e = (b >> 23) & 255u;
    if ((b << 1) == 0u) return __hiloint2double((int)b, 0);
    if (e == 0u || e == 255u) return (double)v;
    return __hiloint2double((int)((b & 0x80000000u) | (((b >> 3) & 0x0fffffffu) + (896u << 20))), (int)(b << 29));
}

// s / scale for a power of two `scale` (NaN for the invalid marker).
__device__ __forceinline__ double fx_widen(int s, float scale) {
    const int k = (int)(__float_as_uint(scale) >> 23) - 127;
    if (s == FX_INVALID || k < -126) return fx_to_double(s, scale);
    if (s == 0) return 0.0;
    const uint32_t m = (uint32_t)abs(s);
    const int lz = __clz(m);
    const uint32_t f = m << lz << 1;  // the bits below the leading one
    const uint32_t hi = ((uint32_t)s & 0x80000000u) | ((uint32_t)(1023 + 31 - lz - k) << 20) | (f >> 12);
    return __hiloint2double((int)hi, (int)(f << 20));
}

// Macroscopic state of the cells of a 32 x 8 tile, one per thread: out(i, j,
// phi_fx, c_fx, ux, uy, dP) for those inside the grid (dP: P - P0).  The block
// forms phi, sigma and P* of the tile and two cells around it in shared memory,
// then the normals of the tile and one cell around it, then each cell's forces,
// with the operations of the three-kernel chain in their order (same bits).
//
// Bound by the pulls (1.69 times the tile's, from L2) and their latency.  Serves
// the kernels without bulk-tensor loads; the others have the tile staged as the
// step does (tile_step with an `out`), from their own storage format.
constexpr int MT_X = 32, MT_Y = 8;
template <bool COUPLED, class Out>
__device__ __forceinline__ void macro_tile(const KParams& p, const float* __restrict__ src,
                                           const float* __restrict__ F, Out out) {
    constexpr int WX = MT_X + 4, WY = MT_Y + 4, NX = MT_X + 2, NY = MT_Y + 2;
    const int x0 = blockIdx.x * MT_X, y0 = blockIdx.y * MT_Y;
    const int rows = min(MT_Y, p.ny - y0), cols = min(MT_X, p.nx - x0);
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int i = x0 + tx, j = y0 + ty;
    const bool own = tx < cols && ty < rows;
    const uint32_t seed = step_seed(p);
    if constexpr (!COUPLED) {
        if (!own) return;
        const uint32_t bits = moment_bits(seed, i, j, p.nx);
        const ScalarMoments f = pull_scalar(src, p, 0, i, j), h = pull_scalar(src + 9 * p.plane, p, 1, i, j);
        const int64_t idx = (int64_t)j * p.pitch + i;
        out(i, j, fx_add_sr(f.s0, f.inc, p.fx_scale[0], bits),
            fx_add_sr(h.s0, h.inc, p.fx_scale[1], second_bits(bits)), F[FP_UX * p.plane + idx],
            F[FP_UY * p.plane + idx], 0.0f);
    } else {
        __shared__ int s_phi[WY * WX], s_c[MT_Y * MT_X];
        __shared__ float s_sig[WY * WX], s_dps[WY * WX], s_nx[NY * NX], s_ny[NY * NX], s_gm[NY * NX];
        for (int k = threadIdx.x; k < (rows + 4) * WX; k += MT_X * MT_Y) {
            const int r = k / WX, w = k - r * WX;
            if (w >= cols + 4) continue;
            const int gi = wrap_i(x0 + w - 2, p.nx), gj = ext_row(y0 + r - 2, p.ny, p.walls);
            const uint32_t bits = moment_bits(seed, gi, gj, p.nx);
            const ScalarMoments f = pull_scalar(src, p, 0, gi, gj);
            const ScalarMoments h = pull_scalar(src + 9 * p.plane, p, 1, gi, gj);
            float a[9];
            pull9(src + 18 * p.plane, p, gi, gj, a);
            const int c_fx = fx_add_sr(h.s0, h.inc, p.fx_scale[1], second_bits(bits));
            s_phi[k] = fx_add_sr(f.s0, f.inc, p.fx_scale[0], bits);
            s_sig[k] = sigma_of_c(p, (float)c_fx * p.fx_inv[1]);
            s_dps[k] = sum9(a);
            if (r >= 2 && r < rows + 2 && w >= 2 && w < cols + 2) s_c[(r - 2) * MT_X + w - 2] = c_fx;
        }
        __syncthreads();
        for (int k = threadIdx.x; k < (rows + 2) * NX; k += MT_X * MT_Y) {
            const int r = k / NX, w = k - r * NX;
            if (w >= cols + 2) continue;
            int v[3][3];
            for (int a = 0; a < 3; ++a)
                for (int b = 0; b < 3; ++b) v[a][b] = s_phi[(r + a) * WX + w + b];
            float gx, gy;
            iso_grad_fx(v, p.fx_inv[0], gx, gy);
            unit_normal(gx, gy, s_nx[k], s_ny[k], s_gm[k]);
        }
        __syncthreads();
        if (!own) return;
        auto around = [&](const auto* s, int stride, int at, auto(&v)[3][3]) {
#pragma unroll
            for (int a = 0; a < 3; ++a)
#pragma unroll
                for (int b = 0; b < 3; ++b) v[a][b] = s[at + (a - 1) * stride + b - 1];
        };
        const int at = (ty + 2) * WX + tx + 2, an = (ty + 1) * NX + tx + 1;
        CellGeom g;
        float vx[3][3], vy[3][3], v[3][3];
        g.phi_fx = s_phi[at];
        g.phi = (float)g.phi_fx * p.fx_inv[0];
        g.c = (float)s_c[ty * MT_X + tx] * p.fx_inv[1];
        g.nx = s_nx[an];
        g.ny = s_ny[an];
        g.gm = s_gm[an];
        g.sig = s_sig[at];
        g.dps = s_dps[at];
        around(s_nx, NX, an, vx);
        around(s_ny, NX, an, vy);
        g.kappa = iso_div(vx, vy);
        around(s_sig, WX, at, v);
        iso_grad(v, g.sgx, g.sgy);
        around(s_dps, WX, at, v);
        iso_grad(v, g.pgx, g.pgy);
        g.fgx = g.fgy = 0.0f;
        if (!p.rho_uniform) {
            int vi[3][3];
            around(s_phi, WX, at, vi);
            iso_grad_fx(vi, p.fx_inv[0], g.fgx, g.fgy);
        }
        float gg[9];
        pull9(src + 18 * p.plane, p, i, j, gg);
        const CellOut r = collide_flow_cell(p, g, j, gg, false);
        out(i, j, g.phi_fx, s_c[ty * MT_X + tx], r.ux, r.uy, r.dP);
    }
}

// ST: storage format of the state that `tmap` loads, or ST_NONE: plain pulls from
// the FP32 state `src`.
constexpr int ST_NONE = -1;
template <bool COUPLED, int ST, class Out>
__device__ __forceinline__ void macro_cells(const CUtensorMap* tmap, const KParams& p, const float* __restrict__ src,
                                            const float* __restrict__ F, int* err, Out out) {
    if constexpr (ST == ST_NONE) {
        macro_tile<COUPLED>(p, src, F, out);
    } else {
        static_assert(MT_X == TILE_TX && MT_X * MT_Y == TILE_NT && MT_Y == TILE_SEG, "one cell per thread");
        tile_step<COUPLED, ST>(tmap, p, nullptr, F, MT_Y, blockIdx.x, blockIdx.y, [&] { return step_seed(p); }, err,
                               out);
    }
}

// Fields as three kernels through global planes, then as plain pulls, then by
// staged tiles: 128 runs of 384 x 128 23, 13 and 10 us a run, 768 x 256 16 us.
template <bool COUPLED, int ST>
__global__ void __launch_bounds__(MT_X * MT_Y)
k_macro_out(const __grid_constant__ CUtensorMap tmap, KParams p, const float* __restrict__ src,
            const float* __restrict__ F, int* __restrict__ err, double* __restrict__ ophi, double* __restrict__ oc,
            double* __restrict__ oux, double* __restrict__ ouy, double* __restrict__ oP) {
    macro_cells<COUPLED, ST>(&tmap, p, src, F, err, [&](int i, int j, int phi_fx, int c_fx, float ux, float uy, float dP) {
        const int64_t o = (int64_t)j * p.nx + i;
        if (ophi) ophi[o] = fx_widen(phi_fx, p.fx_scale[0]);
        if (oc) oc[o] = fx_widen(c_fx, p.fx_scale[1]);
        if (oux) oux[o] = widen(ux);
        if (ouy) ouy[o] = widen(uy);
        if (oP) oP[o] = COUPLED ? (double)p.P0 + widen(dP) : 0.0;
    });
}

// ---------------------------------------------------------------------------
// fused sweep kernel
// ---------------------------------------------------------------------------

constexpr int RING = 5;    // rows kept of phi, c, sigma, P* (current row and four behind)
constexpr int NRING = 3;   // rows kept of n and |grad phi|
constexpr int PRING = 3;   // rows of interior cells waiting for their collision
constexpr int PSLOT = 15;  // per waiting cell: f (jx, jy), h (S, jx, jy), g (9 populations)

size_t fused_smem_bytes(int bx) {
    return sizeof(float) * (size_t)bx * (4 * RING + 3 * NRING + PSLOT * PRING);
}

// Block = bx threads = bx - 4 interior columns plus two halo columns each side.
// Rows [y0, y1) are collided; rows y0-2 .. y1+1 are streamed for phi and rows
// y0-1 .. y1 for c, sigma and P* (ghost rows beyond walls hold the mirrored
// values, so the stencils there reproduce the mirrored extended field).
template <bool COUPLED>
__global__ void __launch_bounds__(128) k_fused_sweep(KParams p, const float* __restrict__ src,
                                                     float* __restrict__ dst,
                                                     const float* __restrict__ F, int seg) {
    extern __shared__ float sm[];
    const int bx = blockDim.x;
    const int t = threadIdx.x;
    int* s_phi = reinterpret_cast<int*>(sm);  // [RING][bx] phi, fixed point
    float* s_c = sm + RING * bx;
    float* s_sig = s_c + RING * bx;
    float* s_dps = s_sig + RING * bx;
    float* s_nx = s_dps + RING * bx;         // [NRING][bx]
    float* s_ny = s_nx + NRING * bx;
    float* s_gm = s_ny + NRING * bx;
    float* s_pop = s_gm + NRING * bx;        // [PRING][PSLOT][bx]

    const int tx = bx - 4;
    const int x0 = blockIdx.x * tx;
    const int xend = min(x0 + tx, p.nx);
    const int y0 = blockIdx.y * seg;
    const int y1 = min(y0 + seg, p.ny);
    const int col = x0 - 2 + t;
    // role: 3 interior, 2 first halo column, 1 second halo column, 0 idle
    int role = 0;
    if (col >= x0 && col < xend) role = 3;
    else if (col == x0 - 1 || col == xend) role = 2;
    else if (col == x0 - 2 || col == xend + 1) role = 1;
    const int i = wrap_i(col, p.nx);
    const uint32_t seed = step_seed(p);

    for (int r = y0 - 2; r <= y1 + 1; ++r) {
        // A: stream row r and form its moments
        const int slot = (r + 2 * RING) % RING;
        if (role > 0) {
            const int jj = ext_row(r, p.ny, p.walls);
            const bool keep = role == 3 && r >= y0 && r < y1;
            float* pp = s_pop + ((r + 3 * PRING) % PRING) * PSLOT * bx;
            const uint32_t bits = moment_bits(seed, i, jj, p.nx);
            ScalarMoments m = pull_scalar(src, p, 0, i, jj);
            s_phi[slot * bx + t] = fx_add_sr(m.s0, m.inc, p.fx_scale[0], bits);
            if (keep) {
                pp[0 * bx + t] = m.jx;
                pp[1 * bx + t] = m.jy;
            }
            if (role >= 2 && r >= y0 - 1 && r <= y1) {
                m = pull_scalar(src + 9 * p.plane, p, 1, i, jj);
                const int c_fx = fx_add_sr(m.s0, m.inc, p.fx_scale[1], second_bits(bits));
                const float c = (float)c_fx * p.fx_inv[1];
                s_c[slot * bx + t] = c;
                s_sig[slot * bx + t] = sigma_of_c(p, c);
                if (keep) {
                    pp[2 * bx + t] = __int_as_float(c_fx);
                    pp[3 * bx + t] = m.jx;
                    pp[4 * bx + t] = m.jy;
                }
                if (COUPLED) {
                    float a[9];
                    pull9(src + 18 * p.plane, p, i, jj, a);
                    s_dps[slot * bx + t] = sum9(a);
                    if (keep) {
#pragma unroll
                        for (int q = 0; q < 9; ++q) pp[(6 + q) * bx + t] = a[q];
                    }
                }
            }
        }
        __syncthreads();
        // B: normal at row r-1 (needs phi rows r-2 .. r)
        const int rn = r - 1;
        if (role >= 2 && rn >= y0 - 1 && rn <= y1) {
            const int sm1 = (rn - 1 + 2 * RING) % RING, s0 = (rn + 2 * RING) % RING,
                      sp1 = (rn + 1 + 2 * RING) % RING;
            int v[3][3];
            v[0][0] = s_phi[sm1 * bx + t - 1]; v[0][1] = s_phi[sm1 * bx + t]; v[0][2] = s_phi[sm1 * bx + t + 1];
            v[1][0] = s_phi[s0 * bx + t - 1];  v[1][1] = s_phi[s0 * bx + t];  v[1][2] = s_phi[s0 * bx + t + 1];
            v[2][0] = s_phi[sp1 * bx + t - 1]; v[2][1] = s_phi[sp1 * bx + t]; v[2][2] = s_phi[sp1 * bx + t + 1];
            float gx, gy, nx, ny, gm;
            iso_grad_fx(v, p.fx_inv[0], gx, gy);
            unit_normal(gx, gy, nx, ny, gm);
            const int ns = (rn + 3 * NRING) % NRING;
            s_nx[ns * bx + t] = nx;
            s_ny[ns * bx + t] = ny;
            s_gm[ns * bx + t] = gm;
        }
        __syncthreads();
        // C: collide row r-2
        const int jc = r - 2;
        if (role == 3 && jc >= y0 && jc < y1) {
            const int cm1 = (jc - 1 + 2 * RING) % RING, c0 = (jc + 2 * RING) % RING,
                      cp1 = (jc + 1 + 2 * RING) % RING;
            const int nm1 = (jc - 1 + 3 * NRING) % NRING, n0 = (jc + 3 * NRING) % NRING,
                      np1 = (jc + 1 + 3 * NRING) % NRING;
            CellGeom g;
            g.phi_fx = s_phi[c0 * bx + t];
            g.phi = (float)g.phi_fx * p.fx_inv[0];
            g.c = s_c[c0 * bx + t];
            g.sig = s_sig[c0 * bx + t];
            g.nx = s_nx[n0 * bx + t];
            g.ny = s_ny[n0 * bx + t];
            g.gm = s_gm[n0 * bx + t];
            if (COUPLED) {
                g.dps = s_dps[c0 * bx + t];
                float vx[3][3], vy[3][3], v[3][3];
                const int nr[3] = {nm1, n0, np1};
                const int cr[3] = {cm1, c0, cp1};
#pragma unroll
                for (int d = 0; d < 3; ++d) {
#pragma unroll
                    for (int e = 0; e < 3; ++e) {
                        vx[d][e] = s_nx[nr[d] * bx + t - 1 + e];
                        vy[d][e] = s_ny[nr[d] * bx + t - 1 + e];
                    }
                }
                g.kappa = iso_div(vx, vy);
#pragma unroll
                for (int d = 0; d < 3; ++d)
#pragma unroll
                    for (int e = 0; e < 3; ++e) v[d][e] = s_sig[cr[d] * bx + t - 1 + e];
                iso_grad(v, g.sgx, g.sgy);
#pragma unroll
                for (int d = 0; d < 3; ++d)
#pragma unroll
                    for (int e = 0; e < 3; ++e) v[d][e] = s_dps[cr[d] * bx + t - 1 + e];
                iso_grad(v, g.pgx, g.pgy);
                if (!p.rho_uniform) {
                    int vi[3][3];
#pragma unroll
                    for (int d = 0; d < 3; ++d)
#pragma unroll
                        for (int e = 0; e < 3; ++e) vi[d][e] = s_phi[cr[d] * bx + t - 1 + e];
                    iso_grad_fx(vi, p.fx_inv[0], g.fgx, g.fgy);
                } else {
                    g.fgx = g.fgy = 0.0f;
                }
            } else {
                g.dps = 0.0f;
                g.kappa = g.sgx = g.sgy = g.pgx = g.pgy = g.fgx = g.fgy = 0.0f;
            }
            const float* pp = s_pop + ((jc + 3 * PRING) % PRING) * PSLOT * bx;
            const float fjx = pp[0 * bx + t], fjy = pp[1 * bx + t];
            const int h_fx = __float_as_int(pp[2 * bx + t]);
            const float hjx = pp[3 * bx + t], hjy = pp[4 * bx + t];
            float gg[9], df[9], dh[9];
#pragma unroll
            for (int q = 0; q < 9; ++q) gg[q] = COUPLED ? pp[(6 + q) * bx + t] : 0.0f;
            const int64_t idx = (int64_t)jc * p.pitch + i;
            float ufx = 0.0f, ufy = 0.0f;
            if (!COUPLED) {
                ufx = F[FP_UX * p.plane + idx];
                ufy = F[FP_UY * p.plane + idx];
            }
            collide_cell<COUPLED>(p, g, jc, ufx, ufy, fjx, fjy, hjx, hjy, gg, df, dh, true);
            store_dev(dst, p, idx, i, g.phi_fx, df);
            store_dev(dst + 9 * p.plane, p, idx, i, h_fx, dh);
            if (COUPLED) store9(dst + 18 * p.plane, p, idx, i, gg);
        }
    }
}

// ---------------------------------------------------------------------------
// initialisation and population import / export
// ---------------------------------------------------------------------------

__global__ void k_init_fields(KParams p, const double* __restrict__ phi,
                              const double* __restrict__ c, const double* __restrict__ ux,
                              const double* __restrict__ uy, const double* __restrict__ P,
                              float* __restrict__ F) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y;
    if (i >= p.nx) return;
    const int64_t idx = (int64_t)j * p.pitch + i;
    const int64_t o = (int64_t)j * p.nx + i;
    const float fphi = (float)phi[o];
    const float fc = (float)c[o];
    F[FP_PHI * p.plane + idx] = __int_as_float(fx_from_double(phi[o], p.fx_scale[0]));
    F[FP_C * p.plane + idx] = __int_as_float(fx_from_double(c[o], p.fx_scale[1]));
    F[FP_SIG * p.plane + idx] = sigma_of_c(p, fc);
    F[FP_UX * p.plane + idx] = (float)ux[o];
    F[FP_UY * p.plane + idx] = (float)uy[o];
    // default pressure: uniform, the rest pressure P0 = cs2 (rho_a + rho_b) / 2
    // (with equal densities, rho cs2 everywhere)
    const double Pv = P ? P[o] : (double)p.P0;
    F[FP_DPS * p.plane + idx] = (float)(Pv - (double)p.P0);
}

// Equilibrium post-streaming populations into `pre` (dense-pitched [nlat*9]).
template <bool COUPLED>
__global__ void k_init_pre(KParams p, const float* __restrict__ F, float* __restrict__ pre) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y;
    if (i >= p.nx) return;
    const int64_t idx = (int64_t)j * p.pitch + i;
    const int phi_fx = __float_as_int(F[FP_PHI * p.plane + idx]);
    const float phi = (float)phi_fx * p.fx_inv[0];
    const float c = (float)__float_as_int(F[FP_C * p.plane + idx]) * p.fx_inv[1];
    const float nx = F[FP_NX * p.plane + idx];
    const float ny = F[FP_NY * p.plane + idx];
    const float ux = F[FP_UX * p.plane + idx];
    const float uy = F[FP_UY * p.plane + idx];
    float theta, theta_c;
    interface_coeffs(p, phi_fx, c, theta, theta_c);
    float a[9];
    eq_scalar(a, phi, p.M_phi * theta * nx, p.M_phi * theta * ny, ux, uy);
    store9_plain(pre, p, idx, a);
    eq_scalar(a, c, p.D_s * theta_c * nx, p.D_s * theta_c * ny, ux, uy);
    store9_plain(pre + 9 * p.plane, p, idx, a);
    if (COUPLED) {
        const float rho = p.rho_uniform ? p.rho_a : lerp_phase(p, phi, p.rho_a, p.rho_b);
        eq_flow_shifted(a, F[FP_DPS * p.plane + idx], rho, ux, uy);
        store9_plain(pre + 18 * p.plane, p, idx, a);
    }
}

// Deviation form of nine slots: returns their sum S rounded to fixed point (scale:
// a power of two, inv its reciprocal) and d_q = u_q - w_q S, as FP64 gives them
// (the slots added in their order, each d_q by one fused multiply-add).  FP64
// instructions issue at two lanes a cycle and SM, and those of a cell made the kernel
// 140 us at 1024 x 512, so it is done in 64-bit whole numbers, in units of 2^-27
// of the fixed point's, or 2^-47 where all slots are small: w_1 = 4 w_5 is whole
// there, and so are the slots of nearly all cells.  Exact sums and products below
// 2^53 are what FP64 has, too; the cells for which that is not so, or whose S is so
// close to a tie that the rounding of the FP64 sum could decide it, take FP64
// itself: 32 us.  (Pairs of floats, 27 us, lose bits where a slot all but cancels
// its share.)
__device__ __forceinline__ int deviations(const float (&u)[9], float scale, float inv, float (&d)[9]) {
    constexpr long long W1 = 14913081;  // 2^27 w_1
    static_assert((float)W1 / 134217728.0f == wq(1) && wq(5) * 4.0f == wq(1), "weights in these units");
    float one = scale * 134217728.0f, unit = inv / 134217728.0f;
    bool none = true, fine = true, whole = true;  // S is certainly 0; slots are below 16 units; certainly exact
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        const float f = fabsf(u[q] * one);
        none = none && f < 7.0e6f;  // 9 of them: 0.47 of a fixed-point unit
        fine = fine && f < 2.1e9f;  // below 2^31
    }
    const int more = fine ? 20 : 0;
    if (fine) one *= 1048576.0f, unit *= 1.0f / 1048576.0f;
    long long U[9], sum = 0;
    if (!none) {
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            const float f = u[q] * one;
            whole = whole && fabsf(f) < 7.2e16f && truncf(f) == f;  // below 2^56
            U[q] = __float2ll_rn(f);
            sum += U[q];
        }
    }
    // eight roundings to 53 bits of sums below 9 * 2^56: less than 2^10 units
    const long long half = 1LL << (26 + more);
    const long long S64 = (sum + half) >> (27 + more);
    whole = whole && llabs((sum & (2 * half - 1)) - half) > 1024 && llabs(S64) <= FX_RANGE;
    int S = (int)S64;
    if (none || (whole && S == 0)) {  // (with the sign of a zero)
#pragma unroll
        for (int q = 1; q < 9; ++q) d[q] = u[q];
        return 0;
    }
    const long long T = W1 * S << more;  // below 2^57
#pragma unroll
    for (int q = 1; q < 9; ++q) {
        const long long D = (q <= 4 ? U[q] : 4 * U[q]) - T;
        whole = whole && llabs(D) < 1LL << 53;
        d[q] = __ll2float_rn(D) * (q <= 4 ? unit : 0.25f * unit);
    }
    if (!whole) {
        double s = 0.0;
        for (int q = 0; q < 9; ++q) s += (double)u[q];
        S = fx_from_double(s, scale);
        const double Sr = fx_to_double(S, scale);
#pragma unroll
        for (int q = 1; q < 9; ++q) d[q] = (float)__fma_rn(-(double)wq(q), Sr, (double)u[q]);
    }
    return S;
}

// Stored (post-collision, pull-ready) form from post-streaming populations:
// slot q at y is read by the pull of cell y + e_q, or, when y + e_q lies
// beyond a wall, by the bounce-back of direction opp(q) at y.  The two
// advection-diffusion lattices are then written in deviation form
// (S = sum of the slots, d_q = slot_q - w_q S); the flow lattice as is.
__global__ void k_unstream(KParams p, int nlat, const float* __restrict__ pre,
                           float* __restrict__ dst) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y;
    if (i >= p.nx) return;
    const int64_t idx = (int64_t)j * p.pitch + i;
    for (int l = 0; l < nlat; ++l) {
        const float* pl = pre + (int64_t)l * 9 * p.plane;
        float* dl = dst + (int64_t)l * 9 * p.plane;
        float u[9];
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            const int ti = wrap_i(i + ex(q), p.nx);
            const int tj = j + ey(q);
            if (p.walls && (tj < 0 || tj >= p.ny)) {
                u[q] = pl[opp(q) * p.plane + idx];
            } else {
                u[q] = pl[q * p.plane + (int64_t)wrap_i(tj, p.ny) * p.pitch + ti];
            }
        }
        if (l < 2) {
            float d[9];
            const int S_fx = deviations(u, p.fx_scale[l], p.fx_inv[l], d);
            store_dev(dl, p, idx, i, S_fx, d);
        } else {
            store9(dl, p, idx, i, u);
        }
    }
}

// Post-streaming populations of the stored state, into a pitched float buffer.
__global__ void k_pull_pre(KParams p, int nlat, const float* __restrict__ src,
                           float* __restrict__ pre) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y;
    if (i >= p.nx) return;
    const int64_t idx = (int64_t)j * p.pitch + i;
    for (int l = 0; l < nlat; ++l) {
        float a[9];
        if (l < 2)
            pull9_dev<float>(src + (int64_t)l * 9 * p.plane, p, l, i, j, a);
        else
            pull9(src + (int64_t)l * 9 * p.plane, p, i, j, a);
        store9_plain(pre + (int64_t)l * 9 * p.plane, p, idx, a);
    }
}

// Post-streaming populations as float64 dense [nlat*9][ny][nx], unshifted.
__global__ void k_export_pops(KParams p, int nlat, const float* __restrict__ src,
                              double* __restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y;
    if (i >= p.nx) return;
    const int64_t n = (int64_t)p.nx * p.ny;
    const int64_t o = (int64_t)j * p.nx + i;
    for (int l = 0; l < nlat; ++l) {
        double a[9];
        if (l < 2) {
            pull9_dev<double>(src + (int64_t)l * 9 * p.plane, p, l, i, j, a);
        } else {
            float b[9];
            pull9(src + (int64_t)l * 9 * p.plane, p, i, j, b);
#pragma unroll
            for (int q = 0; q < 9; ++q) a[q] = (double)b[q] + (double)wq(q) * (double)p.P0;
        }
#pragma unroll
        for (int q = 0; q < 9; ++q) out[(l * 9 + q) * n + o] = a[q];
    }
}

// One lattice of float64 dense post-streaming populations into the pitched
// float pre-form (flow lattice shifted by w P0).
__global__ void k_f64_to_pre(KParams p, int lat, const double* __restrict__ in,
                             float* __restrict__ pre) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y;
    if (i >= p.nx) return;
    const int64_t idx = (int64_t)j * p.pitch + i;
    const int64_t n = (int64_t)p.nx * p.ny;
    const int64_t o = (int64_t)j * p.nx + i;
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        double v = in[q * n + o];
        if (lat == 2) v -= (double)wq(q) * (double)p.P0;
        pre[(lat * 9 + q) * p.plane + idx] = (float)v;
    }
}

// ---------------------------------------------------------------------------
// diagnostics: totals and the shape moments of the drop
// ---------------------------------------------------------------------------

// The drop indicator w, (phi - phi_b) / (phi_a - phi_b) clipped to [0, 1], in
// units of phi's fixed point.  The shape moments (centroid, Ixx, Iyy, Ixy;
// D = (L - B) / (L + B) of Sec. 4.3) belong to the drop region: the clip keeps
// the small over- and undershoot of phi away from the interface, which its
// distance would weigh heavily, out.
__device__ __forceinline__ int drop_indicator(const KParams& p, int phi_fx) {
    const int span = p.phi_a_fx - p.phi_b_fx, v = phi_fx - p.phi_b_fx;
    return span > 0 ? min(max(v, 0), span) : min(max(-v, 0), -span);
}

// Everything that is summed over cells is a whole number (fixed-point values and
// counts), so the sums are exact whatever their order and can be made by atomic
// adds; w is summed by column and by row, from which the centroid, Ixx and Iyy
// follow with one term per column or row.  Only Ixy needs the cells again.  With
// FP64 sums, and the sines and cosines taken per cell, the two passes took 272 us
// at 1024 x 512 after 72 us for the fields; now 78 and 17 us with the fields.
constexpr int DIAG_THREADS = 256;
constexpr double TWO_PI = 6.283185307179586476925286766559;
enum DiagWord { DW_PHI = 0, DW_C, DW_NONFINITE, DW_SIGMA_NEG, DW_UMAX2, DW_DONE1, DW_DONE2, DW_COUNT = 8 };
using u64 = unsigned long long;

// Blocks of pass 2, each with a partial sum of Ixy: about 16 rows a thread, long
// enough for the loads and short enough to fill the chip.
static int ixy_strips(const KParams& p) { return (p.nx + DIAG_THREADS - 1) / DIAG_THREADS; }
static int ixy_bands(const KParams& p) {
    const int most = 1024 / ixy_strips(p), bands = (p.ny + 15) / 16;
    return most < 1 ? 1 : bands < most ? bands : most;
}
size_t diag_words(const KParams& p) {
    return DW_COUNT + 3 * ((size_t)p.nx + p.ny) + (size_t)ixy_strips(p) * ixy_bands(p);
}

// Sum over a warp of signed 32-bit values, exact.
__device__ __forceinline__ long long warp_sum(int v) {
    const unsigned lo = __reduce_add_sync(0xffffffffu, (unsigned)v & 0xffffu);
    const int hi = __reduce_add_sync(0xffffffffu, v >> 16);
    return (long long)hi * 65536 + (long long)lo;
}

template <int NK>
__device__ __forceinline__ void block_sum(double (&v)[NK]) {
    __shared__ double red[NK][DIAG_THREADS / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < NK; ++k) {
        for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_down_sync(0xffffffffu, v[k], o);
        if (lane == 0) red[k][w] = v[k];
    }
    __syncthreads();
    for (int k = 0; k < NK; ++k) {
        v[k] = 0.0;
        for (int q = 0; q < DIAG_THREADS / 32; ++q) v[k] += red[k][q];
    }
    __syncthreads();
}

__device__ __forceinline__ double min_image(double d, int n, bool periodic) {
    if (!periodic) return d;
    while (d >= 0.5 * n) d -= n;
    while (d < -0.5 * n) d += n;
    return d;
}

// True in the block that is the last of the grid to come here; what the others
// wrote before is then visible to it.
__device__ __forceinline__ bool last_block(u64* done) {
    __shared__ bool last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(done, 1ull) + 1 == (u64)gridDim.x * gridDim.y;
        __threadfence();
    }
    __syncthreads();
    return last;
}

// result layout: [0] sum_phi [1] sum_c [2] xc [3] yc [4] nonfinite [5] sigma_neg [6] umax
//                [7] Ixx [8] Iyy [9] Ixy [10] L [11] B [12] D [13] sum w
// Pass 1: fields of every cell, all sums but Ixy's, w of every cell into `wmap`
// (0 where a field is not finite).  arg_lo, arg_hi: 1 - c / c_max between which
// sigma is positive for certain.
template <bool COUPLED, int ST>
__global__ void __launch_bounds__(DIAG_THREADS)
k_diag1(const __grid_constant__ CUtensorMap tmap, KParams p, const float* __restrict__ src,
        const float* __restrict__ F, int* __restrict__ err, float arg_lo, float arg_hi, int* __restrict__ wmap,
        u64* __restrict__ words, double* __restrict__ res) {
    static_assert(MT_X * MT_Y == DIAG_THREADS && MT_Y * 32 == DIAG_THREADS, "one warp per tile row");
    // cosines and sines of the columns and rows: formed by the blocks at the grid's
    // edges, spread over the SMs (FP64 on the finishing block's one SM is slow)
    double2* xtrig = reinterpret_cast<double2*>(words + DW_COUNT);
    double2* ytrig = xtrig + p.nx;
    u64* col = reinterpret_cast<u64*>(ytrig + p.ny);
    u64* row = col + p.nx;
    int phi = 0, c = 0, w = 0, nonfinite = 0, sigma_neg = 0;
    float u2 = 0.0f, a = 0.0f, b = 0.0f;
    macro_cells<COUPLED, ST>(&tmap, p, src, F, err, [&](int i, int j, int phi_fx, int c_fx, float ux, float uy, float) {
        const int64_t o = (int64_t)j * p.nx + i;
        if (phi_fx == FX_INVALID || c_fx == FX_INVALID || !isfinite(ux) || !isfinite(uy)) {
            nonfinite = 1;
            wmap[o] = 0;
            return;
        }
        phi = phi_fx;
        c = c_fx;
        w = drop_indicator(p, phi_fx);
        wmap[o] = w;
        a = ux;
        b = uy;
        u2 = ux * ux + uy * uy;
        if (p.beta != 0.0f) {
            const float near = 1.0f - (float)c_fx * p.fx_inv[1] * p.inv_cmax;
            if (!(near > arg_lo && near < arg_hi)) {
                const double arg = 1.0 - fx_to_double(c_fx, p.fx_scale[1]) * (double)p.inv_cmax;
                sigma_neg = arg <= 0.0 || 1.0 + (double)p.beta * log(arg) < 0.0;
            }
        }
    });
    __shared__ int sw[MT_Y][MT_X];
    __shared__ u64 su[MT_Y];
    __shared__ long long ssum[2][MT_Y];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int i = blockIdx.x * MT_X + tx, j = blockIdx.y * MT_Y + ty;
    sw[ty][tx] = w;
    const long long sphi = warp_sum(phi), sc = warp_sum(c), sr = warp_sum(w);
    const unsigned bad = __popc(__ballot_sync(0xffffffffu, nonfinite)),
                   neg = __popc(__ballot_sync(0xffffffffu, sigma_neg));
    // the largest |u|^2 of the warp: in FP64 for the cells that may have it
    const float most = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(u2)));
    double top = 0.0;
    if ((a != 0.0f || b != 0.0f) && (most < 1e-30f || u2 >= most * 0.999999f)) top = widen(a) * widen(a) + widen(b) * widen(b);
    u64 tb = (u64)__double_as_longlong(top);
    for (int o = 16; o > 0; o >>= 1) tb = max(tb, __shfl_xor_sync(0xffffffffu, tb, o));
    if (tx == 0) {
        su[ty] = tb;
        ssum[0][ty] = sphi;
        ssum[1][ty] = sc;
        if (sr) atomicAdd(row + j, (u64)sr);
        if (bad) atomicAdd(words + DW_NONFINITE, (u64)bad);
        if (neg) atomicAdd(words + DW_SIGMA_NEG, (u64)neg);
    }
    __syncthreads();
    if (ty == 0 && i < p.nx) {
        long long s = 0;
        for (int r = 0; r < MT_Y; ++r) s += sw[r][tx];
        if (s) atomicAdd(col + i, (u64)s);
    }
    if (threadIdx.x == DIAG_THREADS - 1) {
        u64 m = 0;
        for (int r = 0; r < MT_Y; ++r) m = max(m, su[r]);
        if (m) atomicMax(words + DW_UMAX2, m);
    }
    // one add a block: atomics on one address are served one after the other
    if (threadIdx.x >= 64 && threadIdx.x < 66) {
        long long t = 0;
        for (int r = 0; r < MT_Y; ++r) t += ssum[threadIdx.x - 64][r];
        if (t) atomicAdd(words + (threadIdx.x == 64 ? DW_PHI : DW_C), (u64)t);
    }
    if (blockIdx.y == 0 && ty == 0 && i < p.nx) sincos(TWO_PI * (i + 0.5) / p.nx, &xtrig[i].y, &xtrig[i].x);
    const int jt = blockIdx.y * MT_Y + tx;
    if (blockIdx.x == 0 && ty == 1 && tx < MT_Y && jt < p.ny && !p.walls)
        sincos(TWO_PI * (jt + 0.5) / p.ny, &ytrig[jt].y, &ytrig[jt].x);
    if (!last_block(words + DW_DONE1)) return;

    // the centroid and the moments that follow from the column and row sums, by
    // one block, in units of w
    double v[6] = {0, 0, 0, 0, 0, 0};  // sum w, cos x, sin x; rows: cos y, sin y, y
    for (int k = threadIdx.x; k < p.nx; k += DIAG_THREADS) {
        const double s = (double)(long long)__ldcg(col + k);
        if (s == 0.0) continue;
        const double2 t = __ldcg(xtrig + k);
        v[0] += s;
        v[1] += s * t.x;
        v[2] += s * t.y;
    }
    for (int k = threadIdx.x; k < p.ny; k += DIAG_THREADS) {
        const double s = (double)(long long)__ldcg(row + k);
        if (s == 0.0) continue;
        if (p.walls) {
            v[5] += s * (k + 0.5);
            continue;
        }
        const double2 t = __ldcg(ytrig + k);
        v[3] += s * t.x;
        v[4] += s * t.y;
    }
    block_sum<6>(v);
    __shared__ double centre[2];
    if (threadIdx.x == 0) {  // (one thread: FP64 by all 256 would take the SM 12 us)
        double xc = 0.5 * p.nx, yc = 0.5 * p.ny;
        if (v[0] != 0.0) {
            double ax = atan2(v[2], v[1]);
            if (ax < 0) ax += TWO_PI;
            xc = ax * p.nx / TWO_PI;
            if (p.walls) {
                yc = v[5] / v[0];
            } else {
                double ay = atan2(v[4], v[3]);
                if (ay < 0) ay += TWO_PI;
                yc = ay * p.ny / TWO_PI;
            }
        }
        centre[0] = xc;
        centre[1] = yc;
    }
    __syncthreads();
    const double xc = centre[0], yc = centre[1];
    double I[2] = {0.0, 0.0};
    for (int k = threadIdx.x; k < p.nx; k += DIAG_THREADS) {
        const double d = min_image(k + 0.5 - xc, p.nx, true);
        I[0] += (double)(long long)__ldcg(col + k) * d * d;
    }
    for (int k = threadIdx.x; k < p.ny; k += DIAG_THREADS) {
        const double d = min_image(k + 0.5 - yc, p.ny, !p.walls);
        I[1] += (double)(long long)__ldcg(row + k) * d * d;
    }
    block_sum<2>(I);
    if (threadIdx.x != 0) return;
    const double sw0 = v[0] != 0.0 ? v[0] : 1.0;
    res[0] = (double)(long long)__ldcg(words + DW_PHI) / (double)p.fx_scale[0];
    res[1] = (double)(long long)__ldcg(words + DW_C) / (double)p.fx_scale[1];
    res[2] = xc;
    res[3] = yc;
    res[4] = (double)__ldcg(words + DW_NONFINITE);
    res[5] = (double)__ldcg(words + DW_SIGMA_NEG);
    res[6] = sqrt(__longlong_as_double((long long)__ldcg(words + DW_UMAX2)));
    res[7] = I[0] / sw0;
    res[8] = I[1] / sw0;
    res[13] = v[0];
}

// Pass 2: Ixy about the centroid, then the axes of the drop.  A thread owns a
// column of a band of rows: one multiply-add a cell.
__global__ void __launch_bounds__(DIAG_THREADS)
k_diag2(KParams p, const int* __restrict__ wmap, u64* __restrict__ words, double* __restrict__ res) {
    double* partial = reinterpret_cast<double*>(words + DW_COUNT + 3 * ((size_t)p.nx + p.ny));
    const double xc = res[2], yc = res[3];
    const int strips = (p.nx + DIAG_THREADS - 1) / DIAG_THREADS;
    const int band = blockIdx.x / strips, bands = gridDim.x / strips;
    const int i = (blockIdx.x - band * strips) * DIAG_THREADS + threadIdx.x;
    const int j0 = (int)((int64_t)p.ny * band / bands), j1 = (int)((int64_t)p.ny * (band + 1) / bands);
    double v[1] = {0.0};
    __shared__ double dy[32];
    for (int jb = j0; jb < j1; jb += 32) {
        __syncthreads();
        if (threadIdx.x < 32) dy[threadIdx.x] = min_image(jb + (int)threadIdx.x + 0.5 - yc, p.ny, !p.walls);
        __syncthreads();
        if (i >= p.nx) continue;
        for (int j = jb; j < min(j1, jb + 32); ++j) {
            const int w = wmap[(int64_t)j * p.nx + i];
            if (w) v[0] += fx_widen(w, 1.0f) * dy[j - jb];
        }
    }
    if (i < p.nx) v[0] *= min_image(i + 0.5 - xc, p.nx, true);
    block_sum<1>(v);
    if (threadIdx.x == 0) partial[blockIdx.x] = v[0];
    if (!last_block(words + DW_DONE2)) return;
    double t[1] = {0.0};
    for (int k = threadIdx.x; k < (int)gridDim.x; k += DIAG_THREADS) t[0] += __ldcg(partial + k);
    block_sum<1>(t);
    if (threadIdx.x != 0) return;
    const double I[3] = {res[7], res[8], res[13] != 0.0 ? t[0] / res[13] : 0.0};
    const double tr = I[0] + I[1], det = I[0] * I[1] - I[2] * I[2];
    const double disc = sqrt(fmax(0.25 * tr * tr - det, 0.0));
    const double l1 = 0.5 * tr + disc, l2 = fmax(0.5 * tr - disc, 0.0);
    const double L = 4.0 * sqrt(l1), B = 4.0 * sqrt(l2);
    res[9] = I[2];
    res[10] = L;
    res[11] = B;
    res[12] = (L + B) > 0.0 ? (L - B) / (L + B) : 0.0;
}

// ---------------------------------------------------------------------------
// FP64 statistics of given fields (fixed order: per-block partials, one
// finishing block)
// ---------------------------------------------------------------------------

__device__ __forceinline__ bool finite_cell(double a, double b, double c, double d) {
    return isfinite(a) && isfinite(b) && isfinite(c) && isfinite(d);
}

template <int NS>
__device__ void block_partial(double (&v)[NS], double* partial_out) {
    __shared__ double red[NS][DIAG_THREADS / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < NS; ++k) {
        double x = v[k];
        for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
        if (lane == 0) red[k][w] = x;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 0; k < NS; ++k) {
            double s = 0.0;
            for (int q = 0; q < DIAG_THREADS / 32; ++q) s += red[k][q];
            partial_out[k] = s;
        }
    }
}

// The drop indicator (see `drop_indicator`) of an FP64 phi.
__device__ __forceinline__ double drop_indicator_of(const KParams& p, double phi) {
    const double w = (phi - (double)p.phi_b) / ((double)p.phi_a - (double)p.phi_b);
    return fmin(fmax(w, 0.0), 1.0);
}

// Pass 1 sums: phi, c, w cos/sin(2 pi x / nx), w cos/sin(2 pi y / ny), w y,
// nonfinite count, sigma<0 count, max |u| (as max), w (w: drop indicator).
constexpr int STATS_SW = 10;  // slot of sum w; after pass 1, block 0's slot holds the total
__global__ void k_stats1(KParams p, const double* __restrict__ phi, const double* __restrict__ c,
                        const double* __restrict__ ux, const double* __restrict__ uy,
                        double* __restrict__ partial) {
    double v[STATS_NSUM];
    for (int k = 0; k < STATS_NSUM; ++k) v[k] = 0.0;
    double umax = 0.0;
    const int64_t n = (int64_t)p.nx * p.ny;
    for (int64_t o = (int64_t)blockIdx.x * DIAG_THREADS + threadIdx.x; o < n;
         o += (int64_t)gridDim.x * DIAG_THREADS) {
        const int i = (int)(o % p.nx), j = (int)(o / p.nx);
        const double f = phi[o], cc = c[o], a = ux[o], b = uy[o];
        if (!finite_cell(f, cc, a, b)) {
            v[7] += 1.0;
            continue;
        }
        const double ax = TWO_PI * (i + 0.5) / p.nx, ay = TWO_PI * (j + 0.5) / p.ny;
        const double w = drop_indicator_of(p, f);
        v[0] += f;
        v[1] += cc;
        v[2] += w * cos(ax);
        v[3] += w * sin(ax);
        v[4] += w * cos(ay);
        v[5] += w * sin(ay);
        v[6] += w * (j + 0.5);
        v[STATS_SW] += w;
        const double arg = 1.0 - cc * (double)p.inv_cmax;
        if (p.beta != 0.0f && (arg <= 0.0 || 1.0 + (double)p.beta * log(arg) < 0.0)) v[8] += 1.0;
        umax = fmax(umax, sqrt(a * a + b * b));
    }
    for (int o = 16; o > 0; o >>= 1) umax = fmax(umax, __shfl_down_sync(0xffffffffu, umax, o));
    __shared__ double smax[DIAG_THREADS / 32];
    if ((threadIdx.x & 31) == 0) smax[threadIdx.x >> 5] = umax;
    block_partial<STATS_NSUM>(v, partial + (int64_t)blockIdx.x * STATS_NSUM);
    if (threadIdx.x == 0) {
        double m = 0.0;
        for (int q = 0; q < DIAG_THREADS / 32; ++q) m = fmax(m, smax[q]);
        partial[(int64_t)blockIdx.x * STATS_NSUM + 9] = m;
    }
}

// result layout: [0] sum_phi [1] sum_c [2] xc [3] yc [4] nonfinite [5] sigma_neg [6] umax
//                [7] Ixx [8] Iyy [9] Ixy [10] L [11] B [12] D
// Sums over the nb partial rows (slot 9 by max instead when MAX9) by one
// block of STATS_FINISH threads: thread t adds rows t, t + STATS_FINISH, ... in
// order, then a fixed tree over the threads, so the result does not depend
// on scheduling.  Thread 0 receives the totals in s.
constexpr int STATS_FINISH = 256;
template <int NK, bool MAX9>
__device__ __forceinline__ void finish_sums(const double* __restrict__ partial, int nb,
                                            double s[NK]) {
    __shared__ double red[NK][STATS_FINISH];
    for (int k = 0; k < NK; ++k) s[k] = 0.0;
    for (int b = threadIdx.x; b < nb; b += STATS_FINISH)
        for (int k = 0; k < NK; ++k) {
            const double v = partial[(int64_t)b * STATS_NSUM + k];
            s[k] = (MAX9 && k == 9) ? fmax(s[k], v) : s[k] + v;
        }
    for (int k = 0; k < NK; ++k) red[k][threadIdx.x] = s[k];
    __syncthreads();
    for (int w = STATS_FINISH / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w)
            for (int k = 0; k < NK; ++k)
                red[k][threadIdx.x] = (MAX9 && k == 9)
                                          ? fmax(red[k][threadIdx.x], red[k][threadIdx.x + w])
                                          : red[k][threadIdx.x] + red[k][threadIdx.x + w];
        __syncthreads();
    }
    for (int k = 0; k < NK; ++k) s[k] = red[k][0];
}

__global__ void __launch_bounds__(STATS_FINISH) k_stats_finish1(KParams p, double* __restrict__ partial,
                                                              int nb, double* __restrict__ res) {
    double s[STATS_NSUM];
    finish_sums<STATS_NSUM, true>(partial, nb, s);
    if (threadIdx.x != 0) return;
    const double m = s[9];
    res[0] = s[0];
    res[1] = s[1];
    double xc = 0.5 * p.nx, yc = 0.5 * p.ny;
    if (s[STATS_SW] != 0.0) {
        double ax = atan2(s[3], s[2]);
        if (ax < 0) ax += TWO_PI;
        xc = ax * p.nx / TWO_PI;
        if (p.walls) {
            yc = s[6] / s[STATS_SW];
        } else {
            double ay = atan2(s[5], s[4]);
            if (ay < 0) ay += TWO_PI;
            yc = ay * p.ny / TWO_PI;
        }
    }
    res[2] = xc;
    res[3] = yc;
    res[4] = s[7];
    res[5] = s[8];
    res[6] = m;
    // the normalisation of pass 2 (the result array has no free slot)
    partial[STATS_SW] = s[STATS_SW];
}

__global__ void k_stats2(KParams p, const double* __restrict__ phi, const double* __restrict__ c,
                        const double* __restrict__ ux, const double* __restrict__ uy,
                        const double* __restrict__ res, double* __restrict__ partial) {
    double v[3] = {0.0, 0.0, 0.0};
    const double xc = res[2], yc = res[3];
    const int64_t n = (int64_t)p.nx * p.ny;
    for (int64_t o = (int64_t)blockIdx.x * DIAG_THREADS + threadIdx.x; o < n;
         o += (int64_t)gridDim.x * DIAG_THREADS) {
        const int i = (int)(o % p.nx), j = (int)(o / p.nx);
        const double f = phi[o];
        if (!finite_cell(f, c[o], ux[o], uy[o])) continue;
        const double dx = min_image(i + 0.5 - xc, p.nx, true);
        const double dy = min_image(j + 0.5 - yc, p.ny, !p.walls);
        const double w = drop_indicator_of(p, f);
        v[0] += w * dx * dx;
        v[1] += w * dy * dy;
        v[2] += w * dx * dy;
    }
    block_partial<3>(v, partial + (int64_t)blockIdx.x * STATS_NSUM);
}

__global__ void __launch_bounds__(STATS_FINISH) k_stats_finish2(const double* __restrict__ partial,
                                                              int nb, double* __restrict__ res) {
    double I[3];
    finish_sums<3, false>(partial, nb, I);
    if (threadIdx.x != 0) return;
    const double s0 = partial[STATS_SW];  // sum of the drop indicator (pass 1)
    if (s0 != 0.0)
        for (int k = 0; k < 3; ++k) I[k] /= s0;
    const double tr = I[0] + I[1], det = I[0] * I[1] - I[2] * I[2];
    const double disc = sqrt(fmax(0.25 * tr * tr - det, 0.0));
    const double l1 = 0.5 * tr + disc, l2 = fmax(0.5 * tr - disc, 0.0);
    const double L = 4.0 * sqrt(l1), B = 4.0 * sqrt(l2);
    res[7] = I[0];
    res[8] = I[1];
    res[9] = I[2];
    res[10] = L;
    res[11] = B;
    res[12] = (L + B) > 0.0 ? (L - B) / (L + B) : 0.0;
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------

static dim3 row_grid(const KParams& p, int bx) { return dim3((p.nx + bx - 1) / bx, p.ny); }

void launch_fields(const KParams& p, const DevState& s, int src, cudaStream_t st) {
    const int bx = 128;
    if (p.coupled)
        k_fields<true><<<row_grid(p, bx), bx, 0, st>>>(p, s.pop[src], s.fields);
    else
        k_fields<false><<<row_grid(p, bx), bx, 0, st>>>(p, s.pop[src], s.fields);
    k_normals<<<row_grid(p, bx), bx, 0, st>>>(p, s.fields);
}

void launch_step_split(const KParams& p, const DevState& s, int src, cudaStream_t st) {
    launch_fields(p, s, src, st);
    const int bx = 128;
    if (p.coupled)
        k_collide<true><<<row_grid(p, bx), bx, 0, st>>>(p, s.pop[src], s.pop[1 - src], s.fields);
    else
        k_collide<false><<<row_grid(p, bx), bx, 0, st>>>(p, s.pop[src], s.pop[1 - src], s.fields);
}

void launch_step_fused(const KParams& p, const DevState& s, int src, const FusedShape& sh,
                       cudaStream_t st) {
    const int tx = sh.bx - 4;
    dim3 grid((p.nx + tx - 1) / tx, (p.ny + sh.seg - 1) / sh.seg);
    const size_t smem = fused_smem_bytes(sh.bx);
    if (p.coupled)
        k_fused_sweep<true><<<grid, sh.bx, smem, st>>>(p, s.pop[src], s.pop[1 - src], s.fields,
                                                      sh.seg);
    else
        k_fused_sweep<false><<<grid, sh.bx, smem, st>>>(p, s.pop[src], s.pop[1 - src], s.fields,
                                                       sh.seg);
}

cudaError_t configure_fused_smem() {
    const int maxb = (int)fused_smem_bytes(128);
    cudaError_t e = cudaFuncSetAttribute(k_fused_sweep<true>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, maxb);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(k_fused_sweep<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                maxb);
}

namespace {

// f(coupled, storage format) as constants, and the shared memory of that form.
template <typename F>
cudaError_t with_macro(bool coupled, int st, F&& f) {
    using std::integral_constant;
    auto go = [&](auto C) {
        if (st == ST_F32) return f(C, integral_constant<int, ST_F32>{}, TileLayout<C(), ST_F32>::bytes(MT_Y));
        if (st == ST_F16) return f(C, integral_constant<int, ST_F16>{}, TileLayout<C(), ST_F16>::bytes(MT_Y));
        if (st == ST_BF16) return f(C, integral_constant<int, ST_BF16>{}, TileLayout<C(), ST_BF16>::bytes(MT_Y));
        return f(C, integral_constant<int, ST_NONE>{}, (size_t)0);
    };
    return coupled ? go(std::true_type{}) : go(std::false_type{});
}

dim3 macro_grid(const KParams& p) { return dim3((p.nx + MT_X - 1) / MT_X, (p.ny + MT_Y - 1) / MT_Y); }

}  // namespace

cudaError_t configure_macro_smem() {
    cudaError_t e = cudaSuccess;
    for (bool coupled : {false, true})
        for (int st : {ST_F32, ST_F16, ST_BF16})
            if (e == cudaSuccess)
                e = with_macro(coupled, st, [](auto C, auto S, size_t smem) {
                    cudaError_t a = cudaFuncSetAttribute(k_macro_out<C(), S()>,
                                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
                    return a != cudaSuccess ? a
                                            : cudaFuncSetAttribute(k_diag1<C(), S()>,
                                                                   cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                                   (int)smem);
                });
    return e;
}

void launch_macro_out(const KParams& p, const MacroSource& m, double* phi, double* c, double* ux, double* uy,
                      double* P, cudaStream_t st) {
    with_macro(p.coupled, m.map ? m.st : ST_NONE, [&](auto C, auto S, size_t smem) {
        k_macro_out<C(), S()><<<macro_grid(p), MT_X * MT_Y, smem, st>>>(m.map ? *m.map : CUtensorMap{}, p, m.pop,
                                                                        m.fields, m.err, phi, c, ux, uy, P);
        return cudaSuccess;
    });
}

void launch_init(const KParams& p, const DevState& s, int dst, const double* phi,
                 const double* c, const double* ux, const double* uy, const double* P,
                 cudaStream_t st) {
    const int bx = 128;
    k_init_fields<<<row_grid(p, bx), bx, 0, st>>>(p, phi, c, ux, uy, P, s.fields);
    k_normals<<<row_grid(p, bx), bx, 0, st>>>(p, s.fields);
    float* tmp = s.pop[1 - dst];
    if (p.coupled)
        k_init_pre<true><<<row_grid(p, bx), bx, 0, st>>>(p, s.fields, tmp);
    else
        k_init_pre<false><<<row_grid(p, bx), bx, 0, st>>>(p, s.fields, tmp);
    k_unstream<<<row_grid(p, bx), bx, 0, st>>>(p, s.nlat, tmp, s.pop[dst]);
}

void launch_get_pops(const KParams& p, const DevState& s, int src, double* out, cudaStream_t st) {
    const int bx = 128;
    k_export_pops<<<row_grid(p, bx), bx, 0, st>>>(p, s.nlat, s.pop[src], out);
}

void launch_set_pops(const KParams& p, const DevState& s, int dst, const double* f,
                     const double* h, const double* g, cudaStream_t st) {
    const int bx = 128;
    float* tmp = s.pop[1 - dst];
    k_pull_pre<<<row_grid(p, bx), bx, 0, st>>>(p, s.nlat, s.pop[dst], tmp);
    const double* in[3] = {f, h, g};
    for (int l = 0; l < s.nlat; ++l)
        if (in[l]) k_f64_to_pre<<<row_grid(p, bx), bx, 0, st>>>(p, l, in[l], tmp);
    k_unstream<<<row_grid(p, bx), bx, 0, st>>>(p, s.nlat, tmp, s.pop[dst]);
}

cudaError_t launch_diag(const KParams& p, const MacroSource& m, int* wmap, unsigned long long* words,
                        double* result, cudaStream_t st) {
    const cudaError_t e = cudaMemsetAsync(words, 0, sizeof(u64) * diag_words(p), st);
    if (e != cudaSuccess) return e;
    // 1 + beta log(arg) > 0 between these, with a margin for the FP32 arg
    const double span = p.beta != 0.0f ? 1.0 / std::fabs((double)p.beta) : 0.0;
    const float lo = (float)(std::exp(-span) + 1e-5), hi = (float)(std::exp(std::fmin(span, 80.0)) * 0.99999);
    with_macro(p.coupled, m.map ? m.st : ST_NONE, [&](auto C, auto S, size_t smem) {
        k_diag1<C(), S()><<<macro_grid(p), DIAG_THREADS, smem, st>>>(m.map ? *m.map : CUtensorMap{}, p, m.pop,
                                                                     m.fields, m.err, lo, hi, wmap, words, result);
        return cudaSuccess;
    });
    k_diag2<<<ixy_strips(p) * ixy_bands(p), DIAG_THREADS, 0, st>>>(p, wmap, words, result);
    return cudaSuccess;
}

int stats_blocks(const KParams& p) {
    const int64_t n = (int64_t)p.nx * p.ny;
    int64_t b = (n + DIAG_THREADS * 8 - 1) / (DIAG_THREADS * 8);
    if (b < 1) b = 1;
    if (b > 1024) b = 1024;
    return (int)b;
}

void launch_field_stats(const KParams& p, const double* phi, const double* c, const double* ux,
                        const double* uy, double* partial, int nb, double* result, cudaStream_t st) {
    k_stats1<<<nb, DIAG_THREADS, 0, st>>>(p, phi, c, ux, uy, partial);
    k_stats_finish1<<<1, STATS_FINISH, 0, st>>>(p, partial, nb, result);
    k_stats2<<<nb, DIAG_THREADS, 0, st>>>(p, phi, c, ux, uy, result, partial);
    k_stats_finish2<<<1, STATS_FINISH, 0, st>>>(partial, nb, result);
}

// ---------------------------------------------------------------------------
// 4-connected components of {phi > level}, periodic in x, and in y without walls
// ---------------------------------------------------------------------------
// Union-find on the cells, joined by atomic minima (Playne and Hawick, "A New
// Algorithm for Parallel Connected-Component Labelling on GPUs", IEEE TPDS 29(6),
// 2018): label[k] <= k points towards the smallest cell of k's tree.  Cells start pointing at the first cell of their run within 32 aligned
// columns; then every run is joined to its neighbours, each pair of runs once.
// Components = trees at the start - joins.  Bound by the latency of the chains of
// loads and atomics.  (Propagating the least label sweep by sweep, with a host
// read after each, took 234 us a call at 1024 x 512; now 68, 25 of them here.)

constexpr int LABEL_ROWS = 8;  // rows a block handles, one warp each

__global__ void __launch_bounds__(32 * LABEL_ROWS)
k_label_init(const KParams p, const float* __restrict__ src, float level, int* __restrict__ label,
             int* __restrict__ count) {
    const int tx = threadIdx.x & 31;
    const int i = blockIdx.x * 32 + tx, j = blockIdx.y * LABEL_ROWS + (threadIdx.x >> 5);
    bool in = false;
    if (i < p.nx && j < p.ny) {
        const ScalarMoments m = pull_scalar(src, p, 0, i, j);
        const int phi_fx = fx_add_sr(m.s0, m.inc, p.fx_scale[0], moment_bits(step_seed(p), i, j, p.nx));
        in = phi_fx != FX_INVALID && (float)phi_fx * p.fx_inv[0] > level;
    }
    const unsigned set = __ballot_sync(0xffffffffu, in);
    // the run's first lane: just above the highest clear bit below this lane
    const unsigned gap = ~set & ((1u << tx) - 1u);
    const int first = gap ? 32 - __clz(gap) : 0;
    const int k = j * p.nx + i;
    if (i < p.nx && j < p.ny) label[k] = in ? k - (tx - first) : -1;
    const int trees = __syncthreads_count(in && first == tx);
    if (threadIdx.x == 0 && trees) atomicAdd(count, trees);
}

// Join the trees of a and b; 1 if they were two.  Labels only ever fall and a
// label is below its cell, so the walks and the retries end.
__device__ __forceinline__ int join(int* label, int a, int b) {
    volatile int* L = label;
    while (true) {
        for (int n = L[a]; n != a; n = L[a]) a = n;
        for (int n = L[b]; n != b; n = L[b]) b = n;
        if (a == b) return 0;
        if (a < b) {
            const int t = a;
            a = b;
            b = t;
        }
        const int old = atomicMin(label + a, b);
        if (old == a) return 1;  // a was a root until now
        a = old;                 // it had a parent already: join that one
    }
}

__global__ void __launch_bounds__(32 * LABEL_ROWS)
k_label_join(const KParams p, int* __restrict__ label, int* __restrict__ count) {
    const int tx = threadIdx.x & 31;
    const int i = blockIdx.x * 32 + tx, j = blockIdx.y * LABEL_ROWS + (threadIdx.x >> 5);
    int joins = 0;
    if (i < p.nx && j < p.ny) {
        const int k = j * p.nx + i;
        auto inside = [&](int at) { return label[at] >= 0; };
        if (inside(k)) {
            const int left = j * p.nx + wrap_i(i - 1, p.nx);
            if ((tx == 0 || i == 0) && inside(left)) joins += join(label, k, left);
            if (j > 0 || !p.walls) {
                const int above = wrap_i(j - 1, p.ny) * p.nx;
                // the cell to the left has joined the same two runs already
                const bool again = tx > 0 && inside(left) && inside(above + i - 1);
                if (inside(above + i) && !again) joins += join(label, k, above + i);
            }
        }
    }
    for (int o = 16; o > 0; o >>= 1) joins += __shfl_down_sync(0xffffffffu, joins, o);
    if (tx == 0 && joins) atomicSub(count, joins);
}

cudaError_t launch_components(const KParams& p, const DevState& s, int src, float level, int* label, int* count,
                              cudaStream_t st) {
    const cudaError_t e = cudaMemsetAsync(count, 0, sizeof(int), st);
    if (e != cudaSuccess) return e;
    const dim3 grid((p.nx + 31) / 32, (p.ny + LABEL_ROWS - 1) / LABEL_ROWS);
    k_label_init<<<grid, 32 * LABEL_ROWS, 0, st>>>(p, s.pop[src], level, label, count);
    k_label_join<<<grid, 32 * LABEL_ROWS, 0, st>>>(p, label, count);
    return cudaSuccess;
}

}  // namespace lbm

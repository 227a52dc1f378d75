// One time step of one 32 x seg tile per block: the same cell arithmetic as
// the row sweep (lbm_sweep2.cuh), with all rows of the tile in flight at once
// instead of one row after the other.
//
// The sweep walks a strip row by row, and a row costs about 1.2 us whatever
// the grid (load, moments, barrier, normals, barrier, collisions), so a grid
// that does not fill the chip with long strips pays for the walk: 37 rows,
// 52 us, on any grid up to 512 x 256.  Here one thread issues the bulk-tensor
// loads of all staged rows of the tile (its own rows and three more each
// side), and the block then forms
//   A  phi, sigma and P* of every window cell (two columns and rows of halo),
//   B  the unit normal of the own cells and one ring around them,
//   C  the flow, phase-field and surfactant collisions of the own cells,
// one cell per thread and pass, with a barrier between the phases.  The halo
// costs 1.69 times the moments of the own cells at 32 x 8 but none of the
// collisions, and there is no ring to address: fewer instructions per cell
// than the sweep.  What bounds it is issue while three blocks per SM (shared
// memory) cover one another's loads.
#pragma once

#include <utility>

#include "lbm_sweep2.cuh"

namespace lbm {

constexpr int TILE_TX = 32;             // own columns: one warp per row of the tile
constexpr int TILE_WW = TILE_TX + 4;    // window columns x0-2 .. x0+33
constexpr int TILE_W = TILE_TX + 8;     // staged columns x0-4 .. x0+35 (16-byte aligned)
constexpr int TILE_NT = 256;
constexpr int TILE_SEG = 8;             // most rows of a tile

template <bool COUPLED, int ST>
struct TileLayout {
    static constexpr int NL = store_planes(ST, COUPLED);
    static constexpr int SLOT = (NL * TILE_W + 31) / 32 * 32;  // floats per staged row
    // window fields: phi (fixed point), and coupled sigma and P*
    static constexpr int NFIELD = COUPLED ? 3 : 1;
    __host__ __device__ static constexpr size_t bytes(int seg) {
        return 128 + sizeof(float) * ((size_t)(seg + 6) * SLOT + (size_t)NFIELD * (seg + 4) * TILE_WW +
                                      (size_t)5 * seg * TILE_TX);
    }
    // B writes the normals over the first words of the staged rows, which
    // belong to the scalar lattices and are read in A only
    static_assert((ST == ST_F32 ? 18 : 10) * TILE_W >= 3 * TILE_WW, "room for nx, ny, |grad phi|");
};

// Programmatic dependent launch: a step lets the next one be scheduled while its
// own last tiles run, and waits for the whole of the step before (and its writes)
// ahead of its first read.  Hides the launch latency of these short steps: us per
// step with snapshots, 512 x 256 14.8 -> 14.1, 301 x 167 BF16 7.5 -> 6.9, 128 x 128
// fixed velocity 4.8 -> 4.2.  The next step may start once a tile's loads have
// landed: let in at the kernel's first instruction, its waiting blocks cost more
// than they hide on the smallest grids (14.5, 6.9, 5.0).
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Launch with that attribute.
template <class... P, class... A>
void launch_after(void (*kernel)(P...), dim3 grid, size_t smem, cudaStream_t st, A&&... args) {
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(TILE_NT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}

// Tile (bxi, byi) of a run.  seg: rows per tile (4 .. TILE_SEG); seed_of(): the
// hash of the step (step_seed); err: device flag of the bounded wait.  With an
// `out` the block takes no step: it hands out(i, j, phi_fx, c_fx, ux, uy, P - P0)
// of its cells to it, one cell per thread at 8 rows.
struct TakeStep {};
template <bool COUPLED, int ST, class Seed, class Out = TakeStep>
__device__ __forceinline__ void tile_step(const CUtensorMap* tmap, const KParams& p, float* __restrict__ dst,
                                          const float* __restrict__ F, int seg, int bxi, int byi,
                                          Seed seed_of, int* __restrict__ err, Out out = Out()) {
    constexpr bool STEP = std::is_same<Out, TakeStep>::value;
    using L = TileLayout<COUPLED, ST>;
    constexpr int W = TILE_W, WW = TILE_WW, TX = TILE_TX, SLOT = L::SLOT;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    if (smem_u32(smem_raw) & 127u) {
        wait_for_previous();
        if (threadIdx.x == 0) atomicExch(err, 2);
        return;
    }
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem_raw);
    float* raw = reinterpret_cast<float*>(smem_raw + 128);
    int* s_phi = reinterpret_cast<int*>(raw + (seg + 6) * SLOT);
    float* s_sig = reinterpret_cast<float*>(s_phi) + (seg + 4) * WW;
    float* s_dps = s_sig + (seg + 4) * WW;
    float* mom = reinterpret_cast<float*>(s_phi) + L::NFIELD * (seg + 4) * WW;  // [5][seg * TX]

    const int t = threadIdx.x;
    const int x0 = bxi * TX, xend = min(x0 + TX, p.nx);
    const int y0 = byi * seg, y1 = min(y0 + seg, p.ny);
    const int rows = y1 - y0;
    if (t == 0) {
        mbar_init(bar, 1);
        mbar_init(bar + 1, 1);  // the failure-path test hook
        fence_barrier_init();
    }
    wait_for_previous();
    const uint32_t seed = seed_of();
    if (t == 0) {
        mbar_arrive_expect_tx(bar, (uint32_t)((rows + 6) * L::NL * W * sizeof(float)));
        for (int k = 0; k < rows + 6; ++k) {
            const int row = y0 - 3 + k;  // staged row k; rows beyond walls read fill values
            const int y = p.walls ? row : wrap_i(row, p.ny);
            tma_load_3d(raw + k * SLOT, tmap, x0 - 4 + XGHOST, y, 0, bar);
        }
    }
    __syncthreads();  // the barrier is initialised
    bool ok = mbar_wait_bounded(bar, 0);
    // failure-path test: wait on a barrier that no copy completes
    if (p.stall_test) ok = mbar_wait_bounded(bar + 1, 0, 4096) && ok;

    let_next_start();

    // ---------------- A: moments of the window ----------------
    if (ok) {
        for (int k = t; k < (rows + 4) * WW; k += TILE_NT) {
            const int r = k / WW, w = k - r * WW;
            const int col = x0 - 2 + w, row = y0 - 2 + r;
            if (col > xend + 1) continue;  // beyond a ragged last tile
            // a row beyond a wall is the mirror image of one of the tile
            const int jj = ext_row(row, p.ny, p.walls);
            const float* R0 = raw + (p.walls ? jj - y0 + 3 : r + 1) * SLOT;
            const float *Rm = R0 - SLOT, *Rp = R0 + SLOT;
            const bool bot = p.walls && jj == 0, top = p.walls && jj == p.ny - 1;
            const int cs = w + 2;
            ScalarMomentsV<f2, i2> m;
            if constexpr (ST == ST_F32)
                m = pull_scalars_fh<W>(Rm, R0, Rp, cs, bot, top, f2(p.fx_inv[0], p.fx_inv[1]));
            else
                m = pull_scalars_fh16<ST, W>(Rm, R0, Rp, cs, bot, top, p);
            const uint32_t b = moment_bits(seed, rmodm_rt(col, p.nx), jj, p.nx);
            s_phi[k] = fx_add_sr(m.s0.x, m.inc.x, p.fx_scale[0], b);
            const int c_fx = fx_add_sr(m.s0.y, m.inc.y, p.fx_scale[1], second_bits(b));
            if (w >= 2 && w < TX + 2 && r >= 2 && r < rows + 2) {
                float* o = mom + (r - 2) * TX + (w - 2);
                o[0] = m.jx.x;
                o[seg * TX] = m.jy.x;
                o[2 * seg * TX] = m.jx.y;
                o[3 * seg * TX] = m.jy.y;
                o[4 * seg * TX] = __int_as_float(c_fx);
            }
            if constexpr (COUPLED) {
                s_sig[k] = sigma_of_c(p, (float)c_fx * p.fx_inv[1]);
                float a[9];
                if constexpr (ST == ST_F32)
                    pull_flow_v<1, W>(Rm + 18 * W, R0 + 18 * W, Rp + 18 * W, cs, bot, top, a);
                else
                    pull_flow16_v<1, ST, W>(Rm, R0, Rp, cs, bot, top, p.qinv[2], a);
                s_dps[k] = sum9(a);
            }
        }
    }
    if (__syncthreads_or(!ok)) {
        // a staged row never landed: report, and let the copies in flight finish
        if (t == 0) {
            atomicExch(err, 1);
            mbar_wait_bounded(bar, 0);
        }
        return;
    }

    // normal of window cell (r, w) from the phi window
    auto normal_at = [&](int r, int w, float& nx, float& ny, float& gm) {
        int v[3][3];
#pragma unroll
        for (int d = 0; d < 3; ++d) stencil3i<1>(s_phi + (r - 1 + d) * WW, w, v[d]);
        float gx, gy;
        iso_grad_fx(v, p.fx_inv[0], gx, gy);
        unit_normal(gx, gy, nx, ny, gm);
    };
    // normals of window row r: nx, ny, |grad phi| in staged row r
    auto n_row = [&](int r) { return raw + r * SLOT; };

    // ---------------- B: normals ----------------
    if constexpr (COUPLED) {
        constexpr int BW = TX + 2;
        for (int k = t; k < (rows + 2) * BW; k += TILE_NT) {
            const int r = 1 + k / BW, w = 1 + k - (r - 1) * BW;
            float nx, ny, gm;
            normal_at(r, w, nx, ny, gm);
            float* o = n_row(r) + w;
            o[0] = nx;
            o[WW] = ny;
            o[2 * WW] = gm;
        }
        __syncthreads();
    }

    // ---------------- C: collisions of the own cells ----------------
    for (int k = t; k < rows * TX; k += TILE_NT) {
        const int j = k / TX, w = 2 + k - j * TX, r = j + 2;
        const int i = x0 + w - 2, jc = y0 + j;
        if (i >= xend) continue;
        const int at = r * WW + w;
        const int gi[1] = {i};
        const EdgeInfo<1> E(p, i, x0, xend, gi);
        const int phi_fx = s_phi[at];
        const float phi = i2f(phi_fx) * p.fx_inv[0];
        const int c_fx = __float_as_int(mom[4 * seg * TX + k]);
        float ux, uy, nx, ny;
        if constexpr (COUPLED) {
            CellGeomT<float> g;
            g.phi_fx = phi_fx;
            g.phi = phi;
            g.sig = s_sig[at];
            g.dps = s_dps[at];
            g.nx = n_row(r)[w];
            g.ny = n_row(r)[WW + w];
            g.gm = n_row(r)[2 * WW + w];
            float vx[3][3], vy[3][3], v[3][3];
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                stencil3<1>(n_row(r - 1 + d), w, vx[d]);
                stencil3<1>(n_row(r - 1 + d) + WW, w, vy[d]);
            }
            g.kappa = iso_div(vx, vy);
#pragma unroll
            for (int d = 0; d < 3; ++d) stencil3<1>(s_sig + (r - 1 + d) * WW, w, v[d]);
            iso_grad(v, g.sgx, g.sgy);
#pragma unroll
            for (int d = 0; d < 3; ++d) stencil3<1>(s_dps + (r - 1 + d) * WW, w, v[d]);
            iso_grad(v, g.pgx, g.pgy);
            if (!p.rho_uniform) {
                int vi[3][3];
#pragma unroll
                for (int d = 0; d < 3; ++d) stencil3i<1>(s_phi + (r - 1 + d) * WW, w, vi[d]);
                iso_grad_fx(vi, p.fx_inv[0], g.fgx, g.fgy);
            } else {
                g.fgx = g.fgy = 0.0f;
            }
            const float* R0 = raw + (j + 3) * SLOT;
            const bool bot = p.walls && jc == 0, top = p.walls && jc == p.ny - 1;
            float gg[9];
            if constexpr (ST == ST_F32)
                pull_flow_v<1, W>(R0 - SLOT + 18 * W, R0 + 18 * W, R0 + SLOT + 18 * W, w + 2, bot, top, gg);
            else
                pull_flow16_v<1, ST, W>(R0 - SLOT, R0, R0 + SLOT, w + 2, bot, top, p.qinv[2], gg);
            const CellOutT<float> o =
                collide_flow_cell(p, g, jc, gg, STEP, ST == ST_F32 ? 1.0f : p.qs[2]);
            if constexpr (!STEP) {
                out(i, jc, phi_fx, c_fx, o.ux, o.uy, o.dP);
                continue;
            }
            ux = o.ux;
            uy = o.uy;
            nx = g.nx;
            ny = g.ny;
            if constexpr (ST == ST_F32) {
                direct_stores<1, 9>(dst, p, 18, jc, gi, E, [&](int m) { return gg[m]; });
            } else {
                uint32_t wv[5];
                const uint32_t h = cell_bits(seed ^ 0x80000000u, i, jc, p.nx);
#pragma unroll
                for (int m = 0; m < 5; ++m)
                    wv[m] = pack2_sr<ST>(gg[2 * m], 2 * m + 1 < 9 ? gg[2 * m + 1 < 9 ? 2 * m + 1 : 8] : 0.0f,
                                         word_bits(h, 9 + m));
                direct_stores<1, 5>(dst, p, 10, jc, gi, E,
                                    [&](int m) { return __uint_as_float(wv[m]); });
            }
        } else {
            const int64_t idx = (int64_t)jc * p.pitch + i;
            ux = F[FP_UX * p.plane + idx];
            uy = F[FP_UY * p.plane + idx];
            if constexpr (!STEP) {
                out(i, jc, phi_fx, c_fx, ux, uy, 0.0f);
                continue;
            }
            float gm;
            normal_at(r, w, nx, ny, gm);
        }
        float df[9], dh[9];
        collide_scalars_pair(p, phi_fx, phi, (float)c_fx * p.fx_inv[1], nx, ny, ux, uy,
                             f2(mom[k], mom[2 * seg * TX + k]),
                             f2(mom[seg * TX + k], mom[3 * seg * TX + k]), df, dh,
                             ST == ST_F32 ? 1.0f : p.qs[0], ST == ST_F32 ? 1.0f : p.qs[1]);
        const float s_f = __int_as_float(phi_fx), s_h = __int_as_float(c_fx);
        if constexpr (ST == ST_F32) {
            direct_stores<1, 18>(dst, p, 0, jc, gi, E, [&](int m) {
                return m == 0 ? s_f : m == 9 ? s_h : m < 9 ? df[m] : dh[m - 9];
            });
        } else {
            uint32_t wv[8];
            const uint32_t h = cell_bits(seed, i, jc, p.nx);
#pragma unroll
            for (int q = 1; q < 9; ++q) wv[q - 1] = pack2_sr<ST>(df[q], dh[q], word_bits(h, q));
            direct_stores<1, 10>(dst, p, 0, jc, gi, E, [&](int m) {
                return m == 0 ? s_f : m == P16_SH ? s_h : __uint_as_float(wv[m >= P16_FH ? m - P16_FH : 0]);
            });
        }
    }
}

template <bool COUPLED, int ST>
__global__ void __launch_bounds__(TILE_NT, 3)
    k_tile(const __grid_constant__ CUtensorMap tmap, KParams p, float* __restrict__ dst,
           const float* __restrict__ F, int seg, int* __restrict__ err) {
    tile_step<COUPLED, ST>(&tmap, p, dst, F, seg, blockIdx.x, blockIdx.y, [&] { return step_seed(p); },
                           err);
}

}  // namespace lbm

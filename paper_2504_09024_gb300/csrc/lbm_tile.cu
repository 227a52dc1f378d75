// The tile-parallel step (lbm_tile.cuh): shapes and launches.
#include <type_traits>

#include "lbm_tile.cuh"

namespace lbm {

namespace {

template <typename F>
auto with_tile(bool coupled, int st, F&& f) {
    using std::integral_constant;
    auto go = [&](auto C) {
        if (st == ST_F16) return f(C, integral_constant<int, ST_F16>{});
        if (st == ST_BF16) return f(C, integral_constant<int, ST_BF16>{});
        return f(C, integral_constant<int, ST_F32>{});
    };
    return coupled ? go(std::true_type{}) : go(std::false_type{});
}

}  // namespace

int tile_map_bx() { return TILE_W - 4; }

cudaError_t configure_tile_smem() {
    cudaError_t e = cudaSuccess;
    for (bool coupled : {false, true})
        for (int st : {ST_F32, ST_F16, ST_BF16})
            if (e == cudaSuccess)
                e = with_tile(coupled, st, [](auto C, auto S) {
                    return cudaFuncSetAttribute(k_tile<C(), S()>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                (int)TileLayout<C(), S()>::bytes(TILE_SEG));
                });
    return e;
}

void launch_step_tile(const KParams& p, float* dst, const float* fields, int seg, const CUtensorMap& load_map,
                      int st, int* err, cudaStream_t s) {
    const dim3 grid((p.nx + TILE_TX - 1) / TILE_TX, (p.ny + seg - 1) / seg);
    with_tile(p.coupled, st, [&](auto C, auto S) {
        launch_after(k_tile<C(), S()>, grid, TileLayout<C(), S()>::bytes(seg), s, load_map, p, dst, fields, seg, err);
        return 0;
    });
}

}  // namespace lbm

// The launch rules as the library takes them, for tests/test_launch_rules.py:
// host code only, linked against the built library.
#include "lbm_launch.cuh"

namespace lbmk {
LBMK_EXTERN(MODE_F64)
LBMK_EXTERN(MODE_F32)
LBMK_EXTERN(MODE_F16)
LBMK_EXTERN(MODE_BF16)
}  // namespace lbmk

template <int M>
static lbmk::StepLaunch launch_of(int qt, int flow, int bounce, int nx, int ny, int form, dim3 b, bool chosen) {
    lbmk::StepParams<typename lbmk::ModeTraits<M>::R> P = {};
    P.nx = nx;
    P.ny = ny;
    P.solid_scheme = bounce;
    return lbmk::step_launch<M>(P, qt, flow, form, b, false, chosen);
}

// The one-step kernel's grid and block in columns and rows (out[0..3]) for a run
// in the given step form, with the run's own block shape or the chosen (bx, by).
extern "C" void rule_step(int mode, int qt, int flow, int bounce, int nx, int ny, int form, int bx, int by, int* out) {
    using namespace lbmk;
    const dim3 b = bx ? dim3(bx, by) : step_block(mode, nx, ny);
    const StepLaunch L = mode == MODE_F64   ? launch_of<MODE_F64>(qt, flow, bounce, nx, ny, form, b, bx != 0)
                         : mode == MODE_F32 ? launch_of<MODE_F32>(qt, flow, bounce, nx, ny, form, b, bx != 0)
                         : mode == MODE_F16 ? launch_of<MODE_F16>(qt, flow, bounce, nx, ny, form, b, bx != 0)
                                            : launch_of<MODE_BF16>(qt, flow, bounce, nx, ny, form, b, bx != 0);
    out[0] = (int)L.grid.x;
    out[1] = (int)L.grid.y;
    out[2] = (int)L.block.x;
    out[3] = (int)L.block.y;
}

// Whether grouped launches over `nodes` nodes take node pairs.
extern "C" int rule_group_pairs(int mode, int qt, int flow, long long nodes) {
    return lbmk::group_pairs(mode, qt, flow, nodes) ? 1 : 0;
}

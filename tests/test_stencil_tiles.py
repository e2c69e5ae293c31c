"""The vector stencil needs the level's tile list: without one it is an argument error, not a
product that was never formed."""
from native import run_without_device

SOURCE = r"""
#include <cstdio>
#include "dm_common.cuh"
int main() {
    const dm::VecOp<double, double> op{dm::Grid3{}, nullptr, nullptr, nullptr, nullptr, 0.0};
    for (int mode = 0; mode < dm::kStencilModes; ++mode) {
        int code = 0;
        try { dm::vec_stencil<double, double>(op, mode, nullptr, nullptr, nullptr, 0.0, nullptr); }
        catch (const dm::Error& e) { code = e.code; }
        std::printf("%d ", code);
    }
    return 0;
}
"""


def test_missing_tiles_are_an_error(tmp_path):
    assert run_without_device(SOURCE, tmp_path).split() == ["1"] * 4   # DM_ERR_INVALID_ARG

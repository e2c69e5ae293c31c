"""An allocation that fails leaves nothing behind that a later call would take for
a buffer: run without a device, where every allocation fails."""
from native import run_without_device

SOURCE = r"""
#include <cstdio>
#include "dm_common.cuh"
#include "dm_learned.cuh"
template <class F> int throws(F&& f) { try { f(); } catch (const dm::Error&) { return 1; } return 0; }
int main() {
    dm::DBuf<double> b;
    std::printf("%d ", throws([&] { b.alloc(100); }));
    std::printf("%d ", b.get() == nullptr && b.n == 0);
    // a buffer kept between calls: asked for again, it is allocated again
    std::printf("%d ", throws([&] { b.ensure(100); }));
    std::printf("%d ", throws([&] { b.ensure(100); }));
    dm::LearnedNet net;
    dm::Grid3 g{};
    g.nx = g.ny = g.nz = 4;
    g.sx = 8; g.sxy = 64; g.np = 512; g.off0 = 73;
    std::printf("%d ", throws([&] { net.alloc(g); }));
    std::printf("%d\n", throws([&] { net.alloc(g); }));
    return 0;
}
"""


def test_failed_allocations_are_asked_for_again(tmp_path):
    assert run_without_device(SOURCE, tmp_path).split() == ["1"] * 6

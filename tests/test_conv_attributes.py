"""The convolutions' shared-memory opt-in belongs to the device that is current, so
every launch needs it on its own device: checked on the host with faked device calls."""
from native import run_without_device

SOURCE = r"""
#include <cuda_runtime.h>
#include <cstdio>
#include <set>
namespace {
int g_dev = 0;
std::set<std::pair<int, const void*>> g_set;   // (device, kernel) that have the opt-in
cudaError_t fake_get(int* d) { *d = g_dev; return cudaSuccess; }
cudaError_t fake_attr(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
template <class K> cudaError_t fake_set(K* k, cudaFuncAttribute, int) {
    g_set.insert({g_dev, (const void*)k});
    return cudaSuccess;
}
}
#define cudaGetDevice fake_get
#define cudaDeviceGetAttribute fake_attr
#define cudaFuncSetAttribute fake_set
#include "dm_conv_tc.cu"
int main() {
    dm::Grid3 g{};
    g.nx = g.ny = g.nz = 4;
    g.sx = 8; g.sxy = 64; g.np = 512; g.off0 = 73;
    const dm::ActLayout L = dm::act_layout(g);
    int counts[2];
    for (g_dev = 0; g_dev < 2; ++g_dev) {
        auto launch = [&](auto&& f) { try { f(); } catch (const dm::Error&) {} };   // (no device: the launch itself fails)
        for (int cb = 1; cb <= 2; ++cb)
            for (int epi = 0; epi < (cb == 1 ? 2 : 3); ++epi)
                launch([&] { dm::conv_tc(g, L, cb, epi, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr); });
        for (int cb = 1; cb <= 2; ++cb)
            launch([&] { dm::conv_dw_tc(g, L, cb, 8, nullptr, 1, 3, nullptr, nullptr, nullptr, nullptr, nullptr); });
        counts[g_dev] = 0;
        for (const auto& e : g_set) counts[g_dev] += e.first == g_dev;
    }
    std::printf("%d %d\n", counts[0], counts[1]);
    return 0;
}
"""


def test_opt_in_on_every_device(tmp_path):
    first, second = map(int, run_without_device(SOURCE, tmp_path).split())
    assert first == second == 7   # five convolutions and two weight gradients

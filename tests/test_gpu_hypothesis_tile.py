"""The hypothesis tile is a build option (PILOT_HYP_TILE: 2, 4 or 8 hypotheses per build-pass CTA):
the reductions of the build pass follow it.  A small library is compiled per value; sums of whole
numbers are exact, so they are compared with equality."""
import ctypes as ct
import os
import subprocess

import numpy as np
import pytest

from paper_2606_31098_gb300 import build_ext

from gpu_support import require_cuda

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "pilot_build_impl.cuh"
using namespace pilot;
__device__ float value(int lane, int warp, int i) { return (float)((lane * 37 + warp * 11 + i * 5) % 101); }
template <int APB, bool SCATTER> __global__ void slots(float* out) {
    __shared__ __align__(16) float red[kBuildThreads / 32][kHypTile][kAcc];
    float acc[kNumSums];
    for (int i = 0; i < kNumSums; ++i) acc[i] = value(threadIdx.x & 31, threadIdx.x >> 5, i);
    const float v = cta_reduce_slots<kBuildThreads, APB, SCATTER>(acc, red);
    if (threadIdx.x < kHypTile * kAcc) out[threadIdx.x] = v;
}
template <int APB> __global__ void spread(float* out, int* roles) {
    __shared__ float red[kBuildThreads / 32][kAcc];
    constexpr int n = sizeof(RoleTable::sum) / kHypTile;
    float acc[n];
    for (int i = 0; i < n; ++i) acc[i] = value(threadIdx.x & 31, threadIdx.x >> 5, i);
    const float v = cta_reduce_spread<APB>(acc, red);
    if (threadIdx.x < kAcc) out[threadIdx.x] = v;
    if (threadIdx.x == 0)
        for (int k = 0; k < kHypTile * n; ++k) roles[k] = kRoles.sum[k / n][k % n];
}
extern "C" int run(int apb, float* a, float* b, float* c, int* roles) {
    if (apb == 1) slots<1, true><<<1, kBuildThreads>>>(a), slots<1, false><<<1, kBuildThreads>>>(b), spread<1><<<1, kBuildThreads>>>(c, roles);
    if (apb == 2) slots<2, true><<<1, kBuildThreads>>>(a), slots<2, false><<<1, kBuildThreads>>>(b), spread<2><<<1, kBuildThreads>>>(c, roles);
#if PILOT_HYP_TILE == 2
    if (apb == 4) slots<4, true><<<1, kBuildThreads>>>(a), slots<4, false><<<1, kBuildThreads>>>(b), spread<4><<<1, kBuildThreads>>>(c, roles);
#endif
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.mark.parametrize("tile", [2, 4, 8])
def test_reductions_follow_the_hypothesis_tile(tile, tmp_path):
    torch = require_cuda()
    src, lib = tmp_path / "tile.cu", tmp_path / f"libtile{tile}.so"
    src.write_text(SOURCE)
    flags = [f for f in build_ext.NVCC_FLAGS if f != "-lineinfo"]
    subprocess.run([build_ext.nvcc(), *build_ext.ARCH, *flags, f"-DPILOT_HYP_TILE={tile}", "-shared", str(src), "-o", str(lib)],
                   check=True, capture_output=True, text=True)
    fn = ct.CDLL(os.fspath(lib)).run
    fn.argtypes = [ct.c_int] + [ct.c_void_p] * 4
    lane, warp = np.arange(32)[:, None, None], np.arange(8)[None, :, None]
    for apb in [a for a in (1, 2, 4) if a * tile <= 8]:        # the channel layouts' (anchors per group batch)
        slot = (np.arange(32) // apb) % tile
        value = (lane * 37 + warp * 11 + np.arange(32) * 5) % 101
        want = np.zeros((tile, 32))
        for h in range(tile):
            want[h, :29] = value[slot == h][:, :, :29].sum((0, 1))
        a, b = torch.zeros((tile, 32), device="cuda"), torch.zeros((tile, 32), device="cuda")
        c, roles = torch.zeros(32, device="cuda"), torch.zeros(32, device="cuda", dtype=torch.int32)
        assert fn(apb, a.data_ptr(), b.data_ptr(), c.data_ptr(), roles.data_ptr()) == 0
        np.testing.assert_array_equal(a.cpu().numpy(), want)
        np.testing.assert_array_equal(b.cpu().numpy(), want)
        # one hypothesis: every sum belongs to one slot's lanes
        r = roles.cpu().numpy().reshape(tile, 32 // tile)
        assert sorted(r[r < 29]) == list(range(29))
        got = c.cpu().numpy()
        for h in range(tile):
            for i, s in enumerate(r[h]):
                if s < 29:
                    assert got[s] == value[slot == h][:, :, i].sum()

"""The radix passes and the active list when a tile's wait for the tiles before
it runs out: the sources built with a limit of no polls at all
(SPH_WAIT_POLLS = 0), so that a tile that does not find its predecessors' words
at the first look counts their items itself. The results are numpy's exactly."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

SRC = r"""
#define SPH_WAIT_POLLS 0
#include "grid.cu"
#include "noalloc.cu"
// work: flag_work_bytes(n) bytes, cleared
extern "C" int flags_to_list(const uint8_t* flag, int n, long long tick, int max_bin, unsigned long long* work,
                             int32_t* list, uint32_t* count) {
    sph::k_flag_list<<<(n + sph::kCpTile - 1) / sph::kCpTile, sph::kCpT>>>(flag, n, tick, max_bin, work, list, count,
                                                                         sph::CallBegin());
    return (int)cudaGetLastError();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2003_10850_gb300 import build
    d = tmp_path_factory.mktemp("waits")
    (d / "waits.cu").write_text(SRC)
    subprocess.run([build.nvcc(), *build.ARCH, *build.NVCC_FLAGS, "-shared", "-o", str(d / "waits.so"),
                    str(d / "waits.cu")], check=True, capture_output=True, text=True)
    return ctypes.CDLL(os.path.join(d, "waits.so"))


def _p(t):
    return ctypes.c_void_p(t.data_ptr())


# two tiles, more than the eight read at a time, more than run at once
@pytest.mark.parametrize("n", [8193, 40_960, 300_007, 1 << 20])
@pytest.mark.parametrize("values", [1, 5000])
def test_sort(lib, n, values):
    rng = np.random.default_rng(n + values)
    keys = rng.integers(0, 2**64, size=values, dtype=np.uint64)[rng.integers(0, values, size=n)]
    order = np.argsort(keys, kind="stable")
    k = torch.from_numpy(keys.view(np.int64)).cuda()
    out, perm = torch.full_like(k, -1), torch.full((n,), -1, dtype=torch.int32, device="cuda")
    assert lib.sph_sort_keys_static(_p(k), ctypes.c_int64(n), _p(out), _p(perm), None) == 0
    torch.cuda.synchronize()
    assert np.array_equal(out.cpu().numpy().view(np.uint64), keys[order])
    assert np.array_equal(perm.cpu().numpy(), order.astype(np.int32))


@pytest.mark.parametrize("n", [4097, 140_003, 2_000_003])
@pytest.mark.parametrize("max_bin", [-1, 5])
def test_active_list(lib, n, max_bin):
    rng = np.random.default_rng(n)
    flag = rng.integers(0, 7, n).astype(np.uint8) if max_bin >= 0 else (rng.random(n) < 0.3).astype(np.uint8)
    tick = 12   # a multiple of 4: bins from max_bin - 2 up are active
    on = np.minimum(flag, max_bin) >= max_bin - 2 if max_bin >= 0 else flag != 0
    f = torch.from_numpy(flag).cuda()
    work = torch.zeros((n + 4095) // 4096 + 1, dtype=torch.int64, device="cuda")
    lst = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    count = torch.zeros(1, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    assert lib.flags_to_list(_p(f), n, ctypes.c_longlong(tick), max_bin, _p(work), _p(lst), _p(count)) == 0
    torch.cuda.synchronize()
    want = np.nonzero(on)[0]
    got = lst.cpu().numpy()
    assert int(count) == len(want)
    assert np.array_equal(got[: len(want)], want) and np.all(got[len(want):] == -1)

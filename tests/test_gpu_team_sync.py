"""The team barrier and sums of csrc/common.cuh between the CTAs of a
cluster team and of a global-memory team, on the GPU.

* A barrier orders the whole block's writes, not only those of the warp that
  posts: every warp but the first stores late, and the next CTA reads each word
  after a plain barrier.  Words and sums are whole numbers, compared exactly.
* A status word that one CTA sets before its post ends the team on every CTA at
  that sync or the next one, even when all of them arrive.
* What tells such a launch: cluster_matches.
"""
import ctypes
import os
import subprocess

import pytest
import torch

from paper_2210_06874_gb300 import build_lib

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
HERE = os.path.dirname(os.path.abspath(__file__))
P = ctypes.c_void_p


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("team") / "libteam_sync_probe.so")
    subprocess.run([build_lib.nvcc(), *build_lib.ARCH, *build_lib.FLAGS, "-shared", "-o", so,
                    os.path.join(HERE, "team_sync_probe.cu")], check=True)
    lib = ctypes.CDLL(so)
    lib.probe_control_bytes.restype = ctypes.c_ulonglong
    lib.probe_exchange.argtypes = [P, P, P] + [ctypes.c_int] * 4
    lib.probe_status.argtypes = [P, P] + [ctypes.c_int] * 4
    lib.probe_matches.argtypes = [P] + [ctypes.c_int] * 3
    return lib


def control(lib):
    return torch.zeros(lib.probe_control_bytes(), dtype=torch.uint8, device=DEV)


@pytest.mark.parametrize("grid,threads,cluster", [(2, 256, 1), (8, 640, 1), (16, 640, 1),
                                                  (2, 256, 0), (16, 640, 0), (96, 256, 0)])
def test_barrier_orders_every_warp(probe, grid, threads, cluster):
    ctl = control(probe)
    data = torch.zeros(grid * threads, dtype=torch.int32, device=DEV)
    bad = torch.zeros(1, dtype=torch.int32, device=DEV)
    torch.cuda.synchronize()
    assert probe.probe_exchange(ctl.data_ptr(), data.data_ptr(), bad.data_ptr(), grid, threads,
                                200, cluster) == 0
    assert int(bad) == 0


@pytest.mark.parametrize("kind", [0, 1, 2])
@pytest.mark.parametrize("grid,setter", [(2, 1), (33, 0), (96, 95)])
def test_status_ends_the_sync(probe, grid, setter, kind):
    ctl = control(probe)
    res = torch.full((grid,), -1, dtype=torch.int32, device=DEV)
    torch.cuda.synchronize()
    assert probe.probe_status(ctl.data_ptr(), res.data_ptr(), grid, 256, setter, kind) == 0
    assert set(res.tolist()) <= {2, 3}          # of 8 syncs


@pytest.mark.parametrize("grid,launched,size,want", [(8, 4, 4, 1), (8, 8, 8, 1), (8, 4, 2, 0),
                                                     (8, 2, 4, 0), (8, 0, 2, 0), (8, 0, 1, 1)])
def test_launch_without_its_clusters_is_told(probe, grid, launched, size, want):
    res = torch.full((grid,), -1, dtype=torch.int32, device=DEV)
    torch.cuda.synchronize()
    assert probe.probe_matches(res.data_ptr(), grid, launched, size) == 0
    assert res.tolist() == [want] * grid

"""The kernels that the bench says ran: its copies of the library's launch
rules at the rules' edges (152 SMs), template arguments as many as the
kernels have, and the grid check's bytes."""
import os
import re

import pytest

import bench

CSRC = os.path.join(os.path.dirname(os.path.abspath(bench.__file__)), "paper_1904_06680_gb300", "csrc")
SMS = 152


@pytest.mark.parametrize("W,N,want", [
    (16, 133 * 16, "16,8,4,6,0,4,0,0"), (16, 133 * 16 + 1, "16,4,4,4,0,4,0,0"), (16, 16 * 8 * SMS, "16,4,4,4,0,4,0,0"),
    (16, 16 * 8 * SMS + 1, "16,4,20,1,0,4,0,1"), (16, 20480, "16,4,20,1,0,4,0,1"), (16, 20 * 8 * SMS, "16,4,20,1,0,4,0,1"),
    (16, 20 * 8 * SMS + 1, "16,4,4,4,0,4,0,0"), (32, 133 * 8, "32,16,4,5,0,8,0,0"), (32, 133 * 8 + 1, "32,8,4,4,0,8,0,0"),
    (64, 16383, "64,32,4,4,0,16,0,0"), (64, 16384, "64,16,4,3,0,8,8,0")])
def test_trajectory_kernels(W, N, want):
    assert bench.traj_kernel_name(W, N, SMS) == "traj_tmem_kernel<%s>" % want
    assert bench.traj_kernel_name(W, N, SMS, var=True, option=3).startswith("traj_tmem_kernel<%d," % W)
    assert bench.traj_kernel_name(W, N, SMS, option=3).startswith("traj_kernel<%d," % W)


@pytest.mark.parametrize("N,want", [(160 * SMS - 1, "64,32,4,4,1,16,0,8,4"), (160 * SMS, "64,32,24,1,1,10,6,8,4")])
def test_windowed_kernels(N, want):
    assert bench.fused_kernel_name(64, N, SMS, var=True) == "fused_tmem_kernel<%s>" % want
    assert bench.fused_kernel_name(64, N, SMS, option=1) == "fused_tmem_kernel<64,32,24,1,0,10,6,8,4>"


@pytest.mark.parametrize("N,M,T,want", [(8192, 63, 127, 16), (8191, 63, 127, 32), (8192, 64, 127, 32), (8192, 63, 128, 32),
                                        (20480, 20, 200, 32)])
def test_states_check(N, M, T, want):
    assert bench.check_kernel_name(M, N, T, -1) == "collide_states_kernel<%d>" % want


def test_binned_checks():
    name = bench.check_kernel_name
    assert name(8702, 1024, 40, 5) == "collide_grid_kernel"
    for M, N, T, chunks in ((8703, 1024, 40, 1), (8702, 1023, 40, 1), (8702, 1024, 65535, 1), (8702, 1024, 40, 2)):
        assert name(M, N, T, 5, chunks=chunks) == "collide_binned_kernel<0>"
    assert name(2000, 9999, 40, -1, poly=True) == "collide_binned_kernel<1>"
    assert name(2000, 9999, 40, 2, poly=True) == "collide_poly_kernel"


def test_as_many_template_arguments_as_the_kernels_have():
    text = open(os.path.join(CSRC, "npp_rollout.cuh")).read()
    for kernel, name in (("traj_tmem_kernel", bench.traj_kernel_name(16, 20480, SMS)),
                         ("traj_kernel", bench.traj_kernel_name(16, 20480, SMS, option=3)),
                         ("fused_tmem_kernel", bench.fused_kernel_name(64, 20480, SMS)),
                         ("fused_kernel", bench.fused_kernel_name(32, 20480, SMS))):
        args = re.search(r"template <([^>]*)>\s*__global__[^;{]*\b%s\(" % kernel, text).group(1)
        assert name.startswith(kernel + "<") and name.count(",") == args.count(","), kernel


def test_grid_check_bytes():
    """The course: 16 chunks of 1024 samples at 41 steps."""
    assert bench.GRID_POINTS == 8702
    blocks = 16 * 41 * (32768 + 8 * 2000)
    assert bench.grid_check_bytes(16384, 40, 2000, SMS, 1000) == blocks + 20 * 1000 + 12 * 16384
    # chunks of at most 1024 samples, at most 1024 of them
    assert bench.grid_check_bytes(2048, 200, 0, SMS, 0) == 2 * 201 * 32768 + 12 * 2048
    assert bench.grid_check_bytes(1 << 21, 1, 0, SMS, 0) == 1024 * 2 * 32768 + 12 * (1 << 21)

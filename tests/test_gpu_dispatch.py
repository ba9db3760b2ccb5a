"""Which kernels a step launches: the path that tfkt_step_path names is the one that
tfkt_step switches on (the counters of tfkt_step_profiled name the first and second
launch of a step, whichever kernels they are)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    import torch
    assert torch.cuda.is_available()
    from paper_2201_10132_gb300 import build, tfkt
    build.build()
    return tfkt


def _params(T, prec, nx, ny, S=6, R=3.0, stress=False):
    return T.Params(nx, ny, S, R, 5.0, 2.0 if stress else 0.5, 0.5 if stress else 0.2, 0.05, 1,
                    0.03 if stress else 0.0, 0.0, 1, getattr(T, prec), 0.0, int(stress))


@pytest.mark.parametrize("prec,nx,ny,path", [
    ("FP64", 64, 32, "split"), ("FP64", 70, 19, "two_pass"), ("FP64", 640, 64, "split"),
    ("FP64", 609, 57, "two_pass"),
    ("FP32", 64, 32, "split"), ("FP32", 160, 160, "split"), ("FP32", 416, 64, "fused"),   # 100, 104 tiles
    ("FP32", 601, 58, "two_pass"), ("FP32", 609, 57, "fused"),                            # 152, 160 tiles
    ("FP16", 416, 64, "split"), ("FP16", 608, 64, "split"), ("FP16", 640, 64, "fused"),   # 152, 160 tiles
    ("FP16", 601, 58, "two_pass"), ("FP16", 609, 57, "fused")])
@pytest.mark.parametrize("stress", [False, True])
def test_step_path(T, prec, nx, ny, path, stress):
    with T.Solver(_params(T, prec, nx, ny, stress=stress)) as s:
        assert s.step_path() == path
        ms, n = np.zeros(len(T.KERNELS)), np.zeros(len(T.KERNELS), np.int64)
        s.step_profiled(2, ms, n)
        assert s.step_path() == path
    assert n.tolist() == ([1, 2, 0, 0] if path == "two_pass" else [0, 0, 2, 2])


@pytest.mark.parametrize("prec,nx,ny,path", [("FP64", 64, 16, "two_pass"), ("FP32", 416, 64, "two_pass")])
def test_large_disks_take_two_passes(T, prec, nx, ny, path):
    """156 Q-nodes are more than a tile's shared memory holds."""
    with T.Solver(_params(T, prec, nx, ny, 14, 7.0)) as s:
        assert s.step_path() == path


def test_a_slab_steps_as_its_whole_run(T):
    with T.Slab(_params(T, "FP32", 416, 64), 0, 32) as a, T.Slab(_params(T, "FP32", 160, 160), 0, 80) as b:
        assert a.step_path() == "fused" and b.step_path() == "split"


def test_the_step_after_a_learned_block_is_fused(T):
    p = T.Params(64, 32, 6, 3.0, 10.0, 1.0, 0.2, 0.05, 1, 0.0, 0.0, 1, T.FP32)
    with T.Solver(p) as s:
        s.step(2)
        T.lpm_run(s, None, 1, K=4, mode=T.LPM_FROZEN)
        assert s.step_path() == "fused"
        s.step(1)
        assert s.step_path() == "split"

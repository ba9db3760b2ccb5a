"""FP64 runs of one Q-node on grids that fill the GPU form U in a pass of its own before the
collision (from 77824 nodes on); others in the collision. Same results: 1e-12 against the
oracle on both sides of the line, and slabs, each of which alone is below it, bit for bit."""
import numpy as np
import pytest

from test_gpu_paths import _check, _params
from test_gpu_slabs import FIELDS, _run_slabs, _single

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    import torch
    assert torch.cuda.is_available()
    from paper_2201_10132_gb300 import build, tfkt
    build.build()
    return tfkt


@pytest.mark.parametrize("nx,ny", [(288, 272), (301, 263), (256, 288)])   # 78336, 79163, 73728 nodes
@pytest.mark.parametrize("stress", [False, True])
def test_matches_oracle(T, oracle_mod, nx, ny, stress):
    _check(T, oracle_mod, _params(T, nx, ny, 1, 1.0, "FP64", stress), 4, "FP64")


@pytest.mark.parametrize("nx,ny,parts", [(288, 272, 2), (301, 263, 3)])
def test_slabs_are_bit_identical(T, nx, ny, parts):
    from paper_2201_10132_gb300.inputs import perturbation
    p = _params(T, nx, ny, 1, 1.0, "FP64")
    pert = perturbation(nx, ny, 9, 0.05, 0.05)
    ref, ref_psi, ref_pops = _single(T, p, pert, 8)
    got, psi, pops, _ = _run_slabs(T, p, pert, parts, 8)
    for k in FIELDS:
        assert np.array_equal(got[k], ref[k], equal_nan=True), k
    assert np.array_equal(psi, ref_psi) and np.array_equal(pops, ref_pops)

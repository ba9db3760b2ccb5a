"""The fused kernel, mostly on whole tiles, which every large run takes: FP32 grids of more than 100
and FP16 grids of more than 152 tiles of 32 x 8. Parity with the oracle over the physical
options, slabs, checkpoints, batches of single-run kernels and captured steps: the cases of
the other files, whose grids are small enough for the Q-split kernels, above that line.
Tolerances are those of tests/test_gpu_parity.py and test_gpu_paths.py (FP32 2e-5, FP16
storage 3e-3 of the field's scale); the others are bit for bit."""
import numpy as np
import pytest

from test_checkpoint import test_resume_is_bit_exact as _resume
from test_gpu_paths import TOL, SCALE, _check, test_steps_captured_in_a_graph as _captured
from test_gpu_slabs import FIELDS, _params as _slab_params, _run_slabs, _single

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    import torch
    assert torch.cuda.is_available()
    from paper_2201_10132_gb300 import build, tfkt
    build.build()
    return tfkt


def _grid(prec, shape):
    """104 and 160 tiles; one column and one row of tiles, which are their own neighbours."""
    return {"block": {"FP32": (416, 64), "FP16": (640, 64)}, "column": {"FP32": (32, 840), "FP16": (32, 1240)},
            "row": {"FP32": (3360, 8), "FP16": (4960, 8)}}[shape][prec]


# S, R, re, wi, beta, tau2, ic, fene_b, stress (as in tests/test_gpu_parity.py)
OPTIONS = {
    "momentum": (6, 3.0, 5.0, 0.5, 0.2, 0.0, 1, 0.0, 0),
    "rest-52": (8, 4.0, 5.0, 0.5, 0.2, 0.0, 0, 0.0, 0),
    "tau2": (6, 3.0, 4.0, 1.0, 0.5, 0.3, 1, 0.0, 0),
    "newtonian": (4, 2.0, 3.0, 0.0, 1.0, 0.0, 1, 0.0, 0),
    "all-bounce": (2, 1.0, 5.0, 0.5, 0.2, 0.0, 1, 0.0, 0),
    "fene": (6, 3.0, 5.0, 2.0, 0.2, 0.0, 1, 3.1, 0),
    "stress": (6, 3.0, 5.0, 2.0, 0.5, 0.03, 1, 0.0, 1),
    "stress-fene": (6, 3.0, 5.0, 2.0, 0.5, 0.03, 1, 3.1, 1),
}


@pytest.mark.parametrize("prec", ["FP32", "FP16"])
@pytest.mark.parametrize("shape,option", [("block", o) for o in OPTIONS] +
                         [("column", "momentum"), ("column", "stress"), ("row", "momentum")])
def test_matches_oracle(T, oracle_mod, prec, shape, option):
    from paper_2201_10132_gb300.inputs import perturbation
    nx, ny = _grid(prec, shape)
    S, R, re, wi, beta, tau2, ic, fene, qe = OPTIONS[option]
    pert = perturbation(nx, ny, 7, 0.05, 0.05)
    o = oracle_mod.Oracle(oracle_mod.map_params(nx, ny, S, R, re, wi, beta, 0.05, 1, tau2, 0.0, fene, qe))
    o.init(pert, ic)
    o.step(4)
    f = o.fields()
    p = T.Params(nx, ny, S, R, re, wi, beta, 0.05, 1, tau2, 0.0, ic, getattr(T, prec), fene, qe)
    with T.Solver(p, pert) as s:
        assert s.step_path() == "fused"
        s.step(4)
        g = s.moments(list(SCALE))
    scale = {}
    for k, t in SCALE.items():
        scale[t] = max(scale.get(t, 0.0), np.abs(f[k]).max())
    for k, t in SCALE.items():
        err = np.abs(g[k] - f[k]).max() / max(scale[t], 1e-300)
        assert err < TOL[prec], (k, err)


@pytest.mark.parametrize("nx,ny", [(609, 57), (33, 617), (1, 1225)])
@pytest.mark.parametrize("prec,beta", [("FP16", 0.2), ("FP16", 1.0), ("FP32", 1.0)])
def test_partial_tiles_with_one_q_node(T, oracle_mod, nx, ny, prec, beta):
    """The form of the kernel for a few Q-nodes in FP16 storage."""
    p = T.Params(nx, ny, 1, 1.0, 5.0, 0.0 if beta == 1.0 else 0.5, beta, 0.05, 1, 0.0, 0.0, 1, getattr(T, prec))
    with T.Solver(p) as s:
        assert s.step_path() == "fused"
    _check(T, oracle_mod, p, 3, prec)


@pytest.mark.parametrize("nx,ny,parts,prec,stress", [
    (416, 64, 2, "FP32", False), (416, 72, 3, "FP32", False), (640, 64, 2, "FP16", False),
    (416, 64, 2, "FP32", True), (640, 64, 2, "FP16", True)])
def test_slabs_are_bit_identical(T, nx, ny, parts, prec, stress):
    from paper_2201_10132_gb300.inputs import perturbation
    p = _slab_params(T, nx, ny, prec, stress)
    pert = perturbation(nx, ny, 9, 0.05, 0.05)
    with T.Solver(p) as s:
        assert s.step_path() == "fused"
    ref, ref_psi, ref_pops = _single(T, p, pert, 12)
    got, psi, pops, _ = _run_slabs(T, p, pert, parts, 12)
    for k in FIELDS:
        assert np.array_equal(got[k], ref[k], equal_nan=True), k
    assert np.array_equal(psi, ref_psi)
    assert np.array_equal(pops, ref_pops)


@pytest.mark.parametrize("case", [(416, 64, 6, 3.0, 5.0, 0.5, 0.2, 1, 1, "FP32", 0),
                                  (640, 64, 6, 3.0, 5.0, 0.5, 0.2, 1, 0, "FP16", 0),
                                  (609, 57, 4, 1.6, 5.0, 0.5, 0.2, 1, 1, "FP32", 0)],   # partial tiles
                         ids=lambda c: f"{c[9]}-{c[0]}x{c[1]}")
def test_resume_is_bit_exact(T, tmp_path, case):
    with T.Solver(T.Params(*case[:7], 0.05, case[7], 0.0, 0.0, case[8], getattr(T, case[9]))) as s:
        assert s.step_path() == "fused"
    _resume(T, tmp_path, case)


@pytest.mark.parametrize("nx,ny,prec", [(416, 64, "FP32"), (640, 64, "FP16"), (609, 57, "FP32")])
def test_steps_captured_in_a_graph(T, nx, ny, prec):
    with T.Solver(T.Params(nx, ny, 6, 3.0, 5.0, 0.5, 0.2, 0.05, 1, precision=getattr(T, prec))) as s:
        assert s.step_path() == "fused"
    _captured(T, nx, ny, prec)


@pytest.mark.parametrize("steps", [1, 6, 7])
def test_per_run_batch_is_bit_identical(T, steps, monkeypatch):
    """Single-run kernels as graph branches: two runs on the fused kernel, one on the Q-split
    kernels."""
    from paper_2201_10132_gb300.inputs import perturbation
    monkeypatch.setenv("TFKT_BATCH_PER_RUN", "1")
    grids = [(416, 64, 6, 3.0), (64, 32, 6, 3.0), (352, 96, 3, 1.5)]
    params = [T.Params(nx, ny, S, R, 5.0, 0.5, 0.2, 0.05, 1, 0.0, 0.0, 1, T.FP32) for nx, ny, S, R in grids]
    perts = [perturbation(g[0], g[1], 3 + k, 0.05, 0.05) for k, g in enumerate(grids)]
    with T.Batch(params, perts) as b:
        assert b.plan()["per_run"]
        assert [b.run(k).step_path() for k in range(3)] == ["fused", "split", "fused"]
        b.step(steps)
        got = [b.run(k).moments() for k in range(3)]
    for p, pert, g in zip(params, perts, got):
        with T.Solver(p, pert) as s:
            s.step(steps)
            ref = s.moments()
        for k in ref:
            assert np.array_equal(g[k], ref[k], equal_nan=True), k

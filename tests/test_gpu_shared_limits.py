"""Contexts and batches of different Q-disks alive together: a kernel's shared-memory limit is
shared by all of them, so none may lower it under what another one launches with."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

DISK = {32: (6, 3.0), 9: (3, 1.5)}


@pytest.fixture(scope="module")
def T():
    import torch
    assert torch.cuda.is_available()
    from paper_2201_10132_gb300 import build, tfkt
    build.build()
    return tfkt


def _params(T, nq, nx, ny):
    return T.Params(nx, ny, *DISK[nq], 5.0, 0.5, 0.2, 0.05, 1, 0.0, 0.0, 1, T.FP32)


def _alone(T, p, steps):
    with T.Solver(p) as s:
        s.step(steps)
        return s.moments()


def _close(got, ref):
    u = max(np.abs(ref[k]).max() for k in ("ux", "uy"))
    for k in ref:
        scale = u if k in ("ux", "uy", "vort") else np.abs(ref[k]).max()
        assert np.abs(got[k] - ref[k]).max() <= 2e-5 * max(scale, 1e-30), k


@pytest.mark.parametrize("first", [32, 9])
@pytest.mark.parametrize("plan", [{"TFKT_BATCH_PER_RUN": "1"}, {"TFKT_BATCH_TILE_HEIGHT": "8"}])
def test_two_live_batches(T, monkeypatch, first, plan):
    """Both are created before either steps (its graph is captured at the first step of two);
    416 x 64 nodes take the fused kernel in the per-run plan too."""
    for k, v in plan.items():
        monkeypatch.setenv(k, v)
    second = 41 - first
    p = {n: _params(T, n, 416, 64) for n in (first, second)}
    with T.Batch([p[first]]) as a, T.Batch([p[second]]) as b:
        a.step(3)
        b.step(3)
        a.step(1)
        got = {first: a.run(0).moments(), second: b.run(0).moments()}
    _close(got[first], _alone(T, p[first], 4))
    _close(got[second], _alone(T, p[second], 3))


def test_solver_with_fewer_q_nodes_between_steps_of_a_batch(T, monkeypatch):
    monkeypatch.setenv("TFKT_BATCH_PER_RUN", "1")
    p, q = _params(T, 32, 416, 64), _params(T, 9, 416, 64)
    with T.Batch([p]) as b, T.Solver(q) as s:
        for _ in range(3):
            s.step(1)
            b.step(1)       # an odd step launches without the graph
        _close(b.run(0).moments(), _alone(T, p, 3))
        _close(s.moments(), _alone(T, q, 3))

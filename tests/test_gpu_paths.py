"""Kernel paths of the step at the sizes where they can go wrong, against the oracle:
the Q-split kernels (small grids, ragged grids, FP64) at node counts around a group
of 32 nodes, Q-node counts around the warps of a block and grids on both sides of
the line to the fused kernel, and the fused kernel just above that line and with
partial tiles, also split into slabs.
Tolerances are those of tests/test_gpu_parity.py: FP64 1e-12, FP32 2e-5, FP16
storage 3e-3 of the field's scale."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TOL = {"FP64": 1e-12, "FP32": 2e-5, "FP16": 3e-3}
SCALE = {"ux": "u", "uy": "u", "cxx": "c", "cxy": "c", "cyy": "c", "thxx": "t", "thxy": "t",
         "thyy": "t", "rho_s": "rho_s", "psi_tot": "psi_tot"}


@pytest.fixture(scope="module")
def T():
    import torch
    assert torch.cuda.is_available()
    from paper_2201_10132_gb300 import build, tfkt
    build.build()
    return tfkt


def _params(T, nx, ny, S, R, prec, stress=False, fene=0.0):
    return T.Params(nx, ny, S, R, 5.0, 2.0 if stress or fene else 0.5, 0.5 if stress else 0.2, 0.05, 1,
                    0.03 if stress else 0.0, 0.0, 1, getattr(T, prec), fene, int(stress))


def _check(T, O, p, steps, prec):
    from paper_2201_10132_gb300.inputs import perturbation
    pert = perturbation(p.nx, p.ny, 7, 0.05, 0.05) if p.nx * p.ny > 1 else None
    o = O.Oracle(O.map_params(p.nx, p.ny, p.q_side, p.q_radius, p.re, p.wi, p.beta, p.u0,
                              p.k_periods, p.tau2, 0.0, p.fene_b, p.qe_model))
    o.init(pert, p.ic_mode)
    o.step(steps)
    f = o.fields()
    with T.Solver(p, pert) as s:
        s.step(steps)
        g = s.moments(list(SCALE))
    scale = {}
    for k, t in SCALE.items():
        scale[t] = max(scale.get(t, 0.0), np.abs(f[k]).max())
    for k, t in SCALE.items():
        err = np.abs(g[k] - f[k]).max() / max(scale[t], 1e-300)
        assert err < TOL[prec], (k, err)


# 1, 4, 5 and 9 Q-nodes, then 12, 32, 29 and 52
SIZES = [(1, 33, 1, 1.0), (31, 1, 2, 1.0), (32, 8, 3, 1.0), (11, 3, 3, 1.5),
         (33, 31, 4, 2.0), (5, 13, 6, 3.0), (97, 50, 7, 3.0), (72, 72, 8, 4.0)]


# (FP16 storage leaves out the one-row grid: its viscous length is 1/(2 pi) node, its stress
# mode hardly damped, and the rounding of the stored populations reaches 1e-2 of the
# velocity with any of the kernels.)
@pytest.mark.parametrize("prec,nx,ny,S,R", [(prec,) + c for prec in TOL for c in SIZES
                                            if not (prec == "FP16" and c[1] == 1)])
def test_q_split_sizes(T, oracle_mod, nx, ny, S, R, prec):
    _check(T, oracle_mod, _params(T, nx, ny, S, R, prec), 6, prec)


@pytest.mark.parametrize("prec,stress,fene", [("FP32", False, 0.0), ("FP16", False, 0.0),
                                              ("FP32", True, 0.0), ("FP16", True, 0.0),
                                              ("FP32", False, 3.1), ("FP32", True, 3.1)])
@pytest.mark.parametrize("nx,ny", [(160, 160), (416, 64), (601, 58), (609, 57)])   # 100, 104, 152, 160 tiles of 32 x 8
def test_both_sides_of_the_tile_line(T, oracle_mod, nx, ny, prec, stress, fene):
    _check(T, oracle_mod, _params(T, nx, ny, 6, 3.0, prec, stress, fene), 4, prec)


# Partial tiles of the fused kernel (more than 152 tiles): last tiles of 1, 3, 31 and 30 by 1, 7
# and 2 nodes, and grids of one tile column or row, whose tile is its own neighbour.
PARTIAL = [(33, 617), (99, 311), (639, 63), (1, 1225), (4898, 5), (62, 610)]


# (the stress model refuses this momentum relaxation time on five rows)
@pytest.mark.parametrize("nx,ny,prec,stress,fene", [
    c + k for c in PARTIAL for k in (("FP32", False, 0.0), ("FP16", False, 0.0), ("FP32", True, 0.0),
                                     ("FP16", True, 3.1)) if not (k[1] and c[1] == 5)])
def test_fused_partial_tiles(T, oracle_mod, nx, ny, prec, stress, fene):
    p = _params(T, nx, ny, 4, 1.6, prec, stress, fene)
    with T.Solver(p) as s:
        k, ms = np.zeros(len(T.KERNELS), np.int64), np.zeros(len(T.KERNELS))
        s.step_profiled(1, ms, k)
    assert k[T.KERNELS.index("fused")] == 1     # the fused kernel ran
    _check(T, oracle_mod, p, 3, prec)


@pytest.mark.parametrize("nx,ny,parts,prec", [(575, 70, 3, "FP32"), (575, 70, 2, "FP16"),
                                              (576, 65, 4, "FP32"), (33, 620, 5, "FP32")])
def test_slabs_of_partial_tiles_are_bit_identical(T, nx, ny, parts, prec):
    """Slabs keep the whole run's tile rows wherever they start."""
    import torch
    from paper_2201_10132_gb300 import slabs as S
    from paper_2201_10132_gb300.inputs import perturbation
    p = _params(T, nx, ny, 4, 1.6, prec)
    pert = perturbation(nx, ny, 9, 0.05, 0.05)
    with T.Solver(p, pert) as s:
        s.step(9)
        ref = s.populations()
    slabs = [T.Slab(p, y0, n, S.local_perturbation(pert, y0, n)) for y0, n in S.partition(ny, parts)]
    bufs = [[torch.empty(s.halo_bytes(), dtype=torch.uint8, device="cuda") for _ in (0, 1)] for s in slabs]
    S.exchange_local(slabs, bufs)
    for _ in range(9):
        for s in slabs:
            s.step(1)
        S.exchange_local(slabs, bufs)
    got = np.concatenate([s.owned(s.populations()) for s in slabs], axis=1)
    for s in slabs:
        s.close()
    assert np.array_equal(got, ref)


@pytest.mark.parametrize("prec", ["FP32", "FP16"])
@pytest.mark.parametrize("S,R", [(1, 1.0), (3, 1.0), (3, 1.5), (6, 3.0), (7, 3.0)])
def test_field_sums_of_fp32_contexts(T, S, R, prec):
    """psi_tot, C and Q_rms against FP64 sums over the same psi(r, q): both sides round a
    sum of positive terms at most nq + 4 times."""
    from paper_2201_10132_gb300.inputs import perturbation
    p = _params(T, 45, 19, S, R, prec)
    with T.Solver(p, perturbation(45, 19, 5, 0.05, 0.05)) as s:
        s.step(4)
        psi, f = s.psi(), s.moments(["psi_tot", "cxx", "cxy", "cyy", "qrms"])
    h = 0.5 * (S - 1)
    Q = np.array([(i - h, j - h) for j in range(S) for i in range(S)
                  if (i - h) ** 2 + (j - h) ** 2 <= R * R + 1e-9])
    pt = psi.sum(-1)
    c = {k: 2.0 * (psi * w).sum(-1) / pt for k, w in
         (("cxx", Q[:, 0] ** 2), ("cxy", Q[:, 0] * Q[:, 1]), ("cyy", Q[:, 1] ** 2))}
    tr = c["cxx"] + c["cyy"]
    eps = 2 * (len(Q) + 4) * 2.0 ** -53
    assert np.abs(f["psi_tot"] - pt).max() <= eps * np.abs(pt).max()
    for k in c:
        assert np.abs(f[k] - c[k]).max() <= 2 * eps * np.abs(tr).max(), k
    assert np.abs(f["qrms"] ** 2 - tr).max() <= 4 * eps * np.abs(tr).max()


@pytest.mark.parametrize("nx,ny,prec", [(64, 32, "FP32"), (40, 24, "FP32"), (416, 64, "FP16")])
def test_steps_captured_in_a_graph(T, nx, ny, prec):
    """tfkt_step under the caller's stream capture: three replays of two captured steps
    leave the state of six plain steps."""
    import torch
    from paper_2201_10132_gb300.inputs import perturbation
    p = _params(T, nx, ny, 6, 3.0, prec)
    pert = perturbation(nx, ny, 3, 0.05, 0.05)
    with T.Solver(p, pert) as s:
        s.step(6)
        ref = s.moments()
    st = torch.cuda.Stream()
    with T.Solver(p, pert, stream=st.cuda_stream) as s:
        s.sync()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            s.step(2)
        with torch.cuda.stream(st):
            for _ in range(3):
                g.replay()
        st.synchronize()
        got = s.moments()
    for k in ref:
        assert np.array_equal(got[k], ref[k], equal_nan=True), k


@pytest.mark.parametrize("n", [1, 127, 128, 129, 152 * 128, 152 * 128 + 1, 40000])
def test_training_gradient_over_tile_counts(T, n):
    """Loss and gradient for sample counts at the edges of a tile of 128 samples and of one
    tile per block, against FP64 autograd with the same bfloat16 matrices (1e-4 of each
    tensor's largest magnitude, as in tests/test_gpu_lpm.py); the caller's copy of the
    gradient may be at any 4-byte boundary, and so may the samples."""
    import torch
    from paper_2201_10132_gb300 import train_lpm
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    vec, _ = train_lpm.load()
    w = {k: torch.from_numpy(np.array(v)).cuda() for k, v in T.unpack_mlp(vec).items()}
    X = torch.empty(n * T.MLP_IN + 1, device="cuda")[1:].view(n, T.MLP_IN)
    X.copy_(torch.randn((n, T.MLP_IN), generator=g, device="cuda") * w["sx"] + w["mx"])
    Y = torch.randn((n, T.MLP_OUT), generator=g, device="cuda") * w["st"] + w["mt"]
    grad = torch.empty(T.MLP_NWEIGHTS + 1, device="cuda")[1:]
    net = T.Mlp(vec)
    loss = net.loss_grad(X.data_ptr(), Y.data_ptr(), n, grad.data_ptr())
    net.close()
    p = [(w[k].bfloat16() if k[0] == "W" else w[k]).double().requires_grad_()
         for k in ("W1", "b1", "W2", "b2", "W3", "b3")]
    act = torch.nn.functional.gelu
    x = (X.double() - w["mx"].double()) / w["sx"].double()
    t = (Y.double() - w["mt"].double()) / w["st"].double()
    o = act(act(x @ p[0].T + p[1]) @ p[2].T + p[3]) @ p[4].T + p[5]
    ref = ((o - t) ** 2).sum() / n
    assert loss == pytest.approx(float(ref), rel=1e-4)
    k = 0
    for r in torch.autograd.grad(ref, p):
        got = grad[k:k + r.numel()].double().view_as(r)
        k += r.numel()
        assert (got - r).abs().max() <= 1e-4 * r.abs().max()

"""A context's workspace holds what its kernels read, and not what only others' do."""
import pytest


@pytest.fixture(scope="module")
def T():
    from paper_2201_10132_gb300 import build, tfkt
    build.build()
    return tfkt


@pytest.mark.parametrize("nx,ny,S,R,nq,buffers", [(64, 64, 8, 4.0, 52, 2), (512, 512, 6, 3.0, 32, 2),
                                                  (70, 64, 8, 4.0, 52, 1), (64, 64, 14, 7.0, 156, 1)])
def test_fp64_workspace_holds_no_fused_kernel_data(T, nx, ny, S, R, nq, buffers):
    """Two population buffers, the moment planes (double-buffered on whole tiles up to 58
    Q-nodes), U, and tables of at most 1 kB per Q-node, 32 bytes per row and 0.1 MB of partial
    sums; no ring exports and table images, which only the fused kernel reads."""
    p = T.Params(nx, ny, S, R, 5.0, 0.5, 0.2, 0.05, 1, precision=T.FP64)
    pitch = -(-nx // 32) * 32
    planes = (2 * (9 + 25 * nq) + buffers * (nq + 6) + 2) * 8 * pitch * ny
    extra = T.required_bytes(p) - planes
    assert 0 < extra < 1024 * nq + 32 * ny + 100_000

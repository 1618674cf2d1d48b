"""Backprojection of ragged tiles, where whole warps (8 x 4 columns of a 16 x
16 tile) lie outside the square and take no part: squares that end 1 to 15
voxels into a tile along each axis, with and without shared views, whole
volumes and slabs, against the oracle (bars as in test_gpu_parity.py:
rel-RMSE <= 1e-5, max error <= 2e-4 of the largest value)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

REL_RMSE = 1e-5
MAX_REL = 2e-4


@pytest.fixture(scope="module")
def fd():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_1708_07515_gb300 as fd
    fd.load()
    return fd


def _cmp(got, want, what):
    err = got.astype(np.float64) - want
    rel = np.linalg.norm(err) / np.linalg.norm(want)
    mx = np.abs(err).max() / np.abs(want).max()
    assert rel <= REL_RMSE and mx <= MAX_REL, f"{what}: rel-RMSE {rel:.3e}, max-rel {mx:.3e}"


@pytest.mark.parametrize("N,P,s,D,split", [
    (17, 24, 0, 1, 4),     # one column and one row past a tile
    (20, 24, 0, 2, 2),     # 4: the last rows fill one row of warps
    (41, 24, 1, 1, 4),     # 20 and 21
    (24, 8, 0, 1, 1),      # 8: the last columns fill one warp
    (57, 8, 1, 1, 1),      # 28 and 29
    (31, 8, 0, 1, 1),      # 15: no warp idle
    (5, 12, 1, 2, 1),      # smaller than a warp
])
def test_every_remainder(fd, oracle_mod, N, P, s, D, split):
    R, Nu = 3.0 * N, N + 3 + (-(N + 3)) % 4
    Q = np.random.default_rng(N).standard_normal((P, N + 1, Nu)).astype(np.float32)
    Qd = torch.from_numpy(Q).cuda()
    want = oracle_mod.fdkod(Q, R, N, s, D)
    with fd.Plan(R, N, Nu, N + 1, P, s, D) as plan:
        assert fd.fdkod_get_forms(plan.handle)["bp_split"] == split
        got = plan.backproject(Qd).cpu().numpy()
        z0, nz = N // 3, max(1, N // 2)
        v0, nr = plan.slab_rows(z0, nz)
        work = torch.empty(max(1, plan.slab_workspace_elems(nr)), device="cuda")
        slab = plan.backproject_slab(Qd[:, v0:v0 + nr].contiguous(), v0, work, z0, nz).cpu().numpy()
        assert plan.device_status() == 0
    _cmp(got, want, f"N={N}")
    _cmp(slab, want[z0:z0 + nz], f"slab of N={N}")

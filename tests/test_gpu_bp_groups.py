"""The staged backprojection's forms against the FP64 oracle.

The pair kernel walks its slices in groups of 16, 8 or 4, or one by one, by
the view's largest row drift |1/U - 1| per slice (below 1/15, 1/7, 1/3, or
any), and holds 16 or 32 slice pairs per thread by the number of CTAs.  The
source distances here make each group size occur (R = 40 N: 16 only; 4 N: 16,
8 and 4; 2 N and 1.2 N: all), at sizes whose tiles and slabs end ragged.
Bars as in test_gpu_parity.py: rel-RMSE <= 1e-5, max error <= 2e-4 of the
largest value (float32 arithmetic on identical Q)."""
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


def _smooth_q(rng, P, Nv, Nu):
    """Random filtered projections, smooth along rows and columns."""
    Q = rng.standard_normal((P, Nv, Nu))
    for ax in (1, 2):
        Q = Q + np.roll(Q, 1, ax) + np.roll(Q, -1, ax)
    return Q.astype(np.float32)


@pytest.mark.parametrize("ratio", [40.0, 4.0, 2.0, 1.2])
@pytest.mark.parametrize("N,P,s,D", [(33, 24, 0, 1), (48, 24, 1, 2), (65, 36, 2, 3)])
def test_every_group_size(fd, oracle_mod, N, P, s, D, ratio):
    R = ratio * N
    Q = _smooth_q(np.random.default_rng(int(10 * ratio) + N), P, N + 3, N + 3 + (-(N + 3)) % 4)
    with fd.Plan(R, N, Q.shape[2], Q.shape[1], P, s, D) as plan:
        got = plan.backproject(torch.from_numpy(Q).cuda()).cpu().numpy()
        assert plan.device_status() == 0
    _cmp(got, oracle_mod.fdkod(Q, R, N, s, D), f"N={N} R={ratio}N")


@pytest.mark.parametrize("N,P,s,D,qtype", [
    (16, 10, 0, 1, "f32"),     # clusters of 2 (5 views each)
    (33, 43, 1, 1, "bf16"),    # of 8, uneven ranges of views
    (96, 90, 1, 2, "f32"),     # of 4
    (130, 128, 1, 2, "f32"),   # of 4 in two waves, ragged tiles
    (131, 66, 0, 2, "f32"),    # of 2
    (64, 45, 1, 1, "f16"),
])
def test_views_shared_by_a_cluster(fd, oracle_mod, N, P, s, D, qtype):
    R = 3.0 * N
    Q = _smooth_q(np.random.default_rng(P), P, N, N + (-N) % 8)
    t = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}[qtype]
    Qd = torch.from_numpy(Q).to(t).cuda()
    with fd.Plan(R, N, Q.shape[2], N, P, s, D, qtype=qtype) as plan:
        got = plan.backproject(Qd)
        again = plan.backproject(Qd)
        assert plan.device_status() == 0
    assert torch.equal(got, again)   # the ranges are added in a fixed order
    _cmp(got.cpu().numpy(), oracle_mod.fdkod(Qd.float().cpu().numpy(), R, N, s, D), f"N={N} P={P}")


@pytest.mark.parametrize("ratio", [4.0, 1.6])
@pytest.mark.parametrize("qtype", ["f32", "f16"])
def test_many_tiles_sampled_slices(fd, oracle_mod, qtype, ratio):
    """An odd volume with enough tiles for 32 slice pairs per thread: the
    first and last slices, the middle one (its own mirror image) and both
    sides of a slab's end; FDK-OD and plain FDK."""
    N, P, s, D = 245, 24, 2, 2
    R = ratio * N
    Q = _smooth_q(np.random.default_rng(77), P, N, 248)
    zs = np.array([0, 31, 32, 122, 213, 244])
    Qd = torch.from_numpy(Q).to({"f32": torch.float32, "f16": torch.float16}[qtype]).cuda()
    Qr = Qd.float().cpu().numpy()
    with fd.Plan(R, N, 248, N, P, s, D, qtype=qtype) as plan:
        sel = torch.from_numpy(zs).cuda()
        got = plan.backproject(Qd)[sel].cpu().numpy()
        plain = plan.backproject_plain(Qd)[sel].cpu().numpy()
        assert plan.device_status() == 0
    _cmp(got, oracle_mod.fdkod_slices(Qr, R, N, s, D, zs), f"FDK-OD {qtype} R={ratio}N")
    _cmp(plain, oracle_mod.fdk_slices(Qr, R, N, zs), f"plain FDK {qtype} R={ratio}N")


@pytest.mark.parametrize("ratio", [4.0, 1.6, 1.2])
@pytest.mark.parametrize("N,s,D,z0,nz", [
    (245, 2, 2, 30, 192),   # 32 slices per slab and thread
    (245, 2, 1, 228, 17),   # the volume's last slices, a second slab wholly past the end
    (61, 1, 3, 0, 33),      # one slice past a CTA's slabs
    (61, 1, 1, 20, 1),
])
def test_slabs_equal_the_whole_volume(fd, N, s, D, z0, nz, ratio):
    """Slabs (two slabs per CTA, not mirrored) from just the detector rows
    they read, against the whole volume's mirrored pairs: float32 rounding of
    the same sums (rel-RMSE 1e-5, as slabs against whole volumes elsewhere)."""
    P, Nv = 24, N + 2
    Nu = N + (-N) % 4
    Q = torch.from_numpy(_smooth_q(np.random.default_rng(N + nz), P, Nv, Nu)).cuda()
    with fd.Plan(ratio * N, N, Nu, Nv, P, s, D) as plan:
        whole = plan.backproject(Q)
        v0, nr = plan.slab_rows(z0, nz)
        rows = Q[:, v0:v0 + nr].contiguous()
        work = torch.empty(max(1, plan.slab_workspace_elems(nr)), device="cuda")
        slab = plan.backproject_slab(rows, v0, work, z0, nz)
        assert plan.device_status() == 0
    want = whole[z0:z0 + nz]
    err = (slab.double() - want.double()).norm() / want.double().norm()
    assert float(err) <= 1e-5, float(err)

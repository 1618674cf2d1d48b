"""A staging-window width selected with fdkod_set_tile changes the layout in
shared memory, never the result: bit for bit the same volume at every valid
width, also where the wider windows leave no room for the ring of the
32-slice form (volumes with enough tiles for it), for slabs, and for 16-bit
windows."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

_TYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}


@pytest.fixture(scope="module")
def fd():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_1708_07515_gb300 as fd
    fd.load()
    return fd


@pytest.mark.parametrize("N,P,s,D,r,qtype", [
    (245, 24, 2, 2, 4.0, "f32"),    # 32 slices per slab
    (245, 24, 2, 1, 4.0, "f16"),
    (245, 24, 2, 2, 1.3, "f32"),    # larger windows
    (200, 12, 2, 1, 4.0, "f32"),    # 16, no shared views
    (72, 40, 1, 2, 3.0, "f32"),     # views shared by a cluster
])
def test_every_width_gives_the_same_bits(fd, N, P, s, D, r, qtype):
    from paper_1708_07515_gb300 import autotune
    Nu = N + (-N) % 8
    gen = torch.Generator(device="cuda").manual_seed(N)
    Q = torch.randn((P, N, Nu), device="cuda", generator=gen).to(_TYPES[qtype])
    with fd.Plan(r * N, N, Nu, N, P, s, D, qtype=qtype) as plan:
        z0, nz = N // 3, 40
        v0, nr = plan.slab_rows(z0, nz)
        rows = Q[:, v0:v0 + nr].contiguous()
        work = torch.empty(max(1, plan.slab_workspace_elems(nr)), device="cuda")

        def both():
            return plan.backproject(Q).clone(), plan.backproject_slab(rows, v0, work, z0, nz).clone()

        want = both()
        widths = autotune.tile_candidates(plan.tile[1], count=5)
        assert len(widths) >= 2
        for w in widths:
            plan.set_tile(w)
            assert plan.tile[0] == w
            got = both()
            for a, b, what in zip(got, want, ("volume", "slab")):
                assert torch.equal(a, b), (w, what, float((a - b).abs().max()))
        assert plan.device_status() == 0


def test_the_tuner_times_the_widths_that_launches_take(fd):
    """choose_tile leaves out widths for which a launch would keep the default
    one (their times say nothing about the width, and the batch's persistent
    kernel would take them), and detectors the staged kernel cannot read."""
    from paper_1708_07515_gb300 import autotune
    with fd.Plan(4.0 * 245, 245, 248, 245, 24, 2, 2) as plan:
        taken = []
        for w in autotune.tile_candidates(plan.tile[1], count=5):
            plan.set_tile(w)
            if fd.fdkod_get_forms(plan.handle)["bp_columns"] == w:
                taken.append(w)
        assert taken and taken != autotune.tile_candidates(plan.tile[1], count=5)
        plan.set_tile(0)
        best, times = autotune.choose_tile(plan, count=5)
        assert sorted(times) == taken and plan.tile[0] == best and best in taken
    with fd.Plan(4.0 * 64, 64, 63, 64, 24, 1, 1) as plan:
        assert autotune.choose_tile(plan) == (plan.tile[1], {})

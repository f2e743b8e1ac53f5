"""Ensembles of members with and without x/y transforms on the tensor cores: the ones without stay in the
grouped launches of those stages, the others make their own.

A grouped launch uses the ensemble's radix schedules, a grid's own launches the grid's; for a padded
length of 192 points the two differ (4 4 4 3 and 8 8 3, and with them the last bits), so such a member
evolves bit for bit as in an ensemble without the others only if it stayed grouped."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2406_01322_gb300 import inputs  # noqa: E402

pytestmark = pytest.mark.gpu

PHYS = dict(re_tau=150.0, we=1.0, ch=0.05, pe=20.0, dt=1e-4)
SMALL, LARGE = dict(nx=128, ny=8, nz=33, **PHYS), dict(nx=64, ny=64, nz=33, **PHYS)   # 2^14, 2^16 modes


@pytest.fixture(scope="module")
def binding():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_01322_gb300 import build
    build.build_library()
    from paper_2406_01322_gb300 import binding as b
    b.lib()
    return b


def evolve(ens, seeds):
    for g, m, s in zip(ens.grids, ens.members, seeds):
        f = inputs.initial_fields(m["nx"], m["ny"], m["nz"], 150.0, 0.05, 1, 0.4, s)
        g.set_fields(*[torch.from_numpy(np.ascontiguousarray(a)) for a in f])
    ens.step(3)
    out = [g.get_state() for g in ens.grids]
    ens.close()
    return out


def ensemble(binding, members):
    e = binding.Ensemble(members)
    e.members = members
    return e


def test_members_without_tensor_core_xy_stay_grouped(binding):
    mixed = evolve(ensemble(binding, [SMALL, LARGE, SMALL]), (1, 2, 3))
    small = evolve(ensemble(binding, [SMALL, SMALL]), (1, 3))
    large = evolve(ensemble(binding, [LARGE]), (2,))
    for a, b in zip(mixed, (small[0], large[0], small[1])):
        assert torch.equal(a, b)


def test_stages_without_grouped_members_keep_their_defaults(binding):
    e = ensemble(binding, [LARGE, dict(LARGE, nx=72)])
    evolve_seeds = (4, 5)
    for g, m, s in zip(e.grids, e.members, evolve_seeds):
        f = inputs.initial_fields(m["nx"], m["ny"], m["nz"], 150.0, 0.05, 1, 0.4, s)
        g.set_fields(*[torch.from_numpy(np.ascontiguousarray(a)) for a in f])
    t = e.autotune(2)
    assert t["tuned"] == 1
    assert t["radix_style"]["x"] == 0 and t["radix_style"]["y"] == 0
    assert t["ctas_per_sm"][3:] == [0, 0, 0]
    e.close()


def test_members_of_few_long_x_lines_are_grouped_there(binding):
    """512 x 8 x 17: a grid of its own has its x line on the tensor cores, a member the grouped FFT (the last
    bits tell them apart); both agree to the float64 bar of the step, 1e-10, and a member evolves the
    same bit for bit whatever is beside it."""
    m = dict(nx=512, ny=8, nz=17, **PHYS)
    alone = evolve(ensemble(binding, [m]), (7,))[0]
    among = evolve(ensemble(binding, [LARGE, m, SMALL]), (8, 7, 9))[1]
    assert torch.equal(alone, among)
    e = ensemble(binding, [m])
    g = binding.Grid(**m)
    assert g.launches_per_step() == 9
    f = [torch.from_numpy(np.ascontiguousarray(a))
         for a in inputs.initial_fields(512, 8, 17, 150.0, 0.05, 1, 0.4, 7)]
    for x in (g, e.grids[0]):
        x.set_fields(*f)
    g.step(3)
    e.step(3)
    assert not torch.equal(g.get_state(), e.grids[0].get_state())
    for a, b in zip(g.get_fields(), e.grids[0].get_fields()):
        assert float((a - b).abs().max()) <= 1e-10 * float(b.abs().max())
    e.close()
    g.close()

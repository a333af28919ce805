"""lpm_set_auto takes lpm_set_launch and lpm_set_sort back: the context then launches what one
that never had those calls launches, with the same results; and a tuned small run may keep the
library's own choice."""
import numpy as np
import pytest

import lpm_inputs as li

pytestmark = pytest.mark.gpu


def _run(sim, steps):
    from paper_0912_3223_gb300 import lpm
    sim.reset().step(steps).reset()              # (a changed interval sends particles home once)
    lpm.lpm_stats(sim.ctx)
    sim.step(steps)
    launches = lpm.lpm_stats(sim.ctx)[0]
    return [launches, *sim.particles(), *(a for s in range(sim.cfg.n_scenarios)
                                          for a in sim.fixed_state(s)[:3])]


@pytest.mark.parametrize("scenarios", [1, 4])
def test_the_choice_by_size_again(scenarios):
    from paper_0912_3223_gb300 import Sim, lpm
    cfg = (li.make_cfg3(n_particles=70000, n_steps=250) if scenarios == 1 else
           li.make_cfg2(n_scenarios=4, n_steps=250, n_min=1000, n_max=5000))
    with Sim(cfg) as sim:
        want = _run(sim, 250)
    with Sim(cfg, launch=(128, 1, 1), sort_every=20) as sim:
        fixed = _run(sim, 250)
        assert fixed[0] != want[0]
        lpm.lpm_set_auto(sim.ctx, launch=False, sort=False)
        assert _run(sim, 250)[0] == fixed[0]
        lpm.lpm_set_auto(sim.ctx)
        got = _run(sim, 250)
        lpm.lpm_set_sort(sim.ctx, 20)            # in the middle of a sorted run
        sim.reset()
        sim.step(130)
        lpm.lpm_set_auto(sim.ctx)
        sim.step(120)
        piece = [sim.particles()[0], sim.fixed_state()[0]]
    assert got[0] == want[0]
    for a, b in zip(got[1:], want[1:]):
        assert np.array_equal(a, b)
    assert np.array_equal(piece[0], want[1]) and np.array_equal(piece[1], want[3])


def test_a_tuned_small_run_may_keep_it(tmp_path, monkeypatch):
    from paper_0912_3223_gb300 import Sim
    from paper_0912_3223_gb300.autotune import autotune_with_sort
    monkeypatch.setenv("LPM_AUTOTUNE_CACHE", str(tmp_path / "tune.json"))
    cfg = li.make_cfg3(n_particles=2160, n_steps=360)
    with Sim(cfg) as sim:
        want = _run(sim, 360)
        shape, every, ms = autotune_with_sort(sim, shapes=[None, (512, 1, 2)],
                                              sort_intervals=(None, 60), reps=1)
        assert set(ms) == {"auto/sortauto", "512x1x2/sortauto", "auto/sort60", "512x1x2/sort60"}
        assert min(ms, key=ms.get) == "auto/sortauto" or (shape, every) != (None, None)
        got = _run(sim, 360)
    for a, b in zip(got[1:], want[1:]):
        assert np.array_equal(a, b)

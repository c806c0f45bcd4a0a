"""The batch's host copy of its lattices' state is read from the device only after steps: calls
between steps, and table uploads after them (a new schedule, tuning, members joining and leaving),
see and keep the current state."""
import numpy as np
import pytest

from paper_1908_09235_gb300 import lbm, workloads

pytestmark = pytest.mark.gpu


def _parts(w):
    eos = lbm.make_eos(lbm.EOS_CS, **dict(w["eos"], T_over_Tc=0.87))
    rl, rv = lbm.lbm_coexistence(eos)
    eos.rho_wall = rv
    return eos, tuple(w["drop"]) + (rl, rv)


def test_state_between_steps_and_across_uploads(gpu_lib):
    ws = workloads.batched_domains(n=3, seed=workloads.SEED, side_lo=40, side_hi=90)
    b = lbm.Batch(lbm.FP32_DEV, lbm.EOS_CS, max_domains=3)
    slots = []
    for w in ws[:2]:
        eos, drop = _parts(w)
        slots.append(b.add(lbm.make_domain(w["nx"], w["ny"], 1.0, "mod_b", circles=[w["cyl"]],
                                           eos=eos, droplet=drop), 100))
    b.step(21)
    assert [b.progress(s) for s in slots] == [(21, 79)] * 2
    b.set_schedule(16, lbm.SCHED_STRIDED)  # uploads the tables at the next step
    b.step(3)
    assert b.poll(3) == [76, 76, -1]
    b.tune(1)
    eos, drop = _parts(ws[2])
    late = b.add(lbm.make_domain(ws[2]["nx"], ws[2]["ny"], 1.0, "mls", circles=[ws[2]["cyl"]],
                                 eos=eos, droplet=drop), 5)
    assert b.poll(3) == [76, 76, 5]
    b.step(17)
    b.remove(late)
    b.step(2)
    assert [b.progress(s) for s in slots] == [(43, 57)] * 2
    for s, w in zip(slots, ws):
        eos, drop = _parts(w)
        lat = lbm.Lattice(w["nx"], w["ny"], 1.0, "mod_b", circles=[w["cyl"]], eos=eos,
                          precision=lbm.FP32_DEV)
        lat.init_droplet(*drop)
        lat.step(43)
        for _ in range(2):  # twice without a step between
            for x, y in zip(b.fields(s), lat.fields()):
                assert np.array_equal(np.nan_to_num(x, nan=-7.0), np.nan_to_num(y, nan=-7.0))
        lat.close()
    b.close()

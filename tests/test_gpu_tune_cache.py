"""Cached layout choices (Plan.tune) where plans of one shape differ in the solves they have."""
import json

import numpy as np
import pytest

from oracle import rexi_coeffs as rc
from paper_1812_03431_gb300 import inputs

pytestmark = pytest.mark.gpu
N, B = 21, 3
ORDER = 1e-13  # the same sums in another order


@pytest.fixture(scope="module")
def rexi():
    from paper_1812_03431_gb300 import rexi
    rexi.load()
    return rexi


def plan_of(rexi, al, be, max_batch):
    return rexi.Plan(N, 36, 72, tau=1800.0, max_batch=max_batch, layout="spectral", alpha=al, beta=be)


def alike(n=45):
    al, be, _ = rc.rexi_coefficients(64, 0.2)
    k = (al.size - n) // 2
    return al[k:k + n], be[k:k + n]


def unlike(n=45):
    """Poles whose couplings differ by more than the fixed-point factors cover."""
    k = np.arange(n)
    return -(2.0 ** (k % 3 * 10.0 - 10.0)) + 1j * k, np.full(n, 1.0 / n) + 0j


def result(plan):
    import torch
    return plan.step(torch.from_numpy(inputs.random_spectral(N, B, 3)).cuda()).cpu().numpy()


def test_plans_with_other_solves_do_not_share_an_entry(rexi, tmp_path):
    cache = str(tmp_path / "tune.json")
    for al, be, max_batch in (alike() + (4,), alike() + (8,), unlike() + (4,)):  # limbs, digits, neither
        ref = rexi.Plan(N, 36, 72, tau=1800.0, max_batch=B, layout="spectral", alpha=al, beta=be, pole_slots=1)
        plan = plan_of(rexi, al, be, max_batch)
        plan.tune(B, cache=cache)
        a, b = result(plan), result(ref)
        assert np.linalg.norm(a - b) < ORDER * np.linalg.norm(b)
        plan.close()
        ref.close()
    assert len(json.load(open(cache))) == 3


def test_an_entry_that_the_plan_refuses_is_a_miss(rexi, tmp_path):
    cache = tmp_path / "tune.json"
    plan = plan_of(rexi, *unlike(), 4)
    plan.tune(B, cache=str(cache))
    (key, kept), = json.loads(cache.read_text()).items()
    assert kept[1] != 5
    cache.write_text(json.dumps({key: [4, 5]}))
    plan.tune(B, cache=str(cache))
    assert json.loads(cache.read_text())[key][1] != 5
    plan.close()


@pytest.mark.parametrize("max_batch", [3, 8])
def test_pole_slots_are_those_of_the_solve_in_use(rexi, max_batch):
    """A slot layout chosen earlier is not reported once the fixed-point solve has been."""
    plan = plan_of(rexi, *alike(), max_batch)
    used = plan.set_pole_slots(max_batch, 4, 0)
    assert plan.info()["pole_slots"] == used > 0
    plan.set_pole_slots(max_batch, 0, 5)
    assert plan.info()["pole_slots"] == 0
    plan.close()

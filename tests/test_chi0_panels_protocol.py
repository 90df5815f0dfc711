"""The barrier protocol of k_pn_gram on the CPU: the model of the tensor-core kernels (test_chi0_protocol) with the roles
of that kernel, persistent over items and with separate drain warps, for items of one to a few stages."""
import os
import re

import pytest

from tests.test_chi0_protocol import _run

SRC = open(os.path.join(os.path.dirname(__file__), "..", "paper_2603_12326_gb300", "csrc", "chi0_panels.cu")).read()


def _constant(name):
    return int(re.search(r"constexpr int %s = (\d+);" % name, SRC).group(1))


@pytest.mark.parametrize("kstages", [1, 2, 3, 5, 8])
@pytest.mark.parametrize("fault", [{}, {"timeouts": True}, {"withhold": True, "timeouts": True}])
def test_persistent_items_with_drain_warps(kstages, fault):
    for seed in range(6):
        errors, aborted = _run(kstages, _constant("PG_NSTAGE"), _constant("PG_PROMOTE"), seed, ngroups=1, ntile=6,
                               drain_warps=8, **fault)
        assert not errors, (kstages, seed, errors[:3])
        assert bool(aborted) <= bool(fault)


def test_register_budgets_fit_the_launch():
    regs, threads = _constant("PG_LAUNCH_REGS"), _constant("PG_THREADS")
    m = re.search(r"PG_REG_CTRL = (\d+), PG_REG_AGEN = (\d+), PG_REG_DRAIN = (\d+)", SRC)
    ctrl, agen, drain = map(int, m.groups())
    assert 128 * ctrl + 256 * agen + 256 * drain <= threads * regs and threads == 128 + 256 + 256

"""The barrier protocol of k_pn_gram with its A warps in groups on alternate stages, on the CPU (the model of
test_chi0_protocol: a group starts every item at its own parity, as the kernel does for items of an even number of stages,
and over one long item for an odd one), for both ring lengths."""
import re

import pytest

from tests.test_chi0_panels_protocol import SRC, _constant
from tests.test_chi0_protocol import _run


@pytest.mark.parametrize("kstages,ntile", [(2, 6), (4, 5), (8, 4), (14, 3), (1, 1), (33, 1)])
@pytest.mark.parametrize("extra", [0, 1])
@pytest.mark.parametrize("fault", [{}, {"timeouts": True}, {"withhold": True, "timeouts": True}])
def test_two_groups_of_a_warps(kstages, ntile, extra, fault):
    warps = _constant("PG_AWARPS")
    assert warps == 4 and re.search(r"mbar_init\(&full_a\[s\], PG_AWARPS\)", SRC)
    for seed in range(6):
        errors, aborted = _run(kstages, _constant("PG_NSTAGE") + extra, _constant("PG_PROMOTE"), seed, ngroups=2,
                               ntile=ntile, drain_warps=8, **fault)
        assert not errors, (kstages, seed, errors[:3])
        assert bool(aborted) <= bool(fault)

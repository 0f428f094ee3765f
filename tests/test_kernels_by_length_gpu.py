"""The tests of the short, mid and team kernels with those kernels: at the sizes an oracle can follow the general
kernels are the faster ones, and tile 0 takes them."""
import types

import pytest
import torch

from tests.test_mid_window_gpu import *        # noqa: F401,F403  (their cases run here with this module's fixture)
from tests.test_short_window_gpu import *      # noqa: F401,F403
from tests.test_team_window_gpu import *       # noqa: F401,F403

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def native():
    from paper_2510_18136_gb300 import build
    build.build()
    from paper_2510_18136_gb300 import native as nat
    assert torch.cuda.is_available()

    class ByLength(nat.Plan):
        def __init__(self, *a, **k):
            super().__init__(*a, **k)
            assert nat.lib.nsfrb_dbg_plan_by_length(self.handle, 1) == nat.OK

    return types.SimpleNamespace(**{**vars(nat), "Plan": ByLength})

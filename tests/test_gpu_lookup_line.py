"""The lookup forms of test_gpu_lookup_forms.py at table sizes on both sides of the
line between them (240 MB of buckets)."""

import pytest

import test_gpu_lookup_forms as forms

pytestmark = pytest.mark.gpu

LINE = (240 << 20) // 256


@pytest.mark.parametrize("nb", [LINE, LINE + 1])
@pytest.mark.parametrize("timers", [False, True])
def test_lookup_forms_agree_around_their_line(nb, timers):
    forms.test_lookup_forms_agree(nb, timers)

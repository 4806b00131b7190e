"""Results that are kept bit for bit (tests/recorded.py says why)."""
import json

import pytest

from tests import recorded

pytestmark = pytest.mark.gpu
with open(recorded.GOLDEN) as f:
    GOLDEN = json.load(f)


@pytest.mark.parametrize("name", sorted(recorded.RECORDS))
def test_recorded_outputs(name):
    assert recorded.RECORDS[name]() == GOLDEN[name]

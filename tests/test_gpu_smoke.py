"""The smoke entry point: a small bucket through the bulk-copy pipeline and one through the gather pipeline, against the oracle."""
import pytest

import __graft_entry__

pytestmark = pytest.mark.gpu


def test_smoke():
    __graft_entry__.smoke()

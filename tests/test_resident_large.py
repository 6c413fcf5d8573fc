"""The resident kernel on bytes at the largest edges whose slabs fit the shared memory of a cluster of eight."""
import pytest

import paper_1508_06268_gb300 as rf
from tests.test_resident import test_resident_bytes_match_oracle as _check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [110, 112, 114, 116])
@pytest.mark.parametrize("kind", [rf.FIELD_BIMODAL, rf.FIELD_EXPLICIT])
def test_largest_edges_match_oracle(L, kind, monkeypatch):
    _check(L, 2, "8,1,4,512,b", kind, monkeypatch)

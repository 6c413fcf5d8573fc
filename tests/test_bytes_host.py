"""Host-side check of the resident kernel on bytes (no GPU): its divisions by reciprocals are exact, with every
argument inside the range that guarantees it, for every block of every L it may take."""
import pytest


@pytest.mark.parametrize("L", range(4, 146, 2))
def test_block_places_are_exact(L):
    import paper_1508_06268_gb300 as rf
    assert rf.selftest_bytes(L) == (0 if L <= 144 else -1)

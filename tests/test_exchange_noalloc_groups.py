"""rfim_exchange_noalloc where its replica groups, slabs and state leave their simplest form: partial
groups of four replicas, both fields, slabs of uneven sizes, and more replicas than the last CTA
keeps in shared memory.  Bounds as in test_zz_no_alloc: integers and bimodal energies equal, float
energies to 1e-9 relative."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1508_06268_gb300 as rf  # noqa: E402
from tests.test_zz_no_alloc import test_noalloc_exchange_matches_allocating_entry_point as _check  # noqa: E402


@pytest.mark.parametrize("L,R,kind,pre,measure_from", [
    (8, 2, rf.FIELD_GAUSSIAN, 0, 0), (16, 2, rf.FIELD_GAUSSIAN, 0, 0), (32, 39, rf.FIELD_GAUSSIAN, 0, 0),
    (32, 41, rf.FIELD_BIMODAL, 2, 0), (64, 5, rf.FIELD_BIMODAL, 0, 0), (64, 7, rf.FIELD_GAUSSIAN, 2, 3),
    (16, 1031, rf.FIELD_GAUSSIAN, 0, 0), (8, 1024, rf.FIELD_BIMODAL, 1, 0),
])
def test_noalloc_replica_groups(L, R, kind, pre, measure_from):
    _check(L, R, kind, pre, measure_from)

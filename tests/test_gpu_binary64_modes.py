"""The binary64 update stores the same bits whether a step is reduced or not, for the instantiations
that the force-series test leaves out (lattices, walls and couplings)."""
import pytest

from test_gpu_force_series import _cuda, test_fused_reduction_pass_updates_bit_identically as _same_bits  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("q,walls,coupling", [(15, 0, 0), (19, 4, 0), (15, 0, 1), (15, 4, 1), (19, 0, 1)])
def test_binary64_update_is_the_same_reduced_or_not(q, walls, coupling):
    _same_bits(q, 3, walls, coupling)

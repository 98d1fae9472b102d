"""prx_get_bonds on both sides of the number of records from which the device
sorts them (1,536 and below: the host), and at the edges of its tiles there."""
import pytest

from test_gpu_bond_order import test_initial_bonds_come_back_sorted as check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [1535, 1536, 1537, 2047, 2048, 3072, 3073, 4096, 4097])
def test_edges(m):
    check(m)

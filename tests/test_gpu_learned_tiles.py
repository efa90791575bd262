"""The learned step where the order in which its warpgroups take tiles changes: tiles
of 32 x 4 cells for some of the CTAs, for every warpgroup of 152 SMs exactly, and
one row of tiles more."""
import pytest

import test_gpu_learned as L

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(32, 8, 152), (64, 40, 38), (64, 40, 39), (32, 4, 151)])
def test_every_cell_whichever_warpgroup_takes_its_tile(dims):
    L.test_learned_step_on_every_cell_and_all_bits_of_the_biases(dims)

"""Host-side checks of the adjoint sweep's binding (no GPU: nothing reaches the library)."""
import numpy as np
import pytest

import paper_1512_03210_gb300 as fse


@pytest.mark.parametrize("gammas", [None, np.ones((4, 2)), np.ones(12), np.ones((4, 4)), np.ones((2, 2, 3)), 1.0])
def test_sweep_wants_a_row_of_dim_frequencies_per_step(gammas):
    """The library reads nsteps rows of dim values from the host array."""
    with pytest.raises(ValueError, match="gammas"):
        fse.fse_adjoint_sweep(None, None, None, None, 0.0, gammas, 3)

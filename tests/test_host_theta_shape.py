"""Parameters that are not a vector are refused, as their entries are no numbers (CPU)."""
import numpy as np
import pytest

import paper_2605_04178_gb300 as pm


@pytest.mark.parametrize("shape", [(3, 6), (18, 1), (1, 18)])
def test_theta_is_a_vector(shape):
    with pytest.raises(TypeError):
        pm.params(np.ones(shape))
    with pytest.raises((TypeError, AssertionError)):
        pm._params_f64(np.ones(shape))

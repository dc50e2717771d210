"""Array arguments of the binding, on CPU: every kind of numpy array that has an
address is taken, silently, at that address."""
import warnings

import numpy as np
import pytest


@pytest.fixture(scope="module")
def R():
    from paper_2408_14070_gb300 import rid
    return rid


def _arrays():
    own = np.arange(6, dtype=np.float32).reshape(2, 3)
    frozen = own.copy()
    frozen.flags.writeable = False
    broadcast, _ = np.broadcast_arrays(np.ones(3, np.float32), np.ones((1, 3), np.float32))
    return dict(own=own, view=own[1:], frozen=frozen, broadcast=broadcast, empty=np.zeros((0, 3), np.float32),
                scalar=np.ones((), np.float32), masked=np.ma.zeros((2, 3), dtype=np.float32))


@pytest.mark.parametrize("kind", list(_arrays()))
def test_inputs_are_taken_at_their_address_without_a_warning(R, kind):
    a = _arrays()[kind]
    with warnings.catch_warnings():
        warnings.simplefilter("error")
        p = R._Args().address(a, np.float32, a.shape)
    assert p == a.ctypes.data


def test_read_only_outputs_and_wrong_layouts_are_refused(R):
    a = np.zeros((2, 3), np.float32)
    a.flags.writeable = False
    with pytest.raises(ValueError, match="read-only"):
        R._Args().address(a, np.float32, (2, 3), True)
    with pytest.raises(TypeError):
        R._Args().address(np.zeros((3, 2), np.float32).T, np.float32, (2, 3))
    with pytest.raises(TypeError):
        R._Args().address(np.zeros((2, 3), ">f4"), np.float32, (2, 3))
    with pytest.raises(ValueError, match="elements"):
        R._Args().address(np.zeros((2, 3), np.float32), np.float32, (3, 3))

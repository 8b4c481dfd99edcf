"""Number lists taken by the binding: what it refuses and what it converts (no GPU)."""
import numpy as np
import pytest

import paper_1505_00344_gb300 as ff


def values(v):
    a, address = ff._dbl(v)
    return [float(x) for x in a], address


def test_lists_of_numbers_are_taken_as_numpy_takes_them():
    for v in ([1, 2.5, True], (np.float32(0.1), 3), [[1, 2], [3, 4]], ["1.5"], [None], [], 3.0, range(3), [np.float64(2)],
              [np.array(1.0), np.array([2.0])[0]], [2 ** 70, -0.0, float("inf")]):
        want = np.asarray(v, dtype=np.float64).reshape(-1)
        np.testing.assert_array_equal(values(v)[0], want)


def test_tensors_that_carry_gradients_are_refused_in_lists():
    """A parameter list of tensors that require gradients is an error, as in numpy: its values would
    enter the integration with their gradients silently dropped."""
    torch = pytest.importorskip("torch")
    with pytest.raises(RuntimeError):
        values([torch.tensor(10.0, requires_grad=True), 28.0, 8 / 3])
    assert values([torch.tensor(10.0), 28.0])[0] == [10.0, 28.0]

"""What the layer API's host code enqueues, checks and refuses, on a CUDA runtime that only writes down what it is asked."""
import pytest

import fake_runtime


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return fake_runtime.load(fake_runtime.build_library(str(tmp_path_factory.mktemp("host"))))


@pytest.fixture(autouse=True)
def clean(lib):
    lib.fake_reset()
    yield
    lib.fake_reset()


BAD_ARG, CUDA = -1, -16


def test_one_layer_under_two_indices_never_shares_a_launch_with_itself(lib):
    """Two actions of a kind on one layer in one launch would commit its scales twice, and two indices' weight gradients
    would be added up in one sum, beyond the products that a sum has room for."""
    s = fake_runtime.Stage(lib, [(256, 256)], M=16, slots=16, window=8)
    acts = [(k, m // 8, m) for k in ("F", "dI", "dW") for m in (0, 8, 1, 9, 2, 10, 3, 11, 4, 12, 5, 13, 6, 14, 7, 15)]
    assert s.step(acts, layers=[0, 0]) == BAD_ARG and "same layer" in s.error()
    assert b"launch" not in lib.fake_log()
    s.close()
    s = fake_runtime.Stage(lib, [(256, 256)], M=2, slots=2, window=1)  # action by action the list is a legal one
    assert s.step([("F", 0, 0), ("F", 1, 1), ("dI", 0, 0), ("dI", 1, 1), ("dW", 0, 0), ("dW", 1, 1)], layers=[0, 0]) == 0
    s.close()

"""The square roots of the FP64 path against CUDA's correctly rounded ones.  Before its last rounding a
root is off by the product of two relative errors below 2^-38, a 2^-20th of a unit in the last place at most,
so about one root in 2^20 may round the other way; 0.05% did without the step for the reciprocal."""
import pytest

pytestmark = pytest.mark.gpu


def test_roots_are_correctly_rounded():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1305_4650_gb300 import build, bf
    build.build()
    n = 1 << 24
    assert bf.selfcheck_sqrt(n) <= 4 * (n >> 20)

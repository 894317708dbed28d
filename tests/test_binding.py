"""The packed descriptors that the calls hand over (no GPU needed): the same bytes
as the ctypes structures, and the same errors for fields that are no integers."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2609_21849_gb300 import qlin

Z = torch.zeros(64, dtype=torch.uint8)


def _nvfp4(rows, K):
    return qlin.NVFP4Tensor(Z, Z, Z, rows, K)


def _fp8(rows, K, per_channel):
    return qlin.FP8Tensor(Z, Z, rows, K, per_channel)


@pytest.mark.parametrize("rows", [4, True, -1, np.int64(4), torch.tensor(4), 2**63, 2**70])
def test_packed_rows_are_the_structures_bytes(rows):
    for t in (_nvfp4(rows, 64), _fp8(rows, 64, 1)):
        assert t.packed() == bytes(t.desc())


@pytest.mark.parametrize("per_channel", [0, 1, True, 2**31, 2**40])
def test_packed_per_channel_is_the_structures_bytes(per_channel):
    t = _fp8(4, 64, per_channel)
    assert t.packed() == bytes(t.desc())


@pytest.mark.parametrize("bad", [4.0, "4", None])
def test_fields_that_are_no_integers(bad):
    for t in (_nvfp4(bad, 64), _nvfp4(4, bad), _fp8(bad, 64, 0), _fp8(4, bad, 0), _fp8(4, 64, bad)):
        with pytest.raises(TypeError):
            t.packed()

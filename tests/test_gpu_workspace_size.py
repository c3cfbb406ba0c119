"""Workspaces of tiled plans ask for no more than they once did, so that a budget that held a probe still holds it.

The sizes are those of plans on 152 SMs whose eigen-steps logged their rotations and whose passes summed their partial
Grams in groups of 16.
"""
import ctypes

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# (complex, precision, frames, pixels): bytes
SIZES = {
    (0, 0, 20, 262144): 21270016, (0, 0, 33, 4096): 1109504, (0, 0, 65, 20000): 8997888, (0, 0, 96, 87880): 41938176,
    (0, 0, 100, 20000): 16887296, (0, 1, 100, 87880): 44301312, (0, 0, 128, 87880): 59531264, (0, 0, 132, 87880): 61858816,
    (0, 0, 160, 4096): 22445312, (0, 0, 192, 262144): 233983488, (0, 0, 224, 500): 13969920, (0, 0, 224, 20000): 62352640,
    (1, 0, 10, 4096): 547072, (1, 1, 50, 20000): 17149184, (1, 0, 50, 87880): 44039424, (1, 0, 90, 20000): 43108608,
    (1, 0, 112, 262144): 279313664,
}


@pytest.mark.parametrize("key", sorted(SIZES))
def test_workspace_is_no_larger(key):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the sizes are those of 152 SMs")
    from paper_2506_10257_gb300 import rpca
    cplx, precision, T, m = key
    p = rpca.default_params(m, T, dtype=cplx, precision=precision)
    n = ctypes.c_size_t()
    assert rpca.load().rpca_workspace_size(ctypes.byref(p), ctypes.byref(n)) == rpca.OK
    assert n.value <= SIZES[key]

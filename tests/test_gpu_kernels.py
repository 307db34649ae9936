"""Kernels of the step against the FP64 oracle at the sizes where their tiling can go wrong.

Bounds as in test_gpu_parity.py, per field max |got - want| / max |want|: explicit terms of the
FP64 path 1e-12, its Jacobian action 1e-11, explicit terms of the mixed path 2e-5 (FP32 transforms).
"""
import numpy as np
import pytest

import seeded_inputs as si
from oracle.shell import Shell

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as _t
    if not _t.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    return _t


def _errors(s, got, want):
    g, w = s.to_complex(got), s.to_complex(want)
    return [float(np.abs(g[i] - w[i]).max() / np.abs(w[i]).max()) for i in range(3)]


# Longitudes per sector by K = L / M_s: 4 (one wavenumber), 8, 27 (odd), 54 (not a multiple of
# four), 81 (odd), 96 (three quads per thread); latitudes 6 to 48.
@pytest.mark.parametrize("L,Ms", [(3, 2), (4, 2), (8, 1), (17, 1), (25, 1), (31, 1)])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_products_longitude_counts(torch, L, Ms, precision):
    from paper_2508_16635_gb300 import RotatingShell
    Nr, Ek, Ra = 9, 1e-3, 80.0
    s = Shell(L, Ms, Nr, Ek, Ra)
    gpu = RotatingShell(L, Ms, Nr, Ek, Ra, precision=precision)
    x = s.conductive_state() + si.perturbation(L, Ms, Nr, seed=31, amp=3e-2)
    got = gpu.explicit_terms(torch.tensor(x, device="cuda")).cpu().numpy()
    want = s.to_real(s.explicit_terms(s.to_complex(x)))
    assert max(_errors(s, got, want)) < (1e-12 if precision == "fp64" else 2e-5)
    u = si.random_vector(L, Ms, Nr, seed=32)
    J = s.real_index("T", Ms, Ms, 1, 1)
    got = gpu.apply_jacobian(torch.tensor(x, device="cuda"), 0.4, J, torch.tensor(u, device="cuda"),
                             200.0).cpu().numpy()
    assert max(_errors(s, got, s.jvp(x, 0.4, J, u, 200.0))) < (1e-11 if precision == "fp64" else 1e-5)
    gpu.close()

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


# FP64 Legendre transforms on digit slices: degrees per parity class 16 and 17 (one and two 16-term
# steps), m = L (one degree, an empty odd class), radii that leave part of a 3- and 4-radius tile,
# more than 128 north latitudes (two row tiles).
@pytest.mark.parametrize("L,Ms,Nr", [(31, 31, 8), (32, 16, 9), (33, 11, 7), (47, 24, 6), (191, 95, 8)])
def test_sliced_transforms(torch, L, Ms, Nr):
    from paper_2508_16635_gb300 import RotatingShell
    s = Shell(L, Ms, Nr, 1e-3, 80.0)
    gpu = RotatingShell(L, Ms, Nr, 1e-3, 80.0)
    x = s.conductive_state() + si.perturbation(L, Ms, Nr, seed=33, amp=3e-2, l_decay=30.0)
    got = gpu.explicit_terms(torch.tensor(x, device="cuda")).cpu().numpy()
    want = s.to_real(s.explicit_terms(s.to_complex(x)))
    assert max(_errors(s, got, want)) < 1e-12
    # columns of zeros (one field only) and of very different sizes
    y = x.reshape(3, s.P, Nr, 2).copy()
    y[0] = 0.0
    y[1] *= 1e-150
    got = gpu.explicit_terms(torch.tensor(y.reshape(-1), device="cuda")).cpu().numpy()
    want = s.to_real(s.explicit_terms(s.to_complex(y.reshape(-1))))
    assert max(_errors(s, got, want)[1:]) < 1e-12
    gpu.close()


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_sliced_transforms_pass_on_what_is_not_finite(torch, bad):
    from paper_2508_16635_gb300 import RotatingShell
    L, Ms, Nr = 15, 4, 10
    gpu = RotatingShell(L, Ms, Nr, 1e-3, 80.0)
    U = gpu.conductive_state()
    U[gpu.phase_slot(Ms, 2) - 1] = bad          # Re T at l = m = M_s
    U[gpu.n // 3 + 2 * Nr] = 1e-2               # some velocity
    N = gpu.explicit_terms(U).view(3, gpu.P, Nr, 2)
    assert not torch.isfinite(N[2, L + 1]).any()
    gpu.close()


# Radial stages by reflection: odd and even N_r and N_d (N_r = 6 the smallest, 128 the largest), one
# and several pairs per block, the last block part full.  The bounds of the explicit terms and of a
# step and Jacobian action; the second-order step (its boundary rows) 2e-11 as in test_step2_parity.
@pytest.mark.parametrize("L,Ms,Nr", [(5, 2, 6), (6, 3, 7), (9, 4, 13), (7, 3, 33), (6, 2, 66), (3, 1, 97), (2, 1, 128)])
def test_radial_stages_by_reflection(torch, L, Ms, Nr):
    from paper_2508_16635_gb300 import RotatingShell
    s = Shell(L, Ms, Nr, 1e-3, 80.0)
    gpu = RotatingShell(L, Ms, Nr, 1e-3, 80.0)
    x = s.conductive_state() + si.perturbation(L, Ms, Nr, seed=35, amp=3e-2)
    dev = lambda a: torch.tensor(a, device="cuda")  # noqa: E731
    got = gpu.explicit_terms(dev(x)).cpu().numpy()
    assert max(_errors(s, got, s.to_real(s.explicit_terms(s.to_complex(x))))) < 1e-12
    got = gpu.step(dev(x), 0.4, 1e-3).cpu().numpy()
    assert max(_errors(s, got, s.step(x, 0.4, 1e-3))) < 1e-11
    got = gpu.step2(dev(x), 1e-3).cpu().numpy()
    assert max(_errors(s, got, s.step2(x, 1e-3))) < 2e-11
    u = si.random_vector(L, Ms, Nr, seed=36)
    J = s.real_index("T", Ms, Ms, 1, 1)
    got = gpu.apply_jacobian(dev(x), 0.4, J, dev(u), 1e-3).cpu().numpy()
    assert max(_errors(s, got, s.jvp(x, 0.4, J, u, 1e-3))) < 1e-11
    gpu.close()


# Passes of the odd-even reduced chain solve: rows that fill part of a warp, one, two passes of
# rows, columns that end inside a chunk, odd N_r (a middle row of its own), a chain of one and of two
# blocks (no even or odd neighbour), and 612 CTAs (between four and five per SM of 152).  Bounds as
# test_implicit_solve_backward_error_* of test_gpu_parity.py.
@pytest.mark.parametrize("L,Ms,Nr", [(4, 4, 6), (9, 3, 17), (12, 5, 33), (7, 7, 64), (8, 8, 65),
                                     (5, 4, 128), (34, 1, 8)])
@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_reduced_chain_passes(torch, L, Ms, Nr, precision):
    from paper_2508_16635_gb300 import RotatingShell
    from tests.test_gpu_parity import U48, U64, _random_rhs, _solve_errors
    s = Shell(L, Ms, Nr, 1e-3, 80.0)
    gpu = RotatingShell(L, Ms, Nr, 1e-3, 80.0, precision=precision)
    b = _random_rhs(s, 41)
    x = gpu.implicit_solve(torch.tensor(s.to_real(b), device="cuda"), 2e-3).cpu().numpy()
    eta, fwd, fwd_T = _solve_errors(s, 2e-3, b, s.to_complex(x))
    assert eta < 64 * (U48 if precision == "mixed" else U64)
    assert fwd < (32 * 1e-10 if precision == "mixed" else 1e-11)
    assert fwd_T < 1e-12
    gpu.close()


# Residual of the refined FP64 solve: rows in pairs (odd N_r: a middle row alone), row pairs that fill
# part of a warp, pairs past the last block.  A second refinement leaves the solution where the first
# puts it (within the bounds of the FP64 solve in test_gpu_parity.py): a wrong residual moves it by O(1).
@pytest.mark.parametrize("L,Ms,Nr", [(4, 4, 6), (9, 3, 17), (13, 1, 33), (7, 7, 64), (8, 8, 65), (5, 4, 128)])
def test_chain_residual(torch, L, Ms, Nr):
    from paper_2508_16635_gb300 import RotatingShell
    from tests.test_gpu_parity import U64, _random_rhs, _solve_errors
    s = Shell(L, Ms, Nr, 1e-4, 80.0)
    gpu = RotatingShell(L, Ms, Nr, 1e-4, 80.0)
    b = _random_rhs(s, 43)
    B = torch.tensor(s.to_real(b), device="cuda")
    t0 = gpu.tuning()
    for refine in (1, 2):
        gpu.set_tuning(dict(t0, refine=refine))
        eta, fwd, fwd_T = _solve_errors(s, 2e-3, b, s.to_complex(gpu.implicit_solve(B, 2e-3).cpu().numpy()))
        assert eta < 64 * U64
        assert fwd < 1e-11
        assert fwd_T < 1e-12
    gpu.close()


# Kernels that start while the one ahead ends: steps in a row, with nothing between the launches, give the
# bits of traced ones (an event before and after every launch, the temperature solve in line).
@pytest.mark.parametrize("L,Ms,Nr,n", [(7, 4, 10, 40), (31, 4, 24, 10), (52, 8, 60, 4)])
@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_launches_in_a_row_and_one_by_one(torch, L, Ms, Nr, n, precision):
    from paper_2508_16635_gb300 import RotatingShell
    gpu = RotatingShell(L, Ms, Nr, 1e-3, 80.0, precision=precision)
    U0 = gpu.conductive_state() + torch.tensor(si.perturbation(L, Ms, Nr, seed=47, amp=3e-2), device="cuda")
    out = []
    for traced in (False, True):
        U = U0.clone()
        gpu.profile(traced)
        for _ in range(n):
            gpu.step(U, 1e-3)
        torch.cuda.synchronize()
        gpu.profile(False)
        out.append(U)
    assert torch.equal(out[0], out[1])
    gpu.close()


# The FP64 transforms hold every input to its own 53 bits, whatever else stands in its row or column.
# An action is linear, so scaled by 2^-1035 (every entry subnormal, 39 bits left of an entry of 1) it
# gives the scaled result.  Rounding to multiples of 2^-1074 at each stage is 2^-39 of 1; fields and
# intermediates down to 2^-20 of 1 keep 2^-19: bound 2^-19 per field.  A transform that reads
# subnormals as zero loses the products, which are most of the action of this state.
@pytest.mark.parametrize("L,Ms,Nr", [(15, 4, 10), (47, 12, 13)])
def test_action_scaled_into_subnormals(torch, L, Ms, Nr):
    from paper_2508_16635_gb300 import RotatingShell
    s = Shell(L, Ms, Nr, 1e-1, 80.0)
    gpu = RotatingShell(L, Ms, Nr, 1e-1, 80.0)
    x = torch.tensor(s.conductive_state() + si.perturbation(L, Ms, Nr, seed=49, amp=10.0), device="cuda")
    u = torch.tensor(si.random_vector(L, Ms, Nr, seed=50), device="cuda")
    want = gpu.apply_jacobian(x, 0.4, -1, u, 200.0).cpu().numpy()
    linear = gpu.apply_jacobian(torch.zeros_like(x), 0.4, -1, u, 200.0).cpu().numpy()
    us = torch.tensor(np.ldexp(u.cpu().numpy(), -1035), device="cuda")
    got = gpu.apply_jacobian(x, 0.4, -1, us, 200.0).cpu().numpy()
    assert min(_errors(s, linear, want)) > 1e-2          # the products matter in every field
    assert max(_errors(s, np.ldexp(got, 1035), want)) < 2.0 ** -19
    gpu.close()


def _leave_free(torch, nbytes):
    """Device memory held so that about nbytes stay free (1 MB tensors, two to a block of the allocator)."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    held = [torch.empty(torch.cuda.mem_get_info()[0] - nbytes - (64 << 20), dtype=torch.uint8, device="cuda")]
    while torch.cuda.mem_get_info()[0] >= nbytes + (2 << 20):
        try:
            held.append(torch.empty(1 << 20, dtype=torch.uint8, device="cuda"))
        except torch.cuda.OutOfMemoryError:
            break
    return held


# No room for the reduced factorisation (441 MB of scratch at this size): the FP64 solve runs on the
# unreduced chains (294 MB of factors) and says nothing of the failed try.  Both solutions are refined,
# each within 1e-11 of the oracle's at the sizes of test_chain_residual.
def test_fp64_solve_without_room_for_the_reduced_factors(torch):
    from paper_2508_16635_gb300 import RotatingShell
    L, Ms, Nr = 127, 12, 64
    s = Shell(L, Ms, Nr, 1e-4, 80.0)
    roomy, tight = (RotatingShell(L, Ms, Nr, 1e-4, 80.0) for _ in range(2))
    b = torch.tensor(si.random_vector(L, Ms, Nr, seed=51), device="cuda")
    want = roomy.implicit_solve(b, 2e-3).cpu().numpy()
    got = torch.empty_like(b)
    held = _leave_free(torch, 380 << 20)
    tight.profile(True)
    tight.implicit_solve(b, 2e-3, out=got)
    del held
    torch.cuda.empty_cache()
    launches = {k: v["launches"] for k, v in tight.profile_report().items()}
    tight.profile(False)
    assert launches["chain_reduced"] == 0 and launches["chain_sweep"] == 4, launches
    assert tight.lib.rsc_last_error(tight._ctx) == b""
    assert max(_errors(s, got.cpu().numpy(), want)) < 2e-11
    assert torch.equal(tight.implicit_solve(b, 2e-3), got)      # the slot keeps its choice
    roomy.close()
    tight.close()


# No room for a context's own tables of the reduced passes (3 MB) while the slot it shares holds the
# reduced factors: an error while there is no room for the unreduced factors either, then a solve on
# those; the other context goes on with the reduced ones.
def test_shared_factors_without_room_for_the_tables(torch):
    from paper_2508_16635_gb300 import Batch
    from paper_2508_16635_gb300.rsc import RscError
    L, Ms, Nr = 127, 12, 64
    s = Shell(L, Ms, Nr, 1e-4, 80.0)
    batch = Batch([dict(L=L, Ms=Ms, Nr=Nr, Ek=1e-4, Ra=ra) for ra in (80.0, 90.0)])
    a, c = batch.shells
    b = torch.tensor(si.random_vector(L, Ms, Nr, seed=51), device="cuda")
    want, got = torch.empty_like(b), torch.empty_like(b)
    torch.cuda.synchronize()
    a.implicit_solve(b, 2e-3, out=want)
    torch.cuda.synchronize()
    held = _leave_free(torch, 0)
    for _ in range(2):
        with pytest.raises(RscError) as e:
            c.implicit_solve(b, 2e-3, out=got)
        assert e.value.status == 2                               # RSC_ENOMEM
    del held
    torch.cuda.empty_cache()
    c.implicit_solve(b, 2e-3, out=got)
    torch.cuda.synchronize()
    assert max(_errors(s, got.cpu().numpy(), want.cpu().numpy())) < 2e-11
    again = torch.empty_like(b)
    torch.cuda.synchronize()
    a.profile(True)
    a.implicit_solve(b, 2e-3, out=again)
    launches = a.profile_report()["chain_reduced"]["launches"]
    a.profile(False)
    torch.cuda.synchronize()
    assert launches == 6 and torch.equal(again, want)
    batch.close()


# Only the factors that the solves of a context read are built, on the host (N_r > 96, factor_gpu = 0) as
# on the device.  A set is the 2 P blocks of N_r x N_r complex numbers, FP64 or double-float: reduced
# chains D^-1 of half the blocks and G, H, W of the other half (2 sets per precision), unreduced ones
# 3.  Half a set (20 MB) is left to the tables and to kernels loaded on first use.
@pytest.mark.parametrize("Nr,precision,tuning,sets", [
    (97, "fp64", {}, 2), (96, "fp64", {"factor_gpu": 0}, 2), (96, "fp64", {}, 2),
    (97, "mixed", {}, 4), (96, "mixed", {}, 4), (96, "mixed", {"chain_cr": 0}, 6)])
def test_factors_that_nothing_reads_are_not_built(torch, Nr, precision, tuning, sets):
    from paper_2508_16635_gb300 import RotatingShell
    L, Ms = 31, 4
    gpu = RotatingShell(L, Ms, Nr, 1e-3, 80.0, precision=precision)
    gpu.set_tuning(dict(gpu.tuning(), **tuning))
    U = gpu.conductive_state()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    gpu.step(U, dt=1e-3)
    torch.cuda.synchronize()
    one = 2 * gpu.P * Nr * Nr * 16
    assert free - torch.cuda.mem_get_info()[0] < (sets + 0.5) * one
    b = torch.tensor(si.random_vector(L, Ms, Nr, seed=53), device="cuda")
    x = gpu.implicit_solve(b, 1e-3)
    G = gpu.factor_block(1e-3, "G", 0)          # the unreduced chains', built now
    assert np.isfinite(G).all() and np.abs(G).max() > 0
    assert torch.equal(gpu.implicit_solve(b, 1e-3), x)
    gpu.close()


# The autotuner times the block shape of the right-hand side where it has one (explicit Coriolis): eight
# pairs per block, the first choice at this size, take 1.6 times as long as one, two or four.
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_autotune_of_the_explicit_right_hand_side(torch, precision):
    from paper_2508_16635_gb300 import RotatingShell
    gpu = RotatingShell(31, 4, 24, 1e-3, 80.0, precision=precision, coriolis="explicit")
    gpu.set_tuning(dict(gpu.tuning(), rhs_pairs=[8, 8]))
    assert 8 not in list(gpu.autotune()["rhs_pairs"])
    gpu.close()


# Many wavenumbers: 48 and 64 (the shapes of a tuning go back in as they came out, in a batch too), 72, the
# most that the FP64 products hold; 74 is refused in words.  Bounds as test_products_longitude_counts.
@pytest.mark.parametrize("K,precision", [(47, "fp64"), (63, "fp64"), (63, "mixed"), (71, "fp64")])
def test_many_wavenumbers(torch, K, precision):
    from paper_2508_16635_gb300 import Batch, RotatingShell
    s = Shell(K, 1, 6, 1e-3, 80.0)
    gpu = RotatingShell(K, 1, 6, 1e-3, 80.0, precision=precision)
    gpu.set_tuning(gpu.tuning())
    x = s.conductive_state() + si.perturbation(K, 1, 6, seed=55, amp=3e-2)
    got = gpu.explicit_terms(torch.tensor(x, device="cuda")).cpu().numpy()
    want = s.to_real(s.explicit_terms(s.to_complex(x)))
    assert max(_errors(s, got, want)) < (1e-12 if precision == "fp64" else 2e-5)
    gpu.close()
    if K == 47:
        batch = Batch([dict(L=K, Ms=1, Nr=6, Ek=1e-3, Ra=ra) for ra in (80.0, 90.0)])
        batch.autotune()
        batch.close()


def test_too_many_wavenumbers_for_the_products(torch):
    from paper_2508_16635_gb300 import RotatingShell
    from paper_2508_16635_gb300.rsc import RscError
    gpu = RotatingShell(73, 1, 6, 1e-3, 80.0)
    U = gpu.conductive_state()
    with pytest.raises(RscError, match="too many wavenumbers"):
        gpu.explicit_terms(U)
    b = torch.tensor(si.random_vector(73, 1, 6, seed=57), device="cuda")
    assert torch.isfinite(gpu.implicit_solve(b, 1e-3)).all()      # what needs no products runs
    gpu.close()


def test_factor_time_is_that_of_the_last_factorisation(torch):
    """Each dt's own parts: the unreduced chains added to one dt do not count for the other."""
    import time
    from paper_2508_16635_gb300 import RotatingShell
    gpu = RotatingShell(31, 4, 64, 1e-3, 80.0)
    gpu.set_tuning(dict(gpu.tuning(), factor_gpu=0))
    b = torch.tensor(si.random_vector(31, 4, 64, seed=59), device="cuda")
    t = {}
    for dt in (1e-3, 2e-3):
        gpu.implicit_solve(b, dt)
        t[dt] = gpu.factor_time()[0]
    for dt in (1e-3, 2e-3):
        t0 = time.perf_counter()
        gpu.factor_block(dt, "G", 0)
        wall = time.perf_counter() - t0
        assert t[dt] < gpu.factor_time()[0] <= t[dt] + wall
    gpu.close()


# The build of the passes with fewer registers runs where it alone puts all CTAs on the device at once: 630
# CTAs of 256 threads (four or five per SM of 152).
@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_reduced_chain_passes_in_one_wave(torch, precision):
    test_reduced_chain_passes(torch, 34, 1, 64, precision)


# Without refinement the FP64 solve on reduced chains holds the bounds of the double-float one, which is not
# refined either and has the same passes in fewer bits (test_reduced_chain_passes).
@pytest.mark.parametrize("L,Ms,Nr", [(9, 3, 17), (12, 5, 33), (7, 7, 64)])
def test_reduced_chain_passes_unrefined(torch, L, Ms, Nr):
    from paper_2508_16635_gb300 import RotatingShell
    from tests.test_gpu_parity import U48, _random_rhs, _solve_errors
    s = Shell(L, Ms, Nr, 1e-3, 80.0)
    gpu = RotatingShell(L, Ms, Nr, 1e-3, 80.0)
    gpu.set_tuning(dict(gpu.tuning(), refine=0))
    b = _random_rhs(s, 41)
    x = gpu.implicit_solve(torch.tensor(s.to_real(b), device="cuda"), 2e-3).cpu().numpy()
    eta, fwd, fwd_T = _solve_errors(s, 2e-3, b, s.to_complex(x))
    assert eta < 64 * U48
    assert fwd < 32 * 1e-10
    assert fwd_T < 1e-12
    gpu.close()


# The unreduced factors that the autotuner tries are given back: 4 sets stay on a mixed context that it
# leaves on the reduced chains (sets as above), 6 more if the unreduced ones win.
def test_autotune_gives_back_the_factors_it_tried(torch):
    from paper_2508_16635_gb300 import RotatingShell
    L, Ms, Nr = 31, 4, 96
    gpu = RotatingShell(L, Ms, Nr, 1e-3, 80.0, precision="mixed")
    U = gpu.conductive_state()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    t = gpu.autotune()
    gpu.step(U, dt=200.0)
    torch.cuda.synchronize()
    one = 2 * gpu.P * Nr * Nr * 16
    assert free - torch.cuda.mem_get_info()[0] < ((4 if t["chain_cr"] else 10) + 0.5) * one
    gpu.close()

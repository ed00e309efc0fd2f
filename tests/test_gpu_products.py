"""The products behind the forms, on both sides of each size rule that picks them."""
import numpy as np
import pytest

from oracle import tdb_oracle as O
from paper_1912_03174_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    import __graft_entry__ as g
    g.build()
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1912_03174_gb300 import binding
    return binding


# N = 4 (less than one 8 x 8 tile), 36, 188 (largest DFMA size), 192 (smallest sliced size: whole
# tiles), 260 (ragged tiles, K not a multiple of the 128-deep exact chunk)
@pytest.mark.parametrize("n_atoms,seed", [(1, 3), (9, 3), (47, 8), (48, 8), (65, 8)])
def test_fp64_form_matches_the_oracle_on_both_sides_of_the_slice_rule(B, n_atoms, seed):
    # FP64 products either way: the form differs from the oracle in summation order only, so the
    # bounds are those of the FP64 parity tests (1e-10)
    sysm = I.small_flake(n_atoms, seed=seed)
    run = I.Run(dt=0.2, n_steps=0, scc=True, kick=1e-2, kT=I.SCC_KT)
    n = 100
    with B.Propagator(sysm, run, "fp64") as p:
        p.setup()
        rho0 = B.tdb_get_rho(p.ctx)
        p.step(n)
        hist = B.tdb_dipole_history(p.ctx, n)
        obs = p.observables()
        rho = B.tdb_get_rho(p.ctx)
    ref, _, _, _ = O.setup(sysm, run)
    tr = O.propagate(sysm, run, ref, n)
    assert np.max(np.abs(rho0 - ref)) < 1e-10
    assert np.max(np.abs(np.vstack([hist, obs["dipole"][None]]) - tr.dipole)) < 1e-10
    assert np.max(np.abs(rho - tr.rho)) < 1e-10
    assert obs["herm_err"] == 0.0


def _exact(A, Bm):
    return (A.astype(np.longdouble) @ Bm.astype(np.longdouble)).astype(np.float64)


# 1: one element; 129 x 65 x 1025: one row, column and K element past the tiles; 4096: the
# largest K; "spread" gives a row's elements 60 binades (digits far below the row maximum)
@pytest.mark.parametrize("M,N,K,spread", [(1, 1, 1, 0), (129, 65, 1025, 0), (128, 64, 512, 60),
                                          (5, 7, 4096, 0), (33, 40, 31, 60)])
def test_slice_gemm_keeps_its_error_bound(B, M, N, K, spread):
    rng = np.random.default_rng(M + N + K)
    A = rng.normal(size=(M, K)) * 2.0 ** rng.integers(-spread, 1, (M, K))
    Bm = rng.normal(size=(K, N)) * 2.0 ** rng.integers(-spread, 1, (K, N))
    C, _ = B.tdb_slice_gemm(A, Bm)
    bound = 7 * 2.0 ** -42 * K * np.abs(A).max(1)[:, None] * np.abs(Bm).max(0)[None]
    assert np.all(np.abs(C - _exact(A, Bm)) <= bound)


def test_slice_gemm_of_non_finite_rows_is_nan_there_and_only_there(B):
    rng = np.random.default_rng(5)
    A, Bm = rng.normal(size=(130, 70)), rng.normal(size=(70, 66))
    ref, _ = B.tdb_slice_gemm(A, Bm)
    A[129, 3], A[7, 0], Bm[5, 65] = np.inf, np.nan, -np.inf
    C, _ = B.tdb_slice_gemm(A, Bm)
    bad = np.zeros(C.shape, bool)
    bad[[7, 129]] = True
    bad[:, 65] = True
    assert np.all(np.isnan(C[bad]))
    assert np.array_equal(C[~bad], ref[~bad])
    assert np.all(B.tdb_slice_gemm(np.zeros((3, 5)), np.zeros((5, 2)))[0] == 0.0)

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


# N = 4, 64 (one whole tile), 68 (one tile and a ragged one), 196
@pytest.mark.parametrize("n_atoms", [1, 16, 17, 49])
def test_fp32_form_matches_the_oracle_at_tile_edges(B, n_atoms):
    # FP32 products on rho - rho_gs: the 1e-6 bounds of the reduced-form parity tests
    sysm = I.small_flake(n_atoms, seed=8)
    run = I.Run(dt=0.2, n_steps=0, scc=True, kick=1e-3, kT=I.SCC_KT)
    n = 100
    with B.Propagator(sysm, run, "fp32") as p:
        p.setup()
        p.step(n)
        hist = B.tdb_dipole_history(p.ctx, n)
        rho = B.tdb_get_rho(p.ctx)
    ref, _, _, _ = O.setup(sysm, run)
    tr = O.propagate(sysm, run, ref, n)
    assert np.max(np.abs(hist - tr.dipole[:n])) < 1e-6
    assert np.max(np.abs(rho - tr.rho)) < 1e-6


# N = 532 (32 x 32 tiles for X: 64 x 32 ones would leave a nearly empty round), 772 (the smallest
# aligned size past one 64 x 64 tile per SM); the bounds of the test above
@pytest.mark.parametrize("n_atoms", [133, 193])
def test_fp32_form_matches_the_oracle_past_its_tile_rules(B, n_atoms):
    sysm = I.small_flake(n_atoms, seed=8)
    run = I.Run(dt=0.2, n_steps=0, scc=True, kick=1e-3, kT=I.SCC_KT)
    n = 10
    with B.Propagator(sysm, run, "fp32") as p:
        p.setup()
        p.step(n)
        hist = B.tdb_dipole_history(p.ctx, n)
        rho = B.tdb_get_rho(p.ctx)
    ref, _, _, _ = O.setup(sysm, run)
    tr = O.propagate(sysm, run, ref, n)
    assert np.max(np.abs(hist - tr.dipole[:n])) < 1e-6
    assert np.max(np.abs(rho - tr.rho)) < 1e-6


@pytest.mark.parametrize("dt_over_damp", [0.0, 0.004, 0.5])
@pytest.mark.parametrize("nsig,K,nw", [(1, 513, 24000), (3, 4608, 901), (10, 1023, 1300)])
def test_damped_transform_of_large_problems_matches_the_oracle(B, nsig, K, nw, dt_over_damp):
    # past the size from which samples go in blocks of 512 (one sample past a block, whole
    # blocks, one short), undamped, damped, and damped too strongly within a block for that path;
    # bound of the kernel's test at small sizes
    from oracle import tdb_spectra as SP
    rng = np.random.default_rng(nsig + K)
    x = rng.normal(size=(nsig, K))
    om = rng.uniform(0.0, 5.0, size=nw)
    dt = 0.2
    t_damp = dt / dt_over_damp if dt_over_damp else 0.0
    got = B.tdb_damped_transform(x, dt, t_damp, om)
    ref = SP.damped_transform(x, dt, t_damp or np.inf, om)
    scale = dt * np.sum(np.abs(x), axis=1, keepdims=True)
    assert np.max(np.abs(got - ref) / scale) < 1e-13


# one sample; shares of a 16-CTA cluster that leave CTAs empty, one chunk of 32 per CTA, two
# chunks with a ragged second; batch sizes that do not divide the samples; hidden and feature
# counts that are not multiples of 4, and the largest network
@pytest.mark.parametrize("F,H,n,batch", [(1, 1, 1, 1), (5, 7, 40, 9), (16, 64, 1100, 512),
                                         (32, 64, 2000, 700), (3, 33, 600, 600)])
def test_training_epochs_match_the_oracle_gradients_and_adam(B, F, H, n, batch):
    # FP32 sums of at most 700 terms against FP64 agree to ~1e-6 of the largest gradient
    # component; a master weight within that of a tie may round to the other bfloat16, which moves
    # the gradient by up to ~3e-4 of its largest component.  Adam divides by sqrt(v): a parameter
    # with a small gradient may differ by up to its whole step (2 lr), others by that error over
    # sqrt(v) (factor 50: two moments over the steps), and the mean stays below 2% of a step.
    rng = np.random.default_rng(F * 100 + H)
    p = (rng.normal(size=F * H + H + H * H + 2 * H + 1) * 0.3).astype(np.float32)
    X = rng.normal(size=(n, F)).astype(np.float32)
    Y = rng.normal(size=n).astype(np.float32)
    lr = 1e-3
    with B.ShiftNet(F, H) as net:
        net.set_params(p)
        loss = net.train(X, Y, epochs=2, batch=batch, lr=lr)
        got = net.params()
    q, m, v, t = p.astype(np.float64), 0.0, 0.0, 0
    allowed = 2.0 ** -22 * np.abs(q) + 1e-8
    for ep in range(2):
        sse = 0.0
        for s in range(0, n, batch):
            x, y = X[s:s + batch].astype(np.float64), Y[s:s + batch].astype(np.float64)
            l, g = O.shiftnet_loss_grad(q, x, y, F, H)
            sse += l * len(y)
            t += 1
            m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
            rms = np.sqrt(v / (1 - 0.999 ** t)) + 1e-8
            q = q - lr * (m / (1 - 0.9 ** t)) / rms
            allowed = allowed + lr * np.minimum(2.0, 50 * 3e-4 * np.max(np.abs(g)) / rms)
    assert abs(loss - sse / n) < 1e-4 * (sse / n)
    assert np.all(np.abs(got - q) <= allowed)
    assert np.mean(np.abs(got - q)) < 0.02 * lr * t


# N = 188, 192 (the largest size of the library's own inverse), 196 (cuSOLVER / Newton-Schulz)
@pytest.mark.parametrize("form,tol", [("fp64", 1e-9), ("fp64s", 1e-8)])
@pytest.mark.parametrize("n_atoms", [47, 48, 49])
def test_ehrenfest_matches_the_oracle_on_both_sides_of_the_inverse_rule(B, n_atoms, form, tol):
    # bounds of the Ehrenfest parity tests of the two forms
    sysm = I.small_cluster(n_atoms, seed=7, T=3000.0, rep_A=60.0)
    run = I.Run(dt=0.2, n_steps=0, scc=True, move_nuclei=True, kick=1e-2, kT=I.SCC_KT)
    n = 40
    with B.Propagator(sysm, run, form) as p:
        p.setup()
        p.step(n // 2)
        p.observables()                 # the next step keeps what this evaluated
        p.step(n // 2)
        hist = B.tdb_dipole_history(p.ctx, n)
        obs = p.observables(forces=True)
        again = p.observables(forces=True)
        rho = B.tdb_get_rho(p.ctx)
    rho0, gs, S, Sinv = O.setup(sysm, run)
    tr = O.propagate(sysm, run, rho0, n, keep_forces=True)
    assert np.max(np.abs(hist - tr.dipole[:n])) < tol
    assert np.max(np.abs(obs["forces"] - tr.forces[-1])) < tol
    assert np.max(np.abs(rho - tr.rho)) < tol
    assert abs(obs["work"] - tr.work[-1]) < 1e-9
    assert np.array_equal(obs["forces"], again["forces"])


@pytest.mark.parametrize("s0", [0.3, np.float64(7.1373463)])
def test_ill_conditioned_overlaps_are_inverted_in_fp64(B, s0):
    # the overlap amplitude of the other systems and one that brings the smallest eigenvalue of S
    # to ~1e-6 of the largest: past what two Newton-Schulz steps from an FP32 inverse reach.  Forces of the ground
    # state against the oracle: an inverse accurate to cond(S) 2^-52 of its largest element (1e6
    # here) leaves about cond^2 2^-52 of S^-1 H rho's terms, which are O(1).
    import dataclasses
    sysm = dataclasses.replace(I.small_cluster(12, seed=5), s0=s0)
    S, H0 = O.model_matrices(sysm, sysm.R)
    ev = np.linalg.eigvalsh(S)
    cond = ev[-1] / ev[0]
    run = I.Run(dt=1e-6, n_steps=0, scc=False, move_nuclei=True, kT=I.SCC_KT)
    with B.Propagator(sysm, run, "fp64") as p:
        p.setup()
        f = p.observables(forces=True)["forces"]
    rho, gs, S, Sinv = O.setup(sysm, run)
    G = O.gamma_matrix(sysm, sysm.R)
    q = O.mulliken(sysm, rho, S) - O.reference_populations(sysm)
    E = np.zeros(3)
    v = O.atom_potential(G, q, sysm.R, E, False)
    H = O.scc_hamiltonian(sysm, H0, S, v)
    ref = O.forces(sysm, rho, S, Sinv, H, G, q, v, sysm.R, E, False)
    assert np.all(np.isfinite(f))
    assert np.max(np.abs(f - ref)) < 1e-10 + 100 * cond ** 2 * 2.0 ** -52 * np.max(np.abs(ref))


# N = 4 (fewer rows than CTAs), 36 (rows that do not divide), 64 (the largest); a laser and one
# orbital per atom
@pytest.mark.parametrize("n_atoms,n_species,laser,per", [(1, 1, False, 4), (9, 2, True, 4),
                                                         (16, 1, False, 4), (13, 1, True, 1)])
def test_cluster_steps_give_the_bits_of_the_separate_kernels(B, n_atoms, n_species, laser, per):
    # tdb_step runs small FP64 systems in one launch, tdb_step_profiled always step by step in the
    # separate kernels; the same steps taken either way, in pieces or at once, agree bit for bit
    import dataclasses
    sysm = I.small_flake(n_atoms, seed=8, n_species=n_species)
    if per == 1:
        sysm = dataclasses.replace(sysm, orbs_per_atom=1, n_electrons=1.0 * n_atoms)
    fld = I.Field(E0=0.02, omega=0.3, phase=0.3, t_center=4.0, fwhm=3.0, envelope=1,
                  dir=np.array([0.6, 0.8, 0.0])) if laser else None
    run = I.Run(dt=0.2, n_steps=0, scc=True, kick=1e-2, field=fld, kT=I.SCC_KT)
    out = []
    for how in ("at once", "pieces", "profiled"):
        with B.Propagator(sysm, run, "fp64") as p:
            p.setup()
            if how == "at once":
                p.step(38)
            elif how == "pieces":
                for n in (1, 2, 1, 3, 31):
                    p.step(n)
            else:
                for _ in range(38):
                    B.tdb_step_profiled(p.ctx)
            out.append((B.tdb_get_state(p.ctx), B.tdb_dipole_history(p.ctx, 38),
                        p.observables()["E_total"]))
    for o in out[1:]:
        assert o[0] == out[0][0] and np.array_equal(o[1], out[0][1]) and o[2] == out[0][2]


# one orbital per atom gives N that is no multiple of 4 or 2: rows without 16-byte alignment in
# every form (N = 13, 70 and 193, the last with the FP64 form's sliced products)
@pytest.mark.parametrize("form,n_atoms,tol", [
    ("fp64", 193, 1e-10), ("fp64s", 13, 2e-8), ("fp64s", 70, 2e-8), ("fp32", 13, 1e-6),
    ("fp32", 70, 1e-6), ("fp32", 193, 1e-6), ("fp16x6", 13, 1e-6), ("fp16x6", 70, 1e-6), ("bf16x3", 13, 2e-5),
    ("bf16x3", 70, 2e-5)])
def test_rows_without_alignment_match_the_oracle(B, form, n_atoms, tol):
    # the bounds of each form's parity tests; a clone half way steps to the same bits
    import dataclasses
    sysm = dataclasses.replace(I.small_flake(n_atoms, seed=8), orbs_per_atom=1,
                               n_electrons=1.0 * n_atoms)
    run = I.Run(dt=0.2, n_steps=0, scc=True, kick=1e-3, kT=I.SCC_KT)
    n = 60
    with B.Propagator(sysm, run, form) as p:
        p.setup()
        p.step(n // 2)
        c = B.tdb_clone(p.ctx)
        p.step(n - n // 2)
        B.tdb_step(c, n - n // 2)
        hist = B.tdb_dipole_history(p.ctx, n)
        rho = B.tdb_get_rho(p.ctx)
        same = B.tdb_get_state(p.ctx) == B.tdb_get_state(c)
        B.tdb_destroy(c)
    tr = O.propagate(sysm, run, O.setup(sysm, run)[0], n)
    assert np.max(np.abs(hist - tr.dipole[:n])) < tol
    assert np.max(np.abs(rho - tr.rho)) < tol
    assert same


# less than a block of 128 samples, one block and a ragged one, two whole ones (a sum of two does not
# depend on its order); more batches than one launch takes; hidden and feature counts that are
# no multiples of 4
@pytest.mark.parametrize("F,H,n,batch", [(16, 64, 2048, 256), (5, 7, 400, 100), (32, 64, 1250, 250),
                                         (3, 33, 390, 130), (1, 1, 300, 1)])
def test_training_epochs_give_the_bits_of_the_gradient_kernel_and_adam(B, F, H, n, batch):
    # the same steps from tdb_shiftnet_gradient (same block sums) and Adam in FP32: moments by one
    # fused multiply-add each, bias corrections from powers rounded once
    f, d = np.float32, np.float64
    rng = np.random.default_rng(F * 100 + H)
    p = (rng.normal(size=F * H + H + H * H + 2 * H + 1) * 0.3).astype(f)
    X = rng.normal(size=(n, F)).astype(f)
    Y = rng.normal(size=n).astype(f)
    lr, b1, b2 = f(2e-3), f(0.9), f(0.999)
    with B.ShiftNet(F, H) as net:
        net.set_params(p)
        net.train(X, Y, epochs=1, batch=batch, lr=lr)
        got = net.params()
        q, m, v = p, np.zeros_like(p), np.zeros_like(p)
        for t, s in enumerate(range(0, n, batch), 1):
            net.set_params(q)
            g = net.gradient(X[s:s + batch], Y[s:s + batch])[1]
            m = (d(b1) * m + ((f(1) - b1) * g).astype(d)).astype(f)
            v = (d(b2) * v + ((f(1) - b2) * g * g).astype(d)).astype(f)
            c1, c2 = (f(1) - f(float(b) ** t) for b in (b1, b2))
            q = q - (lr * (m / c1)) / (np.sqrt(v / c2) + f(1e-8))
            assert q.dtype == f
    assert np.array_equal(got, q)


@pytest.mark.parametrize("H", [5, 64])
def test_an_infinite_feature_saturates_its_units_and_no_others(B, H):
    # tanh takes +-inf to +-1, so the loss stays finite and only the gradient of the infinite
    # feature's weights (inf times a derivative of zero) is NaN, as in the gradient kernel
    F, n = 3, 100
    rng = np.random.default_rng(H)
    p = (rng.normal(size=F * H + H + H * H + 2 * H + 1) * 0.3).astype(np.float32)
    X = rng.normal(size=(n, F)).astype(np.float32)
    X[17, 1] = np.inf
    Y = rng.normal(size=n).astype(np.float32)
    with B.ShiftNet(F, H) as net:
        net.set_params(p)
        loss, g = net.gradient(X, Y)
        net.set_params(p)
        assert net.train(X, Y, epochs=1, batch=n, lr=1e-3) == pytest.approx(loss, rel=1e-6)
        q = net.params()
    assert np.isfinite(loss) and np.isfinite(g).sum() == len(g) - H
    assert np.array_equal(np.isfinite(q), np.isfinite(g))


@pytest.mark.parametrize("form,n_atoms", [("fp64", 12), ("fp64s", 12), ("fp64s", 49)])
@pytest.mark.parametrize("failures", [1, 2])
def test_a_failed_graph_leaves_an_ehrenfest_run_as_it_was(B, form, n_atoms, failures):
    # the calls that would capture a step fail on the host (out of memory, say); the same steps taken
    # afterwards give the bits of an undisturbed run
    sysm = I.small_cluster(n_atoms, seed=7, T=3000.0, rep_A=60.0)
    run = I.Run(dt=0.2, n_steps=0, scc=True, move_nuclei=True, kick=1e-2, kT=I.SCC_KT)
    out = []
    for fail in (0, failures):
        with B.Propagator(sysm, run, form) as p:
            p.setup()
            done = 0
            while done < 12:
                if fail:
                    B.load().tdb_test_fail_once(1)
                try:
                    p.step(1)
                    done += 1
                except B.TdbError as e:
                    assert e.status == 3 and "graph" in str(e)
                    fail -= 1
            B.load().tdb_test_fail_once(0)
            assert fail == 0
            out.append((B.tdb_get_state(p.ctx), B.tdb_dipole_history(p.ctx, 12)))
    assert out[0][0] == out[1][0] and np.array_equal(out[0][1], out[1][1])


def test_damped_transform_of_large_problems_takes_infinite_samples_as_fp64_does(B):
    # an infinite sample times the cosine and sine of its phase: infinities of their signs (those
    # above 1e-9 keep them: the twiddles are good to tens of ulps); a NaN makes its own signal NaN,
    # other signals are as without them
    from oracle import tdb_spectra as SP
    rng = np.random.default_rng(3)
    x = rng.normal(size=(4, 4608))
    om = rng.uniform(0.1, 5.0, size=901)
    dt, t_damp = 0.2, 200.0
    x[1, 700], x[2, 3000], x[3, 4607] = np.inf, -np.inf, np.nan
    re, im = np.empty((4, 901)), np.empty((4, 901))   # (a complex array has no infinite parts of its own)
    assert B.load().tdb_damped_transform(4, 4608, B._ptr(x), dt, t_damp, 901, B._ptr(om), B._ptr(re),
                                         B._ptr(im)) == 0
    ref = SP.damped_transform(x[:1], dt, t_damp, om)
    assert np.max(np.abs(re[0] + 1j * im[0] - ref[0])) < 1e-13 * dt * np.sum(np.abs(x[0]))
    for s, n, sign in ((1, 700, 1.0), (2, 3000, -1.0)):
        c, d = np.cos(om * n * dt), np.sin(om * n * dt)
        assert np.min(np.abs(c)) > 1e-9 and np.min(np.abs(d)) > 1e-9
        assert np.array_equal(re[s], sign * np.sign(c) * np.inf)
        assert np.array_equal(im[s], sign * np.sign(d) * np.inf)
    assert np.all(np.isnan(re[3])) and np.all(np.isnan(im[3]))


def test_contexts_and_clones_without_product_slices_step_with_fp64_products(B):
    # the slices' memory cannot be had, for the source, the clone or both: every call is served, a pair
    # of the same kind steps to the same bits and any two of them within the form's bound; the clone of
    # a source without slices has none either
    sysm = I.small_flake(49, seed=8)
    run = I.Run(dt=0.2, n_steps=0, scc=True, kick=1e-2, kT=I.SCC_KT)
    n = 40
    ends = []
    for no_src, no_clone in ((0, 0), (0, 1), (1, 0), (1, 1)):
        B.load().tdb_test_fail_once(2 * no_src)
        with B.Propagator(sysm, run, "fp64") as p:
            p.setup()
            p.step(n // 2)
            B.load().tdb_test_fail_once(2 * no_clone)
            c = B.tdb_clone(p.ctx)
            B.load().tdb_test_fail_once(0)
            p.step(n // 2)
            B.tdb_step(c, n // 2)
            same = B.tdb_get_state(p.ctx) == B.tdb_get_state(c)
            assert same == (no_src or not no_clone)
            ends += [B.tdb_get_rho(p.ctx), B.tdb_get_rho(c)]
            B.tdb_destroy(c)
    assert not np.array_equal(ends[0], ends[4])     # (slices and DFMA products differ in the last bits)
    for e in ends[1:]:
        assert np.max(np.abs(e - ends[0])) < 1e-10


def test_damped_transform_needs_no_more_memory_than_its_samples_and_results(B):
    # 320 MB of results where 420 MB are free; damped too strongly within a block for the blocked
    # path; two samples, so that the reference is a closed form
    import torch
    rng = np.random.default_rng(9)
    x, om = rng.normal(size=(100, 2)), rng.uniform(0.0, 5.0, size=200000)
    dt, t_damp = 0.2, 0.5
    B.tdb_damped_transform(x, dt, t_damp, om[:1])
    torch.cuda.empty_cache()
    fill = torch.empty(torch.cuda.mem_get_info()[0] - (420 << 20), dtype=torch.uint8, device="cuda")
    try:
        got = B.tdb_damped_transform(x, dt, t_damp, om)
    finally:
        del fill
        torch.cuda.empty_cache()
    ref = dt * (x[:, :1] + x[:, 1:] * np.exp((1j * om - 1 / t_damp) * dt)[None])
    assert np.max(np.abs(got - ref) / (dt * np.sum(np.abs(x), axis=1, keepdims=True))) < 1e-13


def test_clones_step_with_the_tuned_tile_width_of_their_source(B):
    # a width is tuned once (tens of launches); the clone of a context that has none tunes its own
    sysm = I.small_flake(40, seed=8)
    run = I.Run(dt=0.2, n_steps=0, scc=True, kick=1e-3, kT=I.SCC_KT)
    with B.Propagator(sysm, run, "bf16x3") as p:
        p.setup()
        early = B.tdb_clone(p.ctx)
        B.tdb_set_x_tile(p.ctx, 176)
        p.step(3)
        c = B.tdb_clone(p.ctx)
        assert B.tdb_x_tile(early) == 0 and B.tdb_x_tile(c) == 176
        for x in (p.ctx, c):
            B.tdb_step(x, 10)
        B.tdb_step(early, 13)
        assert B.tdb_x_tile(c) == 176 and B.tdb_x_tile(early) in (128, 176, 256)
        state = B.tdb_get_state(p.ctx)
        assert B.tdb_get_state(c) == state and B.tdb_get_state(early) == state
        for x in (c, early):
            B.tdb_destroy(x)


# N = 48, 188 and 192 (the largest size of that inverse)
@pytest.mark.parametrize("n_atoms,s0", [(12, 7.1373463), (47, 6.7347821), (48, 6.8602551)])
def test_the_fp64_repair_of_an_ill_conditioned_inverse_is_needed_and_taken(B, n_atoms, s0):
    # cond(S) = 1.09e6.  A stable FP64 inverse and ground state leave a small multiple of N cond 2^-52
    # of the forces (three eigensolvers differ by 2e-9); two Newton-Schulz steps from an FP32 inverse
    # without the repair leave 1e-6 to 4e-5, at least 19 times the bound
    import dataclasses
    sysm = dataclasses.replace(I.small_cluster(n_atoms, seed=5), s0=s0)
    S, H0 = O.model_matrices(sysm, sysm.R)
    ev = np.linalg.eigvalsh(S)
    run = I.Run(dt=1e-6, n_steps=0, scc=False, move_nuclei=True, kT=I.SCC_KT)
    with B.Propagator(sysm, run, "fp64") as p:
        p.setup()
        f = p.observables(forces=True)["forces"]
    rho, gs, S, Sinv = O.setup(sysm, run)
    G = O.gamma_matrix(sysm, sysm.R)
    q = O.mulliken(sysm, rho, S) - O.reference_populations(sysm)
    E = np.zeros(3)
    v = O.atom_potential(G, q, sysm.R, E, False)
    ref = O.forces(sysm, rho, S, Sinv, O.scc_hamiltonian(sysm, H0, S, v), G, q, v, sysm.R, E, False)
    assert np.max(np.abs(f - ref)) < 10 * sysm.n_orb * ev[-1] / ev[0] * 2.0 ** -52 * np.max(np.abs(ref))


@pytest.mark.parametrize("n_atoms", [47, 48, 65])
def test_windows_of_the_fp64_form_match_the_oracle_on_both_sides_of_the_slice_rule(B, n_atoms):
    # N = 188 (DFMA products), 192 and 260 (slices); the FP64 form's bound of the window tests
    sysm = I.small_flake(n_atoms, seed=8)
    run = I.Run(dt=0.2, n_steps=0, scc=True, kick=0.02, kT=I.SCC_KT)
    with B.Propagator(sysm, run, "fp64") as p:
        p.setup()
        p.step(5)
        rho, prev = B.tdb_get_rho(p.ctx, prev=True)
        v = B.tdb_scc_shift(p.ctx)
        B.tdb_step_window(p.ctx, v, 9)
        got, got_prev = B.tdb_get_rho(p.ctx, prev=True)
    S, H0 = O.model_matrices(sysm, np.asarray(sysm.R))
    a, b = O.window_propagate(prev, rho, S, O.scc_hamiltonian(sysm, H0, S, v), run.dt, 9)
    assert np.max(np.abs(got_prev - a)) < 1e-10
    assert np.max(np.abs(got - b)) < 1e-10


# one element; one K element short of, at and past the exact chunk of 128; ragged tiles; the largest K;
# "spread" gives a row's elements 60 binades, "extreme" makes every digit product as large as it gets
# (x0: digits -127, -128, ..., -128) with one sign, which fills the FP32 accumulators and 64-bit sums,
# "cancel" leaves 2^-40 of the terms' size
@pytest.mark.parametrize("M,N,K,kind", [(1, 1, 1, "normal"), (5, 7, 127, "normal"), (130, 66, 128, "normal"),
                                        (129, 65, 129, "spread"), (129, 65, 1025, "normal"),
                                        (3, 5, 4096, "spread"), (3, 5, 4096, "extreme"),
                                        (130, 66, 128, "extreme"), (33, 40, 1000, "cancel")])
def test_seven_digit_slice_products_keep_their_error_bound(B, M, N, K, kind):
    # operands to 2^-55 of their row's largest value (twice, over K terms), digit pairs from 2^-64 of the
    # row scales on dropped (20.1 2^-64 of the largest values a term), the sum rounded once
    import ctypes
    rng = np.random.default_rng(M + N + K)
    A, Bt = rng.normal(size=(M, K)), rng.normal(size=(N, K))
    if kind == "spread":
        A *= 2.0 ** rng.integers(-60, 1, A.shape)
        Bt *= 2.0 ** rng.integers(-60, 1, Bt.shape)
    if kind == "extreme":
        x0 = (127 + sum(128 * 2.0 ** (-8 * s) for s in range(1, 7))) / 128
        A[:], Bt[:] = -x0, -x0
    if kind == "cancel":
        A[:, K // 2:], Bt[:, K // 2:] = -A[:, :K // 2], Bt[:, :K // 2]
        A[:, 0] *= 1 + 2.0 ** -40
    C = np.zeros((M, N))
    dp = ctypes.POINTER(ctypes.c_double)
    fn = B.load().tdb_test_slice_gemm7
    fn.restype, fn.argtypes = ctypes.c_int, [ctypes.c_int] * 3 + [dp] * 3
    assert fn(M, N, K, B._ptr(A), B._ptr(Bt), B._ptr(C)) == 0
    ref = A.astype(np.longdouble) @ Bt.T.astype(np.longdouble)
    eps = float(np.finfo(np.longdouble).eps)   # of the reference's own sums
    big = K * np.abs(A).max(1)[:, None] * np.abs(Bt).max(1)[None]
    bound = big * (2.0 ** -54 + 20.1 * 2.0 ** -64 + K * eps) + 2.0 ** -53 * np.abs(ref)
    assert np.all(np.abs(C - ref) <= bound)

"""GPU checks of the split-precision tensor-core path (tcgen05, FP16x3/BF16x3/TF32x3).

The product engine is checked against the FP64 product; the density, charges,
forces and kernel against the oracle.  Tolerances of the mixed forms: charges
1e-5 e, forces 1e-4 eV/A.
"""
import os

import numpy as np
import pytest

import oracle as O
import synth

pytestmark = pytest.mark.gpu

ALPHA_MIX = 0.06


@pytest.fixture(scope="module")
def X():
    import paper_1705_10845_gb300 as X
    X.build.build()
    X.load()
    return X


def sysdict(s):
    return dict(natoms=s.natoms, L=s.L, R=s.R, V=s.V, Z=s.Z, mass=s.mass)


@pytest.mark.parametrize("n", [128, 256, 384, 1024, 2944, 4096, 8192])
@pytest.mark.parametrize("sym", [False, True])
@pytest.mark.parametrize("prec,bound", [("fp16x3", 1e-6), ("bf16x3", 2e-5), ("tf32x3", 1e-6)])
def test_tensor_core_product_matches_fp64(X, n, sym, prec, bound):
    err, flag, ms = X.binding.selftest_gemm(n, prec, sym)
    assert flag == 0
    # entries are sums of n products of U(-1, 1) numbers; the tensor-core FP32
    # accumulation loses up to ~2^-23 of the running sum per step, so the
    # error bound grows linearly with n (a wrong operand layout gives O(1)).
    print(prec, n, sym, err, ms)
    assert err < bound * n, (err, ms)


@pytest.mark.parametrize("n", [256, 384, 1024, 4096, 8192])
@pytest.mark.parametrize("prec,bound", [("fp16x3", 1e-6), ("bf16x3", 2e-5), ("tf32x3", 1e-6)])
def test_pair_product_matches_fp64(X, n, prec, bound):
    # C = A B^T + B A^T as one symmetric-output product over two K ranges (the
    # A1 = T T1 + T1 T of the response chains); twice the sums of one product
    err, flag, ms = X.binding.selftest_gemm(n, prec, 2)
    print(prec, n, "pair", err, ms)
    assert flag == 0
    assert err < 2 * bound * n, (err, ms)


@pytest.mark.parametrize("n", [384, 2944, 4096, 6144, 8192])
@pytest.mark.parametrize("sym", [0, 1, 2])
@pytest.mark.parametrize("prec,u", [("fp16x3", 2.0 ** -11), ("bf16x3", 2.0 ** -8), ("tf32x3", 2.0 ** -11)])
def test_single_product_matches_fp64(X, n, sym, prec, u):
    # one product of the hi operands (FP16 and TF32 keep 11 significant bits, BF16 8), the
    # product of the single-product chains; below
    # n = 8192 consecutive tiles of a CTA alternate between the two TMEM accumulators, at
    # n = 8192 the hi*hi sum splits over both.  Each operand carries a relative rounding error of
    # at most u, so an entry's error is a sum of n terms a db + b da with standard deviation about
    # u sqrt(2 n / 27) for U(-1, 1) inputs; the bound is 8 of those (twice that for the pair
    # product), far below the O(sqrt(n)) error of a wrong tile or accumulator
    err, flag, ms = X.binding.selftest_gemm(n, prec, sym if sym != 2 else 2, single=True)
    bound = 8.0 * u * np.sqrt(2.0 * n / 27.0) * (2.0 if sym == 2 else 1.0)
    print(prec, n, "single", sym, err, bound, ms)
    assert flag == 0
    assert err < bound, (err, bound, ms)


@pytest.mark.parametrize("prec", ["fp16x3", "bf16x3", "tf32x3"])
@pytest.mark.parametrize("case", ["tiny24", "ragged37"])
@pytest.mark.parametrize("mu_prec", [0, 1])
def test_split_density_against_oracle(X, prec, case, mu_prec):
    # mu_prec = 1: the chemical-potential chain at one hi*hi product (the mu start is 0.01 eV
    # off, so the Newton steps and the first-order correction both use it)
    s = synth.make_system(24, 1705, L=7.0) if case == "tiny24" else synth.make_system(37, 11)
    p = X.default_params(mix_alpha=ALPHA_MIX, kernel_c=1 - 1 / ALPHA_MIX, prec=prec, mu_tol=1e-3,
                         mu_prec=mu_prec)
    m = O.Model(Te=p.Te, n_sq=p.n_sq)
    rng = np.random.default_rng(2)
    n = rng.normal(scale=0.02, size=s.natoms)
    n -= n.mean()
    xl = O.XLParams(rank_m=p.rank_m, kernel_c=p.kernel_c)
    ref = O.evaluate(s.R, s.L, s.Z, n, m, xl)
    with X.Context(p, [sysdict(s)]) as ctx:
        ctx.set(0, X.N, n)
        ctx.set(0, X.MU, [ref.dens.mu + 0.01])
        ctx.build_H(0)
        ctx.density(0)
        ctx.kernel_update(0)
        ctx.energy(0)
        q, F, Kr = ctx.get(0, X.Q), ctx.get(0, X.F), ctx.get(0, X.KR)
        E = ctx.get(0, X.ENERGY)
    # FP16x3 and TF32x3 meet the mixed-precision bounds (1e-5 e, 1e-4 eV/A): both hi/lo pairs
    # keep 22 significant bits.  BF16x3 does not: its pair keeps 16, and its charges measure
    # 1.1-1.4e-5 e here (2-3e-5 e at 1536-2048 atoms), so it is held to its own measured level
    # (3e-5 e) and is not used by the bench, batch or serving workloads
    tol_q = 3e-5 if prec == "bf16x3" else 1e-5
    tol_f = 1e-4
    print(prec, case, "mu_prec", mu_prec, "dq", np.abs(q - ref.q).max(), "dF", np.abs(F - ref.F).max(), "dKr",
          np.abs(Kr - ref.Kr).max())
    assert np.max(np.abs(q - ref.q)) < tol_q
    assert np.max(np.abs(F - ref.F)) < tol_f
    assert np.max(np.abs(Kr - ref.Kr)) < 100 * tol_q
    # energy monitor: Omega and its parts against the oracle (eV)
    print(prec, case, "dOmega", E[0] - ref.Omega, "dS", E[3] - ref.parts["entropy"])
    assert abs(E[3] - ref.parts["entropy"]) < 1e-3
    assert abs(E[0] - ref.Omega) < (2e-2 if prec == "bf16x3" else 2e-3)


@pytest.mark.parametrize("mu_prec", [0, 1])
def test_full_size_charges_against_oracle(X, mu_prec):
    # the bench workload: 1536 atoms (N = 6144), Te = 1500 K, 14 squarings,
    # FP16x3, at the t0 ground state that the MD starts from (kernel SCF with
    # the automatic J_0); the oracle diagonalises H on the host at the same
    # (R, n) and the charges must agree to 1e-5 e, with the mu chain at three
    # products or at one
    s = synth.make_system(1536, 1705)
    p = X.default_params(Te=1500.0, n_sq=14, rank_m=4, mix_alpha=ALPHA_MIX, kernel_c=1 - 1 / ALPHA_MIX,
                         prec="fp16x3", mu_tol=1e-3, scf_mode=1, kernel_auto=1, scf_tol=1e-5,
                         scf_max_iter=200, mu_prec=mu_prec)
    with X.Context(p, [sysdict(s)]) as ctx:
        ctx.scf(0)
        n = ctx.get(0, X.N)
        ctx.build_H(0)
        ctx.density(0)
        q = ctx.get(0, X.Q)
    q_ref = O.charges_at(s.R, s.L, s.Z, n, O.Model(Te=1500.0, n_sq=14))
    err = np.max(np.abs(q - q_ref))
    print("full size fp16x3 mu_prec", mu_prec, "|dq|", err)
    assert err < 1e-5


@pytest.fixture(scope="module")
def ref2048():
    """The oracle's evaluation of the 2048-atom state (one eigendecomposition for every precision)."""
    s = synth.make_system(2048, 1705)
    m = O.Model(Te=1000.0, n_sq=10, rep_A=40.0, rep_rho=0.3)
    rng = np.random.default_rng(2048)
    n = rng.normal(scale=0.01, size=s.natoms)
    n -= n.mean()
    ref = O.evaluate(s.R, s.L, s.Z, n, m, O.XLParams(rank_m=4, kernel_c=1 - 1 / ALPHA_MIX))
    return s, n, ref


@pytest.mark.parametrize("prec", ["fp16x3", "tf32x3"])
def test_accumulator_split_size_against_oracle(X, ref2048, prec):
    # 2048 atoms (N = 8192): the first size whose products split their hi*hi sums over both
    # TMEM accumulators.  At a seeded (R, n) with the Newton search started 5 meV off the
    # oracle's mu (no SCF needed), the split path with the bench's chain precisions (probe and
    # mu chains at one hi*hi product) must match the oracle's eigendecomposition element by
    # element: charges to 1e-5 e, forces to 1e-4 eV/A; Omega and the rank-4 K r are reported
    # against it too.  Te = 1000 K and 10 squarings are the 4096-atom precision workload's.
    s, n, ref = ref2048
    p = X.default_params(Te=1000.0, n_sq=10, rank_m=4, mix_alpha=ALPHA_MIX, kernel_c=1 - 1 / ALPHA_MIX,
                         prec=prec, mu_tol=1e-3, rep_A=40.0, rep_rho=0.3, kernel_prec=1, mu_prec=1)
    with X.Context(p, [sysdict(s)]) as ctx:
        assert ctx.sizes(0)[2] == 8192
        ctx.set(0, X.N, n)
        ctx.set(0, X.MU, [ref.dens.mu + 0.005])
        ctx.build_H(0)
        ctx.density(0)
        ctx.kernel_update(0)
        ctx.energy(0)
        q, F, Kr, E = ctx.get(0, X.Q), ctx.get(0, X.F), ctx.get(0, X.KR), ctx.get(0, X.ENERGY)
    dq, dF = np.abs(q - ref.q).max(), np.abs(F - ref.F).max()
    dK = np.abs(Kr - ref.Kr).max() / np.abs(ref.Kr).max()
    print("2048 atoms", prec, ": |dq|", dq, "|dF|", dF, "dOmega", E[0] - ref.Omega, "K r rel", dK)
    assert dq < 1e-5
    assert dF < 1e-4
    assert abs(E[0] - ref.Omega) < 1e-6 * abs(ref.Omega)
    assert dK < 2e-3


@pytest.mark.parametrize("prec,tol", [("fp16x3", 1e-4), ("bf16x3", 1e-3), ("tf32x3", 1e-4)])
def test_split_exact_kernel_against_oracle(X, prec, tol):
    s = synth.make_system(37, 11)
    p = X.default_params(mix_alpha=ALPHA_MIX, kernel_c=1 - 1 / ALPHA_MIX, prec=prec, mu_tol=1e-3, kernel_mode=1)
    m = O.Model(Te=p.Te, n_sq=p.n_sq)
    rng = np.random.default_rng(8)
    n = rng.normal(scale=0.02, size=s.natoms)
    n -= n.mean()
    ev = O.evaluate(s.R, s.L, s.Z, n, m, None, with_kernel=False, with_forces=False)
    Kref = O.kernel_exact(ev.dens, ev.gamma)
    with X.Context(p, [sysdict(s)]) as ctx:
        ctx.set(0, X.N, n)
        ctx.set(0, X.MU, [ev.dens.mu])
        ctx.build_H(0)
        ctx.density(0)
        ctx.kernel_exact(0)
        K = ctx.get(0, X.KMAT)
    err = np.max(np.abs(K - Kref)) / np.abs(Kref).max()
    print(prec, "exact kernel rel err", err)
    assert err < tol


@pytest.mark.parametrize("variant", ["classic", "pair"])
def test_other_product_variants_match_fp64(X, variant):
    # the one-CTA-per-tile product kernel (XLBOMD_GEMM=classic) and the two-SM (cta_group::2)
    # kernel (XLBOMD_GEMM=pair, sizes that are multiples of 256) stay checked next to the default
    # one-SM persistent kernel; a fresh process reads the variant once
    import json
    import os
    import subprocess
    import sys
    code = ("import json, paper_1705_10845_gb300 as X; X.load(); "
            "print(json.dumps([[X.binding.selftest_gemm(n, p, s) for n in (256, 384, 2048) "
            "for p in ('fp16x3', 'bf16x3') for s in (False, True)], "
            "[X.binding.selftest_gemm(8192, 'fp16x3', s) for s in (False, True, 2)], "
            "[X.binding.selftest_gemm(4096, 'fp16x3', s, single=True) for s in (False, True, 2)]]))")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    out = subprocess.run([sys.executable, "-c", code], cwd=root, capture_output=True, text=True,
                         env=dict(os.environ, XLBOMD_GEMM=variant), timeout=300)
    assert out.returncode == 0, out.stderr[-2000:]
    res, large, single = json.loads(out.stdout.strip().splitlines()[-1])
    k = 0
    for n in (256, 384, 2048):
        for bound in (1e-6, 2e-5):
            for _sym in (False, True):
                err, flag, ms = res[k]
                k += 1
                assert flag == 0 and err < bound * n, (n, err)
    # n = 8192 split products (dense, symmetric, pair) with the bounds of the default kernel's tests
    for (err, flag, ms), bound in zip(large, (1e-6, 1e-6, 2e-6)):
        print(variant, "fp16x3 8192", err, ms)
        assert flag == 0 and err < bound * 8192, (err, ms)
    # single products (one 16-bit product) at n = 4096
    for (err, flag, ms), f in zip(single, (1.0, 1.0, 2.0)):
        bound = 8.0 * 2.0 ** -11 * np.sqrt(2.0 * 4096 / 27.0) * f
        assert flag == 0 and err < bound, (err, bound)


@pytest.mark.parametrize("prec", ["fp16x3", "bf16x3", "tf32x3"])
def test_single_product_probe_chains(X, prec):
    # kernel_prec = 1: the kernel's response chains run one hi*hi product per
    # step; charges and forces (expansion and mu chain at three products) do not
    # change, and K r is checked against the oracle's exact-response kernel
    s = synth.make_system(37, 11)
    out = {}
    ref = None
    for kp in (0, 1):
        p = X.default_params(mix_alpha=ALPHA_MIX, kernel_c=1 - 1 / ALPHA_MIX, prec=prec, mu_tol=1e-3,
                             kernel_prec=kp)
        m = O.Model(Te=p.Te, n_sq=p.n_sq)
        rng = np.random.default_rng(2)
        n = rng.normal(scale=0.02, size=s.natoms)
        n -= n.mean()
        ref = O.evaluate(s.R, s.L, s.Z, n, m, O.XLParams(rank_m=p.rank_m, kernel_c=p.kernel_c))
        with X.Context(p, [sysdict(s)]) as ctx:
            ctx.set(0, X.N, n)
            ctx.set(0, X.MU, [ref.dens.mu + 0.01])
            ctx.build_H(0)
            ctx.density(0)
            ctx.kernel_update(0)
            out[kp] = (ctx.get(0, X.Q), ctx.get(0, X.F), ctx.get(0, X.KR))
    q0, F0, K0 = out[0]
    q1, F1, K1 = out[1]
    assert np.array_equal(q0, q1) and np.array_equal(F0, F1)
    rel = np.abs(K1 - ref.Kr).max() / np.abs(ref.Kr).max()
    print(prec, "single-product probes: K r rel err", rel, "three products:",
          np.abs(K0 - ref.Kr).max() / np.abs(ref.Kr).max())
    assert rel < (2e-2 if prec == "bf16x3" else 2e-3)


def test_graph_replay_matches_direct_launches(X):
    # params.graphs = 1: chemical-potential passes and probe responses are
    # captured on their second run and replayed afterwards; a run through the
    # kernel SCF and 15 MD steps must equal the run with direct launches bitwise
    import torch
    s = synth.make_system(64, 3)
    res = {}
    stream = torch.cuda.Stream()      # the legacy default stream cannot be captured
    for g in (0, 1):
        p = X.default_params(mix_alpha=ALPHA_MIX, kernel_c=1 - 1 / ALPHA_MIX, prec="fp16x3", Te=1000.0,
                             n_sq=12, rank_m=2, scf_mode=1, kernel_auto=1, scf_tol=1e-5, mu_tol=1e-3,
                             rep_A=40.0, graphs=g)
        with X.Context(p, [sysdict(s)], stream=stream.cuda_stream) as ctx:
            ctx.scf(0)
            ctx.step(15)
            res[g] = [ctx.get(0, w) for w in (X.Q, X.R, X.NHIST, X.KR, X.F, X.STATS)]
    for a, b in zip(res[0], res[1]):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("n", [256, 384, 1024])
@pytest.mark.parametrize("sym", [0, 1, 2])
@pytest.mark.parametrize("single", [False, True])
@pytest.mark.parametrize("prec", ["fp16x3", "tf32x3"])
def test_grouped_product_equals_single_launches(X, n, sym, single, prec):
    # the grouped launch of the lockstep batch path (several problems' tiles in one persistent
    # launch, per-problem tensor maps and epilogue arguments from a device table, both tile
    # widths as the autotuner tries them) computes every tile exactly as a single launch does
    err, flag = X.binding.selftest_gemm_group(n, prec, sym, single=single, nprob=3)
    print(prec, n, sym, single, err)
    assert flag == 0
    assert err == 0.0


@pytest.mark.parametrize("kernel_prec,tol", [(0, 1e-4), (1, 2e-3)])
def test_grouped_exact_kernel_256_atoms(X, kernel_prec, tol):
    # the exact kernel K = (J - I)^-1 (Eq. KK) of a 256-atom system: its 256 unit-probe response
    # chains run up to 64 at a time in chain slots of their own, every chain product one grouped
    # launch; K against the oracle's eigenbasis kernel, and the cost of one recompute
    import time
    s = synth.make_system(256, 31)
    p = X.default_params(mix_alpha=ALPHA_MIX, kernel_c=1 - 1 / ALPHA_MIX, prec="fp16x3", mu_tol=1e-3,
                         kernel_mode=1, kernel_prec=kernel_prec)
    m = O.Model(Te=p.Te, n_sq=p.n_sq)
    rng = np.random.default_rng(9)
    n = rng.normal(scale=0.01, size=s.natoms)
    n -= n.mean()
    ev = O.evaluate(s.R, s.L, s.Z, n, m, None, with_kernel=False, with_forces=False)
    Kref = O.kernel_exact(ev.dens, ev.gamma)
    with X.Context(p, [sysdict(s)]) as ctx:
        ctx.set(0, X.N, n)
        ctx.set(0, X.MU, [ev.dens.mu])
        ctx.build_H(0)
        ctx.density(0)
        ctx.kernel_exact(0)           # allocates the chain slots
        ctx.get(0, X.MU)
        t = time.perf_counter()
        ctx.kernel_exact(0)
        K = ctx.get(0, X.KMAT)
        dt = time.perf_counter() - t
    err = np.max(np.abs(K - Kref)) / np.abs(Kref).max()
    print("exact kernel 256 atoms, kernel_prec", kernel_prec, "rel err", err, "recompute s", dt)
    assert err < tol


@pytest.mark.parametrize("nat", [32, 33, 224, 320, 352])
def test_density_where_the_tile_width_changes(X, nat):
    # symmetric products take 32-wide tiles up to 1024 padded orbitals, 64-wide ones at 1280 and 1408 (their
    # 32-wide tiles would need two waves of SMs); 128 and 256 are the smallest sizes, one and four
    # tiles.  Every product of the expansion writes its value and its operands in the epilogue, in both
    # triangles, with and without side inputs: charges to 1e-5 e and forces to 1e-4 eV/A of the oracle
    s = synth.make_system(nat, 7)
    p = X.default_params(mix_alpha=ALPHA_MIX, kernel_c=1 - 1 / ALPHA_MIX, prec="fp16x3", mu_tol=1e-3)
    m = O.Model(Te=p.Te, n_sq=p.n_sq)
    rng = np.random.default_rng(nat)
    n = rng.normal(scale=0.01, size=s.natoms)
    n -= n.mean()
    ref = O.evaluate(s.R, s.L, s.Z, n, m, O.XLParams(rank_m=p.rank_m, kernel_c=p.kernel_c))
    with X.Context(p, [sysdict(s)]) as ctx:
        ctx.set(0, X.N, n)
        ctx.set(0, X.MU, [ref.dens.mu + 0.01])
        ctx.build_H(0)
        ctx.density(0)
        ctx.kernel_update(0)
        q, F, Kr, D = ctx.get(0, X.Q), ctx.get(0, X.F), ctx.get(0, X.KR), ctx.get(0, X.D)
    assert np.max(np.abs(q - ref.q)) < 1e-5
    assert np.max(np.abs(F - ref.F)) < 1e-4
    assert np.max(np.abs(Kr - ref.Kr)) < 1e-3
    assert np.array_equal(D, D.T)


@pytest.mark.parametrize("nat,L", [(10, 5.3), (33, None), (255, None), (256, None), (620, None)])
def test_model_of_the_split_path_against_oracle(X, nat, L):
    # H (FP64 with an FP32 pair test before it), gamma and the forces at a given density: a box barely above
    # the cutoff (several images of each pair inside it), a warp's remainder, both sides of the Coulomb
    # force's split over tx (256 atoms) and of the four-atoms-a-block launch (608).  gamma sums 27 FP32
    # terms of order 1/r with relative errors of a few 2^-24 and cancellation between 1/r terms: 1e-5 of
    # its largest entry is loose; a missed or doubled image is 1e-3 and more
    s = synth.make_system(nat, 19, L=L)
    p = X.default_params(mix_alpha=ALPHA_MIX, kernel_c=1 - 1 / ALPHA_MIX, prec="fp16x3", rep_A=40.0, mu_tol=1e-3)
    m = O.Model(Te=p.Te, n_sq=p.n_sq, rep_A=40.0, rep_rho=p.rep_rho)
    rng = np.random.default_rng(nat)
    n = rng.normal(scale=0.01, size=s.natoms)
    n -= n.mean()
    H0, G = O.build_H0(s.R, s.L, m), O.build_gamma(s.R, s.L, m)
    with X.Context(p, [sysdict(s)]) as ctx:
        ctx.set(0, X.N, n)
        ctx.build_H(0)
        H, gam = ctx.get(0, X.H), ctx.get(0, X.GAMMA)
        if nat <= 256:
            ref = O.evaluate(s.R, s.L, s.Z, n, m, None, with_kernel=False)
            ctx.set(0, X.MU, [ref.dens.mu])
            ctx.density(0)
            F = ctx.get(0, X.F)
            # positions moved without a new Hamiltonian: the forces follow R
            ctx.set(0, X.R, s.R + 0.25)
            ctx.density(0)
            F2 = ctx.get(0, X.F)
            assert np.max(np.abs(F - ref.F)) < 1e-4
            assert np.max(np.abs(F2 - F)) < 1e-4
    off = ~np.eye(4 * nat, dtype=bool)
    assert np.max(np.abs(H - H0)[off]) < 1e-11
    assert np.max(np.abs(np.diag(H) - np.diag(H0) - np.repeat(G @ n, 4))) < 1e-4
    assert np.max(np.abs(gam - G)) < 1e-5 * np.max(np.abs(G))


@pytest.mark.parametrize("prec,nat,n_sq,kernel_prec", [("fp16x3", 32, 10, 0), ("fp16x3", 33, 1, 0), ("bf16x3", 33, 10, 0),
                                                       ("tf32x3", 65, 12, 0), ("fp16x3", 353, 10, 0),
                                                       ("fp16x3", 33, 10, 1), ("fp16x3", 33, 2, 1)])
def test_response_chain_by_levels(X, prec, nat, n_sq, kernel_prec):
    # both forms of a chain level (two launches up to 1408 padded orbitals, three at 353 atoms), the first level
    # made from the diagonal and the last one only reduced, also where they are the same (n_sq = 1) or
    # neighbours (2).  Against the oracle's response: 1e-4 with split products (1e-3 in BF16x3), 1e-2 with
    # single ones, whose operands are good to 2^-11
    import torch
    s = synth.make_system(nat, 27)
    Te = 1000.0 if n_sq >= 10 else 200000.0 / n_sq   # |beta (e - mu)| / 2^(n+1) stays below 1
    p = X.default_params(mix_alpha=ALPHA_MIX, kernel_c=1 - 1 / ALPHA_MIX, prec=prec, mu_tol=1e-3, n_sq=n_sq, Te=Te,
                         kernel_prec=kernel_prec)
    m = O.Model(Te=p.Te, n_sq=p.n_sq)
    rng = np.random.default_rng(nat)
    n = rng.normal(scale=0.01, size=nat)
    n -= n.mean()
    v = rng.normal(size=nat)
    v -= v.mean()
    v /= np.linalg.norm(v)
    ref = O.evaluate(s.R, s.L, s.Z, n, m, None, with_kernel=False, with_forces=False)
    wref = O.response(ref.dens, ref.gamma, v)
    with X.Context(p, [sysdict(s)]) as ctx:
        ctx.set(0, X.N, n)
        ctx.set(0, X.MU, [ref.dens.mu])
        ctx.build_H(0)
        ctx.density(0)
        vd = torch.tensor(v, dtype=torch.float64, device="cuda")
        wd = torch.zeros_like(vd)
        ctx.response(0, vd.data_ptr(), wd.data_ptr())
        torch.cuda.synchronize()
        w = wd.cpu().numpy()
    tol = 1e-2 if kernel_prec else 1e-3 if prec == "bf16x3" else 1e-4
    assert np.linalg.norm(w - wref) < tol * np.linalg.norm(wref)


@pytest.mark.parametrize("prec,nat,kernel_prec", [("fp64", 24, 0), ("fp16x3", 33, 0), ("fp16x3", 33, 1), ("bf16x3", 24, 0),
                                                  ("tf32x3", 65, 0), ("fp16x3", 353, 0)])
def test_response_is_linear_in_the_probe(X, prec, nat, kernel_prec):
    # w is linear in v and v has no preferred size: a factor 2^k of the probe is a factor 2^k of every number
    # of the chain, so w changes by exactly that factor (two- and three-launch chains, split and single products)
    import torch
    s = synth.make_system(nat, 27, **({"L": 7.0} if nat == 24 else {}))
    p = X.default_params(mix_alpha=ALPHA_MIX, kernel_c=1 - 1 / ALPHA_MIX, prec=prec, mu_tol=1e-3, kernel_prec=kernel_prec)
    rng = np.random.default_rng(nat)
    n = rng.normal(scale=0.01, size=nat)
    n -= n.mean()
    v = rng.normal(size=nat)
    with X.Context(p, [sysdict(s)]) as ctx:
        ctx.set(0, X.N, n)
        ctx.build_H(0)
        ctx.density(0)
        w = {}
        for k in (0, -60, -83, -300, 40, 66, 300):
            vd = torch.tensor(np.ldexp(v, k), dtype=torch.float64, device="cuda")
            wd = torch.zeros_like(vd)
            ctx.response(0, vd.data_ptr(), wd.data_ptr())
            torch.cuda.synchronize()
            w[k] = np.ldexp(wd.cpu().numpy(), -k)
        zero = torch.zeros(nat, dtype=torch.float64, device="cuda")
        wd = torch.ones_like(zero)
        ctx.response(0, zero.data_ptr(), wd.data_ptr())
        torch.cuda.synchronize()
    assert np.all(np.isfinite(w[0])) and np.max(np.abs(w[0])) > 0.1
    for k in w:
        assert np.array_equal(w[k], w[0]), k
    assert np.all(wd.cpu().numpy() == 0.0)


def hold_all_but(nbytes):
    """A device block that leaves about nbytes of device memory free."""
    import torch
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    return torch.empty(free - nbytes, dtype=torch.uint8, device="cuda")


@pytest.mark.parametrize("nat,left", [(33, 200 << 20), (96, 300 << 20)])
def test_exact_kernel_does_not_depend_on_free_memory(X, nat, left):
    # how many probes run side by side follows the free memory; the arithmetic of a probe must not.  33 atoms
    # (4 tiles each) sit where the form of a chain changes with the number of probes
    import torch
    s = synth.make_system(nat, 12)
    p = X.default_params(mix_alpha=ALPHA_MIX, kernel_c=1 - 1 / ALPHA_MIX, prec="fp16x3", mu_tol=1e-3, kernel_mode=1)
    K = []
    for little in (False, True):
        with X.Context(p, [sysdict(s)]) as ctx:
            ctx.build_H(0)
            ctx.density(0)
            held = hold_all_but(left) if little else None
            try:
                ctx.kernel_exact(0)
                K.append(ctx.get(0, X.KMAT))
            finally:
                del held
                torch.cuda.empty_cache()
    assert np.array_equal(K[0], K[1])


def test_exact_kernel_after_a_failed_allocation(X):
    # one chain slot of 200 atoms (896 padded orbitals, 45 MB) does not fit: ERR_OOM, nothing half-made is kept, and with the memory
    # back the same context gives the kernel that a fresh one gives
    import torch
    s = synth.make_system(200, 13)
    p = X.default_params(mix_alpha=ALPHA_MIX, kernel_c=1 - 1 / ALPHA_MIX, prec="fp16x3", mu_tol=1e-3, kernel_mode=1)
    K = []
    for fail in (False, True):
        with X.Context(p, [sysdict(s)]) as ctx:
            ctx.build_H(0)
            ctx.density(0)
            if fail:
                held = hold_all_but(24 << 20)
                try:
                    with pytest.raises(X.XlbomdError) as e:
                        ctx.kernel_exact(0)
                    assert e.value.status == -2
                finally:
                    del held
                    torch.cuda.empty_cache()
                assert ctx._lib.xlbomd_clear_error(ctx.h) == 0
            ctx.kernel_exact(0)
            K.append(ctx.get(0, X.KMAT))
    assert np.array_equal(K[0], K[1])


@pytest.mark.parametrize("prec", ["fp16x3", "tf32x3"])
def test_entropy_does_not_count_padding(X, prec, tmp_path):
    # 33 atoms: the log-determinants run over 192 rows, 60 of them padding, which must be rows of the identity.
    # What the planned corrections leave of an inverse (below 1e-8, but times up to 2^13) is a function of the
    # eigenvalue; it is computed here for the eigenvalues of the system and for the padding's zero, and
    # the entropy has to be off by the former alone, to within half of the latter (14 squarings: below that
    # the padding's part is no larger than what the error of D puts on the entropy, some 1e-5 eV)
    import shutil
    import subprocess
    n_sq = 14
    if shutil.which("g++") is None:
        pytest.skip("no host compiler")
    s = synth.make_system(33, 27)
    p = X.default_params(mix_alpha=ALPHA_MIX, kernel_c=1 - 1 / ALPHA_MIX, prec=prec, mu_tol=1e-3, n_sq=n_sq)
    m = O.Model(Te=p.Te, n_sq=p.n_sq)
    n = np.zeros(33)
    ref = O.evaluate(s.R, s.L, s.Z, n, m, None, with_kernel=False, with_forces=False)
    with X.Context(p, [sysdict(s)]) as ctx:
        ctx.set(0, X.N, n)
        ctx.set(0, X.MU, [ref.dens.mu])
        ctx.build_H(0)
        ctx.density(0)
        ctx.energy(0)
        S = ctx.get(0, X.ENERGY)[3]
    radius = np.abs(ref.H).sum(1) - np.abs(np.diag(ref.H))
    sc = m.beta / 2.0 ** (n_sq + 1)
    t0 = sc * max((np.diag(ref.H) + radius).max() - ref.dens.mu, ref.dens.mu - (np.diag(ref.H) - radius).min())
    src = tmp_path / "left.cpp"
    src.write_text(r"""
#include "plan.h"
#include <cstdio>
#include <cstdlib>
using namespace xl;
int main(int argc, char** argv) {   // t0, n, then eigenvalues of T_0: sum_k 2^(n-1-k) ln(1 - R_k) of each
  const int n = std::atoi(argv[2]);
  PlanCache cache;
  std::vector<LevelPlan> p;
  plan_expansion(cache, std::atof(argv[1]), n, 1e-8, p);
  for (int i = 3; i < argc; ++i) {
    double t = std::atof(argv[i]), w1 = 0.0, s1 = 0.0, sum = 0.0;
    for (int k = 0; k < n; ++k) {
      const double s = t * t, W0 = p[k].g[0] + p[k].g[1] * w1 + p[k].g[2] * s + p[k].g[3] * s1;
      double R = 1.0 - (1.0 + s) * (1.0 - W0);
      for (int r = 0; r < p[k].inv.n; ++r) R = std::pow(R, p[k].inv.order[r]);
      sum += std::ldexp(std::log1p(-R), n - 1 - k);
      s1 = s;
      w1 = 1.0 - (1.0 - R) / (1.0 + s);
      t = 2.0 * t * (1.0 - w1);
    }
    std::printf("%.17g\n", sum);
  }
}
""")
    exe = tmp_path / "left"
    csrc = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1705_10845_gb300", "csrc")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I" + csrc, str(src), "-o", str(exe)], check=True)
    t = [repr(float(x)) for x in sc * (ref.dens.mu - ref.dens.eps)] + ["0.0"]
    left = [float(x) for x in subprocess.run([str(exe), repr(float(t0)), str(n_sq)] + t, capture_output=True, text=True,
                                             check=True).stdout.split()]
    unit = 2.0 * 8.617333262e-5 * p.Te   # the energy part is -2 kB Te S, S = -sum ln(1 - f) - ..
    own, pad = unit * sum(left[:-1]), unit * 60 * left[-1]
    off = S - ref.parts["entropy"]
    print("entropy off by", off, "corrections of the spectrum", own, "of the padding", pad)
    assert abs(pad) > 1e-4
    assert abs(off - own) < 0.5 * abs(pad)


@pytest.mark.parametrize("n,nprob", [(128, 64), (256, 24), (256, 64), (640, 16), (1024, 3)])
@pytest.mark.parametrize("sym", [0, 1, 2])
@pytest.mark.parametrize("prec,single", [("fp16x3", False), ("fp16x3", True), ("bf16x3", False), ("tf32x3", False)])
def test_group_with_other_tiles_than_one_product(X, n, nprob, sym, prec, single):
    # one product of these sizes takes 32-wide tiles (dense 1024 64-wide), a group 64- or 128-wide ones,
    # by their waves over the SMs: a lockstep group gives the bits of its systems' own runs only if the width does not matter
    err, flag = X.binding.selftest_gemm_group(n, prec, sym, single, nprob)
    assert flag == 0 and err == 0.0

"""GPU parity of the plain-FP64 path against the oracle (through the C ABI).

Tolerances (FP64 path): charges 1e-9 e, energies 1e-8 relative, forces
1e-8 eV/A, Hamiltonian and density elements 1e-10.  Inputs are seeded
synthetic systems; the 37-atom case has a padded orbital count (148 -> 256).
"""
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


def model_params(X, **kw):
    p = X.default_params(mix_alpha=ALPHA_MIX, kernel_c=1.0 - 1.0 / ALPHA_MIX, **kw)
    return p


def oracle_model(p):
    return O.Model(Te=p.Te, n_sq=p.n_sq, rep_A=p.rep_A, rep_rho=p.rep_rho)


CASES = [
    ("tiny24", lambda: synth.make_system(24, 1705, L=7.0)),
    ("ragged37", lambda: synth.make_system(37, 11)),
    ("small8", lambda: synth.make_system(8, 42, L=7.0)),
]


def random_n(nat, seed, scale=0.02):
    rng = np.random.default_rng(seed)
    n = rng.normal(scale=scale, size=nat)
    return n - n.mean()


@pytest.mark.parametrize("name,make", CASES)
def test_build_H_and_gamma(X, name, make):
    s = make()
    p = model_params(X)
    m = oracle_model(p)
    n = random_n(s.natoms, 1)
    with X.Context(p, [sysdict(s)]) as ctx:
        ctx.set(0, X.N, n)
        ctx.build_H(0)
        H = ctx.get(0, X.H)
        G = ctx.get(0, X.GAMMA)
    Gref = O.build_gamma(s.R, s.L, m)
    Href = O.hamiltonian(O.build_H0(s.R, s.L, m), Gref, n)
    assert np.max(np.abs(G - Gref)) < 1e-10 * np.max(np.abs(Gref))
    assert np.max(np.abs(H - Href)) < 1e-11


@pytest.mark.parametrize("name,make", CASES)
def test_density_charges_forces_energy(X, name, make):
    s = make()
    p = model_params(X)
    m = oracle_model(p)
    n = random_n(s.natoms, 2)
    ref = O.evaluate(s.R, s.L, s.Z, n, m, None, with_kernel=False)
    with X.Context(p, [sysdict(s)]) as ctx:
        ctx.set(0, X.N, n)
        ctx.set(0, X.MU, [ref.dens.mu + 0.02])
        ctx.build_H(0)
        ctx.density(0)
        ctx.energy(0)
        q, D, F, mu = ctx.get(0, X.Q), ctx.get(0, X.D), ctx.get(0, X.F), ctx.get(0, X.MU)[0]
        E = ctx.get(0, X.ENERGY)
    assert abs(mu - ref.dens.mu) < 1e-9
    assert np.max(np.abs(D - ref.dens.D)) < 1e-10
    assert np.max(np.abs(q - ref.q)) < 1e-9
    assert np.max(np.abs(F - ref.F)) < 1e-8
    parts = ref.parts
    assert E[1] == pytest.approx(parts["band"], rel=1e-10, abs=1e-9)
    assert E[2] == pytest.approx(parts["coulomb"], rel=1e-9, abs=1e-9)
    assert E[3] == pytest.approx(parts["entropy"], rel=1e-7, abs=1e-8)
    assert E[0] == pytest.approx(ref.Omega, rel=1e-8)


@pytest.mark.parametrize("name,make", CASES[:2])
def test_response_and_kernel(X, name, make):
    import torch
    s = make()
    p = model_params(X, rank_m=4)
    m = oracle_model(p)
    n = random_n(s.natoms, 3)
    xl = O.XLParams(rank_m=4, kernel_c=p.kernel_c)
    ref = O.evaluate(s.R, s.L, s.Z, n, m, xl)
    rng = np.random.default_rng(4)
    v = rng.normal(size=s.natoms)
    v -= v.mean()
    v /= np.linalg.norm(v)
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
        ctx.kernel_update(0)
        Kr = ctx.get(0, X.KR)
        probes = ctx.get(0, X.PROBES)
    assert np.max(np.abs(w - wref)) < 1e-8 * max(1.0, np.max(np.abs(wref)))
    assert np.max(np.abs(Kr - ref.Kr)) < 1e-9
    Vref = np.array(ref.V)
    assert np.max(np.abs(probes[0][:len(Vref)] - Vref)) < 1e-8


def test_scf_ground_state(X):
    s = synth.make_system(24, 1705, L=7.0)
    p = model_params(X)
    m = oracle_model(p)
    n_ref, _ = O.scf(s.R, s.L, s.Z, m, ALPHA_MIX, tol=p.scf_tol)
    with X.Context(p, [sysdict(s)]) as ctx:
        ctx.scf(0)
        n = ctx.get(0, X.N)
        hist = ctx.get(0, X.NHIST)
    assert np.max(np.abs(n - n_ref)) < 1e-9
    assert np.allclose(hist, hist[0][None, :])


@pytest.mark.parametrize("rank", [2, 4])
def test_kernel_scf_ground_state(X, rank):
    # Eq. SCF_K with the rank-m kernel and a fixed c, against the oracle's kernel SCF
    s = synth.make_system(24, 1705, L=7.0)
    p = model_params(X, scf_mode=1, rank_m=rank)
    m = oracle_model(p)
    n_ref, it = O.scf_kernel(s.R, s.L, s.Z, m, rank, p.kernel_c, tol=p.scf_tol)
    with X.Context(p, [sysdict(s)]) as ctx:
        ctx.scf(0)
        n = ctx.get(0, X.N)
    assert np.max(np.abs(n - n_ref)) < 1e-9, it


def test_trajectory_matches_oracle(X):
    s = synth.make_system(24, 1705, L=7.0)
    p = model_params(X)
    m = oracle_model(p)
    xl = O.XLParams(rank_m=p.rank_m, kernel_c=p.kernel_c, mix_alpha=ALPHA_MIX)
    st, ev = O.md_init(s.R, s.V, s.L, s.Z, s.mass, m, xl)
    with X.Context(p, [sysdict(s)]) as ctx:
        ctx.set(0, X.N, st.nhist[0])
        ctx.set(0, X.MU, [ev.dens.mu])
        ctx.build_H(0)
        ctx.density(0)
        ctx.kernel_update(0)
        assert np.max(np.abs(ctx.get(0, X.KR) - st.Kr)) < 1e-9
        for k in range(50):
            st, ev = O.md_step(st, s.L, s.Z, s.mass, m, xl)
            ctx.step(1)
            ctx.energy(0)
            R = ctx.get(0, X.R)
            dR = O.min_image(R - st.R, s.L)
            assert np.max(np.abs(dR)) < 1e-9, k
            assert np.max(np.abs(ctx.get(0, X.Q) - ev.q)) < 1e-9, k
            assert np.max(np.abs(ctx.get(0, X.N) - st.nhist[0])) < 1e-9, k
            E = ctx.get(0, X.ENERGY)
            assert E[0] == pytest.approx(ev.Omega, rel=1e-8), k


@pytest.mark.parametrize("prec,tol_q", [("fp64", 1e-9), ("fp16x3", 1e-5), ("bf16x3", 3e-5)])
def test_mu_search_through_flat_occupation(X, prec, tol_q):
    # (BF16x3 is held to its measured level, 3e-5 e, outside the 1e-5 e bound of FP16x3)
    # 33 atoms at n = 0, Te = 1000 K, 12 squarings: from the first guess (the
    # middle of the Gershgorin interval) the safeguarded Newton search bisects
    # to a mu above every level, where Tr D = N and dTr D/dmu = 0; it must
    # keep bisecting to Tr D = N_occ rather than accept the zero step
    s = synth.make_system(33, 1715)
    p = model_params(X, Te=1000.0, n_sq=12, prec=prec, mu_tol=1e-9 if prec == "fp64" else 1e-3)
    ref = O.evaluate(s.R, s.L, s.Z, np.zeros(s.natoms), O.Model(Te=1000.0, n_sq=12), None, with_kernel=False)
    with X.Context(p, [sysdict(s)]) as ctx:
        ctx.build_H(0)
        ctx.density(0)
        q = ctx.get(0, X.Q)
    print(prec, "dq", np.abs(q - ref.q).max())
    assert abs(q.sum() - ref.q.sum()) < s.natoms * tol_q
    assert np.max(np.abs(q - ref.q)) < tol_q


def test_pair_repulsion_matches_oracle(X):
    s = synth.make_system(24, 1705, L=7.0)
    p = model_params(X, rep_A=40.0, rep_rho=0.3)
    m = oracle_model(p)
    n = random_n(s.natoms, 12)
    ref = O.evaluate(s.R, s.L, s.Z, n, m, None, with_kernel=False)
    with X.Context(p, [sysdict(s)]) as ctx:
        ctx.set(0, X.N, n)
        ctx.set(0, X.MU, [ref.dens.mu])
        ctx.build_H(0)
        ctx.density(0)
        ctx.energy(0)
        F, E = ctx.get(0, X.F), ctx.get(0, X.ENERGY)
    assert ref.parts["repulsion"] > 0.0
    assert E[6] == pytest.approx(ref.parts["repulsion"], rel=1e-12, abs=1e-12)
    assert E[0] == pytest.approx(ref.Omega, rel=1e-8)
    assert np.max(np.abs(F - ref.F)) < 1e-8


def test_single_atom_edge_case(X):
    p = model_params(X)
    s = dict(natoms=1, L=7.0, R=np.array([[1.0, 2.0, 3.0]]), V=np.zeros((1, 3)), Z=np.array([4.0]), mass=12.0)
    with X.Context(p, [s]) as ctx:
        ctx.build_H(0)
        ctx.density(0)
        q = ctx.get(0, X.Q)
        F = ctx.get(0, X.F)
    assert abs(q[0]) < 1e-12
    assert np.max(np.abs(F)) < 1e-12


def test_argument_errors_are_reported(X):
    p = model_params(X)
    s = synth.make_system(8, 42, L=7.0)
    bad = sysdict(s)
    bad["L"] = 4.0           # box not larger than the hopping cutoff
    with pytest.raises(X.XlbomdError) as e:
        X.Context(p, [bad])
    assert e.value.status == -1
    with X.Context(p, [sysdict(s)]) as ctx:
        with pytest.raises(X.XlbomdError) as e:
            ctx.kernel_update(0)     # no density yet
        assert e.value.status == -1
        with pytest.raises(X.XlbomdError):
            ctx.build_H(0)           # sticky until cleared
        ctx._lib.xlbomd_clear_error(ctx.h)
        ctx.build_H(0)


@pytest.mark.parametrize("name,make", CASES[:2])
def test_exact_kernel_matches_oracle(X, name, make):
    # Eq. KK: K = (J - I)^-1 with J from the natoms unit-direction responses
    s = make()
    p = model_params(X, kernel_mode=1)
    m = oracle_model(p)
    n = random_n(s.natoms, 6)
    ev = O.evaluate(s.R, s.L, s.Z, n, m, None, with_kernel=False, with_forces=False)
    Kref = O.kernel_exact(ev.dens, ev.gamma)
    with X.Context(p, [sysdict(s)]) as ctx:
        ctx.set(0, X.N, n)
        ctx.set(0, X.MU, [ev.dens.mu])
        ctx.build_H(0)
        ctx.density(0)
        ctx.kernel_update(0)           # computes the held kernel, then K r
        K = ctx.get(0, X.KMAT)
        Kr = ctx.get(0, X.KR)
        assert ctx.get(0, X.STATS)[2] == s.natoms
    assert np.max(np.abs(K - Kref)) < 1e-9 * max(1.0, np.abs(Kref).max())
    assert np.max(np.abs(Kr - Kref @ ev.r)) < 1e-10


@pytest.mark.parametrize("variant", ["exact_every5", "accumulated", "delta", "kmax6", "kmax7", "repulsion"])
def test_kernel_and_dissipation_variants_follow_oracle(X, variant):
    # the exact kernel held and recomputed every 5 steps (Section VI.A), the
    # accumulated rank-1 kernel (end of Section V.F), K = K_0 only (rank 0), and
    # the K_max = 6, 7 rows of Table I (the library's table against the
    # oracle's, typed independently)
    s = synth.make_system(24, 1705, L=7.0)
    kw, xlkw = {}, {}
    if variant == "exact_every5":
        kw, xlkw = dict(kernel_mode=1, kernel_every=5), dict(kernel_mode="exact", kernel_every=5)
    elif variant == "accumulated":
        kw, xlkw = dict(kernel_mode=2), dict(kernel_mode="accumulated")
    elif variant == "repulsion":
        kw = dict(rep_A=40.0, rep_rho=0.3)
    elif variant == "delta":
        kw, xlkw = dict(rank_m=0), dict(rank_m=0)
    else:
        kmax = int(variant[-1])
        kappa, alpha, c = O.TABLE_I[kmax]
        kw, xlkw = dict(kmax=kmax), dict(kappa=kappa, alpha=alpha, c=tuple(float(x) for x in c))
    p = model_params(X, **kw)
    m = oracle_model(p)
    base = dict(rank_m=p.rank_m, kernel_c=p.kernel_c, mix_alpha=ALPHA_MIX)
    base.update(xlkw)
    xl = O.XLParams(**base)
    assert p.kmax == xl.kmax and abs(p.kappa - xl.kappa) < 1e-15 and abs(p.alpha - xl.alpha) < 1e-15
    assert all(abs(p.c[k] - xl.c[k]) < 1e-15 for k in range(xl.kmax + 1))
    st, ev = O.md_init(s.R, s.V, s.L, s.Z, s.mass, m, xl)
    with X.Context(p, [sysdict(s)]) as ctx:
        ctx.set(0, X.N, st.nhist[0])
        ctx.set(0, X.MU, [ev.dens.mu])
        ctx.build_H(0)
        ctx.density(0)
        ctx.kernel_update(0)
        assert np.max(np.abs(ctx.get(0, X.KR) - st.Kr)) < 1e-9
        for k in range(12):
            st, ev = O.md_step(st, s.L, s.Z, s.mass, m, xl)
            ctx.step(1)
            assert np.max(np.abs(O.min_image(ctx.get(0, X.R) - st.R, s.L))) < 1e-9, k
            assert np.max(np.abs(ctx.get(0, X.Q) - ev.q)) < 1e-9, k
            assert np.max(np.abs(ctx.get(0, X.N) - st.nhist[0])) < 1e-9, k
            assert np.max(np.abs(ctx.get(0, X.KR) - ev.Kr)) < 1e-9, k


def test_residual_and_energy_fluctuations_scale_as_dt_squared_on_gpu(X):
    # Section VI.C, Figs. 9-10, through the C ABI: over the same 10 fs from the t0 ground state,
    # halving dt divides the RMS residual |q[n] - n| and the total-energy fluctuation by about 4
    s = synth.make_system(24, 1705, L=7.0)
    res, fluct = [], []
    for dt in (0.5, 0.25, 0.125):
        p = model_params(X, dt=dt, rank_m=2)
        with X.Context(p, [sysdict(s)]) as ctx:
            ctx.scf(0)
            r, E = [], []
            for _ in range(int(round(10.0 / dt))):
                ctx.step(1)
                ctx.energy(0)
                r.append(np.sqrt(np.mean(ctx.get(0, X.RES) ** 2)))
                E.append(ctx.get(0, X.ENERGY)[5])
        assert np.max(np.abs(np.asarray(E) - E[0])) < 1e-3, dt
        res.append(np.mean(r))
        fluct.append(np.std(E))
    print("dt study: residual RMS", res, "energy std", fluct)
    for a, b in ((res[0], res[1]), (res[1], res[2]), (fluct[0], fluct[1]), (fluct[1], fluct[2])):
        assert 3.0 < a / b < 5.5, (res, fluct)


@pytest.mark.parametrize("nat", [33, 65, 97, 129])
def test_density_and_entropy_at_tile_edges(X, nat):
    # padded orbital counts 256, 384, 512 and 640: products with 8, 16 and 32 wide tiles, symmetric and
    # dense, and the batched log-determinants of the energy (4 to 10 panels of 64)
    s = synth.make_system(nat, 23)
    p = model_params(X)
    m = oracle_model(p)
    n = random_n(s.natoms, nat, scale=0.01)
    ref = O.evaluate(s.R, s.L, s.Z, n, m, O.XLParams(rank_m=p.rank_m, kernel_c=p.kernel_c))
    with X.Context(p, [sysdict(s)]) as ctx:
        ctx.set(0, X.N, n)
        ctx.set(0, X.MU, [ref.dens.mu + 0.01])
        ctx.build_H(0)
        ctx.density(0)
        ctx.kernel_update(0)
        ctx.energy(0)
        q, F, Kr, E = ctx.get(0, X.Q), ctx.get(0, X.F), ctx.get(0, X.KR), ctx.get(0, X.ENERGY)
    assert np.max(np.abs(q - ref.q)) < 1e-9
    assert np.max(np.abs(F - ref.F)) < 1e-8
    assert np.max(np.abs(Kr - ref.Kr)) < 1e-8
    assert abs(E[0] - ref.Omega) < 1e-8 * abs(ref.Omega)
    assert abs(E[3] - ref.parts["entropy"]) < 1e-7


@pytest.mark.parametrize("nat,rank,prec", [(5, 1, "fp64"), (9, 8, "fp64"), (33, 3, "fp64"), (65, 7, "fp64"),
                                           (257, 5, "fp16x3")])
def test_rank_m_update_algebra(X, nat, rank, prec):
    # the FP64 vector algebra of the update from the probes V and responses W it reports itself: one or
    # several warps per sum, one and several rounds of sums, 256 and 512 threads.  Orthonormality to a few
    # hundred roundings; K r through S of condition below 1e3; a candidate loses what the projection cancels
    s = synth.make_system(nat, 31, **({} if nat > 24 else {"L": 7.0}))
    p = model_params(X, rank_m=rank, prec=prec)
    with X.Context(p, [sysdict(s)]) as ctx:
        ctx.set(0, X.N, random_n(nat, 7))
        ctx.build_H(0)
        ctx.density(0)
        ctx.kernel_update(0)
        r, Kr, (V, W) = ctx.get(0, X.RES), ctx.get(0, X.KR), ctx.get(0, X.PROBES)
        used = int(ctx.get(0, X.STATS)[2])
    assert 1 <= used <= rank
    V, W = V[:used], W[:used]
    assert np.max(np.abs(V @ V.T - np.eye(used))) < 1e-13
    ref = O.apply_kernel(r, V, W, p.kernel_c)
    assert np.max(np.abs(Kr - ref)) < 1e-11 * np.max(np.abs(ref))
    for i in range(used):
        x = O.apply_kernel(r, V[:i], W[:i], p.kernel_c)
        left = x - V[:i].T @ (V[:i] @ x)
        left -= V[:i].T @ (V[:i] @ left)
        ratio = np.linalg.norm(left) / np.linalg.norm(x)
        assert np.max(np.abs(V[i] - left / np.linalg.norm(left))) < 1e-12 / ratio


@pytest.mark.parametrize("nat", [2, 5, 9, 64, 65])
def test_exact_kernel_inverse_at_cluster_edges(X, nat):
    # columns dealt to the 8 CTAs of the inverting cluster: fewer than CTAs, one more than a multiple, more
    # than one column per CTA
    s = synth.make_system(nat, 12, **({} if nat > 24 else {"L": 7.0}))
    p = model_params(X, kernel_mode=1)
    n = random_n(nat, 16)
    ev = O.evaluate(s.R, s.L, s.Z, n, oracle_model(p), None, with_kernel=False, with_forces=False)
    Kref = O.kernel_exact(ev.dens, ev.gamma)
    with X.Context(p, [sysdict(s)]) as ctx:
        ctx.set(0, X.N, n)
        ctx.set(0, X.MU, [ev.dens.mu])
        ctx.build_H(0)
        ctx.density(0)
        ctx.kernel_exact(0)
        K = ctx.get(0, X.KMAT)
    assert np.max(np.abs(K - Kref)) < 1e-9 * max(1.0, np.abs(Kref).max())


@pytest.mark.parametrize("nat", [200, 460])
def test_exact_kernel_inverts_the_response(X, nat):
    # K (w - v) = v with w the response along v; 460 atoms are beyond the shared memory of a cluster.  The
    # FP16x3 responses are good to 1e-5 (w and the columns of J alike), K here has a condition below 100
    import torch
    s = synth.make_system(nat, 13)
    p = model_params(X, kernel_mode=1, prec="fp16x3")
    v = random_n(nat, 17)
    with X.Context(p, [sysdict(s)]) as ctx:
        ctx.set(0, X.N, random_n(nat, 18))
        ctx.build_H(0)
        ctx.density(0)
        vd = torch.tensor(v, dtype=torch.float64, device="cuda")
        wd = torch.zeros_like(vd)
        ctx.response(0, vd.data_ptr(), wd.data_ptr())
        torch.cuda.synchronize()
        ctx.kernel_exact(0)
        K = ctx.get(0, X.KMAT)
    assert np.linalg.norm(K @ (wd.cpu().numpy() - v) - v) < 1e-3 * np.linalg.norm(v)


@pytest.mark.parametrize("prec", ["fp64", "fp16x3"])
@pytest.mark.parametrize("coulomb_k", [14.399645, 0.0])
def test_non_finite_positions_are_reported(X, prec, coulomb_k):
    # also without the Coulomb term, whose gamma would carry a NaN into H by itself: the pair search must not lose it
    s = synth.make_system(24, 1705, L=7.0)
    p = model_params(X, prec=prec, coulomb_k=coulomb_k, mu_tol=1e-9 if prec == "fp64" else 1e-3)
    for bad in (np.nan, np.inf):
        R = s.R.copy()
        R[5, 1] = bad
        with X.Context(p, [sysdict(s)]) as ctx:
            ctx.set(0, X.R, R)
            ctx.build_H(0)
            assert np.isnan(ctx.get(0, X.H)).any()
            with pytest.raises(X.XlbomdError) as e:
                ctx.density(0)
            assert e.value.status == -5


@pytest.mark.parametrize("prec", ["fp64", "fp16x3"])
def test_forces_after_a_non_finite_move_are_not_finite(X, prec):
    # positions moved without a new Hamiltonian: D stays that of the old H, the atom's own forces cannot be finite
    s = synth.make_system(24, 1705, L=7.0)
    p = model_params(X, prec=prec, coulomb_k=0.0, rep_A=40.0, mu_tol=1e-9 if prec == "fp64" else 1e-3)
    R = s.R.copy()
    R[5, 1] = np.nan
    with X.Context(p, [sysdict(s)]) as ctx:
        ctx.build_H(0)
        ctx.set(0, X.R, R)
        ctx.density(0)
        assert not np.isfinite(ctx.get(0, X.F)[5]).any()
        ctx.energy(0)
        assert np.isnan(ctx.get(0, X.ENERGY)[6])


@pytest.mark.parametrize("prec", ["fp64", "fp16x3"])
def test_energy_work_area_is_shared_by_the_systems(X, prec):
    # eight systems of 512 padded orbitals: the first energy makes the work area, the others use it.  A context
    # of uneven sizes gives each system the energies of its own context
    import torch
    systems = [sysdict(synth.make_system(100 + i, 40 + i)) for i in range(8)]
    p = model_params(X, prec=prec, mu_tol=1e-9 if prec == "fp64" else 1e-3)
    with X.Context(p, systems) as ctx:
        free = []
        for i in range(8):
            ctx.build_H(i)
            ctx.density(i)
            ctx.energy(i)
            torch.cuda.synchronize()
            free.append(torch.cuda.mem_get_info()[0])
    assert len(set(free)) == 1, free
    mixed = [sysdict(synth.make_system(nat, 60 + nat)) for nat in (40, 24, 100, 33)]
    own = []
    for s in mixed:
        with X.Context(p, [s]) as ctx:
            ctx.density(0)
            ctx.energy(0)
            own.append(ctx.get(0, X.ENERGY))
    with X.Context(p, mixed) as ctx:
        for i in range(len(mixed)):
            ctx.density(i)
            ctx.energy(i)
            assert np.array_equal(ctx.get(i, X.ENERGY), own[i]), i


def test_energy_with_little_free_memory(X):
    # FP64, 1024 padded orbitals: the work area for all levels takes 100 MB, for one 9 MB.  With 60, 20 and 4 MB
    # free the log-determinants run in smaller batches, the last on the engine's own matrices
    import torch
    s = sysdict(synth.make_system(230, 9))
    p = model_params(X, rank_m=0)
    E = []
    for left in (None, 60 << 20, 20 << 20, 4 << 20):
        with X.Context(p, [s]) as ctx:
            ctx.density(0)
            held = None
            if left is not None:
                torch.cuda.synchronize()
                torch.cuda.empty_cache()
                held = torch.empty(torch.cuda.mem_get_info()[0] - left, dtype=torch.uint8, device="cuda")
            try:
                ctx.energy(0)
                E.append(ctx.get(0, X.ENERGY))
            finally:
                del held
                torch.cuda.empty_cache()
    for e in E[1:]:
        assert np.max(np.abs(e - E[0])) < 1e-10 * np.max(np.abs(E[0]))


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-9), ("fp16x3", 1e-5)])
def test_restart_from_host_copies_continues_the_trajectory(X, prec, tol):
    # the first half kick takes F(t) and the first n update K r(t): with both set beside R, V, the history and
    # mu a second context goes on where the first one stands.  Its search for mu starts without a
    # history, so charges agree to the precision of a density (1e-9 e, FP16x3 1e-5 e) and not to the bit
    s = synth.make_system(24, 1705, L=7.0)
    p = model_params(X, prec=prec, mu_tol=1e-9 if prec == "fp64" else 1e-3, rep_A=40.0)
    what = (X.R, X.V, X.NHIST, X.F, X.KR, X.MU)
    with X.Context(p, [sysdict(s)]) as a, X.Context(p, [sysdict(s)]) as b:
        a.set(0, X.N, random_n(s.natoms, 5, scale=0.01))
        a.build_H(0)
        a.density(0)
        a.kernel_update(0)
        a.step(2)
        kept = {w: a.get(0, w) for w in what}
        a.step(1)
        b.build_H(0)
        b.density(0)
        b.kernel_update(0)
        for w in what:
            b.set(0, w, kept[w])
        b.step(1)
        for w in (X.R, X.NHIST):   # functions of what was set alone
            assert np.array_equal(a.get(0, w), b.get(0, w))
        assert np.max(np.abs(a.get(0, X.Q) - b.get(0, X.Q))) < tol
        assert np.max(np.abs(a.get(0, X.F) - b.get(0, X.F))) < 10 * tol
        assert np.max(np.abs(a.get(0, X.V) - b.get(0, X.V))) < 1e-3 * tol   # half a kick: 1e-4 A/fs per eV/A


@pytest.mark.parametrize("prec,nsys,steps", [("fp64", 1, 1), ("fp16x3", 1, 3), ("fp16x3", 3, 2)])
def test_calls_from_one_state_repeat(X, prec, nsys, steps):
    # near the exact kernel K r = n - n*, so a step that takes the K r of the call before multiplies the deviation
    # by -kappa; from a state set whole every call gives the same bits, however many there are
    p = model_params(X, prec=prec, mu_tol=1e-9 if prec == "fp64" else 1e-3, rep_A=40.0)
    systems = [sysdict(synth.make_system(24 - i, 1705 + i)) for i in range(nsys)]
    what = (X.R, X.V, X.NHIST, X.F, X.KR, X.MU)
    with X.Context(p, systems) as ctx:
        state = []
        for i in range(nsys):
            ctx.set(i, X.N, random_n(systems[i]["natoms"], 6 + i, scale=0.01))
            ctx.build_H(i)
            ctx.density(i)
            ctx.kernel_update(i)
            state.append({w: ctx.get(i, w) for w in what})
        first = None
        for call in range(40):
            for i in range(nsys):
                for w in what:
                    ctx.set(i, w, state[i][w])
            ctx.step(steps)
            got = [ctx.get(i, w) for i in range(nsys) for w in what + (X.Q,)]
            first = first or got
            assert all(np.array_equal(a, b) for a, b in zip(first, got)), call


@pytest.mark.parametrize("prec,tol_f", [("fp64", 1e-8), ("fp16x3", 1e-4)])
@pytest.mark.parametrize("nat", [24, 300])
def test_forces_follow_moved_positions(X, prec, tol_f, nat):
    # atoms moved by set(R) without a new Hamiltonian: D, q and n stay those of the old one, every force term is
    # taken at the new R.  A uniform shift cannot tell (the Coulomb terms do not change under it); here the
    # displacements differ, and Coulomb forces of the old R would miss by hundreds of tolerances
    s = synth.make_system(nat, 29, **({"L": 7.0} if nat == 24 else {}))
    p = model_params(X, prec=prec, rep_A=40.0, mu_tol=1e-9 if prec == "fp64" else 1e-3)
    m = oracle_model(p)
    n = random_n(nat, 30, scale=0.3)
    ref = O.evaluate(s.R, s.L, s.Z, n, m, None, with_kernel=False, with_forces=False)
    R2 = s.R + np.random.default_rng(31).normal(scale=0.05, size=(nat, 3))
    want = O.forces(R2, s.L, m, ref.dens.D, ref.q, n)
    bare = O.Model(Te=p.Te, n_sq=p.n_sq, rep_A=p.rep_A, rep_rho=p.rep_rho, coulomb_k=0.0)
    coul = lambda R, F: F - O.forces(R, s.L, bare, ref.dens.D, ref.q, n, np.zeros((nat, nat, 3)))
    stale = want - coul(R2, want) + coul(s.R, O.forces(s.R, s.L, m, ref.dens.D, ref.q, n))
    assert np.max(np.abs(stale - want)) > 100 * tol_f
    with X.Context(p, [sysdict(s)]) as ctx:
        ctx.set(0, X.N, n)
        ctx.set(0, X.MU, [ref.dens.mu])
        ctx.build_H(0)
        ctx.set(0, X.R, R2)
        ctx.density(0)
        F = ctx.get(0, X.F)
        ctx.density(0)   # and again, from what the first call left
        F2 = ctx.get(0, X.F)
    assert np.max(np.abs(F - want)) < tol_f
    assert np.max(np.abs(F2 - want)) < tol_f


def test_exact_kernel_beyond_the_cluster(X):
    # 470 atoms: the inverse by launches (up to 463 fit the shared memory of a cluster).  K (w - v) = v as above
    import torch
    nat = 470
    s = synth.make_system(nat, 13)
    p = model_params(X, kernel_mode=1, prec="fp16x3", kernel_prec=1)
    v = random_n(nat, 17)
    with X.Context(p, [sysdict(s)]) as ctx:
        ctx.set(0, X.N, random_n(nat, 18))
        ctx.build_H(0)
        ctx.density(0)
        before = X.binding.launch_count()
        ctx.kernel_exact(0)
        assert X.binding.launch_count() - before > 2 * nat   # a search and an elimination per step
        K = ctx.get(0, X.KMAT)
        vd = torch.tensor(v, dtype=torch.float64, device="cuda")
        wd = torch.zeros_like(vd)
        ctx.response(0, vd.data_ptr(), wd.data_ptr())
        torch.cuda.synchronize()
    # single products: the responses, and so J and w, are good to a few 2^-11
    assert np.linalg.norm(K @ (wd.cpu().numpy() - v) - v) < 1e-1 * np.linalg.norm(v)

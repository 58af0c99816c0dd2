"""Second propagation round: period averages <A>_T of Floquet states (Eq. 17) through the C ABI,
against the oracle on the same states, and the Floquet Hellmann-Feynman relation
d eps / d f_dc = <H1>_T measured entirely on the GPU path."""
import math

import numpy as np
import pytest

import floquet_inputs as fi
import oracle as o

pytestmark = pytest.mark.gpu
U32 = 2.0 ** -24


@pytest.fixture(scope="module")
def fq():
    import torch
    assert torch.cuda.is_available()
    import paper_1508_07621_gb300 as fq
    return fq


@pytest.mark.parametrize("precision", ["FQ_FP64", "FQ_DF32", "FQ_OZAKI"])
def test_dense_fp64_averages_match_oracle(fq, precision):
    """Period averages through the FP64 chain and the two emulated ones (same FP64 criterion)."""
    n, M = 40, 60
    h0, h1 = fi.goe(n, 1401), fi.goe(n, 1402)
    drv = fi.Drive(0.1, 1.1, 1.2, 0.3)
    plan = fq.Plan.dense(h0, h1, omega=drv.omega, f_ac=drv.f_ac, f_dc=drv.f_dc, phi0=drv.phi0, steps=M,
                         precision=getattr(fq, precision))
    eps, states = fq.floquet_states(plan.build_UT(), drv.period)
    e_avg = plan.average_observable(states, 1.0, 0.0, 1.0).cpu().numpy()       # <H(t)>_T
    h1_avg = plan.average_observable(states, 0.0, 1.0, 0.0).cpu().numpy()      # <H1>_T
    p = o.plan_for_drive_dense(h0, h1, drv, M)
    k = o.commutator_dense(h0, h1)
    step = lambda m, x: o.chebyshev_step(lambda v: o.omega_tilde_dense(h0, h1, k, p, m) @ v, x, p.coeffs, p.phase)
    x0 = states.cpu().numpy().T
    ref_e = o.average_observable(step, o.expect_dense(h0, h1, 1.0, 0.0, 1.0, drv), x0, drv, M)
    ref_h1 = o.average_observable(step, o.expect_dense(h0, h1, 0.0, 1.0, 0.0, drv), x0, drv, M)
    assert np.max(np.abs(e_avg - ref_e)) <= 1e-10
    assert np.max(np.abs(h1_avg - ref_h1)) <= 1e-10


def test_hellmann_feynman_on_gpu(fq):
    """All on the library: U_T at f_dc +- d (FP64 dense), quasienergy slopes vs <H1>_T."""
    n, M = 24, 80
    h0, h1 = fi.goe(n, 1501), fi.goe(n, 1502)

    def run(fdc):
        plan = fq.Plan.dense(h0, h1, omega=1.3, f_ac=0.9, f_dc=fdc, steps=M)
        eps, st = fq.floquet_states(plan.build_UT(), 2 * math.pi / 1.3)
        return plan, eps, st

    fdc, d = 0.2, 1e-4
    plan, eps, states = run(fdc)
    _, ep, _ = run(fdc + d)
    _, em, _ = run(fdc - d)
    near = lambda e0, e1: np.array([e1[np.argmin(np.abs(np.angle(np.exp(1j * (e1 - x) * 2 * math.pi / 1.3))))]
                                    for x in e0])
    slope = (near(eps, ep) - near(eps, em)) / (2 * d)
    h1_avg = plan.average_observable(states, 0.0, 1.0, 0.0).cpu().numpy()
    assert np.max(np.abs(slope - h1_avg)) < 1e-6


@pytest.mark.parametrize("precision,kernel", [(0, 1), (1, 2)])
def test_dimer_average_energy(fq, precision, kernel):
    """Dimer (dim 41, M = 100): <H(t)>_T of its Floquet states (the paper's sorting key, §7), FP64
    streaming and FP32 resident, against the oracle.  A state error e moves <H> by at most
    2 ||H|| e, so the FP32 tolerance is 2 ||H|| min(1e-5, the FP32 rounding bound of the states)."""
    d = fi.config_dimer(nb=40, steps=100)
    plan = fq.Plan.tridiag(d.h0_diag, d.h0_off, d.h1_diag, omega=3.0, f_ac=1.5, steps=d.steps,
                           precision=precision, kernel=kernel)
    ref_plan = fq.Plan.tridiag(d.h0_diag, d.h0_off, d.h1_diag, omega=3.0, f_ac=1.5, steps=d.steps, precision=0,
                               kernel=1)
    eps, states = fq.floquet_states(ref_plan.build_UT(), d.drive.period)
    avg = plan.average_observable(states, 1.0, 0.0, 1.0).cpu().numpy()
    p = o.plan_for_drive_tridiag(d.h0_diag, d.h0_off, d.h1_diag, d.drive, d.steps)
    kl = o.commutator_tridiag(d.h0_off, d.h1_diag)

    def step(m, x):
        dd, lo = o.omega_tilde_tridiag(d.h0_diag, d.h0_off, d.h1_diag, kl, p, m)
        return o.chebyshev_step(lambda v: o.apply_tridiag(dd, lo, v), x, p.coeffs, p.phase)

    ref = o.average_observable(step, o.expect_tridiag(d.h0_diag, d.h0_off, d.h1_diag, 1.0, 0.0, 1.0, d.drive),
                               states.cpu().numpy().T, d.drive, d.steps)
    if precision == 0:
        tol = 1e-9
    else:
        hn = max(abs(plan.info.e_min), abs(plan.info.e_max))
        tol = 2 * hn * min(1e-5, 2 * d.steps * plan.info.R * U32 + 4 * math.sqrt(d.steps) * plan.info.L * U32)
    assert np.max(np.abs(avg - ref)) <= tol
    order = np.argsort(avg)      # the paper sorts Floquet states by mean energy
    assert len(set(order.tolist())) == d.n


def test_floquet_analysis_sorted_by_average_energy(fq):
    """floquet_analysis: U_T, Floquet states, <H(t)>_T by the second round, sorted ascending;
    energies match the oracle's averages of the same states and the order is by energy."""
    n, M = 32, 50
    h0, h1 = fi.goe(n, 1801), fi.goe(n, 1802)
    drv = fi.Drive(0.3, 1.0, 1.4, 0.2)
    plan = fq.Plan.dense(h0, h1, omega=drv.omega, f_ac=drv.f_ac, f_dc=drv.f_dc, phi0=drv.phi0, steps=M)
    avg, eps, states = fq.floquet_analysis(plan)
    assert np.all(np.diff(avg) >= 0)
    p = o.plan_for_drive_dense(h0, h1, drv, M)
    k = o.commutator_dense(h0, h1)
    step = lambda m, x: o.chebyshev_step(lambda v: o.omega_tilde_dense(h0, h1, k, p, m) @ v, x, p.coeffs, p.phase)
    ref = o.average_observable(step, o.expect_dense(h0, h1, 1.0, 0.0, 1.0, drv), states.cpu().numpy().T, drv, M)
    assert np.max(np.abs(avg - ref)) <= 1e-10
    # each row is a Floquet state: U_T phi = e^{-i eps T} phi
    U = plan.build_UT().cpu().numpy()
    phi = states.cpu().numpy()
    res = U @ phi.T - phi.T * np.exp(-1j * eps * drv.period)[None, :]
    assert np.max(np.abs(res)) < 1e-9


def _random_states(n, nc, seed):
    import torch
    x = np.exp(2j * np.pi * fi.uniform(seed, n * nc)).reshape(nc, n) * (0.1 + fi.uniform(seed + 1, n * nc).reshape(nc, n))
    x /= np.linalg.norm(x, axis=1, keepdims=True)
    return torch.from_numpy(x).cuda()


@pytest.mark.parametrize("n,nc", [(1, 1), (2, 5), (31, 4), (32, 9), (33, 3), (64, 1), (65, 65), (100, 30), (161, 2)])
def test_dense_averages_block_edges(fq, n, nc):
    """Sizes around the 32-row blocks of H and the 4 states of a CTA, with an odd (trapezoid) and an
    even number of steps, H0, H1 and the drive all weighted; FP64 against the oracle."""
    h0, h1 = fi.goe(n, 1821), fi.goe(n, 1822)
    drv = fi.Drive(0.3, 1.0, 1.4, 0.2)
    states = _random_states(n, nc, 1823)
    k = o.commutator_dense(h0, h1)
    for M in (7, 10):
        plan = fq.Plan.dense(h0, h1, omega=drv.omega, f_ac=drv.f_ac, f_dc=drv.f_dc, phi0=drv.phi0, steps=M)
        avg = plan.average_observable(states, 0.7, -0.4, 1.3).cpu().numpy()
        assert plan.check_status() == fq.FQ_OK
        p = o.plan_for_drive_dense(h0, h1, drv, M)
        step = lambda m, x: o.chebyshev_step(lambda v: o.omega_tilde_dense(h0, h1, k, p, m) @ v, x, p.coeffs, p.phase)
        ref = o.average_observable(step, o.expect_dense(h0, h1, 0.7, -0.4, 1.3, drv), states.cpu().numpy().T, drv, M)
        assert np.max(np.abs(avg - ref)) <= 1e-12


@pytest.mark.parametrize("n", [1, 33, 100, 128])
def test_dense_averages_few_and_many_states(fq, n):
    """A formed inside the expectation kernel (few states) and by a launch of its own (more CTAs than SMs): the
    same bits for every state."""
    import torch
    plan = fq.Plan.dense(fi.goe(n, 1824), fi.goe(n, 1825), omega=1.4, f_ac=1.0, f_dc=0.3, phi0=0.2, steps=5)
    x = _random_states(n, 5, 1826)
    few = plan.average_observable(x, 0.7, -0.4, 1.3)
    many = plan.average_observable(x.repeat(130, 1).contiguous(), 0.7, -0.4, 1.3)
    assert plan.check_status() == fq.FQ_OK
    assert torch.equal(many, few.repeat(130))


@pytest.mark.parametrize("precision,kernel", [(0, 1), (0, 3), (1, 2), (1, 3), (4, 3), (5, 4)])
@pytest.mark.parametrize("nb,nc", [(1, 1), (2, 5), (60, 61), (511, 3), (512, 6), (1100, 2)])
def test_tridiagonal_averages_by_path(fq, precision, kernel, nb, nc):
    """Averages on every tridiagonal kernel (those with gauge tables take all steps' tables from one
    launch, each step then entering and leaving the original frame), around the 512-row chunks of H and
    the 4 states of a CTA: against the averages of the same plan's own propagation, step by step, in
    FP64 on the host."""
    d = fi.config_dimer(nb=nb)
    n, M = d.n, 5
    h = 2 * math.pi / 3.0 / 2000
    plan = fq.Plan.tridiag(d.h0_diag, d.h0_off, d.h1_diag, omega=3.0, f_ac=1.5, f_dc=0.2, phi0=0.3, steps=M,
                           period=M * h, precision=precision, kernel=kernel)
    states = _random_states(n, nc, 1831)
    avg = plan.average_observable(states, 0.7, -0.4, 1.3).cpu().numpy()
    assert plan.check_status() == fq.FQ_OK
    x, ref, scale = states, 0.0, 0.0
    for m in range(M + 1):
        f = 0.2 + 1.5 * math.cos(3.0 * m * h + 0.3)
        v = x.cpu().numpy()
        dg = 0.7 * d.h0_diag + (-0.4 + 1.3 * f) * d.h1_diag
        e = (np.abs(v) ** 2 @ dg) + 2 * 0.7 * np.real(np.conj(v[:, :-1]) * v[:, 1:]) @ d.h0_off
        ref = ref + (0.5 if m in (0, M) else 1.0) * e / M
        scale = max(scale, np.max(np.abs(dg)) + 2 * np.max(np.abs(d.h0_off), initial=0.0))
        if m < M:
            x = plan.propagate(x, m, m + 1)
    # 64-bit sums of at most 1101 terms below the scale in magnitude
    assert np.max(np.abs(avg - ref)) <= 4 * n * 2.0 ** -53 * scale + 1e-15


@pytest.mark.parametrize("nb", [1, 30, 255, 256, 511, 512, 1100])
def test_tridiagonal_averages_few_and_many_states(fq, nb):
    """A CTA a state for up to three states an SM, four states a CTA for more: a state's average has the same bits
    either way, at row counts around the 256-row rounds, with a partly filled last CTA."""
    import torch
    d = fi.config_dimer(nb=nb)
    plan = fq.Plan.tridiag(d.h0_diag, d.h0_off, d.h1_diag, omega=3.0, f_ac=1.5, f_dc=0.2, phi0=0.3, steps=4,
                           period=4 * 2 * math.pi / 6000, precision=fq.FQ_FP64)
    x = _random_states(d.n, 5, 1835)
    few = plan.average_observable(x, 0.7, -0.4, 1.3)
    many = plan.average_observable(x.repeat(121, 1).contiguous(), 0.7, -0.4, 1.3)
    assert plan.check_status() == fq.FQ_OK
    assert torch.equal(many, few.repeat(121))


@pytest.mark.parametrize("n,k", [(1, 1), (5, 3), (31, 31), (32, 1), (33, 17), (255, 2), (256, 9), (257, 40), (520, 130)])
def test_unitarity_defect_chunks(fq, n, k):
    """The defect over listed columns (unsorted, one of them twice) at the edges of the 32- and 256-column
    blocks and of every chunk size, against the same sums in numpy."""
    import torch
    rng = np.random.default_rng(1841)
    u = fi.haar_unitary(n, 1842) + 1e-3 * (rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n)))
    cols = rng.permutation(n)[:k]
    cols[-1] = cols[0]
    d = u[:, cols].conj().T @ u
    d[np.arange(k), cols] -= 1.0
    U = torch.from_numpy(np.ascontiguousarray(u)).cuda()
    mx, fro = fq.api.unitarity_defect(U, torch.from_numpy(cols.astype(np.int32)).cuda())
    assert abs(mx - np.max(np.abs(d))) <= 1e-14 * (1 + n) and abs(fro - np.linalg.norm(d) / math.sqrt(k)) <= 1e-14 * (1 + n)
    full = u.conj().T @ u - np.eye(n)
    mx, fro = fq.api.unitarity_defect(U)
    assert abs(mx - np.max(np.abs(full))) <= 1e-14 * (1 + n)
    assert abs(fro - np.linalg.norm(full) / math.sqrt(n)) <= 1e-14 * (1 + n)


@pytest.mark.parametrize("n,k", [(40, 40), (257, 33), (520, 520)])
def test_unitarity_defect_least_workspace(fq, n, k):
    """A workspace of the least accepted size (a pair of doubles per 16 listed columns and 256 columns) makes a
    CTA take several column blocks: the defect of the queried size to rounding, and one alignment unit less is
    refused."""
    import torch
    rng = np.random.default_rng(1851)
    u = fi.haar_unitary(n, 1852) + 1e-3 * (rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n)))
    U = torch.from_numpy(np.ascontiguousarray(u)).cuda()
    cols = torch.from_numpy(rng.permutation(n)[:k].astype(np.int32)).cuda()
    least = -(-16 * -(-k // 16) * -(-n // 256) // 256) * 256
    mx, fro = fq.api.unitarity_defect(U, cols)
    a, b = fq.floquet_unitarity_defect(U, n, cols, k, fq.workspace(least))
    assert abs(a - mx) <= 1e-15 and abs(b - fro) <= 1e-14 * fro
    with pytest.raises(fq.FloquetError):
        fq.floquet_unitarity_defect(U, n, cols, k, fq.workspace(least - 256))


@pytest.mark.parametrize("precision", [0, 2])
def test_overlap_phase_error_matches_oracle(fq, precision):
    """Eq. 20 on the library (coarse chain applied to the fine Floquet states by
    floquet_propagate) against the oracle's Sigma from its own U_T's.  FP64 to 1e-9; the BF16X3
    coarse chain to sqrt(N) 1e-5: the split target bounds U_T's entries by 1e-5, hence
    ||dU phi||_2 <= sqrt(N) 1e-5 for a unit phi, and |dSigma| <= ||dU phi||_2."""
    n, M = 24, 40
    h0, h1 = fi.goe(n, 1901), fi.goe(n, 1902)
    drv = fi.Drive(0.2, 1.2, 1.3, 0.4)
    coarse = fq.Plan.dense(h0, h1, omega=drv.omega, f_ac=drv.f_ac, f_dc=drv.f_dc, phi0=drv.phi0, steps=M,
                           precision=precision)
    fine = fq.Plan.dense(h0, h1, omega=drv.omega, f_ac=drv.f_ac, f_dc=drv.f_dc, phi0=drv.phi0, steps=2 * M)
    eps, sig = fq.overlap_phase_error(coarse, fine.build_UT())
    uc = o.build_ut_dense(h0, h1, o.plan_for_drive_dense(h0, h1, drv, M))
    uf = o.build_ut_dense(h0, h1, o.plan_for_drive_dense(h0, h1, drv, 2 * M))
    ref_eps, ref_sig = o.overlap_phase_error(uc, uf, drv.period)
    assert np.max(np.abs(eps - ref_eps)) < 1e-10
    assert np.max(np.abs(sig - ref_sig)) <= (1e-9 if precision == 0 else math.sqrt(n) * 1e-5)
    assert np.max(ref_sig) > 1e-7   # the test resolves the coarse chain's error

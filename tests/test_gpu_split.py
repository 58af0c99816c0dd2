"""Split-precision dense path (tcgen05 BF16 slices, FP32 accumulation) against the FP64 oracle.

Tolerance: max |U - U_oracle| <= min(1e-5, 2 M R eps + 4 sqrt(M L) eps).  1e-5 is the accuracy
target for FP32-level split paths; the second term is the bound of the FP32 tridiagonal path with
eps the relative error of one sliced product:
  * FQ_BF16X3 (2 slices, products hi*hi + hi*lo + lo*hi): a bf16 slice keeps 8 significant bits,
    so two slices represent x to 2^-18 relative, and the dropped lo*lo term is of the same
    size; eps = 2^-17.
  * FQ_BF16X6 (3 slices, 6 products a + b < 3): the representation error is 2^-27, and FP32
    accumulation and the FP32 master copies dominate; eps = 2^-23.
"""
import math

import numpy as np
import pytest

import floquet_inputs as fi
import oracle as o

pytestmark = pytest.mark.gpu

EPS = {2: 2.0 ** -17, 3: 2.0 ** -23}


SPLIT_TARGET = 1e-5


def tol_split(M, L, R, ns):
    e = EPS[ns]
    return min(SPLIT_TARGET, 2.0 * M * R * e + 4.0 * math.sqrt(M * L) * e)


@pytest.fixture(scope="module")
def fq():
    import torch
    assert torch.cuda.is_available()
    import paper_1508_07621_gb300 as fq
    return fq


def cuda_c128(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.complex128)).cuda()


SHAPES = [(2, 2, 64, 0), (2, 2, 64, 32), (3, 3, 64, 0), (2, 2, 128, 0), (3, 3, 128, 0)]  # (prec, NS, width, K stage)


@pytest.mark.parametrize("prec,ns,tile,tk", SHAPES)
def test_split_goe64_build(fq, prec, ns, tile, tk):
    m = fi.config_goe64()
    plan = fq.Plan.dense(m.h0, m.h1, omega=m.drive.omega, f_ac=m.drive.f_ac, steps=m.steps, precision=prec,
                         tile_n=tile, tile_k=tk)
    U = plan.build_UT().cpu().numpy()
    assert plan.check_status() == fq.FQ_OK
    ref = o.build_ut_dense(m.h0, m.h1, o.plan_for_drive_dense(m.h0, m.h1, m.drive, m.steps))
    err = np.max(np.abs(U - ref))
    tol = tol_split(m.steps, plan.info.L, plan.info.R, ns)
    print(f"GOE64 split NS={ns}: max err {err:.3e} (tol {tol:.3e})")
    assert err <= tol


@pytest.mark.parametrize("n", [1, 3, 31, 33, 66, 127, 129, 161])
@pytest.mark.parametrize("prec,ns,tile,tk", SHAPES)
def test_split_tile_edges(fq, prec, ns, tile, tk, n):
    """U_T at the edges of the epilogue's 32-column blocks and 4-column units and of the 64- and
    128-wide tiles, every shape, with a drive of nonzero phase (A of Omega~ = S + i A not small)."""
    M = 10
    h0, h1 = fi.goe(n, 1311), fi.goe(n, 1312)
    drv = fi.Drive(0.2, 1.3, 1.1, 0.6)
    plan = fq.Plan.dense(h0, h1, omega=drv.omega, f_ac=drv.f_ac, f_dc=drv.f_dc, phi0=drv.phi0, steps=M,
                         precision=prec, tile_n=tile, tile_k=tk)
    U = plan.build_UT().cpu().numpy()
    assert plan.check_status() == fq.FQ_OK
    ref = o.build_ut_dense(h0, h1, o.plan_for_drive_dense(h0, h1, drv, M))
    assert np.max(np.abs(U - ref)) <= tol_split(M, plan.info.L, plan.info.R, ns)


@pytest.mark.parametrize("prec", [2, 3])
def test_split_default_tile(fq, prec):
    """Below the line of the default rule a plan without a tile width runs the 64-wide tiles, bit for
    bit as a plan that asks for them, whole and in column blocks."""
    import torch
    n = 150
    kw = dict(omega=1.3, f_ac=1.1, steps=6, precision=prec)
    h0, h1 = fi.goe(n, 1313), fi.goe(n, 1314)
    plan = fq.Plan.dense(h0, h1, **kw)
    U = plan.build_UT()
    assert torch.equal(U, fq.Plan.dense(h0, h1, tile_n=64, **kw).build_UT())
    X = plan.propagate(torch.eye(n, dtype=torch.complex128, device="cuda")[17:20].contiguous())
    assert torch.equal(X.transpose(0, 1), U[:, 17:20])


@pytest.mark.parametrize("prec,n,nc,width", [(3, 700, 700, 64), (3, 700, 3900, 64), (3, 700, 5000, 128), (2, 700, 5000, 64)])
def test_split_default_tile_of_many_states(fq, prec, n, nc, width):
    """More states than levels: BF16X6 plans without a tile width run the wide tiles from a wave and a half of
    them on (228 on 152 SMs: 38 blocks of 128 states at n = 700), bit for bit as a plan that asks for them."""
    import torch
    kw = dict(omega=1.3, f_ac=1.1, steps=64, precision=prec)
    h0, h1 = fi.goe(n, 1319), fi.goe(n, 1320)
    x = torch.eye(n, dtype=torch.complex128, device="cuda").repeat((nc + n - 1) // n, 1)[:nc].contiguous()
    plan = fq.Plan.dense(h0, h1, **kw)
    X = plan.propagate(x, 3, 5)
    assert plan.check_status() == 0
    assert torch.equal(X, fq.Plan.dense(h0, h1, tile_n=width, **kw).propagate(x, 3, 5))


@pytest.mark.parametrize("prec", [2, 3])
@pytest.mark.parametrize("n,nc", [(1, 1), (63, 5), (130, 129), (257, 200), (1024, 1024), (1100, 100)])
def test_split_kept_tiles(fq, prec, n, nc):
    """Chains whose tiles fit one to an SM keep states and accumulator on the SM, larger ones and a
    captured stream's single products keep them in memory: the same bits.  n = 1100 has 162 tiles a
    product for a whole build and 18 for 100 states."""
    import torch
    kw = dict(omega=1.3, f_ac=1.1, f_dc=0.2, phi0=0.4, steps=5, precision=prec, tile_n=64)
    plan = fq.Plan.dense(fi.goe(n, 1315), fi.goe(n, 1316), **kw)
    U = plan.build_UT()
    X = plan.propagate(torch.eye(n, dtype=torch.complex128, device="cuda")[:nc].contiguous())
    assert torch.equal(X.transpose(0, 1), U[:, :nc])
    ws = fq.workspace(plan.workspace_size())
    V = torch.empty_like(U)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        plan.build_UT(V, ws)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(U, V)
    assert plan.check_status() == 0


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_split_kept_tiles_not_finite(fq, bad):
    """A state with an entry that is not finite is reported and leaves the others as they are."""
    import torch
    n = 90
    plan = fq.Plan.dense(fi.goe(n, 1317), fi.goe(n, 1318), omega=1.3, f_ac=1.1, steps=4, precision=2)
    x = torch.eye(n, dtype=torch.complex128, device="cuda")[:40].contiguous()
    clean = plan.propagate(x.clone())
    assert plan.check_status() == 0
    x[17, 3] = bad
    X = plan.propagate(x)
    keep = [j for j in range(40) if j != 17]
    assert torch.equal(X[keep], clean[keep])
    assert not torch.isfinite(X[17].abs()).any()
    assert plan.check_status() != 0


@pytest.mark.parametrize("prec,ns,tile,tk", SHAPES)
def test_split_ragged_propagate(fq, prec, ns, tile, tk):
    """N = 200 (K' padded to 512, output tiles ragged), 37 states (one partial 128-row tile),
    steps 2..9 of 24, non-even drive."""
    n, M = 200, 24
    h0, h1 = fi.goe(n, 1301), fi.goe(n, 1302)
    drv = fi.Drive(0.2, 1.3, 1.1, 0.6)
    x0 = fi.ginibre(n, 1303)[:37]
    x0 /= np.linalg.norm(x0, axis=1, keepdims=True)
    plan = fq.Plan.dense(h0, h1, omega=drv.omega, f_ac=drv.f_ac, f_dc=drv.f_dc, phi0=drv.phi0, steps=M,
                         precision=prec, tile_n=tile, tile_k=tk)
    X = plan.propagate(cuda_c128(x0), 2, 10).cpu().numpy()
    ref = o.propagate_dense(h0, h1, o.plan_for_drive_dense(h0, h1, drv, M), x0.T, 2, 10).T
    err = np.max(np.abs(X - ref))
    assert err <= tol_split(8, plan.info.L, plan.info.R, ns), err


@pytest.mark.slow
def test_split_goe4096_sampled(fq):
    """Dense GOE N = 4096 (seeds 3, 4; A = 2, omega = 2, M = 512), BF16X6: 256 basis states
    through steps 0..7, against the oracle on the same states."""
    import torch
    m = fi.config_goe4096()
    plan = fq.Plan.dense(m.h0, m.h1, omega=m.drive.omega, f_ac=m.drive.f_ac, steps=m.steps, precision=3)
    cols = np.arange(0, 4096, 16)
    x0 = np.zeros((len(cols), 4096), complex)
    x0[np.arange(len(cols)), cols] = 1.0
    X = plan.propagate(cuda_c128(x0), 0, 8).cpu().numpy()
    assert plan.check_status() == fq.FQ_OK
    ref = o.propagate_dense(m.h0, m.h1, o.plan_for_drive_dense(m.h0, m.h1, m.drive, m.steps), x0.T, 0, 8).T
    err = np.max(np.abs(X - ref))
    print(f"GOE4096 BF16X6 8 steps: max err {err:.3e}")
    assert err <= tol_split(8, plan.info.L, plan.info.R, 3)


@pytest.mark.slow
@pytest.mark.parametrize("prec,ns", [(2, 2), (3, 3)])
def test_split_goe4096_full_build_sampled_columns(fq, prec, ns):
    """The dense benchmark workload end to end (GOE N = 4096, M = 512, tile 128): the U_T the
    library builds (one call, all 4096 states) against the oracle's propagation of 6 sampled
    basis states through all 512 steps, and the unitarity defect over 64 columns (stated, and
    checked against what the entry bound implies)."""
    import torch
    m = fi.config_goe4096()
    plan = fq.Plan.dense(m.h0, m.h1, omega=m.drive.omega, f_ac=m.drive.f_ac, steps=m.steps, precision=prec)
    U = plan.build_UT()
    assert plan.check_status() == fq.FQ_OK
    cols = [0, 1, 1000, 2047, 3001, 4095]
    x0 = np.zeros((4096, len(cols)), complex)
    x0[cols, np.arange(len(cols))] = 1.0
    ref = o.propagate_dense(m.h0, m.h1, o.plan_for_drive_dense(m.h0, m.h1, m.drive, m.steps), x0)
    got = U[:, cols].cpu().numpy()
    err = np.max(np.abs(got - ref))
    sample = torch.arange(0, 4096, 64, dtype=torch.int32, device="cuda")
    mx, fro = fq.api.unitarity_defect(U, sample)
    print(f"GOE4096 full build NS={ns}: max err {err:.3e} (tol {SPLIT_TARGET:.0e}); defect max {mx:.2e} fro {fro:.2e}")
    assert err <= SPLIT_TARGET
    # U = U_exact + D with |D_ij| <= e gives |(U^+U - 1)_cj| <= 2 sqrt(N) e + N e^2
    e = SPLIT_TARGET
    assert mx <= 2 * math.sqrt(4096) * e + 4096 * e * e

"""FP64 products by digits, the batched Cholesky sweep and the register tiles of
the FP32 form at the edges of their tiles, against the CPU oracle.

Bounds, fixed from the arithmetic: a product of digits errs by at most one
rounding and a truncation of 2^-61 of its row's largest element, so an FP64
result errs like the oracle's own sums.  chi, W and Sigma take the 1e-10 of the
other oracle tests; S^-1 M S^-1 with cond(S) < 6 and n <= 257 takes
2 n 2^-52 cond^2 = 4e-12, rounded to 1e-11 of the largest element.  The forms
that sum in FP32 take 1e-6.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from oracle import chain as och  # noqa: E402
from oracle import chi as oc  # noqa: E402
from oracle import sigma as osg  # noqa: E402
from synth import System, case_from_system, make_case  # noqa: E402
from synth.chain_inputs import omega_grid, synthetic_w, transform_weights  # noqa: E402


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__ as g

    g.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2104_09857_gb300 as p

    return p


def _basis(ctx, n):
    """A basis of n auxiliary functions, one primary function per atom."""
    ri = np.array([30] * (n // 30) + ([n % 30] if n % 30 else []), dtype=np.int32)
    xyz = np.zeros((len(ri), 3))
    xyz[:, 0] = 1.4 * np.arange(len(ri))
    ctx.set_basis(xyz, np.ones(len(ri), dtype=np.int32), ri)


def _spd(rng, n):
    b = rng.standard_normal((n, n))
    return b @ b.T / n + np.eye(n)


@pytest.mark.parametrize("n", [1, 2, 63, 64, 65, 127, 128, 129, 193, 257])
def test_metric_and_chain_sizes(pkg, n):
    """One matrix and one frequency, and several of each in a batch."""
    from paper_2104_09857_gb300 import _lib

    rng = np.random.default_rng(n)
    s = _spd(rng, n)
    m = rng.standard_normal((2, n, n))
    m = m + m.transpose(0, 2, 1)
    tau = np.array([0.05, 0.7, 6.0])
    gamma, delta = transform_weights(tau, omega_grid(3, 0.3, 2.3), 0.3, 2.3)
    chi = -np.stack([_spd(rng, n) * np.exp(-t) for t in tau])
    w_ref, _ = och.chi_to_w(chi, s, gamma, delta)
    with pkg.Context(0) as ctx:
        _basis(ctx, n)
        nao = len(s) // 30 + (1 if n % 30 else 0)
        c = np.eye(nao) if nao > 1 else np.ones((1, 1))
        got = _lib.gw_ri_metric(ctx.ctx, s, m)
        if nao > 1:
            ctx.set_greens(c, np.linspace(-1.0, 1.0, nao), 1, 0.0, tau)
            w = ctx.chi_to_w(chi, s, gamma, delta).cpu().numpy()
            for j in range(3):
                assert np.linalg.norm(w[j] - w_ref[j]) <= 1e-10 * np.linalg.norm(w_ref[j])
    for k in range(2):
        ref = och.apply_metric(s, m[k])
        assert np.abs(got[k] - ref).max() <= 1e-11 * np.abs(ref).max()


@pytest.mark.parametrize("last,ri", [(13, 63), (14, 64), (15, 65)])
def test_chi_at_the_tile_edges(pkg, last, ri):
    """447, 448 and 449 primary functions (both sides of the first size whose
    Green's functions are digit products), 63 to 65 auxiliary ones, all forms."""
    sysm = System("edge", np.array([[1.4 * i, 0.0, 0.0] for i in range(32)]), ["C"] * 32)
    sysm.n_ao = np.array([14] * 31 + [last], dtype=np.int32)
    sysm.n_ri = np.array([2] * 31 + [ri - 62], dtype=np.int32)
    case = case_from_system(sysm, 2, 1e-9, 7)
    case.tau = np.array([0.3, 2.0])
    ref = oc.chi_dense(case)
    with pkg.Context(0) as ctx:
        ctx.load_case(case)
        for form, tol in (("fp64", 1e-10), ("fp32", 1e-6), ("fp16x3", 1e-6), ("bf16x6", 1e-6)):
            got = ctx.chi_tau(case.thr, form).cpu().numpy()
            for j in range(2):
                assert np.linalg.norm(got[j] - ref[j]) <= tol * np.linalg.norm(ref[j]), (form, j)


@pytest.mark.parametrize("last", [1, 14])
def test_chi_operands_in_segments(pkg, last):
    """519 and 532 primary functions: a batch's reduction length (299 and 306
    thousand) passes one operand segment of the tensor-core forms."""
    sysm = System("long", np.array([[1.4 * i, 0.0, 0.0] for i in range(38)]), ["C"] * 38)
    sysm.n_ao = np.array([14] * 37 + [last], dtype=np.int32)
    sysm.n_ri = np.array([1] * 37 + [3], dtype=np.int32)
    case = case_from_system(sysm, 1, 1e-9, 7)
    case.tau = np.array([0.5])
    ref = oc.chi_dense(case)
    with pkg.Context(0) as ctx:
        ctx.load_case(case)
        for form in ("fp16x3", "bf16x6"):
            got = ctx.chi_tau(case.thr, form).cpu().numpy()
            assert np.linalg.norm(got - ref) <= 1e-6 * np.linalg.norm(ref), form


@pytest.mark.parametrize("form", ["fp64", "fp32"])
@pytest.mark.parametrize("thr", [0.0, 1e-18, 1e4])
def test_filter_outside_the_quick_norms(pkg, form, thr):
    """Thresholds whose square FP32 does not resolve, and one that drops all."""
    case = make_case("chain_CHCH", n_tau=2)
    ref = oc.chi_dense(case, thr=thr)
    with pkg.Context(0) as ctx:
        ctx.load_case(case)
        got = ctx.chi_tau(thr, form).cpu().numpy()
    assert np.abs(got - ref).max() <= (1e-10 if form == "fp64" else 1e-6) * np.abs(ref).max()


@pytest.mark.parametrize("n_orb", [1, 2, 3, 4, 5, 7])
def test_sigma_orbital_counts(pkg, n_orb):
    """B^n of every remainder of the orbitals that one pass takes."""
    case = make_case("benzene", n_tau=2)
    w = synthetic_w(case.system.nri_total, case.tau, 5)
    orbs = list(range(case.n_occ - n_orb // 2, case.n_occ - n_orb // 2 + n_orb))
    ref = osg.sigma_dense(case, w, orbs, thr=0.0)
    with pkg.Context(0) as ctx:
        ctx.load_case(case)
        got = ctx.sigma_tau(w, orbs, 0.0)
    assert np.abs(got - ref).max() <= 1e-10 * np.abs(ref).max()


def test_sigma_non_finite_rows(pkg):
    """A row that no fixed-point form holds takes the plain sums: the NaN shows
    at its tau point and the other one is as without it."""
    case = make_case("benzene", n_tau=2)
    w = synthetic_w(case.system.nri_total, case.tau, 5)
    orbs = [case.n_occ - 1, case.n_occ]
    with pkg.Context(0) as ctx:
        ctx.load_case(case)
        want = ctx.sigma_tau(w, orbs, 0.0)
        w[1, 3, :] = w[1, :, 3] = np.nan
        got = ctx.sigma_tau(w, orbs, 0.0)
    assert np.isnan(got[:, 1]).all()
    assert np.abs(got[:, 0] - want[:, 0]).max() <= 1e-14 * np.abs(want).max()

"""FP64 by digit products at its limits: time-outs, scratch memory, row chunks,
non-finite operands and elements far below the largest, against the CPU oracle."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from oracle import chi as oc  # noqa: E402
from synth import make_case  # noqa: E402


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__ as g

    g.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2104_09857_gb300 as p

    return p


def _rel(got, ref):
    return max(np.linalg.norm(a - b) / np.linalg.norm(b) for a, b in zip(got, ref))


def test_stall_times_out_and_context_recovers(pkg):
    """A dependency that is never met ends every kernel of the FP64 form after
    its bounded wait; the same context then computes chi."""
    from paper_2104_09857_gb300 import _lib

    case = make_case("benzene", n_tau=1)
    ref = oc.chi_dense(case)
    with pkg.Context(0) as ctx:
        ctx.load_case(case)
        ctx.set_option("test_stall_tc", 1)
        with pytest.raises(_lib.GwError) as e:
            ctx.chi_tau(case.thr, "fp64")
        assert e.value.code == -7  # GW_ERR_TIMEOUT
        ctx.set_option("test_stall_tc", 0)
        got = ctx.chi_tau(case.thr, "fp64").cpu().numpy()
    assert _rel(got, ref) <= 1e-10


def test_cholesky_pivots_are_rounded_roots(pkg):
    """With chi = 0, W^c = L L^T - V is the factorisation's own error.  For a
    diagonal V a correctly rounded root errs by 2^-53 of itself, its square by
    twice that and one more rounding: 3 2^-53 of V, to first order."""
    n, tau = 300, np.array([1.0])
    v = np.exp(np.random.default_rng(3).uniform(np.log(1e-6), np.log(1e6), n))
    with pkg.Context(0) as ctx:
        ctx.set_basis(np.arange(30.0).reshape(10, 3), np.ones(10, dtype=np.int32), np.full(10, n // 10, dtype=np.int32))
        ctx.set_greens(np.eye(10), np.linspace(-1.0, 1.0, 10), 5, 0.0, tau)
        w = ctx.chi_to_w(np.zeros((1, n, n)), np.diag(v), np.ones((1, 1)), np.ones((1, 1))).cpu().numpy()[0]
    assert not np.any(w - np.diag(np.diag(w)))
    assert np.abs(np.diag(w) / v).max() <= 3 * 2.0 ** -53 * (1 + 1e-9)

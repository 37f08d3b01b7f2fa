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

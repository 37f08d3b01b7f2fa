"""FP64 by digit products at its limits: time-outs, scratch memory, row chunks,
non-finite operands and elements far below the largest, against the CPU oracle."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from oracle import chi as oc  # noqa: E402
from synth import System, case_from_system, make_case  # noqa: E402


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


def test_chi_of_distant_functions(pkg):
    """Every element of chi along a chain of 33 Angstrom, over which chi falls by
    1e-10, to an FP64 sum's accuracy: with S = sum |X| |Y| (Green's functions of
    positive orbitals, so that their sums do not cancel), n operations of
    rounding 2^-53 each err by n 2^-53 S; chi is K = n_AO^2 of them, X and Y each
    n_AO + n_AO (G), the oracle's own sums the same again."""
    n, rng = 24, np.random.default_rng(9)
    sysm = System("chain", np.array([[1.4 * i, 0.0, 0.0] for i in range(n)]), ["C"] * n)
    sysm.n_ao = np.full(n, 2, dtype=np.int32)
    sysm.n_ri = np.full(n, 2, dtype=np.int32)
    case = case_from_system(sysm, 1, 0.0, 7)
    nao, tau = 2 * n, 0.5
    x = np.repeat(sysm.xyz[:, 0], 2)
    at = np.concatenate([sysm.xyz[:, 0], sysm.xyz[:, 0]])  # one occupied, one virtual orbital per atom
    c = rng.uniform(0.5, 1.0, (nao, nao)) * np.exp(-0.8 * np.abs(x[:, None] - at[None]))
    eps = np.concatenate([np.linspace(-1.0, -0.2, n), np.linspace(0.2, 1.0, n)])
    t = case.t3c
    d = oc.dense_three_center(sysm.n_ao, sysm.n_ri, t.blocks, t.offsets, t.data)
    h = c * np.exp(-0.5 * tau * np.abs(eps))
    go, gv = h[:, :n] @ h[:, :n].T, h[:, n:] @ h[:, n:].T

    def sums(t3):
        m = np.einsum("ml,lsp->msp", go, t3).reshape(nao * nao, -1)
        q = np.einsum("sl,mlq->msq", gv, t3).reshape(nao * nao, -1)
        return m.T @ q

    ref, bound = -sums(d), sums(np.abs(d))
    with pkg.Context(0) as ctx:
        ctx.set_basis(sysm.xyz, sysm.n_ao, sysm.n_ri)
        ctx.set_3c_tensor(t.blocks, t.data)
        ctx.set_greens(c, eps, n, 0.0, np.array([tau]))
        got = ctx.chi_tau(0.0, "fp64").cpu().numpy()[0]
    up = np.arange(nao)[:, None] // 2 <= np.arange(nao)[None] // 2
    assert bound[0, -1] <= 1e-9 * bound.max()
    assert (np.abs(got - ref)[up] / bound[up]).max() <= 2 * (nao * nao + 4 * nao) * 2.0 ** -53


def _digits(ctx):
    """The last call's products were digits (36 of them per multiply-add)."""
    s = ctx.stats()
    return s["flops_issued"] > 16 * s["flops_useful"]


def test_chi_without_room_for_a_batch_of_digits(pkg):
    """A batch whose digits do not fit goes through the CUDA-core kernels; the
    call fails only where their operands do not fit either."""
    from paper_2104_09857_gb300 import _lib

    case = make_case("benzene", n_tau=2)
    ref = oc.chi_dense(case)
    seen = []
    for limit in 2e6 * 1.25 ** np.arange(24):
        with pkg.Context(0) as ctx:
            ctx.load_case(case)
            ctx.set_option("batch_atoms", 1)
            ctx.chi_tau(case.thr, "fp64", 0, 1)  # the panels' digits are there
            ctx.set_option("batch_atoms", 0)
            ctx.set_option("test_device_bytes", limit)
            try:
                got = ctx.chi_tau(case.thr, "fp64").cpu().numpy()
            except _lib.GwError as e:
                assert e.code == -5  # GW_ERR_OOM
                seen.append("none")
            else:
                assert _rel(got, ref) <= 1e-10
                seen.append("digits" if _digits(ctx) else "cores")
            ctx.set_option("test_device_bytes", 0)
            got = ctx.chi_tau(case.thr, "fp64").cpu().numpy()
            assert _rel(got, ref) <= 1e-10 and _digits(ctx)
    order = [k for i, k in enumerate(seen) if i == 0 or seen[i - 1] != k]
    assert order == ["none", "cores", "digits"], seen


def test_route_does_not_depend_on_earlier_calls(pkg):
    """The memory that a plan with digits needs is not counted twice where the
    context holds its buffers already: the smallest device on which the digits
    are taken serves a second threshold as well."""
    case = make_case("ribbon28", n_tau=2)

    def routes(limit):
        with pkg.Context(0) as ctx:
            ctx.load_case(case)
            ctx.set_option("test_device_bytes", limit)
            out = []
            for thr in (1e-6, 1e-9, 1e-6):
                got = ctx.chi_tau(thr, "fp64", 0, 1).cpu().numpy()
                out.append(_digits(ctx))
            return out, got

    ref = oc.chi_dense(case, thr=1e-6)[:1]
    lo, hi = 1.5e9, 2e10  # the CUDA cores' X and Y fit; everything does
    assert routes(hi)[0] == [True] * 3
    for _ in range(7):
        mid = (lo * hi) ** 0.5
        taken, got = routes(mid)
        assert _rel(got, ref) <= 1e-10
        assert taken[2] == taken[0]
        # 1e-9 keeps more blocks than 1e-6: it may need more
        lo, hi = (lo, mid) if taken[0] else (mid, hi)


def test_other_calls_get_the_panel_digits_memory(pkg):
    """A call that finds no memory takes back the panels' digits of an earlier
    FP64 chi before it gives up: afterwards there are device sizes at which chi
    has to do without them (were they still there, it would need nothing new)."""
    from paper_2104_09857_gb300 import _lib
    from synth.chain_inputs import synthetic_w

    case = make_case("benzene", n_tau=1)
    ref = oc.chi_dense(case)
    w = synthetic_w(case.system.nri_total, case.tau, 5)
    taken = []
    for limit in 2e7 * 1.2 ** np.arange(24):
        with pkg.Context(0) as ctx:
            ctx.load_case(case)
            ctx.chi_tau(case.thr, "fp64")
            assert _digits(ctx)
            ctx.set_option("test_device_bytes", 1)
            with pytest.raises(_lib.GwError) as e:
                ctx.sigma_tau(w, [case.n_occ], case.thr)
            assert e.value.code == -5  # GW_ERR_OOM
            ctx.set_option("test_device_bytes", limit)
            try:
                got = ctx.chi_tau(case.thr, "fp64").cpu().numpy()
            except _lib.GwError as e:
                assert e.code == -5
            else:
                assert _rel(got, ref) <= 1e-10
                taken.append(_digits(ctx))
    assert not taken[0] and taken[-1], taken


def _spd(rng, n):
    b = rng.standard_normal((n, n))
    return b @ b.T / n + np.eye(n)


@pytest.fixture(scope="module")
def dense_inputs():
    """chi(i tau), V, transforms, S and M of n = 300 auxiliary functions."""
    rng = np.random.default_rng(21)
    n = 300
    m = rng.standard_normal((2, n, n))
    return {"n": n, "tau": np.array([0.1, 1.0, 8.0]), "chi": -np.stack([_spd(rng, n) * f for f in (1.0, 0.5, 0.1)]),
            "v": _spd(rng, n), "gamma": rng.standard_normal((3, 3)) ** 2, "delta": rng.standard_normal((3, 3)),
            "m": m + m.transpose(0, 2, 1)}


def _dense_calls(ctx, d):
    from paper_2104_09857_gb300 import _lib

    w = ctx.chi_to_w(d["chi"], d["v"], d["gamma"], d["delta"]).cpu().numpy()
    return w, np.asarray(_lib.gw_ri_metric(ctx.ctx, d["v"], d["m"]))


def _dense_context(pkg, d):
    ctx = pkg.Context(0)
    ctx.set_basis(np.arange(30.0).reshape(10, 3), np.ones(10, dtype=np.int32),
                  np.full(10, d["n"] // 10, dtype=np.int32))
    ctx.set_greens(np.eye(10), np.linspace(-1.0, 1.0, 10), 5, 0.0, d["tau"])
    return ctx


def test_row_chunks_and_frequency_groups_change_nothing(pkg, dense_inputs):
    """Products in chunks of 128 rows and sweeps of one frequency at a time: sums
    of digits are exact, so every bit is that of the whole product."""
    from paper_2104_09857_gb300 import _lib
    from synth.chain_inputs import synthetic_w

    case = make_case("benzene", n_tau=1)
    w = synthetic_w(case.system.nri_total, case.tau, 5)
    nao = case.system.nao_total
    got = []
    for limit in (0, 7e5):
        with _dense_context(pkg, dense_inputs) as ctx:
            ctx.set_option("test_digit_bytes", limit)
            got.append(list(_dense_calls(ctx, dense_inputs)))
        with pkg.Context(0) as ctx:
            ctx.load_case(case)
            ctx.set_option("test_digit_bytes", limit)
            got[-1].append(np.asarray(_lib.gw_sigma_ao_tau(ctx.ctx, w, 1, nao, case.thr)))
    for whole, chunks in zip(*got):
        assert np.array_equal(whole, chunks)


def test_products_without_room_for_whole_digits(pkg, dense_inputs):
    """On a device that does not hold an operand's digits whole the products go
    in smaller chunks: chi_to_w and the metric run, to the same bits, with less
    than their matrices, the partial sums and both operands' digits."""
    from paper_2104_09857_gb300 import _lib

    d, n = dense_inputs, dense_inputs["n"]
    nn, digits = 8.0 * n * n, 16.0 * n * 320
    with _dense_context(pkg, d) as ctx:
        ref = _dense_calls(ctx, d)
    ran = []
    for limit in 6 * nn * 1.05 ** np.arange(40):
        with _dense_context(pkg, d) as ctx:
            ctx.set_option("test_device_bytes", limit)
            try:
                got = _dense_calls(ctx, d)
            except _lib.GwError as e:
                assert e.code == -5, limit
            else:
                assert all(np.array_equal(a, b) for a, b in zip(got, ref))
                ran.append(limit)
    # V, L, [eps; L] of one frequency and two products; a sweep's panel as digits
    # and the partial sums of its update; two operands
    rows = 2 * n - 64
    assert ran and ran[0] < 6 * nn + rows * (64 + n - 64) * 16 + 2 * digits, ran


@pytest.mark.parametrize("n", [2, 29, 30])
def test_chain_of_one_frequency_and_few_functions(pkg, n):
    """Two atoms, one frequency: the smallest chains."""
    from oracle import chain as och

    rng = np.random.default_rng(n)
    v, chi = _spd(rng, n), -_spd(rng, n)[None]
    one = np.ones((1, 1))
    ref, _ = och.chi_to_w(chi, v, one, one)
    with pkg.Context(0) as ctx:
        ctx.set_basis(np.array([[0.0, 0.0, 0.0], [1.4, 0.0, 0.0]]), np.ones(2, dtype=np.int32),
                      np.array([n - n // 2, n // 2], dtype=np.int32))
        ctx.set_greens(np.eye(2), np.array([-1.0, 1.0]), 1, 0.0, np.array([1.0]))
        got = ctx.chi_to_w(chi, v, one, one).cpu().numpy()
    assert np.linalg.norm(got - ref) <= 1e-10 * np.linalg.norm(ref)


@pytest.mark.parametrize("where", ["tensor", "orbitals"])
def test_non_finite_chi(pkg, where):
    """Operands that no fixed-point form holds take the plain sums, in the panels
    and in step C: elements of magnitude 1e200 overflow G (to Inf) or T's
    products, and what they do not reach is as without them."""
    case = make_case("chain_CHCH", n_tau=1)
    with pkg.Context(0) as ctx:
        ctx.load_case(case)
        want = ctx.chi_tau(0.0, "fp64").cpu().numpy()[0]
        big = 1e200 if where == "tensor" else 1e160
        if where == "tensor":  # T^2 overflows: the elements of chi with the last auxiliary function
            data = case.t3c.data.copy()
            last = case.t3c.blocks[:, 2] == case.system.n_atoms - 1
            for i in np.nonzero(last)[0]:
                blk = data[case.t3c.offsets[i]:case.t3c.offsets[i + 1]].reshape(-1, case.system.n_ri[-1])
                blk[:, -1] *= big
            ctx.set_3c_tensor(case.t3c.blocks, data)
        else:  # G overflows
            c = case.C.copy()
            c[0] *= big
            ctx.set_greens(c, case.eps, case.n_occ, case.mu_fermi, case.tau)
        got = ctx.chi_tau(0.0, "fp64").cpu().numpy()[0]
    if where == "tensor":
        assert not np.isfinite(got[-1, -1])
        assert np.abs(got[:-1, :-1] - want[:-1, :-1]).max() <= 1e-14 * np.abs(want).max()
        assert np.abs(got[:-1, -1] / big - want[:-1, -1]).max() <= 1e-13 * np.abs(want).max()
    else:
        assert not np.isfinite(got).any()


def test_segments_stay_within_the_operand_budget(pkg):
    """X and Y of 519 functions take one batch of exactly batch_bytes without the
    padding of their segments: with it they take two."""
    sysm = System("long", np.array([[1.4 * i, 0.0, 0.0] for i in range(38)]), ["C"] * 38)
    sysm.n_ao = np.array([14] * 37 + [1], dtype=np.int32)
    sysm.n_ri = np.array([1] * 37 + [3], dtype=np.int32)
    case = case_from_system(sysm, 1, 1e-9, 7)
    case.tau = np.array([0.5])
    ref = oc.chi_dense(case)
    plain = 4 * (40 + 40) * (576 * 519)  # two 16-bit slices, rows of X and Y, padded functions x functions
    with pkg.Context(0) as ctx:
        ctx.load_case(case)
        for room, batches in ((1.2, 1), (1.0, 2)):
            ctx.set_option("batch_bytes", plain * room)
            got = ctx.chi_tau(case.thr, "fp16x3").cpu().numpy()
            assert ctx.stats()["n_batches"] == batches
            assert np.linalg.norm(got - ref) <= 1e-6 * np.linalg.norm(ref)


@pytest.mark.parametrize("nao,nri", [(255, 257), (256, 256), (257, 257)])
def test_long_rows_of_digits(pkg, nao, nri):
    """The last product of the AO self-energy at n_AO n_RI = 65535, 65536 and
    66049: rows of digits, the first length in blocks, an odd one."""
    from oracle import sigma as osg
    from paper_2104_09857_gb300 import _lib
    from synth.chain_inputs import synthetic_w

    n = 17
    sysm = System("chain", np.array([[1.4 * i, 0.0, 0.0] for i in range(n)]), ["C"] * n)
    sysm.n_ao = np.array([15] * 16 + [nao - 240], dtype=np.int32)
    sysm.n_ri = np.array([15] * 16 + [nri - 240], dtype=np.int32)
    case = case_from_system(sysm, 1, 1e-9, 7)
    w = synthetic_w(nri, case.tau, 5)
    ref = osg.sigma_ao_dense(case, w, thr=case.thr)
    with pkg.Context(0) as ctx:
        ctx.load_case(case)
        got = np.asarray(_lib.gw_sigma_ao_tau(ctx.ctx, w, 1, nao, case.thr)).reshape(np.shape(ref))
    assert np.linalg.norm(got - ref) <= 1e-10 * np.linalg.norm(ref)

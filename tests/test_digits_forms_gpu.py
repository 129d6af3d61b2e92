"""Digit-split products as a program uses a handle: precisions in turn, CUDA graphs of its own."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from tests import gpu_cases as G  # noqa: E402
from tests.test_digits_gpu import _one_block_case, _oracle, TOL  # noqa: E402
from tests.test_heff_gpu import _dev  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_1512_03318_gb300 as P
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return P.Context(0, torch.cuda.current_stream())


def test_precisions_in_turn_keep_their_operands(ctx):
    """FP64 and float-float applications in turn on one handle: once each has run, a change of precision
    launches nothing besides the application (no second planning or packing of the environments), and the
    results stay the same bits."""
    import paper_1512_03318_gb300 as P
    case = _one_block_case(91, 256, 200, 4)
    ref = _oracle(case)
    h = P.Heff(ctx, **G.heff_args(case))
    h.set_env(_dev(case["lflat"]), _dev(case["rflat"]))
    T = _dev(case["tflat"])
    out = torch.empty_like(T)
    first, launches = {}, {}
    for prec in (0, 0, 3, 3, 0, 3, 0, 0, 3):
        n = P.launch_count()
        h.apply(T, out, prec)
        h.status()
        launches.setdefault(prec, []).append(P.launch_count() - n)
        got = out.cpu().numpy()
        assert np.max(np.abs(got - ref)) <= TOL[prec] * np.max(np.abs(ref))
        assert np.array_equal(got, first.setdefault(prec, got))
    for prec in (0, 3):
        assert len(set(launches[prec][1:])) == 1, launches
    # new environments are packed once for each precision
    h.set_env(_dev(2.0 * case["lflat"]), _dev(case["rflat"]))
    for prec in (0, 3):
        h.apply(T, out, prec)
        assert np.array_equal(out.cpu().numpy(), 2.0 * first[prec])
    h.close()


@pytest.mark.parametrize("warm", [False, True])
def test_fp64_in_a_callers_graph(warm):
    """An FP64 application captured by the caller, with or without an earlier one: a replay multiplies the
    environments and theta of its own time, and applications outside the graph stay right."""
    import paper_1512_03318_gb300 as P
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    s = torch.cuda.Stream()
    case = _one_block_case(93, 256, 200, 4)
    ref = _oracle(case)
    ok = lambda x, f: np.max(np.abs(x.cpu().numpy() - f * ref)) <= TOL[0] * f * np.max(np.abs(ref))
    with torch.cuda.stream(s):
        ctx = P.Context(0, s)
        h = P.Heff(ctx, **G.heff_args(case))
        L, R, T = _dev(case["lflat"]), _dev(case["rflat"]), _dev(case["tflat"])
        L2, out, out2 = 2.0 * L, torch.empty_like(T), torch.empty_like(T)
        h.set_env(L, R)
        if warm:
            h.apply(T, out2, 0)
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            h.apply(T, out, 0)
        g.replay()
        assert ok(out, 1.0)
        h.set_env(L2, R)
        g.replay()
        assert ok(out, 2.0)
        h.apply(T, out2, 0)
        assert ok(out2, 2.0)
        # the environment load captured too: its replays change what the next application multiplies
        g2 = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g2, stream=s):
            h.set_env(L, R)
            h.apply(T, out, 0)
        for f in (1.0, 3.0):
            L.copy_(f * _dev(case["lflat"]))
            g2.replay()
            assert ok(out, f)
            h.apply(T, out2, 0)
            assert ok(out2, f)
            e, steps = h.lanczos(T.clone(), 2, 0.0, 0)
            assert steps == 2 and np.isfinite(e)
        h.close()
        del g, g2


@pytest.mark.parametrize("prec", [0, 3])
def test_lanczos_after_captured_loads(prec):
    """Lanczos on environments that a replay changed: the same energy as on a handle of their own."""
    import paper_1512_03318_gb300 as P
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    s = torch.cuda.Stream()
    case = _one_block_case(95, 256, 200, 4)
    with torch.cuda.stream(s):
        ctx = P.Context(0, s)
        L, R, T = _dev(case["lflat"]), _dev(case["rflat"]), _dev(case["tflat"])

        def fresh(x):
            h = P.Heff(ctx, **G.heff_args(case))
            h.set_env(x, R)
            e = h.lanczos(T.clone(), 3, 0.0, prec)[0]
            h.close()
            return e

        h = P.Heff(ctx, **G.heff_args(case))
        h.set_env(L, R)
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            h.set_env(L, R)
        for f in (1.0, -1.5):
            L.copy_(f * _dev(case["lflat"]))
            g.replay()
            assert h.lanczos(T.clone(), 3, 0.0, prec)[0] == fresh(L)
        h.close()
        del g


def test_float_float_in_a_callers_graph_keeps_its_panels():
    """A captured float-float application reads panels of the handle: they stay while other precisions, options
    and a run that would release panels come and go, and a replay gives the same bits."""
    import paper_1512_03318_gb300 as P
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    s = torch.cuda.Stream()
    case = _one_block_case(107, 256, 200, 4)
    with torch.cuda.stream(s):
        ctx = P.Context(0, s)
        h = P.Heff(ctx, **G.heff_args(case))
        h.set_option(P.MRD_OPT_DIGITS, 2)
        h.set_env(_dev(case["lflat"]), _dev(case["rflat"]))
        T = _dev(case["tflat"])
        out, out2 = torch.empty_like(T), torch.empty_like(T)
        h.apply(T, out2, 3)
        assert h.form() == 1
        first = out2.cpu().numpy()
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            h.apply(T, out, 3)
        for change in range(4):
            if change == 1:
                h.apply(T, out2, 0)
            elif change == 2:
                h.set_option(P.MRD_OPT_PER_TASK_LAUNCH, 1)
                h.apply(T, out2, 3)
                h.set_option(P.MRD_OPT_PER_TASK_LAUNCH, 0)
            elif change == 3:
                h.lanczos(T.clone(), 2, 0.0, 3)
            out.fill_(0.0)
            g.replay()
            assert np.array_equal(out.cpu().numpy(), first)
        h.close()
        del g

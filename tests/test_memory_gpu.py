"""Device memory at its limit: what the library keeps for speed (cached blocks, panels of digit-split
products) makes way for what a call cannot do without."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import synth  # noqa: E402
from tests import gpu_cases as G  # noqa: E402
from tests.test_digits_gpu import _one_block_case, _oracle, TOL  # noqa: E402
from tests.test_heff_gpu import _dev  # noqa: E402

pytestmark = pytest.mark.gpu

MB = 1 << 20


class Hog:
    """All free device memory but `leave` bytes, while the block runs."""

    def __init__(self, leave):
        self.leave = leave

    def __enter__(self):
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        free, _ = torch.cuda.mem_get_info()
        assert free > self.leave
        self.x = torch.empty((free - self.leave) // (2 * MB) * (2 * MB), dtype=torch.uint8, device="cuda")

    def __exit__(self, *a):
        torch.cuda.synchronize()
        del self.x
        torch.cuda.empty_cache()


@pytest.fixture()
def ctx():
    import paper_1512_03318_gb300 as P
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = P.Context(0, torch.cuda.current_stream())
    c.release_cached()
    yield c
    c.release_cached()


def _state(ctx, chi):
    """A half-filled 4 x 8 cylinder with the bond sectors of a converged state, centre in the middle."""
    import paper_1512_03318_gb300 as P
    mpo = P.MPO(None, 4, 8, 1, 8, 1.0, 1.0, P.MRD_BASIS_MIXED)
    caps = [[(q[0], q[1], d) for q, d in synth.bond_sectors(chi, 8, round(j / 2), synth.substream(97, 7, j), min_dim=1)]
            if 2 <= j <= 30 else [] for j in range(33)]
    return P.DMRG(ctx, mpo, 16, 0, chi, seed=5, center=16, caps=caps)


def test_panels_make_way_for_lanczos(ctx):
    """FP64 applications hold panels of hundreds of MB; the Lanczos basis (65 MB here) that then finds no
    memory gets theirs, and the applications go on."""
    import paper_1512_03318_gb300 as P
    case = _one_block_case(97, 160, 160, 40)
    ref = _oracle(case)
    h = P.Heff(ctx, **G.heff_args(case))
    h.set_env(_dev(case["lflat"]), _dev(case["rflat"]))
    T = _dev(case["tflat"])
    out, v = torch.empty_like(T), T.clone()
    ok = lambda: np.max(np.abs(out.cpu().numpy() - ref)) <= TOL[0] * np.max(np.abs(ref))
    h.apply(T, out, 0)
    assert ok()
    with Hog(24 * MB):
        e, steps = h.lanczos(v, 3, 0.0, 0)
        assert steps == 3 and np.isfinite(e)
        h.apply(T, out, 0)
        assert ok()
    h.set_env(_dev(case["lflat"]), _dev(case["rflat"]))
    h.apply(T, out, 0)
    assert ok()
    h.close()


def test_cached_blocks_make_way_for_a_state(ctx):
    """Blocks of a freed H_eff are cached; a DMRG state whose own buffers find no memory gets theirs."""
    import paper_1512_03318_gb300 as P
    case = _one_block_case(99, 700, 700, 30)
    h = P.Heff(ctx, **G.heff_args(case))
    h.set_env(_dev(case["lflat"]), _dev(case["rflat"]))
    T = _dev(case["tflat"])
    out = torch.empty_like(T)
    h.apply(T, out, 0)
    torch.cuda.synchronize()
    h.close()
    with Hog(10 * MB):
        d = _state(ctx, 800)
        e, _ = d.update(16, +1, P.DMRG.params(800, 0.0, 2, 0.0, 0, 0, 1e-13))
        assert np.isfinite(e)
        d.close()


def test_idle_state_keeps_no_panels(ctx):
    """After an environment update the panels of its products are in the cache, which a program can give back."""
    import paper_1512_03318_gb300 as P
    d = _state(ctx, 800)
    ctx.release_cached()
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    size = 16 * d.env_len(16, 0)
    d.env_update(15, +1, P.MRD_PREC_FF)
    torch.cuda.synchronize()
    ctx.release_cached()
    # what stays: the state's own scratch (T, tables), a few times the environment's size at most
    assert before - torch.cuda.mem_get_info()[0] <= 4 * size
    d.close()


@pytest.mark.parametrize("prec,tol", [(2, 1e-4), (3, TOL[3])])
def test_application_after_one_that_found_no_memory(ctx, prec, tol):
    """Split BF16 operands that find no memory: the application is refused, and the next one, with room, is
    right (half-built tables are not taken for built). Float-float ones alike, whichever kernels run."""
    import paper_1512_03318_gb300 as P
    case = _one_block_case(103, 160, 160, 40)
    ref = _oracle(case)
    h = P.Heff(ctx, **G.heff_args(case))
    h.set_env(_dev(case["lflat"]), _dev(case["rflat"]))
    T = _dev(case["tflat"])
    out = torch.empty_like(T)
    with Hog(10 * MB):
        with pytest.raises(P.MrdError) as ex:
            h.apply(T, out, prec)
        assert ex.value.code == -4
        h.status()
    h.apply(T, out, prec)
    h.status()
    assert np.max(np.abs(out.cpu().numpy() - ref)) <= tol * np.max(np.abs(ref))
    h.close()

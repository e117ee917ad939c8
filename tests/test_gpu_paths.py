"""Which kernel steps a box: the automatic choice, and that a handle's reports say what runs."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2507_08820_gb300 import build
    build.build()
    from paper_2507_08820_gb300 import rflbm
    return rflbm


def _waits_for_copies(R, box):
    """True when the next step runs a TMA kernel: with bytes expected that never arrive, its wait expires, while the
    general kernel has no copies to wait for."""
    R.rflbm_init_rest(box.h)
    R.rflbm_testing_expect_extra_bytes(box.h, 16)
    R.rflbm_step(box.h, 1)
    try:
        R.rflbm_synchronize(box.h)
        return False
    except R.RflbmError as e:
        assert e.status == R.RFLBM_ETIMEOUT
        return True
    finally:
        R.rflbm_testing_expect_extra_bytes(box.h, 0)


@pytest.mark.parametrize("shape,tma", [((32, 32, 32), False), ((64, 8, 8), False), ((64, 9, 7), True)])
@pytest.mark.parametrize("pattern", [0, 1])
def test_a_testing_hook_does_not_change_the_kernel(R, shape, tma, pattern):
    """The automatic choice takes the general kernel for small boxes from 4096 sites, whatever hook is set."""
    box = R.Box(*shape, tau=0.8, kT=1e-4, pattern=pattern)
    assert _waits_for_copies(R, box) is tma
    box.close()


AUTO, GATHER, TMA = 0, 1, 2


@pytest.mark.parametrize("shape,kw,path,sites", [
    ((32, 32, 32), dict(kT=1e-4), (GATHER, 0), (1, 1)),              # small boxes: the general kernel
    ((32, 32, 32), dict(kT=1e-4, storage=1), (GATHER, 0), (1, 1)),
    ((32, 32, 32), dict(kT=0.0), (GATHER, 0), (1, 1)),
    ((32, 32, 32), dict(kT=0.0, storage=1), (TMA, 32), (2, 2)),
    ((32, 32, 32), dict(kT=1e-4, kernel=TMA), (TMA, 32), (1, 1)),
    ((100, 12, 11), dict(kT=1e-4, pattern=1), (GATHER, 0), (1, 1)),
    ((100, 12, 11), dict(kT=1e-4, kernel=TMA), (TMA, 128), (1, 1)),  # a ragged segment
    ((64, 6, 5), dict(kT=0.0), (TMA, 64), (2, 2)),
    ((256, 64, 9), dict(kT=1e-4, pattern=1), (TMA, 128), (1, 2)),    # row segments
    ((150, 50, 41), dict(kT=1e-4), (TMA, 0), (1, 1)),                # flat tiles
    ((150, 50, 41), dict(kT=1e-4, storage=2), (TMA, 0), (2, 2)),
    ((150, 50, 41), dict(kT=1e-4, pattern=1), (TMA, 0), (1, 2)),
    ((151, 50, 41), dict(kT=1e-4, pattern=1), (TMA, 0), (1, 1)),
    ((160, 50, 41), dict(kT=1e-4, kernel=TMA), (TMA, 0), (1, 1)),
    ((160, 50, 41), dict(kT=1e-4, kernel=GATHER), (GATHER, 0), (1, 1)),
    ((150, 50, 41), dict(kT=0.0), (GATHER, 0), (1, 1)),              # too small for flat tiles without noise
    ((160, 8, 2), dict(kT=1e-4, nz_global=4), (TMA, 32), (1, 1)),    # a z-slab
])
def test_reports_say_what_runs(R, shape, kw, path, sites):
    """The path and the sites per thread of the first and the second step of each rule's sides."""
    box = R.Box(*shape, tau=0.8, **kw)
    assert R.rflbm_step_path(box.h) == path
    R.rflbm_init_rest(box.h)
    got = [R.rflbm_step_sites_per_thread(box.h)]
    if not kw.get("nz_global"):
        R.rflbm_step(box.h, 1)
        got.append(R.rflbm_step_sites_per_thread(box.h))
        assert tuple(got) == sites
        assert _waits_for_copies(R, box) is (path[0] == TMA)
    else:
        assert got[0] == sites[0]
    box.close()

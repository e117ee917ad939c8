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

"""The kernels that carry FP64 results on float32 and integer pipes (csrc/wide.cuh): initial
fields, moments, global statistics, mode sums and shell sums, at the edges of the ranges where
they change to plain FP64 and at sizes around their blocks, against FP64 numpy.

A population is stored as the float32 g = f - w rho0, so an FP64 export returns it to one FP64
rounding of f, and sums of 27 of them agree with numpy's to 27 roundings of their terms."""
import numpy as np
import pytest

from oracle import rflbm_oracle as o
from paper_2507_08820_gb300 import workloads as W

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -53


@pytest.fixture(scope="module")
def R():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2507_08820_gb300 import build
    build.build()
    from paper_2507_08820_gb300 import rflbm
    return rflbm


@pytest.mark.parametrize("du", [0.0, 1e-30, 1e-12, 1e-8, 1e-3, 0.3, 1e5])
@pytest.mark.parametrize("rho0", [1.0, 0.37])
@pytest.mark.parametrize("pattern", [0, 1])
def test_initial_fields_round_once(R, du, rho0, pattern):
    """g is the float32 nearest to f - w rho0 up to the FP64 roundings of f, for velocities from
    zero to beyond the split's range (at 2^16), a site of each kind in every warp."""
    shape = (33, 5, 3)
    n = int(np.prod(shape))
    rho, u = W.random_fields(*shape, seed=3, drho=min(du, 0.02), du=du, rho0=rho0)
    u[:, ::7] = 0.0
    rho[::5] = rho0
    box = R.Box(*shape, tau=0.8, rho0=rho0, pattern=pattern)
    R.rflbm_init_field(box.h, rho, np.ascontiguousarray(u))
    got = box.populations()
    box.close()
    rho0 = float(np.float32(rho0))
    f = o.equilibrium_state(rho, u)
    rest = o.weights()[:, None] * rho0
    scale = np.abs(rho) * np.prod([1.0 + 3 * np.abs(v) + 3 * v * v for v in u], axis=0) * o.weights()[:, None]
    assert np.all(np.abs(got - f) <= 2.0 ** -24 * np.abs(f - rest) + 256 * EPS * scale)

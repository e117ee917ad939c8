"""Flat tiles (csrc/step_flat.cuh): boxes that take them step bit for bit like the general gather
kernel, for rows shorter and longer than a tile, rows that fill no 16-byte units, last tiles
of few sites, boxes of one row or one slab of rows, and rows that segments divide."""
from functools import lru_cache

import numpy as np
import pytest

from oracle import rflbm_oracle as o
from paper_2507_08820_gb300 import workloads as W

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


SHAPES = [(16, 121, 110), (17, 113, 109), (150, 44, 31), (131, 1, 1600), (401, 503, 1), (100, 50, 51), (30, 93, 91),
          (160, 40, 33), (288, 32, 31), (320, 30, 29), (1000, 2, 131), (250001, 1, 1),
          (83, 77, 75), (100, 70, 66)]
VARIANTS = [dict(kT=1e-4), dict(kT=0.0), dict(kT=1e-4, model=1), dict(kT=0.0, model=1, storage=1), dict(kT=1e-4, storage=1),
            dict(kT=0.0, storage=1), dict(kT=3e-4, storage=2), dict(kT=1e-4, model=1, storage=2)]


@lru_cache(maxsize=1)
def _start(shape):
    rho, u = W.random_fields(*shape, seed=5, drho=0.02, du=0.03)
    return o.equilibrium_state(rho, u) + W.population_perturbation(rho.size, 6, 2e-4)


def _agree(R, shape, kw, steps=(1, 1, 3)):
    import torch
    f0 = torch.tensor(_start(shape), device="cuda")
    n = f0.shape[1]
    out = []
    for kernel in (R.RFLBM_KERNEL_AUTO, R.RFLBM_KERNEL_GATHER):
        box = R.Box(*shape, tau=0.7, seed=3, kernel=kernel, **kw)
        R.rflbm_set_populations(box.h, f0)
        R.rflbm_set_step(box.h, 5)
        snaps = []
        for s in steps:
            R.rflbm_step(box.h, s)
            f = torch.empty((27, n), dtype=torch.float32, device="cuda")
            R.rflbm_get_populations_f32(box.h, f)
            snaps.append(f)
        out.append(snaps)
        box.close()
    for a, b in zip(*out):
        assert torch.equal(a, b), float((a - b).abs().max())


@pytest.mark.parametrize("pattern", [0, 1])
@pytest.mark.parametrize("kw", VARIANTS)
@pytest.mark.parametrize("shape", SHAPES)
def test_flat_tiles_match_the_gather_kernel_bitwise(R, shape, kw, pattern):
    _agree(R, shape, dict(kw, pattern=pattern))


@pytest.mark.parametrize("kw", [dict(kT=1e-4, omega_g=0.7), dict(kT=0.0, omega_g=1.3), dict(kT=1e-4, phi_rho=1),
                                dict(kT=1e-4, omega_g=0.7, phi_rho=1), dict(kT=1e-4, model=1, phi_rho=1)])
@pytest.mark.parametrize("shape", [(83, 77, 75)])
def test_flat_tiles_of_every_variant(R, shape, kw):
    _agree(R, shape, kw)


def test_flat_tiles_report_an_expired_wait(R):
    for kw in (dict(kT=1e-4), dict(kT=1e-4, pattern=1), dict(kT=0.0, storage=1)):
        box = R.Box(150, 50, 40, tau=0.8, **kw)
        R.rflbm_init_rest(box.h)
        R.rflbm_testing_expect_extra_bytes(box.h, 16)
        R.rflbm_step(box.h, 1)
        with pytest.raises(R.RflbmError) as e:
            R.rflbm_synchronize(box.h)
        assert e.value.status == R.RFLBM_ETIMEOUT
        R.rflbm_testing_expect_extra_bytes(box.h, 0)
        R.rflbm_init_rest(box.h)
        R.rflbm_step(box.h, 3)
        st, status = R.rflbm_stats(box.h)
        assert status == R.RFLBM_OK and abs(st.mass - box.n) < 1e-5 * box.n
        box.close()


# without noise flat tiles start at 450,000 sites in float32 and 230,000 in 16-bit storage: the edge geometries above that
# line (the shortest rows, one row of a box, one slab of rows, a single row, a last tile of one site, rows of 30 sites)
STILL_SHAPES = [(16, 121, 240), (17, 113, 240), (131, 1, 3500), (401, 1151, 1), (460033, 1, 1), (30, 160, 96), (100, 50, 91),
                (1002, 2, 231), (150, 44, 70)]


@pytest.mark.parametrize("pattern", [0, 1])
@pytest.mark.parametrize("kw", [dict(), dict(storage=1), dict(storage=2), dict(model=1), dict(model=1, storage=2),
                                dict(omega_g=1.3)])
@pytest.mark.parametrize("shape", STILL_SHAPES)
def test_flat_tiles_without_noise_match_the_gather_kernel_bitwise(R, shape, kw, pattern):
    if pattern == 1 and "omega_g" in kw:
        pytest.skip("AA steps run Reg-FLBM with omega_g = 1, or BGK")
    kw = dict(kw, kT=0.0, pattern=pattern)
    box = R.Box(*shape, tau=0.7, **kw)
    assert R.rflbm_step_path(box.h) == (R.RFLBM_KERNEL_TMA, 0)
    box.close()
    _agree(R, shape, kw)


@pytest.mark.parametrize("shape", [s for s in SHAPES if s[0] not in (288, 320, 1000)])
@pytest.mark.parametrize("kw", [kw for kw in VARIANTS if kw["kT"] > 0])
def test_the_boxes_with_noise_above_run_flat_tiles(R, shape, kw):
    """What the comparisons with the gather kernel rest on (rows in segments of 64 or 96 sites run flat tiles in some
    variants only, rows of 1000 ragged segments)."""
    box = R.Box(*shape, tau=0.7, **kw)
    assert R.rflbm_step_path(box.h) == (R.RFLBM_KERNEL_TMA, 0)
    box.close()

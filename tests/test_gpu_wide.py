"""The kernels that carry FP64 results on float32 and integer pipes (csrc/wide.cuh): initial
fields, moments, global statistics, mode sums and shell sums, at the edges of the ranges where
they change to plain FP64 and at sizes around their blocks, against FP64 numpy.

A population is stored as the float32 g = f - w rho0, so an FP64 export returns it to one FP64
rounding of f, and sums of 27 of them agree with numpy's to 27 roundings of their terms."""
import numpy as np
import pytest

from oracle import rflbm_oracle as o
from paper_2507_08820_gb300 import workloads as W
from test_gpu_diag import _shells_numpy

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


def _state(shape, seed, scale):
    g = np.random.default_rng(seed)
    return scale * g.standard_normal((27, int(np.prod(shape)))) * 10.0 ** g.uniform(-6, 0, (27, int(np.prod(shape))))


@pytest.mark.parametrize("scale", [0.0, 1e-28, 1e-16, 1e-3, 1e20, 1e36])
@pytest.mark.parametrize("shape", [(1, 1, 1), (17, 9, 5), (256, 2, 1)])
def test_moments_match_fp64_sums(R, scale, shape):
    """rho0 = 1e-30 leaves g = f to one rounding, so that the sums of tiny and huge states are
    compared at their own scale (outside 2^-66 .. 2^114 the kernel sums in FP64)."""
    rho0 = 1e-30
    f = _state(shape, 5, scale)
    box = R.Box(*shape, tau=0.8, rho0=rho0)
    R.rflbm_set_populations(box.h, np.ascontiguousarray(f))
    f = box.populations()
    rho, u, pi = box.macroscopic()
    box.close()
    wrho, wu, wpi = o.macroscopic(f)
    s = np.abs(f).sum(axis=0) + 1e-30
    assert np.all(np.abs(rho - wrho) <= 64 * EPS * s)
    assert np.all(np.abs(pi - wpi) <= 64 * EPS * s)
    ok = np.abs(wrho) > 1e-3 * s  # (a quotient by a density that cancels has no digits)
    assert np.all(np.abs(u - wu)[:, ok] <= 1e-10 * (1.0 + np.abs(wu[:, ok])))


def test_moments_of_non_finite_sites(R):
    shape = (32, 3, 2)
    f = o.rest_state(int(np.prod(shape)))
    f[5, 17], f[0, 40] = np.nan, np.inf
    box = R.Box(*shape, tau=0.8)
    R.rflbm_set_populations(box.h, np.ascontiguousarray(f))
    rho, u, pi = box.macroscopic()
    st, status = R.rflbm_stats(box.h)
    box.close()
    assert np.isnan(rho[17]) and np.isinf(rho[40]) and np.all(np.isnan(u[:, 17]))
    others = np.setdiff1d(np.arange(rho.size), [17, 40])
    assert np.all(np.isfinite(rho[others])) and np.all(u[:, others] == 0.0)
    assert status == R.RFLBM_EUNSTABLE and st.nonfinite == 2 and st.max_speed == 0.0


@pytest.mark.parametrize("scale", [0.0, 1e-20, 1e-3, 1e18, 1e31, 1e36])
@pytest.mark.parametrize("shape", [(1, 1, 1), (255, 1, 1), (257, 3, 1), (64, 48, 70)])
def test_statistics_match_fp64_sums(R, scale, shape):
    """Positive populations, so that every site is stable; values of 2^100 and more, and momenta
    outside 2^-40 .. 2^60, take the FP64 branches. The sums of a site are float32."""
    f = np.abs(_state(shape, 7, scale)) + o.weights()[:, None] * 1e-30
    box = R.Box(*shape, tau=0.8, rho0=1e-30)
    R.rflbm_set_populations(box.h, np.ascontiguousarray(f))
    f = box.populations()
    first, status = R.rflbm_stats(box.h)
    st, _ = R.rflbm_stats(box.h)  # the count of finished blocks starts from zero again
    box.close()
    assert status == R.RFLBM_OK and st.nonfinite == 0
    assert (first.mass, list(first.momentum), first.max_speed) == (st.mass, list(st.momentum), st.max_speed)
    rho, u, _ = o.macroscopic(f)
    s = np.abs(f).sum()
    assert abs(st.mass - rho.sum()) <= 27 * 2.0 ** -24 * s
    assert np.all(np.abs(np.array(st.momentum) - (rho * u).sum(axis=1)) <= 27 * 2.0 ** -24 * s)
    speed = np.sqrt((u * u).sum(axis=0)).max()
    assert abs(st.max_speed - speed) <= 60 * 2.0 ** -24 * max(1.0, speed)


@pytest.mark.parametrize("n", [1, 31, 4095, 4096, 4097, 9001])
def test_mode_sums_at_block_edges(R, n):
    f = o.rest_state(n) + W.population_perturbation(n, 9, 1e-3)
    box = R.Box(n, 1, 1, tau=0.8)
    R.rflbm_set_populations(box.h, np.ascontiguousarray(f))
    m = o.moments(box.populations())
    m[0] -= 1.0
    s1, s2 = R.rflbm_mode_sums(box.h)
    box.close()
    # per-site values to 27 float32 roundings of at most sum |g|, then sums of 16 sites in float32
    tol = 64 * 2.0 ** -24 * np.abs(W.population_perturbation(n, 9, 1e-3)).sum(axis=0).max()
    assert np.all(np.abs(s1 - m.sum(axis=1)) <= n * tol)
    assert np.all(np.abs(s2 - (m * m).sum(axis=1)) <= n * tol * np.abs(m).max() * 4)


@pytest.mark.parametrize("shape", [(2, 3, 5), (33, 31, 7), (64, 3, 2), (7, 64, 9), (130, 4, 3), (3, 2, 100),
                                   (768, 3, 1), (2, 5, 770), (11, 26, 8), (35, 9, 2), (1, 1, 6)])
@pytest.mark.parametrize("nshell", [None, 3])
def test_shell_sums_of_uneven_boxes(R, shape, nshell):
    """Spectrum rows shorter and longer than a warp, fewer shells than the box has, every radix of
    the library's transform, its longest edge, and edges it leaves to cuFFT (31, 770)."""
    n = int(np.prod(shape))
    f = o.rest_state(n) + W.population_perturbation(n, 11, 1e-3)
    box = R.Box(*shape, tau=0.8)
    R.rflbm_set_populations(box.h, np.ascontiguousarray(f))
    r, u, pi = o.macroscopic(box.populations())
    ns = R.rflbm_shell_count(box.h)
    for k, phi in ((0, r - 1.0), (2, u[1] * r), (5, pi[1]), (9, pi[5])):
        want_s, want_c = _shells_numpy(phi, shape, ns)
        got_s, got_c = R.rflbm_structure_factor(box.h, k, nshell)
        assert np.array_equal(got_c, want_c[:got_c.size]), k
        assert np.allclose(got_s, want_s[:got_s.size], rtol=1e-5, atol=1e-6 * want_s.max()), k
    box.close()


@pytest.mark.parametrize("scale", [1e-25, 1e-12, 1e-3, 1e15, 1e25])
@pytest.mark.parametrize("shape", [(24, 10, 9), (31, 4, 3)])
def test_structure_factors_at_every_scale(R, scale, shape):
    """Fields whose squares leave the range of float32 (and edges that are none of the library's
    lengths) take cuFFT, usual ones the library's transform."""
    f = _state(shape, 13, scale)
    box = R.Box(*shape, tau=0.8, rho0=1e-30)
    R.rflbm_set_populations(box.h, np.ascontiguousarray(f))
    f = box.populations()
    cx = o.velocities()[:, 0].astype(float)
    ns = R.rflbm_shell_count(box.h)
    got_s, _ = R.rflbm_structure_factor(box.h, 1)
    again, _ = R.rflbm_structure_factor(box.h, 1)
    box.close()
    want_s, _ = _shells_numpy(cx @ f, shape, ns)
    assert np.array_equal(got_s, again)
    assert np.allclose(got_s, want_s, rtol=1e-4, atol=1e-5 * want_s.max())


def test_structure_factor_of_a_fluid_at_rest_is_zero(R):
    box = R.Box(24, 10, 9, tau=0.8)
    R.rflbm_init_rest(box.h)
    s, count = R.rflbm_structure_factor(box.h, 0)
    box.close()
    assert not s.any() and count.sum() == 24 * 10 * 9


def _sites_of_sums():
    """Populations (27, n) whose sums come near the bound of their terms: all equal, of either sign, within 30 % of each
    other, equal where c_x != 0, w_i times one density deviation, and equal values far below one that sets the scale,
    with mantissas near all ones (each part of a split is then near its largest, with one sign)."""
    g = np.random.default_rng(17)
    one = np.ones((27, 1))
    cx = o.velocities()[:, 0][:, None]
    full = 1.0 - 2.0 ** -22
    blocks = [s * v * one for s in (1.0, -1.0) for v in (0.1, 0.12, 0.5, full)]
    blocks += [s * (0.05 * (1.0 + 0.3 * g.uniform(-1.0, 1.0, (27, 400)))) for s in (1.0, -1.0)]
    blocks += [s * v * (cx != 0) for s in (1.0, -1.0) for v in (0.12, full)]
    blocks += [o.weights()[:, None] * g.uniform(-0.1, 0.1, (1, 2000))]
    low = np.repeat(full * 2.0 ** -np.arange(64)[None, :], 27, axis=0)
    low[26] = 0.99
    return np.float64(np.float32(np.concatenate(blocks + [low, -low], axis=1)))


@pytest.mark.parametrize("scale", [2.0 ** -40, 1.0, 2.0 ** 90])
def test_moments_of_sums_near_the_bound_of_their_terms(R, scale):
    """Against FP64 sums at the tolerance of test_moments_match_fp64_sums, in both views of a site."""
    f = scale * _sites_of_sums()
    for pattern in (0, 1):
        box = R.Box(f.shape[1], 1, 1, tau=0.8, rho0=1e-30, pattern=pattern)
        R.rflbm_set_populations(box.h, np.ascontiguousarray(f))
        got = box.populations()
        rho, _, pi = box.macroscopic()
        box.close()
        wrho, _, wpi = o.macroscopic(got)
        s = np.abs(got).sum(axis=0) + 1e-30
        assert np.all(np.abs(rho - wrho) <= 64 * EPS * s)
        assert np.all(np.abs(pi - wpi) <= 64 * EPS * s)


@pytest.mark.parametrize("others", [0.0, 0.1])
def test_initial_fields_where_a_velocity_term_cancels(R, others):
    """Near |u| = 1 the factor 1 - 3 |u| + 3 u^2 of a population is near 1 with large terms. g is the float32
    nearest to f - w rho0 up to the FP64 roundings of f: three of each of the three factors' terms, and four of
    their product with the density and its difference from the rest value."""
    g = np.random.default_rng(23)
    n = 6000
    near = lambda: g.choice([-1.0, 1.0], n) * (1.0 + g.choice([-1.0, 1.0], n) * 2.0 ** -g.uniform(1, 50, n))  # noqa: E731
    u = np.stack([near(), others * g.uniform(-1, 1, n), others * near()])
    for k in range(1, 3):  # every axis
        u[:, k::3] = np.roll(u[:, k::3], k, axis=0)
    rho = np.ones(n)
    box = R.Box(n, 1, 1, tau=0.8)
    R.rflbm_init_field(box.h, rho, np.ascontiguousarray(u))
    got = box.populations()
    box.close()
    w = o.weights()[:, None].astype(np.longdouble)
    v = u.astype(np.longdouble)
    f, size = w * rho, w * rho
    for a, c in enumerate(o.velocities().T):
        c = c[:, None]
        f = f * np.where(c == 0, 1 - 1.5 * v[a] ** 2, 1 + 3 * c * v[a] + 3 * v[a] ** 2)
        size = size * (1 + 3 * np.abs(v[a]) + 3 * v[a] ** 2)
    stored = (got.astype(np.longdouble) - w).astype(np.float32)  # (the export rounds f to FP64)
    tol = 0.5000001 * np.spacing(np.abs(stored)).astype(float) + 16 * EPS * size
    assert np.all(np.abs(stored.astype(np.longdouble) - (f - w)) <= tol)


@pytest.mark.parametrize("unit", [2.0 ** -40, 2.0 ** -22, 2.0 ** 40, 2.0 ** 85])
def test_velocities_are_fp64_quotients(R, unit):
    """Populations of whole units, so that the sums are exact in FP64 and so is their conversion: u is then the quotient of
    the same two numbers, to 2 units in the last place of the correctly rounded one (a reciprocal by Newton steps, a
    quotient corrected once by its remainder). 2^12 to 2^20 units a population; at 2^85 densities pass 2^107."""
    g = np.random.default_rng(29)
    n = 20000
    k = g.integers(2 ** 12, 2 ** 20, (27, n)) * g.choice([-1, 1], (27, n))
    k[:, : n // 2] = np.abs(k[:, : n // 2])  # half of the sites with densities far from zero
    v = k * unit
    f = o.weights()[:, None] + v  # rounds to FP64; g = f - w rho0 is v again in float32
    box = R.Box(n, 1, 1, tau=0.8)
    R.rflbm_set_populations(box.h, np.ascontiguousarray(f))
    rho, u, _ = box.macroscopic()
    box.close()
    wrho = 1.0 + k.sum(axis=0) * unit
    assert np.array_equal(rho, wrho)
    j = (o.velocities().T @ k) * unit
    want = j / wrho
    assert np.all(np.abs(u - want) <= 2 * np.spacing(np.abs(want)))


@pytest.mark.parametrize("rho0,rho,u", [
    (1.0, 1.0, (-666.7065315539121, 335.5127149724657, 134.1717761152097)),
    (0.37, float(np.float32(0.37)), (396.84542754641285, -256.2102318772882, -36.53873304552258)),
    (0.37, float(np.float32(0.37)), (-451.7177706589363, 575.1681675438398, 132.75070061364414)),
    (2.5, 2.5132507072454056, (791.9933978206979, 236.0201251622538, 757.5623402964293)),
    (1e-3, 0.0009941081360488576, (30.00013269037117, -29.999999852552524, 29.999999999686505)),
])
def test_initial_fields_at_large_velocities(R, rho0, rho, u):
    """Sites with a population so near the middle of two float32 values that the error of a form in float32 pairs, larger
    here than for flows, decides between them: the FP64 form rounds to the nearer one, up to its own
    roundings (as in test_initial_fields_where_a_velocity_term_cancels)."""
    box = R.Box(1, 1, 1, tau=0.8, rho0=rho0)
    R.rflbm_init_field(box.h, np.array([rho]), np.array(u)[:, None].copy())
    got = box.populations()[:, 0]
    box.close()
    rho0 = float(np.float32(rho0))
    w = o.weights().astype(np.longdouble)
    f, size = w * rho, w * rho
    for a, c in enumerate(o.velocities().T):
        v = np.longdouble(u[a])
        f = f * np.where(c == 0, 1 - 1.5 * v ** 2, 1 + 3 * c * v + 3 * v ** 2)
        size = size * (1 + 3 * abs(v) + 3 * v ** 2)
    stored = (got.astype(np.longdouble) - w * rho0).astype(np.float32)  # (the export rounds f to FP64)
    tol = 0.5000001 * np.spacing(np.abs(stored)).astype(float) + 16 * EPS * size
    assert np.all(np.abs(stored.astype(np.longdouble) - (f - w * rho0)) <= tol)


@pytest.mark.parametrize("rho0", [1.0, 0.37])
@pytest.mark.parametrize("kind", ["rest", "slow", "near one"])
def test_initial_fields_store_the_spelled_out_fp64_form(R, kind, rho0):
    """Where the pair form leaves sites open, the stored value is the FP64 form's with the roundings that the kernel spells
    out: r psi_x psi_y in turn, then one rounding of its product with psi_z less w rho0 (exact fractions here)."""
    from fractions import Fraction
    g = np.random.default_rng(31)
    n, rho0 = 300, float(np.float32(rho0))
    sign = lambda: g.choice([-1.0, 1.0], (3, n))  # noqa: E731
    u = {"rest": np.zeros((3, n)), "slow": sign() * 10.0 ** g.uniform(-9, -6, (3, n)),
         "near one": np.concatenate([sign()[:1] * (1.0 + sign()[:1] * 2.0 ** -g.uniform(20, 30, (1, n))), np.zeros((2, n))])}[kind]
    rho = rho0 * (1.0 + 1e-9 * g.integers(-1, 2, n))
    box = R.Box(n, 1, 1, tau=0.8, rho0=rho0)
    R.rflbm_init_field(box.h, rho, np.ascontiguousarray(u))
    got = box.populations()
    box.close()
    w1 = {0: 2.0 / 3.0, 1: 1.0 / 6.0, -1: 1.0 / 6.0}
    psi = [{c: 2.0 / 3.0 - v * v if c == 0 else 0.5 * ((1.0 / 3.0 + c * v) + v * v) for c in (-1, 0, 1)} for v in u]
    want = np.empty((27, n))
    for i, (cx, cy, cz) in enumerate(o.velocities().tolist()):
        w = w1[cx] * w1[cy] * w1[cz]
        f = (rho * psi[0][cx]) * psi[1][cy]
        for s in range(n):
            x = Fraction(f[s]) * Fraction(psi[2][cz][s]) - Fraction(w * rho0)
            want[i, s] = float(np.float32(x.numerator / x.denominator)) + w * rho0  # (as the export returns it)
    assert np.array_equal(got, want)

"""The FP64 operator's hops on integer and float limbs at the edges of their range: spinors of very different
magnitude next to one another, zero and tiny and huge ones, and links that are not unitary
(which go through FP64 arithmetic), against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1810_04201_gb300 import gen

pytestmark = pytest.mark.gpu
DIMS, KAPPA = (4, 3, 5, 6), 0.12


def lattice(U, dims=DIMS, recon=18):
    from paper_1810_04201_gb300 import wd
    lat = wd.Lattice(dims)
    lat.set_gauge(U, recon=recon)
    return lat


def apply(lat, psi, dagger=False):
    fo = lat.new_field()
    lat.apply(KAPPA, lat.pack(psi), fo, dagger=dagger)
    return lat.unpack(fo)


def neighbourhood_max(psi, dims):
    """Largest component of each site and its eight neighbours."""
    m = np.abs(psi.view(np.float64)).reshape(*dims[::-1], -1).max(-1)
    out = m.copy()
    for ax in range(4):
        out = np.maximum(out, np.maximum(np.roll(m, 1, ax), np.roll(m, -1, ax)))
    return out.reshape(-1)


@pytest.mark.parametrize("recon", [18, 12])
@pytest.mark.parametrize("decades", [0, 3, 20, 120])
def test_magnitudes_that_differ_between_neighbours(recon, decades):
    """Sites scaled by 10^(+-decades): each site's error is bounded by its own neighbourhood's
    largest component M.  The unit is at most 2 M; the FP32 products are off by 2^-24 of 12 terms
    of 2^-30 units a hop, eight hops at kappa = 0.12 by 2e-15 / 5 M; the FP64 rounding of the oracle
    and of the result stays below the rest of 2e-15 M."""
    U = gen.haar_links(DIMS, seed=3)
    psi = gen.gaussian_source(DIMS, seed=4)
    s = 10.0 ** (decades * (2.0 * gen.uniform(5, gen.STREAM_MISC, 0, psi.shape[0]) - 1.0))
    psi = psi * s[:, None, None]
    lat = lattice(U, recon=recon)
    for dagger in (False, True):
        got = apply(lat, psi, dagger)
        ref = oracle.apply_D(U, psi, KAPPA, DIMS, dagger=dagger)
        err = np.abs(got - ref).reshape(psi.shape[0], -1).max(1)
        assert np.all(err <= 2e-15 * neighbourhood_max(psi, DIMS))


@pytest.mark.parametrize("scale", [1e-306, 1e-290, 1e-269, 1e-260, 1e290, 1e302, 1e304])
def test_scales_at_the_ends_of_the_double_range(scale):
    U = gen.haar_links(DIMS, seed=3)
    psi = gen.gaussian_source(DIMS, seed=4)
    ref = oracle.apply_D(U, psi, KAPPA, DIMS)
    got = apply(lattice(U), psi * scale)
    # multiplying by the scale rounds; subnormal products below 1e-306 lose up to 5e-324 each
    assert oracle.rel_err(got / scale, ref) < (1e-13 if scale > 1e-300 else 1e-12)


def test_zeros_stay_exact():
    """A point source reaches its neighbours and nothing else; with unit links the other
    colours stay exactly zero."""
    psi = gen.point_source(DIMS, 17, 2, 1)
    got = apply(lattice(gen.haar_links(DIMS, seed=3)), psi)
    far = neighbourhood_max(psi, DIMS) == 0
    assert far.any() and np.all(got[far] == 0)
    psi = gen.gaussian_source(DIMS, seed=4)
    psi[:, :, (0, 2)] = 0
    got = apply(lattice(gen.unit_links(DIMS)), psi)
    assert np.all(got[:, :, (0, 2)] == 0)
    assert oracle.rel_err(got, oracle.apply_D(gen.unit_links(DIMS), psi, KAPPA, DIMS)) < 1e-13


@pytest.mark.parametrize("factor", [1.0 + 2.0 ** -13, 1.01, 3.0, 1e-3])
def test_links_that_are_not_unitary(factor):
    U = gen.haar_links(DIMS, seed=3)
    U[2, 7] *= factor
    psi = gen.gaussian_source(DIMS, seed=4)
    lat = lattice(U)
    for dagger in (False, True):
        assert oracle.rel_err(apply(lat, psi, dagger), oracle.apply_D(U, psi, KAPPA, DIMS, dagger=dagger)) < 1e-13


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_non_finite_spinors_reach_their_neighbours_only(bad):
    U = gen.haar_links(DIMS, seed=3)
    psi = gen.gaussian_source(DIMS, seed=4)
    psi[29, 1, 0] = bad
    got = apply(lattice(U), psi)
    near = ~np.isfinite(neighbourhood_max(psi, DIMS))
    clean = psi.copy()
    clean[29, 1, 0] = 0
    ref = oracle.apply_D(U, clean, KAPPA, DIMS)
    assert not np.isfinite(got[near].reshape(near.sum(), -1)).all(1).any()
    assert oracle.rel_err(got[~near], ref[~near]) < 1e-13


@pytest.mark.parametrize("small", [1e-6, 1e-10, 1e-14, 1e-19, 1e-120])
@pytest.mark.parametrize("recon", [18, 12])
def test_colours_far_below_the_others_keep_their_digits(small, recon):
    """Unit links do not mix colours, so every colour is right to its own rounding: what falls below
    2^-14 of the lane's unit is computed with IEEE arithmetic."""
    U = gen.unit_links(DIMS)
    psi = gen.gaussian_source(DIMS, seed=4)
    psi[:, :, 1] *= small
    psi[:, :, 2] *= small ** 2 if small > 1e-100 else 0.0
    lat = lattice(U, recon=recon)
    for dagger in (False, True):
        got, ref = apply(lat, psi, dagger), oracle.apply_D(U, psi, KAPPA, DIMS, dagger=dagger)
        for c in range(3):
            assert np.linalg.norm(got[:, :, c] - ref[:, :, c]) <= 1e-15 * np.linalg.norm(ref[:, :, c])


@pytest.mark.parametrize("spin", range(4))
def test_spins_far_below_the_others_keep_their_digits(spin):
    """The hops into a spin never read the other spin of its chirality, but its lane takes its unit from
    that one too: with only that one large, the spin keeps its own digits."""
    U = gen.haar_links(DIMS, seed=3)
    psi = gen.gaussian_source(DIMS, seed=4)
    psi[:, spin] *= 1e10
    lat = lattice(U)
    for dagger in (False, True):
        got = apply(lat, psi, dagger)[:, spin ^ 1]
        ref = oracle.apply_D(U, psi, KAPPA, DIMS, dagger=dagger)[:, spin ^ 1]
        assert np.linalg.norm(got - ref) <= 1e-15 * np.linalg.norm(ref)


def test_components_above_the_limit_are_within_the_stated_bound():
    """Colours 1e-4 and 1e-2 of the largest on unit links.  A hop is off by at most 2^-56 of the unit
    for its low limb's 24 bits and 2^-57 for the rounding of its sums, eight hops by 24 x 2^-57, and the
    unit is at most twice the largest component of the neighbourhood."""
    U = gen.unit_links(DIMS)
    psi = gen.gaussian_source(DIMS, seed=4)
    psi[:, :, 1] *= 1e-4
    psi[:, :, 2] *= 1e-2
    err = np.abs(apply(lattice(U), psi) - oracle.apply_D(U, psi, KAPPA, DIMS))[:, :, 1].reshape(len(psi), -1).max(1)
    assert np.all(err <= 24 * 2.0 ** -56 * KAPPA * neighbourhood_max(psi, DIMS))


@pytest.mark.parametrize("dims", [DIMS, (16, 8, 8, 8)])
def test_sparse_fields_are_exact_zeros_and_right(dims):
    """One colour of one spin on unit links: most sums are zeros, which are looked at again."""
    U = gen.unit_links(dims)
    psi = gen.gaussian_source(dims, seed=4)
    psi[:, :, 1:] = 0
    psi[:, 1:] = 0
    got, ref = apply(lattice(U, dims), psi), oracle.apply_D(U, psi, KAPPA, dims)
    assert np.all(got[ref == 0] == 0)
    assert oracle.rel_err(got, ref) < 1e-15


def crooked_links(dims, seed):
    """Haar links with two of them scaled: the FP64 kernels keep such links as doubles."""
    U = gen.haar_links(dims, seed=seed)
    U[2, 7] *= 1.2
    U[0, 3] *= 0.9
    return U


@pytest.mark.parametrize("recon", [18, 12])
def test_every_fp64_kernel_on_links_that_are_not_unitary(recon):
    """recon 12 rebuilds row 2 of a scaled link as the square of the scale: its reference has that."""
    from paper_1810_04201_gb300 import wd
    dims = (4, 4, 6, 4)
    U = crooked_links(dims, 3)
    lat = lattice(U, dims, recon)
    if recon == 12:
        U = U.copy()
        U[..., 2, :] = np.cross(U[..., 0, :], U[..., 1, :]).conj()
    B = gen.gaussian_source(dims, seed=4, nrhs=2)
    X = np.stack([oracle.cgnr(U, b, KAPPA, dims, tol=1e-13)[0] for b in B])
    fb = lat.pack(B)
    for kw in (dict(), dict(precondition=1), dict(block=1), dict(inner=1), dict(inner=1, precondition=1), dict(normal_eq=1)):
        fx = lat.new_field(nrhs=2)
        lat.cg(KAPPA, fb, fx, tol=1e-11, nrhs=2, **kw)
        assert oracle.rel_err(lat.unpack(fx, nrhs=2), X) < 1e-9, kw
    fo = lat.new_field()
    lat.normal_apply_noalloc(KAPPA, lat.pack(B[0]), fo)
    assert oracle.rel_err(lat.unpack(fo), oracle.apply_normal(U, B[0], KAPPA, dims)) < 1e-13
    straight = lattice(gen.haar_links(DIMS, seed=5), recon=recon)
    b5 = gen.gaussian_source(DIMS, seed=6)
    xs = [lat.new_field(), straight.new_field()]
    res, st = wd.cg_batched([lat, straight], [KAPPA, KAPPA], [lat.pack(B[0]), straight.pack(b5)], xs, tol=1e-11)
    assert st == 0
    assert oracle.rel_err(lat.unpack(xs[0]), X[0]) < 1e-9
    x5, _ = oracle.cgnr(gen.haar_links(DIMS, seed=5), b5, KAPPA, DIMS, tol=1e-13)
    assert oracle.rel_err(straight.unpack(xs[1]), x5) < 1e-9


def test_fp64_arithmetic_has_its_own_launch_shape():
    """Where the FP64 units bound the operator (links not unitary, recon 8) blocks stay small."""
    dims = (16, 16, 32, 32)
    V = int(np.prod(dims))
    U = np.tile(gen.haar_links((4, 4, 4, 4), seed=9), (1, V // 256, 1, 1))
    lat = lattice(U, dims)
    assert lat.tiles(0, 1) == (256, 1, 1)
    lat.set_gauge(U, recon=8)
    assert lat.tiles(0, 1) == (64, 1, 1)
    U[2, 7] *= 1.2
    lat.set_gauge(U)
    assert lat.tiles(0, 1) == (64, 1, 1)
    lat.set_gauge(U, recon=12)
    assert lat.tiles(0, 1) == (64, 1, 1)


def spread(psi, decades, seed):
    """psi with its sites scaled by 10^(+-decades)."""
    s = 10.0 ** (decades * (2.0 * gen.uniform(seed, gen.STREAM_MISC, 0, psi.shape[0]) - 1.0))
    return psi * s[:, None, None]


def test_rows_of_very_different_magnitude():
    """Three right-hand sides, each in its own units: the bound of each site in its own row."""
    U = gen.haar_links(DIMS, seed=3)
    B = gen.gaussian_source(DIMS, seed=4, nrhs=3)
    B = np.stack([spread(B[0], 20, 5), B[1] * 1e-200, spread(B[2], 3, 6) * 1e200])
    lat = lattice(U)
    fo = lat.new_field(nrhs=3)
    lat.apply(KAPPA, lat.pack(B), fo, nrhs=3)
    got = lat.unpack(fo, nrhs=3, squeeze=False)
    for k in range(3):
        err = np.abs(got[k] - oracle.apply_D(U, B[k], KAPPA, DIMS)).reshape(len(B[k]), -1).max(1)
        assert np.all(err <= 2e-15 * neighbourhood_max(B[k], DIMS))


@pytest.mark.parametrize("decades", [0, 3, 20])
@pytest.mark.parametrize("bad_link", [False, True])
def test_checkerboard_hops_of_different_magnitudes(decades, bad_link):
    """The even-odd operator 1 - kappa^2 H_eo H_oe on sites of very different magnitude, unitary
    links and not: D on the even field gives the odd half -kappa H_oe, D on that the even half; two
    hops, each with the bound above (2e-15 of the largest value within two sites)."""
    dims = (4, 4, 2, 6)
    U = gen.haar_links(dims, seed=3)
    if bad_link:
        U[1, 9] *= 1.5
    psi = spread(gen.gaussian_source(dims, seed=4), decades, 5)
    x, y, z, t = np.meshgrid(*[np.arange(n) for n in dims], indexing="ij")
    odd = ((x + y + z + t) & 1).transpose(3, 2, 1, 0).reshape(-1).astype(bool)
    even_in = np.where(odd[:, None, None], 0.0, psi)
    lat = lattice(U, dims)
    for dagger in (False, True):
        fo = lat.new_field()
        lat.apply_schur(KAPPA, lat.pack(psi), fo, dagger=dagger)
        got = lat.unpack(fo)
        # D takes an even field to -kappa H_oe of it on the odd sites, and that to kappa^2 H_eo H_oe
        h = oracle.apply_D(U, even_in, KAPPA, dims, dagger=dagger)
        h[~odd] = 0
        want = even_in - oracle.apply_D(U, h, KAPPA, dims, dagger=dagger)
        near = neighbourhood_max(even_in, dims).reshape(*dims[::-1])
        near2 = near.copy()
        for ax in range(4):
            near2 = np.maximum(near2, np.maximum(np.roll(near, 1, ax), np.roll(near, -1, ax)))
        err = np.abs(got - want).reshape(len(psi), -1).max(1)
        assert np.all(err[~odd] <= 4e-15 * near2.reshape(-1)[~odd])
        assert np.all(got[odd] == 0)

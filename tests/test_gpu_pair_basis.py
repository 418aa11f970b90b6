"""The Legendre kernels' own edges (parity-pair basis, blocks of 16 steps, tiles of
ring pairs), against the oracle: J = (lmax - m) / 2 + 1 around multiples of 16, a
partial warp of ring pairs, the forms of the recurrence and, in FP32, more ring pairs
than one tile of the analysis holds.  Tolerances as in the tests of the transforms,
relative to the largest output: 1e-12 in FP64, u (64 + 2 nside sqrt(lmax+1)) in FP32."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TOL64 = 1e-12
U = 2.0 ** -24


def tol32(nside, lmax):
    return U * (64.0 + 2.0 * nside * np.sqrt(lmax + 1.0))


# (11, 32): 17 steps at m = 0; (21, 62): a partial second block, 42 pairs;
# (100, 66): 200 pairs, the last tile of the synthesis in the equatorial form;
# (50, 30) and (50, 31): exactly one block at m = 0
SMALL = [(11, 32), (21, 62), (50, 30), (50, 31), (100, 66)]


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1702_08852_gb300 import build
    build.build()
    return torch


def rand_alm(lmax, seed):
    from paper_1702_08852_gb300 import inputs
    rng = np.random.default_rng(seed)
    n = inputs.nalm(lmax)
    a = rng.standard_normal(n) + 1j * rng.standard_normal(n)
    _, ms = inputs.lm_of_slots(lmax)
    a[ms == 0] = a[ms == 0].real
    return a


@pytest.mark.parametrize("nside,lmax", SMALL)
def test_block_and_tile_edges(torch_cuda, osht, nside, lmax):
    torch = torch_cuda
    from paper_1702_08852_gb300 import wf
    a = rand_alm(lmax, nside + lmax)
    m = np.random.default_rng(nside * lmax).standard_normal(12 * nside * nside)
    ref, refb = osht.alm2map(a, nside, lmax), osht.map2alm(m, nside, lmax)
    with wf.Plan(nside, lmax, np.ones(lmax + 1)) as p:
        got = p.alm2map(torch.from_numpy(a).cuda()).cpu().numpy()
        gotb = p.map2alm(torch.from_numpy(m).cuda()).cpu().numpy()
        got32 = p.alm2map_f32(torch.from_numpy(a).cuda()).cpu().numpy()
        got32b = p.map2alm_f32(torch.from_numpy(m).cuda()).cpu().numpy()
    t32 = tol32(nside, lmax)
    assert np.max(np.abs(got - ref)) <= TOL64 * np.max(np.abs(ref))
    assert np.max(np.abs(gotb - refb)) <= TOL64 * np.max(np.abs(refb))
    assert np.max(np.abs(got32 - ref)) <= t32 * np.max(np.abs(ref))
    assert np.max(np.abs(got32b - refb)) <= t32 * np.max(np.abs(refb))


def test_more_pairs_than_a_tile(torch_cuda, osht):
    """Nside 1030: 2060 ring pairs, so the analysis adds up two tiles."""
    torch = torch_cuda
    from paper_1702_08852_gb300 import wf, inputs
    nside, lmax = 1030, 6
    npix = 12 * nside * nside
    a = rand_alm(lmax, 3)
    rng = np.random.default_rng(4)
    m = rng.standard_normal(npix)
    pix = np.concatenate([rng.integers(0, npix, 40), [0, 3, npix - 1, npix // 2]])
    ref = osht.alm2map_pixels(a, nside, lmax, pix)
    ls, ms = inputs.lm_of_slots(lmax)
    refb = 4 * np.pi / npix * osht.adjoint_modes(m, nside, lmax, ls, ms)
    with wf.Plan(nside, lmax, np.ones(lmax + 1)) as p:
        got = p.alm2map_f32(torch.from_numpy(a).cuda()).cpu().numpy()
        gotb = p.map2alm_f32(torch.from_numpy(m).cuda()).cpu().numpy()
    assert np.max(np.abs(got[pix] - ref)) <= tol32(nside, lmax) * np.max(np.abs(got))
    assert np.max(np.abs(gotb - refb)) <= tol32(nside, lmax) * np.max(np.abs(refb))

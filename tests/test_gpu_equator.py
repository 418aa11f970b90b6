"""Accuracy on the rings next to the equator, ring by ring.

There Q_j = lam / z of the parity-pair basis amplifies rounding by up to 1/z, so the
Legendre kernels switch to the one-step recurrence; the norm over a whole map does not
show whether they do.  Its lmax + 1 steps each leave a rounding of at most u of an O(1)
value, in a recurrence that neither grows nor shrinks there, and the sums as many again:
they add like a random walk, so the error is held to 4 u sqrt(lmax + 1) of the rms.  u is
2^-53 in FP64, 2^-24 in FP32 and 2^-47 in double-float (an operation's bound)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

UNIT = {"f64": 2.0 ** -53, "f32": 2.0 ** -24, "df64": 2.0 ** -47}


def tol(prec, lmax):
    return 4.0 * UNIT[prec] * np.sqrt(lmax + 1.0)


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


def walk(osht, nside, lmax, i):
    """(l, lam_lm(z) of m = 0 .. l) for l = 0 .. lmax on ring i, the textbook recurrence in
    long double, from the oracle's lam_mm (its rounding scales a whole m and is not the
    recurrence's)."""
    ld = np.longdouble
    m = np.arange(lmax + 1, dtype=ld)
    _, _, z, sth, _ = osht.ring_info(nside, i)
    z = ld(z)
    k = np.arange(lmax + 1)
    mm = osht.lambda_all(lmax, z, sth)[osht.alm_index(lmax, k, k)].astype(ld)
    prev, cur = np.zeros(lmax + 1, ld), np.zeros(lmax + 1, ld)
    cur[0] = mm[0]
    yield 0, cur[:1]
    for l in range(1, lmax + 1):
        k = m[:l]
        a = np.sqrt((4 * ld(l) * l - 1) / (ld(l) * l - k * k))
        b = np.sqrt(((ld(l) - 1) ** 2 - k * k) / (4 * (ld(l) - 1) ** 2 - 1))
        nxt = np.zeros(lmax + 1, ld)
        nxt[:l] = a * (z * cur[:l] - b * prev[:l])
        nxt[l] = mm[l]
        prev, cur = cur, nxt
        yield l, cur[:l + 1]


def slots(lmax, l):
    m = np.arange(l + 1)
    return m * (2 * lmax + 1 - m) // 2 + l


def ring(nside, i):
    """(first pixel, phase step num: phi_0 = pi num / (4 nside)) of the belt's ring i
    (nside <= i <= 3 nside), 4 nside pixels."""
    return 2 * nside * (nside - 1) + (i - nside) * 4 * nside, 0 if (i + nside) & 1 else 1


def phase(nside, lmax, num):
    m = np.arange(lmax + 1)
    return np.exp(1j * np.pi * ((m * num) % (8 * nside)) / (4.0 * nside))


def synth_rings(osht, a, nside, lmax, i):
    """The belt's rings i and 4 nside - i (i <= 2 nside) of Y a."""
    _, num = ring(nside, i)
    f = np.zeros((2, lmax + 1), np.clongdouble)
    for l, lam in walk(osht, nside, lmax, i):
        v = lam * a[slots(lmax, l)]
        s = 1 - 2 * ((np.arange(l + 1) + l) & 1)
        f[0, :l + 1] += v
        f[1, :l + 1] += s * v
    f = f.astype(np.complex128) * phase(nside, lmax, num)
    n = 4 * nside
    out = []
    for row in f:
        c = np.zeros(n, complex)
        np.add.at(c, np.arange(lmax + 1) % n, row)
        np.add.at(c, -np.arange(1, lmax + 1) % n, row[1:].conj())
        out.append((np.fft.ifft(c) * n).real)
    return out


def check_synthesis(torch, osht, prec, nside, lmax, variant=None, rings=None):
    from paper_1702_08852_gb300 import wf
    a = rand_alm(lmax, nside + lmax)
    rings = rings or [2 * nside, 2 * nside - 1, 2 * nside - 2, 2 * nside - 4]
    with wf.Plan(nside, lmax, np.ones(lmax + 1)) as p:
        if variant:
            p.set_tuning(**variant)
        f = {"f64": p.alm2map, "f32": p.alm2map_f32, "df64": p.alm2map_df64}[prec]
        got = f(torch.from_numpy(a).cuda()).cpu().numpy()
    for i in rings:
        for j, ref in zip((i, 4 * nside - i), synth_rings(osht, a, nside, lmax, i)):
            first = ring(nside, j)[0]
            err = got[first:first + 4 * nside] - ref
            assert np.sqrt(np.mean(err ** 2)) <= tol(prec, lmax) * np.sqrt(np.mean(ref ** 2)), j


# whole warps of pairs from the equator on (64, 128, 192), a part of one (75), the pairs
# per thread that a plan may run
@pytest.mark.parametrize("nside,lmax", [(64, 128), (75, 150), (128, 256), (192, 384), (512, 1024)])
@pytest.mark.parametrize("np_", [1, 2, 4])
def test_synthesis_f64(torch_cuda, osht, nside, lmax, np_):
    check_synthesis(torch_cuda, osht, "f64", nside, lmax, {"syn_np": [np_, 2]})


@pytest.mark.parametrize("nside,lmax", [(75, 150), (128, 256), (192, 384)])
def test_synthesis_df64(torch_cuda, osht, nside, lmax):
    check_synthesis(torch_cuda, osht, "df64", nside, lmax)


@pytest.mark.parametrize("nside,lmax", [(64, 128), (75, 150), (128, 256), (256, 512), (512, 1024)])
@pytest.mark.parametrize("np_", [1, 2, 4])
def test_synthesis_f32(torch_cuda, osht, nside, lmax, np_):
    check_synthesis(torch_cuda, osht, "f32", nside, lmax, {"syn_np": [1, np_]})


def strip(nside, seed):
    """A map that is zero but on the equator and the four rings on each side of it."""
    m = np.zeros(12 * nside * nside)
    a, b = ring(nside, 2 * nside - 4)[0], ring(nside, 2 * nside + 5)[0]
    m[a:b] = np.random.default_rng(seed).standard_normal(b - a)
    return m


def analyse_strip(osht, m, nside, lmax):
    from paper_1702_08852_gb300 import inputs
    out = np.zeros(inputs.nalm(lmax), np.clongdouble)
    n = 4 * nside
    for i in range(2 * nside - 4, 2 * nside + 1):
        g = []
        for j in sorted({i, 4 * nside - i}):
            first, num = ring(nside, j)
            x = np.fft.fft(m[first:first + n])
            g.append(x[np.arange(lmax + 1) % n] * phase(nside, lmax, num).conj())
        for l, lam in walk(osht, nside, lmax, i):
            s = 1 - 2 * ((np.arange(l + 1) + l) & 1)
            v = g[0][:l + 1] + (s * g[1][:l + 1] if len(g) > 1 else 0)
            out[slots(lmax, l)] += lam * v
    return (4 * np.pi / m.size * out).astype(np.complex128)


# (64, 128) .. (256, 512): whole warps of equatorial pairs; 75: a part of one; 16: a
# few pairs; 4: every pair
@pytest.mark.parametrize("nside,lmax", [(4, 9), (16, 33), (64, 128), (75, 150), (256, 512)])
@pytest.mark.parametrize("prec", ["f64", "f32", "df64"])
def test_analysis(torch_cuda, osht, prec, nside, lmax):
    torch = torch_cuda
    from paper_1702_08852_gb300 import wf
    m = strip(nside, nside + lmax)
    with wf.Plan(nside, lmax, np.ones(lmax + 1)) as p:
        f = {"f64": p.map2alm, "f32": p.map2alm_f32, "df64": p.map2alm_df64}[prec]
        got = f(torch.from_numpy(m).cuda()).cpu().numpy()
    ref = analyse_strip(osht, m, nside, lmax)
    assert np.linalg.norm(got - ref) <= tol(prec, lmax) * np.linalg.norm(ref)


# the first rings of the belt (z = 2/3): the recurrence's form for their z^2, whatever
# other pairs their thread, warp or CTA holds
FORMS = [(p, n, l, k) for p, n, l in [("f64", 128, 256), ("f64", 512, 1024), ("f32", 128, 256)]
         for k in (1, 2, 4)] + [("df64", 512, 1024, 1)]


@pytest.mark.parametrize("prec,nside,lmax,np_", FORMS)
def test_form_of_each_pair(torch_cuda, osht, prec, nside, lmax, np_):
    check_synthesis(torch_cuda, osht, prec, nside, lmax, {"syn_np": [np_, np_]},
                    [nside, nside + 1, nside + nside // 8])


def test_half_tiles(torch_cuda):
    """Nside 1024, lmax 2600: the FP64 and double-float analysis take the ring pairs in two
    halves; the coefficients that a plan of lmax 2048 has (one tile) are the same but for
    the order of the sums, 2048 pairs' roundings at random."""
    torch = torch_cuda
    from paper_1702_08852_gb300 import wf
    nside, l0, l1 = 1024, 2048, 2600
    m = torch.from_numpy(np.random.default_rng(3).standard_normal(12 * nside * nside)).cuda()
    out = []
    for lmax in (l0, l1):
        with wf.Plan(nside, lmax, np.ones(lmax + 1)) as p:
            out.append([f(m).cpu().numpy() for f in (p.map2alm, p.map2alm_df64)])
    i, j = (np.concatenate([slots(lmax, l) for l in range(l0 + 1)]) for lmax in (l0, l1))
    for a, b, u in zip(out[0], out[1], (UNIT["f64"], UNIT["df64"])):
        assert np.linalg.norm(a[i] - b[j]) <= 4 * u * np.sqrt(2048) * np.linalg.norm(a)


def test_small_terms_f32(torch_cuda, osht):
    """Terms between 2^-100 and 2^-80 count in FP32 too: m = 20 on the ring next to the
    pole, where lam_lm first reaches 2^-99 at l = 41 and 2^-92 at l = 51, the end of the
    analysis' first block.  Tolerance as for the FP32 transforms, of each coefficient."""
    torch = torch_cuda
    from paper_1702_08852_gb300 import wf
    nside, lmax = 64, 128
    m = np.zeros(12 * nside * nside)
    m[:4] = [1.0, -2.0, 0.5, 3.0]
    ls = np.arange(44, 52)
    ms = np.full(ls.size, 20)
    ref = 4 * np.pi / m.size * osht.adjoint_modes(m, nside, lmax, ls, ms)
    with wf.Plan(nside, lmax, np.ones(lmax + 1)) as p:
        got = p.map2alm_f32(torch.from_numpy(m).cuda()).cpu().numpy()
    err = np.abs(got[ms * (2 * lmax + 1 - ms) // 2 + ls] - ref)
    assert np.all(err <= UNIT["f32"] * (64 + 2 * nside * np.sqrt(lmax + 1.0)) * np.abs(ref))


def test_large_plan(torch_cuda):
    """Nside 2048: only the FP32 ring FFTs fit shared memory, so a plan has no FP64
    checkpoints.  Without them it holds 6.2 GB (maps 1.4, ring coefficients 0.8, chirps 1.4,
    FP32 checkpoints 2.2 and less than half a GB of others), with them 10.7 GB."""
    torch = torch_cuda
    from paper_1702_08852_gb300 import wf
    nside, lmax = 2048, 2048
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    with wf.Plan(nside, lmax, np.ones(lmax + 1)) as p:
        assert free - torch.cuda.mem_get_info()[0] < 8.5e9
        a = torch.zeros(p.nalm, dtype=torch.complex128, device="cuda")
        a[3] = 1.0  # l = 3, m = 0
        with pytest.raises(wf.WFError) as e:
            p.alm2map(a)
        assert e.value.status == wf.WF_ERR_CUDA
        m = p.alm2map_f32(a)
        b = p.map2alm_f32(m)
        assert torch.linalg.vector_norm(b - a) < 1e-3  # quadrature


def test_synthesis_in_separate_blocks(torch_cuda):
    """Nside 1024, lmax 2600: too much shared memory for both kinds of pairs in a block of
    the FP32 synthesis.  A field of l <= 2048 comes out as from the plan of lmax 2048, whose
    blocks are common: the same sums."""
    torch = torch_cuda
    from paper_1702_08852_gb300 import wf
    nside, l0, l1 = 1024, 2048, 2600
    a = rand_alm(l0, 5)
    b = np.zeros((l1 + 1) * (l1 + 2) // 2, complex)
    for l in range(l0 + 1):
        b[slots(l1, l)] = a[slots(l0, l)]
    out = []
    for lmax, x in ((l0, a), (l1, b)):
        with wf.Plan(nside, lmax, np.ones(lmax + 1)) as p:
            out.append(p.alm2map_f32(torch.from_numpy(x).cuda()))
    assert torch.linalg.vector_norm(out[0] - out[1]) <= UNIT["f32"] * torch.linalg.vector_norm(out[0])

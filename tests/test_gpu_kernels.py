"""Kernels at the edges of their ranges (tile remainders, chunk borders, the
smallest and largest sizes of a dispatch rule) against the FP64 oracle or
against the general path, through the C ABI."""
import numpy as np
import pytest

import synth
from oracle import dda as odda

from _cases import Case, random_case

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda"
EPS = 2.0 ** -53


@pytest.fixture(scope="module")
def dda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0908_0863_gb300 as m
    return m


# ------------------------------------------------ incident field, cross sections

# rows of 1 to 512 sites (lattices of one x site take their rows along y), fewer
# and more sites than a CTA's threads, and 40,000 and 160,000 rows (the latter
# more than one round of 512 rows x 304 CTAs)
@pytest.mark.parametrize("shape,fill", [((1, 1, 1), 1.0), ((129, 3, 2), 0.5), ((512, 2, 3), 0.3), ((33, 17, 5), 0.6),
                                        ((3, 200, 200), 0.4), ((1, 400, 400), 0.3), ((2, 400, 400), 0.1),
                                        ((512, 1, 9), 0.8)])
def test_incident_field_edges(dda, shape, fill):
    case = random_case(shape, seed=sum(shape), fill=fill, two_materials=False)
    kh = synth.random_direction(7)[0]
    e = np.array([0.3 + 0.1j, -0.5j, 0.7])
    with case.lattice() as lat:
        E = torch.empty((3, case.nd), dtype=torch.complex128, device=DEV)
        lat.incident_field(kh, e, E)
        ref = odda.incident_field(case.coords, case.k, kh, e)
        # the phase is an FP64 angle of up to k sum(n): its own rounding on
        # both sides (three products and sums), plus the complex products
        bound = 8 * EPS * (1.0 + case.k * sum(shape))
        assert np.abs(E.cpu().numpy() - ref).max() <= bound * np.abs(e).sum()


# right-hand sides below, at and above the 32 of one launch
@pytest.mark.parametrize("two", [False, True])
@pytest.mark.parametrize("nb", [1, 32, 33, 70])
def test_cross_sections_batches(dda, nb, two):
    case = random_case((9, 7, 11), seed=nb, fill=0.7, two_materials=two)
    E = synth.complex_normal(nb, (nb, 3, case.nd))
    P = (0.2 - 0.1j) * E + 0.05 * synth.complex_normal(nb + 1, (nb, 3, case.nd))
    with case.lattice() as lat:
        got = lat.cross_sections_batch(torch.from_numpy(E).to(DEV), torch.from_numpy(P).to(DEV))
    for b in range(nb):
        ext, ab = odda.c_ext(E[b], P[b], case.k), odda.c_abs(case.ainv, P[b], case.k)
        # sums of 3 N_d terms of either sign: their rounding is below N_d eps times the sum of their sizes
        f = 4 * np.pi * case.k * EPS * 6 * case.nd
        w = np.abs(case.ainv.T.imag) + case.k**3
        assert abs(got[b, 0] - ext) <= f * np.abs(E[b] * P[b]).sum()
        assert abs(got[b, 1] - ab) <= f * (w * np.abs(P[b]) ** 2).sum()
        assert got[b, 2] == got[b, 0] - got[b, 1]


# a right-hand side's sums are added in one order, alone or at any place of a
# batch (21,600 dipoles or 24,000 sites: 43 and 94 blocks a right-hand side)
@pytest.mark.parametrize("two", [False, True])
@pytest.mark.parametrize("nb", [2, 32, 33, 40])
def test_cross_sections_do_not_depend_on_the_batch(dda, nb, two):
    case = random_case((40, 30, 20), seed=nb, fill=0.9, two_materials=two)
    E = torch.from_numpy(synth.complex_normal(nb, (nb, 3, case.nd))).to(DEV)
    P = (0.2 - 0.1j) * E + 0.05 * torch.from_numpy(synth.complex_normal(nb + 1, (nb, 3, case.nd))).to(DEV)
    with case.lattice() as lat:
        got = lat.cross_sections_batch(E, P)
        for b in range(nb):
            assert np.array_equal(got[b], lat.cross_sections(E[b], P[b])), b


# ------------------------------------------------------ dependent launches

# products queued back to back with other work of the same stream between
# them, on the current stream and on another one: the passes may be scheduled
# early but must see all earlier writes
@pytest.mark.parametrize("side", [False, True])
@pytest.mark.parametrize("shape", [(6, 5, 4), (40, 24, 33)])
def test_products_in_stream_order(dda, shape, side):
    case = random_case(shape, seed=3, fill=0.8)
    with case.lattice() as lat:
        p0 = torch.from_numpy(synth.complex_normal(5, (3, case.nd), np.complex64)).to(DEV)
        torch.cuda.synchronize()
        want, p = [], p0.clone()
        for _ in range(6):
            y = torch.empty_like(p)
            lat.matvec(p, y)
            torch.cuda.synchronize()
            want.append(y.clone())
            p = y * 0.25
            torch.cuda.synchronize()
        stream = torch.cuda.Stream() if side else torch.cuda.current_stream()
        with torch.cuda.stream(stream):
            got, p = [], p0.clone()
            for _ in range(6):
                y = torch.empty_like(p)
                lat.matvec(p, y)
                got.append(y.clone())
                p = y * 0.25
        stream.synchronize()
        for a, b in zip(got, want):
            assert torch.equal(a, b)


# products that read the previous product's output with nothing between them,
# in all three arithmetics, against the same sequence replayed from a captured
# graph, where every pass is an ordinary launch.  (64, 64, 48) is just below
# the block limit of dependent launches in the complex64 x passes (4608 of
# 4864) and (64, 64, 52) just above it, with the other passes below; a batch
# of five takes the 16-byte arithmetics through several chunks, each one's last
# pass followed by the first of the next
@pytest.mark.parametrize("shape,nb", [((6, 5, 4), 1), ((6, 5, 4), 5), ((40, 24, 33), 1), ((40, 24, 33), 3),
                                      ((64, 64, 48), 1), ((64, 64, 52), 1), ((17, 60, 49), 5)])
@pytest.mark.parametrize("dtype", ["c64", "c128", "c128df"])
def test_dependent_products_equal_captured(dda, shape, nb, dtype):
    case = random_case(shape, seed=nb, fill=0.8)
    real = np.complex64 if dtype == "c64" else np.complex128
    kind = "c128df" if dtype == "c128df" else None
    with case.lattice() as lat:
        p = torch.from_numpy(synth.complex_normal(6, (nb, 3, case.nd), real)).to(DEV)
        a, b = torch.empty_like(p), torch.empty_like(p)

        def chain():
            dda.dda_matvec_batch(lat.ctx, p, a, dtype=kind)
            for _ in range(3):
                dda.dda_matvec_batch(lat.ctx, a, b, dtype=kind)
                dda.dda_matvec_batch(lat.ctx, b, a, dtype=kind)

        chain()   # the workspace grows here, not under capture
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            chain()
        graph.replay()
        torch.cuda.synchronize()
        want = a.clone(), b.clone()
        assert torch.isfinite(torch.view_as_real(want[0])).all()
        for _ in range(4):
            a.zero_()
            b.zero_()
            chain()
            torch.cuda.synchronize()
            assert torch.equal(a, want[0]) and torch.equal(b, want[1])


# ------------------------------------------------------------ double-float

# vectors below, at the lower end of and inside the range that is split and
# widened on the integer units (2^-70 .. 2^126; products of larger vectors leave
# the range of a float), of both signs with exact zeros
@pytest.mark.parametrize("exponent", [-90, -71, -70, -66, 0, 60, 100, 112])
def test_double_float_product_scales(dda, exponent):
    case = random_case((6, 5, 7), seed=11, fill=0.7)
    p = synth.complex_normal(12, (3, case.nd))
    p[:, ::3] = 0.0
    p[:, 1::3] *= 2.0 ** -20   # entries of two sizes
    p *= 2.0 ** exponent
    with case.lattice() as lat:
        x = torch.from_numpy(p).to(DEV)
        y, z = torch.empty_like(x), torch.empty_like(x)
        lat.matvec(x, y)
        dda.dda_matvec(lat.ctx, x, z, dtype="c128df")
    # five times the 2e-15 of this lattice, three times what the largest show
    assert float((z - y).norm() / y.norm()) <= 1e-14


# short x rows share a CTA for 8-byte reals; z counts that do not fill it
@pytest.mark.parametrize("K", [1, 2, 4, 7, 16, 32])
@pytest.mark.parametrize("P", [1, 3, 17])
def test_short_rows(dda, K, P):
    case = random_case((K, 3, P), seed=K + P, fill=0.9)
    p = synth.complex_normal(K * P, (3, case.nd))
    ref = odda.direct_matvec(case.coords, case.ainv, case.k, p)
    with case.lattice() as lat:
        x = torch.from_numpy(p).to(DEV)
        for dtype, tol in ((None, 1e-13), ("c128df", 1e-12)):
            y = torch.empty_like(x)
            dda.dda_matvec(lat.ctx, x, y, dtype=dtype)
            assert np.abs(y.cpu().numpy() - ref).max() <= tol * np.abs(ref).max()


# fewer z tiles than a CTA of the x passes holds (it then has those alone), as
# many, and one more, in batches
@pytest.mark.parametrize("K", [2, 6, 14, 50])
@pytest.mark.parametrize("P", [1, 2, 5, 8, 9, 33])
@pytest.mark.parametrize("dtype", ["c64", "c128", "c128df"])
def test_few_z_tiles(dda, K, P, dtype):
    case = random_case((K, 5, P), seed=K * P, fill=0.9)
    p = synth.complex_normal(K + P, (3, 3, case.nd), np.complex64 if dtype == "c64" else np.complex128)
    ref = np.stack([odda.direct_matvec(case.coords, case.ainv, case.k, q.astype(np.complex128)) for q in p])
    with case.lattice() as lat:
        x = torch.from_numpy(p).to(DEV)
        y = torch.empty_like(x)
        dda.dda_matvec_batch(lat.ctx, x, y, dtype="c128df" if dtype == "c128df" else None)
    tol = {"c64": 2e-6, "c128": 1e-13, "c128df": 1e-12}[dtype]
    assert np.abs(y.cpu().numpy() - ref).max() <= tol * np.abs(ref).max()


# --------------------------------------------------------- tensor spectrum

# every component against its own size, lines of one site among them.  Each
# component by itself is within 4.2e-16 of the reference's transform; where two
# shared one, the smaller was off by up to 7.7e-16.  A component that is odd on
# an axis of one site vanishes exactly.
@pytest.mark.parametrize("shape", [(1, 7, 3), (13, 1, 5), (6, 5, 1), (2, 2, 1), (40, 24, 9), (9, 33, 65)])
def test_tensor_spectrum_components(dda, shape):
    from oracle import circulant
    K, J, P = shape
    k = 0.7
    case = Case(np.ones((P, J, K), dtype=np.uint8), [1.5 + 0.1j], k)
    L = tuple(circulant.padded_length(v) for v in shape)
    half = circulant.half_spectrum(circulant.tensor_section1(k, K, J, P), L) / (L[0] * L[1] * L[2])
    half = np.ascontiguousarray(half.transpose(2, 3, 1, 0))
    with case.lattice() as lat:
        out = torch.empty(half.shape, dtype=torch.complex128, device=DEV)
        lat.tensor_spectrum(out)
        got = out.cpu().numpy()
    for q, odd in enumerate([(), (0, 1), (0, 2), (), (1, 2), ()]):   # xx, xy, xz, yy, yz, zz
        g, h = got[..., q], half[..., q]
        if any(shape[a] == 1 for a in odd):
            assert not g.any()
        else:
            assert np.linalg.norm(g - h) <= 5e-16 * np.linalg.norm(h)


# ------------------------------------------------- z pass, split columns

# 128-point columns at the ends of their site counts (and the lengths either
# side, which keep the general kernels), lattices of one x site (fewer columns
# than a CTA holds) up to several CTAs, tile widths below and above a warp's
# two columns, a batch
@pytest.mark.parametrize("P", [48, 49, 57, 64, 65])
@pytest.mark.parametrize("K,J", [(1, 1), (3, 2), (9, 5)])
def test_split_columns(dda, P, K, J):
    case = random_case((K, J, P), seed=P + K, fill=0.8)
    p = synth.complex_normal(P * K, (2, 3, case.nd), np.complex64)
    ref = np.stack([odda.direct_matvec(case.coords, case.ainv, case.k, q.astype(np.complex128)) for q in p])
    with case.lattice() as lat:
        assert (lat.padded[2] == 128) == (49 <= P <= 64)
        x = torch.from_numpy(p).to(DEV)
        got, t0 = [], list(lat.tiles("c64"))
        for width in ((0, t0[1], t0[1] + 2) if lat.padded[2] == 128 else (t0[1],) * 3):
            lat.tiles("c64", [t0[0], width, t0[2]])
            y = torch.empty_like(x)
            lat.matvec_batch(x, y)
            got.append(y)
        assert np.abs(got[0].cpu().numpy() - ref).max() <= 2e-6 * np.abs(ref).max()
        assert torch.equal(got[0], got[1]) and torch.equal(got[0], got[2])


"""The FP64 apply in fixed point (csrc/dslash_fx.cu): at the sizes where its
split of the hop list changes, on site ranges, with fields that span many
orders of magnitude, with links that are not unitary, and with infinities and
NaN (where it runs the FP64 loop), against the oracle.

Tolerance: every row is known to about 2^-54 of its class's largest neighbour,
the final FP64 operations round a few times: 1e-15 of the largest result, and
4e-15 of each site's own largest component (weights 1/16 to 1/432 times up to
32 hops a class)."""
import numpy as np
import pytest
import torch

import oracle
from paper_1012_3615_gb300 import Brillouin, synth

pytestmark = pytest.mark.gpu
AP = (1, 1, 1, -1)


def _op(L, U, gpu):
    """the operator, and its 81 fields in the oracle's order (W_{-d}(x) = W_d(x - d)^dagger)"""
    op = Brillouin(L, AP)
    op.build_hops(torch.as_tensor(U, device=gpu))
    h = op.hops().cpu().numpy()
    x = synth.coordinates(L)
    W = np.zeros((len(x), 81, 3, 3), complex)
    W[:, 40] = np.eye(3)
    for j in range(40):
        d = [((j + 41) // 3 ** mu) % 3 - 1 for mu in range(4)]
        back = ((x - d) % L) @ np.cumprod((1,) + tuple(L[:3]))
        W[:, 41 + j] = h[:, j]
        W[:, 39 - j] = h[back, j].conj().transpose(0, 2, 1)
    return op, W


# volumes on both sides of the lines between 4, 2 and 1 splits of the hop list
# (2 ceil(V / 32) warps at 1216 and 2432), ragged last groups
@pytest.mark.parametrize("L,nrhs", [((3, 3, 3, 3), 1), ((5, 3, 7, 3), 2), ((11, 12, 12, 12), 1), ((11, 11, 12, 13), 1),
                                    ((13, 14, 14, 15), 1), ((14, 14, 14, 15), 1), ((4, 5, 3, 4), 40)])
def test_splits_against_oracle(gpu, L, nrhs):
    U = synth.random_su3_links(L, 0.4, 5)
    psi = synth.gaussian_spinor(L, nrhs, 6)
    op, W = _op(L, U, gpu)
    x = torch.as_tensor(psi, device=gpu)
    for r in (0, nrhs - 1):
        for dag in (False, True):
            out = op.apply(x, m0=0.1, dagger=dag)[r].cpu().numpy()
            ref = oracle.apply(L, AP, W, 0.1, psi[r], dagger=dag)
            assert np.abs(out - ref).max() <= 1e-15 * np.abs(ref).max() * 4  # the oracle rounds ~480 sums in FP64


def test_orders_of_magnitude(gpu):
    """a field falling by e^-2 per step in every direction, a point source and a
    tiny and a huge field: each site to rounding of its own size"""
    L = (5, 4, 6, 4)
    U = synth.random_su3_links(L, 0.3, 7)
    op, W = _op(L, U, gpu)
    psi = np.repeat(synth.gaussian_spinor(L, 1, 8), 4, axis=0)
    psi[0] *= np.exp(-2.0 * synth.coordinates(L).sum(1))[:, None, None]
    psi[1] = 0
    psi[1, 17, 2, 1] = 1.0
    psi[2] *= 1e-290
    psi[3] *= 1e290
    out = op.apply(torch.as_tensor(psi, device=gpu), m0=0.1).cpu().numpy()
    for r in range(4):
        ref = oracle.apply(L, AP, W, 0.1, psi[r])
        size = np.abs(ref).max(axis=(1, 2), keepdims=True)
        assert (np.abs(out[r] - ref) <= 4e-15 * size).all(), r
        assert ((out[r] == 0) == (ref == 0)).all()


@pytest.mark.parametrize("scale", [1.0, 3.7, 1e-3, 1e60])
def test_links_that_are_not_unitary(gpu, scale):
    """one-hop fields are the links as given (at 1e60 the path sums overflow in the
    projection and nothing is finite)"""
    L = (4, 3, 5, 4)
    U = synth.random_su3_links(L, 0.3, 9)
    rng = np.random.default_rng(10)
    U = scale * (U + 0.2 * (rng.standard_normal(U.shape) + 1j * rng.standard_normal(U.shape)))
    op, W = _op(L, U, gpu)
    psi = synth.gaussian_spinor(L, 1, 11)
    out = op.apply(torch.as_tensor(psi, device=gpu), m0=0.1).cpu().numpy()[0]
    ref = oracle.apply(L, AP, W, 0.1, psi[0])
    fine = np.isfinite(ref)
    assert np.array_equal(np.isfinite(out), fine) and (fine.all() or scale == 1e60)
    assert (np.abs(out - ref)[fine] <= 4e-15 * np.abs(ref[fine]).max(initial=0.0)).all()


def test_infinities_and_nan_stay_local(gpu):
    """sites that see an infinity or a NaN are as the FP64 loop gives them (not
    finite where the oracle is not), the others are untouched"""
    L = (6, 7, 6, 8)
    U = synth.random_su3_links(L, 0.3, 12)
    op, _ = _op(L, U, gpu)
    psi = synth.gaussian_spinor(L, 1, 13)
    clean = op.apply(torch.as_tensor(psi, device=gpu)).cpu().numpy()[0]
    psi[0, 100, 1, 2] = np.inf
    psi[0, 900, 3, 0] = np.nan
    out = op.apply(torch.as_tensor(psi, device=gpu)).cpu().numpy()[0]
    x = synth.coordinates(L)
    far = np.ones(len(x), bool)
    for s in (100, 900):
        d = np.abs(x - x[s])
        far &= (np.minimum(d, np.array(L) - d) > 1).any(1)
    assert np.array_equal(out[far], clean[far])
    assert not np.isfinite(out[~far]).all(axis=(1, 2)).any()


def test_capture_and_streams(gpu):
    """The work space of an apply follows its stream: equal bits from a captured
    apply, replayed on new input, and from two streams at once."""
    L = (8, 6, 6, 8)
    op, _ = _op(L, synth.random_su3_links(L, 0.3, 14), gpu)
    x = torch.as_tensor(synth.gaussian_spinor(L, 8, 15), device=gpu)
    want = [op.apply(x[r:r + 1], m0=0.1) for r in range(8)]
    static = x[:1].clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = op.apply(static, m0=0.1)
    for r in (1, 2, 3):
        static.copy_(x[r:r + 1])
        graph.replay()
        assert torch.equal(out, want[r])
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    torch.cuda.synchronize()
    got = []
    for r in range(8):
        with torch.cuda.stream(streams[r % 2]):
            got.append(op.apply(x[r:r + 1], m0=0.1))
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(got, want))


@pytest.mark.parametrize("classes", [(1, 3), (1, 3, 4), (2,), (4,), (1, 2, 4), (2, 3, 4)])
def test_classes_switched_off(gpu, oracle_weights, classes):
    """Weights that leave out whole hop classes move the ends of the splits: with
    classes 1, 3 and with 1, 3, 4 the last pair of a split is the only one of its
    class, so that its sums follow the class before with no pair between."""
    lam = [1.9] + [-0.1 * n if n in classes else 0.0 for n in range(1, 5)]
    rho = [0.0] + [0.3 / n if n in classes else 0.0 for n in range(1, 5)]
    L = (4, 5, 3, 4)  # four splits
    U = synth.random_su3_links(L, 0.3, 16)
    psi = synth.gaussian_spinor(L, 9, 17)
    op, W = _op(L, U, gpu)
    op.set_weights(lam, rho)
    oracle_weights(lam, rho)
    x = torch.as_tensor(psi, device=gpu)
    for dag in (False, True):
        out = op.apply(x, m0=0.1, dagger=dag).cpu().numpy()
        for r in range(9):
            ref = oracle.apply(L, AP, W, 0.1, psi[r], dagger=dag)
            assert np.abs(out[r] - ref).max() <= 4e-15 * np.abs(ref).max()


@pytest.mark.parametrize("size", [2.0**10, 2.0**30, 2.0**62, 2.0**200])
def test_one_large_link_stays_local(gpu, size):
    """a link of any norm takes no digits from the sites that do not see it, nor
    from the unitary fields of those that do"""
    L = (6, 5, 7, 6)
    U = synth.random_su3_links(L, 0.3, 18)
    psi = synth.gaussian_spinor(L, 1, 19)
    U[100, 1] *= size
    op, W = _op(L, U, gpu)
    out = op.apply(torch.as_tensor(psi, device=gpu), m0=0.1).cpu().numpy()[0]
    ref = oracle.apply(L, AP, W, 0.1, psi[0])
    assert (np.abs(out - ref) <= 4e-15 * np.abs(ref).max(axis=(1, 2), keepdims=True)).all()


@pytest.mark.parametrize("scale", [1e-3, 1e-9, 1e-100])
def test_small_links_keep_their_digits(gpu, oracle_weights, scale):
    """links of a small norm where they are the whole result: Wilson weights,
    diagonal zero"""
    L = (4, 3, 5, 4)
    lam, rho = [4.0, -0.5, 0, 0, 0], [0, 0.5, 0, 0, 0]
    U = scale * synth.random_su3_links(L, 0.3, 20)
    psi = synth.gaussian_spinor(L, 1, 21)
    op, W = _op(L, U, gpu)
    op.set_weights(lam, rho)
    oracle_weights(lam, rho)
    out = op.apply(torch.as_tensor(psi, device=gpu), m0=-4.0).cpu().numpy()[0]
    ref = oracle.apply(L, AP, W, -4.0, psi[0])
    assert np.abs(out - ref).max() <= 4e-15 * np.abs(ref).max()


@pytest.mark.parametrize("size", [1e-290, 1e-200, 1e200])
def test_weights_of_any_size(gpu, oracle_weights, size):
    """weights whose products with the spinors' scales would leave the range of
    normal FP64 numbers lose no digits"""
    L = (4, 3, 5, 4)
    lam, rho = [0] + [size * v for v in (-0.5, -0.2, 0.1, 0.3)], [0] + [size * v for v in (0.3, 0.2, 0.1, 0.05)]
    U = synth.random_su3_links(L, 0.3, 22)
    psi = synth.gaussian_spinor(L, 1, 23) * 1e-10
    op, W = _op(L, U, gpu)
    op.set_weights(lam, rho)
    oracle_weights(lam, rho)
    out = op.apply(torch.as_tensor(psi, device=gpu), m0=0.0).cpu().numpy()[0]
    ref = oracle.apply(L, AP, W, 0.0, psi[0])
    assert np.abs(out - ref).max() <= 4e-15 * np.abs(ref).max()


def _scaled_weights(op, oracle_weights, f):
    lam, rho = op.weights()
    lam, rho = [f * v for v in lam], [f * v for v in rho]
    op.set_weights(lam, rho)
    oracle_weights(lam, rho)


@pytest.mark.parametrize("L,nrhs", [((3, 3, 3, 3), 1), ((4, 5, 3, 4), 7), ((11, 12, 12, 12), 1), ((14, 14, 14, 15), 1)])
@pytest.mark.parametrize("f", [2.0**-61, 2.0**-59])
def test_fp64_kernel_and_fixed_point(gpu, oracle_weights, L, nrhs, f):
    """The operator times a power of 2, just out of and just in the range of the
    fixed-point apply: the FP64 kernel, which also runs without memory for the
    fixed-point copy, and the fixed-point one, through D, D^dagger, the overlap
    kernel, the clover term and slabs of time slices"""
    U = synth.random_su3_links(L, 0.3, 24)
    psi = synth.gaussian_spinor(L, nrhs, 25)
    op, W = _op(L, U, gpu)
    _scaled_weights(op, oracle_weights, f)
    x = torch.as_tensor(psi, device=gpu)

    def check(out, ref):
        assert np.abs(out - ref).max() <= 4e-15 * np.abs(ref).max()

    r = nrhs - 1
    for dag in (False, True):
        ref = oracle.apply(L, AP, W, 0.1 * f, psi[r], dagger=dag)
        check(op.apply(x, m0=0.1 * f, dagger=dag)[r].cpu().numpy(), ref)
    host = op.apply_host(torch.as_tensor(psi).pin_memory(), m0=0.1 * f, dagger=True)
    torch.cuda.synchronize()
    check(host[r].numpy(), ref)
    check(op.overlap_kernel(x, rho=1.5 * f)[r].cpu().numpy(), oracle.overlap_kernel(L, AP, W, 0.0, 1.5 * f, psi[r]))
    if len(psi[0]) < 1000:
        op.set_clover(f)
        check(op.apply(x, m0=0.1 * f)[r].cpu().numpy(), oracle.apply_clover(L, AP, W, U, 0.1 * f, f, psi[r]))


@pytest.mark.parametrize("f", [2.0**61, 2.0**59])
@pytest.mark.parametrize("mode,nrhs", [(0, 1), (1, 2), (4, 3)])
def test_solves_with_either_apply(gpu, oracle_weights, f, mode, nrhs):
    """solver iterations and residuals (with right-hand sides skipped as they
    converge) on the FP64 kernel and on the fixed-point apply"""
    L = (4, 4, 5, 4)
    U = synth.random_su3_links(L, 0.3, 26)
    b = synth.z2_spinor(L, nrhs, 27)
    b[-1] = 0
    b[-1, 5, 1, 2] = 1.0
    op, W = _op(L, U, gpu)
    _scaled_weights(op, oracle_weights, f)
    op.store_hops("f32", "2row")
    x, info = op.solve(torch.as_tensor(b, device=gpu), m0=0.1 * f, tol=1e-10, mode=mode)
    assert all(i["status"] == "BRI_OK" for i in info)
    for r in range(nrhs):
        res = b[r] - oracle.apply(L, AP, W, 0.1 * f, x.cpu().numpy()[r])
        assert np.linalg.norm(res) <= 1.01e-10 * np.linalg.norm(b[r])


@pytest.mark.parametrize("what", ["spin", "colour", "zero beside small", "laplacian", "near the line"])
def test_components_of_different_size(gpu, oracle_weights, what):
    """Components that stay apart (one chirality and its spins, colours over unit
    links, chiralities without gamma terms) keep their own digits next to ones
    that are many orders larger: against the largest result of their own kind.
    Within the line of 2^-20 the block exponent takes at most that factor, 2^-54
    of the largest component and 80 hops of weight 1/16 or less."""
    L = (4, 4, 3, 5)
    U = synth.unit_links(L) if what in ("colour", "near the line") else synth.random_su3_links(L, 0.3, 28)
    psi = synth.gaussian_spinor(L, 1, 29)
    if what in ("spin", "zero beside small"):
        psi[:, :, 2:] = 0
    if what == "spin":
        psi[:, :, 1] *= 1e-14
    elif what == "colour":
        psi[..., 2] *= 1e-14
    elif what == "near the line":
        psi[..., 2] *= 1e-4
    elif what == "zero beside small":
        psi *= 1e-14
        psi[0, 100] = 0
        psi[0, 100, 0, 0] = 1.0
    else:
        psi[:, :, 2:] *= 1e-14
    op, W = _op(L, U, gpu)
    if what == "laplacian":
        lam, rho = [1.9, -0.1, -0.05, -0.02, -0.01], [0] * 5
        op.set_weights(lam, rho)
        oracle_weights(lam, rho)
    out = op.apply(torch.as_tensor(psi, device=gpu), m0=0.1).cpu().numpy()[0]
    ref = oracle.apply(L, AP, W, 0.1, psi[0])
    size = np.abs(ref).max(axis=0)
    tol = 4e-15 if what != "near the line" else 4e-15 + 2.0**-54 * 5 * np.abs(psi).max() / size
    assert (np.abs(out - ref).max(axis=0) <= tol * size).all()
    if what == "zero beside small":  # far from the point, each site by itself
        far = np.abs(ref).max(axis=(1, 2)) < 1e-10
        assert far.any()
        assert (np.abs(out - ref)[far] <= 4e-15 * np.abs(ref[far]).max(axis=(1, 2), keepdims=True)).all()


@pytest.mark.parametrize("rho2", [0.0, 1e-12])
def test_class_without_gamma_terms(gpu, oracle_weights, rho2):
    """the chiralities of a site that is seen through a class without (or with tiny)
    gamma terms do not mix: what the small one gives keeps its digits"""
    L = (4, 4, 3, 5)
    U = synth.random_su3_links(L, 0.3, 30)
    psi = 1e-14 * synth.gaussian_spinor(L, 1, 31)
    psi[0, 100, :2] *= 1e14
    op, W = _op(L, U, gpu)
    lam, rho = [0, -0.1, -0.05, -0.02, -0.01], [0, 0.1, rho2, 0.02, 0.01]
    op.set_weights(lam, rho)
    oracle_weights(lam, rho)
    out = op.apply(torch.as_tensor(psi, device=gpu), m0=0.0).cpu().numpy()[0]
    ref = oracle.apply(L, AP, W, 0.0, psi[0])
    x = synth.coordinates(L)
    d = np.abs(x - x[100])
    d = np.minimum(d, np.array(L) - d)
    seen = (d.max(1) == 1) & (d.sum(1) == 2)  # by a two-hop offset only
    size = np.abs(ref[:, 2:]).max(axis=(1, 2), keepdims=True)
    assert seen.sum() == 24 and size[seen].max() < 1e-11
    assert (np.abs(out - ref)[:, 2:] <= 4e-15 * size)[seen].all()

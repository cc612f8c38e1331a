"""GPU link precompute (path sums, Sec. 5.1; SU(3) projection, Sec. 5.2)
against the CPU oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_1012_3615_gb300 import Brillouin, synth

pytestmark = pytest.mark.gpu
AP = (1, 1, 1, -1)


@pytest.mark.parametrize("L,eps,seed", [((4, 4, 4, 4), 0.4, 1), ((3, 5, 4, 6), 0.3, 2), ((3, 3, 3, 3), 0.8, 3)])
def test_hops_match_oracle(gpu, L, eps, seed):
    U = synth.random_su3_links(L, eps, seed)
    W = oracle.build_hops(L, U)
    op = Brillouin(L, AP)
    op.build_hops(torch.as_tensor(U, device=gpu))
    Wg = op.hops().cpu().numpy()
    for j in range(40):
        assert np.abs(Wg[:, j] - W[:, j + 41]).max() < 1e-12, j


def _su3_check(Y, tol=1e-13):
    eye = np.eye(3)
    assert np.abs(np.einsum("nji,njk->nik", Y.conj(), Y) - eye).max() < tol
    assert np.abs(np.linalg.det(Y) - 1).max() < tol


def test_projection_generic_matrices(gpu):
    rng = np.random.default_rng(4)
    n = 3000
    A = (synth.random_su3(n, 5) + 1.5 * (rng.standard_normal((n, 3, 3)) + 1j * rng.standard_normal((n, 3, 3))))
    A[:500] *= 1e-3  # scale invariance over magnitudes
    A[500:1000] = synth.random_su3(500, 6) * (1 + 1e-7 * rng.standard_normal((500, 1, 1)))  # near-degenerate s
    op = Brillouin((3, 3, 3, 3), AP)
    Y = op.project_su3(torch.as_tensor(A, device=gpu)).cpu().numpy()
    _su3_check(Y)
    ref = oracle.project_su3(A)
    assert np.abs(Y - ref).max() < 1e-11


def test_projection_negative_determinant_sums(gpu):
    """Footnote of Sec. 5.2: det(U+V) can be negative real; then two phase
    choices tie, so compare the maximised objective and check Y in SU(3)."""
    As = []
    for t in range(6000):
        U, V = synth.random_su3(2, 5000 + t)
        A = U + V
        if np.linalg.det(A).real < -1e-3:
            As.append(A)
        if len(As) >= 40:
            break
    A = np.array(As)
    op = Brillouin((3, 3, 3, 3), AP)
    Y = op.project_su3(torch.as_tensor(A, device=gpu)).cpu().numpy()
    _su3_check(Y)
    ref = oracle.project_su3(A)
    fg = np.real(np.einsum("nij,nij->n", A.conj(), Y))
    fo = np.real(np.einsum("nij,nij->n", A.conj(), ref))
    assert np.abs(fg - fo).max() < 1e-12


def test_projection_branch_b_inputs(gpu):
    """det A with phase near pi and well separated singular values: the
    maximum needs the smallest singular value's phase beyond pi/2."""
    rng = np.random.default_rng(7)
    A = []
    for _ in range(200):
        s = np.sort(rng.uniform(0.05, 2.0, 3))[::-1]
        Uq = synth.random_su3(1, int(rng.integers(1 << 30)))[0]
        Vq = synth.random_su3(1, int(rng.integers(1 << 30)))[0]
        ph = np.exp(1j * rng.uniform(2.6, 3.1) / 3)
        A.append(Uq @ np.diag(s * ph) @ Vq.conj().T)
    A = np.array(A)
    op = Brillouin((3, 3, 3, 3), AP)
    Y = op.project_su3(torch.as_tensor(A, device=gpu)).cpu().numpy()
    _su3_check(Y)
    ref = oracle.project_su3(A)
    fg = np.real(np.einsum("nij,nij->n", A.conj(), Y))
    fo = np.real(np.einsum("nij,nij->n", A.conj(), ref))
    assert np.abs(fg - fo).max() < 1e-12
    assert np.abs(Y - ref).max() < 1e-9


def test_empty_projection_batch(gpu):
    op = Brillouin((3, 3, 3, 3), AP)
    A = torch.zeros((0, 3, 3), dtype=torch.complex128, device=gpu)
    assert op.project_su3(A).shape == (0, 3, 3)


@pytest.mark.parametrize("what", ["smooth", "rough", "haar", "gauss", "tiny", "huge", "identity", "near singular", "det phase"])
def test_projection_seeds(gpu, what):
    """Matrices that the FP32-seeded projection takes and ones that it hands to
    the general form (any scale, either branch, nearly singular), mixed in one
    launch: special unitary, stationary (the traceless anti-hermitian part of
    A^dagger Y vanishes) and no worse than the oracle's maximum.  Bounds: a few
    roundings of 3x3 products, 16 2^-52, relative to |A| for the last two."""
    rng = np.random.default_rng(77)
    n = 400

    def near(eps):
        return synth.random_su3_links((n, 1, 1, 1), eps, int(rng.integers(1 << 30)))[:, 0]

    A = sum(near(0.5) for _ in range(4)) / 4
    if what == "rough":
        A = sum(near(2.0) for _ in range(4)) / 4
    elif what == "haar":
        A = sum(synth.random_su3(n, s) for s in range(3))
    elif what == "gauss":
        A = rng.standard_normal((n, 3, 3)) + 1j * rng.standard_normal((n, 3, 3))
    elif what == "tiny":
        A = A * 1e-40
    elif what == "huge":
        A = A * 1e40
    elif what == "identity":
        A = A * 0 + np.eye(3)
    elif what == "near singular":
        A[:, 2] = A[:, 1] + 1e-7 * A[:, 2]
    elif what == "det phase":
        A = A * np.exp(1j * np.linspace(0, 2 * np.pi, n))[:, None, None]  # through branch A, its edge and branch B
    op = Brillouin((3, 3, 3, 3), (1, 1, 1, 1))
    Y = op.project_su3(torch.as_tensor(np.ascontiguousarray(A), device=gpu)).cpu().numpy()
    eps = 16 * 2.0 ** -52
    size = np.abs(A).max(axis=(1, 2))
    assert np.abs(Y.conj().transpose(0, 2, 1) @ Y - np.eye(3)).max() <= eps
    assert np.abs(np.linalg.det(Y) - 1).max() <= eps
    B = A.conj().transpose(0, 2, 1) @ Y
    T = 0.5 * (B - B.conj().transpose(0, 2, 1))
    T -= np.eye(3) * (np.trace(T, axis1=1, axis2=2) / 3)[:, None, None]
    assert (np.abs(T).max(axis=(1, 2)) <= eps * size).all()
    for i in range(0, n, 40):
        best = np.trace(A[i].conj().T @ oracle.project_su3(A[i])).real
        assert np.trace(B[i]).real >= best - eps * size[i]


@pytest.mark.parametrize("what", ["unitary", "rough", "norm 1 + 1e-4", "scaled", "one bad link"])
def test_path_sums_fixed_point_and_fp64(gpu, what):
    """Unit-norm links take the fixed-point path sums, any others the FP64 ones
    (also when a single link is the reason): fields and force against the
    oracle, to the bounds of the other tests."""
    L = (3, 4, 5, 3)
    U = synth.random_su3_links(L, 2.0 if what == "rough" else 0.3, 91)
    if what == "norm 1 + 1e-4":
        U = U * (1 + 1e-4)
    elif what == "scaled":
        U = U * 1e-3
    elif what == "one bad link":
        U[17, 2] *= 1.5
    op = Brillouin(L, AP)
    op.build_hops(torch.as_tensor(U, device=gpu))
    W = oracle.build_hops(L, U)
    Wg = op.hops().cpu().numpy()
    for j in range(40):
        assert np.abs(Wg[:, j] - W[:, j + 41]).max() < 1e-12, j
    chi, psi = synth.gaussian_spinor(L, 2, 92)
    ref = oracle.force(L, AP, U, 0.0, chi, psi)
    dU = op.force(torch.as_tensor(chi, device=gpu), torch.as_tensor(psi, device=gpu)).cpu().numpy()
    assert np.abs(dU - ref).max() <= 1e-10 * np.abs(ref).max()


@pytest.mark.parametrize("L,eps", [((4, 3, 3, 3), 0.3), ((3, 5, 3, 3), 1.0), ((3, 3, 3, 4), 3.0)])
def test_projection_of_fixed_point_sums(gpu, L, eps):
    """The off-axis fields of unitary links, projected in fixed point where the
    FP32 seed settles and in the general form elsewhere: special unitary,
    stationary and no worse than the oracle's maximum at the oracle's path sums.
    Bounds as for the projection of single matrices, 16 2^-52."""
    U = synth.random_su3_links(L, eps, 95)
    op = Brillouin(L, AP)
    op.build_hops(torch.as_tensor(U, device=gpu))
    W = op.hops().cpu().numpy()
    tol = 16 * 2.0**-52
    for j in range(40):
        d = [(j + 41) // 3**m % 3 - 1 for m in range(4)]
        if sum(map(abs, d)) < 2:
            continue
        Y = W[:, j]
        A = np.stack([a / n for a, n in (oracle.path_sum(L, U, s, d) for s in range(len(W)))])
        assert np.abs(Y.conj().transpose(0, 2, 1) @ Y - np.eye(3)).max() <= tol
        assert np.abs(np.linalg.det(Y) - 1).max() <= tol
        B = A.conj().transpose(0, 2, 1) @ Y
        T = 0.5 * (B - B.conj().transpose(0, 2, 1))
        T -= np.eye(3) * (np.trace(T, axis1=1, axis2=2) / 3)[:, None, None]
        assert np.abs(T).max() <= tol
        for s in range(0, len(W), 20):
            assert np.trace(B[s]).real >= np.trace(A[s].conj().T @ oracle.project_su3(A[s])).real - tol


@pytest.mark.parametrize("a,b", [(0.0, 3**-0.5), (0.612, 0.296), (0.3, 0.46)])
def test_unit_norms_without_orthogonality(gpu, a, b):
    """Links whose rows and columns have norm 1 without being unitary, a + b J in
    any order with any phases: path sums of norm up to 1.73^4, beyond the bounds
    of the fixed-point form.  They take the FP64 form, like twice those links,
    whose off-axis fields are therefore the same bits (all steps scale by powers
    of 2; an entry in a hundred may differ where a threshold of the projection
    does not), and agree with the oracle's to the bound of the other tests."""
    L = (3, 4, 3, 5)
    rng = np.random.default_rng(96)
    n = synth.volume(L) * 4
    A = a * np.eye(3) + b * np.ones((3, 3))
    A = A / np.linalg.norm(A[0])
    perm = np.array([rng.permutation(3) for _ in range(n)])
    ph = np.exp(0.4j * rng.standard_normal((2, n, 3)))
    U = (A[perm] * ph[0][:, :, None] * ph[1][:, None, :]).reshape(-1, 4, 3, 3)
    assert np.allclose(np.linalg.norm(U, axis=-1), 1) and np.allclose(np.linalg.norm(U, axis=-2), 1)
    op = Brillouin(L, AP)
    off = [j for j in range(40) if sum((j + 41) // 3**m % 3 != 1 for m in range(4)) > 1]
    op.build_hops(torch.as_tensor(U, device=gpu))
    W = op.hops().cpu().numpy()[:, off]
    op.build_hops(torch.as_tensor(2 * U, device=gpu))
    assert (op.hops().cpu().numpy()[:, off] == W).mean() > 0.99
    ref = oracle.build_hops(L, U)[:, [j + 41 for j in off]]
    # where the maximum is unique to 64 bits: the path sum's singular values apart from zero
    fine = np.isfinite(ref).all(axis=(-1, -2))
    for i, j in enumerate(off):
        d = [(j + 41) // 3**m % 3 - 1 for m in range(4)]
        for s in range(0, len(W), 7):
            P, m = oracle.path_sum(L, U, s, d)
            sv = np.linalg.svd(P / m, compute_uv=False)
            if fine[s, i] and sv[2] > 1e-3:
                assert np.abs(W[s, i] - ref[s, i]).max() < 1e-12 / sv[2], (s, j)

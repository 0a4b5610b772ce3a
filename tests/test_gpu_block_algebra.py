"""Block algebra and L x L steps (C ABI) at the sizes where their kernels
change: the row kernels up to 12 columns, the tiled ones above, odd column
counts, lattices that fill no tile, and the FP64 operator on either side of
its split over four warps."""
import numpy as np
import pytest

import synth
from oracle import dense, dirac

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

# sums of n products of unit-size terms: sqrt(n) roundings of the arithmetic, with a factor of ten to spare
GRAM_TOL = {"fp64": 1e-13, "fp32": 1e-5, "fp16": 2e-3}
XMY_TOL = {"fp64": 2e-14, "fp32": 2e-6, "fp16": 2e-3}


def _rel(a, b):
    return float(np.max(np.abs(a - b)) / np.max(np.abs(b)))


def _lat(dims, seed=1):
    import paper_0903_4936_gb300 as bk
    lat = bk.Lattice(dims)
    U = synth.random_su3_field(dims, 0.4, seed)
    lat.upload_gauge(U)
    lat.build_clover(1.0)
    return lat, U


@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("dims,L", [((3, 5, 4, 6), 1), ((3, 5, 4, 6), 5), ((2, 2, 2, 2), 6), ((3, 5, 4, 6), 7),
                                    ((3, 5, 4, 6), 12), ((3, 5, 4, 6), 13), ((2, 2, 2, 2), 27), ((4, 4, 4, 6), 48),
                                    ((3, 5, 4, 6), 63), ((3, 5, 2, 6), 97), ((2, 3, 4, 6), 130), ((2, 3, 4, 6), 259)])
def test_gram_and_xmy(prec, dims, L):
    """G = A^H B and Y = Z + c X M against numpy in FP64."""
    lat, _ = _lat(dims)
    A = synth.gaussian_sources(dims, L, 21)
    B = synth.gaussian_sources(dims, L, 22)
    Fa, Fb = lat.pack(torch.from_numpy(A).cuda(), prec), lat.pack(torch.from_numpy(B).cuda(), prec)
    G = lat.gram(Fa, Fb, L, prec).cpu().numpy()
    a, b = A.reshape(L, -1), B.reshape(L, -1)
    assert _rel(G, a.conj() @ b.T) < GRAM_TOL[prec]
    rng = np.random.default_rng(5)
    M = (rng.standard_normal((L, L)) + 1j * rng.standard_normal((L, L))) / np.sqrt(2 * L)
    for c, Z in ((1.0, None), (0.3 - 0.7j, Fb)):
        Y = lat.unpack(lat.xmy(Fa, torch.from_numpy(M).cuda(), L, c=c, Z=Z, prec=prec), L, prec).cpu().numpy()
        ref = c * (M.T @ a) + (b if Z is not None else 0.0)
        assert _rel(Y.reshape(L, -1), ref) < XMY_TOL[prec]


@pytest.mark.parametrize("method", ["bicggr", "bicgstab"])
@pytest.mark.parametrize("Ls", [(1,), (2, 5), (7,), (11, 3), (12, 6), (13,)])
def test_fp64_solves_by_system_size(method, Ls):
    """FP64 solves whose systems are on either side of 6 and 12 columns against dense LU."""
    dims = (4, 4, 4, 4)
    lat, U = _lat(dims, 7)
    B = synth.z4_noise(dims, sum(Ls), 31)
    X, infos = lat.block_solve_batched(torch.from_numpy(B).cuda(), [0.12] * len(Ls), list(Ls), method=method,
                                       prec="fp64", tol=1e-11, maxiter=500)
    D = dense.dense_matrix(U, 0.12, 1.0)
    ref = np.linalg.solve(D, dense.to_columns(B))
    got = dense.to_columns(X.cpu().numpy())
    assert all(i["converged"] == 1 for i in infos)
    # ||x - x*|| <= ||D^-1|| ||r||, ||D^-1|| < 20 at this kappa
    assert np.max(np.linalg.norm(got - ref, axis=0) / np.linalg.norm(B.reshape(sum(Ls), -1).T, axis=0)) < 2e-10


@pytest.mark.parametrize("dims,L", [((2, 2, 2, 2), 1), ((3, 5, 4, 6), 3), ((8, 8, 8, 8), 9), ((8, 8, 8, 8), 10)])
def test_fp64_operator_split_over_warps(dims, L):
    """Site-columns below (38912 of them) and above the limit of the four-warp form, with a residual solve's path."""
    lat, U = _lat(dims, 9)
    X = synth.gaussian_sources(dims, L, 3)
    kap = np.linspace(0.11, 0.13, L)
    Y = lat.dslash(torch.from_numpy(X).cuda(), list(kap), "fp64").cpu().numpy()
    assert _rel(Y, dirac.apply_dirac(U, X, kap, 1.0)) < 1e-13


@pytest.mark.parametrize("prec,Ls", [("fp64", (3, 2, 4)), ("fp64", (6, 20, 5)), ("fp64", (12, 12, 12)),
                                     ("fp64", (30, 24, 6)), ("fp32", (3, 2, 4)), ("fp32", (6, 6, 6)),
                                     ("fp32", (2, 12, 2))])
def test_systems_around_a_converged_one(prec, Ls):
    """The middle system (small kappa) converges first; the others go on with its columns between theirs."""
    dims = (4, 4, 4, 4)
    lat, U = _lat(dims, 11)
    B = synth.z4_noise(dims, sum(Ls), 33)
    kappas = [0.12, 0.03, 0.12]
    X, infos = lat.block_solve_batched(torch.from_numpy(B).cuda(), kappas, list(Ls), method="bicgstab", prec=prec,
                                       tol=1e-10, maxiter=500, delta=0.0 if prec == "fp64" else 0.03)
    assert all(i["converged"] == 1 for i in infos)
    assert infos[1]["iterations"] < min(infos[0]["iterations"], infos[2]["iterations"])
    got = dense.to_columns(X.cpu().numpy())
    rhs = dense.to_columns(B)
    c = 0
    for kappa, L in zip(kappas, Ls):
        ref = np.linalg.solve(dense.dense_matrix(U, kappa, 1.0), rhs[:, c:c + L])
        # ||x - x*|| <= ||D^-1|| ||r||, ||D^-1|| < 20 at these kappas
        err = np.linalg.norm(got[:, c:c + L] - ref, axis=0) / np.linalg.norm(rhs[:, c:c + L], axis=0)
        assert np.max(err) < 2e-9
        c += L


@pytest.mark.parametrize("L", [5, 6, 7, 12])
@pytest.mark.parametrize("eps", [0.0, 1e-5, 1e-3])
def test_cholesky_basis_of_nearly_dependent_columns(L, eps):
    """P^H P is singular or nearly so when two sources differ by eps times noise: the basis is then left alone (the
    L x L system of equal columns breaks down) or changed to an orthonormal one, the same in every run, bit for bit."""
    dims = (4, 4, 4, 4)
    lat, U = _lat(dims, 13)
    B = synth.gaussian_sources(dims, L, 51)
    B[L - 1] = B[1] + eps * synth.gaussian_sources(dims, 1, 52)[0]
    Bt = torch.from_numpy(B).cuda()
    runs = [lat.block_solve(Bt, 0.12, method="bicgstab", prec="fp64", tol=1e-10, maxiter=300, orth=True,
                            raise_on_fail=False) for _ in range(3)]
    X, info = runs[0]
    for Y, other in runs[1:]:
        assert other["iterations"] == info["iterations"] and torch.equal(torch.view_as_real(X), torch.view_as_real(Y))
    if eps == 0.0:
        assert info["breakdown"] == 1
        return
    assert info["converged"] == 1
    ref = np.linalg.solve(dense.dense_matrix(U, 0.12, 1.0), dense.to_columns(B))
    got = dense.to_columns(X.cpu().numpy())
    # ||x - x*|| <= ||D^-1|| ||r||, ||D^-1|| < 20 at this kappa; the recursive residual of a basis of condition
    # 1 / eps may differ from the true one by rounding times that
    assert np.max(np.linalg.norm(got - ref, axis=0) / np.linalg.norm(dense.to_columns(B), axis=0)) < 20 * (
        1e-10 + 1e-13 / eps)


@pytest.mark.parametrize("L", [889, 1000, 1024])
def test_gram_of_the_widest_blocks(L):
    """FP32 Gram matrices up to the width (1024) at which 256 threads a block fill the work list."""
    dims = (2, 2, 2, 2)
    lat, _ = _lat(dims)
    A, B = (synth.gaussian_sources(dims, L, s) for s in (61, 62))
    G = lat.gram(lat.pack(torch.from_numpy(A).cuda(), "fp32"), lat.pack(torch.from_numpy(B).cuda(), "fp32"), L,
                 "fp32").cpu().numpy()
    assert _rel(G, A.reshape(L, -1).conj() @ B.reshape(L, -1).T) < GRAM_TOL["fp32"]


@pytest.mark.parametrize("nsys,L", [(64, 112), (48, 122), (64, 128)])
def test_many_wide_systems(nsys, L):
    """Partitions whose Gram matrices fill the work list are accepted: one iteration of each system."""
    dims = (2, 2, 2, 2)
    lat, _ = _lat(dims)
    B = torch.from_numpy(synth.gaussian_sources(dims, L, 63)).cuda().repeat(nsys, 1, 1, 1, 1, 1, 1)
    _, infos = lat.block_solve_batched(B, [0.1] * nsys, [L] * nsys, method="bicgstab", prec="fp64", tol=1e-10,
                                       maxiter=1, raise_on_fail=False)
    assert infos[0]["status"] == "BK_ERR_NOT_CONVERGED"
    assert all(i["iterations"] == 1 and np.isfinite(i["rec_res_max"]) for i in infos)


def test_wide_gram_workspace_on_a_small_lattice():
    """The partial sums of a wide Gram matrix take no more memory than a few blocks of its operands' size."""
    dims, L = (4, 4, 4, 4), 512
    lat, _ = _lat(dims)
    A = lat.pack(torch.from_numpy(synth.gaussian_sources(dims, L, 64)).cuda(), "fp64")
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    G = lat.gram(A, A, L, "fp64")
    torch.cuda.synchronize()
    # G, its partial sums (two operands' worth) and a 2 MB allocation granule for each, with room for one block more
    assert before - torch.cuda.mem_get_info()[0] <= 4 * A.numel() + 16 * L * L + (4 << 20)
    a = lat.unpack(A, L, "fp64").cpu().numpy().reshape(L, -1)
    assert _rel(G.cpu().numpy(), a.conj() @ a.T) < GRAM_TOL["fp64"]


@pytest.mark.parametrize("dims,L", [((8, 8, 8, 8), 2), ((8, 8, 8, 8), 6), ((8, 8, 8, 8), 12), ((16, 16, 16, 8), 13),
                                    ((16, 16, 16, 8), 48)])
def test_fp32_gram_beyond_the_fp32_range(dims, L):
    """Sums of at most 96 rows are in FP32 and the rest in FP64: 96 rows of these blocks stay within FP32's range
    (2.8e38 of 3.4e38), all of them are 500 times above it."""
    lat, _ = _lat(dims)
    c = np.float32(1.2e18)
    F = lat.empty_field(L, "fp32")
    F.view(torch.float32).fill_(float(c))
    G = lat.gram(F, F, L, "fp32").cpu().numpy()
    want = 2.0 * float(c) ** 2 * 12 * np.prod(dims)  # conj(c + ic)(c + ic) per row
    assert np.all(np.isfinite(G)) and np.max(np.abs(G - want)) < GRAM_TOL["fp32"] * want


@pytest.mark.parametrize("prec,Ls", [("fp64", (30, 4)), ("fp64", (20, 8)), ("fp64", (3, 40, 1)), ("fp32", (30, 4))])
def test_wide_systems_beside_narrow_ones(prec, Ls):
    """Updates of one launch whose systems stage different numbers of columns (3 and 4 columns take tiles of 1024
    rows), against dense LU."""
    dims = (4, 4, 4, 4)
    lat, U = _lat(dims, 17)
    B = synth.z4_noise(dims, sum(Ls), 35)
    X, infos = lat.block_solve_batched(torch.from_numpy(B).cuda(), [0.11] * len(Ls), list(Ls), method="bicgstab",
                                       prec=prec, tol=1e-10, maxiter=1000, delta=0.0 if prec == "fp64" else 0.03)
    assert all(i["converged"] == 1 for i in infos)
    ref = np.linalg.solve(dense.dense_matrix(U, 0.11, 1.0), dense.to_columns(B))
    got = dense.to_columns(X.cpu().numpy())
    # ||x - x*|| <= ||D^-1|| ||r||, ||D^-1|| < 20 at this kappa
    assert np.max(np.linalg.norm(got - ref, axis=0) / np.linalg.norm(dense.to_columns(B), axis=0)) < 2e-9

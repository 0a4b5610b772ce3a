"""The FP32 / FP16 operators (C ABI) on ragged and extreme lattices and column
counts (one pair, more than one launch), and over part of a block's columns."""
import numpy as np
import pytest

import synth
from oracle import dense, dirac, evenodd

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

# as for the other operator tests: FP32 unit roundoff times about 50 terms; FP16 storage at 11 bits
TOL = {"fp32": 2e-6, "fp16": 2e-3}
SCHUR_TOL = {"fp32": 5e-6, "fp16": 5e-3}  # two operators and a temporary in that storage


def _rel(a, b):
    return float(np.max(np.abs(a - b)) / np.max(np.abs(b)))


def _lat(dims, seed):
    import paper_0903_4936_gb300 as bk
    lat = bk.Lattice(dims)
    U = synth.random_su3_field(dims, 0.5, seed)
    lat.upload_gauge(U)
    lat.build_clover(1.0)
    return lat, U


@pytest.mark.parametrize("prec", ["fp32", "fp16"])
@pytest.mark.parametrize("dims,L", [((2, 2, 2, 2), 1), ((3, 3, 3, 3), 6), ((5, 4, 7, 3), 12), ((7, 3, 2, 5), 29),
                                    ((9, 5, 3, 4), 3), ((4, 6, 5, 3), 97), ((3, 2, 3, 4), 130), ((4, 2, 2, 2), 256),
                                    ((4, 2, 2, 2), 259)])
def test_operator_shapes(prec, dims, L):
    lat, U = _lat(dims, 11 + L)
    X = synth.gaussian_sources(dims, L, 5)
    kap = np.linspace(0.10, 0.13, L)
    Y = lat.dslash(torch.from_numpy(X).cuda(), list(kap), prec).cpu().numpy()
    assert _rel(Y, dirac.apply_dirac(U, X, kap, 1.0)) < TOL[prec]


@pytest.mark.parametrize("prec", ["fp32", "fp16"])
@pytest.mark.parametrize("dims,L", [((2, 2, 2, 2), 1), ((6, 4, 6, 4), 12), ((10, 4, 2, 4), 29), ((6, 6, 4, 4), 3),
                                    ((4, 4, 6, 2), 97), ((4, 2, 2, 4), 259)])
def test_schur_shapes(prec, dims, L):
    lat, U = _lat(dims, 21 + L)
    X = synth.gaussian_sources(dims, L, 6)
    kap = np.repeat(np.linspace(0.10, 0.13, (L + 1) // 2), 2)[:L]
    Y = lat.schur_dslash(torch.from_numpy(X).cuda(), list(kap), prec).cpu().numpy()
    odd = evenodd.parity_mask(dims, 1)
    for j in sorted({0, L // 2, L - 1}):
        ref = evenodd.schur_apply(U, X[j:j + 1], kap[j], 1.0)
        assert np.all(Y[j][odd] == 0)
        assert _rel(Y[j:j + 1], ref) < SCHUR_TOL[prec]


@pytest.mark.parametrize("eo", [False, True])
@pytest.mark.parametrize("prec", ["fp32", "fp16"])
def test_runs_of_columns(prec, eo):
    """Systems that stop at different iterations leave runs of columns that are not whole rows."""
    dims = (4, 4, 4, 4)
    lat, U = _lat(dims, 7)
    kappas, Ls = [0.02, 0.12, 0.06, 0.125, 0.03], [5, 6, 2, 4, 6]
    B = synth.z4_noise(dims, sum(Ls), 31)
    X, infos = lat.block_solve_batched(torch.from_numpy(B).cuda(), kappas, Ls, method="bicgstab", prec=prec, tol=1e-10,
                                       maxiter=500, eo=eo, delta=0.01)
    assert all(i["converged"] == 1 and i["true_res_max"] <= 1e-10 for i in infos)
    assert len({i["iterations"] for i in infos}) > 2
    got, c0 = dense.to_columns(X.cpu().numpy()), 0
    for k, L in zip(kappas, Ls):
        b = B[c0:c0 + L]
        ref = np.linalg.solve(dense.dense_matrix(U, k, 1.0), dense.to_columns(b))
        dev = np.linalg.norm(got[:, c0:c0 + L] - ref, axis=0) / np.linalg.norm(ref, axis=0)
        assert dev.max() <= 1e-8
        c0 += L


# One warp a block up to 152 * 3 * 128 = 58368 (site, pair) items, four above: items on that line, the last block full
# or not.
@pytest.mark.parametrize("prec", ["fp32", "fp16"])
@pytest.mark.parametrize("dims,L", [((8, 8, 6, 8), 38), ((8, 8, 6, 8), 39), ((5, 7, 9, 13), 28), ((5, 7, 9, 13), 29)])
def test_operator_block_sizes(prec, dims, L):
    lat, U = _lat(dims, 31 + L)
    X = synth.gaussian_sources(dims, L, 7)
    kap = np.linspace(0.10, 0.13, L)
    Y = lat.dslash(torch.from_numpy(X).cuda(), list(kap), prec).cpu().numpy()
    for j in (0, 1, L // 2, L - 1):
        assert _rel(Y[j:j + 1], dirac.apply_dirac(U, X[j:j + 1], kap[j:j + 1], 1.0)) < TOL[prec]


@pytest.mark.parametrize("prec", ["fp32", "fp16"])
@pytest.mark.parametrize("dims,L", [((8, 8, 6, 16), 38), ((8, 8, 6, 16), 39), ((10, 10, 6, 14), 26),
                                    ((10, 10, 6, 14), 27)])
def test_schur_block_sizes(prec, dims, L):
    lat, U = _lat(dims, 41 + L)
    X = synth.gaussian_sources(dims, L, 8)
    kap = np.repeat(np.linspace(0.10, 0.13, (L + 1) // 2), 2)[:L]
    Y = lat.schur_dslash(torch.from_numpy(X).cuda(), list(kap), prec).cpu().numpy()
    odd = evenodd.parity_mask(dims, 1)
    for j in (0, L - 1):
        assert np.all(Y[j][odd] == 0)
        assert _rel(Y[j:j + 1], evenodd.schur_apply(U, X[j:j + 1], kap[j], 1.0)) < SCHUR_TOL[prec]


# 32 columns of one site to a block: 456 blocks fill 152 SMs three times; the split over four warps and the form with
# one thread each take turns above that
@pytest.mark.parametrize("L", [57, 58, 77, 96, 128, 140])
def test_fp64_operator_forms(L):
    dims = (4, 4, 4, 4)
    lat, U = _lat(dims, 51 + L)
    X = synth.gaussian_sources(dims, L, 9)
    kap = np.linspace(0.10, 0.13, L)
    Y = lat.dslash(torch.from_numpy(X).cuda(), list(kap), "fp64").cpu().numpy()
    assert _rel(Y, dirac.apply_dirac(U, X, kap, 1.0)) < 1e-13


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("L", [1, 2, 3, 4, 8, 9, 15, 16, 17, 18, 31, 33])
def test_layout_conversions(prec, L):
    """Canonical to device layout and back: tiles of 8 sites and 16 columns, 90 sites, every column exact."""
    import paper_0903_4936_gb300 as bk
    dims, V = (3, 5, 2, 3), 90
    lat = bk.Lattice(dims)
    X = synth.gaussian_sources(dims, L, 10)
    X = X.astype(np.complex64).astype(np.complex128) if prec == "fp32" else X
    F = lat.pack(torch.from_numpy(X).cuda(), prec)
    v = F.cpu().numpy().view(np.float64 if prec == "fp64" else np.float32)  # (its size is rounded up)
    v = v[:V * 12 * ((L + 1) // 2) * 4].reshape(V * 12, (L + 1) // 2, 2, 2)
    x = X.reshape(L, V * 12)
    for j in range(L):
        assert np.array_equal(v[:, j // 2, 0, j % 2], x[j].real) and np.array_equal(v[:, j // 2, 1, j % 2], x[j].imag)
    assert np.array_equal(lat.unpack(F, L, prec).cpu().numpy(), X)

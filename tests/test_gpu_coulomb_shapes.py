"""rho and J at the shapes that stress their work split, through the C ABI.

rho streams the strictly upper elements of each B_P in row-pair order (pair q
is row q followed by row nao-1-q; for odd nao the middle row comes last
alone), thread t of a CTA taking elements t, t + 256, ...; J takes its
elements in chunks of a row pair.  Odd nao (the lone middle row), nao below
the CTA's 256 threads (a thread's next element lies several pairs ahead),
nao = 1, 2 and 3 (the Coulomb build alone), and a naux that is not a
multiple of J's eight loads in flight: rho and J against the oracle's
definitions within the FP64 summation bound, dense and packed layouts equal to
each other bit for bit, and df_build_JK's short grids (items taken from a
counter) equal to df_build_J's full grids bit for bit.
"""
import numpy as np
import pytest
import torch

from oracle import df_oracle as O
from paper_2601_08077_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def df():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2601_08077_gb300 import build, df as dfmod
    build.build_all()
    return dfmod


def _random(seed, naux, nao, nocc):
    rng = np.random.default_rng(seed)
    B = rng.standard_normal((naux, nao, nao))
    B = 0.5 * (B + B.transpose(0, 2, 1))
    C = np.linalg.qr(rng.standard_normal((nao, nao)))[0][:, :nocc] if nocc <= nao else None
    return B, np.ascontiguousarray(C)


def _check(df, B, C, jk=True):
    naux, nao, _ = B.shape
    nocc = C.shape[1]
    D = inputs.density(C)
    rho_ref = O.rho(B, D)
    J_ref = O.coulomb(B, rho_ref)
    # FP64 reordering bounds of the sums (both sides' roundings): rho_P sums nao^2 terms of size
    # |B||D|; J_mn sums naux terms of size |B||rho|, plus |B| times rho's own error per term
    eps, bmax = np.finfo(float).eps, np.max(np.abs(B))
    tol_rho = 4 * nao * nao * eps * bmax * np.max(np.abs(D))
    tol_J = 4 * naux * eps * bmax * np.max(np.abs(rho_ref)) + naux * bmax * tol_rho
    Dg, Cg = torch.from_numpy(D).cuda(), torch.from_numpy(C).cuda()
    Bg = torch.from_numpy(B).cuda()
    Bp = torch.from_numpy(inputs.pack_upper(B)).cuda()
    out = []
    for packed in (False, True):
        ctx = df.Context(nao, naux, nocc)
        if packed:
            ctx.setup_packed(Bp)
        else:
            ctx.setup(Bg)
        J, rho = ctx.build_J(Dg)
        J, rho = J.clone(), rho.clone()
        if jk:
            J2, rho2, _, _ = ctx.build_JK(Dg, Cg, 5)
            assert torch.equal(J, J2) and torch.equal(rho, rho2)
        ctx.sync_status()
        out.append((J.cpu().numpy(), rho.cpu().numpy()))
    (Jd, rd), (Jp, rp) = out
    assert np.array_equal(Jd, Jp) and np.array_equal(rd, rp)
    assert np.max(np.abs(rd - rho_ref)) <= tol_rho
    assert np.max(np.abs(Jd - J_ref)) <= tol_J
    assert np.array_equal(Jd, Jd.T)


@pytest.mark.parametrize("nao, naux", [(33, 29), (255, 13), (257, 11)])
def test_coulomb_random_shapes(df, nao, naux):
    B, C = _random(500 + nao, naux, nao, 1)
    _check(df, B, C)


@pytest.mark.parametrize("nao, naux", [(1, 5), (2, 3), (3, 7)])
def test_coulomb_tiny(df, nao, naux):
    """No or one or three off-diagonal elements per B_P (the Coulomb build alone: an exchange
    build of a 1-3 function basis is not a case the slice GEMM's tiles are meant for)."""
    B, C = _random(600 + nao, naux, nao, 1)
    _check(df, B, C, jk=False)


def test_coulomb_odd_molecule(df):
    """27 atoms: nao 135 (odd), naux 405 (a ragged fourth block of 21 functions)."""
    mol, B, C, D = inputs.make_inputs(inputs.Workload("df-27atom-nao135-naux405-nocc27", 27, 27, 7300))
    _check(df, B, C)


@pytest.mark.parametrize("naux", [1, 7, 8, 9, 15, 16, 17, 31, 32, 33, 48])
def test_coulomb_at_the_edges_of_its_load_ring(df, naux):
    """J's sum over P keeps 8 (alone) or 16 (beside the second exchange GEMM) loads ahead: below one
    ring, one, two and three of them, and remainders.  Both give the same bits; against FP64 within
    the rounding of naux additions."""
    nao = 40
    rng = np.random.default_rng(naux)
    B = rng.standard_normal((naux, nao, nao))
    B = B + B.transpose(0, 2, 1)
    D = rng.standard_normal((nao, nao))
    D = D + D.T
    ctx = df.Context(nao, naux, 4, 3)
    ctx.setup(torch.from_numpy(B).cuda())
    Dg = torch.from_numpy(D).cuda()
    J, rho = ctx.build_J(Dg)
    J2, rho2, _, _ = ctx.build_JK(Dg, torch.from_numpy(rng.standard_normal((nao, 4))).cuda(), 3)
    assert torch.equal(J, J2) and torch.equal(rho, rho2)
    J, rho = J.cpu().numpy(), rho.cpu().numpy()
    ref = np.einsum("pij,p->ij", B, rho)
    assert np.all(np.abs(J - ref) <= 2 * naux * 2.0 ** -52 * np.einsum("pij,p->ij", np.abs(B), np.abs(rho)))


def test_energies_after_overlapping_calls(df):
    """Energies of one context asked for from four threads on their own streams (their launches
    share the context's partial sums and its count of finished blocks), then alone: the count must
    be back at zero, so the later call reduces all of its blocks and returns the usual values."""
    from concurrent.futures import ThreadPoolExecutor

    B, C = _random(5, 40, 96, 12)
    ctx = df.Context(96, 40, 12, 3)
    ctx.setup(torch.from_numpy(B).cuda())
    D = torch.from_numpy(C @ C.T).cuda()
    J, rho, K, _ = ctx.build_JK(D, torch.from_numpy(C).cuda(), 3)
    torch.cuda.synchronize()
    want = ctx.energy(D, J, K, rho)
    streams = [torch.cuda.Stream() for _ in range(4)]

    def ask(st):
        for _ in range(200):
            ctx.energy(D, J, K, rho, stream=st)

    with ThreadPoolExecutor(4) as ex:
        list(ex.map(ask, streams))
    assert all(ctx.energy(D, J, K, rho) == want for _ in range(3))


@pytest.mark.parametrize("naux", [608, 609, 760, 761, 1216, 1217, 1520])
def test_rho_at_the_edges_of_whole_waves(df, naux):
    """rho alone runs four or five CTAs an SM by the waves that naux takes (152 SMs: 608 and 760
    CTAs a wave): the same bits on either side of each edge as beside the exchange GEMM, dense and
    packed, and the FP64 sums within their rounding."""
    nao = 35
    B, C = _random(naux, naux, nao, 4)
    D = torch.from_numpy(C @ C.T).cuda()
    Bg = torch.from_numpy(B).cuda()
    iu = torch.triu_indices(nao, nao, device="cuda")
    Bp = Bg[:, iu[0], iu[1]].contiguous()
    got = []
    for packed in (False, True):
        ctx = df.Context(nao, naux, 4, 2)
        ctx.setup_packed(Bp) if packed else ctx.setup(Bg)
        got.append(ctx.build_J(D)[1].cpu().numpy())
        got.append(ctx.build_JK(D, torch.from_numpy(C).cuda(), 2)[1].cpu().numpy())
    for r in got[1:]:
        assert np.array_equal(r, got[0])
    Dn = D.cpu().numpy()
    ref, mag = np.einsum("pij,ij->p", B, Dn), np.einsum("pij,ij->p", np.abs(B), np.abs(Dn))
    assert np.all(np.abs(got[0] - ref) <= 2 * nao * 2.0 ** -52 * mag)

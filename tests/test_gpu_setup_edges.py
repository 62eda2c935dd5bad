"""df_setup's one pass over a dense B at the edges of its 32-row strips: the
symmetry check (one ulp off, or a NaN, anywhere), the digits of every row (K at
3 slices equals the oracle's emulation bit for bit, with and without an order of
the auxiliary functions) and the 64-wide chunk masks (the fractions worked out
from B)."""
import numpy as np
import pytest
import torch

from oracle import df_oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def df():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2601_08077_gb300 import build, df as dfmod
    build.build_all()
    return dfmod


def _tensor(seed, naux, nao):
    rng = np.random.default_rng(seed)
    B = rng.standard_normal((naux, nao, nao)) * np.exp2(rng.integers(-6, 1, (naux, nao, 1)))
    return np.triu(B) + np.triu(B, 1).transpose(0, 2, 1)


@pytest.mark.parametrize("nao", [1, 31, 32, 33, 64, 65, 130])
def test_setup_checks_symmetry_everywhere(df, nao):
    B = _tensor(nao, 3, nao)
    ctx = df.Context(nao, 3, 1, 2)
    ctx.setup(torch.from_numpy(B).cuda())
    spots = {(0, nao - 1), (nao - 1, 0), (nao // 2, nao - 1), (min(31, nao - 1), min(32, nao - 1))}
    for i, j in spots:
        if i != j:
            bad = B.copy()
            bad[2, i, j] = np.nextafter(bad[2, i, j], 10.0)
            with pytest.raises(df.DFError) as e:
                ctx.setup(torch.from_numpy(bad).cuda())
            assert e.value.status == -1
    bad = B.copy()
    bad[1, nao - 1, nao - 1] = np.nan
    with pytest.raises(df.DFError) as e:
        ctx.setup(torch.from_numpy(bad).cuda())
    assert e.value.status == -1


@pytest.mark.parametrize("naux,nao", [(2, 3), (130, 33), (5, 64), (4, 97)])
def test_setup_digits_and_masks(df, naux, nao):
    B = _tensor(7 * nao, naux, nao)
    pair = np.random.default_rng(nao).random((nao, nao)) < 0.05  # a screened B
    pair = pair | pair.T | np.eye(nao, dtype=bool)
    C = np.random.default_rng(1).standard_normal((nao, 5))
    perm = np.random.default_rng(2).permutation(naux)
    for T, order in ((B, None), (np.where(pair, B, 0.0), None), (B, perm)):
        ctx = df.Context(nao, naux, 5, 3)
        ctx.setup(torch.from_numpy(T).cuda(), perm=order)
        K, _ = ctx.build_K(torch.from_numpy(C).cuda(), 3)
        ref = O.emulated_exchange(T if order is None else T[order], C, 3)
        assert np.array_equal(K.cpu().numpy(), ref)
        on = (T != 0).any(0)
        nk = (nao + 63) // 64
        chunk = np.array([[on[m, 64 * k:64 * k + 64].any() for k in range(nk)] for m in range(nao)])
        upper = [chunk[m, k] for m in range(nao) for k in range(m // 64, nk)]
        rows = np.tile(chunk, (naux, 1))
        tiles = [rows[r:r + 128].any(0).sum() for r in range(0, naux * nao, 128)]
        kt, ch = ctx.sparsity()
        assert ch == pytest.approx(np.mean(upper), abs=1e-12)
        assert kt == pytest.approx(sum(tiles) / (len(tiles) * nk), abs=1e-12)


@pytest.mark.parametrize("cols", [150, 2100])
def test_rounding_at_every_exponent(df, cols):
    # digits (round to nearest even of v 2^(63-e)) of values from the row's maximum
    # down to far below its last digit, ties among them, subnormals, signed zeros and
    # a row that is subnormal throughout; 2100 columns: a whole block per row
    from oracle import crt_oracle as CO
    rng = np.random.default_rng(cols)
    j = np.arange(cols)
    A = np.zeros((6, cols))
    A[0] = np.ldexp(rng.integers(2 ** 52, 2 ** 53, cols).astype(float), -52 - j % 75)
    A[1] = np.ldexp(2.0 * rng.integers(0, 2 ** (1 + j % 51)) + 1.0, -65)   # odd multiples of half a unit (e = 0)
    A[2] = np.ldexp(2.0 * rng.integers(0, 2 ** (1 + j % 51)) + 1.0, -66 + j % 3)
    A[1, 0] = A[2, 0] = 0.75
    A[3] = rng.integers(1, 2 ** 40, cols) * 5e-324
    A[4] = 5e-324
    A[4, 1] = -0.0
    A *= rng.choice([-1.0, 1.0], (6, cols))
    e_ref, d_ref = O.split_rows(A, 8)
    e, d = df.split_int8(torch.from_numpy(A).cuda(), 8)
    assert np.array_equal(e.cpu().numpy(), e_ref.astype(np.int32))
    assert np.array_equal(d.cpu().numpy(), d_ref)
    e_ref, Ai = CO.scaled_integers(A, CO.operand_bits(cols, 9))
    e, R = df.crt_split_rows(torch.from_numpy(A).cuda(), 9)
    assert np.array_equal(e.cpu().numpy(), e_ref)
    for i, m in enumerate(CO.moduli(9)):
        assert np.array_equal(R[i].cpu().numpy(), CO.residues(Ai, m)), m


def test_refused_order_leaves_the_context_as_it_was(df):
    # a set-up context that is offered another B (packed) with an order that is no
    # permutation: DF_ERR_ARG, and the builds go on with the B that it holds
    nao, naux = 65, 20
    B = torch.from_numpy(_tensor(1, naux, nao)).cuda()
    iu = torch.triu_indices(nao, nao, device="cuda")
    other = torch.from_numpy(_tensor(2, naux, nao)).cuda()[:, iu[0], iu[1]].contiguous()
    rng = np.random.default_rng(3)
    D = torch.from_numpy(rng.standard_normal((nao, nao))).cuda()
    D = D + D.T
    C = torch.from_numpy(rng.standard_normal((nao, 7))).cuda()
    ctx = df.Context(nao, naux, 7, 3)
    ctx.setup(B)
    J, rho, K, _ = ctx.build_JK(D, C, 3)
    del B  # the context keeps it
    for perm in (np.zeros(naux, dtype=np.int32), np.arange(1, naux + 1, dtype=np.int32)):
        with pytest.raises(df.DFError) as e:
            ctx.setup_packed(other, perm)
        assert e.value.status == -1
        junk = torch.full((naux, nao, nao), float("nan"), dtype=torch.float64, device="cuda")  # takes freed memory
        J1, rho1 = ctx.build_J(D)
        K1, _ = ctx.build_K(C, 3)
        assert torch.equal(J1, J) and torch.equal(rho1, rho) and torch.equal(K1, K)


@pytest.mark.parametrize("nao", [1, 2, 15, 16, 17, 33, 129])
def test_packed_digits_at_row_ends(df, nao):
    # rows that end inside a lane's pair, inside a digit row's padding or fill it: K and the
    # masks of a packed B are the dense ones, bit for bit
    B = _tensor(50 + nao, 5, nao)
    B[:, nao // 2, :] = 0.0
    B[:, :, nao // 2] = 0.0
    Bg = torch.from_numpy(B).cuda()
    iu = torch.triu_indices(nao, nao, device="cuda")
    C = torch.from_numpy(np.random.default_rng(nao).standard_normal((nao, 3))).cuda()
    perm = [3, 0, 4, 1, 2]
    for s in (3, 6):
        dense, packed = df.Context(nao, 5, 3, s), df.Context(nao, 5, 3, s)
        dense.setup(Bg, perm)
        packed.setup_packed(Bg[:, iu[0], iu[1]].contiguous(), perm)
        assert dense.sparsity() == packed.sparsity()
        assert torch.equal(dense.build_K(C, s)[0], packed.build_K(C, s)[0])

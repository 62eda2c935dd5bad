"""The exchange build at the edges of the slice GEMM's tiles and schedule.

The first GEMM cuts nocc into tiles of a multiple of 32 columns (up to 8 digits
stacked in one MMA at 32 columns, 2 at 128), pads an odd nocc with a zero
orbital, takes nao in 64-wide K tiles, at most 5 to a chunk, and lets up to
16 / chunk steps share their accumulators; row tiles (256 rows on CTA pairs)
end at every auxiliary block.  Up to 5 slices both GEMMs are exact, so K equals
the oracle's emulation bit for bit; at 8 the fixed-point sums drop low bits
(2^-61 of their bound, with K <= 2^13 terms each far below 1e-14 of max|K|).
"""
import numpy as np
import pytest
import torch

from oracle import df_oracle as O

pytestmark = pytest.mark.gpu

SHAPES = [  # naux, nao, nocc, slices
    (130, 33, 1, 3),    # two blocks, one orbital, one K tile with 3 of 4 steps used
    (129, 35, 31, 5),   # odd nao and nocc: a pair's row tile overhangs its block
    (8, 64, 32, 4),     # one full K tile, one full 32-column tile
    (8, 65, 33, 5),     # a K tile with one value, 64-column tiles
    (6, 128, 64, 1),    # one slice: a single pass of one step
    (6, 193, 65, 2),    # 4 K tiles: four steps may share an accumulator
    (4, 320, 96, 5),    # 5 K tiles: one full chunk
    (4, 321, 97, 5),    # 6 K tiles: two chunks of 3
    (4, 100, 127, 3),   # 128-column tile, odd nocc
    (4, 130, 129, 5),   # two orbital tiles, two AO tiles
    (3, 72, 161, 8),    # two orbital tiles of 96 columns, truncated sums
    (3, 260, 40, 8),    # three AO tiles, truncated sums
]


@pytest.fixture(scope="module")
def df():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2601_08077_gb300 import build, df as dfmod
    build.build_all()
    return dfmod


@pytest.mark.parametrize("naux,nao,nocc,s", SHAPES)
def test_exchange_at_tile_edges(df, naux, nao, nocc, s):
    rng = np.random.default_rng(naux * 1000 + nao)
    B = rng.standard_normal((naux, nao, nao)) * np.exp2(rng.integers(-8, 1, (naux, nao, nao)))
    B = np.triu(B) + np.triu(B, 1).transpose(0, 2, 1)
    C = rng.standard_normal((nao, nocc)) * np.exp2(rng.integers(-4, 1, (1, nocc)))
    Bg, Cg = torch.from_numpy(B).cuda(), torch.from_numpy(C).cuda()
    ref = O.emulated_exchange(B, C, s)
    got = []
    for pairs in (0, 1, 2):
        ctx = df.Context(nao, naux, nocc, s)
        ctx.set_cluster_pairs(pairs)
        ctx.setup(Bg)
        K, _ = ctx.build_K(Cg, s)
        ctx.sync_status()
        got.append(K.cpu().numpy())
    assert np.array_equal(got[0], got[1]) and np.array_equal(got[0], got[2])
    if s <= 5:
        assert np.array_equal(got[1], ref)
    else:
        assert np.max(np.abs(got[1] - ref)) <= 1e-14 * np.max(np.abs(ref))


def _both_builds(df, naux, nao, nocc, s, modes):
    """J, rho and K of build_JK (512 threads, the Coulomb passes in the GEMMs' spare warps) under
    each pair mode, and of the separate builds."""
    rng = np.random.default_rng(naux * 1000 + nao + 1)
    B = rng.standard_normal((naux, nao, nao)) * np.exp2(rng.integers(-8, 1, (naux, nao, nao)))
    B = np.triu(B) + np.triu(B, 1).transpose(0, 2, 1)
    D = rng.standard_normal((nao, nao))
    Bg, Dg = torch.from_numpy(B).cuda(), torch.from_numpy(D + D.T).cuda()
    Cg = torch.from_numpy(rng.standard_normal((nao, nocc)) * np.exp2(rng.integers(-4, 1, (1, nocc)))).cuda()
    got = []
    for mode in modes:
        ctx = df.Context(nao, naux, nocc, s)
        if mode is not None:
            ctx.set_cluster_pairs(mode)
        ctx.setup(Bg)
        J, rho = ctx.build_J(Dg)
        K, _ = ctx.build_K(Cg, s)
        got.append([t.clone() for t in (J, rho, K)])
        J, rho, K, _ = ctx.build_JK(Dg, Cg, s)
        ctx.sync_status()
        got.append([J, rho, K])
    return got


@pytest.mark.parametrize("naux,nao,nocc,s", SHAPES)
def test_coulomb_beside_the_gemms_at_tile_edges(df, naux, nao, nocc, s):
    # both GEMMs on single CTAs, the first on pairs, both on pairs
    got = _both_builds(df, naux, nao, nocc, s, (0, 1, 2))
    for other in got[1:]:
        for x, y in zip(got[0], other):
            assert torch.equal(x, y)


@pytest.mark.parametrize("nao", [769, 800, 897])
def test_second_gemm_on_pairs_by_default(df, nao):
    # from 7 AO tile rows on (nao > 768) the default pairs the second GEMM too; an odd row
    # count leaves a pair whose second tile lies past the last row
    got = _both_builds(df, 20, nao, 9, 3, (None, 0))
    for other in got[1:]:
        for x, y in zip(got[0], other):
            assert torch.equal(x, y)


@pytest.mark.parametrize("M", [1930, 2060])
def test_product_of_many_row_tiles_on_pairs(df, M):
    # 16 tile rows, and 17, whose last CTA lies wholly past M; odd N, a ragged K
    rng = np.random.default_rng(M)
    A, B = rng.standard_normal((M, 70)), rng.standard_normal((67, 70))
    got = df.emulated_gemm(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), 3).cpu().numpy()
    assert np.array_equal(got, O.emulated_matmul(A, B.T, 3))

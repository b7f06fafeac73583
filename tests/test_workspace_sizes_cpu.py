"""Sizes of the FP64 exchange's scratch (no GPU needed)."""
import pytest


@pytest.fixture(scope="module")
def lib():
    import paper_2506_06661_gb300 as dfscf
    return dfscf.lib()


@pytest.mark.parametrize("nao,naux", [(5, 15), (100, 300), (600, 1800), (1500, 4500)])
def test_coulomb_alone_holds_no_exchange_buffers(lib, nao, naux):
    ld = lib.df_B_ld(nao)
    slices = (naux + 255) // 256
    assert lib.df_jk_work_bytes(nao, naux, 0, 0) <= 8 * (ld * (1 + slices) + naux) + 4 * 256 + 1024


@pytest.mark.parametrize("centres", [10, 20, 40, 63, 77, 120, 200, 300])
def test_exchange_scratch_is_bounded(lib, centres):
    """Digits of B: two waves of 128-row tiles, or one where two take more than 5/4 of B; X and its
    digits: 1 GB (and less than a block of B's rows above it); partial sums of K."""
    nao, naux, nocc = 5 * centres, 15 * centres, centres // 2
    digits = 14 * ((nao + 7) // 8 * 8)  # bytes of one row of B or X^T over nao, 7 BF16 planes
    wave = 152 * 128 * digits
    x = min(2 ** 30, 22 * nao * naux * nocc)
    kpart = 64 * 8 * nao * nao
    extra = lib.df_jk_work_bytes(nao, naux, nocc, 0) - lib.df_jk_work_bytes(nao, naux, 0, 0)
    b = min(2 * wave, max(lib.df_B_bytes(nao, naux, 0) * 5 // 4, wave))
    assert extra <= b + 1.05 * x + kpart + 16 * nocc * nao + 2 ** 20


@pytest.mark.parametrize("centres", [40, 63, 77, 120, 300])
def test_mixed_scf_shares_its_exchange_scratch(lib, centres):
    """The scratch of the FP64 builds, of the mixed builds and of the whitening is one region."""
    nao, naux, nocc = 5 * centres, 15 * centres, centres // 2
    fp64, mixed = (lib.df_jk_work_bytes(nao, naux, nocc, p) for p in (0, 1))
    b = [lib.df_B_bytes(nao, naux, p) for p in (0, 1)]
    scf = [lib.scf_work_bytes(nao, naux, nocc, p) for p in (0, 1)]
    assert scf[1] - scf[0] <= b[1] - b[0] + max(0, mixed - fp64) + 4096

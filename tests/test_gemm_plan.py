"""The rule that picks a projection's tiles, computed on the host (no GPU needed)."""
import pytest

from paper_2609_03311_gb300 import build as libbuild
from paper_2609_03311_gb300 import dopr

SMS = 152
# (epilogue, N, K) of the projections of hidden 1,024, 2,560 and 4,096, and small ones
WIDTHS = [(dopr.EPI_QKV, 4096, 1024), (dopr.EPI_RESID_ADD, 1024, 2048), (dopr.EPI_SWIGLU, 6144, 1024),
          (dopr.EPI_RESID_ADD, 1024, 3072), (dopr.EPI_QKV, 6144, 2560), (dopr.EPI_RESID_ADD, 2560, 4096),
          (dopr.EPI_SWIGLU, 19456, 2560), (dopr.EPI_RESID_ADD, 2560, 9728), (dopr.EPI_QKV, 6144, 4096),
          (dopr.EPI_RESID_ADD, 4096, 4096), (dopr.EPI_SWIGLU, 24576, 4096), (dopr.EPI_RESID_ADD, 4096, 12288),
          (dopr.EPI_STORE, 256, 64), (dopr.EPI_RESID_ADD, 256, 256), (dopr.EPI_SWIGLU, 256, 256)]


@pytest.fixture(scope="module", autouse=True)
def lib():
    libbuild.build()


@pytest.mark.parametrize("epi,N,K", WIDTHS)
@pytest.mark.parametrize("sms", [2, 16, SMS])
def test_tiles_are_ones_that_a_kernel_exists_for(epi, N, K, sms):
    for M in list(range(1, 1100, 7)) + [1023, 1024, 1025, 2304, 2400, 3800, 5650, 8800, 26800]:
        p = dopr.gemm_plan(epi, M, N, K, sms)
        if p["few"] or p["wide_rows"]:
            assert (p["rows"], p["cols"]) in {(r, 128) for r in (32, 64, 96, 128)} | \
                ({(r, 64) for r in (32, 64, 96)} if epi == dopr.EPI_RESID_ADD else set())
        else:
            assert (p["rows"], p["cols"]) == (128, 256)
        rest = M - p["wide_rows"] if p["wide_rows"] else M if p["few"] else 0
        assert rest <= 1024 and p["wide_rows"] % 256 == 0
        if p["wide_rows"]:  # the rows beside make one round of narrow tiles
            tiles = -(-rest // (2 * p["rows"])) * (N // p["cols"])
            assert not p["few"] and 0 < p["wide_rows"] < M and tiles <= max(sms // 2, 1)


def test_bad_arguments_are_refused():
    for args in ((4, 1, 256, 64), (-1, 1, 256, 64), (0, 0, 256, 64), (0, 1, 256, 32), (0, 1, 128, 64)):
        with pytest.raises(dopr.DoprError):
            dopr.gemm_plan(*args, SMS)

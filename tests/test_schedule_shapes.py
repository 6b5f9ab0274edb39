"""Described schedules are those that run (host only).

P5 of the tuned passes is the projection's, which writes a caller's field:
fewer rows per block on the grids whose blocks would not fill the chip, at
least 256 blocks where a block of four rows leaves that many, and the variants
with half and twice the rows are relative to it.
"""
import pytest

from paper_1601_05970_gb300 import build, fftg

GRIDS = (3, 5, 9, 15, 25, 27, 45, 75, 81, 125, 135, 225, 243)


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    fftg.load()


@pytest.mark.parametrize("N", GRIDS)
def test_projection_rows(N):
    d = [fftg.schedule_describe(N, "p5", v) for v in range(fftg.SCHED_VARIANTS)]
    rows = [x["rows"] for x in d]
    assert rows[0] == 4 or d[0]["blocks"] >= 256
    assert rows[1] == rows[0]
    assert rows[2] == max(4, rows[0] // 2) and rows[3] == 2 * rows[0]
    for x in d:
        assert x["blocks"] == -(-N * N // x["rows"])
        assert x["split"][0] * x["split"][1] == N

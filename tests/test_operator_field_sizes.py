"""A tensor that is too small for an operator's field is refused on the host."""
import pytest

from paper_1601_05970_gb300 import fftg

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,offset,nbytes,fits", [(54, 0, 432, True), (53, 0, 432, False), (54, 1, 432, False),
                                                  (55, 1, 432, True), (108, 0, 864, True), (107, 0, 864, False)])
def test_storage_room(n, offset, nbytes, fits):
    t = torch.zeros(n, dtype=torch.float64)[offset:]
    if fits:
        assert fftg._field(t, nbytes, "call").value == t.data_ptr()
    else:
        with pytest.raises(RuntimeError):
            fftg._field(t, nbytes, "call")

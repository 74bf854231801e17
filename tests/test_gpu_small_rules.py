"""FP64 solves with one block per column go back to the panels when the sliced rows do
not fit the memory.  Same posteriors either way (both solves stop at a relative
residual of 1e-13, amplified by K_ii / Sigma_ii <= 1e4: rtol 1e-9)."""
import pytest

from synth import make_catalogue
from test_gpu_tc64_fallback import _Pool, _posterior, _same

pytestmark = pytest.mark.gpu


def test_no_memory_for_the_sliced_rows(monkeypatch):
    cat = make_catalogue("c1_plain_400", n=400, truth="mean")
    base, free, short = _Pool(), _Pool(), _Pool()
    monkeypatch.setenv("GM_SPMM", "simt")
    want = _posterior(base, monkeypatch, cat)[0]
    monkeypatch.delenv("GM_SPMM")
    _same(_posterior(free, monkeypatch, cat)[0], want)
    short.limit = base.peak + 16384                 # the sliced rows take 160 KB at least
    assert free.peak > short.limit
    _same(_posterior(short, monkeypatch, cat)[0], want)
    assert short.refused > 0

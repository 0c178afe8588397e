"""Every call that returns results of a run reports its device error word: a bounded wait that gave up (bit 0,
HEOM_E_TIMEOUT) or a failed bounds check of the debug build (bit 1, HEOM_E_BOUNDS) leaves a half-advanced state, which
must not come back as a result.  The word is set here from the host, in the run's workspace; it follows the counter of
records, which is found by its value."""
import numpy as np
import pytest

from paper_1803_03498_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def heom():
    from paper_1803_03498_gb300.build import build
    build()
    from paper_1803_03498_gb300 import heom as h
    h.load()
    return h


def _error_word(r):
    """The workspace as 64-bit words and the index of the error word."""
    import torch
    ws = r._ws[(-r._ws.data_ptr()) % 256:]
    words = ws[: ws.numel() // 8 * 8].view(torch.int64)
    r.propagate(1.0, 36, 1)  # the start and 36 steps
    torch.cuda.synchronize()
    at = set(torch.nonzero(words == 37)[:, 0].tolist())
    r.propagate(1.0, 6, 1)
    torch.cuda.synchronize()
    at &= set(torch.nonzero(words == 43)[:, 0].tolist())
    assert len(at) == 1
    return words, at.pop() + 1


@pytest.mark.parametrize("bit,name", [(1, "HEOM_E_TIMEOUT"), (2, "HEOM_E_BOUNDS")])
@pytest.mark.parametrize("precision", ["fp64", "fp32_mixed"])
def test_readers_report_the_error_word(heom, bit, name, precision):
    p = wl.dimer()
    r = heom.Run(p.system, p.rho0_re, p.rho0_im, precision=precision, max_records=64)
    words, at = _error_word(r)
    rho = r.sigma0()
    words[at] = bit
    for call in (r.observables, r.sigma0, lambda: r.get_ados(0, r.n_ado), lambda: r.rhs_eval(0, r.n_ado)):
        with pytest.raises(heom.HeomError) as ei:
            call()
        assert ei.value.code == getattr(heom, name)
    words[at] = 0
    assert np.array_equal(r.sigma0(), rho) and r.observables().shape[0] == 43
    r.close()

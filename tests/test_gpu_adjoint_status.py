"""A bounded wait that runs out in one of the adjoint's passes reaches the caller:
NLSE_ETIMEOUT from the sweep it happened in, no loss and no gradient, and the
context stays usable for the next handle."""
import numpy as np
import pytest

from paper_2306_15678_gb300 import beams, capi, configs
from paper_2306_15678_gb300.adjoint import AdjointMarch

pytestmark = pytest.mark.gpu

COL, ROW, BACK = "NLSE_DEBUG_COL_EXTRA_TX", "NLSE_DEBUG_ROW_EXTRA_TX", "NLSE_DEBUG_ADJ_BACK_EXTRA_TX"
STAGED = {"cols": capi.NLSE_COL_TMA | 2, "row_radix": capi.NLSE_ROW_STAGED | 16}


def problem(n):
    cfg = configs.scaled(configs.cfg_dense_fp32(), n)
    U0 = beams.make_field(cfg).astype(np.complex64)
    return cfg, U0, 1.1 * np.abs(U0.astype(np.complex128)) ** 2


def sweep(cfg, U0, D, prec, launch):
    fit = AdjointMarch(cfg, 1, 1, precision=prec)
    if launch:
        fit.set_launch(launch)
    fit.set_target(D)
    return fit


@pytest.mark.parametrize("prec,n,launch,hook", [("fp32", 512, None, COL), ("fp32", 2048, STAGED, ROW),
                                                ("fp64", 512, None, COL)])
def test_forward_reports_a_wait_that_ran_out(monkeypatch, prec, n, launch, hook):
    """Block 0 of the staged pass expects 16 bytes that its copies never bring."""
    cfg, U0, D = problem(n)
    monkeypatch.setenv(hook, "16")
    fit = sweep(cfg, U0, D, prec, launch)
    with pytest.raises(capi.NlseError) as ei:
        fit.forward(U0)
    assert ei.value.status == capi.NLSE_ETIMEOUT
    with pytest.raises(capi.NlseError) as ei:
        fit.backward()
    assert ei.value.status == capi.NLSE_ESTATE
    fit.close()
    monkeypatch.delenv(hook)
    fit = sweep(cfg, U0, D, prec, launch)
    assert 0.0 < fit.forward(U0) < 1.0
    fit.backward()
    fit.close()


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_backward_reports_a_wait_that_ran_out(monkeypatch, prec):
    cfg, U0, D = problem(512)
    monkeypatch.setenv(BACK, "16")
    fit = sweep(cfg, U0, D, prec, None)
    assert 0.0 < fit.forward(U0) < 1.0
    with pytest.raises(capi.NlseError) as ei:
        fit.backward()
    assert ei.value.status == capi.NLSE_ETIMEOUT
    assert 0.0 < fit.forward(U0) < 1.0  # the word is cleared at the start of a sweep
    fit.close()

"""What the options of the 27-point path read: what a call takes."""
import pytest
import torch

from paper_1901_11350_gb300 import binding as B
from paper_1901_11350_gb300 import inputs as I

SC = I.cfg_sc_128(4)["hamiltonian"]


def _ctx(dims, prec="f32", **options):
    c = B.Context(I.simple_cubic(*dims), SC, prec)
    for k, v in options.items():
        c.set_option(k, v)
    return c


def _read(c):
    return tuple(c.get_option(k) for k in ("heun_lean", "cubic_rows", "cubic_rows_corr"))


def test_columns_and_family_of_a_heun_call():
    assert _read(_ctx((32, 16, 4))) == (1, 2, 2)
    # ragged: the lean passes too, two columns in the predictor alone
    assert _read(_ctx((33, 16, 4))) == (1, 2, 1) and _read(_ctx((32, 24, 4))) == (1, 2, 1)
    assert _read(_ctx((33, 16, 4), cubic_lean=0)) == (0, 1, 1)
    assert _read(_ctx((33, 16, 4), generic_stencil=1))[0] == 0
    assert _read(_ctx((32, 16, 4), "f64")) == (0, 1, 1)
    assert _read(_ctx((32, 16, 4), cubic_rows=1)) == (1, 1, 1)
    with pytest.raises(B.SpinError):
        _ctx((32, 16, 4)).set_option("heun_lean", 1)


@pytest.mark.gpu
def test_split_reads_that_of_the_calls_made():
    for solver in ("depondt", "heun"):
        c = _ctx((33, 16, 40))
        n = c.spins(I.random_spins(c.N, 1))
        assert c.get_option("planes_per_cta") == 0 and c.get_option("planes_per_cta_corr") == 0
        c.llg_step(n, 1, solver=solver)
        assert c.get_option("planes_per_cta") >= 1 and c.get_option("planes_per_cta_corr") >= 1
    torch.cuda.synchronize()


def test_a_choice_for_the_corrector_leaves_the_predictor_alone():
    assert _read(_ctx((33, 16, 4), cubic_rows_corr=2)) == (1, 2, 2)
    assert _read(_ctx((32, 16, 4), cubic_rows_corr=1)) == (1, 2, 1)
    assert _read(_ctx((32, 16, 4), planes_per_cta_corr=3)) == (1, 2, 1)
    assert _read(_ctx((32, 16, 4), planes_per_cta=3)) == (1, 1, 1)
    assert _read(_ctx((32, 16, 4), cubic_rows=1, cubic_rows_corr=2)) == (1, 1, 2)
    assert _read(_ctx((32, 16, 4), cubic_rows_corr=1, cubic_rows=2)) == (1, 2, 2)

"""A constant row is reported as degenerate whatever its value and length: n
copies of a number with few bits have an exact sum, whose division by n gives the
number back (a product with 1 / n need not), so every centred value is zero."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("n", [20, 49, 98, 103, 999])
@pytest.mark.parametrize("value", [1.0, -3.0, 1234.5])
def test_constant_row_is_degenerate(vl, prec, n, value):
    m, row = 6, 2
    g = torch.Generator(device="cuda").manual_seed(n)
    E = torch.randn((m, n), dtype=torch.float64, device="cuda", generator=g)
    E[row] = value
    D, B0 = torch.empty_like(E[:, :m].contiguous()), torch.empty_like(E[:, :m].contiguous())
    order = torch.arange(m, dtype=torch.int32, device="cuda")
    h = vl.Handle(0)
    calls = (lambda: vl.vl_pairwise_measure(h, E, prec, None, None, D),
             lambda: vl.vl_fit_b(h, E, order, None, prec, B0, None),
             lambda: vl.vl_causal_order_standard(h, E, prec, order.clone(), None))
    for call in calls:
        call()
        with pytest.raises(vl.VLError) as ei:
            h.sync()
        assert ei.value.code == 4  # VL_ERR_DEGENERATE
    h.close()

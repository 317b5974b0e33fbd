"""GPU test of the outputs that the binding of rs_lgssm_step_ess returns: given tensors or new ones,
the ESS among them where the caller names neither."""
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("give", ["none", "ess", "log_total", "both"])
def test_outputs_are_returned(rs, give):
    N = 5000
    args = dict(phi=0.9, sigma_x=1.0, y=0.3, sigma_y=0.5, seed=4, step=0)
    out = {k: torch.empty(1, dtype=torch.float64, device=DEV) for k in ("ess", "log_total")
           if give in (k, "both")}
    x = torch.empty(N, dtype=torch.float32, device=DEV)
    with rs.Handle(N) as h:
        logw, ess, log_total = rs.rs_lgssm_step_ess(h, x, None, True, **args, **out)
        want = torch.empty(2, dtype=torch.float64, device=DEV)
        rs.rs_ess(h, logw, out=want[:1], log_total=want[1:])
        assert rs.rs_last_error(h) == rs.RS_OK
    assert logw.numel() == N
    assert (ess is None) == (give == "log_total") and (log_total is None) == (give in ("none", "ess"))
    for got, w, name in ((ess, want[0], "ess"), (log_total, want[1], "log_total")):
        if got is not None:
            assert out.get(name, got) is got
            assert abs(float(got) - float(w)) <= 2.0 ** -39 * abs(float(w))

"""A training run one of whose bounded waits ran out: the tiles' missing sums reach neither the
parameters nor the loss history, the call reports it, and the next run is as if it had not been."""
import pytest
import torch

from paper_2203_15963_gb300 import native

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,steps", [(128, 1), (384, 5), (16384, 40)])
def test_stopped_training_keeps_parameters(batch, steps):
    native.build()
    native.load()
    inp = torch.empty((16384, 3), dtype=torch.float32, device="cuda")
    tg = torch.empty((16384, 7), dtype=torch.float32, device="cuda")
    native.blacklight_mlp_dataset(16384, 7, inp, tg)
    start = torch.empty(native.MLP_PARAMS, dtype=torch.float32, device="cuda")
    native.blacklight_mlp_init(start, 3)
    native.blacklight_mlp_normalise(inp, tg, start)

    def run(call):
        p, hist = start.clone(), torch.full((steps,), -1.0, device="cuda")
        return call(p, inp, tg, batch, steps, 1e-3, 1e-4, loss_history=hist), p, hist

    rc, p, hist = run(native.blacklight_mlp_train)
    assert rc == 0 and not torch.equal(p, start) and float(hist.min()) > 0.0
    stopped, q, none = run(native.blacklight_selftest_train_stopped)
    assert stopped == native.BL_ETIMEOUT
    assert torch.equal(q, start) and bool((none == -1.0).all())
    again = run(native.blacklight_mlp_train)
    assert again[0] == 0 and torch.equal(again[1], p) and torch.equal(again[2], hist)

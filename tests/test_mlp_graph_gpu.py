"""The training step's graph against the plain launches of the same kernels (backward, then adamw): the
weights and losses are equal bit for bit, with new inputs in new buffers each step, batch sizes that
change (ragged ones among them, more of them than graphs are kept), with and without mask and loss,
and on another stream. Shapes include odd multiples that the first layer's 32 x 64 tiles and the
four-element split-K sums do not divide."""
import numpy as np
import pytest

import paper_1910_10391_gb300 as rad

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_in,width,depth,n_out", [(62, 256, 3, 2048), (3, 66, 2, 34), (64, 64, 2, 128)])
def test_graph_step_equals_plain_step(n_in, width, depth, n_out):
    import torch
    g = torch.Generator(device="cuda").manual_seed(1)
    new = lambda *s: torch.randn(*s, generator=g, device="cuda")  # noqa: E731
    nets = [rad.MLP(n_in, width, depth, n_out, max_batch=600, seed=3) for _ in range(2)]
    side = torch.cuda.Stream()
    batches = [600] * 4 + [599, 600, 599, 33, 33, 33, 1, 1, 2, 2, 64, 64, 600, 600, 33, 33]
    for k, B in enumerate(batches):
        x, t = new(B, n_in), new(B, n_out)
        mask = (new(B, n_out) > 0).float() if k % 3 else None
        loss = [torch.zeros(1, device="cuda") if k % 4 else None for _ in nets]
        st = side if k % 5 == 4 else None
        if st is not None:
            st.wait_stream(torch.cuda.current_stream())
        nets[0].train_step(x, t, 1e-3 * (1 + k), 1e-4, loss[0], mask, stream=st)
        nets[1].backward(x, t, loss[1], mask, stream=st)
        nets[1].adamw(1e-3 * (1 + k), weight_decay=1e-4, stream=st)
        torch.cuda.synchronize()
        if loss[0] is not None:
            assert torch.equal(loss[0], loss[1]), (k, B)
        for what in range(4):
            assert np.array_equal(nets[0].get(what), nets[1].get(what)), (k, B, what)
    y = [n.forward(new(40, n_in) * 0 + 0.5) for n in nets]  # the BF16 copies too
    assert torch.equal(y[0], y[1])
    assert rad.rad_device_status(1) == rad.RAD_OK
    for n in nets:
        n.close()

"""The bounded waits of the message kernel: one that runs out is reported, leaves no sums
that look like results and ends the kernel in order, so that the next call is right."""
import numpy as np
import pytest

from tests.test_gpu_mpnn_fused import csr_graph, sg  # noqa: F401  (a fixture)

pytestmark = pytest.mark.gpu


def message_sums(sg, model, g, tries, keep):  # noqa: F811
    import torch
    dev = dict(device="cuda")
    h, p1 = torch.empty((2, g.npad, 128), **dev)
    hb, eb = (torch.empty((r, 128), dtype=torch.int16, **dev) for r in (g.npad, g.Epad))
    Mb = torch.full((g.npad, 128), 0x3F80, dtype=torch.int16, **dev)
    mask = torch.zeros((g.Epad, 4), dtype=torch.int32, **dev) if keep else None
    status = torch.zeros(1, dtype=torch.int32, **dev)
    sg._call("mpnn_encode_edges", g.E, g.ef, model.Wt["edge"], eb, None)
    sg._call("mpnn_encode_nodes", g.n, g.npad, g.nf, model.Wt["node"], model.Wt["msg0"], h, hb,
             p1, None)
    sg._call("mpnn_message_sums_checked", g.n, g.E, g.off, g.nbr, g.dst, hb, eb,
             model.Wt["msg0"], p1, Mb, mask, sg._i32(tries), status, None)
    return int(status.item()), Mb[:g.n]


# a tile a block, a dozen, nodes over several tiles, blocks without edges
@pytest.mark.parametrize("degrees", [[5] * 40, [10] * 22_000, [300] * 80, [0] * 9_000 + [9] * 99],
                         ids=["one_tile", "many_tiles", "wide", "empty_blocks"])
@pytest.mark.parametrize("keep", [False, True])
def test_a_wait_that_runs_out_is_reported(sg, degrees, keep):  # noqa: F811
    import torch
    g, model = csr_graph(sg, np.asarray(degrees, dtype=np.int64), seed=1), sg.MPNN(seed=2)
    rc, ref = message_sums(sg, model, g, -1, keep)
    assert rc == 0
    nan, edges = 0x7FC0, torch.as_tensor(np.asarray(degrees) > 0, device="cuda")
    for tries in (0, 1, 0, 3):
        rc, Mb = message_sums(sg, model, g, tries, keep)
        if tries == 0:  # every block with edges gives up: its nodes say so
            assert rc == 4
            assert bool((Mb[edges] == nan).all())
        elif rc == 0:   # (a try waits for a while itself: it may be enough)
            assert torch.equal(Mb, ref)
        rows = (Mb == nan).all(dim=1)
        assert torch.equal(Mb[~rows], ref[~rows])
        again, Mb = message_sums(sg, model, g, -1, keep)
        assert again == 0 and torch.equal(Mb, ref)


def test_a_pass_whose_wait_ran_out_is_no_result(sg, monkeypatch):  # noqa: F811
    import torch
    rng = np.random.default_rng(7)
    n = 3000
    x = rng.uniform(0, 1.6e-3 * n ** (1 / 3), size=(n, 3))
    state = dict(x=x, v=rng.normal(scale=0.1, size=(n, 3)), w=rng.normal(size=(n, 3)))
    R = np.full(n, 1e-3)
    g = sg.make_graph(state["x"], state["v"], state["w"], R, 1e-3)
    model = sg.MPNN(seed=3)
    T = sg.target_buffer(rng.normal(size=(n, sg.OUT)), g.npad)
    y = model.forward(g, keep=False)
    loss = model.loss_and_grad(g, T)
    G = {k: v.clone() for k, v in model.G.items()}

    monkeypatch.setattr(sg.MPNN, "TRIES", 0)
    for keep in (False, True):
        assert bool(torch.isnan(model.forward(g, keep=keep)[:n, :sg.OUT]).all())
        with pytest.raises(sg._dem.DemError, match="timed out"):
            model.check()
    with pytest.raises(sg._dem.DemError, match="timed out"):
        model.loss_and_grad(g, T)
    with pytest.raises(sg._dem.DemError, match="timed out"):
        sg.predict(model, state, R)

    monkeypatch.setattr(sg.MPNN, "TRIES", -1)
    assert torch.equal(model.forward(g, keep=False), y)
    assert model.loss_and_grad(g, T) == loss
    assert all(torch.equal(model.G[k], v) for k, v in G.items())
    assert np.isfinite(sg.predict(model, state, R)).all()

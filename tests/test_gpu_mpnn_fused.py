"""The fused layers against the layer-by-layer kernels, and the graph kernels at the
edges of their tiles.  Both sides add the same numbers in the same order, so the
comparisons are exact; only the loss is summed in another order, and is held to the
error of an fp32 sum."""
from types import SimpleNamespace

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sg():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2507_12610_gb300 import build
    build.build()
    from paper_2507_12610_gb300 import surrogate
    surrogate.load()
    return surrogate


def bf16_bits(a):
    import torch
    return torch.as_tensor(np.asarray(a, np.float32)).to(torch.bfloat16).view(torch.int16).cuda()


def csr_graph(sg, degrees, seed):
    """A graph with these in-degrees, random senders and random features."""
    import torch
    rng = np.random.default_rng(seed)
    n, E = len(degrees), int(np.sum(degrees))
    npad, Epad = sg.pad64(n), sg.pad64(E)

    def features(rows, padded):
        f = np.zeros((padded, 16))
        f[:rows, :7] = rng.normal(size=(rows, 7))
        f[:rows, 7] = 1.0
        return bf16_bits(f.reshape(-1))

    dev = dict(device="cuda")
    return SimpleNamespace(
        n=n, npad=npad, E=E, Epad=Epad, nf=features(n, npad), ef=features(E, Epad),
        off=torch.as_tensor(np.concatenate([[0], np.cumsum(degrees)]).astype(np.int64), **dev),
        dst=torch.as_tensor(np.repeat(np.arange(n), degrees).astype(np.int32).copy() if E else
                            np.zeros(1, np.int32), **dev),
        nbr=torch.as_tensor(rng.integers(0, n, max(E, 1)).astype(np.int32), **dev))


class Layers:
    """The network from the layer-by-layer kernels."""

    def __init__(self, sg, model, g):
        import torch
        self.sg, self.model, self.g, self.torch = sg, model, g, torch
        self.z = torch.zeros(256, dtype=torch.float32, device="cuda")

    def new(self, rows, cols, dtype=None):
        return self.torch.empty((rows, cols), dtype=dtype or self.torch.float32, device="cuda")

    def product(self, rows, X, name, relu):
        sg, (K, N) = self.sg, self.sg.LAYERS[name]
        C, Cb = self.new(rows, N), self.new(rows, N, self.torch.int16)
        sg._call("mpnn_gemm", rows, N, K, X, self.model.Wt[name], C, Cb, self.z,
                 sg._i32(2 if relu else 0), sg._i32(0), None)
        return C, Cb

    def forward(self):
        sg, g, b16 = self.sg, self.g, self.torch.int16
        h, hb = self.product(g.npad, g.nf, "node", True)
        e, eb = self.product(g.Epad, g.ef, "edge", True)
        self.X, self.Z = {"node": g.nf.view(-1, 16), "edge": g.ef.view(-1, 16)}, {}
        self.Z["node"], self.Z["edge"] = h.clone(), e
        for r in range(sg.ROUNDS):
            Xm = self.new(g.Epad, 400, b16)
            sg._call("mpnn_gather_edges", g.E, g.Epad, sg._i32(128), sg._i32(128), g.dst, g.nbr,
                     hb, eb, Xm, None)
            m, _ = self.product(g.Epad, Xm, f"msg{r}", True)
            M = self.new(g.npad, 128)
            sg._call("mpnn_segment_sum", g.n, g.npad, sg._i32(128), g.off, m, M, None)
            Xu = self.new(g.npad, 272, b16)
            sg._call("mpnn_concat_rows", g.n, g.npad, sg._i32(128), sg._i32(128), hb, M, Xu, None)
            u, _ = self.product(g.npad, Xu, f"upd{r}", True)
            sg._call("mpnn_residual", g.npad * 128, h, u, hb, None)
            self.X[f"msg{r}"], self.Z[f"msg{r}"] = Xm, m
            self.X[f"upd{r}"], self.Z[f"upd{r}"] = Xu, u
        Xd = self.new(g.npad, 144, b16)
        sg._call("mpnn_concat_rows", g.n, g.npad, sg._i32(128), sg._i32(0), hb, None, Xd, None)
        self.X["dec"] = Xd
        return self.product(g.npad, Xd, "dec", False)[0]

    def input_grad(self, name, dZ):
        """dZ through the relu, and the gradient of the layer's inputs."""
        sg, rows = self.sg, dZ.shape[0]
        if name != "dec":
            sg._call("mpnn_relu_backward", dZ.numel(), self.Z[name], dZ, None)
        self.Z[name] = self.new(*dZ.shape, self.torch.int16)
        sg._call("mpnn_to_bf16", dZ.numel(), dZ, self.Z[name], None)
        W = self.model.Wb[name]
        if name in ("edge", "node"):
            return None
        dX = self.new(rows, W.shape[0])
        sg._call("mpnn_gemm", rows, W.shape[0], W.shape[1], self.Z[name], W, dX, None, None,
                 sg._i32(0), sg._i32(0), None)
        return dX

    def weight_grad(self, name):
        """X^T dZ from transposed copies."""
        sg, b16, (kin, nout) = self.sg, self.torch.int16, self.sg.LAYERS[name]
        X, Z, kp = self.X[name], self.Z[name], sg.pad64(kin)
        rows, G = X.shape[0], self.new(kp, nout)
        XT, ZT = self.torch.zeros((kp, rows), dtype=b16, device="cuda"), self.new(nout, rows, b16)
        sg._call("mpnn_transpose_bf16", kin, rows, X, XT, None)
        sg._call("mpnn_transpose_bf16", nout, rows, Z, ZT, None)
        splits = max(1, min(64, rows // 4096))
        sg._call("mpnn_gemm_split", kp, nout, rows, sg._i32(splits), XT, ZT, G, sg._i32(0),
                 self.new(splits * kp, nout), None)
        return G

    def backward(self, dy):
        """The gradients of every layer's output, masked and in bf16, in self.Z."""
        sg, g = self.sg, self.g

        def segment(dX, c0, perm=None):
            out = self.new(g.npad, 128)
            sg._call("mpnn_segment_sum_cols", g.n, g.npad, sg._i32(128), dX.shape[1],
                     sg._i32(c0), g.off, perm, dX, out, None)
            return out

        dh = self.input_grad("dec", dy.clone())[:, :128].clone()
        de = self.torch.zeros((g.Epad, 128), device="cuda")
        for r in reversed(range(sg.ROUNDS)):
            dXu = self.input_grad(f"upd{r}", dh.clone())
            dh += dXu[:, :128]
            dM, dm = dXu[:, 128:256].contiguous(), self.new(g.Epad, 128)
            sg._call("mpnn_gather_rows", g.E, g.Epad, sg._i32(128), g.dst, dM, dm, None)
            dXm = self.input_grad(f"msg{r}", dm)
            dh += segment(dXm, 0)
            dh += segment(dXm, 128, g.perm)
            de += dXm[:, 256:384]
        self.input_grad("edge", de)
        self.input_grad("node", dh.clone())
        return dh


def _degrees(name):
    rng = np.random.default_rng(5)
    return {
        "one_node_no_edge": [0],
        "one_node_one_edge": [1],
        "no_edges": [0] * 65,
        "tiles_of_128": [128] * 7,                       # every node a whole tile
        "over_tiles": [127, 1, 129, 0, 0, 300, 1000, 3],  # nodes over several tiles
        "last_columns": [113, 15, 112, 16, 111, 17],      # runs ending in a tile's last 16
        "one_edge_each": [1] * 300,                       # a run an edge
        "gaps": (rng.random(4000) < 0.1).astype(int),     # mostly nodes without edges
        "bed": rng.integers(0, 17, 6_001),                # more than a tile a block
        "wide": rng.integers(0, 400, 700),
        "63": rng.integers(0, 12, 63), "64": rng.integers(0, 12, 64),
        "19457": rng.integers(0, 3, 152 * 128 + 1),       # a node tile past 2 a block
    }[name]


@pytest.mark.parametrize("name", ["one_node_no_edge", "one_node_one_edge", "no_edges",
                                  "tiles_of_128", "over_tiles", "last_columns", "one_edge_each",
                                  "gaps", "bed", "wide", "63", "64", "19457"])
def test_fused_forward_gives_the_bits_of_the_layers(sg, name):
    import torch
    g = csr_graph(sg, np.asarray(_degrees(name), dtype=np.int64), seed=len(name))
    model = sg.MPNN(seed=2)
    ref = Layers(sg, model, g).forward()
    assert torch.isfinite(ref).all()
    for keep in (False, True):  # the kernels that leave the relu masks are others
        got = model.forward(g, keep=keep)
        assert torch.equal(got.view(torch.int32), ref.view(torch.int32)), keep


@pytest.mark.parametrize("n", [1, 2, 64, 65, 255, 257, 5_000, 8_300])
def test_backward_against_the_layers(sg, n):
    # symmetric graphs (a bed's density; n = 2: one pair)
    import torch
    rng = np.random.default_rng(n)
    x = rng.uniform(0, 1.6e-3 * n ** (1 / 3) if n > 2 else 1e-3, size=(n, 3))
    v, w = rng.normal(scale=0.1, size=(2, n, 3))
    g = sg.Graph(x, v, w, np.full(n, 1e-3), 2.2e-3, 0.1, 1e-3)
    model = sg.MPNN(seed=3)
    T = sg.target_buffer(rng.normal(size=(n, sg.OUT)), g.npad)
    layers = Layers(sg, model, g)
    y = layers.forward()
    dy = 2.0 * (y - T) * np.float32(1.0 / (n * sg.OUT))
    dh = layers.backward(dy)

    loss = model.loss_and_grad(g, T)
    exact = float(((y.double() - T.double()) ** 2).sum()) / (n * sg.OUT)
    assert abs(loss - exact) <= y.numel() * 2.0 ** -23 * exact
    for name, (kin, nout) in sg.LAYERS.items():
        assert torch.equal(model.G[name], layers.weight_grad(name)), name

    # the states' gradients: the same calls as backward() makes
    model.forward(g)
    st, b16 = model.state, torch.int16
    dyb, zb, dMb = layers.Z["dec"], layers.new(g.npad, 128, b16), layers.new(g.npad, 128, b16)
    d, dX, de = layers.new(g.npad, 128), layers.new(g.Epad, 256), layers.new(g.Epad, 128)
    zm, zeb = layers.new(g.Epad, 128, b16), layers.new(g.Epad, 128, b16)
    sg._call("mpnn_grad_decode", g.npad, dyb, model.Wb["dec"], st["u"][-1], d, zb, None)
    for r in reversed(range(sg.ROUNDS)):
        assert torch.equal(zb[:n], layers.Z[f"upd{r}"][:n]), r
        sg._call("mpnn_grad_update", g.npad, zb, model.Wb[f"upd{r}"], d, dMb, None)
        sg._call("mpnn_grad_messages", g.E, g.dst, dMb, st["m"][r], model.Wb[f"msg{r}"], st["eb"],
                 sg._i32(r == sg.ROUNDS - 1), sg._i32(r == 0), zm, dX, de, zeb, None)
        sg._call("mpnn_grad_nodes", n, g.npad, g.off, g.perm, dX, st["u"][r - 1] if r else None,
                 None if r else st["hb"][0], d, zb, None)
        assert torch.equal(zm[:g.E], layers.Z[f"msg{r}"][:g.E]), r
    assert torch.equal(zb[:n], layers.Z["node"][:n])
    assert torch.equal(zeb[:g.E], layers.Z["edge"][:g.E])
    assert torch.equal(d[:n], dh[:n])


@pytest.mark.parametrize("n", [1, 255, 256, 2047, 2048, 2049, 6000])
def test_cell_graph_is_the_all_pairs_graph(sg, n):
    # 2048 nodes a tile of the scans, 8 lanes a node, four nodes a load of the box
    import torch
    rng = np.random.default_rng(n)
    x = rng.uniform(0, 1.2e-3 * n ** (1 / 3), size=(n, 3))
    z, R = np.zeros_like(x), np.full(n, 1e-3)
    a = sg.Graph(x, z, z, R, 2.2e-3, 0.1, 1e-3)
    b = sg.Graph(x, z, z, R, 2.2e-3, 0.1, 1e-3, all_pairs=True)
    assert a.E == b.E and torch.equal(a.off, b.off)
    assert torch.equal(a.nbr[:a.E], b.nbr[:b.E]) and torch.equal(a.dst[:a.E], b.dst[:b.E])
    assert torch.equal(a.nf, b.nf) and torch.equal(a.ef, b.ef)


def test_graph_and_features_take_pointers_off_the_16_byte_grid(sg):
    import ctypes
    import torch
    rng = np.random.default_rng(3)
    n = 1001
    xs, z, R = rng.uniform(0, 0.014, size=(n, 3)), np.zeros((n, 3)), np.full(n, 1e-3)
    g = sg.Graph(xs, z, z, R, 2.2e-3, 0.1, 1e-3)
    i64 = lambda k: torch.empty(k, dtype=torch.int64, device="cuda")
    x = torch.empty(3 * n + 1, dtype=torch.float32, device="cuda")[1:]
    x.copy_(g.x.reshape(-1))
    cells, ne = 1 << 16, ctypes.c_int64(0)
    off, nbr, dst = i64(n + 1), torch.empty_like(g.nbr), torch.empty_like(g.dst)
    sg._call("mpnn_graph_cells", n, x, 2.2e-3, cells, i64(2 * (cells + 1) + 2 * n + 1),
             torch.empty(6, device="cuda"), i64(n), off, nbr, dst, nbr.numel(),
             ctypes.pointer(ne), None)
    assert ne.value == g.E and torch.equal(off, g.off)
    assert torch.equal(nbr[:g.E], g.nbr[:g.E]) and torch.equal(dst[:g.E], g.dst[:g.E])
    nf = torch.empty(g.nf.numel() + 1, dtype=torch.int16, device="cuda")[1:]
    ef = torch.empty(g.ef.numel() + 1, dtype=torch.int16, device="cuda")[1:]
    sg._call("mpnn_features", n, g.npad, g.E, g.Epad, g.dst, g.nbr, x, g.v, g.w, g.R, 0.1, 1e-3,
             nf, ef, None)
    assert torch.equal(nf, g.nf) and torch.equal(ef, g.ef)

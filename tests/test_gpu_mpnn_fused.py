"""The fused forward layers against the layer-by-layer kernels, and the graph
kernels at the edges of their tiles.  Both sides add the same numbers in the same
order, so every comparison is exact."""
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
    ref = model.forward(g, keep=True)
    got = model.forward(g, keep=False)
    assert torch.isfinite(ref).all()
    assert torch.equal(got.view(torch.int32), ref.view(torch.int32))


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

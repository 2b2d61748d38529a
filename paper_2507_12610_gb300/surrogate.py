"""Learned surrogate: a message-passing network over the particle neighbour
graph that predicts each particle's mean linear and angular acceleration
over a stride of DEM steps, trained on trajectories of the GPU DEM itself,
with the DEM as its fallback and as the judge of its error.

Network (hidden width 128, bf16 weights, fp32 accumulation; every layer's
bias is carried by a constant-1 input column):
  node encoder   h  = relu([node features, 1] W_n)                 16 -> 128
  edge encoder   e  = relu([edge features, 1] W_e)                 16 -> 128
  3 rounds       m_ij = relu([h_i, h_j, e_ij, 1] W_m)             400 -> 128
                 M_i  = sum over neighbours j of m_ij (receiver i)
                 h_i += relu([h_i, M_i, 1] W_u)                    272 -> 128
  decoder        y_i = [h_i, 1] W_d   (6 outputs: a_i, R_i alpha_i) 144 -> 6
The neighbour graph joins particles closer than 2.2 R_max.  The graph, the
loss and the Adam update run in the kernels of mpnn.cu, the layers forward in
mpnn_layers.cu and backward in mpnn_grad.cu (include/mpnn.h); this module only
allocates buffers (PyTorch device memory) and sequences the calls.  Sums follow the graph's
CSR order, so forward and backward passes are deterministic.
"""
from __future__ import annotations

import ctypes
import math
import struct

import numpy as np

from . import dem as _dem

EXPORTS = ("mpnn_gemm", "mpnn_gemm_split", "mpnn_transpose_bf16", "mpnn_to_bf16",
           "mpnn_graph", "mpnn_graph_cells", "mpnn_reverse_edges", "mpnn_features", "mpnn_gather_edges",
           "mpnn_concat_rows", "mpnn_residual", "mpnn_gather_rows", "mpnn_segment_sum",
           "mpnn_segment_sum_cols", "mpnn_segment_sum_perm", "mpnn_relu_backward",
           "mpnn_adam", "mpnn_mse", "mpnn_encode_nodes",
           "mpnn_encode_nodes_checked", "mpnn_encode_edges", "mpnn_message_sums",
           "mpnn_message_sums_checked", "mpnn_update_nodes", "mpnn_update_nodes_checked",
           "mpnn_grad_decode", "mpnn_grad_update", "mpnn_grad_messages", "mpnn_grad_nodes",
           "mpnn_grad_weights")

H = 128          # hidden width
ROUNDS = 3       # message-passing rounds
OUT = 6          # a (3), R alpha (3)
# (inputs incl. the constant column, outputs) per layer
LAYERS = {"node": (16, H), "edge": (16, H), "dec": (H + 16, 64)}
for _r in range(ROUNDS):
    LAYERS[f"msg{_r}"] = (3 * H + 16, H)
    LAYERS[f"upd{_r}"] = (2 * H + 16, H)


def pad64(n: int) -> int:
    return max(64, (n + 63) // 64 * 64)


_lib = None


def load():
    global _lib
    if _lib is None:
        lib = _dem.load()
        for name in EXPORTS:
            getattr(lib, name).restype = ctypes.c_int
        import torch
        _CONVERT[torch.Tensor] = lambda t: ctypes.c_void_p(t.data_ptr())
        _lib = lib
    return _lib


# C arguments by Python type (other types: C values as they are, or tensors)
_CONVERT = {int: ctypes.c_int64, float: ctypes.c_float, bool: ctypes.c_int32,
            type(None): lambda _: ctypes.c_void_p(0), ctypes.c_int32: lambda v: v,
            ctypes.c_void_p: lambda v: v}


def _convert(a):
    if isinstance(a, (ctypes._SimpleCData, ctypes._Pointer)):
        return a
    for t in (float, bool, int):  # and types derived from them
        if isinstance(a, t):
            return _CONVERT[t](a)
    return ctypes.c_void_p(a.data_ptr())


def _call(name, *args):
    get = _CONVERT.get
    lib = _lib or load()
    rc = getattr(lib, name)(*[get(type(a), _convert)(a) for a in args])
    if rc != 0:
        raise _dem.DemError(rc, name)


def _i32(v):
    return ctypes.c_int32(int(v))


def _upload(arrays, dev):
    """Float32 copies of host arrays on the device, each from a 16-byte boundary, by
    one transfer (four transfers and numpy's one-thread conversion were 0.4 ms of a
    100,000-sphere stride)."""
    import torch
    arrays = [np.asarray(a) for a in arrays]
    start = np.cumsum([0] + [(a.size + 3) // 4 * 4 for a in arrays]).tolist()
    host = torch.empty(start[-1], dtype=torch.float32)
    for a, k in zip(arrays, start):
        part = host[k:k + a.size].view(a.shape)
        # what torch converts (by its threads); numpy takes the rest
        if a.dtype in (np.float64, np.float32) and a.dtype.isnative and a.flags.writeable \
                and a.flags.aligned and all(st >= 0 and st % a.itemsize == 0 for st in a.strides):
            part.copy_(torch.from_numpy(a))
        else:
            part.numpy()[...] = a
    buf = host.to(dev)
    return [buf[k:k + a.size].view(a.shape) for a, k in zip(arrays, start)]


class Graph:
    """Neighbour graph and network inputs for one particle state (device)."""

    # cells the cell-list graph may use (workspace 2 x 8 B per cell)
    MAX_CELLS = 1 << 24

    def __init__(self, x, v, w, R, cutoff, vs, Rs, max_edges=None, all_pairs=False):
        import torch
        dev = torch.device("cuda")
        n = int(R.shape[0])
        self.n, self.npad = n, pad64(n)
        self.x, self.v, self.w, self.R = _upload((x, v, w, R), dev)
        cnt = torch.empty(n, dtype=torch.int64, device=dev)
        self.off = torch.empty(n + 1, dtype=torch.int64, device=dev)
        ne = ctypes.c_int64(0)
        cap = max_edges or 64 * n
        self.nbr = torch.empty(max(cap, 1), dtype=torch.int32, device=dev)
        self.dst = torch.empty(max(cap, 1), dtype=torch.int32, device=dev)
        if all_pairs:  # O(n^2), kept as the reference of the cell-list graph
            _call("mpnn_graph", n, self.x, float(cutoff), cnt, self.off, self.nbr, self.dst, cap,
                  ctypes.pointer(ne), None)
        else:
            work = torch.empty(2 * (self.MAX_CELLS + 1) + 2 * n + 1, dtype=torch.int64,
                               device=dev)
            box = torch.empty(6, dtype=torch.float32, device=dev)
            _call("mpnn_graph_cells", n, self.x, float(cutoff), self.MAX_CELLS, work, box, cnt,
                  self.off, self.nbr, self.dst, cap, ctypes.pointer(ne), None)
        self.E = int(ne.value)
        self.Epad = pad64(self.E)
        self.perm = torch.empty(max(self.E, 1), dtype=torch.int32, device=dev)
        _call("mpnn_reverse_edges", self.E, self.off, self.nbr, self.dst, self.perm, None)
        self.nf = torch.empty(self.npad * 16, dtype=torch.int16, device=dev)
        self.ef = torch.empty(self.Epad * 16, dtype=torch.int16, device=dev)
        _call("mpnn_features", n, self.npad, self.E, self.Epad, self.dst, self.nbr, self.x,
              self.v, self.w, self.R, float(vs), float(Rs), self.nf, self.ef, None)

    def edges_host(self):
        off = self.off.cpu().numpy()
        return off, self.nbr[:self.E].cpu().numpy(), self.dst[:self.E].cpu().numpy()


class MPNN:
    """The network's parameters (fp32 masters, bf16 copies, Adam moments)."""

    # tries of a wait of the message kernel before it gives up (-1: the library's)
    TRIES = -1

    def __init__(self, seed=0, weights=None):
        import torch
        self.torch = torch
        dev = torch.device("cuda")
        rng = np.random.default_rng(seed)
        self.W, self.Wb, self.Wt, self.m, self.v, self.G = {}, {}, {}, {}, {}, {}
        for name, (kin, nout) in LAYERS.items():
            kp = pad64(kin)
            if weights is not None:
                w = np.zeros((kp, nout), np.float32)
                w[:kin] = weights[name]
            else:
                w = np.zeros((kp, nout), np.float32)
                cols = nout if name != "dec" else OUT
                if kin == 16:   # input layers: 7 features, the constant in column 7
                    w[:7] = rng.normal(scale=math.sqrt(2.0 / 7), size=(7, nout))
                    w[7] = 0.1
                else:           # hidden inputs, then the constant block
                    scale = math.sqrt(2.0 / (kin - 16)) if name != "dec" else 0.1 / math.sqrt(kin)
                    w[:kin - 16, :cols] = rng.normal(scale=scale, size=(kin - 16, cols))
            self.W[name] = torch.as_tensor(w, device=dev)
            self.Wb[name] = torch.empty((kp, nout), dtype=torch.int16, device=dev)
            self.Wt[name] = torch.empty((nout, kin), dtype=torch.int16, device=dev)
            self.m[name] = torch.zeros_like(self.W[name])
            self.v[name] = torch.zeros_like(self.W[name])
            self.G[name] = torch.zeros_like(self.W[name])
            self._refresh(name)
        self.t = 0
        # the last pass: its loss (a float) and, in the high half, its status
        self.report = torch.zeros(1, dtype=torch.int64, device=dev)

    def _refresh(self, name):
        # bf16 copies through a zero-rate Adam step would move the moments;
        # convert directly instead
        kin, nout = LAYERS[name]
        W = self.W[name]
        _call("mpnn_to_bf16", W.numel(), W, self.Wb[name], None)
        Wt32 = W[:kin].t().contiguous()
        _call("mpnn_to_bf16", Wt32.numel(), Wt32, self.Wt[name], None)

    def weights(self) -> dict:
        return {k: self.W[k][:LAYERS[k][0]].cpu().numpy().astype(np.float64) for k in LAYERS}

    # ---- forward -------------------------------------------------------------
    def forward(self, g: Graph, keep=True):
        """The outputs [npad][64] (fp32); keep: also the states and relu masks that
        backward() needs.  Does not wait for the device; should a bounded wait in the
        message kernel run out, all outputs are NaN and check() raises."""
        torch = self.torch
        f32, b16, i32 = torch.float32, torch.int16, torch.int32
        n, npad, E = g.n, g.npad, g.E

        def new(rows, cols, dtype):
            return torch.empty((rows, cols), dtype=dtype, device=torch.device("cuda"))

        self.state = None
        h, hb = new(npad, H, f32), new(npad, H, b16)
        p1, y = new(npad, H, f32), new(npad, 64, f32)
        Mb, eb = new(npad, H, b16), new(g.Epad, H, b16)
        st = dict(hb=[hb], Mb=[], m=[], u=[], eb=eb)
        status = ctypes.c_void_p(self.report.data_ptr() + 4)
        _call("mpnn_encode_edges", E, g.ef, self.Wt["edge"], eb, None)
        _call("mpnn_encode_nodes_checked", n, npad, g.nf, self.Wt["node"], self.Wt["msg0"], h, hb,
              p1, status, None)
        m = u = None
        for r in range(ROUNDS):
            last = r == ROUNDS - 1
            hb_in = hb
            if keep:
                hb, Mb = new(npad, H, b16), new(npad, H, b16)
                m, u = new(g.Epad, H // 32, i32), new(npad, H // 32, i32)
                for key, t in (("hb", hb), ("Mb", Mb), ("m", m), ("u", u)):
                    st[key].append(t)
            _call("mpnn_message_sums_checked", n, E, g.off, g.nbr, g.dst, hb_in, eb,
                  self.Wt[f"msg{r}"], p1, Mb, m, _i32(self.TRIES), status, None)
            _call("mpnn_update_nodes_checked", n, npad, hb_in, Mb, self.Wt[f"upd{r}"],
                  self.Wt["dec" if last else f"msg{r + 1}"], _i32(last), h, hb,
                  y if last else p1, u, status, None)
        if keep:
            self.state = st
        return y

    def check(self):
        """Waits for the last forward pass and raises DemError if it did not run to
        its end; returns the loss, if one was taken."""
        loss, rc = struct.unpack("<fi", struct.pack("<q", self.report.item()))
        if rc != 0:
            raise _dem.DemError(rc, "forward")
        return loss

    # ---- backward ------------------------------------------------------------
    def backward(self, g: Graph, dy):
        torch = self.torch
        f32, b16 = torch.float32, torch.int16
        st = self.state
        n, npad, E = g.n, g.npad, g.E

        def new(rows, cols, dtype):
            return torch.empty((rows, cols), dtype=dtype, device=torch.device("cuda"))

        # a weight's gradient is summed in row ranges of about 4,096 (64 at most)
        splits = {rows: max(1, min(64, rows // 4096)) for rows in (npad, g.Epad)}
        work = new(max(splits[npad], splits[g.Epad]) * pad64(3 * H + 16), H, f32)

        def weights(name, rows, K, segments, X, idx, dZ):
            kin, nout = LAYERS[name]
            X, idx = list(X) + [None] * (3 - len(X)), list(idx) + [None] * (2 - len(idx))
            _call("mpnn_grad_weights", rows, K, _i32(segments), X[0], idx[0], X[1], idx[1], X[2],
                  dZ, _i32(nout), _i32(pad64(kin)), _i32(splits[K]), work, self.G[name], None)

        dyb, zb = new(npad, 64, b16), new(npad, H, b16)
        dh, dMb = new(npad, H, f32), new(npad, H, b16)
        dX, de = new(g.Epad, 2 * H, f32), new(g.Epad, H, f32)
        zm, zeb = new(g.Epad, H, b16), new(g.Epad, H, b16)
        _call("mpnn_to_bf16", npad * 64, dy, dyb, None)
        weights("dec", n, npad, 1, [st["hb"][ROUNDS]], [], dyb)
        _call("mpnn_grad_decode", npad, dyb, self.Wb["dec"], st["u"][-1], dh, zb, None)
        for r in reversed(range(ROUNDS)):
            hb, m = st["hb"][r], st["m"][r]
            weights(f"upd{r}", n, npad, 2, [hb, st["Mb"][r]], [], zb)
            _call("mpnn_grad_update", npad, zb, self.Wb[f"upd{r}"], dh, dMb, None)
            _call("mpnn_grad_messages", E, g.dst, dMb, m, self.Wb[f"msg{r}"], st["eb"],
                  _i32(r == ROUNDS - 1), _i32(r == 0), zm, dX, de, zeb, None)
            weights(f"msg{r}", E, g.Epad, 3, [hb, hb, st["eb"]], [g.dst, g.nbr], zm)
            _call("mpnn_grad_nodes", n, npad, g.off, g.perm, dX, st["u"][r - 1] if r else None,
                  None if r else st["hb"][0], dh, zb, None)
        weights("edge", E, g.Epad, 0, [g.ef], [], zeb)
        weights("node", n, npad, 0, [g.nf], [], zb)

    def loss_and_grad(self, g: Graph, target):
        """MSE over the n x 6 outputs; target fp32 [npad][64] (zeros past 6
        columns and n rows).  Fills G and returns the loss."""
        y = self.forward(g)
        dy = self.torch.empty_like(y)
        _call("mpnn_mse", y.numel(), y, target, 1.0 / (g.n * OUT), dy, self.report, None)
        self.backward(g, dy)
        return self.check() / (g.n * OUT)

    def adam(self, lr=1e-3, b1=0.9, b2=0.999, eps=1e-8):
        self.t += 1
        for name, (kin, nout) in LAYERS.items():
            W = self.W[name]
            _call("mpnn_adam", W.numel(), W, self.m[name], self.v[name], self.G[name], float(lr),
                  float(b1), float(b2), float(eps), self.t, self.Wb[name], self.Wt[name],
                  _i32(W.shape[0]), _i32(nout), _i32(kin), None)


# ---- data from the DEM ---------------------------------------------------------

def targets(v0, w0, v1, w1, R, stride, dt, a_s):
    """Mean accelerations over the stride, scaled: [a, R alpha] / a_s."""
    a = (v1 - v0) / (stride * dt)
    al = (w1 - w0) / (stride * dt) * R[:, None]
    return np.hstack([a, al]) / a_s


def target_buffer(T, npad):
    import torch
    buf = np.zeros((npad, 64), np.float32)
    buf[:T.shape[0], :OUT] = T
    return torch.as_tensor(buf, device=torch.device("cuda"))


SCALES = dict(vs=0.1, Rs=1.0e-3, a_s=10.0)   # velocity, length, acceleration scales


def make_graph(x, v, w, R, rmax):
    return Graph(x, v, w, R, 2.2 * rmax, SCALES["vs"], SCALES["Rs"])


def sample_pairs(scene, n_samples, every=50, stride=10, settle=2000, precision=1):
    """(state at t, state at t + stride) pairs from a GPU DEM run of `scene`
    (dict for dem.Scene.from_dict): settle, then a pair every `every` steps."""
    sc = _dem.Scene.from_dict(scene, precision=precision)
    sc.step(settle)
    R = sc.radii()
    out = []
    for _ in range(n_samples):
        a = sc.state()
        sc.step(stride)
        b = sc.state()
        out.append((a, b))
        sc.step(max(0, every - stride))
    if sc.synchronize() != 0:
        raise RuntimeError("DEM run failed")
    return out, R


def train(model: MPNN, pairs, R, dt, stride=10, iters=300, lr=1e-3, log_every=50, lr_end=None):
    """Adam on the mean-squared error of the scaled mean accelerations,
    cycling through the sample pairs (learning rate decaying geometrically to
    lr_end if given); returns the loss history."""
    rmax = float(R.max())
    graphs = []
    for a, b in pairs:
        g = make_graph(a["x"], a["v"], a["w"], R, rmax)
        T = targets(a["v"], a["w"], b["v"], b["w"], R, stride, dt, SCALES["a_s"])
        graphs.append((g, target_buffer(T, g.npad)))
    hist = []
    for it in range(iters):
        g, T = graphs[it % len(graphs)]
        loss = model.loss_and_grad(g, T)
        rate = lr if lr_end is None else lr * (lr_end / lr) ** (it / max(1, iters - 1))
        model.adam(rate)
        if it % log_every == 0 or it == iters - 1:
            hist.append((it, loss))
    return hist


def predict(model: MPNN, state, R):
    g = make_graph(state["x"], state["v"], state["w"], R, float(R.max()))
    y = model.forward(g, keep=False)[:g.n, :OUT].cpu().numpy()
    if np.isnan(y[:1]).any():  # (all are, if the pass did not run to its end)
        model.check()
    return y.astype(np.float64) * SCALES["a_s"]


def evaluate(model: MPNN, pairs, R, dt, g_vec, stride=10):
    """Mean squared error (scaled units) of the network and of the
    gravity-only guess (a = g, alpha = 0) on held-out pairs."""
    e_net, e_base = [], []
    for a, b in pairs:
        T = targets(a["v"], a["w"], b["v"], b["w"], R, stride, dt, 1.0)
        P = predict(model, a, R)
        base = np.zeros_like(T)
        base[:, :3] = g_vec
        e_net.append(np.mean(((P - T) / SCALES["a_s"]) ** 2))
        e_base.append(np.mean(((base - T) / SCALES["a_s"]) ** 2))
    return float(np.mean(e_net)), float(np.mean(e_base))


def advance(state, acc, R, dt, stride):
    """Semi-implicit Euler over `stride` steps with constant predicted
    accelerations (a, R alpha): v_k = v + k a dt, x += sum_k v_k dt."""
    a, al = acc[:, :3], acc[:, 3:] / R[:, None]
    k = stride
    v1 = state["v"] + k * dt * a
    x1 = state["x"] + k * dt * state["v"] + dt * dt * a * (k * (k + 1) / 2.0)
    w1 = state["w"] + k * dt * al
    return dict(x=x1, v=v1, w=w1, q=state["q"])


def max_overlap(x, R, rmax):
    """Largest overlap / radius among neighbours (from the surrogate's graph)."""
    g = make_graph(x, np.zeros_like(x), np.zeros_like(x), R, rmax)
    off, nbr, dst = g.edges_host()
    if len(nbr) == 0:
        return 0.0
    d = np.linalg.norm(x[nbr] - x[dst], axis=1)
    return float(np.max((R[nbr] + R[dst] - d) / np.minimum(R[nbr], R[dst])))


def rollout(model: MPNN, state, R, params, strides, stride=10, overlap_growth=0.02,
            energy_limit=0.5, precision=1):
    """Hybrid run: each stride, the network's accelerations advance the state
    unless the largest overlap grows by more than overlap_growth R_min or the
    kinetic energy changes by more than energy_limit (relative); then the DEM
    takes that stride from the state before it.  Also runs the DEM alone
    alongside and returns the per-stride position error of the hybrid
    (RMS / R_max)."""
    import time
    dt = params["dt"]
    rmax = float(R.max())
    rho = params["rho"]
    m = 4.0 / 3.0 * math.pi * rho * R ** 3

    def ke(s):
        return 0.5 * float(np.sum(m * np.einsum("ij,ij->i", s["v"], s["v"])))

    def dem_stride(s):
        sc = _dem.Scene(params, R, s["x"], s["v"], s["w"], s["q"], precision=precision,
                        **_mesh_kw)
        sc.step(stride)
        out = sc.state()
        sc.close()
        return out

    ref = dict(state)
    cur = dict(state)
    rows = []
    t_net = t_dem = 0.0
    falls = 0
    for k in range(strides):
        t0 = time.perf_counter()
        acc = predict(model, cur, R)
        nxt = advance(cur, acc, R, dt, stride)
        ov0 = max_overlap(cur["x"], R, rmax)
        ov = max_overlap(nxt["x"], R, rmax)
        e0, e1 = ke(cur), ke(nxt)
        t_net += time.perf_counter() - t0
        if ov > ov0 + overlap_growth or abs(e1 - e0) > energy_limit * max(e0, 1e-30):
            t0 = time.perf_counter()
            nxt = dem_stride(cur)
            t_dem += time.perf_counter() - t0
            falls += 1
        cur = nxt
        ref = dem_stride(ref)
        err = float(np.sqrt(np.mean(np.sum((cur["x"] - ref["x"]) ** 2, axis=1)))) / rmax
        rows.append((k + 1, err, ov))
    return {"strides": strides, "fallbacks": falls, "pos_error_rms_over_rmax": rows,
            "net_s": t_net, "dem_fallback_s": t_dem}


_mesh_kw = {}


def experiment(n_scenes=16, n_train=80, n_eval=16, iters=3000, lr=1e-3, drum_n=100_000,
               strides=10, seed=0):
    """Train on hopper-discharge trajectories (the batched workload), evaluate
    on held-out pairs against the gravity-only guess, then run the network on
    a rotating drum with DEM fallback.  Returns a dict of the results."""
    import time
    from . import batch, scenes
    rng = np.random.default_rng(seed)
    ns = [int(n) for n in np.exp(rng.uniform(math.log(800), math.log(3000), n_scenes))]
    mus = [(float(rng.uniform(0.2, 0.8)), float(rng.uniform(0, 0.2)),
            float(rng.uniform(0, 0.2))) for _ in ns]
    b = batch.combine([batch.hopper_scene(n, 700 + k, mus[k]) for k, n in enumerate(ns)])
    dt = b["params"]["dt"]
    t0 = time.perf_counter()
    pairs, R = sample_pairs(b, n_train + n_eval, every=100, settle=3000)
    t_data = time.perf_counter() - t0
    model = MPNN(seed=seed)
    t0 = time.perf_counter()
    hist = train(model, pairs[:n_train], R, dt, iters=iters, lr=lr, lr_end=lr / 10,
                 log_every=max(1, iters // 12))
    t_train = time.perf_counter() - t0
    gv = np.asarray(b["params"]["g"])
    e_net, e_base = evaluate(model, pairs[n_train:], R, dt, gv)
    t_net_mse, t_base_mse = evaluate(model, pairs[:n_train], R, dt, gv)
    # the network on a drum (another geometry), with DEM fallback
    d = scenes.drum_scene(n=drum_n, seed=5, n_theta=64, n_rings=8, nn_dist=2.15e-3, speed=0.02)
    sc = _dem.Scene.from_dict(d, precision=1)
    sc.step(1500)
    st = sc.state()
    # DEM time for one stride of the drum, graph replay (device)
    sc.synchronize()
    t0 = time.perf_counter()
    sc.step(100)
    sc.synchronize()
    dem_stride_ms = (time.perf_counter() - t0) * 1e3 / 10
    sc.close()
    _mesh_kw.clear()
    _mesh_kw.update(verts=d["verts"], tris=d["tris"], tri_radius=d["tri_radius"],
                    max_mesh_contacts=d["max_mesh_contacts"])
    roll = rollout(model, st, d["R"], d["params"], strides)
    # network time for one stride of the drum: graph + forward
    import torch
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for _ in range(5):
        predict(model, st, d["R"])
    torch.cuda.synchronize()
    net_stride_ms = (time.perf_counter() - t0) * 1e3 / 5
    return {"train_particles": int(len(R)), "train_pairs": n_train, "eval_pairs": n_eval,
            "iters": iters, "loss_history": hist, "eval_mse_net": e_net,
            "eval_mse_gravity_only": e_base, "train_mse_net": t_net_mse,
            "train_mse_gravity_only": t_base_mse, "data_s": t_data, "train_s": t_train,
            "drum_particles": drum_n, "rollout": roll,
            "net_ms_per_stride": net_stride_ms, "dem_ms_per_stride": dem_stride_ms}


def main():
    import json
    import argparse
    ap = argparse.ArgumentParser(description="train and run the surrogate")
    ap.add_argument("--iters", type=int, default=3000)
    ap.add_argument("--drum-n", type=int, default=100_000)
    ap.add_argument("--strides", type=int, default=10)
    a = ap.parse_args()
    print(json.dumps(experiment(iters=a.iters, drum_n=a.drum_n, strides=a.strides)))


if __name__ == "__main__":
    main()

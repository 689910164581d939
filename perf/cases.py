"""What a user of the tracer-box library has it do, as timed cases.

Six kinds of work, each through the public binding:

  replay    tracer boxes stepped from their initial condition on: boundary
            samples pushed, steps run (a captured graph or plain calls), the
            density and velocity fields read out, the chain trajectory left in
            its ring.  Storage formats, time interpolations, zoomed and
            co-moving boxes, one box or a batch of uneven ones.
  upsample  replay of boxes whose boundary comes from the learned upsampler.
  thermal   replay of a box with the fluctuating collision.
  train     one training step of the upsampler (forward, backward, Adam).
  evaluate  features, targets and prediction of the upsampler on face sets.
  observe   the observables of a box between steps: conservation sums, mean
            vorticity of the sub-volume and its centre, the fields.

Sizes: the configurations of the benchmark (32^3, 128^3, 256^3, 512 uneven
boxes, 64^3 upsampler boxes, batches of 16384 rows) and what lies between.

The boundary record of a box holds RECORD samples; the replay runs through it
forwards and backwards, so that a long run meets no jump.  Fields of the
16-bit formats are handed on in that format, and chain trajectories and mean
vorticities of runs in FP32 arithmetic in FP32: what the run itself carries.

exact() repeats a first pass in FP64 with plain torch operations.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_0809_4958_gb300 import inputs, lbtracer as lbt

RECORD = 24  # boundary samples a replay keeps in device memory
U_MAX = 0.05  # velocity scale of the coarse flow (lattice units)
STORE = {"f64": lbt.LB_STORE_F64, "f32": lbt.LB_STORE_F32, "f16": lbt.LB_STORE_F16DEV, "bf16": lbt.LB_STORE_BF16DEV}
BYTES = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2}
INTERP = {"linear": lbt.LB_TIME_LINEAR, "hermite": lbt.LB_TIME_HERMITE, "mlp": lbt.LB_TIME_MLP}
BATCH_EDGES = (24, 32, 48, 64)


def _replay(name, storage="f32", E=128, boxes=1, beads=0, kT=0.0, interp="linear", K=1, zoom=1, frame=False, tau=0.8,
            steps=16, graph=True):
    """boxes = 1: one box of E^3; more: uneven boxes with edges up to E, each
    with a chain of `beads` at most when beads > 0."""
    return dict(name=name, kind="replay", storage=storage, E=E, boxes=boxes, beads=beads, kT=kT, interp=interp, K=K,
                zoom=zoom, frame=frame, tau=tau, steps=steps, graph=graph)


def listed():
    return [
        # the smallest call: one step of the 32^3 validation box in FP64, its 16-bead chain, fields out
        _replay("box32_f64", storage="f64", E=32, beads=16, steps=1, graph=False),
        # production run of one tracer: 128^3 FP32, 64-bead chain with thermal noise, graphs of 8 steps
        _replay("box128_f32", E=128, beads=64, kT=1e-4, steps=8),
        # the same box in FP64, for reference runs: plain steps
        _replay("box128_f64", storage="f64", E=128, beads=64, kT=1e-4, steps=4, graph=False),
        # the paper's replay: a zoomed box in the tracer's co-moving frame, one coarse sample every 113 steps
        _replay("paper128_f32", E=128, beads=64, kT=1e-4, K=113, zoom=6, frame=True, tau=1.0, steps=8),
        # an ensemble: 512 uneven boxes, each with its own flow and chain, graphs of 4 steps
        _replay("batch512_f32", E=64, boxes=512, beads=128, kT=1e-4, steps=4),
        # a large box in half precision, stepped plainly
        _replay("box256_f16", storage="f16", E=256, steps=4, graph=False),
        # a box of middling, uneven size in bfloat16, coarse samples every four steps, Hermite in time
        _replay("box144_bf16", storage="bf16", E=144, interp="hermite", K=4, steps=8, graph=False),
        # boxes fed through the learned upsampler: one coarse interval of 16 steps
        dict(name="upsample128x64_f32", kind="upsample", E=64, boxes=128, K=16, tau=0.8),
        # one training step on the benchmark's batch
        dict(name="train16384", kind="train", K=16, rows=16384),
        # a held-out interval of twelve boxes: features, targets, prediction
        dict(name="evaluate12x64", kind="evaluate", E=64, boxes=12, K=16),
        # a thermal fluid without a chain, graphs of 16 steps
        dict(name="thermal96_f32", kind="thermal", storage="f32", E=96, kT=1e-4, tau=0.8, steps=16, periodic=True),
        # what is looked at between the steps of a run
        dict(name="observe128_f32", kind="observe", storage="f32", E=128),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _edge(rng, lo, hi):
    return 8 * _log_int(rng, lo // 8, hi // 8)


def draw(rng):
    kind = rng.choice(["box", "box", "box64", "paper", "batch", "wide", "wide", "upsample", "train", "train", "evaluate",
                       "thermal", "observe"])
    if kind == "box":
        E = _edge(rng, 16, 160)
        plain = rng.random() < 0.4
        return _unnamed(_replay("", E=E, beads=rng.randint(0, min(96, E - 8)), kT=rng.choice([0.0, 1e-4, 1e-3]),
                                K=rng.choice([1, 1, 3]), interp=rng.choice(["linear", "linear", "hermite"]),
                                tau=rng.choice([0.7, 0.8, 1.0]), steps=rng.randint(1, 6) if plain else rng.choice([4, 8]),
                                graph=not plain))
    if kind == "box64":
        E = _edge(rng, 16, 128)
        return _unnamed(_replay("", storage="f64", E=E, beads=rng.randint(0, min(64, E - 8)), kT=rng.choice([0.0, 1e-4]),
                                tau=rng.choice([0.7, 0.8]), steps=rng.randint(1, 4), graph=False))
    if kind == "paper":
        E = _edge(rng, 48, 128)
        return _unnamed(_replay("", E=E, beads=rng.randint(8, min(64, E - 8)), kT=1e-4, K=rng.randint(20, 120),
                                zoom=rng.randint(2, 8), frame=rng.random() < 0.7, tau=1.0, steps=rng.choice([4, 8])))
    if kind == "batch":
        return _unnamed(_replay("", E=rng.choice([32, 48, 64]), boxes=_log_int(rng, 8, 400),
                                beads=rng.choice([0, 32, 64, 128]), kT=1e-4, steps=rng.choice([2, 4])))
    if kind == "wide":
        return _unnamed(_replay("", storage=rng.choice(["f16", "f16", "bf16", "f32"]), E=_edge(rng, 48, 256),
                                interp=rng.choice(["linear", "hermite"]), K=rng.randint(1, 8), steps=rng.randint(1, 6),
                                graph=False))
    if kind == "upsample":
        return dict(kind="upsample", E=rng.choice([24, 32, 40, 64]), boxes=_log_int(rng, 1, 100), K=rng.choice([8, 16]),
                    tau=0.8)
    if kind == "train":
        return dict(kind="train", K=rng.choice([8, 16]), rows=_log_int(rng, 300, 200000))
    if kind == "evaluate":
        return dict(kind="evaluate", E=_edge(rng, 16, 96), boxes=_log_int(rng, 1, 24), K=rng.choice([8, 16]))
    if kind == "thermal":
        return dict(kind="thermal", storage=rng.choice(["f32", "f32", "f16"]), E=_edge(rng, 24, 128), kT=1e-4,
                    tau=rng.choice([0.7, 0.8, 1.0]), steps=rng.choice([4, 8, 16]), periodic=rng.random() < 0.5)
    return dict(kind="observe", storage=rng.choice(["f32", "f32", "f64", "f16"]), E=_edge(rng, 32, 160))


def _unnamed(case):
    del case["name"]
    return case


# ---- inputs ------------------------------------------------------------------
class _Flow:
    """Random-phase flow u(x, t) = sum_m amp_m cos(kvec_m . (x - xc) + omega_m t + phi_m)
    with a Kolmogorov spectrum, divergence free, root-mean-square 0.4 U_MAX."""

    M = 48

    def __init__(self, rng, E, k_max):
        M = self.M
        k = np.exp(np.linspace(0.0, math.log(k_max), M))
        khat = rng.normal(size=(M, 3))
        khat /= np.linalg.norm(khat, axis=1, keepdims=True)
        e = np.cross(khat, rng.normal(size=(M, 3)))
        e /= np.linalg.norm(e, axis=1, keepdims=True)
        A = k ** (-5.0 / 6.0) * np.exp(-0.5 * (k / 16.0) ** 2) * np.sqrt(k)
        A *= 0.4 * U_MAX / math.sqrt(0.5 * float((A * A).sum()))
        self.E = E
        self.kvec = (2.0 * np.pi * k / E)[:, None] * khat
        self.amp = A[:, None] * e
        self.omega = U_MAX * (2.0 * np.pi / E) * k ** (2.0 / 3.0)
        self.phi = rng.uniform(0.0, 2.0 * np.pi, M)

    def _dev(self, a):
        return torch.from_numpy(np.ascontiguousarray(a)).cuda()

    def faces(self, zoom, times, real):
        """[J][6][3][Ec][Ec] samples at the given times."""
        E, Ec = self.E, _coarse(self.E, zoom)
        g = torch.arange(Ec, device="cuda", dtype=torch.float64) * zoom
        q, p = torch.meshgrid(g, g, indexing="ij")
        pts = []
        for f in range(6):
            n = torch.full_like(p, float(E - 1) if f & 1 else 0.0)
            pts.append(torch.stack([(n, p, q), (p, n, q), (p, q, n)][f // 2], dim=-1).reshape(-1, 3))
        ph = (torch.cat(pts) - 0.5 * (E - 1)) @ self._dev(self.kvec).T + self._dev(self.phi)
        wt = self._dev(np.asarray(times, np.float64)[:, None] * self.omega[None, :])
        amp = self._dev(self.amp).T
        a = (amp[None] * wt.cos()[:, None, :]).reshape(-1, self.M).to(real)
        b = (amp[None] * wt.sin()[:, None, :]).reshape(-1, self.M).to(real)
        u = a @ ph.cos().to(real).T - b @ ph.sin().to(real).T  # [J 3][6 Ec^2]
        return u.view(len(times), 3, 6, Ec, Ec).transpose(1, 2).contiguous()

    def volume(self, zoom, real):
        """[3][Ec][Ec][Ec] at t = 0."""
        E, Ec = self.E, _coarse(self.E, zoom)
        cx = torch.complex128 if real == torch.float64 else torch.complex64
        g = torch.arange(Ec, device="cuda", dtype=torch.float64) * zoom - 0.5 * (E - 1)
        ex = [torch.polar(torch.ones((), dtype=torch.float64, device="cuda"), self._dev(self.kvec[:, a])[:, None] * g).to(cx)
              for a in range(3)]
        ph = torch.polar(self._dev(self.amp).abs(), self._dev(np.where(self.amp < 0, np.pi, 0.0) + self.phi[:, None])).to(cx)
        zy = (ex[2][:, :, None] * ex[1][:, None, :]).view(self.M, -1)
        return torch.stack([((zy * ph[:, c:c + 1]).T @ ex[0]).real.reshape(Ec, Ec, Ec) for c in range(3)]).contiguous()

    def tracer(self, times):
        """Velocity of the box centre and the frame acceleration -dv/dt."""
        a = np.asarray(times, np.float64)[:, None] * self.omega + self.phi
        return np.cos(a) @ self.amp, (self.omega * np.sin(a)) @ self.amp


def _coarse(E, zoom):
    return (E - 1 + zoom - 1) // zoom + 1 if zoom > 1 else E


def _tri(j):
    """Record index of sample j: forwards and backwards through the record."""
    k = j % (2 * RECORD - 2)
    return k if k < RECORD else 2 * RECORD - 2 - k


def _gammas(tau):
    """Relaxation factors of the fluctuating collision: shear by tau, the bulk and the higher modes faster."""
    g = np.zeros(19)
    g[4] = 0.2
    g[5:10] = 1.0 - 1.0 / tau
    return g


def _boxes(case, seed):
    """Edges and chain lengths of a replay, from the case; flows and chain starts, from the seed."""
    n = case.get("boxes", 1)
    E = case["E"]
    rng = np.random.default_rng([n, E, case.get("beads", 0)])
    if n == 1 or case["kind"] != "replay":
        edges = [E] * n
    else:
        edges = [int(e) for e in rng.choice([e for e in BATCH_EDGES if e <= E], n)]
    beads = [0] * n
    if case.get("beads"):
        if n == 1:
            beads = [case["beads"]]
        else:
            beads = [int(rng.integers(32, max(33, min(case["beads"], 3 * e // 2) + 1))) for e in edges]
    rng = np.random.default_rng([int(seed), 11])
    flows = [_Flow(rng, e, 10.0 if case.get("frame") else min(e / 2.0, 64.0)) for e in edges]
    starts = [inputs.chain_start(int(seed) * 1000 + b, nb, e) if nb else None for b, (e, nb) in enumerate(zip(edges, beads))]
    return edges, beads, flows, starts


def _record(case, flows, real):
    """[RECORD][all boxes' faces back to back], and the frame samples of one co-moving box."""
    times = np.arange(RECORD) * case["K"]
    zoom = case.get("zoom", 1)
    parts = [f.faces(zoom, times, real) for f in flows]
    acc = None
    if case.get("frame"):
        v, acc = flows[0].tracer(times)
        parts[0] -= torch.from_numpy(v).to(parts[0])[:, None, :, None, None]
    return torch.cat([p.view(RECORD, -1) for p in parts], dim=1), acc


def _start_field(case, flow, real):
    u0 = flow.volume(case.get("zoom", 1), real)
    if case.get("frame"):
        u0 -= torch.from_numpy(flow.tracer([0.0])[0][0]).to(u0)[:, None, None, None]
    return u0


def _train_rows(case, seed):
    """Features and targets with the shape of the face data: four samples along a smooth track, in-face
    differences, and a residual that vanishes at the samples."""
    K, rows = case["K"], case["rows"]
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    n = lambda *s: torch.randn(*s, device="cuda", generator=g)  # noqa: E731
    base, slope, curv = 0.4 * n(rows, 1, 3), 0.1 * n(rows, 1, 3), 0.03 * n(rows, 1, 3)
    a = torch.tensor([-1.0, 0.0, 1.0, 2.0], device="cuda").view(1, 4, 1)
    smp = base + slope * a + curv * a * a
    grad = 0.1 * n(rows, 1, 6) + 0.02 * n(rows, 2, 6)
    X = torch.zeros((rows, 32), device="cuda")
    X[:, :24] = torch.cat([smp.reshape(rows, 12), grad.reshape(rows, 12)], dim=1)
    th = torch.arange(1, K + 1, device="cuda").view(1, K, 1) / K
    T = (th * (1 - th)) ** 2 * 16.0 * (0.4 * n(rows, 1, 3) + 4.0 * curv * slope + torch.sin(3.0 * base) * 0.3)
    return X.to(torch.bfloat16), T.reshape(rows, 3 * K).contiguous()


# ---- the cases -----------------------------------------------------------------
class _State:
    """What a replaying program keeps: the context, the sample record, the read-out buffers."""


def prepare(case, seed):
    lbt.load()
    return {"replay": _prepare_replay, "upsample": _prepare_replay, "thermal": _prepare_replay, "train": _prepare_train,
            "evaluate": _prepare_evaluate, "observe": _prepare_replay}[case["kind"]](case, seed)


def _full(case):
    """The replay that a case of another kind steps."""
    if case["kind"] == "upsample":
        return dict(case, storage="f32", interp="mlp", steps=case["K"], graph=True)
    if case["kind"] == "thermal":
        return dict(case, interp="linear", K=1, graph=True)
    if case["kind"] == "observe":
        return dict(case, interp="linear", K=1, steps=2, graph=False, tau=0.8)
    return case


def _prepare_replay(case, seed):
    case = _full(case)
    edges, beads, flows, starts = _boxes(case, seed)
    G, K = case["steps"], case["K"]
    st = _State()
    st.case, st.edges = case, edges
    periodic = (True,) * 3 if case.get("periodic") else (False,) * 3
    descs = [lbt.box_desc(e, case["tau"], periodic=periodic, time_interp=INTERP[case["interp"]], K=K, nbeads=nb,
                          zoom=case.get("zoom", 1), frame_accel=case.get("frame", False)) for e, nb in zip(edges, beads)]
    st.tr = tr = lbt.Tracers(descs, STORE[case["storage"]], ring_slots=(G + K - 1) // K + 4 if case["graph"] else 0)
    st.faces, st.acc = (None, None) if all(periodic) else _record(case, flows, tr.real)
    for b, f in enumerate(flows):
        tr.lb_init(b, _start_field(case, f, tr.real))
        if beads[b]:
            tr.chain_couple(b, lbt.chain_desc(beads[b], kT=case["kT"], seed=int(seed) * 1000 + b), starts[b])
    if case["kind"] == "thermal":
        tr.lb_set_fluctuation(0, case["kT"], int(seed), _gammas(case["tau"]))
    if case["interp"] == "mlp":
        st.up = lbt.Upsampler(K=K, batch_rows=1024, master=inputs.mlp_init(seed, K))
        tr.lb_mlp_bind(st.up.export(), U_MAX)
    sites = sum(e ** 3 for e in edges)
    # of an ensemble only the velocities are read
    st.rho = torch.empty(sites, dtype=tr.real, device="cuda") if len(edges) == 1 else None
    st.u = torch.empty(3 * sites, dtype=tr.real, device="cuda")
    st.hist = None
    if sum(beads):
        st.hist = torch.zeros((G, sum(beads), 3), dtype=torch.float64, device="cuda")
        tr.lb_set_chain_history(st.hist, G)
    st.pushed, st.n = -1, 0
    tr.lb_sync()
    if case["kind"] == "observe":
        _steps(st, 2)
    elif case["graph"]:
        tr.lb_graph_capture(G)
    tr.lb_sync()
    return st


def _push(st, n):
    """Samples needed by the steps up to the one that starts at step n."""
    if st.faces is None:
        return
    case = st.case
    j = n // case["K"] + (1 if case["interp"] == "linear" else 2)
    while st.pushed < j:
        st.pushed += 1
        k = _tri(st.pushed)
        st.tr.lb_set_boundary(lbt.LB_ALL_BOXES, st.pushed, st.faces[k])
        if st.acc is not None:
            st.tr.lb_set_frame_accel(0, st.pushed, st.acc[k])


def _steps(st, count):
    for _ in range(count):
        _push(st, st.n)
        st.tr.lb_step(1)
        st.n += 1


def _fields(st):
    o = 0
    for b, e in enumerate(st.edges):
        n3 = e ** 3
        if st.rho is not None:
            st.tr.lb_read_fields(b, lbt.LB_FIELD_RHO | lbt.LB_FIELD_ASYNC, st.rho[o:o + n3])
        st.tr.lb_read_fields(b, lbt.LB_FIELD_U | lbt.LB_FIELD_ASYNC, st.u[3 * o:3 * (o + n3)])
        o += n3


_KEPT = {"f64": torch.float64, "f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}


def run(state):
    if isinstance(state, _State):
        return _run_replay(state)
    return state()


def _run_replay(st):
    case, tr = st.case, st.tr
    with torch.cuda.stream(tr.stream):  # what follows on torch's side runs behind the steps
        if case["kind"] == "observe":
            E = case["E"]
            c = (E - 1) / 2.0
            half = 1.25 / 12.0 * E
            sums = tr.lb_conservation(0)
            vort = [tr.lb_vorticity(0, 1, E - 2), tr.lb_vorticity(0, math.ceil(c - half), math.floor(c + half))]
            _fields(st)
            return {"sums": sums, "vorticity": np.array(vort, tr.np_real), "rho": st.rho, "u": st.u.to(_KEPT[case["storage"]])}
        G = case["steps"]
        if case["graph"]:
            _push(st, st.n + G - 1)
            tr.lb_graph_launch()
            st.n += G
        else:
            _steps(st, G)
        _fields(st)
        out = {"u": st.u.to(_KEPT[case["storage"]])}
        if st.rho is not None:
            out["rho"] = st.rho
        if st.hist is not None:
            out["beads"] = st.hist.to(tr.real)
        return out


def _prepare_train(case, seed):
    K, rows = case["K"], case["rows"]
    X, T = _train_rows(case, seed)
    up = lbt.Upsampler(K=K, batch_rows=rows, master=inputs.mlp_init(seed, K))
    at = _param_sections(K)

    def one():
        loss = up.step(X, T, 2e-3)
        p = up.export()
        out = {k: p[o:o + n].view(d) for k, (o, n, d) in at.items()}
        out["loss"] = loss.float()
        return out
    return one


def _param_sections(K):
    """Offset, bytes and type of the sections of the inference parameters (each aligned to 256 bytes)."""
    at, o = {}, 0
    for name, count, dtype in (("w1", 128 * 32, torch.bfloat16), ("w2", 128 * 128, torch.bfloat16),
                               ("w3", 3 * K * 128, torch.bfloat16), ("b1", 128, torch.float32), ("b2", 128, torch.float32),
                               ("b3", 3 * K, torch.float32)):
        n = count * (2 if dtype == torch.bfloat16 else 4)
        at[name] = (o, n, dtype)
        o = (o + n + 255) // 256 * 256
    return at


def _evaluate_data(case, seed):
    """Per box: the boundary at every step from sample j - 1 to sample j + 2 of an interval, [3 K + 1][6][3][E][E]."""
    rng = np.random.default_rng([int(seed), 12])
    K, E = case["K"], case["E"]
    return [_Flow(rng, E, E / 2.0).faces(1, np.arange(3 * K + 1), torch.float32) for _ in range(case["boxes"])]


def _prepare_evaluate(case, seed):
    K, E, n = case["K"], case["E"], case["boxes"]
    fine = _evaluate_data(case, seed)
    params = lbt.Upsampler(K=K, batch_rows=1024, master=inputs.mlp_init(seed, K)).export()
    R = 6 * E * E
    X = torch.empty((n * R, 32), dtype=torch.bfloat16, device="cuda")
    T = torch.empty((n * R, 3 * K), dtype=torch.float32, device="cuda")

    def one():
        for b, f in enumerate(fine):
            smp = (f[0], f[K], f[2 * K], f[3 * K])
            lbt.mlp_features(*smp, E, U_MAX, out=X[b * R:(b + 1) * R])
            lbt.mlp_targets(*smp, f[K:2 * K + 1], E, K, 0, U_MAX, out=T[b * R:(b + 1) * R])
        return {"x": X, "t": T, "y": lbt.mlp_forward(params, K, X)}
    return one


# ---- what a pass cannot do without ---------------------------------------------
def work(case):
    kind = case["kind"]
    if kind == "train":
        K, R = case["K"], case["rows"]
        P = 32 * 128 + 128 + 128 * 128 + 128 + 128 * 3 * K + 3 * K
        macs = 32 * 128 + 128 * 128 + 128 * 3 * K
        return {"bytes": R * (64 + 12 * K) + P * (4 * 6 + 2 * 2), "flops": 2.0 * R * (3 * macs - 32 * 128)}
    if kind == "evaluate":
        K, R = case["K"], case["boxes"] * 6 * case["E"] ** 2
        return {"bytes": R * (4 * 12 + 12 * K + 64 + 12 * K + 12 * K),
                "flops": 2.0 * R * (32 * 128 + 128 * 128 + 128 * 3 * K)}
    c = _full(case)
    if kind == "replay" and c["boxes"] > 1:  # the mean over the edges
        es = [e for e in BATCH_EDGES if e <= c["E"]]
        edges = [(e, c["boxes"] / len(es)) for e in es]
    else:
        edges = [(c["E"], c.get("boxes", 1))]
    s, r = BYTES[c["storage"]], 8 if c["storage"] == "f64" else 4
    by = fl = 0.0
    for E, n in edges:
        sites = E ** 3
        inner = sites if c.get("periodic") else (E - 2) ** 3
        step = inner * 2 * 19 * s + (sites - inner) * (19 * s + 3 * r * (2 if c["interp"] == "linear" else 4))
        steps = 1 if kind == "observe" else c["steps"]  # observe: the state read once
        if kind == "upsample":  # the residuals of the interval
            fl += n * 6 * E * E * 2.0 * (32 * 128 + 128 * 128 + 128 * 3 * c["K"])
            by += n * 6 * E * E * 2 * 12 * c["K"]
        by += n * ((sites * 19 * s if kind == "observe" else steps * step) + sites * (4 if c.get("boxes", 1) == 1 else 3) * r)
        fl += n * steps * inner * (900.0 if kind == "thermal" else 250.0)
        if c.get("beads"):
            fl += n * steps * 50 * min(c["beads"], E) * 300.0
    return {"bytes": by, "flops": fl}


# ---- the first pass in FP64 --------------------------------------------------------
_C = np.array([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
               (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1),
               (0, -1, 1)])
_W = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)


def _philox(x0, x1, x2, x3, seed):
    """Philox4x32-10 on int64 tensors holding 32-bit words."""
    m = 0xFFFFFFFF
    k0, k1 = seed & m, (seed >> 32) & m
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & m, (k1 + 0xBB67AE85) & m
        p0, p1 = x0 * 0xD2511F53, x2 * 0xCD9E8D57
        x0, x1, x2, x3 = ((p1 >> 32) & m) ^ x1 ^ k0, p1 & m, ((p0 >> 32) & m) ^ x3 ^ k1, p0 & m
    return x0, x1, x2, x3


def _unit(v, storage):
    """Unit-variance uniform of a word: all 32 bits in FP64, the top 24 otherwise."""
    u = v.double() * 2.0 ** -32 if storage == "f64" else (v >> 8).double() * 2.0 ** -24
    return math.sqrt(3.0) * (2.0 * u - 1.0)


def _dev64(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()


def _moments(g):
    """Density deviation and momentum of populations [19][n, z, y, x]."""
    r = sum(g)
    return r, [sum(float(_C[i, a]) * g[i] for i in range(19) if _C[i, a]) for a in range(3)]


def _equilibrium(i, drho, u, usq):
    cu = sum(float(_C[i, a]) * u[a] for a in range(3) if _C[i, a]) if i else 0.0
    return float(_W[i]) * (drho + (1.0 + drho) * (3.0 * cu + 4.5 * cu * cu - usq)), cu


def _modes19():
    """The orthogonal D3Q19 polynomials [19 modes][19 velocities]."""
    x, y, z = (_C[:, a].astype(np.float64) for a in range(3))
    c2 = x * x + y * y + z * z
    return np.array([np.ones(19), x, y, z, c2 - 1, 3 * x * x - c2, y * y - z * z, x * y, y * z, z * x, (3 * c2 - 5) * x,
                     (3 * c2 - 5) * y, (3 * c2 - 5) * z, (y * y - z * z) * x, (z * z - x * x) * y, (x * x - y * y) * z,
                     3 * c2 * c2 - 6 * c2 + 1, (2 * c2 - 3) * (3 * x * x - c2), (2 * c2 - 3) * (y * y - z * z)])


class _Reference:
    """The boxes of one edge length, stepped together in FP64."""

    def __init__(self, case, seed, E, ids, beads, starts, u0, record, acc, residual):
        self.case, self.seed, self.E, self.ids = case, int(seed), E, ids
        self.om, self.acc, self.residual = 1.0 / case["tau"], acc, residual
        z = case.get("zoom", 1)
        self.per = bool(case.get("periodic"))
        if z > 1:  # linear interpolation from the coarse points
            P = torch.zeros((E, _coarse(E, z)), dtype=torch.float64, device="cuda")
            for s in range(E):
                P[s, s // z] += 1.0 - (s % z) / z
                P[s, min(s // z + 1, P.shape[1] - 1)] += (s % z) / z
            u0 = torch.einsum("zc,ye,xf,ncef->nzyx", P, P, P, u0.view(-1, *u0.shape[2:])).view(*u0.shape[:2], E, E, E)
            record = torch.einsum("qc,pd,ncd->nqp", P, P, record.reshape(-1, *record.shape[-2:])).view(*record.shape[:-2], E, E)
        self.record = record  # [boxes][J][6][3][q][p]
        u = [u0[:, a] for a in range(3)]
        usq = 1.5 * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2)
        self.d = [_equilibrium(i, torch.zeros_like(usq), u, usq)[0] for i in range(19)]
        self.mask = None
        if not self.per:
            self.mask = torch.ones((E, E, E), dtype=torch.bool, device="cuda")
            self.mask[1:-1, 1:-1, 1:-1] = False
        self.N = max(beads) if beads else 0
        if self.N:
            self.nb = torch.tensor(beads, device="cuda")
            self.own = torch.arange(self.N, device="cuda")[None, :] < self.nb[:, None]
            self.pos = torch.zeros((len(ids), self.N, 3), dtype=torch.float64, device="cuda")
            for k, p in enumerate(starts):
                self.pos[k, :len(p)] = _dev64(p)
            self.vel = torch.zeros_like(self.pos)

    def accel(self, n):
        if self.acc is None:
            return [0.0, 0.0, 0.0]
        K = self.case["K"]
        j, th = n // K, (n % K) / K
        return [float(v) for v in (1.0 - th) * self.acc[_tri(j)] + th * self.acc[_tri(j + 1)]]

    def boundary(self, n):
        """Velocity of the outer layer at t = n + 1: [boxes][6][3][q][p]."""
        K, S = self.case["K"], lambda j: self.record[:, _tri(j)]
        j = n // K
        s = n + 1 - j * K
        th = s / K
        if self.case["interp"] == "linear":
            return (1.0 - th) * S(j) + th * S(j + 1)
        h00, h10 = 2 * th ** 3 - 3 * th ** 2 + 1, th ** 3 - 2 * th ** 2 + th
        h01, h11 = -2 * th ** 3 + 3 * th ** 2, th ** 3 - th ** 2
        m0 = 0.5 * (S(j + 1) - S(j - 1)) if j > 0 else S(1) - S(0)
        u = h00 * S(j) + h10 * m0 + h01 * S(j + 1) + h11 * 0.5 * (S(j + 2) - S(j))
        return u if self.residual is None else u + self.residual[:, s - 1]  # interval 0 only

    def pulled(self):
        return [torch.roll(self.d[i], (int(_C[i, 2]), int(_C[i, 1]), int(_C[i, 0])), (1, 2, 3)) for i in range(19)]

    def velocity(self, n):
        """Pulled moments: density deviation and velocity with the half body force."""
        g = self.pulled()
        r, j = _moments(g)
        a = self.accel(n)
        return g, r, j, [j[c] / (1.0 + r) + 0.5 * a[c] for c in range(3)]

    def chain(self, n, u):
        """Moves the beads over step n; the force density they leave, [3][boxes][sites]."""
        E, N, dt = self.E, self.N, 1.0 / 50
        nbox = len(self.ids)
        base = self.pos.floor()
        dlt = self.pos - base
        base = base.long()
        flat = torch.stack(u).view(3, nbox, -1)
        at, wt = [], []
        for c in range(8):
            b = [(c >> a) & 1 for a in range(3)]
            at.append(((base[..., 2] + b[2]) * E + base[..., 1] + b[1]) * E + base[..., 0] + b[0])
            wt.append(math.prod(dlt[..., a] if b[a] else 1.0 - dlt[..., a] for a in range(3)) * self.own)
        ub = torch.zeros_like(self.pos)
        for c in range(8):
            at[c] = at[c].clamp(0, E ** 3 - 1)
            for a in range(3):
                ub[..., a] += wt[c] * torch.gather(flat[a], 1, at[c])
        amp = math.sqrt(2.0 * self.case["kT"] / dt)
        pair = (self.own[:, :, None] & self.own[:, None, :]) & ~torch.eye(N, dtype=torch.bool, device="cuda")
        bond = self.own[:, 1:, None]
        mom = torch.zeros_like(self.pos)
        x1 = torch.arange(N, device="cuda")[None, :].expand(nbox, N)
        box = torch.tensor(self.ids, device="cuda")[:, None].expand(nbox, N)
        for sub in range(50):
            dx = self.pos[:, :, None, :] - self.pos[:, None, :, :]
            r2 = (dx * dx).sum(-1)
            near = pair & (r2 < 2.0 ** (1.0 / 3.0))
            inv = torch.where(near, 1.0 / torch.where(near, r2, 1.0), 0.0)
            s6 = inv ** 3
            F = ((24.0 * (2.0 * s6 * s6 - s6) * inv)[..., None] * dx).sum(2)
            b = self.pos[:, 1:] - self.pos[:, :-1]
            f = torch.where(bond, -30.0 * b / (1.0 - (b * b).sum(-1, keepdim=True) / 2.25), 0.0)
            F[:, 1:] += f
            F[:, :-1] -= f
            fric = ub - self.vel
            if amp:
                # the seed of a box is the first's plus its index
                key = torch.tensor([self.seed * 1000 + i for i in self.ids], device="cuda")[:, None]
                r = _philox_keyed(torch.full_like(x1, n), torch.full_like(x1, sub), x1, box, key)
                w = [_unit(r[a], self.case["storage"]) for a in range(3)]
                fric = fric + amp * torch.stack(w, -1)
            self.vel = torch.where(self.own[..., None], self.vel + dt * (F + fric), 0.0)
            self.pos = self.pos + dt * self.vel
            mom = mom - dt * fric
        cnt = self.nb[:, None].double()
        com = (self.pos * self.own[..., None]).sum(1) / cnt
        vcm = (self.vel * self.own[..., None]).sum(1) / cnt
        self.pos = torch.where(self.own[..., None], self.pos + (0.5 * (E - 1) - com)[:, None], 0.0)
        self.vel = torch.where(self.own[..., None], self.vel - vcm[:, None], 0.0)
        g = torch.zeros_like(flat)
        for c in range(8):
            for a in range(3):
                g[a].scatter_add_(1, at[c], wt[c] * mom[..., a])
        return g

    def step(self, n):
        E, om = self.E, self.om
        g, r, j, u = self.velocity(n)
        rho, a = 1.0 + r, self.accel(n)
        F = [rho * a[c] if a[c] else 0.0 for c in range(3)]
        if self.N:
            gb = self.chain(n, u)
            F = [F[c] + gb[c].view(-1, E, E, E) for c in range(3)]
        forced = self.N > 0 or self.acc is not None
        if self.case["kind"] == "thermal":
            new = self.thermal(n, g, r, j)
        else:
            u = [(j[c] + 0.5 * F[c]) / rho for c in range(3)]
            usq = 1.5 * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2)
            uF = sum(u[c] * F[c] for c in range(3))
            new = []
            for i in range(19):
                e, cu = _equilibrium(i, r, u, usq)
                v = g[i] + om * (e - g[i])
                if forced:
                    cF = sum(float(_C[i, c]) * F[c] for c in range(3) if _C[i, c]) if i else 0.0
                    v = v + (1.0 - 0.5 * om) * float(_W[i]) * (3.0 * (cF - uF) + 9.0 * cu * cF)
                new.append(v)
        if not self.per:  # the outer layer: a site on several faces belongs to the first
            s = self.boundary(n)
            ub = [torch.zeros_like(r) for _ in range(3)]
            for c in range(3):
                ub[c][:, -1], ub[c][:, 0] = s[:, 5, c], s[:, 4, c]
                ub[c][:, :, -1], ub[c][:, :, 0] = s[:, 3, c], s[:, 2, c]
                ub[c][..., -1], ub[c][..., 0] = s[:, 1, c], s[:, 0, c]
            usq = 1.5 * (ub[0] ** 2 + ub[1] ** 2 + ub[2] ** 2)
            zero = torch.zeros_like(r)
            new = [torch.where(self.mask, _equilibrium(i, zero, ub, usq)[0], new[i]) for i in range(19)]
        self.d = new

    def thermal(self, n, g, r, j):
        e = _modes19()
        b = (e * e * _W).sum(1)
        gam = _gammas(self.case["tau"])
        rho = 1.0 + r
        u = [j[c] / rho for c in range(3)]
        usq = 1.5 * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2)
        eq = [_equilibrium(i, r, u, usq)[0] for i in range(19)]
        new = list(eq)
        site = torch.arange(self.E ** 3, device="cuda").view(1, self.E, self.E, self.E)
        for blk in range(4):
            x = _philox(torch.full_like(site, n), site, torch.full_like(site, blk), torch.full_like(site, 0xF1), self.seed)
            for w in range(4):
                k = 4 + 4 * blk + w
                if k > 18:
                    break
                m = sum(float(e[k, i]) * (g[i] - eq[i]) for i in range(19) if e[k, i])
                m = gam[k] * m + math.sqrt(3.0 * self.case["kT"] * b[k] * (1.0 - gam[k] ** 2)) * rho.sqrt() * _unit(x[w], self.case["storage"])
                for i in range(19):
                    if e[k, i]:
                        new[i] = new[i] + float(_W[i] * e[k, i] / b[k]) * m
        return new

    def fields(self, n):
        """Density deviation and velocity as they are read out at step n."""
        _, r, _, u = self.velocity(n)
        if self.per:
            return r, u
        r0, j0 = _moments(self.d)
        return torch.where(self.mask, r0, r), [torch.where(self.mask, j0[c] / (1.0 + r0), u[c]) for c in range(3)]


def _philox_keyed(x0, x1, x2, x3, key):
    """_philox with a tensor of seeds."""
    m = 0xFFFFFFFF
    k0, k1 = key & m, (key >> 32) & m
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & m, (k1 + 0xBB67AE85) & m
        p0, p1 = x0 * 0xD2511F53, x2 * 0xCD9E8D57
        x0, x1, x2, x3 = ((p1 >> 32) & m) ^ x1 ^ k0, p1 & m, ((p0 >> 32) & m) ^ x3 ^ k1, p0 & m
    return x0, x1, x2, x3


def _net(master, K, rounded):
    """Weights of a master vector in FP64; rounded: the weights as the bf16 the network runs with."""
    m = torch.from_numpy(master).cuda()
    out, o = [], 0
    for shape in ((32, 128), (128,), (128, 128), (128,), (128, 3 * K), (3 * K,)):
        n = int(np.prod(shape))
        w = m[o:o + n].view(shape)
        out.append((w.to(torch.bfloat16) if rounded and len(shape) == 2 else w).double())
        o += n
    return out


def _predict(net, x):
    w1, b1, w2, b2, w3, b3 = net
    return (torch.relu(torch.relu(x @ w1 + b1) @ w2 + b2) @ w3) + b3


def _exact_features(smp):
    """[6 E^2][24] of samples j - 1 .. j + 2, each [6][3][E][E]."""
    cols = list(smp)
    for s in smp[1:3]:
        gp = torch.cat([s[..., 1:2] - s[..., :1], 0.5 * (s[..., 2:] - s[..., :-2]), s[..., -1:] - s[..., -2:-1]], -1)
        gq = torch.cat([s[..., 1:2, :] - s[..., :1, :], 0.5 * (s[..., 2:, :] - s[..., :-2, :]), s[..., -1:, :] - s[..., -2:-1, :]], -2)
        cols += [gp, gq]
    return torch.cat(cols, 1).permute(0, 2, 3, 1).reshape(-1, 24) / U_MAX


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "evaluate":
        return _exact_evaluate(case, seed)
    c = _full(case)
    edges, beads, flows, starts = _boxes(c, seed)
    real = torch.float64 if c["storage"] == "f64" else torch.float32
    per, zoom, K, G = bool(c.get("periodic")), c.get("zoom", 1), c["K"], c["steps"]
    net = _net(inputs.mlp_init(seed, K), K, True) if kind == "upsample" else None
    offs = np.concatenate([[0], np.cumsum([e ** 3 for e in edges])])
    boff = np.concatenate([[0], np.cumsum(beads)]).astype(int)
    rho = torch.empty(int(offs[-1]), dtype=torch.float64, device="cuda")
    u = torch.empty(3 * int(offs[-1]), dtype=torch.float64, device="cuda")
    hist = torch.zeros((G, int(boff[-1]), 3), dtype=torch.float64, device="cuda")
    extra = {}
    for E in sorted(set(edges)):
        every = [b for b, e in enumerate(edges) if e == E]
        room = max(1, int(6e9 // (19 * 8 * E ** 3)))
        for ids in (every[k:k + room] for k in range(0, len(every), room)):
            rec, acc, res = None, None, None
            if not per:
                parts = [_record(c, [flows[b]], real) for b in ids]
                acc = parts[0][1]
                Ec = _coarse(E, zoom)
                rec = torch.stack([p[0].view(RECORD, 6, 3, Ec, Ec) for p in parts]).double()
            u0 = torch.stack([_start_field(c, flows[b], real) for b in ids]).double()
            if net is not None:  # interval 0: sample -1 is sample 0
                res = []
                for k in range(len(ids)):
                    x = _exact_features([rec[k, 0], rec[k, 0], rec[k, 1], rec[k, 2]])
                    y = _predict([net[0][:24]] + net[1:], x) * (U_MAX / 64.0)
                    res.append(y.view(6, E, E, K, 3).permute(3, 0, 4, 1, 2))
                res = torch.stack(res)
            ref = _Reference(c, seed, E, ids, [beads[b] for b in ids], [starts[b] for b in ids] if sum(beads) else [],
                             u0, rec, acc, res)
            del u0, rec
            for n in range(G):
                ref.step(n)
                if ref.N:
                    for k, b in enumerate(ids):
                        hist[(n + 1) % G, boff[b]:boff[b] + beads[b]] = ref.pos[k, :beads[b]]
            r, v = ref.fields(G)
            for k, b in enumerate(ids):
                rho[offs[b]:offs[b + 1]] = r[k].reshape(-1)
                u[3 * offs[b]:3 * offs[b + 1]] = torch.stack([v[a][k] for a in range(3)]).reshape(-1)
            if kind == "observe":
                tot, mom = _moments(ref.d)
                extra = {"sums": torch.tensor([float(E ** 3 + tot.sum())] + [float(m.sum()) for m in mom] + [0.0] * 3).double(),
                         "vorticity": np.array(_exact_vorticity(v, E))}
            del ref, r, v
            torch.cuda.empty_cache()
    if kind == "observe":
        return dict(extra, rho=rho + 1.0, u=u)
    out = {"u": u} if len(edges) > 1 else {"rho": rho + 1.0, "u": u}
    if sum(beads):
        out["beads"] = hist
    return out


def _exact_vorticity(v, E):
    x, y, z = (v[a][0] for a in range(3))
    d = lambda f, a: 0.5 * (torch.roll(f, -1, 2 - a) - torch.roll(f, 1, 2 - a))  # noqa: E731
    w = ((d(z, 1) - d(y, 2)) ** 2 + (d(x, 2) - d(z, 0)) ** 2 + (d(y, 0) - d(x, 1)) ** 2).sqrt()
    c, half = (E - 1) / 2.0, 1.25 / 12.0 * E
    lo, hi = math.ceil(c - half), math.floor(c + half) + 1
    return [float(w[1:-1, 1:-1, 1:-1].mean()), float(w[lo:hi, lo:hi, lo:hi].mean())]


def _exact_train(case, seed):
    """One Adam step from the master weights, the gradient through the bf16 weights the network runs with."""
    K, lr = case["K"], 2e-3
    X, T = _train_rows(case, seed)
    master = inputs.mlp_init(seed, K)
    net = [w.requires_grad_() for w in _net(master, K, True)]
    loss = ((_predict(net, X.double()) - T.double()) ** 2).mean()
    grads = torch.autograd.grad(loss, net)
    new = [w - lr * (g / (g.abs() + 1e-8)) for w, g in zip(_net(master, K, False), grads)]
    w1, b1, w2, b2, w3, b3 = new
    return {"w1": w1.T.reshape(-1), "w2": w2.T.reshape(-1), "w3": w3.T.reshape(-1), "b1": b1, "b2": b2, "b3": b3,
            "loss": loss.detach().view(1)}


def _exact_evaluate(case, seed):
    K, E = case["K"], case["E"]
    net = _net(inputs.mlp_init(seed, K), K, True)
    xs, ts = [], []
    for f in _evaluate_data(case, seed):
        f = f.double()
        smp = [f[0], f[K], f[2 * K], f[3 * K]]
        xs.append(torch.nn.functional.pad(_exact_features(smp), (0, 8)))
        m0, m1 = 0.5 * (smp[2] - smp[0]), 0.5 * (smp[3] - smp[1])
        t = []
        for s in range(1, K + 1):
            th = s / K
            h = ((2 * th ** 3 - 3 * th ** 2 + 1) * smp[1] + (th ** 3 - 2 * th ** 2 + th) * m0 + (-2 * th ** 3 + 3 * th ** 2) * smp[2]
                 + (th ** 3 - th ** 2) * m1)
            t.append((f[K + s] - h).permute(0, 2, 3, 1).reshape(-1, 3))
        ts.append(torch.cat(t, 1) * (64.0 / U_MAX))
    x = torch.cat(xs)
    return {"x": x, "t": torch.cat(ts), "y": _predict(net, x)}

"""The work that users of the library have it do, as measurable cases through its public entry points.

Six kinds of case:
  layer    one SSM layer, forward + backward (a training step of the sequence model), or forward only
  stack    the stacked sequence model, forward + backward
  block    the paper's sequence block (SSM layer, then the half-GLU gate), one or two of them, forward + backward
  rollout  single steps with the state handed on, optionally after a forward pass over a context (imagination, serving)
  scan     the two scan entry points on their own

Inputs follow the distributions of paper_2502_20168_b200/inputs.py; sizes are those of the repository's
workloads, tests and benchmark, or ragged neighbours of them.
"""
import math

import torch

from paper_2502_20168_b200 import binding as sb, harness, inputs as I

IO = {"f32": torch.float32, "bf16": torch.bfloat16}


def listed():
    return [
        # the smallest training call: a unit-test sized layer, all latency and launches
        {"name": "tiny_layer_fp32", "kind": "layer", "B": 1, "T": 64, "H": 32, "P": 16, "io": "f32", "p_done": 0.0,
         "states": False, "backward": True},
        # a world-model batch in fp32 with episode ends
        {"name": "wm_batch_fp32", "kind": "layer", "B": 16, "T": 64, "H": 256, "P": 128, "io": "f32", "p_done": 0.01,
         "states": False, "backward": True},
        # the four-layer stacked sequence model
        {"name": "stack4_bf16", "kind": "stack", "B": 16, "T": 64, "H": 512, "P": 256, "io": "bf16", "p_done": 0.01, "layers": 4},
        # the paper's training batch, state task: one block of layer and gate
        {"name": "state_block_bf16", "kind": "block", "B": 32, "T": 128, "H": 512, "P": 256, "io": "bf16", "p_done": 0.01,
         "layers": 1},
        # the same for the vision task: two blocks of twice the width
        {"name": "vision_blocks_bf16", "kind": "block", "B": 32, "T": 128, "H": 1024, "P": 512, "io": "bf16", "p_done": 0.01,
         "layers": 2},
        # few long sequences with episode ends
        {"name": "long_horizon_bf16", "kind": "layer", "B": 16, "T": 1024, "H": 512, "P": 256, "io": "bf16", "p_done": 0.002,
         "states": False, "backward": True},
        # the largest: the middle of the scan-scaling sweep, the benchmark's headline
        {"name": "sweep_T1024_bf16", "kind": "layer", "B": 256, "T": 1024, "H": 512, "P": 256, "io": "bf16", "p_done": 0.0,
         "states": False, "backward": True},
        # lengths and widths off the tile sizes, with initial states and final-state gradients (truncated backpropagation)
        {"name": "ragged_bf16", "kind": "layer", "B": 150, "T": 200, "H": 384, "P": 192, "io": "bf16", "p_done": 0.01,
         "states": True, "backward": True},
        # imagination: 15 steps of as many trajectories as a training batch has steps
        {"name": "imagination_bf16", "kind": "rollout", "B": 4096, "T": 0, "H": 512, "P": 256, "io": "bf16", "p_done": 0.01,
         "steps": 15},
        # serving a few trajectories: forward over a context, then single steps from its final state
        {"name": "context_steps_fp32", "kind": "rollout", "B": 16, "T": 64, "H": 256, "P": 128, "io": "f32", "p_done": 0.01,
         "steps": 15},
        # a full fp32 training step of a large batch, the length off the tile sizes
        {"name": "large_fp32", "kind": "layer", "B": 64, "T": 1000, "H": 512, "P": 256, "io": "f32", "p_done": 0.002,
         "states": True, "backward": True},
        # the scans alone on very long sequences
        {"name": "scan_T16384_fp32", "kind": "scan", "B": 16, "T": 16384, "P": 256, "p_done": 0.0},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


WIDTHS = ((256, 128), (256, 256), (384, 192), (512, 128), (512, 256), (768, 256), (1024, 512))


def draw(rng):
    kind = rng.choice(("layer", "layer", "layer", "stack", "block", "rollout", "scan"))
    p_done = rng.choice((0.0, 0.002, 0.01))
    if kind == "layer":
        io = rng.choice(("f32", "bf16", "bf16"))
        odd = rng.random() < 0.2
        H, P = (8 * rng.randint(2, 24), 8 * rng.randint(1, 16)) if odd else rng.choice(WIDTHS)
        most = 1 << (14 if odd else 15 if io == "f32" else 18)   # rows
        rows = min(_log_int(rng, 64, most), (1 << 35) // (H * P))
        T = min(rows, rng.choice((16, 32, 64, 128, 256, 1024, 4096, 16384, _log_int(rng, 1, 5000), _log_int(rng, 30, 1000))))
        return {"kind": kind, "B": max(1, rows // T), "T": T, "H": H, "P": P, "io": io, "p_done": p_done,
                "states": rng.random() < 0.4, "backward": rng.random() < 0.75}
    if kind == "stack":
        H, P = rng.choice(((256, 128), (512, 256)))
        return {"kind": kind, "B": rng.randint(4, 32), "T": rng.choice((32, 50, 64, 100, 128)), "H": H, "P": P,
                "io": rng.choice(("f32", "bf16")), "p_done": p_done, "layers": rng.randint(2, 6)}
    if kind == "block":
        H, P = rng.choice(((256, 128), (512, 256), (1024, 512)))
        return {"kind": kind, "B": rng.randint(8, 64), "T": rng.choice((50, 64, 100, 128, 200)), "H": H, "P": P, "io": "bf16",
                "p_done": p_done, "layers": rng.randint(1, 2)}
    if kind == "rollout":
        H, P = rng.choice(((256, 128), (512, 256), (1024, 512)))
        B = _log_int(rng, 1, 4096)
        T = rng.choice((0, rng.randint(1, 100))) if B <= 256 else 0
        return {"kind": kind, "B": B, "T": T, "H": H, "P": P, "io": rng.choice(("f32", "bf16")), "p_done": p_done,
                "steps": rng.randint(1, 15)}
    rows = _log_int(rng, 1024, 1 << 18)
    T = min(rows, _log_int(rng, 16, 16384))
    return {"kind": kind, "B": max(1, rows // T), "T": T, "P": 8 * rng.randint(4, 32), "p_done": p_done}


# ---- states --------------------------------------------------------------------------------------
def _workload(case, seed, T=None):
    return I.Workload("case", B=case["B"], T=case["T"] if T is None else T, H=case["H"], P=case["P"], io_dtype=case["io"],
                      p_done=case["p_done"], n_layers=case.get("layers", 1), seed=int(seed))


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) + 1)
    return g


def _complex_normal(g, *shape):
    return torch.view_as_complex(torch.randn((*shape, 2), device="cuda", generator=g))


def _flags(g, p_done, *shape):
    return (torch.rand(shape, device="cuda", generator=g) < p_done).to(torch.uint8) if p_done > 0 else None


def _layer(case, seed):
    buf = harness.LayerBuffers(harness.device_drawn(_workload(case, seed)), case["io"])
    if case["states"]:
        g = _generator(seed)
        buf.x0 = _complex_normal(g, case["B"], case["P"])
        buf.gxT = _complex_normal(g, case["B"], case["P"])
    return buf


class _Blocks:
    """A chain of the paper's blocks: per block one layer and one gate."""

    def __init__(self, case, seed):
        n, B, T, H, P = case["layers"], case["B"], case["T"], case["H"], case["P"]
        self.shape = sb.make_shape(B, T, H, P, case["io"])
        d = harness.device_drawn(_workload(case, seed))
        params = d["params"] if n > 1 else [{k: d[k] for k in ("Lambda", "Delta", "Bc", "Cc", "D")}]
        g = _generator(seed)
        self.u, self.gout = d["u"], d["gy"]
        self.layers = [harness.LayerBuffers(dict(p, u=d["u"], gy=d["gy"], done=d["done"]), case["io"]) for p in params]
        self.W = [torch.randn((H, H), device="cuda", generator=g) / math.sqrt(H) for _ in params]
        self.dW = [torch.empty_like(W) for W in self.W]
        self.out = [torch.empty_like(d["u"]) for _ in params]
        self.gv = [torch.empty_like(d["u"]) for _ in params]
        self.gate_ws = [sb.alloc_workspace(sb.ssm_glu_workspace_bytes(self.shape)) for _ in params]
        x = self.u
        for l, layer in enumerate(self.layers):   # the chain's buffers
            layer.u, layer.gy = x, self.gv[l]
            x = self.out[l]

    def step(self):
        for l, layer in enumerate(self.layers):
            layer.forward()
            sb.ssm_glu_fwd(self.shape, self.W[l], layer.y, self.out[l], self.gate_ws[l])
        g = self.gout
        for l in reversed(range(len(self.layers))):
            layer = self.layers[l]
            sb.ssm_glu_bwd(self.shape, self.W[l], layer.y, g, self.gate_ws[l], self.gv[l], self.dW[l])
            layer.backward()
            g = layer.du
        return [self.out[-1], self.layers[0].du, self.dW,
                [[q.dLambda, q.dDelta, q.dB, q.dC, q.dD] for q in self.layers]]


class _Rollout:
    """Single steps for B trajectories from a prepared step workspace; with a context, from its final state."""

    def __init__(self, case, seed):
        B, H, P, n = case["B"], case["H"], case["P"], case["steps"]
        g = _generator(seed)
        self.context = None
        if case["T"] > 0:
            self.context = harness.LayerBuffers(harness.device_drawn(_workload(case, seed)), case["io"])
            q = self.context
        else:
            q = harness.LayerBuffers(harness.device_drawn(_workload(case, seed, T=1)), case["io"])
        self.D = q.D
        self.shape = sb.make_shape(B, 1, H, P, case["io"])
        self.ws = sb.alloc_workspace(sb.ssm_step_workspace_bytes(self.shape))
        sb.ssm_step_prepare(self.shape, q.Lambda, q.Delta, q.Bc, q.Cc, self.ws)
        self.u = torch.randn((n, B, H), device="cuda", generator=g).to(IO[case["io"]])
        self.done = _flags(g, case["p_done"], n, B)
        # flags are handed over by pointer, 16-byte aligned: one row per step
        self.done = [None] * n if self.done is None else [self.done[t].clone() for t in range(n)]
        self.u = [self.u[t].clone() for t in range(n)]
        self.y = [torch.empty_like(u) for u in self.u]
        self.x0 = q.xT if self.context is not None else _complex_normal(g, B, P)
        self.x = torch.empty_like(self.x0)

    def steps(self):
        if self.context is not None:
            self.context.forward()
        x = self.x0
        for u, done, y in zip(self.u, self.done, self.y):
            sb.ssm_step(self.shape, self.D, u, done, x, self.x, y, self.ws)
            x = self.x
        return [self.y, self.x] + ([self.context.y, self.context.xT] if self.context is not None else [])


class _Scan:
    def __init__(self, case, seed):
        B, T, P = case["B"], case["T"], case["P"]
        g = _generator(seed)
        self.shape = sb.make_shape(B, T, 8, P, "f32")
        lam = torch.complex(torch.rand(P, device="cuda", generator=g) * -0.99 - 0.01,
                            torch.rand(P, device="cuda", generator=g) * math.pi)
        delta = torch.exp(math.log(1e-3) + torch.rand(P, device="cuda", generator=g) * math.log(1e2))
        self.Abar = torch.exp(lam * delta)
        self.Bu = _complex_normal(g, B, T, P)
        self.gx = _complex_normal(g, B, T, P)
        self.done = _flags(g, case["p_done"], B, T)
        self.x0, self.gxT = _complex_normal(g, B, P), _complex_normal(g, B, P)
        self.x, self.gBu = torch.empty_like(self.Bu), torch.empty_like(self.Bu)
        self.xT, self.gx0 = torch.empty_like(self.x0), torch.empty_like(self.x0)
        self.gAbar = torch.empty_like(self.Abar)
        self.ws = sb.alloc_workspace(sb.ssm_scan_workspace_bytes(self.shape))

    def both(self):
        sb.ssm_scan_fwd(self.shape, self.Abar, self.Bu, self.done, self.x0, self.x, self.xT, self.ws)
        sb.ssm_scan_bwd(self.shape, self.Abar, self.done, self.x0, self.x, self.gx, self.gxT, self.gBu, self.gAbar,
                        self.gx0, self.ws)
        return [self.x, self.xT, self.gBu, self.gAbar, self.gx0]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "layer":
        state = _layer(case, seed)
    elif kind == "stack":
        state = harness.StackBuffers(harness.device_drawn(_workload(case, seed)), case["io"])
    elif kind == "block":
        state = _Blocks(case, seed)
    elif kind == "rollout":
        state = _Rollout(case, seed)
    else:
        state = _Scan(case, seed)
    return case, state


def run(prepared):
    case, s = prepared
    kind = case["kind"]
    if kind == "layer":
        s.forward()
        if not case["backward"]:
            return [s.y, s.xT]
        s.backward()
        return [s.y, s.xT, s.du, s.dLambda, s.dDelta, s.dB, s.dC, s.dD] + ([s.dx0] if case["states"] else [])
    if kind == "stack":
        s.forward()
        s.backward()
        return [s.out, s.du, s.grads]
    if kind == "block":
        return s.step()
    if kind == "rollout":
        return s.steps()
    return s.both()


# ---- what a pass cannot do without ------------------------------------------------------------------
def work(case):
    kind, B, P = case["kind"], case["B"], case["P"]
    if kind == "scan":   # Bu, gx in, x, gBu out (complex fp32); one multiply-add forward, two backward per element
        n = B * case["T"] * P
        return {"bytes": 4 * 8 * n, "flops": 24 * n}
    H, es = case["H"], 4 if case["io"] == "f32" else 2
    rows, n = B * case["T"], case.get("layers", 1)
    weights = 16 * H * P + 12 * P + 4 * H   # B, C, Lambda, Delta, D
    if kind == "rollout":
        rows += B * case["steps"]
        return {"bytes": 2 * rows * H * es + weights + 16 * B * P, "flops": rows * (8 * H * P + 8 * P)}
    flags = rows if case["p_done"] > 0 else 0
    if kind == "layer" and not case["backward"]:
        return {"bytes": 2 * rows * H * es + flags + weights, "flops": rows * (8 * H * P + 8 * P)}
    # input and output gradient in, output and input gradient out; six products of 4 H P flops, two scans
    moved, flops = 4 * rows * H * es + flags + 2 * n * weights, n * rows * (24 * H * P + 24 * P)
    if kind == "block":   # and the gate's three products
        return {"bytes": moved + 8 * n * H * H, "flops": flops + n * rows * 6 * H * H}
    return {"bytes": moved, "flops": flops}


def tolerance(case):
    """About four times what the path differs by from the same computation in 64 bits (sequential recurrence, the
    roundings of bf16 tensors kept), worst output of the listed cases and two dozen drawn ones."""
    if case["kind"] == "scan":          # 1.2e-6 (gAbar over 262144 rows) / 1.4e-5
        return {"rel": 5e-6, "max": 6e-5}
    if case["io"] == "f32":             # 3.9e-6 (gradients summed over 64000 rows) / 2.6e-5
        return {"rel": 1.6e-5, "max": 1e-4}
    if case["kind"] == "block":         # 2.9e-3 / 0.12: bf16 values that round the other way between layer and gate
        return {"rel": 1.2e-2, "max": 0.5}
    if case["kind"] == "stack":         # 1.7e-3 / 3.9e-3: output and input gradient are bf16, all else fp32
        return {"rel": 7e-3, "max": 1.6e-2}
    return {"rel": 9e-3, "max": 4.5e-2}   # 2.3e-3 / 1.1e-2: bf16 output of a bf16 product of the states

"""What the performance of this library is measured on: the calls its users make, over the range of sizes they make
them at.

A case is one pass of one of these kinds, through the Python binding:

  topk     dgs_topk_encode_static on a vector: the selection for callers that may not allocate.
  select   a vector is loaded as a worker's difference and selected from (state_load, worker_pull).
  events   arrivals of workers at the server (push, apply, pull with secondary compression), then one flush.  One
           arrival per pass is a training loop that computes the next gradient from the result of this one; a round
           of all workers per pass is the replay of an arrival schedule, where consecutive events overlap.
  full     the same with worker_pull_all (no secondary compression, the paper's normal case) as three calls.
  host     one arrival through dgs_event_host: gradient from pinned host memory, pull packet back to the host.
  server   the server alone, fed with packets that other processes made (server_apply of a caller's packet,
           worker_pull).

Shapes are those of the workloads of this repository or generic ones; gradients are synthetic (see workloads/), made
on the GPU.  Every context has served two rounds of its workers before it is measured, as a running job has.  All
results are defined bit for bit (one rounded operation per step, a total order in the selection), so outputs are
compared exactly.
"""
import math

import numpy as np
import torch

import paper_1910_10929_b200 as dgs
import workloads
from workloads import shapes

DEV = "cuda:0"
GRADIENT_BYTES = 3.6e9   # room for the distinct gradients that a state keeps
TENSORS = {"resnet18": shapes.resnet18_shapes, "resnet50": shapes.resnet50_shapes, "gpt2": shapes.gpt2_small_shapes}
PACKET_FLAG = {"f32": 0, "bf16": dgs.DGS_PACKET_BF16, "fp16": dgs.DGS_PACKET_FP16}


def _case(name, kind, **kw):
    c = {"kind": kind, "shape": "flat", "n": 0, "layers": 1, "per_layer": False, "workers": 1, "events": 1,
         "ppm": 1000, "grad": "normal", "arrivals": "cyclic", "packet": "f32", "rule": "momentum", "keep": False}
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest cell of the kernel sweep: a call inside a loop whose memory plan is frozen, where launches count
        _case("topk 2^16 0.1%", "topk", n=1 << 16, ppm=1000),
        # the same call near its limit, with an odd length and a dense packet
        _case("topk 1000003 5%", "topk", n=1_000_003, ppm=50_000),
        # the small flat model with four workers that arrive at random, one at a time
        _case("event flat 2^20 4w", "events", n=1 << 20, ppm=1000, workers=4, arrivals="uniform"),
        # training 8 workers of an ordinary model on one GPU, one arrival at a time, local models kept (Eq. 5)
        _case("event resnet50 8w keep", "events", shape="resnet50", ppm=1000, workers=8, grad="laplace", keep=True),
        # the benchmark's configuration: a round of 32 workers, one selection over the whole model
        _case("round resnet50 32w", "events", shape="resnet50", ppm=1000, workers=32, events=32, grad="laplace"),
        # the paper's model and density: a selection per layer, 1 %
        _case("round resnet18 layers 32w", "events", shape="resnet18", per_layer=True, ppm=10_000, workers=32, events=32,
              grad="laplace"),
        # the largest model: sparse embedding gradients, heavy tails, 0.1 %
        _case("round gpt2 32w", "events", shape="gpt2", ppm=1000, workers=32, events=32, grad="student_t"),
        # the same with a selection per layer, few workers, and bfloat16 packets
        _case("round gpt2 layers 8w bf16", "events", shape="gpt2", per_layer=True, ppm=1000, workers=8, events=8,
              grad="student_t", packet="bf16"),
        # Algorithm 1 with the whole difference sent back (gradient dropping without secondary compression)
        _case("full resnet18 layers 8w", "full", shape="resnet18", per_layer=True, ppm=10_000, workers=8, events=8,
              grad="laplace", rule="residual", keep=True),
        # a worker process without device buffers of its own: gradient in and packet out through host memory
        _case("host resnet18 layers 4w", "host", shape="resnet18", per_layer=True, ppm=10_000, workers=4, grad="laplace"),
        # a server that remote workers send their packets to
        _case("server resnet50 16w", "server", shape="resnet50", ppm=1000, workers=16, events=16, grad="laplace"),
        # a large cell of the kernel sweep: one selection from a loaded vector
        _case("select 2^26 1%", "select", n=1 << 26, ppm=10_000, grad="sweep"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["topk", "topk", "events", "events", "events", "events", "full", "host", "server", "select"])
    if kind == "topk":
        return _case(None, kind, n=_log(rng, 1 << 12, 1 << 20), ppm=_log(rng, 100, 100_000))
    if kind == "select":
        return _case(None, kind, n=_log(rng, 1 << 16, 1 << 27), ppm=_log(rng, 100, 100_000), grad="sweep")
    n = _log(rng, 1 << 16, 1 << 25)
    layers = rng.choice([1, _log(rng, 2, 200)])
    workers = _log(rng, 2, 32)
    # at most about as many entries in a packet as the largest workloads send
    ppm = _log(rng, 300, min(30_000, max(1000, int(2e11 / n))))
    return _case(None, kind, n=n, layers=layers, per_layer=layers > 1 and rng.random() < 0.7, workers=workers,
                 events=1 if kind == "host" else rng.choice([1, workers, workers]), ppm=ppm,
                 grad=rng.choice(["normal", "laplace", "student_t"]), arrivals=rng.choice(["cyclic", "cyclic", "uniform"]),
                 packet=rng.choice(["f32", "f32", "bf16", "fp16"]), rule=rng.choice(["momentum", "momentum", "residual"]),
                 keep=rng.random() < 0.3)


# ---- sizes -------------------------------------------------------------------------------------------------------
def _tensor_sizes(case):
    if case["shape"] != "flat":
        return shapes.sizes(TENSORS[case["shape"]]())
    n, layers = case["n"], case["layers"]
    if layers == 1:
        return [n]
    # layers of very different sizes, the small ones of a few elements, as biases and norms are
    w = np.random.RandomState(layers + n).lognormal(0.0, 2.0, layers)
    size = np.maximum(1, np.floor(w / w.sum() * n)).astype(np.int64)
    size[int(size.argmax())] += n - int(size.sum())
    return [int(x) for x in size]


def _segments(case):
    """(lengths, entries kept) of the slices that are selected from on their own."""
    sizes = _tensor_sizes(case)
    seg = sizes if case["per_layer"] else [sum(sizes)]
    return seg, [workloads.k_of(x, case["ppm"]) for x in seg]


def work(case):
    if case["kind"] == "topk":
        n, k = case["n"], workloads.k_of(case["n"], case["ppm"])
        return {"bytes": 4 * n + 8 * k, "flops": n}
    seg, ks = _segments(case)
    n, K, N, E = sum(seg), sum(ks), case["workers"], case["events"]
    if case["kind"] == "select":
        return {"bytes": 8 * n + 8 * K, "flops": n}        # the vector in, the difference and the packet out
    push = 12 * n + 8 * K                                  # velocity and gradient in, velocity and packet out
    apply = 8 * K + 8 * K * (N + 1)                        # packet in; model and every worker's difference, both ways
    pull = 4 * n + 12 * K                                  # difference in; packet out, sent entries cleared
    if case["keep"]:
        pull += 8 * K
    per_event = apply + pull + (0 if case["kind"] == "server" else push)
    return {"bytes": E * per_event, "flops": E * (K * (N + 2) + n + (0 if case["kind"] == "server" else 4 * n))}


def tolerance(case):
    return "exact"


# ---- inputs ------------------------------------------------------------------------------------------------------
class _Source:
    """Vectors of the case's distribution."""

    def __init__(self, case, gen):
        self.case, self.gen = case, gen
        self.sizes = _tensor_sizes(case)
        self.n = sum(self.sizes)
        if case["grad"] == "laplace":   # a scale per tensor, over three decades
            b = torch.pow(10.0, -5.0 + 3.0 * self._uniform(len(self.sizes)))
            self.scale = torch.repeat_interleave(b, torch.tensor(self.sizes, device=DEV))

    def _uniform(self, n):
        return torch.rand(n, generator=self.gen, device=DEV)

    def _normal(self, n):
        return torch.randn(n, generator=self.gen, device=DEV)

    def vector(self):
        n, grad = self.n, self.case["grad"]
        if grad == "laplace":
            x = torch.empty(n, device=DEV).exponential_(generator=self.gen).mul_(self.scale)
            return torch.copysign(x, self._uniform(n) - 0.5)
        if grad == "student_t":
            chi = self._normal(n).square_()
            for _ in range(2):
                chi.add_(self._normal(n).square_())
            x = self._normal(n).div_(chi.mul_(1.0 / 3.0).sqrt_().clamp_(min=1e-6)).mul_(1e-4)
            if self.case["shape"] == "gpt2":   # 99 % of the embedding's rows are not in the batch
                rows, cols = shapes.gpt2_small_shapes()[0][1]
                x[:rows * cols].view(rows, cols).mul_((self._uniform(rows) < 0.01).view(rows, 1))
            return x
        x = self._normal(n)
        if grad == "sweep":
            return torch.where(self._uniform(n) < 0.01, x * 100.0, x)
        return x.mul_(1e-3)


def _distinct(case, n):
    """How many gradients are kept and handed out in turn: with a common factor with the number of workers a worker
    would only ever see some of them."""
    g = int(max(3, min(31, GRADIENT_BYTES // (4 * n))))
    while math.gcd(g, case["workers"]) > 1:
        g += 1
    return g


def _context(case, theta0):
    seg, ks = _segments(case)
    flags = PACKET_FLAG[case["packet"]]
    flags |= dgs.DGS_KEEP_LOCAL_MODEL if case["keep"] else 0
    flags |= dgs.DGS_RESIDUAL_MODE if case["rule"] == "residual" else 0
    flags |= dgs.DGS_HOST_IO if case["kind"] == "host" else 0
    offset = np.concatenate([[0], np.cumsum(seg)[:-1]])
    return dgs.Context(sum(seg), case["workers"], 0.1, 0.9, offset, seg, ks, ks, theta0, flags=flags,
                       pull_all_capacity=sum(seg) if case["kind"] == "full" else 0)


def prepare(case, seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed))
    if case["kind"] == "topk":
        n, k = case["n"], workloads.k_of(case["n"], case["ppm"])
        return {"case": case, "n": n, "k": k, "x": _Source(case, gen).vector(),
                "idx": torch.empty(k, dtype=torch.int32, device=DEV), "val": torch.empty(k, device=DEV),
                "stream": torch.cuda.current_stream().cuda_stream}
    src = _Source(case, gen)
    n, N = src.n, case["workers"]
    s = {"case": case, "at": 0}
    theta0 = torch.randn(n, generator=gen, device=DEV).mul_(0.05)
    s["ctx"] = ctx = _context(case, theta0)
    s["D"] = [ctx.state(dgs.DGS_D, w) for w in range(N)]
    s["local"] = [ctx.state(dgs.DGS_THETA_LOCAL, w) for w in range(N)] if case["keep"] else None
    s["theta"] = ctx.state(dgs.DGS_THETA)
    rng = np.random.RandomState(int(seed) % (1 << 32))
    s["arrivals"] = [int(w) for w in (rng.permutation(N) if case["arrivals"] == "cyclic" else rng.randint(0, N, 4099))]
    inputs = [src.vector() for _ in range(3 if case["kind"] in ("host", "select") else _distinct(case, n))]
    if case["kind"] == "host":
        inputs = [torch.empty(n, pin_memory=True).copy_(g) for g in inputs]
        s["idx"] = torch.empty(ctx.K_pull, dtype=torch.int32, pin_memory=True)
        s["val"] = torch.empty(ctx.K_pull, pin_memory=True)
    elif case["kind"] == "full":     # what the caller sends the packets from, whatever their length
        s["idx"] = torch.zeros(n, dtype=torch.int32, device=DEV)
        s["val"] = torch.zeros(n, device=DEV)
        s["count"] = 0
    elif case["kind"] == "server":   # the packets of remote workers, made elsewhere
        inputs = [_remote_packet(case, g) for g in inputs]
    s["inputs"] = inputs
    for _ in range(-(-2 * N // case["events"])):
        run(s)
    return s


def _remote_packet(case, g):
    """The entries of largest magnitude of each slice, in index order, as a packet in the caller's memory."""
    at, idx = 0, []
    for length, k in zip(*_segments(case)):
        idx.append(torch.topk(g[at:at + length].abs(), k, sorted=False).indices + at)
        at += length
    idx = torch.cat(idx).sort().values
    val = g[idx] * 0.1
    if case["packet"] != "f32":
        val = val.to(torch.bfloat16 if case["packet"] == "bf16" else torch.float16).float()
    idx = idx.to(torch.int32)
    return idx, val, dgs.dgs_packet(idx.data_ptr(), val.data_ptr(), idx.numel())


# ---- a pass ------------------------------------------------------------------------------------------------------
def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "topk":
        dgs.dgs_topk_encode_static(s["x"].data_ptr(), s["n"], s["k"], s["idx"].data_ptr(), s["val"].data_ptr(), s["stream"])
        return s["idx"], s["val"]
    ctx = s["ctx"]
    if kind == "select":
        ctx.state_load(dgs.DGS_D, 0, s["inputs"][s["at"] % 3])
        s["at"] += 1
        return ctx.packet(ctx.worker_pull(0)) + (s["D"][0],)
    arrivals, inputs, at = s["arrivals"], s["inputs"], s["at"]
    push = pull = None
    for e in range(at, at + case["events"]):
        w, g = arrivals[e % len(arrivals)], inputs[e % len(inputs)]
        if kind == "events":
            push, pull = ctx.event(w, g)
        elif kind == "full":
            push = ctx.worker_push(w, g)
            ctx.server_apply(w, push)
            pull = ctx.worker_pull_all(w)
        elif kind == "host":
            ctx.event_host(w, g, s["idx"], s["val"])
        else:
            ctx.server_apply(w, g[2])
            pull = ctx.worker_pull(w)
    s["at"] = at + case["events"]
    # the model, and what the last arrival has produced and changed
    out = {"theta": s["theta"], "D": s["D"][w]}
    if case["keep"]:
        out["local"] = s["local"][w]
    if kind == "host":
        out["pull"] = (s["idx"], s["val"])
        return out
    if push is not None:
        out["push"] = ctx.packet(push)
    if kind == "full":
        # the caller waits for the number of entries, and moves that many into its send buffer
        idx, val = ctx.var_packet(pull)
        count = idx.numel()
        s["idx"][:count].copy_(idx)
        s["val"][:count].copy_(val)
        if count < s["count"]:
            s["idx"][count:s["count"]].zero_()
            s["val"][count:s["count"]].zero_()
        s["count"] = count
        out["pull"] = (s["idx"], s["val"], count)
    else:
        out["pull"] = ctx.packet(pull)
    return out

"""The workloads by which the library's speed is judged: what a program that
serves or converts packed ternary models has it do, through the public Python
entry points, from one small call to a whole decode step.

listed() names the cases, draw() makes more of the same ranges, prepare() /
run() execute one, work() counts what a pass cannot do without and exact()
states its result in 64-bit arithmetic with torch alone.

Inputs are synthetic, drawn on the device from a seed: trits 0.3 / 0.4 / 0.3,
lognormal(-4, 0.5) scales, N(0, 1e-3) offsets, a tenth of the groups salient
(the workload of tests and bench), dense weights with a scale per row and one
outlier in a thousand, activations N(0, 1) with one channel in 256 ten times
as large, as a transformer's normalised activations have them.
"""
from __future__ import annotations

import math

import torch

from paper_2609_09240_gb300 import tq

GROUP = 128
# The projections (N, K) of one layer of the two models of the benchmark.
LAYER = {
    "qwen3-4b": [(4096, 2560), (1024, 2560), (1024, 2560), (2560, 4096), (9728, 2560), (9728, 2560), (2560, 9728)],
    "qwen3-8b": [(4096, 4096), (1024, 4096), (1024, 4096), (4096, 4096), (12288, 4096), (12288, 4096),
                 (4096, 12288)],
}
# The same layer with q/k/v and gate/up as one projection each: the order in
# which a model depends on them.
FUSED = {
    "qwen3-4b": [(6144, 2560), (2560, 4096), (19456, 2560), (2560, 9728)],
    "qwen3-8b": [(6144, 4096), (4096, 4096), (24576, 4096), (4096, 12288)],
}
# Mask coverage of the element-wise form (masks 0..2, mask 3 the rest).
COVERAGE = (0.005, 0.031, 0.10)


def listed():
    return [
        # One small projection for one token: latency and launches.
        {"name": "linear_512x1024_m1", "kind": "linear", "M": 1, "N": 512, "K": 1024, "salient": 0.0, "index": True,
         "f32": False},
        # A small odd shape for five tokens without the optional second-plane
        # index, fp32 results: what a caller outside the tuned shapes gets.
        {"name": "linear_1000x1408_m5_noindex", "kind": "linear", "M": 5, "N": 1000, "K": 1408, "salient": 0.1,
         "index": False, "f32": True},
        # A layer's projections called one by one, one token: a program whose
        # layers call the linear function each for itself.
        {"name": "calls_4b_m1", "kind": "calls", "model": "qwen3-4b", "M": 1},
        # The decode step of the larger model, every projection in one call:
        # the headline workload.
        {"name": "step_8b_m1", "kind": "batch", "model": "qwen3-8b", "layers": 36, "M": 1},
        # Batched decode of a few sequences, and of the most that the decode
        # path takes (a third of the model: weights larger than L2).
        {"name": "layers12_8b_m4", "kind": "batch", "model": "qwen3-8b", "layers": 12, "M": 4},
        {"name": "layers12_8b_m16", "kind": "batch", "model": "qwen3-8b", "layers": 12, "M": 16},
        # The decode step in a model's order, each projection after the one
        # it depends on.
        {"name": "sequence_8b", "kind": "sequence", "model": "qwen3-8b", "layers": 36},
        # Prefill of a long prompt, one layer, and of a short odd one, one
        # projection.
        {"name": "prefill_layer_8b_m2048", "kind": "batch", "model": "qwen3-8b", "layers": 1, "M": 2048},
        {"name": "prefill_9728x2560_m200", "kind": "linear", "M": 200, "N": 9728, "K": 2560, "salient": 0.1,
         "index": True, "f32": False},
        # The element-wise four-mask form of one layer, one token.
        {"name": "elementwise_8b_m1", "kind": "elementwise", "model": "qwen3-8b", "M": 1},
        # Conversion: a dense projection to the packed format, and the codec
        # (pack and unpack) on a projection's trits.
        {"name": "ternarize_4096x12288", "kind": "ternarize", "N": 4096, "K": 12288},
        {"name": "codec_12288x4096", "kind": "codec", "N": 12288, "K": 4096},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["linear", "linear", "prefill", "calls", "batch", "batch", "sequence", "elementwise", "ternarize",
                       "codec"])
    model = rng.choice(sorted(LAYER))
    if kind == "linear":
        return {"kind": "linear", "M": _log(rng, 1, 16), "N": _log(rng, 128, 12288), "K": GROUP * _log(rng, 4, 96),
                "salient": rng.choice([0.0, 0.1, 0.1]), "index": rng.random() < 0.75, "f32": rng.random() < 0.3}
    if kind == "prefill":
        return {"kind": "linear", "M": _log(rng, 17, 2048), "N": _log(rng, 128, 9728), "K": GROUP * _log(rng, 8, 32),
                "salient": rng.choice([0.0, 0.1, 0.1]), "index": True, "f32": rng.random() < 0.3}
    if kind == "calls":
        return {"kind": "calls", "model": model, "M": _log(rng, 1, 16)}
    if kind == "batch":
        return {"kind": "batch", "model": model, "layers": _log(rng, 1, 12), "M": _log(rng, 1, 16)}
    if kind == "sequence":
        return {"kind": "sequence", "model": model, "layers": _log(rng, 1, 30)}
    if kind == "elementwise":
        return {"kind": "elementwise", "model": model, "M": rng.choice([1, 1, 2, 4])}
    return {"kind": kind, "N": _log(rng, 256, 4096), "K": GROUP * _log(rng, 8, 96)}


# ------------------------------------------------------------------ inputs
def _gen(seed, *ids):
    s = seed
    for i in ids:
        s = (s * 1000003 + i + 1) % (1 << 62)
    g = torch.Generator(device="cuda")
    g.manual_seed(s)
    return g


def _trits(g, N, K):
    u = torch.rand((N, K), generator=g, device="cuda", dtype=torch.float16)
    return (u >= 0.7).to(torch.int8) - (u < 0.3).to(torch.int8)


def _lognormal(g, *shape):
    return torch.exp(torch.randn(shape, generator=g, device="cuda") * 0.5 - 4.0).half()


def _params(g, *shape):
    return (torch.randn(shape, generator=g, device="cuda") * 1e-3).half()


def _x(seed, i, M, K):
    g = _gen(seed, 7, i)
    x = torch.randn((M, K), generator=g, device="cuda")
    big = torch.rand((K,), generator=g, device="cuda") < 1.0 / 256
    return torch.where(big, x * 10, x).half()


def _weight(seed, i, N, K, salient):
    """Codes and parameters of one projection: T1, T2, the salience map (dense
    and as words), s1, off and s2 in (row, group) order."""
    G = K // GROUP
    g = _gen(seed, 1, i)
    T1 = _trits(g, N, K)
    s1, off = _lognormal(g, N, G), _params(g, N, G)
    nnz = int(round(salient * N * G))
    order = torch.rand((N * G,), generator=g, device="cuda").argsort()
    dense = torch.zeros((N * G,), dtype=torch.bool, device="cuda")
    dense[order[:nnz]] = True
    dense = dense.view(N, G)
    words = torch.zeros((N, (G + 31) // 32 * 32), dtype=torch.int64, device="cuda")
    words[:, :G] = dense
    words = (words.view(N, -1, 32) << torch.arange(32, device="cuda")).sum(-1)
    sal = (words - ((words >> 31) << 32)).to(torch.int32)
    T2 = _trits(g, N, K).view(N, G, GROUP).mul_(dense[:, :, None]).view(N, K) if nnz else None
    s2 = _lognormal(g, max(nnz, 1))
    return T1, T2, dense, sal, s1, off, s2, nnz


def _packed(seed, i, N, K, salient, index=True):
    T1, T2, _, sal, s1, off, s2, _ = _weight(seed, i, N, K, salient)
    return tq.pack_weight(T1, T2, sal, s1, off, s2, check=False, index=index)


def _dense64(seed, i, N, K, salient):
    T1, T2, dense, _, s1, off, s2, nnz = _weight(seed, i, N, K, salient)
    G = K // GROUP
    W = T1.view(N, G, GROUP).double() * s1.double()[:, :, None] + off.double()[:, :, None]
    if nnz:
        S2 = torch.zeros((N, G), dtype=torch.float64, device="cuda")
        S2[dense] = s2.double()
        W += T2.view(N, G, GROUP).double() * S2[:, :, None]
    return W.view(N, K)


def _ew(seed, i, N, K):
    """Codes and parameters of one projection of the element-wise form."""
    g = _gen(seed, 2, i)
    u = torch.rand((N, K), generator=g, device="cuda")
    c0, c1, c2 = COVERAGE
    ids = ((u >= c0).to(torch.uint8) + (u >= c0 + c1).to(torch.uint8) + (u >= c0 + c1 + c2).to(torch.uint8))
    T0 = _trits(g, N, K)
    T1 = _trits(g, N, K) * (ids < 2)
    return T0, T1, ids, _params(g, N, 4), _lognormal(g, N, 4), _lognormal(g, N, 2)


def _dense_source(seed, N, K):
    """A dense projection to convert: Gaussian rows of their own scale and a
    small mean, one weight in a thousand eight times as large."""
    g = _gen(seed, 3)
    sd = torch.exp(torch.randn((N, 1), generator=g, device="cuda") * 0.25 + math.log(0.02))
    mean = torch.randn((N, 1), generator=g, device="cuda") * 1e-3
    W = torch.randn((N, K), generator=g, device="cuda") * sd + mean
    big = torch.rand((N, K), generator=g, device="cuda") < 1e-3
    return torch.where(big, W * 8, W).half()


def _shapes(case):
    if case["kind"] == "sequence":
        return FUSED[case["model"]] * case["layers"]
    return LAYER[case["model"]] * case.get("layers", 1)


def _outputs(case):
    """One buffer for every projection's result [M][N], one after the other as
    a decode loop lays them out, and the results as views of it."""
    M = case.get("M", 1)
    sizes = [M * N for N, _ in _shapes(case)]
    out = torch.empty(sum(sizes), dtype=torch.float16, device="cuda")
    return out, [y.view(M, -1) for y in out.split(sizes)]


def _nnz(N, K):
    return int(round(0.1 * N * (K // GROUP)))


# ------------------------------------------------------------------- a pass
def prepare(case, seed):
    kind = case["kind"]
    if kind == "linear":
        M, N, K = case["M"], case["N"], case["K"]
        w = _packed(seed, 0, N, K, case["salient"], case["index"])
        y = torch.empty((M, N), dtype=torch.float32 if case["f32"] else torch.float16, device="cuda")
        return {"kind": kind, "w": w, "x": _x(seed, 0, M, K), "y": y, "f32": case["f32"],
                "ws": tq.workspace(tq.tq_workspace_bytes(M, N, K), "cuda")}
    if kind in ("calls", "batch", "sequence"):
        M = case.get("M", 1)
        out, ys = _outputs(case)
        items = [(_packed(seed, i, N, K, 0.1), _x(seed, i, M, K), ys[i]) for i, (N, K) in enumerate(_shapes(case))]
        if kind == "calls":
            need = max(tq.tq_workspace_bytes(M, w.N, w.K) for w, _, _ in items)
            return {"kind": kind, "items": items, "out": out, "ws": tq.workspace(need, "cuda")}
        return {"kind": kind, "batch": tq.Batch(M, items), "out": out}
    if kind == "elementwise":
        M = case["M"]
        out, ys = _outputs(case)
        items = []
        for i, (N, K) in enumerate(_shapes(case)):
            w = tq.ew_index(tq.pack_ew_weight(*_ew(seed, i, N, K), check=False), check=False)
            items.append((w, _x(seed, i, M, K), ys[i]))
        return {"kind": kind, "batch": tq.EwBatch(M, items), "out": out}
    N, K = case["N"], case["K"]
    if kind == "ternarize":
        return {"kind": kind, "W": _dense_source(seed, N, K), "nnz": _nnz(N, K),
                "ws": tq.workspace(tq.tq_ternarize_workspace_bytes(N, K), "cuda")}
    T1, T2, _, sal, _, _, _, nnz = _weight(seed, 0, N, K, 0.1)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    rowptr = torch.empty(N + 1, dtype=torch.int32, device="cuda")
    tq.tq_salience_rowptr(N, K, sal, rowptr, status)
    return {"kind": kind, "N": N, "K": K, "T1": T1, "T2": T2, "sal": sal, "rowptr": rowptr, "status": status,
            "plane1": torch.empty((N, tq.tq_row_bytes(K)), dtype=torch.uint8, device="cuda"),
            "plane2": torch.empty((nnz, tq.TQ_GROUP_BYTES), dtype=torch.uint8, device="cuda"),
            "U1": torch.empty_like(T1), "U2": torch.empty_like(T2)}


def run(state):
    kind = state["kind"]
    if kind == "linear":
        fn = tq.tq_linear_f32out if state["f32"] else tq.tq_linear
        return fn(state["x"], state["w"], y=state["y"], ws=state["ws"])
    if kind == "calls":
        for w, x, y in state["items"]:
            tq.tq_linear(x, w, y=y, ws=state["ws"])
        return state["out"]
    if kind in ("batch", "sequence", "elementwise"):
        fn = {"batch": tq.tq_linear_batched, "sequence": tq.tq_linear_sequence,
              "elementwise": tq.tq_ew_linear_batched}[kind]
        fn(state["batch"])
        return state["out"]
    if kind == "ternarize":
        w = tq.ternarize(state["W"], state["nnz"], ws=state["ws"])
        return [w.plane1, w.salience, w.rowptr, w.plane2, w.scale1, w.offset, w.scale2, w.p2index]
    s = state
    tq.tq_pack(s["N"], s["K"], s["T1"], s["T2"], s["sal"], s["rowptr"], s["plane1"], s["plane2"], s["status"])
    tq.tq_unpack(s["N"], s["K"], s["plane1"], s["plane2"], s["sal"], s["rowptr"], s["U1"], s["U2"], s["status"])
    return [s["plane1"], s["plane2"], s["U1"], s["U2"], s["status"]]


# --------------------------------------------------------- least work, exact
def _packed_bytes(N, K, nnz):
    """Plane 1 with its row padding, scale and offset of every group, the
    salience words and row pointers, and the records with their scales."""
    G = K // GROUP
    return N * ((26 * G + 15) // 16 * 16 + 4 * G + 4 * ((G + 31) // 32)) + 4 * (N + 1) + 28 * nnz


def work(case):
    kind = case["kind"]
    if kind == "linear":
        M, N, K = case["M"], case["N"], case["K"]
        nnz = int(round(case["salient"] * N * (K // GROUP)))
        return {"bytes": _packed_bytes(N, K, nnz) + 2 * M * K + (4 if case["f32"] else 2) * M * N,
                "flops": 2 * M * (N * K + nnz * GROUP)}
    if kind in ("calls", "batch", "sequence"):
        M = case.get("M", 1)
        shapes = _shapes(case)
        return {"bytes": sum(_packed_bytes(N, K, _nnz(N, K)) + 2 * M * (N + K) for N, K in shapes),
                "flops": sum(2 * M * (N * K + _nnz(N, K) * GROUP) for N, K in shapes)}
    if kind == "elementwise":
        M = case["M"]
        second = COVERAGE[0] + COVERAGE[1]
        return {"bytes": int(sum(N * ((26 * (K // GROUP) + 15) // 16 * 16 + K / 4 + second * K / 5 + 4 + 20)
                                 + 2 * M * (N + K) for N, K in _shapes(case))),
                "flops": int(sum(2 * M * N * K * (1 + second) for N, K in _shapes(case)))}
    N, K = case["N"], case["K"]
    G, nnz = K // GROUP, _nnz(N, K)
    if kind == "ternarize":
        index = 4 * (G + 1) + 32 * (nnz + 8 * G)
        # per weight: 15 operations of the statistics, 5 of a block's planes, 11 more of a salient block's
        return {"bytes": 2 * N * K + _packed_bytes(N, K, nnz) + index, "flops": 20 * N * K + 11 * nnz * GROUP}
    codes = 2 * N * K  # T1 and T2, read once by pack and written once by unpack
    packed = N * ((26 * G + 15) // 16 * 16) + 26 * nnz
    return {"bytes": 2 * (codes + packed + N * 4 * ((G + 31) // 32) + 4 * (N + 1)), "flops": 20 * N * K}


def exact(case, seed):
    kind = case["kind"]
    if kind == "linear":
        M, N, K = case["M"], case["N"], case["K"]
        return _x(seed, 0, M, K).double() @ _dense64(seed, 0, N, K, case["salient"]).T
    if kind in ("calls", "batch", "sequence"):
        M = case.get("M", 1)
        return torch.cat([(_x(seed, i, M, K).double() @ _dense64(seed, i, N, K, 0.1).T).flatten()
                          for i, (N, K) in enumerate(_shapes(case))])
    if kind == "elementwise":
        out = []
        for i, (N, K) in enumerate(_shapes(case)):
            T0, T1, ids, mu, a0, a1 = _ew(seed, i, N, K)
            q = ids.long()
            a1 = torch.cat([a1.double(), torch.zeros((N, 2), dtype=torch.float64, device="cuda")], 1)
            W = mu.double().gather(1, q) + a0.double().gather(1, q) * T0 + a1.gather(1, q) * T1
            out.append((_x(seed, i, case["M"], K).double() @ W.T).flatten())
        return torch.cat(out)
    if kind == "ternarize":
        return _ternarized64(_dense_source(seed, case["N"], case["K"]), _nnz(case["N"], case["K"]))
    return None  # bytes and whole numbers


def _ternarized64(W, nnz, sweeps=4):
    """alpha0 and mu of every block (threshold 0.75 of the mean magnitude,
    least-squares scales, the residual's support where its energy is among the
    nnz largest, then the alternating sweeps).  The planes and the salience are
    whole numbers, and the places of the second scales follow from these."""
    N, K = W.shape
    w = W.double().view(-1, GROUP)

    def support(r):
        d = 0.75 * r.abs().mean(1, keepdim=True)
        return (r > d).double() - (r < -d).double()

    def scale(r, T):
        return (r * T).sum(1, keepdim=True) / T.abs().sum(1, keepdim=True).clamp_min(1)

    mu = w.mean(1, keepdim=True)
    c = w - mu
    T0 = support(c)
    a0 = scale(c, T0)
    r = c - a0 * T0
    top = r.square().sum(1).argsort(descending=True, stable=True)[:nnz]
    T1 = torch.zeros_like(w)
    T1[top] = support(r[top])
    a1 = scale(r, T1)
    for _ in range(sweeps):
        mu = (w - a0 * T0 - a1 * T1).mean(1, keepdim=True)
        a0 = scale(w - mu - a1 * T1, T0)
        a1 = scale(w - mu - a0 * T0, T1)
    G = K // GROUP
    return [None, None, None, None, a0.view(N, G), mu.view(N, G), None, None]

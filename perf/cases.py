"""The workloads whose speed this repository is judged by, as data and small
functions: what a program that trains or queries Forward-Forward nets calls,
through the public entry points of ``paper_2404_08573_gb300.ff``.

A case is a dict of plain values:

  kind    "ff"        steps of the FF net (``Net.train_step`` or, with
                      ``images``, ``Net.train_step_images``) on layer streams
          "po"        steps of the Performance-Optimized net (``PoNet``)
          "head"      softmax-head training (``Head.train_epoch``)
          "head_pred" softmax prediction (``Head.predict``)
          "predict"   goodness prediction over the 10 label overlays
          "adaptive"  AdaptiveNEG negative labels
  dims    layer widths, "784,2000,2000": input first
  prec    "bf16" (bf16 operands, fp32 accumulation and masters) or "fp32"
  n       rows: pairs per step ("ff"), rows per step ("po"), or rows per call
  steps   train steps per pass; ``tail``: rows of the last one (0: n)
  batch   rows per step of the head
  graph   the pass's steps captured once as a CUDA graph, as the benchmark's
          headline runs them; else one host call per step

A training pass returns the losses and every layer's updated weights, bias
and first moment (which holds the pass's gradients).  Training starts from a
mid-run state (Adam moments of the gradients' size, step 100): from a fresh
state the first update is lr * sign(g), which says little about g.
"""

from __future__ import annotations

import ctypes
import math

import torch

from paper_2404_08573_gb300 import ff

THETA, LR, HEAD_LR = 2.0, 1e-3, 1e-4
B1, B2, EPS = 0.9, 0.999, 1e-8
STEP0 = 100  # Adam steps taken before the pass


def _case(name, kind, dims, prec, n, steps=1, tail=0, batch=0, graph=False, images=False):
    return dict(name=name, kind=kind, dims=dims, prec=prec, n=n, steps=steps, tail=tail, batch=batch, graph=graph,
                images=images)


def listed():
    return [
        # the small exact-precision net, 16 steps of 64 pairs: launch latency and tiny GEMMs
        _case("ff_fp32_784-500x2_b64", "ff", "784,500,500", "fp32", 64, steps=16),
        # the paper's net at the paper's batch of 64: Adam's state traffic and latency
        _case("ff_bf16_784-2000x4_b64", "ff", "784,2000,2000,2000,2000", "bf16", 64, steps=16, graph=True, images=True),
        # the benchmark's epoch, its first and its ragged last batches
        _case("ff_bf16_784-2000x4_b1024", "ff", "784,2000,2000,2000,2000", "bf16", 1024, steps=8, tail=608, graph=True),
        # the paper's net in exact precision, a medium batch
        _case("ff_fp32_784-2000x4_b256", "ff", "784,2000,2000,2000,2000", "fp32", 256, steps=2),
        # the wide CIFAR-shaped net: the largest GEMMs
        _case("ff_bf16_3072-8192x2_b4096", "ff", "3072,8192,8192", "bf16", 4096, steps=2),
        # test-set evaluation
        _case("predict_bf16_784-2000x4_n10000", "predict", "784,2000,2000,2000,2000", "bf16", 10000),
        # an interactive query of a few samples
        _case("predict_bf16_784-2000x4_n8", "predict", "784,2000,2000,2000,2000", "bf16", 8),
        # validation in exact precision
        _case("predict_fp32_784-2000x4_n1000", "predict", "784,2000,2000,2000,2000", "fp32", 1000),
        # negatives for part of a training set, odd sizes
        _case("adaptive_bf16_784-1500x3_n4097", "adaptive", "784,1500,1500,1500", "bf16", 4097),
        # softmax-head training over two forward passes and a ragged last step
        _case("head_bf16_784-2000x4_n20000", "head", "784,2000,2000,2000,2000", "bf16", 20000, batch=1024),
        # softmax evaluation of a validation set
        _case("head_pred_bf16_784-2000x4_n1000", "head_pred", "784,2000,2000,2000,2000", "bf16", 1000),
        # Performance-Optimized training at the benchmark's batch
        _case("po_bf16_784-2000x4_b1024", "po", "784,2000,2000,2000,2000", "bf16", 1024, steps=8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the same ranges: 1 to 5 layers of 64 to 4096 units (multiples
    of 8, of 4, and odd), 1 to 20000 rows, all kinds."""
    while True:
        kind = rng.choice(["ff", "ff", "ff", "po", "head", "head_pred", "predict", "adaptive"])
        prec = rng.choice(["bf16", "bf16", "fp32"])
        first = rng.choice([784, 784, 3072, _log_int(rng, 64, 3072)])
        width = _log_int(rng, 64, 4096)
        width = max(width - width % rng.choice([8, 8, 4, 1]), 16)
        depth = rng.randint(1, 5)
        dims = [first] + [width if rng.random() < 0.8 else max(64, width // 2 + rng.randint(0, 9))
                          for _ in range(depth)]
        train = kind in ("ff", "po")
        n = _log_int(rng, 8, 2048) if train else _log_int(rng, 256 if kind == "head" else 1, 20000)
        steps = _log_int(rng, 1, 16) if train else 1
        tail = rng.randint(1, n) if train and rng.random() < 0.3 else 0
        batch = min(n, _log_int(rng, 32, 2048)) if kind == "head" else 0
        case = dict(kind=kind, dims=",".join(map(str, dims)), prec=prec, n=n, steps=steps, tail=tail, batch=batch,
                    graph=kind == "ff" and rng.random() < 0.5, images=kind == "ff" and rng.random() < 0.5)
        w = work(case)
        if kind == "predict" or kind == "adaptive":
            limit = 2e12 if prec == "bf16" else 2e11
        else:
            limit = 2e12 if prec == "bf16" else 4e10
        params = sum(k * m for k, m in zip(dims, dims[1:]))
        rounds = -(-n // batch) if batch else steps
        if w["flops"] <= limit and params * rounds <= 3e8:
            return case


# ------------------------------------------------------------------- inputs
def _dims(case):
    return [int(d) for d in case["dims"].split(",")]


def _gen(seed, what):
    return torch.Generator(device="cuda").manual_seed((int(seed) * 1000003 + what) % (1 << 62))


def _steps(case):
    """Rows (or pairs) of each train step."""
    s = [case["n"]] * case["steps"]
    if case["tail"]:
        s[-1] = case["tail"]
    return s


def _images(n, features, seed, what):
    """MNIST-shaped rows (80 % zeros, else U(0, 1)); CIFAR-shaped ones (3072
    features) are dense U(0, 1)."""
    g = _gen(seed, what)
    x = torch.rand(n, features, device="cuda", generator=g)
    if features != 3072:
        x *= torch.rand(n, features, device="cuda", generator=g) < 0.2
    return x


def _labels(n, seed, what):
    return torch.randint(0, 10, (n,), device="cuda", dtype=torch.int32, generator=_gen(seed, what))


def _wrong_labels(y, seed, what):
    off = torch.randint(1, 10, (y.shape[0],), device="cuda", dtype=torch.int32, generator=_gen(seed, what))
    return (y + off) % 10


def _layer_state(K, N, seed, k, train):
    """He-uniform W, a small bias; for training, Adam moments of the size of
    such a layer's gradients (a mean over pairs of h x / (K N)-sized terms)."""
    g = _gen(seed, 100 + k)
    st = {"W": (torch.rand(N, K, device="cuda", generator=g) * 2 - 1) * math.sqrt(6.0 / K),
          "b": (torch.rand(N, device="cuda", generator=g) * 2 - 1) * 0.02}
    if train:
        for name, shape, size in (("W", (N, K), 0.5 / K), ("b", (N,), 0.5 / math.sqrt(K))):
            st["m" + name] = torch.randn(shape, device="cuda", generator=g) * (0.2 * size)
            st["v" + name] = (torch.rand(shape, device="cuda", generator=g) + 0.5) * size ** 2
    return st


def _head_state(F, seed, k, train, scale):
    g = _gen(seed, 200 + k)
    st = {"V": torch.randn(10, F, device="cuda", generator=g) * scale,
          "c": torch.randn(10, device="cuda", generator=g) * 0.05}
    if train:
        for name, shape in (("V", (10, F)), ("c", (10,))):
            st["m" + name] = torch.randn(shape, device="cuda", generator=g) * 2e-4
            st["v" + name] = (torch.rand(shape, device="cuda", generator=g) + 0.5) * 1e-6
    return st


def _ptr(t):
    return None if t is None else ctypes.c_void_p(t.data_ptr())


def _ok(status):
    if status != 0:
        raise ff.FFError(status, "state copy")


def _set_layer(layer, st):
    _ok(ff.lib().ff_layer_set_state(layer.handle, *[_ptr(st.get(n)) for n in ("W", "b", "mW", "vW", "mb", "vb")],
                                    STEP0 if "mW" in st else 0))


def _set_head(head, st):
    _ok(ff.lib().ff_head_set_state(head._h, *[_ptr(st.get(n)) for n in ("V", "c", "mV", "vV", "mc", "vc")],
                                   STEP0 if "mV" in st else 0))


def _head_features(dims):
    return sum(dims[2:]) if len(dims) > 2 else dims[1]


def _data(case, seed):
    """The inputs of a pass: per train step (x, labels), or x (and labels)."""
    dims, kind = _dims(case), case["kind"]
    if kind == "ff":
        out = []
        for t, b in enumerate(_steps(case)):
            x = _images(b, dims[0], seed, 1000 + 4 * t)
            y = _labels(b, seed, 1001 + 4 * t)
            lab = torch.cat([y, _wrong_labels(y, seed, 1002 + 4 * t)])
            out.append((x if case["images"] else torch.cat([x, x]), lab))
        return out
    if kind == "po":
        return [(_images(b, dims[0], seed, 1000 + 4 * t), _labels(b, seed, 1001 + 4 * t))
                for t, b in enumerate(_steps(case))]
    return _images(case["n"], dims[0], seed, 1000), _labels(case["n"], seed, 1001)


def prepare(case, seed):
    dims, kind = _dims(case), case["kind"]
    L = len(dims) - 1
    train = kind in ("ff", "po")
    s = {"case": case, "dims": dims, "data": _data(case, seed)}
    rows = 2 * case["n"] if kind == "ff" else case["n"] if kind == "po" else 0
    s["layers"] = [ff.Layer(dims[k], dims[k + 1], prec=case["prec"], theta=THETA, lr=LR, max_rows=rows)
                   for k in range(L)]

    def set_states():
        for k, l in enumerate(s["layers"]):
            _set_layer(l, _layer_state(dims[k], dims[k + 1], seed, k, train))

    set_states()
    torch.cuda.synchronize()  # the states just set are temporaries of this function
    if train:
        s["state"] = [{"W": torch.empty(l.out_features, l.in_features, device="cuda"),
                       "b": torch.empty(l.out_features, device="cuda"),
                       "mW": torch.empty(l.out_features, l.in_features, device="cuda")} for l in s["layers"]]
        s["loss"] = torch.empty(case["steps"], L, device="cuda")
    if kind == "ff":
        s["net"] = ff.Net(s["layers"], max_B=case["n"])
        if case["graph"]:
            # warm up (workspaces), capture one pass, start from the same state again
            _net_steps(s, None)
            torch.cuda.synchronize()
            stream = torch.cuda.Stream()
            s["graph"] = torch.cuda.CUDAGraph()
            with torch.cuda.graph(s["graph"], stream=stream):
                _net_steps(s, stream)
            torch.cuda.synchronize()
            set_states()
    elif kind == "po":
        s["blocks"] = [ff.Head(d, lr=HEAD_LR, max_rows=case["n"]) for d in dims[1:]]
        s["head_state"] = []
        for k, h in enumerate(s["blocks"]):
            _set_head(h, _head_state(dims[k + 1], seed, k, True, 1.0))
            s["head_state"].append({"V": torch.empty(10, dims[k + 1], device="cuda"),
                                    "c": torch.empty(10, device="cuda")})
        s["net"] = ff.PoNet(s["layers"], s["blocks"], max_rows=case["n"])
    elif kind in ("head", "head_pred"):
        F = _head_features(dims)
        s["head"] = ff.Head(F, lr=HEAD_LR, max_rows=case["batch"])
        _set_head(s["head"], _head_state(F, seed, 0, kind == "head", 1.0))
        if kind == "head":
            s["loss"] = torch.empty(-(-case["n"] // case["batch"]), device="cuda")
            s["head_state"] = [{"V": torch.empty(10, F, device="cuda"), "c": torch.empty(10, device="cuda"),
                                "mV": torch.empty(10, F, device="cuda")}]
        else:
            s["pred"] = torch.empty(case["n"], dtype=torch.int32, device="cuda")
            s["logits"] = torch.empty(case["n"], 10, device="cuda")
    else:
        s["pred"] = torch.empty(case["n"], dtype=torch.int32, device="cuda")
        s["goodness"] = torch.empty(case["n"], 10, device="cuda")
    torch.cuda.synchronize()
    return s


def _net_steps(s, stream):
    net, loss = s["net"], s["loss"]
    step = net.train_step_images if s["case"]["images"] else net.train_step
    for t, (x, lab) in enumerate(s["data"]):
        step(x, lab, loss=loss[t], stream=stream)
    net.sync(stream)


def _read_layers(s):
    """Every layer's weights, bias and first moment into the program's own buffers."""
    for l, st in zip(s["layers"], s["state"]):
        _ok(ff.lib().ff_layer_get_state(l.handle, _ptr(st["W"]), _ptr(st["b"]), _ptr(st["mW"]), None, None, None,
                                        None))
    return s["state"]


def _read_heads(heads, states):
    for h, st in zip(heads, states):
        _ok(ff.lib().ff_head_get_state(h._h, _ptr(st["V"]), _ptr(st["c"]), _ptr(st.get("mV")), None, None, None, None))
    return states


def run(s):
    kind = s["case"]["kind"]
    if kind == "ff":
        if "graph" in s:
            s["graph"].replay()
        else:
            _net_steps(s, None)
        return {"loss": s["loss"], "layers": _read_layers(s)}
    if kind == "po":
        for t, (x, lab) in enumerate(s["data"]):
            s["net"].train_step(x, lab, loss=s["loss"][t])
        s["net"].sync()
        return {"loss": s["loss"], "layers": _read_layers(s), "blocks": _read_heads(s["blocks"], s["head_state"])}
    x, y = s["data"]
    if kind == "head":
        s["head"].train_epoch(s["layers"], x, y, s["case"]["batch"], loss=s["loss"])
        return {"loss": s["loss"], "head": _read_heads([s["head"]], s["head_state"])}
    if kind == "head_pred":
        s["head"].predict(s["layers"], x, pred=s["pred"], logits=s["logits"])
        return {"logits": s["logits"], "pred": s["pred"]}
    if kind == "adaptive":
        ff.adaptive_negatives(s["layers"], x, y, neg=s["pred"], goodness=s["goodness"])
    else:
        ff.predict(s["layers"], x, pred=s["pred"], goodness=s["goodness"])
    return {"goodness": s["goodness"], "pred": s["pred"]}


def work(case):
    """FLOPs of the matrix products; bytes: the inputs and outputs once, and
    per train step the parameters and both moments read and written (the big
    nets' state exceeds the caches)."""
    dims, kind = _dims(case), case["kind"]
    kn = [k * m for k, m in zip(dims, dims[1:])]
    params = sum(kn)
    wb = 2 if case["prec"] == "bf16" else 4
    if kind in ("ff", "po"):
        rows = sum(_steps(case))
        images = rows
        if kind == "ff":
            rows, images = 2 * rows, rows if case["images"] else 2 * rows
        return {"flops": 4.0 * rows * params, "bytes": 24.0 * params * case["steps"] + 4.0 * images * dims[0]}
    n = case["n"]
    if kind in ("head", "head_pred"):
        F = _head_features(dims)
        flops = 2.0 * n * params + (4.0 if kind == "head" else 2.0) * n * 10 * F
        nbytes = 4.0 * n * dims[0] + wb * params + 40.0 * F
        if kind == "head":
            nbytes += 240.0 * F * -(-n // case["batch"])
        else:
            nbytes += 44.0 * n
        return {"flops": flops, "bytes": nbytes}
    return {"flops": 2.0 * n * kn[0] + 20.0 * n * sum(kn[1:]), "bytes": 4.0 * n * dims[0] + wb * params + 44.0 * n}


def tolerance(case):
    """About four times the measured distance from ``exact``: fp32 2e-5
    (goodness; three TF32 products a term) and 1e-4 (a first moment after 16
    steps); bf16 operands 2e-4 (goodness), 2e-3 to 8e-3 (first moments,
    logits).  A unit at its kink, or a bf16 rounding that falls the other
    way, moves a single element by more than the norm: "max".  Labels whose
    scores tie within the rounding may differ."""
    if case["kind"] in ("predict", "adaptive"):
        return {"rel": 1e-3 if case["prec"] == "bf16" else 1e-4, "differ": 0.01}
    if case["prec"] == "bf16":
        return {"rel": 1e-2, "max": 0.5, "differ": 0.01}
    return {"rel": 4e-4, "max": 0.05, "differ": 0.01}


# ------------------------------------------------------- 64-bit restatement
def _overlay(x, labels):
    x = x.double().clone()
    if labels is None:
        x[:, :10] = 0.1
    else:
        x[:, :10] = torch.nn.functional.one_hot(labels.long(), 10).double()
    return x


def _unit(x):
    return x / torch.linalg.vector_norm(x, dim=1, keepdim=True).clamp_min(1e-12)


def _adam(p, m, v, g, t, lr):
    m.mul_(B1).add_(g, alpha=1 - B1)
    v.mul_(B2).addcmul_(g, g, value=1 - B2)
    p.sub_(lr * (m / (1 - B1 ** t)) / ((v / (1 - B2 ** t)).sqrt() + EPS))


def _double(st):
    return {k: v.double() for k, v in st.items()}


def _block_step(st, feats, labels, t):
    """Softmax cross-entropy of the linear block, its Adam update; returns the
    loss and the gradient at the features (weights before the update)."""
    z = feats @ st["V"].T + st["c"]
    lse = torch.logsumexp(z, 1)
    n = z.shape[0]
    loss = (lse - z[torch.arange(n, device="cuda"), labels.long()]).mean()
    dz = (torch.softmax(z, 1) - torch.nn.functional.one_hot(labels.long(), 10).double()) / n
    back = dz @ st["V"]
    _adam(st["V"], st["mV"], st["vV"], dz.T @ feats, t, HEAD_LR)
    _adam(st["c"], st["mc"], st["vc"], dz.sum(0), t, HEAD_LR)
    return loss, back


def _exact_train(case, seed):
    dims, kind = _dims(case), case["kind"]
    L = len(dims) - 1
    layers = [_double(_layer_state(dims[k], dims[k + 1], seed, k, True)) for k in range(L)]
    blocks = [_double(_head_state(d, seed, k, True, 1.0)) for k, d in enumerate(dims[1:])] if kind == "po" else []
    losses = torch.zeros(case["steps"], L, dtype=torch.float64, device="cuda")
    for t, (x, lab) in enumerate(_data(case, seed)):
        if kind == "ff":
            B = lab.shape[0] // 2
            a = _overlay(torch.cat([x, x]) if case["images"] else x, lab)
        else:
            a = _overlay(x, None)
        for k, st in enumerate(layers):
            xh = _unit(a)
            h = torch.relu(xh @ st["W"].T + st["b"])
            if kind == "ff":
                g = (h * h).sum(1)
                sign = torch.ones_like(g)
                sign[:B] = -1.0  # positive rows: softplus(theta - g)
                losses[t, k] = torch.nn.functional.softplus(sign * (g - THETA)).sum() / B
                dz = (sign * torch.sigmoid(sign * (g - THETA)) * (2.0 / B)).unsqueeze(1) * h
            else:
                losses[t, k], back = _block_step(blocks[k], h, lab, STEP0 + 1 + t)
                dz = back * (h > 0)
            _adam(st["W"], st["mW"], st["vW"], dz.T @ xh, STEP0 + 1 + t, LR)
            _adam(st["b"], st["mb"], st["vb"], dz.sum(0), STEP0 + 1 + t, LR)
            a = h
    out = {"loss": losses, "layers": [{n: st[n] for n in ("W", "b", "mW")} for st in layers]}
    if kind == "po":
        out["blocks"] = [{n: st[n] for n in ("V", "c")} for st in blocks]
    return out


def exact(case, seed):
    dims, kind = _dims(case), case["kind"]
    if work(case)["flops"] > 8e12:
        return None  # over about 20 seconds in 64 bits
    if kind in ("ff", "po"):
        return _exact_train(case, seed)
    x, y = _data(case, seed)
    layers = [_double(_layer_state(dims[k], dims[k + 1], seed, k, False)) for k in range(len(dims) - 1)]
    n = case["n"]
    if kind in ("head", "head_pred"):
        feats, a = [], _overlay(x, None)
        for k, st in enumerate(layers):
            a = torch.relu(_unit(a) @ st["W"].T + st["b"])
            if k >= 1 or len(layers) == 1:
                feats.append(_unit(a))
        feats = torch.cat(feats, 1)
        st = _double(_head_state(feats.shape[1], seed, 0, kind == "head", 1.0))
        if kind == "head_pred":
            z = feats @ st["V"].T + st["c"]
            return {"logits": z, "pred": None}
        losses = [_block_step(st, feats[r:r + case["batch"]], y[r:r + case["batch"]], STEP0 + 1 + i)[0]
                  for i, r in enumerate(range(0, n, case["batch"]))]
        return {"loss": torch.stack(losses), "head": [{k: st[k] for k in ("V", "c", "mV")}]}
    G = torch.zeros(n, 10, dtype=torch.float64, device="cuda")
    for c in range(10):
        a = _overlay(x, torch.full((n,), c, device="cuda"))
        for k, st in enumerate(layers):
            a = torch.relu(_unit(a) @ st["W"].T + st["b"])
            if k >= 1 or len(layers) == 1:
                G[:, c] += (a * a).sum(1)
    return {"goodness": G, "pred": None}

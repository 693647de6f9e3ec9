"""The measured cases: what a user of this framework has it do.

A training run alternates the forward product, the transposed product and an
update of each layer; the prox phase updates from the dense gradient (fused
with its GEMM, or as separate calls for a gradient the caller keeps and for
the adaptive methods), the debias phase from the gradient at the stored
entries; the trained network is then served. The cases are these calls at the
sizes of the workloads (the 784-300-100-10 MLP, LeNet-5, the 9216-4096-4096-1000
classifier head, the 4096 x 4096 sweep at 1-50% density and 1-1024 columns) and
two whole calls: LeNet-5 inference and a debias step of the classifier head.
Single-layer calls are issued one by one, as the eager training loop does.
"""

import math
from statistics import NormalDist

import numpy as np
import torch

from paper_1905_07931_gb300 import csrtrain as C
from paper_1905_07931_gb300 import infer, synth, train

ETA = 0.01       # step size of the prox phase (the workloads' value)
LAMBDA = 1e-4    # l1 weight of the workloads
STEP = 10        # step number of the adaptive methods' bias corrections


def listed():
    return [
        # the smallest call: the single FC layer 784 -> 300 (10%, 64 samples), forward with bias and ReLU
        dict(name="fwd_300x784_n64", op="forward", m=300, k=784, n=64, density=0.10, zipf=False),
        # serving one sample through the classifier head's first layer
        dict(name="fwd_4096x9216_n1", op="forward", m=4096, k=9216, n=1, density=0.05, zipf=False),
        # a hidden layer's products of one training step: forward, then transposed with the ReLU of the layer below
        dict(name="fwdbwd_4096_5pct_n256", op="forward_backward", m=4096, k=4096, n=256, density=0.05, zipf=False),
        # the same for a small batch on power-law rows at the sweep's 20%
        dict(name="fwdbwd_4096_zipf_20pct_n32", op="forward_backward", m=4096, k=4096, n=32, density=0.20, zipf=True),
        # the same for the sweep's densest layer and largest batch (early training, little compressed yet)
        dict(name="fwdbwd_4096_50pct_n1024", op="forward_backward", m=4096, k=4096, n=1024, density=0.50, zipf=False),
        # a layer's debias update: gradient at the stored entries, values and transposed copy updated
        dict(name="debias_4096_20pct_n256", op="debias", m=4096, k=4096, n=256, density=0.20, zipf=False),
        # the dense gradient in full float32 (the call's default precision), a ragged batch: the last of an epoch
        dict(name="grad_fp32_4096_n250", op="gradient", m=4096, k=4096, n=250),
        # the head's first layer in the prox phase: gradient + prox + compaction in one call, no transposed copy
        dict(name="gradprox_4096x9216_n256", op="gradient_prox", m=4096, k=9216, n=256, density=0.05, out_density=0.25,
             transposed=False),
        # prox + compaction of a gradient the caller holds, at the l1 weight that keeps the density, with the copy
        dict(name="prox_4096_5pct", op="prox", m=4096, k=4096, density=0.05, out_density=0.05, transposed=True,
             method="sgd"),
        # the same along the Prox-ADAM direction, a hidden layer at 20%
        dict(name="adam_1000x4096_20pct", op="prox", m=1000, k=4096, density=0.20, out_density=0.20, transposed=True,
             method="adam"),
        # whole call: LeNet-5 inference with compressed weights, a batch of 1000 images
        dict(name="infer_lenet_b1000", op="lenet", n=1000),
        # whole call: one debias step of the classifier head, batch 256, eager as the training loop runs it
        dict(name="step_head_debias_n256", op="head_debias", inputs=9216, hidden=4096, classes=1000, n=256),
    ]


def _size(rng, lo, hi):
    """A size between lo and hi, uniform in its logarithm; half of them rounded to whole multiples of 32 as layer
    widths mostly are, the others as they fall (odd ones among them)."""
    v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    if rng.random() < 0.5 and v >= 32:
        v = v // 32 * 32
    return max(lo, min(hi, v))


def draw(rng):
    op = rng.choice(["forward", "forward_backward", "forward_backward", "debias", "gradient", "gradient_prox", "prox",
                     "prox", "lenet", "head_debias"])
    if op == "lenet":
        return dict(op=op, n=_size(rng, 16, 2000))
    if op == "head_debias":
        return dict(op=op, inputs=_size(rng, 784, 9216), hidden=_size(rng, 300, 4096), classes=_size(rng, 10, 1000),
                    n=_size(rng, 16, 256))
    m, k, n = _size(rng, 64, 4096), _size(rng, 64, 9216), _size(rng, 1, 1024)
    if m * k > 4096 * 4096 and n > 256:
        n = 256          # no more than the largest listed case
    density = round(math.exp(rng.uniform(math.log(0.01), math.log(0.5))), 4)
    if op in ("forward", "forward_backward", "debias"):
        if m * k > 4096 * 4096:
            density = min(density, 0.2)
        return dict(op=op, m=m, k=k, n=n, density=density, zipf=rng.random() < 0.25)
    if op == "gradient":
        return dict(op=op, m=m, k=k, n=n)
    transposed = rng.random() < 0.5
    out = round(math.exp(rng.uniform(math.log(0.02), math.log(0.9))), 4)
    if op == "gradient_prox":
        return dict(op=op, m=m, k=k, n=n, density=density, out_density=out, transposed=transposed)
    return dict(op=op, m=m, k=k, density=density, out_density=out, transposed=transposed,
                method=rng.choice(["sgd", "sgd", "rmsprop", "adam"]))


# ---------------------------------------------------------------------------
# Inputs: plain dense tensors, made on the GPU from the seed
# ---------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda")


def _weights(g, m, k, density, zipf=False, seed=0):
    """Dense M x K weights, He normal on a Bernoulli mask, or on power-law row lengths over permuted rows."""
    score = torch.rand(m, k, generator=g, device="cuda")
    if zipf:
        lengths = synth.zipf_row_lengths(m, k, int(round(density * m * k)))
        lengths = np.random.default_rng(seed).permutation(lengths)
        order = score.argsort(dim=1).argsort(dim=1)
        mask = order < torch.from_numpy(lengths).cuda()[:, None]
    else:
        mask = score < density
    return torch.where(mask, _randn(g, m, k) * math.sqrt(2.0 / k), torch.zeros((), device="cuda"))


def _features(g, k, n):
    """ReLU features: about half of them zero."""
    return _randn(g, k, n).relu_()


def _upstream(g, m, n, scale):
    """A gradient that came through a ReLU: about half of it zero."""
    return _randn(g, m, n) * (torch.rand(m, n, generator=g, device="cuda") < 0.5) * scale


def _threshold(density):
    """The normal quantile that |N(0, 1)| exceeds with this probability."""
    return NormalDist().inv_cdf(1.0 - density / 2.0)


def _head_sizes(case):
    return [(case["hidden"], case["inputs"], 0.05), (case["hidden"], case["hidden"], 0.05),
            (case["classes"], case["hidden"], 0.15)]


def _inputs(case, seed):
    g = _gen(seed)
    op = case["op"]
    if op == "lenet":
        ws, bs = infer.lenet_weights(int(seed))
        return dict(W=ws, b=bs, images=torch.rand(case["n"], 28, 28, generator=g, device="cuda"))
    if op == "head_debias":
        W = [_weights(g, m, k, d) for m, k, d in _head_sizes(case)]
        return dict(W=W, b=[0.01 * _randn(g, w.shape[0]) for w in W],
                    x=_randn(g, case["inputs"], case["n"]).abs_(),
                    labels=torch.randint(0, case["classes"], (case["n"],), generator=g, device="cuda",
                                         dtype=torch.int32),
                    eta=1e-4)
    m, k, n = case["m"], case["k"], case.get("n", 1)
    s = dict(eta=ETA)
    if op != "gradient":
        s["W"] = _weights(g, m, k, case["density"], case.get("zipf", False), int(seed))
    if op in ("forward", "forward_backward", "debias"):
        s["x"] = _features(g, k, n)
        s["dy"] = _upstream(g, m, n, 1.0 / n)
        s["b"] = 0.01 * _randn(g, m)
    elif op == "gradient":
        s["x"], s["dy"] = _features(g, k, n), _upstream(g, m, n, 1.0 / n)
    elif op == "gradient_prox":
        # gradient entries are about N(0, scale^2 n / 4): the scale at which LAMBDA keeps out_density of them
        scale = LAMBDA / (_threshold(case["out_density"]) * math.sqrt(n / 4.0))
        s["x"], s["dy"] = _features(g, k, n), _upstream(g, m, n, scale)
        s["lam"] = LAMBDA
    else:
        s["G"] = _randn(g, m, k)
        s["lam"] = _threshold(case["out_density"])
        if case["method"] != "sgd":
            # a few steps into the run: moments of earlier gradients (the search direction is about N(0, 1) then)
            bc1, bc2 = (1.0 - 0.9 ** STEP, 1.0 - 0.999 ** STEP) if case["method"] == "adam" else (1.0, 1.0)
            s["v"] = bc2 * (0.5 + torch.rand(m, k, generator=g, device="cuda"))
            if case["method"] == "adam":
                s["m"] = bc1 * _randn(g, m, k)
    return s


# ---------------------------------------------------------------------------
# The framework's objects, and one pass
# ---------------------------------------------------------------------------

def prepare(case, seed):
    op = case["op"]
    s = _inputs(case, seed)
    s["op"] = op
    if op == "lenet":
        net = infer.Compressed(s["W"], s["b"], case["n"])
        net.x.copy_(s.pop("images").reshape(1, -1))
        return dict(op=op, net=net)
    if op == "head_debias":
        net = train.SparseNet(train.mlp_layers(3), [w.cpu().numpy() for w in s["W"]], [b.cpu().numpy() for b in s["b"]],
                              case["n"], (case["inputs"],))
        net.x_in.copy_(s["x"])
        net.labels.copy_(s["labels"])
        return dict(op=op, net=net, eta=s["eta"])
    m, k, n = case["m"], case["k"], case.get("n", 1)
    s["ws"] = C.Workspace(m, k, n)
    if op == "gradient":
        s["g"] = torch.empty(m, k, device="cuda")
        return s
    keep_copy = op in ("forward_backward", "debias")
    W = C.CSR(m, k, transposed=keep_copy)
    C.csr_from_dense(s["W"], W, s["ws"])
    s["W"] = W
    if op in ("forward", "forward_backward"):
        s["y"], s["dx"] = torch.empty(m, n, device="cuda"), torch.empty(k, n, device="cuda")
    elif op == "debias":
        s["g"] = torch.zeros(W.capacity, device="cuda")
    else:
        s["out"] = C.CSR(m, k, transposed=case["transposed"])
        s["scratch"] = None
        if op == "gradient_prox":
            s["scratch"] = torch.empty(m, k, device="cuda")
        else:
            s["method"] = case["method"]
    return s


def _csr(w):
    out = dict(row_ptr=w.row_ptr, col_idx=w.col_idx, val=w.val)
    if w.transposed:
        out.update(t_row_ptr=w.t_row_ptr, t_col_idx=w.t_col_idx, t_val=w.t_val, t_pos=w.t_pos)
    return out


def run(s):
    op = s["op"]
    if op == "lenet":
        s["net"].forward()
        return dict(logits=s["net"].logits)
    if op == "head_debias":
        net = s["net"]
        loss = net.step("debias", s["eta"], 0.0)
        out = dict(logits=net.logits, loss=loss)
        for i, L in enumerate(net.params):
            W = net.weights(i)
            out["val%d" % i], out["bias%d" % i] = W.val, L["b"]
            if W.transposed:
                out["t_val%d" % i] = W.t_val
        return out
    ws = s["ws"]
    if op == "gradient":
        C.weight_grad_dense(s["dy"], s["x"], s["g"], ws)
        return dict(g=s["g"])
    W = s["W"]
    if op == "forward":
        C.spmm_fwd_bias_act(W, s["x"], s["b"], True, s["y"], ws)
        return dict(y=s["y"])
    if op == "forward_backward":
        C.spmm_fwd_bias_act(W, s["x"], s["b"], True, s["y"], ws)
        C.spmm_bwd_t_relu(W, s["dy"], s["x"], s["dx"], ws)
        return dict(y=s["y"], dx=s["dx"])
    if op == "debias":
        C.weight_grad_sddmm(W, s["dy"], s["x"], s["g"], ws)
        C.debias_update(W, s["g"], s["eta"])
        return dict(g=s["g"], val=W.val, t_val=W.t_val)
    out = s["out"]
    if op == "gradient_prox":
        C.weight_grad_prox_update(W, s["dy"], s["x"], s["eta"], s["lam"], out, ws, g_scratch=s["scratch"])
        return _csr(out)
    if s["method"] == "sgd":
        C.prox_update_compact(W, s["G"], s["eta"], s["lam"], out, ws)
        return _csr(out)
    if s["method"] == "rmsprop":
        C.prox_rmsprop_update_compact(W, s["G"], s["v"], s["eta"], s["lam"], 0.9, 1e-8, out, ws)
        return dict(_csr(out), v=s["v"])
    C.prox_adam_update_compact(W, s["G"], s["m"], s["v"], STEP, s["eta"], s["lam"], 0.9, 0.999, 1e-8, out, ws)
    return dict(_csr(out), m=s["m"], v=s["v"])


# ---------------------------------------------------------------------------
# Work that the path cannot do without
# ---------------------------------------------------------------------------

def work(case):
    op = case["op"]
    if op == "lenet":
        taps = (158, 2101, 10804, 270)                  # stored weights of the four layers
        n = case["n"]
        flops = 2.0 * n * (taps[0] * 576 + taps[1] * 64 + taps[2] + taps[3])
        return dict(bytes=4.0 * n * (784 + 10) + 8.0 * sum(taps), flops=flops)
    if op == "head_debias":
        n, total, flops = case["n"], 0.0, 0.0
        for i, (m, k, d) in enumerate(_head_sizes(case)):
            nnz = d * m * k
            # the layer's columns, values read and written (both copies where there is one), its input and output
            total += nnz * (12.0 if i == 0 else 24.0) + 4.0 * n * (m + k)
            flops += 2.0 * nnz * n * (2 if i == 0 else 3)
        return dict(bytes=total, flops=flops)
    m, k, n = case["m"], case["k"], case.get("n", 1)
    nnz = case.get("density", 0.0) * m * k
    io = 4.0 * n * (m + k)
    if op == "forward":
        return dict(bytes=8.0 * nnz + 4.0 * (2 * m + 1) + io, flops=2.0 * nnz * n)
    if op == "forward_backward":
        return dict(bytes=16.0 * nnz + 4.0 * (2 * m + k + 2) + 2 * io, flops=4.0 * nnz * n)
    if op == "debias":
        # columns and positions read, values of both copies written, the old values read, the gradient written
        return dict(bytes=24.0 * nnz + 4.0 * (m + 1) + io, flops=2.0 * nnz * n + 2.0 * nnz)
    if op == "gradient":
        return dict(bytes=4.0 * m * k + io, flops=2.0 * m * k * n)
    # a stored weight is kept about as often as an unstored one, or always: near enough
    kept = case["out_density"] * m * k
    total = 8.0 * nnz + (8.0 + (12.0 if case["transposed"] else 0.0)) * kept + 8.0 * (m + 1)
    if case["transposed"]:
        total += 4.0 * (k + 1)
    if op == "gradient_prox":
        return dict(bytes=total + io, flops=2.0 * m * k * n)
    moments = {"sgd": 0, "rmsprop": 1, "adam": 2}[case["method"]]
    return dict(bytes=total + 4.0 * m * k * (1 + 2 * moments), flops=float((4 + 8 * moments) * m * k))


# ---------------------------------------------------------------------------
# The same in 64 bits, from plain torch
# ---------------------------------------------------------------------------

def _padded(v, size):
    """A CSR's values in a buffer of its capacity, zero past the stored entries."""
    return torch.nn.functional.pad(v, (0, size - v.numel()))


def exact(case, seed):
    op = case["op"]
    s = _inputs(case, seed)
    if op == "lenet":
        F = torch.nn.functional
        w = [torch.from_numpy(t).cuda().double() for t in s["W"]]
        b = [torch.from_numpy(t).cuda().double() for t in s["b"]]
        y = s["images"].double()[:, None]
        for i, ci in ((0, 1), (1, 20)):
            cols = F.unfold(y, 5)                       # samples x (c 5 5) x pixels
            side = int(math.isqrt(cols.shape[2]))
            y = (w[i] @ cols + b[i][:, None]).reshape(y.shape[0], -1, side, side)
            y = F.max_pool2d(y, 2)
        h = torch.relu(y.reshape(y.shape[0], 800) @ w[2].T + b[2])
        return dict(logits=(h @ w[3].T + b[3]).T.contiguous())
    if op == "head_debias":
        W, b, n, eta = [w.double() for w in s["W"]], [t.double() for t in s["b"]], case["n"], s["eta"]
        ys = [s["x"].double()]
        for i in range(3):
            y = W[i] @ ys[-1] + b[i][:, None]
            ys.append(torch.relu(y) if i < 2 else y)
        logp = torch.log_softmax(ys[3], 0)
        hot = torch.nn.functional.one_hot(s["labels"].long(), case["classes"]).T
        per = -(logp * hot).sum(0)
        d = (logp.exp() - hot) / n
        out = dict(logits=ys[3], loss=torch.cat([per.mean()[None], per]))
        for i in (2, 1, 0):
            mask = s["W"][i] != 0
            new = W[i] - eta * (d @ ys[i].T)
            out["val%d" % i], out["bias%d" % i] = _padded(new[mask], mask.numel()), b[i] - eta * d.sum(1)
            if i:
                out["t_val%d" % i] = _padded(new.T[mask.T], mask.numel())
                d = (W[i].T @ d) * (ys[i] > 0)
        return out
    if op == "gradient":
        return dict(g=s["dy"].double() @ s["x"].double().T)
    if op == "gradient_prox":
        return None      # which entries are kept follows the tensor cores' rounding of the gradient
    W = s["W"].double()
    if op in ("forward", "forward_backward"):
        out = dict(y=torch.relu(W @ s["x"].double() + s["b"].double()[:, None]))
        if op == "forward_backward":
            out["dx"] = (W.T @ s["dy"].double()) * (s["x"] > 0)
        return out
    if op == "debias":
        mask = s["W"] != 0
        G = s["dy"].double() @ s["x"].double().T
        new = W - s["eta"] * G
        size = mask.numel()
        return dict(g=_padded(G[mask], size), val=_padded(new[mask], size), t_val=_padded(new.T[mask.T], size))
    # prox: which entries are kept is a rule on float32 values (the header's); their values in 64 bits
    f32 = lambda v: float(np.float32(v))  # noqa: E731
    eta, lam, G = f32(s["eta"]), f32(s["lam"]), s["G"]
    d32, d64, extra = G, G.double(), {}
    if case["method"] != "sgd":
        B1, B2 = f32(0.9), f32(0.999 if case["method"] == "adam" else 0.9)
        for kind, r in ((torch.float32, f32), (torch.float64, float)):
            c = lambda v: torch.tensor(r(v), dtype=kind, device="cuda")  # noqa: E731
            g = G.to(kind)
            v = c(B2) * s["v"].to(kind) + c(1.0 - B2) * (g * g)
            eps = c(f32(1e-8))
            if case["method"] == "adam":
                mm = c(B1) * s["m"].to(kind) + c(1.0 - B1) * g
                d = (mm / c(1.0 - B1 ** STEP)) / ((v / c(1.0 - B2 ** STEP)).sqrt() + eps)
                extra = dict(m=mm, v=v)
            else:
                d = g / (v.sqrt() + eps)
                extra = dict(v=v)
            if kind == torch.float32:
                d32 = d
        d64 = d
    thr = np.float32(eta) * np.float32(lam)
    z = s["W"] - d32 * eta
    keep = z.abs() > float(thr)
    z = W - d64 * eta
    new = z - torch.copysign(torch.full_like(z, eta * lam), z)
    size = case["m"] * case["k"]
    out = dict(row_ptr=None, col_idx=None, val=_padded(new[keep], size))
    if case["transposed"]:
        out.update(t_row_ptr=None, t_col_idx=None, t_val=_padded(new.T[keep.T], size), t_pos=None)
    return dict(out, **extra)

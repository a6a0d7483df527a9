"""Timed cases of the library: the calls that a training loop makes, over the sizes it makes them at.

A training loop that uses this library does the following things, and each of them is a `kind` here:

  step     fira.step over all 2-D weights of a model (Fira.step), every iteration;
  single   the same step of one matrix without caller-provided buffers (fira_step_single_noalloc);
  refresh  a new projection for every matrix from its gradient (Fira.refresh_projection), every T steps;
  dense    plain Adam over what is not projected: embedding, output head, norm gains (adam_dense);
  host     the step with weights and gradients in page-locked host memory (Fira.step_host).

A model is a list of layers with four hidden x hidden, two hidden x mlp and one mlp x hidden weights
(the shape lists of paper_2410_01623_b200/workloads.py), or one hidden x mlp matrix when layers = 0.
Gradients are Gaussian with one log-normal scale per column, in some models with 1 % of the columns
twenty times larger; weights are N(0, 0.02^2); the moments are those of a run under way (no matrix is
on its first step), and the remembered norm is such that the limiter acts on one matrix in eight.
"""
from __future__ import annotations

import ctypes
import math

import torch

from paper_2410_01623_b200 import binding as fb
from paper_2410_01623_b200.workloads import llama_shapes

#: Options of a step beside the default one: flags of the library.
OPTIONS = {
    "": 0,
    "padded": fb.FLAG_ROW_PADDING_WRITABLE,    # rows padded to 8 elements by the caller
    "lowrank_alpha": fb.FLAG_ALPHA_LOWRANK_ONLY,
    "galore": fb.FLAG_NO_RESIDUAL,             # the ablations of the method and the other base optimizers
    "matrix_scaling": fb.FLAG_MATRIX_SCALING,
    "no_scaling": fb.FLAG_NO_SCALING,
    "only_scaling": fb.FLAG_ONLY_SCALING,
    "rmsprop": fb.FLAG_PSI_RMSPROP,
    "adagrad": fb.FLAG_PSI_ADAGRAD,
}
TORCH = {"f32": torch.float32, "bf16": torch.bfloat16}
SIZE = {"f32": 4, "bf16": 2}
ROUNDS = 4                                     # rounds of the refresh (the library's default)


def _model(kind, layers, hidden, mlp, rank, dtype, option="", outliers=False):
    return dict(kind=kind, layers=layers, hidden=hidden, mlp=mlp, rank=rank, dtype=dtype, option=option,
                outliers=outliers)


def listed():
    cases = [
        # The smallest calls: one 512 x 1376 matrix of the smallest model.  Launches and their latency count.
        ("single_512x1376_f32", _model("single", 0, 512, 1376, 128, "f32")),
        ("step_512x1376_f32", _model("step", 0, 512, 1376, 128, "f32")),
        # All weights of the smallest model in fp32 (8 layers, rank a quarter of the hidden size).
        ("step_8x512_f32", _model("step", 8, 512, 1376, 128, "f32")),
        # A small bf16 model whose width and rank fit no tile: ragged rows, odd leading dimensions.
        ("step_4x640_ragged_bf16", _model("step", 4, 640, 1707, 100, "bf16")),
        # The three bf16 models: r = 256 (short products, memory bound), r = 512 with an odd MLP width
        # (rows that start on no 16-byte boundary) and outlier columns, r = 1024 (the largest).
        ("step_24x1024_bf16", _model("step", 24, 1024, 2736, 256, "bf16")),
        ("step_24x2048_bf16", _model("step", 24, 2048, 5461, 512, "bf16", "", True)),
        ("step_32x4096_bf16", _model("step", 32, 4096, 11008, 1024, "bf16")),
        # The projection refresh of the smallest (fp32), the odd-width and the largest model.
        ("refresh_8x512_f32", _model("refresh", 8, 512, 1376, 128, "f32")),
        ("refresh_24x2048_bf16", _model("refresh", 24, 2048, 5461, 512, "bf16", "", True)),
        ("refresh_32x4096_bf16", _model("refresh", 32, 4096, 11008, 1024, "bf16")),
        # Embedding, head and 49 norm gains of the 24-layer model with hidden size 1024.
        ("dense_24x1024_bf16", dict(kind="dense", layers=24, hidden=1024, vocab=32000, dtype="bf16")),
        # Offloaded weights and gradients: the smallest model stepped from host memory.
        ("host_8x512_f32", _model("host", 8, 512, 1376, 128, "f32")),
    ]
    return [dict(name=name, **case) for name, case in cases]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _near(rng, x, multiple):
    """x itself or, as often, the multiple nearest to it."""
    return x if rng.random() < 0.5 else max(multiple, x // multiple * multiple)


def draw(rng):
    kind = rng.choices(["step", "refresh", "dense", "single", "host"], [10, 4, 2, 2, 1])[0]
    if kind == "dense":
        return dict(kind="dense", layers=_log(rng, 1, 32), hidden=_near(rng, _log(rng, 96, 4096), 64),
                    vocab=_near(rng, _log(rng, 50, 32000), 64), dtype=rng.choice(["f32", "bf16"]))
    if kind == "single":                       # max(m, n) * r up to the built-in array's limit
        hidden = _near(rng, _log(rng, 64, 768), 32)
        mlp = int(hidden * rng.uniform(1.0, 3.0))
        rank = min(max(8, int(hidden * rng.uniform(0.1, 0.4))), 900_000 // mlp)
        return _model("single", 0, *((hidden, mlp) if rng.random() < 0.5 else (mlp, hidden)), rank,
                      rng.choice(["f32", "f32", "bf16"]))
    if kind == "host" or rng.random() < 0.4:   # fp32, any width and rank
        hidden = _near(rng, _log(rng, 128, 1024), 64)
        dtype, layers = "f32", _log(rng, 1, 8)
    else:                                      # bf16: small models of any width and rank, large ones of the usual ones
        hidden = _log(rng, 256, 4096)
        hidden = _near(rng, hidden, 64) if hidden < 1024 else hidden // 128 * 128
        dtype, layers = "bf16", _log(rng, 1, 24)
    layers = max(1, min(layers, 8 * 4096 * 4096 // (hidden * hidden)))
    mlp = _near(rng, int(hidden * rng.uniform(2.0, 3.5)), 16)
    rank = max(8, int(hidden * rng.uniform(0.15, 0.35)))
    rank = _near(rng, rank, 128) if dtype == "bf16" and 512 <= hidden < 1024 else max(128, rank // 128 * 128) if hidden >= 1024 else rank
    option = ""
    if kind == "step" and rng.random() < 0.4:
        option = rng.choice(sorted(o for o in OPTIONS if o and (dtype == "bf16" or o != "padded")))
    if kind == "step" and rng.random() < 0.15:
        layers = 0
    return _model(kind, layers, hidden, mlp, rank, dtype, option, rng.random() < 0.2)


# ------------------------------------------------------------------------------------------ inputs
def _shapes(case):
    if case["layers"] == 0:
        return ((case["hidden"], case["mlp"]),)
    return llama_shapes(case["layers"], case["hidden"], case["mlp"])


def _pitch(case, n):
    return (n + 7) // 8 * 8 if case["option"] == "padded" else n


class _Group:
    """The matrices of one shape behind one another in one buffer (each starts on a 256-byte boundary),
    so that a list of any length comes back as a few tensors."""

    def __init__(self, case, shapes, on_host=False):
        self.buffers, self.views = [], [None] * len(shapes)
        for shape in sorted(set(shapes)):
            where = [i for i, s in enumerate(shapes) if s == shape]
            m, n = shape
            ld = _pitch(case, n)
            stride = (m * ld + 127) // 128 * 128
            kw = dict(pin_memory=True) if on_host else dict(device="cuda")
            buf = torch.zeros(len(where), stride, dtype=TORCH[case["dtype"]], **kw)
            self.buffers.append((buf, shape, ld))
            for k, i in enumerate(where):
                self.views[i] = buf[k, :m * ld].view(m, ld)[:, :n]

    def outputs(self):
        return [buf[:, :m * ld].unflatten(1, (m, ld))[..., :n] for buf, (m, n), ld in self.buffers]


def _column_scale(case, n, gen):
    c = torch.exp(torch.randn(n, generator=gen, device="cuda"))
    if case["outliers"]:
        c = torch.where(torch.rand(n, generator=gen, device="cuda") < 0.01, 20.0 * c, c)
    return c


def _weights_and_gradients(case, shapes, gen):
    W, G = _Group(case, shapes), _Group(case, shapes)
    scales = []
    for i, (m, n) in enumerate(shapes):
        W.views[i].copy_(torch.randn(m, n, generator=gen, device="cuda").mul_(0.02))
        scales.append(_column_scale(case, n, gen))
        G.views[i].copy_(torch.randn(m, n, generator=gen, device="cuda").mul_(scales[i]))
    return W, G, scales


def _bases(case, shapes, gen):
    """One orthonormal basis per projected extent, shared by the matrices that have it."""
    out = {}
    for d in sorted({min(s) for s in shapes}):
        q = torch.linalg.qr(torch.randn(d, case["rank"], generator=gen, device="cuda"))[0]
        out[d] = q.to(TORCH[case["dtype"]]).contiguous()
    return out


def _moments(case, shape, scale, gen):
    """M, V (l x r) after 100 steps, and about the norm of the scaled residual that the next step finds."""
    m, n = shape
    l, d, r = max(m, n), min(m, n), case["rank"]
    rms = scale.square().mean().sqrt()
    # R of a column of G has its column's scale; R of a row has the scale that all columns give it
    c = scale[:, None] if m <= n else rms
    M = torch.randn(l, r, generator=gen, device="cuda").mul_(0.25 * c)
    V = torch.rand(l, r, generator=gen, device="cuda").add_(0.5).mul_(c * c)
    V.mul_(100.0 if case["option"] == "adagrad" else 0.1)
    size = {"rmsprop": 3.0, "adagrad": 0.1}.get(case["option"], 0.25)       # of an entry of N
    if case["option"] in ("rmsprop", "adagrad"):
        M.zero_()
    if case["option"] == "no_scaling":
        size = float(rms)
    return M, V, size * math.sqrt(l * max(d - r, 1))


def _context(case, shapes, gen, scales=None):
    hp = fb.make_hparams(lr=1e-2, alpha=0.25, gamma=1.01, flags=OPTIONS[case["option"]])
    lds = [_pitch(case, n) for _, n in shapes]
    f = fb.Fira(shapes, case["rank"], TORCH[case["dtype"]], hp, "cuda", lds=lds)
    if scales is not None:
        bases = _bases(case, shapes, gen)
        for i, shape in enumerate(shapes):
            f.set_projection(i, bases[min(shape)])
            M, V, norm = _moments(case, shape, scales[i], gen)
            f.set_state(i, M, V, norm * (0.5 if i % 8 == 7 else 4.0), 100)
    return f


def _state_sections(case, shapes, f):
    """Views of the state buffer, whose sections (projection, M, V, scalars; each padded to 256 bytes)
    follow one another matrix by matrix: a section of the same matrix of all layers is one view."""
    per_layer = 1 if case["layers"] == 0 else 7
    es, r = SIZE[case["dtype"]], case["rank"]
    pad = lambda b: (b + 255) // 256 * 256                                              # noqa: E731
    at, sections = 0, []
    for m, n in shapes[:per_layer]:
        l, d = max(m, n), min(m, n)
        for what, rows, size, dtype in (("P", d, es, TORCH[case["dtype"]]), ("M", l, 4, torch.float32),
                                        ("V", l, 4, torch.float32)):
            sections.append((what, at, rows, dtype))
            at += pad(rows * r * size)
        at += pad(32)
    layers = len(shapes) // per_layer
    out = {"P": [], "M": [], "V": []}
    for what, start, rows, dtype in sections:
        flat = f.state.view(dtype)
        size = flat.element_size()
        out[what].append(flat.as_strided((layers, rows, r), (at // size, r, 1), start // size))
    return out


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    kind = case["kind"]
    if kind == "dense":
        h = case["hidden"]
        sizes = [case["vocab"] * h] * 2 + [h] * (2 * case["layers"] + 1)
        starts, total = [], 0
        for s in sizes:
            starts.append(total)
            total += (s + 127) // 128 * 128
        dt = TORCH[case["dtype"]]
        flat = [torch.randn(total, generator=gen, device="cuda").mul_(0.02).to(dt),
                torch.randn(total, generator=gen, device="cuda").to(dt),
                torch.randn(total, generator=gen, device="cuda").mul_(0.3),
                torch.rand(total, generator=gen, device="cuda").add_(0.5)]
        lists = [[x[a:a + s] for a, s in zip(starts, sizes)] for x in flat]
        return dict(kind=kind, hp=fb.make_hparams(lr=1e-2), lists=lists, t=100, out=[flat[0], flat[2], flat[3]])
    shapes = _shapes(case)
    W, G, scales = _weights_and_gradients(case, shapes, gen)
    if kind == "single":
        (m, n), r = shapes[0], case["rank"]
        M, V, norm = _moments(case, shapes[0], scales[0], gen)
        P = _bases(case, shapes, gen)[min(m, n)]
        prev, t = torch.full((1,), 4.0 * norm, device="cuda"), torch.full((1,), 100, dtype=torch.int64, device="cuda")
        args = (ctypes.byref(fb.make_hparams(lr=1e-2)),
                ctypes.byref(fb.MatrixDesc(m, n, r, fb.FIRA_BF16 if case["dtype"] == "bf16" else fb.FIRA_F32, 0)),
                W.views[0].data_ptr(), G.views[0].data_ptr(), P.data_ptr(), M.data_ptr(), V.data_ptr(),
                prev.data_ptr(), t.data_ptr(), -1.0, torch.cuda.current_stream().cuda_stream)
        return dict(kind=kind, args=args, keep=(W, G, P), out=[W.views[0], M, V, prev])
    if kind == "refresh":
        f = _context(case, shapes, gen)
        return dict(kind=kind, f=f, G=G.views, out=_state_sections(case, shapes, f)["P"])
    f = _context(case, shapes, gen, scales)
    sections = _state_sections(case, shapes, f)
    moments = sections["V"] if case["option"] in ("rmsprop", "adagrad") else sections["M"] + sections["V"]
    if kind == "host":
        Wh, Gh = _Group(case, shapes, on_host=True), _Group(case, shapes, on_host=True)
        for host, dev in ((Wh, W), (Gh, G)):
            for (h, _, _), (x, _, _) in zip(host.buffers, dev.buffers):
                h.copy_(x)
        staging = torch.empty(f.staging_bytes(), dtype=torch.uint8, device="cuda")
        return dict(kind=kind, f=f, W=Wh.views, G=Gh.views, staging=staging, out=Wh.outputs() + moments)
    return dict(kind=kind, f=f, W=W.views, G=G.views, out=W.outputs() + moments)


def run(state):
    kind = state["kind"]
    if kind == "step":
        state["f"].step(state["W"], state["G"])
    elif kind == "refresh":
        state["f"].refresh_projection(state["G"], seed=1)
    elif kind == "dense":
        fb.adam_dense(state["hp"], *state["lists"], state["t"])
        state["t"] += 1
    elif kind == "single":
        fb.check(fb.lib().fira_step_single_noalloc(*state["args"]))
    else:
        state["f"].step_host(state["W"], state["G"], state["staging"])
    return state["out"]


def work(case):
    es = SIZE[case["dtype"]]
    if case["kind"] == "dense":
        n = 2 * case["vocab"] * case["hidden"] + (2 * case["layers"] + 1) * case["hidden"]
        return {"bytes": n * (3 * es + 16), "flops": 12 * n}
    r, nbytes, flops = case["rank"], 0, 0
    moments = {"rmsprop": 8, "adagrad": 8}.get(case.get("option"), 16)      # M is left alone by these
    for m, n in _shapes(case):
        l, d = max(m, n), min(m, n)
        if case["kind"] == "refresh":          # G in, basis out; 2 rounds + 1 products with G
            nbytes += es * (m * n + d * r)
            flops += (2 * ROUNDS + 1) * 2 * m * n * r
        else:                                  # G and W in, W out, moments in and out, basis in; two products
            nbytes += 3 * es * m * n + moments * l * r + es * d * r
            flops += (2 if case.get("option") == "only_scaling" else 4) * m * n * r
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    if case["dtype"] == "f32":
        return {"rel": 1e-5}                   # sums in fp32, the refreshed basis among them
    if case["kind"] == "refresh":
        # The iterate is rounded to bf16 before all but the last products: two correct roundings of it
        # leave bases that differ by 1.3e-2 to 1.7e-2, in all columns alike.
        return {"rel": 2e-2}
    return {"rel": 1e-2}

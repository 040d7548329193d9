"""What is timed: optimizer steps and the calls around them, through the package's public class ``DesLoc``.

A case says which call a training program makes (``call``), for which optimizer, worker count, tensor list, gradient type,
sync periods, buffer layout and options.  ``listed()`` are fixed cases, ``draw()`` gives others of the same ranges, ``prepare()``
builds what the program has in hand before the call -- M replicas of x, u, v in the middle of a run, one set of gradients, the
``DesLoc`` object -- ``run()`` makes the call once and returns every array that it updates.

Tensor lists are Llama-style (embedding, per block q k v o gate up down and two norms, final norm) or one tensor of ``n``
elements.  ``align`` is the layout of the buffers: 1 or 4 = the tensors follow one another in a flat buffer per worker and array
(packed, or each start rounded up to 4 elements); 0 = every tensor an allocation of its own, that is on a 512-byte boundary,
gradients included.  ``fresh`` = the program hands over nested lists of tensors at every step; otherwise it reuses
its gradient buffers and has bound them once.
"""
import math

import numpy as np
import torch

import paper_2505_22549_b200 as desloc

BASE = dict(call="step", opt="adam", M=4, n=0, layers=0, width=0, kv=0, ffn=0, vocab=0, grads="bf16", heavy=False,
            Kx=16, Ku=32, Kv=64, beta2=0.999, eps=1e-8, rho=0.0, wd=0.0, post=False, align=4, fresh=False)
SMALL = 4096                                                              # parameters of the smallest problem
MODEL_135M = dict(layers=30, width=576, kv=192, ffn=1536, vocab=49152)    # 134.5 M parameters, 272 tensors
MODEL_360M = dict(layers=32, width=960, kv=320, ffn=2560, vocab=49152)    # 361.8 M parameters, 290 tensors
MODEL_25M = dict(layers=3, width=768, kv=256, ffn=2048, vocab=8192)       # 25 M parameters, 29 tensors
MODEL_5M = dict(layers=4, width=256, kv=128, ffn=704, vocab=8192)         # 5 M parameters, 38 tensors
MODEL_MINI = dict(layers=2, width=72, kv=24, ffn=200, vocab=1031)         # 0.2 M parameters, 21 tensors, ragged sizes


def _case(name, **kw):
    return dict(BASE, name=name, **kw)


def listed():
    return [
        # one small tensor, two workers, fp32 gradients: pure latency of a call
        _case("adam_4096_m2", M=2, n=SMALL, grads="f32", Kx=4, Ku=8, Kv=16),
        # the same problem as launch-bound programs run it: a window of lcm(K) = 16 steps in a CUDA graph
        _case("graph_window_4096_m2", call="graph", M=2, n=SMALL, grads="f32", Kx=4, Ku=8, Kv=16),
        # the two-parameter toy problem with 256 workers, each handing over its own gradient tensor
        _case("toy_m256", M=256, n=2, grads="f32", Kx=192, Ku=192, Kv=692, align=1, fresh=True),
        # a tiny model with ragged tensors in packed buffers, nested gradient lists at every step
        _case("mini_packed_m4", **MODEL_MINI, Kx=4, Ku=8, Kv=16, align=1, fresh=True),
        # a small model with one allocation per tensor, autograd's fresh gradients at every step
        _case("adam_5m_m4", **MODEL_5M, align=0, fresh=True),
        # the 135 M-parameter model, four workers, desynced periods
        _case("adam_135m_m4", **MODEL_135M),
        # the same with norm-based clipping in front (the language-model runs), fp32 gradients
        _case("normclip_135m_m4", call="normclip", **MODEL_135M, grads="f32"),
        # eight workers, ADOPT with both clips and heavy-tailed gradients: the largest
        _case("adopt_360m_m8", opt="adopt", M=8, **MODEL_360M, heavy=True, Kx=32, Ku=64, Kv=128, beta2=0.9999, eps=1e-6,
              rho=1.0),
        # momentum SGD that averages everything at every step (the data-parallel baseline)
        _case("sgdm_360m_m8_ddp", opt="sgdm", M=8, **MODEL_360M, heavy=True, Kx=1, Ku=1, Kv=1),
        # sixteen workers, everything averaged at every step
        _case("adam_25m_m16_ddp", M=16, **MODEL_25M, Kx=1, Ku=1, Kv=1),
        # a monitored step: norms of gradient, parameters and update per tensor, rate of change of u since a snapshot
        _case("monitor_135m_m4", call="monitor", **MODEL_135M, wd=0.1),
        # gradients that arrive in pinned host memory
        _case("host_25m_m4", call="host", **MODEL_25M),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    call = rng.choices(["step", "normclip", "monitor", "host", "graph"], [60, 15, 10, 8, 7])[0]
    opt = rng.choices(["adam", "adopt", "sgdm"], [5, 3, 3])[0]
    M = rng.choices([1, 2, 3, 4, 5, 6, 7, 8, 9, 12, 16, 24], [1, 4, 2, 6, 2, 2, 1, 5, 1, 2, 2, 1])[0]
    grads = rng.choices(["bf16", "f32"], [7, 3])[0]
    c = dict(BASE, call=call, opt=opt, M=M, grads=grads, heavy=rng.random() < 0.3)
    # no more bytes than the largest listed case, host copies and graph windows far fewer
    largest = 361_821_120 * 8 * 26
    most = largest / {"step": 1, "normclip": 1.2, "monitor": 1.4, "host": 40, "graph": 400}[call] / (M * _step_bytes(c))
    params = _log_uniform(rng, SMALL, min(most, 600e6))
    if params < 50_000 and rng.random() < 0.5:
        c["n"] = max(1, int(params)) | (1 if rng.random() < 0.5 else 0)
    else:
        # a model of about that size: vocab and depth grow with the width, odd sizes among them
        c["layers"] = rng.randint(1, 6) if params < 20e6 else rng.randint(4, 32)
        share = rng.uniform(0.1, 0.5)                               # of the embedding
        width = math.sqrt(params * (1 - share) / (c["layers"] * 10.67))
        unit = rng.choice([1, 1, 4, 8, 64])
        c["width"] = max(4, int(width) // unit * unit)
        c["kv"] = max(1, c["width"] // rng.choice([1, 3, 4]))
        c["ffn"] = max(2, int(c["width"] * 8 / 3) // unit * unit)
        c["vocab"] = max(1, int(params * share / c["width"]))
    K = rng.choice([1, 2, 4, 16, 32, 64])
    c["Kx"], c["Ku"], c["Kv"] = K, K * rng.choice([1, 2, 4]), K * rng.choice([1, 2, 4, 16])
    if call == "graph":
        c["Kx"], c["Ku"], c["Kv"] = 4, 8, 16
        if M * len(_sizes(c)) > 32:                                 # what a graph takes without a table of pointers
            c.update(layers=0, n=max(1, int(params)))
            c["M"] = min(M, 32)
    c["rho"] = rng.choice([0.0, 0.0, 1.0])
    c["wd"] = rng.choice([0.0, 0.1])
    c["post"] = rng.random() < 0.12
    c["align"] = rng.choice([0, 1, 4])
    c["fresh"] = rng.random() < 0.5
    if opt == "adopt":
        c["beta2"], c["eps"] = 0.9999, 1e-6
    return c


def _sizes(c):
    """Element counts of the tensor list."""
    if not c["layers"]:
        return [c["n"]]
    w, kv, f = c["width"], c["kv"], c["ffn"]
    return [c["vocab"] * w] + [w * w, w * kv, w * kv, w * w, f * w, f * w, w * f, w, w] * c["layers"] + [w]


def _offsets(sizes, unit):
    offs, pos = [], 0
    for n in sizes:
        pos = -(-pos // unit) * unit
        offs.append(pos)
        pos += n
    return offs, pos


def _step_bytes(c):
    """Per worker and parameter: the gradient, and every state array in and out."""
    return (2 if c["grads"] == "bf16" else 4) + (16 if c["opt"] == "sgdm" else 24)


def _normal(out, gen, sd):
    """N(0, sd) into a flat tensor of any type, by pieces."""
    for s in range(0, out.numel(), 1 << 26):
        piece = out[s:s + (1 << 26)]
        z = piece if piece.dtype == torch.float32 else torch.empty(piece.shape, device=piece.device)
        z.normal_(0.0, sd, generator=gen)
        if z is not piece:
            piece.copy_(z)


def _student_t3(out, gen, scale):
    """Student-t with three degrees of freedom, scaled."""
    for s in range(0, out.numel(), 1 << 26):
        piece = out[s:s + (1 << 26)]
        chi, z = torch.zeros(piece.shape, device=piece.device), torch.empty(piece.shape, device=piece.device)
        for _ in range(3):
            z.normal_(generator=gen)
            chi.addcmul_(z, z, value=1.0 / 3.0)
        z.normal_(0.0, scale, generator=gen)
        piece.copy_(z.div_(chi.sqrt_()))


def prepare(case, seed):
    c, dev = case, torch.device("cuda", torch.cuda.current_device())
    gen = torch.Generator(device=dev)
    gen.manual_seed(1_000_003 * seed + 17)
    M, sizes, has_v = c["M"], _sizes(c), c["opt"] != "sgdm"
    gdt = torch.bfloat16 if c["grads"] == "bf16" else torch.float32
    offs, total = _offsets(sizes, c["align"] or 128)                                    # fp32: 128 elements = 512 bytes
    goffs, gtotal = (offs, total) if c["align"] else _offsets(sizes, 512 // gdt.itemsize)

    def buffers(count, dtype):
        # one buffer per worker; beyond 16 workers the rows of one tensor
        if M > 16:
            whole = torch.zeros(M, count, dtype=dtype, device=dev)
            return list(whole.unbind(0)), [whole]
        each = [torch.zeros(count, dtype=dtype, device=dev) for _ in range(M)]
        return each, each

    def views(bufs, at):
        return [[b[o:o + n] for o, n in zip(at, sizes)] for b in bufs]

    # small problems have gradients of order one, models of order 1e-3
    sd = 1.0 if not c["layers"] else 1e-3
    x, x_out = buffers(total, torch.float32)
    u, u_out = buffers(total, torch.float32)
    v, v_out = buffers(total, torch.float32) if has_v else (None, [])
    g, _ = buffers(gtotal, gdt)
    # the middle of a run: workers that drifted apart by a few steps, moments of the gradients' scale
    x0 = torch.empty(total, device=dev)
    _normal(x0, gen, 0.02)
    for m in range(M):
        _normal(x[m], gen, 1e-3)
        x[m].add_(x0)
        _normal(u[m], gen, 0.23 * sd)
        if has_v:
            v[m].uniform_(0.5 * sd * sd, 1.5 * sd * sd, generator=gen)
        (_student_t3 if c["heavy"] else _normal)(g[m], gen, sd)
    del x0
    flags = (desloc.DESLOC_FLAG_ADOPT_NORM_CLIP if c["opt"] == "adopt" else 0) | \
            (desloc.DESLOC_FLAG_POST_AVERAGE if c["post"] else 0)
    eng = desloc.DesLoc(views(x, offs), views(u, offs), views(v, offs) if has_v else None, opt=c["opt"], grad_dtype=c["grads"],
                        beta1=0.9, beta2=c["beta2"], eps=c["eps"], weight_decay=c["wd"], clip_rho=c["rho"],
                        K=(c["Kx"], c["Ku"], c["Kv"]), flags=flags)
    gv = views(g, goffs)
    # the first pass averages everything, later ones follow the periods
    s = dict(case=c, eng=eng, t=math.lcm(c["Kx"], c["Ku"], c["Kv"]), lr=1e-3, grads=gv if c["fresh"] else eng.bind_grads(gv),
             out=[x_out, u_out, v_out], dev=dev)
    if c["call"] == "host":
        # the gradients are on the host, in pinned memory; g is where they land
        hg = [torch.empty(gtotal, dtype=gdt, pin_memory=True) for _ in range(M)]
        for h, b in zip(hg, g):
            h.copy_(b)
            b.zero_()
        s["host"] = views(hg, goffs)
    if c["call"] == "monitor":
        # u as it was some steps ago
        then = []
        for m in range(M):
            b = torch.empty_like(u[m])
            _normal(b, gen, 0.1 * sd)
            then.append(b.add_(u[m]))
        s["then"] = views(then, offs)
    if c["call"] == "graph":
        graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side), torch.cuda.graph(graph, stream=side):
            for t in range(s["t"], s["t"] + 16):
                eng.step(t, s["lr"], s["grads"], clip_bound=_bound(c, t))
        torch.cuda.current_stream().wait_stream(side)
        s["graph"] = graph
    return s


def _bound(c, t):
    return float(t) ** 0.25 if c["opt"] == "adopt" else 0.0


def run(state):
    s, c, eng = state, state["case"], state["eng"]
    t, call = s["t"], c["call"]
    if call == "graph":
        s["graph"].replay()
        return s["out"]
    s["t"] = t + 1
    if call == "step":
        eng.step(t, s["lr"], s["grads"], clip_bound=_bound(c, t))
    elif call == "normclip":
        eng.step_normclip(t, s["lr"], s["grads"], 1.0, clip_bound=_bound(c, t))
    elif call == "host":
        eng.step_host(t, s["lr"], s["host"], s["grads"], clip_bound=_bound(c, t))
    else:
        eng.step_diag(t, s["lr"], s["grads"], clip_bound=_bound(c, t))
        per_tensor, total = eng.diag_norms()
        rate = eng.rel_change(1, s["then"])
        return s["out"] + [np.array(a, dtype=np.float32) for a in (per_tensor, total, rate)]      # for the log
    return s["out"]


def work(case):
    """Algorithmic bytes and operations: gradient in, every state array in and out; 15 operations per coordinate."""
    c = case
    elems = c["M"] * sum(_sizes(c))
    steps = 16 if c["call"] == "graph" else 1
    per = _step_bytes(c)
    if c["call"] == "monitor":
        per += 8                         # u and its snapshot once more
    if c["call"] == "host":
        per += 2 if c["grads"] == "bf16" else 4          # written once on arrival
    return {"bytes": float(elems * per * steps), "flops": float(elems * 15 * steps)}


def tolerance(case):
    """fp32 state and fp32 arithmetic.  One or two steps against the same steps in fp64 (all optimizers, 2 to 16 workers, both
    orderings, clipped and not) were off by up to rel 8e-8, max 7e-7 on five million parameters; more of them reach further."""
    return {"rel": 4e-7, "max": 5e-6}

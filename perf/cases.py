"""What is timed: one optimizer step over a model's whole parameter list.

Each case is one call of the step as a training loop makes it: the state (w,
m, v, the gradients and the optional bf16 weight copy) and the plan are made
once, and a pass runs one step through the public entry points on them.  The
layouts are the repository's workloads and smaller or larger models of the
same kinds; gradients, moments and weights are drawn per tensor as in
workloads.py (weights of the layer's initialisation, gradients of a
per-tensor scale, moments as after some steps), on the GPU.

Learning rates are low enough that a state stays in the range of a training
run when the same gradient is applied some ten thousand times.
"""
from __future__ import annotations

import math

import torch

from paper_1904_00962_gb300 import binding as B
from paper_1904_00962_gb300 import workloads as W
from paper_1904_00962_gb300.state import DeviceState, LambPlan

DEV = "cuda:0"
STEP = 1000            # t of a state's first pass
MU_PRODUCT = 1e-3      # N-LAMB's product of the momentum schedule before it
MU_DECAY = 0.004
SCHEDULE = (2e-3, 3125, 31250)   # eta_0, warm-up and total steps


def _case(name, model, opt="lamb", grad="f32", copy=False, mode="plain",
          entry="plan", align=64, **size):
    """model and size: the parameter list.  mode: step flags.  entry: the
    plan's step, one rank of a sharded step, or the allocation-free call.
    align: elements to which the tensors' offsets in the flat buffers are
    rounded up (1: packed, as flattened parameter buffers are)."""
    return {"name": name, "model": model, "opt": opt, "grad": grad,
            "copy": copy, "mode": mode, "entry": entry, "align": align,
            **size}


def listed():
    return [
        # a tiny model: the call's latency is all there is
        _case("mlp_lamb", "mlp", inputs=64, hidden=32, outputs=10),
        # a small mixed-precision encoder, most of it one embedding
        _case("encoder_small_lamb", "bert", grad="bf16", copy=True, layers=2,
              hidden=256, ffn=1024, vocab=30522),
        # the paper's image workload, with both of its optimizers
        _case("resnet50_lamb", "conv", width=64),
        _case("resnet50_lars", "conv", opt="lars", width=64),
        # the same under an allocator that owns all device memory
        _case("resnet50_noalloc", "conv", entry="noalloc", width=64),
        # the paper's language workloads: fp32, and mixed precision as a
        # large-batch trainer runs it, with the schedule on the device
        _case("bert_base_lamb", "bert", layers=12, hidden=768, ffn=3072,
              vocab=30522),
        _case("bert_large_lamb", "bert", grad="bf16", copy=True,
              mode="schedule", layers=24, hidden=1024, ffn=4096,
              vocab=30522),
        # Nesterov momentum (the appendix's Algorithm 3)
        _case("bert_large_nlamb", "bert", opt="nlamb", grad="bf16", copy=True,
              layers=24, hidden=1024, ffn=4096, vocab=30522),
        # mixed precision with a loss scale: a step with Inf/NaN is skipped
        _case("bert_large_skip", "bert", grad="bf16", copy=True, mode="skip",
              layers=24, hidden=1024, ffn=4096, vocab=30522),
        # one of eight data-parallel ranks that share the optimizer's work
        _case("bert_large_shard8", "bert", grad="bf16", copy=True,
              entry="shard", layers=24, hidden=1024, ffn=4096, vocab=30522),
        # thousands of tensors of every size from 1 to 4M elements
        _case("ragged_4000_lamb", "ragged", tensors=4000, largest=4194304),
        # the same kind in a packed buffer: nothing is aligned
        _case("ragged_packed_lamb", "ragged", grad="bf16", align=1,
              tensors=300, largest=4194304),
    ]


def draw(rng):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    model = rng.choice(["mlp", "bert", "conv", "ragged"])
    if model == "mlp":
        size = dict(inputs=logint(3, 4000), hidden=logint(5, 4000),
                    outputs=logint(2, 2000))
    elif model == "bert":
        hidden = 16 * logint(4, 64) + rng.choice([0, 0, 0, 4, 5])
        size = dict(layers=logint(1, 24), hidden=hidden,
                    ffn=rng.choice([2, 3, 4]) * hidden,
                    vocab=logint(1000, 30522))
    elif model == "conv":
        size = dict(width=logint(4, 128))
    else:
        size = dict(tensors=logint(10, 4000), largest=logint(1000, 4194304))
    opt = rng.choice(["lamb", "lamb", "lamb", "lars", "nlamb", "nnlamb"])
    entry = rng.choice(["plan"] * 6 + ["shard", "noalloc"])
    mode = rng.choice(["plain", "plain", "plain", "schedule", "gradnorm",
                       "skip"])
    if entry == "noalloc":
        opt, mode = "lamb", "plain"
    if entry == "shard" and mode in ("gradnorm", "skip"):
        mode = "plain"
    grad, copy = rng.choice([("f32", False), ("f32", False), ("bf16", True),
                             ("bf16", True), ("bf16", False), ("f32", True)])
    c = _case("", model, opt, grad, copy, mode, entry,
              rng.choice([64, 64, 64, 1]), **size)
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# Layouts and inputs
# ---------------------------------------------------------------------------

def _layout(case):
    model = case["model"]
    if model == "bert":
        return W.bert_layout(case["layers"], case["hidden"], case["ffn"],
                             vocab=case["vocab"])
    if model == "mlp":
        i, h, o = case["inputs"], case["hidden"], case["outputs"]
        L = W.mlp_layout()
        L.shapes = [(i, h), (h,), (h, o), (o,)]
        L.hyper.lr = 1e-4
        return L
    if model == "conv":       # ResNet-50 with other channel counts
        L = W.resnet50_layout()
        f = case["width"] / 64

        def scaled(c):
            return c if c in (3, 1000) else max(1, round(c * f))

        L.shapes = [tuple(scaled(c) if j < 2 else c for j, c in enumerate(s))
                    for s in L.shapes]
        L.hyper.lr = 1e-3
        L.lars_hyper.lr = 0.1
        return L
    return W.ragged_layout(case["tensors"], case["largest"])


def _hyper(case, L):
    """The step's hyperparameters as plain values."""
    lars = case["opt"] == "lars"
    h = L.hyper
    d = dict(lr=h.lr, beta1=h.beta1, beta2=h.beta2, eps=h.eps,
             weight_decay=h.weight_decay, phi=h.phi, gamma_l=h.gamma_l,
             gamma_u=h.gamma_u, trust_coef=1.0, bias_correction=not lars)
    if lars:
        x = L.lars_hyper or W.Hyper(lr=0.1, weight_decay=1e-4, trust_coef=1e-3)
        d.update(lr=x.lr, beta1=x.beta1, weight_decay=x.weight_decay,
                 phi=x.phi, trust_coef=x.trust_coef)
    return d


def _offsets(sizes, align):
    """Element offsets of the tensors in the flat buffers, and their length,
    as DeviceState lays them out."""
    offs, cur = [], 0
    for s in sizes:
        cur = -(-cur // align) * align
        offs.append(cur)
        cur += s
    return offs, max(cur + align, 1)


def _inputs(case, seed, L):
    """Flat w, m, v (fp32) and g, from the seed: w of the layer's
    initialisation, g ~ N(0, s_k), m ~ N(0, 0.3 s_k), v = s_k^2 U(5e-4,
    3e-3), with a tensor's scale s_k; a ragged list starts with m = v = 0 and
    holds some all-zero weights and gradients."""
    sizes = L.sizes
    offs, total = _offsets(sizes, case["align"])
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed) * 1000003 + 17)
    n = len(sizes)
    span = torch.tensor([b - a for a, b in zip(offs, offs[1:] + [total])],
                        device=DEV)

    def per_element(values):
        return torch.repeat_interleave(
            torch.tensor(values, dtype=torch.float32, device=DEV), span,
            output_size=total)

    def normal():
        return torch.empty(total, device=DEV).normal_(generator=gen)

    std = [v if kind == "normal" else 0.0 for kind, v in L.init]
    mean = [v if kind == "const" else 0.0 for kind, v in L.init]
    w = normal().mul_(per_element([0.0 if k in L.zero_w else s
                                   for k, s in enumerate(std)]))
    if any(mean):
        w.add_(per_element(mean))
    scale = per_element([0.0 if k in L.zero_g else float(L.grad_sigma[k])
                         for k in range(n)])
    g = normal().mul_(scale)
    if case["grad"] == "bf16":
        g = g.to(torch.bfloat16)
    if case["model"] == "ragged":
        m, v = torch.zeros_like(w), torch.zeros_like(w)
    else:
        m = normal().mul_(scale).mul_(0.3)
        v = torch.empty(total, device=DEV).uniform_(5e-4, 3e-3, generator=gen)
        v.mul_(scale).mul_(scale)
    return w, m, v, g


class _DeviceArray:
    """A device array of the plan, for torch.as_tensor (no copy).  The tensor
    holds this object, and this object the plan that owns the memory."""

    def __init__(self, plan, address, n, kind):
        self.plan = plan
        self.__cuda_array_interface__ = {"shape": (n,), "typestr": kind,
                                         "data": (address, False),
                                         "version": 3}


def _wrap(plan, address, n, kind="<f8"):
    return torch.as_tensor(_DeviceArray(plan, address, n, kind), device=DEV)


_SHARD_WORLD, _SHARD_RANK = 8, 3
_OPT_CODE = {"lamb": B.LAMB_OPT_LAMB, "lars": B.LAMB_OPT_LARS,
             "nlamb": B.LAMB_OPT_NLAMB, "nnlamb": B.LAMB_OPT_NNLAMB}


def prepare(case, seed):
    L = _layout(case)
    w, m, v, g = _inputs(case, seed, L)
    lars = case["opt"] == "lars"
    st = DeviceState(L.sizes, grad_dtype=case["grad"],
                     copy_dtype="bf16" if case["copy"] else None,
                     with_v=not lars, align_elems=case["align"])
    assert st.total == w.numel()
    st.w, st.m, st.g = w, m, g
    if not lars:
        st.v = v
    d = _hyper(case, L)
    lr = d.pop("lr")
    sched = case["mode"] == "schedule"
    hyper = B.make_hyper(**d, increment_step=True,
                         lr_schedule=SCHEDULE if sched else None,
                         grad_norm=case["mode"] == "gradnorm",
                         skip_nonfinite=case["mode"] == "skip")
    s = {"st": st, "hyper": hyper,
         "step": torch.full((1,), STEP, dtype=torch.int64, device=DEV),
         "lr": torch.full((1,), lr, dtype=torch.float32, device=DEV),
         "mu": torch.full((1,), MU_PRODUCT, dtype=torch.float64, device=DEV)}
    out = {"w": st.w, "m": st.m, "step": s["step"]}
    if not lars:
        out["v"] = st.v
    if st.copy is not None:
        out["copy"] = st.copy
    if case["opt"] in ("nlamb", "nnlamb"):
        out["mu"] = s["mu"]
    if sched:
        out["lr"] = s["lr"]
    n = len(L.sizes)
    nest = case["opt"] in ("nlamb", "nnlamb")
    if case["entry"] == "noalloc":
        out["ratio"] = torch.ones(n, dtype=torch.float64, device=DEV)
        args = (L.sizes, L.decay,
                B.LAMB_BF16 if case["grad"] == "bf16" else B.LAMB_F32,
                B.LAMB_BF16 if case["copy"] else B.LAMB_DTYPE_NONE,
                st.ptrs("w"), st.ptrs("g"), st.ptrs("m"), st.ptrs("v"),
                st.ptrs("copy"), hyper, s["step"].data_ptr(),
                s["lr"].data_ptr(), out["ratio"].data_ptr(),
                torch.cuda.current_stream().cuda_stream)
        s["call"] = lambda: B.lamb_step_noalloc(*args)
    elif case["entry"] == "shard":
        plan = LambPlan(st, L.decay, shard_world=_SHARD_WORLD,
                        shard_rank=_SHARD_RANK)
        code = _OPT_CODE[case["opt"]]
        scalars = (s["step"], s["lr"], s["mu"] if nest else None)
        # the other ranks' sums, as the all-reduce brings them: here those of
        # the first chunk range's kind, one value per chunk
        info = plan.info()
        other = torch.empty(info["n_chunks"], 2, device=DEV)
        gen = torch.Generator(device=DEV)
        gen.manual_seed(int(seed) * 7919 + 3)
        other.uniform_(0.5, 2.0, generator=gen)
        other[info["shard_chunk_begin"]:info["shard_chunk_end"]] = 0
        other = other.reshape(-1)

        def call():
            plan.shard_pass1(hyper, code, *scalars, momentum_decay=MU_DECAY)
            sums = plan.partials()
            sums.add_(other)             # stands for the all-reduce
            plan.set_partials(sums)
            plan.shard_pass2(hyper, code, *scalars, momentum_decay=MU_DECAY)

        s.update(plan=plan, call=call)
    else:
        plan = LambPlan(st, L.decay)
        s["plan"] = plan
        s["call"] = plan.step_call(case["opt"], hyper, s["step"], s["lr"],
                                   s["mu"] if nest else None, MU_DECAY)
    if "plan" in s:
        plan = s["plan"]
        r, wn, un = B.lamb_plan_trust_ratios(plan.handle)
        out["ratio"], out["wnorm"], out["unorm"] = (_wrap(plan, p, n)
                                                    for p in (r, wn, un))
        if case["mode"] in ("gradnorm", "skip"):
            gn, total, bad = B.lamb_plan_grad_norms(plan.handle)
            out["gnorm"] = _wrap(plan, gn, n)
            out["gnorm_all"] = _wrap(plan, total, 1)
            out["nonfinite"] = _wrap(plan, bad, 1, "<i4")
    s["out"] = out
    return s


def run(state):
    state["call"]()
    return state["out"]


# ---------------------------------------------------------------------------
# What a step costs at least, and what it gives
# ---------------------------------------------------------------------------

def work(case):
    """Each operand of the step once: g, m, v, w in, m, v, w and the copy
    out (LARS: no v); a rank of a sharded step has its share of them."""
    L = _layout(case)
    n = L.n_params
    if case["entry"] == "shard":
        n /= _SHARD_WORLD
    state = 8 if case["opt"] == "lars" else 12
    per = (2 if case["grad"] == "bf16" else 4) + 2 * state + \
        (2 if case["copy"] else 0)
    # moments, direction, two sums of squares, update
    flops = 10 if case["opt"] == "lars" else 20
    return {"bytes": n * per, "flops": n * flops}


def tolerance(case):
    """fp32 state, and fp32 sums of squares over up to 16,384 elements: w, m,
    v and the ratios are within 7e-8 of 64 bits (2-norm), so that two correct
    steps are within 1.5e-7 of each other.  A bf16 copy rounds the new w:
    where two correct w lie on either side of a tie it differs by one bf16
    unit (2^-8 of the value at most), which happens to some six elements in a
    million, and to one or two of a small model."""
    if case["copy"]:
        n = _layout(case).n_params
        return {"rel": max(2e-5, 2 * 2 ** -8 / math.sqrt(n)), "max": 1e-2}
    return {"rel": 1e-6, "max": 4e-5}


def exact(case, seed):
    L = _layout(case)
    w, m, v, g = _inputs(case, seed, L)
    d = _hyper(case, L)
    lars, nest = case["opt"] == "lars", case["opt"] in ("nlamb", "nnlamb")
    t, sizes = STEP, L.sizes
    n = len(sizes)
    b1, b2, lam0 = d["beta1"], d["beta2"], d["weight_decay"]
    lr = float(torch.tensor(d["lr"], dtype=torch.float32))
    if case["mode"] == "schedule":
        base, warm, total = SCHEDULE
        lr = base * t / warm if t < warm else base * max(0.0, 1 - t / total)
        lr = float(torch.tensor(lr, dtype=torch.float32))

    def mu(i):
        return b1 * (1 - 0.5 * 0.96 ** (i * MU_DECAY))

    prod = MU_PRODUCT * mu(t)
    offs, _ = _offsets(sizes, case["align"])
    w, m = w.double(), m.double()
    v = None if lars else v.double()
    own = torch.ones(w.numel(), dtype=torch.bool, device=DEV)
    sums = None
    if case["entry"] == "shard":
        # a rank's chunks, 16,384 elements each, and the sums of the others
        chunk = 16384
        counts = [-(-s // chunk) for s in sizes]
        starts, pos, at = [], 0, []
        for k, s in enumerate(sizes):
            for j in range(counts[k]):
                starts.append(pos + j * chunk)
                at.append((k, j))
            pos += s
        lo, hi = (pos * r // _SHARD_WORLD
                  for r in (_SHARD_RANK, _SHARD_RANK + 1))
        mine = [lo <= x < hi for x in starts]
        own.zero_()
        gen = torch.Generator(device=DEV)
        gen.manual_seed(int(seed) * 7919 + 3)
        other = torch.empty(len(starts), 2, device=DEV).uniform_(
            0.5, 2.0, generator=gen)
        other[torch.tensor(mine, device=DEV)] = 0
        # per tensor; a rank's chunks of one tensor are consecutive
        tensor = torch.tensor([k for k, _ in at], device=DEV)
        sums = torch.zeros(n, 2, dtype=torch.float64, device=DEV).index_add_(
            0, tensor, other.double())
        for (k, j), x in zip(at, mine):
            if x:
                a = offs[k] + j * chunk
                own[a:min(a + chunk, offs[k] + sizes[k])] = True
    ratio = torch.ones(n, dtype=torch.float64, device=DEV)
    wn, un, gn = (torch.zeros_like(ratio) for _ in range(3))
    one = torch.ones((), dtype=torch.float64, device=DEV)
    shard = case["entry"] == "shard"
    for k, size in enumerate(sizes):
        if size == 0:
            continue
        sl = slice(offs[k], offs[k] + size)
        lam = lam0 if L.decay[k] else 0.0
        wk, mk, gk = w[sl], m[sl], g[sl].double()
        keep = own[sl] if shard else None
        if lars:
            m_new = b1 * mk + (1 - b1) * (gk + lam * wk)
            u = m_new
        else:
            m_new = b1 * mk + (1 - b1) * gk
            v_new = b2 * v[sl] + (1 - b2) * gk * gk
            if nest:
                mh = (mu(t + 1) * m_new / (1 - prod * mu(t + 1)) +
                      (1 - mu(t)) * gk / (1 - prod))
                vh = (v_new / (1 - b2 ** t) if case["opt"] == "nlamb" else
                      b2 * v_new / (1 - b2 ** (t + 1)) +
                      (1 - b2) * gk * gk / (1 - b2 ** t))
            else:
                mh, vh = m_new / (1 - b1 ** t), v_new / (1 - b2 ** t)
            u = mh / (vh.sqrt() + d["eps"]) + lam * wk
        if shard:
            a = sums[k, 0] + (wk * wk)[keep].sum()
            b = sums[k, 1] + (u * u)[keep].sum()
        else:
            a, b = wk.dot(wk), u.dot(u)
        a, b = a.sqrt(), b.sqrt()
        phi = a.clamp(d["gamma_l"], d["gamma_u"]) if d["phi"] == "clip" else a
        rho = torch.where((a == 0) | (b == 0), one,
                          d["trust_coef"] * phi / b)
        wn[k], un[k], ratio[k] = a, b, rho
        gn[k] = gk.dot(gk).sqrt()
        w_new = wk - lr * rho * u
        if shard:
            w[sl] = torch.where(keep, w_new, wk)
            m[sl] = torch.where(keep, m_new, mk)
            if not lars:
                v[sl] = torch.where(keep, v_new, v[sl])
        else:
            w[sl], m[sl] = w_new, m_new
            if not lars:
                v[sl] = v_new
    out = {"w": w, "m": m, "step": None}
    if not lars:
        out["v"] = v
    if case["copy"]:
        copy = w.to(torch.float32).to(torch.bfloat16).double()
        inside = torch.zeros_like(own)
        for k, size in enumerate(sizes):
            inside[offs[k]:offs[k] + size] = True
        out["copy"] = torch.where(own & inside, copy, torch.zeros_like(copy))
    if nest:
        out["mu"] = torch.tensor([prod], dtype=torch.float64)
    if case["mode"] == "schedule":
        out["lr"] = torch.tensor([lr], dtype=torch.float64)
    out["ratio"] = ratio
    if case["entry"] != "noalloc":
        out["wnorm"], out["unorm"] = wn, un
        if case["mode"] in ("gradnorm", "skip"):
            out["gnorm"] = gn
            out["gnorm_all"] = gn.square().sum().sqrt().reshape(1)
            out["nonfinite"] = None
    return out

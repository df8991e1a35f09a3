"""GPU tests of the one-launch form of the two-pass step (lamb_stash.cu), which
AUTO's two-pass plans take: against the two-pass kernels (the same moments bit
for bit, the norms in another summation order) on grids small enough that a
tensor is kept in part and read again in part, with empty, 1-element, ragged
and unaligned tensors; against itself (repeats, graph replay, two plans at
once); and its bounded wait giving up (nothing faults)."""
import numpy as np
import pytest
import torch

from gpu_util import TOL_RATIO, TOL_STEP, f32
from paper_1904_00962_gb300 import binding as B
from paper_1904_00962_gb300 import build as build_mod
from paper_1904_00962_gb300 import workloads as W
from paper_1904_00962_gb300.state import DeviceState, LambPlan

pytestmark = pytest.mark.gpu

C = 10240     # elements per chunk; a tile is 1,024
# with 4 CTAs a tensor above 16 chunks is read again in part (22 chunks here);
# tiles of every kind: full, partial, the last 1-3 elements, odd and even counts
SIZES = [22 * C + 5, 0, 1, 2, 3, 4, 5, 1023, 1024, 1025, 2047, 2049, C - 1, C,
         C + 1, 4095, 7 * C + 2050, 16 * C, 9 * C + 3, 0, 100003, 65539,
         12 * C + 1022, 3000]


@pytest.fixture(scope="module", autouse=True)
def _lib(gpu):
    build_mod.build()
    B.load()
    yield
    torch.cuda.empty_cache()


def _state(sizes, grad, copy, misalign, with_v, seed=3):
    st = DeviceState(sizes, grad_dtype=grad, copy_dtype=copy,
                     misalign=misalign, with_v=with_v)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    st.w.normal_(0, .02, generator=gen)
    st.g.copy_(torch.empty(st.total, device="cuda").normal_(0, 1e-3,
                                                            generator=gen))
    st.m.normal_(0, 3e-4, generator=gen)
    if with_v:
        st.v.uniform_(5e-10, 3e-9, generator=gen)
    return st


class Run:
    """A state, its plan and a step; launches = kernels of the last step."""

    def __init__(self, sizes, opt="lamb", grad="f32", copy=None, misalign=None,
                 seed=3, flags=None, **plan):
        lars = opt == "lars"
        self.st = _state(sizes, grad, copy, misalign, not lars, seed)
        for k in (0, 9):     # zero w, zero g (and m): the zero-norm rule
            if k < len(sizes):
                self.st.view("w" if k == 0 else "g", k).zero_()
        self.plan = LambPlan(self.st, [k % 2 for k in range(len(sizes))],
                             **plan)
        self.hyper = B.make_hyper(
            weight_decay=.01, phi="clip", gamma_u=10., increment_step=True,
            trust_coef=1e-3 if lars else 1., bias_correction=not lars,
            **(flags or {}))
        dev = "cuda:0"
        self.scalars = (torch.full((1,), 7, dtype=torch.int64, device=dev),
                        torch.full((1,), f32(2e-3), device=dev),
                        torch.full((1,), .6, dtype=torch.float64, device=dev))
        self.step = self.plan.step_call(opt, self.hyper, *self.scalars)
        self.form = B.lamb_plan_step_form(
            self.plan.handle, self.hyper,
            ["lamb", "lars", "nlamb", "nnlamb"].index(opt))

    def launches(self):
        B.lamb_plan_set_timing(self.plan.handle, True)
        self.step()
        n, ms = B.lamb_plan_read_timing(self.plan.handle, 3)
        B.lamb_plan_set_timing(self.plan.handle, False)
        assert n == 1
        return sum(x > 0 for x in ms)

    def out(self):
        st = self.st
        t = [st.w, st.m] + ([st.v] if st.v is not None else []) + \
            ([st.copy.view(torch.int16)] if st.copy is not None else []) + \
            list(self.scalars)
        torch.cuda.synchronize()
        return [x.clone() for x in t], [x.clone() for x in self.plan.results()]


def _same(a, b):
    return all(torch.equal(x.view(torch.uint8), y.view(torch.uint8))
               for x, y in zip(a, b))


@pytest.mark.parametrize("opt", ["lamb", "lars", "nlamb", "nnlamb"])
@pytest.mark.parametrize("grad,copy", [("f32", None), ("bf16", "bf16")])
@pytest.mark.parametrize("misalign", [None, {0, 5, 8, 13, 18, 21}],
                         ids=["aligned", "unaligned"])
@pytest.mark.parametrize("flags", [{}, {"decoupled_decay": True,
                                        "lr_schedule": (2e-3, 10, 100)}],
                         ids=["plain", "decoupled_schedule"])
def test_one_launch_matches_the_two_pass_kernels(opt, grad, copy, misalign,
                                                 flags):
    if opt == "lars":
        flags = {k: v for k, v in flags.items() if k != "decoupled_decay"}
    # 5 CTAs keep 20 chunks of a tensor at most: 7 of the first tensor's 23
    # are read again
    kw = dict(opt=opt, grad=grad, copy=copy, misalign=misalign, flags=flags,
              onchip_max_ctas=5)
    one = Run(SIZES, algorithm=B.LAMB_ALGO_AUTO, **kw)
    two = Run(SIZES, algorithm=B.LAMB_ALGO_TWO_PASS, **kw)
    w0 = two.st.w.clone()
    assert one.form == B.LAMB_FORM_ONE_LAUNCH
    assert one.launches() == 1 and two.launches() == 2
    assert one.plan.info()["algorithm"] == B.LAMB_ALGO_TWO_PASS
    (w1, *s1), r1 = one.out()
    (w2, *s2), r2 = two.out()
    n = len(s1)
    copied = 1 if copy else 0
    keep = [i for i in range(n) if not (copied and i == n - 4)]
    assert _same([s1[i] for i in keep], [s2[i] for i in keep])
    for a, b in zip(r1, r2):
        np.testing.assert_allclose(a.cpu(), b.cpu(), rtol=2 * TOL_RATIO, atol=0)
    scale = torch.maximum(w2.double().abs(), w0.double().abs())
    scale = torch.maximum(scale, (w2.double() - w0.double()).abs())
    assert bool(torch.all((w1.double() - w2.double()).abs() <=
                          TOL_STEP * scale))
    if copied:    # the copy is w rounded to nearest even, bit for bit
        own = torch.zeros(w1.numel(), dtype=torch.bool, device="cuda:0")
        for o, size in zip(one.st.offsets, SIZES):
            own[o:o + size] = True
        assert torch.equal(one.st.copy[own].view(torch.int16),
                           w1.to(torch.bfloat16)[own].view(torch.int16))
    assert one.plan.query() == 0
    for r in (one, two):
        r.plan.destroy()


def _grad_norms(r):
    gn, total, bad = r.plan.grad_norms()
    torch.cuda.synchronize()
    return gn.cpu().numpy(), float(total.item()), int(bad.item())


@pytest.mark.parametrize("opt", ["lamb", "nnlamb"])
@pytest.mark.parametrize("grad,copy", [("f32", None), ("bf16", "bf16")])
@pytest.mark.parametrize("misalign", [None, {0, 5, 8, 13, 18, 21}],
                         ids=["aligned", "unaligned"])
@pytest.mark.parametrize("bad", [None, float("nan"), float("inf")])
@pytest.mark.parametrize("flag", ["grad_norm", "skip_nonfinite"])
def test_gradient_check_matches_the_two_pass_kernels(opt, grad, copy, misalign,
                                                     bad, flag):
    """The check reads g in its own launch; norms, decision, status word and
    what a skipped step leaves and reports are those of the two kernels.  (Both
    are two launches: the sums tell them apart.)"""
    runs = []
    for algo, form in ((B.LAMB_ALGO_AUTO, B.LAMB_FORM_ONE_LAUNCH),
                       (B.LAMB_ALGO_TWO_PASS, B.LAMB_FORM_TWO_PASS)):
        r = Run(SIZES, opt=opt, grad=grad, copy=copy, misalign=misalign,
                flags={flag: True, "lr_schedule": (2e-3, 10, 100)},
                algorithm=algo, onchip_max_ctas=5)
        if bad is not None:
            r.st.view("g", 20)[100002] = bad
        before = r.out()[0]
        assert r.form == form and r.launches() == 2
        after, res = r.out()
        runs.append((before, after, res, _grad_norms(r), r.plan.query()))
        r.plan.destroy()
    (b1, a1, r1, n1, s1), (b2, a2, r2, n2, s2) = runs
    assert s1 == s2 and n1[2] == n2[2] == (bad is not None)
    skipped = bad is not None and flag == "skip_nonfinite"
    assert bool(s1 & B.LAMB_STATUS_SKIPPED) == skipped
    if skipped:
        assert _same(b1, a1) and _same(b2, a2)
    m = slice(1, 2 if opt == "lars" else 3)      # m, v
    assert _same(a1[m], a2[m]) and _same(a1[-3:], a2[-3:])
    # a chunk's sum is fp32 over 40 (kernel: 64) elements, then trees
    np.testing.assert_allclose(n1[0], n2[0], rtol=2 * TOL_RATIO)
    np.testing.assert_allclose(n1[1], n2[1], rtol=2 * TOL_RATIO)
    for a, b in zip(r1, r2):
        np.testing.assert_allclose(a.cpu(), b.cpu(), rtol=2 * TOL_RATIO)
    # ||w||: two floats over a chunk against fp32 sums
    assert not torch.equal(r1[1], r2[1])


@pytest.mark.parametrize("flag", ["grad_norm", "skip_nonfinite"])
def test_lars_with_the_gradient_check_keeps_the_two_kernels(flag):
    """Bit for bit, norms included: their sums' order, not the launch's."""
    outs = []
    for algo in (B.LAMB_ALGO_AUTO, B.LAMB_ALGO_TWO_PASS):
        r = Run(SIZES, opt="lars", flags={flag: True}, algorithm=algo,
                onchip_max_ctas=5)
        r.step()
        a, b = r.out()
        outs.append(a + b)
        r.plan.destroy()
    assert _same(*outs)


def test_gradient_check_of_a_step_with_a_bad_count_does_nothing():
    r = Run(SIZES, flags={"skip_nonfinite": True}, onchip_max_ctas=5)
    r.st.view("g", 20)[5] = float("nan")
    r.scalars[0].fill_(0)
    before = r.out()[0]
    r.step()
    assert _same(before, r.out()[0])
    assert r.plan.query() == B.LAMB_STATUS_BAD_STEP
    assert _grad_norms(r)[2] == 0
    r.plan.destroy()


@pytest.mark.parametrize("misalign", [None, {0, 4, 6}],
                         ids=["aligned", "unaligned"])
def test_on_chip_plans_of_several_rounds(misalign):
    """AUTO's on-chip plan of several rounds runs lamb_step as one launch and
    lars_step on the two-pass kernels; one with mostly short tensors keeps the
    on-chip kernel, whose norms are within the ratio tolerance too."""
    sizes = [100003, 90000, 3000, 0, 65539, 5 * C + 7, 8 * C, 1025, 100001]
    kw = dict(misalign=misalign, onchip_max_ctas=4)
    one = Run(sizes, algorithm=B.LAMB_ALGO_AUTO, **kw)
    two = Run(sizes, algorithm=B.LAMB_ALGO_TWO_PASS, **kw)
    info = one.plan.info()
    assert info["algorithm"] == B.LAMB_ALGO_ON_CHIP and info["n_rounds"] > 1
    assert one.form == B.LAMB_FORM_ONE_LAUNCH and one.launches() == 1 and two.launches() == 2
    (w1, *s1), r1 = one.out()
    (w2, *s2), r2 = two.out()
    assert _same(s1, s2)
    for a, b in zip(r1, r2):
        # fp64 ratios of fp32 chunk sums: an on-chip ratio, rounded to fp32,
        # would not be this close to its own norms
        np.testing.assert_allclose(a.cpu(), b.cpu(), rtol=2 * TOL_RATIO, atol=0)
    rho, wn, un = r1
    live = [k for k in range(1, len(sizes)) if sizes[k]]
    np.testing.assert_allclose((rho * un / wn.clamp(max=10.))[live].cpu(), 1.0,
                               rtol=1e-12)
    for r in (one, two):
        r.plan.destroy()
    lars = Run(sizes, opt="lars", algorithm=B.LAMB_ALGO_AUTO, **kw)
    assert lars.form == B.LAMB_FORM_TWO_PASS and lars.launches() == 2
    lars.plan.destroy()
    short = Run([900] * 400, algorithm=B.LAMB_ALGO_AUTO, onchip_max_ctas=4)
    assert short.plan.info()["n_rounds"] > 1
    assert short.form == B.LAMB_FORM_ON_CHIP and short.launches() == 1
    rho, wn, un = short.out()[1]
    assert not torch.equal(rho * un, wn)     # fp32: the on-chip kernel
    short.plan.destroy()


@pytest.mark.parametrize("kind", ["on_chip", "two_pass"])
@pytest.mark.parametrize("misalign", [None, {0, 4, 6}],
                         ids=["aligned", "unaligned"])
def test_norms_keep_more_than_fp32_sums(kind, misalign):
    """||w|| and ||u|| against 64 bits, the u's elements being exact here (fp32,
    no decay, no corrections).  Squares are added in fp32 over four elements
    only: a norm of n elements is then within 2^-24 / sqrt(n) or so, 4.5e-10 on
    average and 1.6e-9 at most over 400 tensors of 10,240 normal elements by a
    host model; fp32 sums over a chunk gave 2.5e-8 and 6.7e-8.  An on-chip
    plan's norms, in two floats, must not lose by AUTO's choice of kernel."""
    sizes = [C] * 40 + [8192] * 20 + [3 * C + 5, 100001]
    if kind == "two_pass":
        sizes += [22 * C + 5]
    r = Run(sizes, misalign=misalign, onchip_max_ctas=5)
    assert r.plan.info()["algorithm"] == {
        "on_chip": B.LAMB_ALGO_ON_CHIP,
        "two_pass": B.LAMB_ALGO_TWO_PASS}[kind]
    r.hyper = B.make_hyper(weight_decay=0., eps=2.0 ** -20,
                           bias_correction=False)
    r.step = r.plan.step_call("lamb", r.hyper, *r.scalars)
    w = [r.st.download("w", k).astype(np.float64) for k in range(len(sizes))]
    r.step()
    _, wn, un = (x.cpu().numpy() for x in r.out()[1])
    for k in range(len(sizes)):
        u = r.st.download("m", k) / (np.sqrt(r.st.download("v", k)) +
                                     np.float32(2.0 ** -20))
        assert u.dtype == np.float32
        for got, x in ((wn[k], w[k]), (un[k], u.astype(np.float64))):
            want = np.sqrt(np.dot(x, x))
            assert abs(got - want) <= 4e-9 * want, (k, got / want - 1)
    r.plan.destroy()


def test_a_layout_read_again_for_the_most_part_takes_the_two_launches():
    r = Run([60 * C, 5 * C], algorithm=B.LAMB_ALGO_AUTO, onchip_max_ctas=2)
    assert r.launches() == 2
    r.plan.destroy()


def test_repeats_and_graph_replays_give_the_same_bits():
    L = W.bert_layout(2, 768, 3072, vocab=12000)
    outs = []
    for graph in (False, False, True):
        r = Run(L.sizes, grad="bf16", copy="bf16")
        assert r.launches() == 1
        if graph:
            torch.cuda.synchronize()
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                call = r.plan.step_call("lamb", r.hyper, *r.scalars, stream=s)
                g = torch.cuda.CUDAGraph()
                with torch.cuda.graph(g, stream=s):
                    call()
                for _ in range(5):
                    g.replay()
            s.synchronize()
        else:
            for _ in range(5):
                r.step()
        a, b = r.out()
        assert r.plan.query() == 0
        outs.append(a + b)
        r.plan.destroy()
    assert _same(outs[0], outs[1]) and _same(outs[0], outs[2])


def test_steps_of_two_plans_on_two_streams():
    """Each launch needs every SM and waits inside for its own CTAs only; two
    plans' launches on two streams must not wait for each other's."""
    L = W.bert_layout(1, 768, 3072, vocab=8000)
    want, runs, calls = [], [], []
    for seed in (1, 2):
        r = Run(L.sizes, seed=seed, wait_limit_ms=2000)
        assert r.launches() == 1
        for _ in range(29):
            r.step()
        want.append(r.out())
        r.plan.destroy()
    for seed in (1, 2):
        r = Run(L.sizes, seed=seed, wait_limit_ms=2000)
        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())
        runs.append((r, s))
        calls.append(r.plan.step_call("lamb", r.hyper, *r.scalars, stream=s))
    torch.cuda.synchronize()
    for _ in range(30):
        for c in calls:
            c()
    torch.cuda.synchronize()
    for (r, _), (a, b) in zip(runs, want):
        assert r.plan.query() == 0
        x, y = r.out()
        assert _same(x + y, a + b)
        r.plan.destroy()


def test_wait_gives_up_and_a_new_plan_works():
    """A plan whose CTAs wait for ratios tagged for a launch that never comes
    (a test-only option): the wait runs out, every CTA returns, no weight
    changes, later steps do nothing, and a new plan works."""
    sizes = [3 * C, 8 * C + 1, 500, 4 * C]
    r = Run(sizes, test_unmet_wait=True, wait_limit_ms=20, onchip_max_ctas=2)
    w0 = r.st.w.clone()
    r.step()
    torch.cuda.synchronize()
    assert r.plan.query(clear=True) & B.LAMB_STATUS_WAIT_TIMEOUT
    assert torch.equal(r.st.w, w0)
    r.step()
    torch.cuda.synchronize()
    assert torch.equal(r.st.w, w0) and r.plan.query() == 0
    r.plan.destroy()
    outs = []
    for algo in (B.LAMB_ALGO_AUTO, B.LAMB_ALGO_TWO_PASS):
        n = Run(sizes, onchip_max_ctas=2, algorithm=algo)
        n.step()
        outs.append(n.out())
        assert n.plan.query() == 0
        n.plan.destroy()
    assert _same(outs[0][0][1:3], outs[1][0][1:3])     # m, v
    assert not torch.equal(outs[0][0][0], w0)

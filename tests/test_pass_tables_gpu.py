"""GPU tests of what surrounds the two passes: the combine of the chunk sums
into a tensor's norms, at the edges of its batches, and the tables that
lamb_step_noalloc builds, at the sizes where their way to the device
changes."""
import numpy as np
import pytest
import torch

from paper_1904_00962_gb300 import binding as B
from paper_1904_00962_gb300 import build as build_mod
from paper_1904_00962_gb300.state import DeviceState, LambPlan

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib(gpu):
    build_mod.build()
    B.load()
    yield
    torch.cuda.empty_cache()


def _scalars():
    return (torch.full((1,), 3, dtype=torch.int64, device="cuda:0"),
            torch.full((1,), 1e-3, dtype=torch.float32, device="cuda:0"))


def _fixed_order_sum(x, threads):
    """Thread t's slots t, t + threads, ... in order, then the trees of a
    warp and of the warps (the documented order), in float64."""
    acc = np.zeros(threads)
    for i in range(0, len(x), threads):
        part = x[i:i + threads].astype(np.float64)
        acc[:len(part)] += part
    for width in (32, threads // 32):
        acc = acc.reshape(-1, width)
        while acc.shape[1] > 1:
            half = acc.shape[1] // 2
            acc = acc[:, :half] + acc[:, half:]
        acc = acc.reshape(-1)
    return acc[0]


def test_norms_are_the_fixed_order_sums_of_the_slots():
    counts = [0, 1, 31, 32, 33, 255, 256, 257, 511, 513, 2047, 2048, 2049,
              4097]
    st = DeviceState([1024 * c - (7 if c else 0) for c in counts])
    plan = LambPlan(st, chunk_elems=1024, shard_world=2, shard_rank=0,
                    algorithm=B.LAMB_ALGO_TWO_PASS)
    threads = plan.info()["threads_per_block"]
    assert sum(counts) == plan.info()["n_chunks"]
    gen = torch.Generator(device="cuda:0")
    gen.manual_seed(5)
    slots = torch.rand(sum(counts), 2, device="cuda:0", generator=gen) + 1e-3
    step, lr = _scalars()
    hyper = B.make_hyper()
    for t in (st.w, st.g, st.m, st.v):
        t.zero_()
    plan.shard_pass1(hyper, B.LAMB_OPT_LAMB, step, lr)
    plan.set_partials(slots.reshape(-1))
    plan.shard_pass2(hyper, B.LAMB_OPT_LAMB, step, lr)
    ratio, wn, un = (x.cpu().numpy() for x in plan.results())
    host = slots.cpu().numpy()
    first = 0
    for k, c in enumerate(counts):
        if c:
            part = host[first:first + c]
            want = [np.sqrt(_fixed_order_sum(part[:, i], threads))
                    for i in (0, 1)]
            # same adds in the same order, correctly rounded roots: equal
            assert [wn[k], un[k]] == want, c
            assert ratio[k] == pytest.approx(want[0] / want[1], rel=1e-15), c
        first += c
    plan.destroy()


@pytest.mark.parametrize("mask", [False, True])
@pytest.mark.parametrize("n", [1, 192, 193, 640, 641, 1025, 4096])
def test_noalloc_tables_of_many_tensors_match_the_plan(n, mask):
    """192 | 193: two sizes of launch parameter; 640 | 641: parameter and
    copies; 1025: two tensors a thread; 4096: the most the call takes."""
    sizes = [(37 * k) % 3001 for k in range(n)]
    sizes[-1] = 16384 * 3 + 5          # several chunks, in the last tensor
    decay = [k % 3 != 0 for k in range(n)] if mask else None
    a = DeviceState(sizes, grad_dtype="bf16", copy_dtype="bf16")
    b = DeviceState(sizes, grad_dtype="bf16", copy_dtype="bf16")
    gen = torch.Generator(device="cuda:0")
    gen.manual_seed(n)
    for name, scale in (("w", 0.02), ("g", 1e-3), ("m", 1e-3), ("v", 1e-6)):
        t = torch.randn(getattr(a, name).numel(), device="cuda:0",
                        generator=gen) * scale
        if name == "v":
            t = t.abs()
        for s in (a, b):
            getattr(s, name).copy_(t)
    a.copy.zero_()
    b.copy.zero_()
    step, lr = _scalars()
    hyper = B.make_hyper()
    plan = LambPlan(a, decay, algorithm=B.LAMB_ALGO_TWO_PASS)
    plan.lamb_step(hyper, step, lr)
    ratio = torch.empty(n, dtype=torch.float64, device="cuda:0")
    B.lamb_step_noalloc(sizes, decay, B.LAMB_BF16, B.LAMB_BF16, b.ptrs("w"),
                        b.ptrs("g"), b.ptrs("m"), b.ptrs("v"),
                        b.ptrs("copy"), hyper, step.data_ptr(),
                        lr.data_ptr(), ratio.data_ptr(),
                        torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    for name in ("w", "m", "v", "copy"):
        x, y = getattr(a, name), getattr(b, name)
        if x.dtype == torch.bfloat16:
            x, y = x.view(torch.int16), y.view(torch.int16)
        assert torch.equal(x, y), name
    assert torch.equal(ratio, plan.results()[0])
    plan.destroy()


@pytest.mark.parametrize("opt", ["lamb", "lars", "noalloc"])
def test_captured_passes_replay_like_eager_steps(opt):
    """The second pass starts behind the first before it has ended: five
    steps in a row, eager and replayed, on many small tensors (the first pass
    ends late) and one of 2,000 chunks."""
    sizes = [1 + (97 * k) % 5000 for k in range(300)] + [16384 * 2000 + 3]
    out = []
    for captured in (False, True):
        st = DeviceState(sizes)
        gen = torch.Generator(device="cuda:0")
        gen.manual_seed(9)
        for name, scale in (("w", 0.02), ("g", 1e-3), ("m", 1e-3),
                            ("v", 1e-6)):
            t = torch.randn(getattr(st, name).numel(), device="cuda:0",
                            generator=gen) * scale
            getattr(st, name).copy_(t.abs() if name == "v" else t)
        step, lr = _scalars()
        hyper = B.make_hyper(increment_step=True, bias_correction=opt != "lars",
                             trust_coef=1e-2 if opt == "lars" else 1.0)
        plan = LambPlan(st, algorithm=B.LAMB_ALGO_TWO_PASS)
        ptrs = [st.ptrs(x) for x in ("w", "g", "m", "v")]

        def one():
            if opt == "lamb":
                plan.lamb_step(hyper, step, lr)
            elif opt == "lars":
                plan.lars_step(hyper, step, lr)
            else:
                B.lamb_step_noalloc(sizes, None, B.LAMB_F32,
                                    B.LAMB_DTYPE_NONE, *ptrs, None, hyper,
                                    step.data_ptr(), lr.data_ptr(), 0,
                                    torch.cuda.current_stream().cuda_stream)
        one()
        torch.cuda.synchronize()
        if captured:
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph):
                one()
            for _ in range(5):
                graph.replay()
        else:
            for _ in range(5):
                one()
        torch.cuda.synchronize()
        assert int(step.item()) == 3 + 6
        out.append([getattr(st, x).clone() for x in ("w", "m", "v")])
        plan.destroy()
    for a, b in zip(*out):
        assert torch.equal(a, b)

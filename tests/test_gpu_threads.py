"""Host threads: the library keeps its per-call caches per host thread and
initialises each plan's page-locked tables once, so plans may be used from
several threads, each on its own stream (and one plan from two threads with
separate workspaces)."""
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest
import torch

import oracle as O
import workloads as WL

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sc():
    if not torch.cuda.is_available():
        pytest.fail("a GPU test ran without a visible GPU")
    import paper_2007_08056_gb300 as mod
    mod.load()
    return mod


def spec(t):
    return (t.signs, t.charge, t.dims)


def test_two_threads_two_streams(sc):
    c = WL.cc_ladder(8, 128, 64)
    u, v = WL.draw_pair(c)
    o = O.plan(c.einsum, O.Group(c.moduli), O.Sym(*spec(c.u)), O.Sym(*spec(c.v)))
    want = O.contract_blockloop(o, u, v)
    shared = sc.Plan(c.einsum, c.moduli, spec(c.u), spec(c.v), "split_bf16")
    ud, vd = torch.from_numpy(u).cuda(), torch.from_numpy(v).cuda()
    torch.cuda.synchronize()

    def work(k):
        torch.cuda.set_device(0)
        stream = torch.cuda.Stream()
        own = sc.Plan(c.einsum, c.moduli, spec(c.u), spec(c.v), ("split_bf16", "tf32")[k % 2])
        ws = torch.empty(int(shared.info.workspace_bytes), dtype=torch.uint8, device="cuda")
        outs = []
        with torch.cuda.stream(stream):
            for i in range(4):
                p = shared if i % 2 == 0 else own
                outs.append((p.info.precision, p.contract(ud, vd, workspace=ws if p is shared else None)))
            stream.synchronize()
        return [(prec, w.cpu().numpy()) for prec, w in outs]

    with ThreadPoolExecutor(max_workers=3) as ex:
        results = list(ex.map(work, range(3)))
    tol = {1: 1e-10, 2: 1e-2}
    for res in results:
        for prec, got in res:
            assert np.linalg.norm(got - want) <= tol[prec] * np.linalg.norm(want)


@pytest.mark.parametrize("long_k,short_k", [((4, 16, 16), (2, 5, 3)), ((8, 32, 8), (8, 24, 2))],
                         ids=["short_rows", "long_rows"])
def test_shorter_rows_on_another_thread(sc, long_k, short_k):
    """A kernel's shared-memory limit belongs to the function, not to a thread:
    a second thread with shorter rows (autograd's backward thread, say) must not
    lower it below what the first thread has already asked for."""
    def run(dims):
        G, virt, occ = dims
        c = WL.cc_ladder(G, G * virt, G * occ)
        gen = torch.Generator(device="cuda").manual_seed(1)
        p = sc.Plan(c.einsum, c.moduli, spec(c.u), spec(c.v), "split_bf16")
        x = [torch.randn(s, generator=gen, dtype=torch.float64, device="cuda") for s in (p.shape_u, p.shape_v)]
        p.contract(*x)
        torch.cuda.synchronize()
        p.check_device_error()
        return p.info.single_read_prep

    def other():
        torch.cuda.set_device(0)
        return run(short_k)

    kernels = run(long_k)
    with ThreadPoolExecutor(max_workers=1) as ex:
        assert ex.submit(other).result() & kernels   # the same preparation kernel
    assert run(long_k) == kernels

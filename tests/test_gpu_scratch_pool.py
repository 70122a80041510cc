"""The library's scratch pool: what it keeps is bounded while a geometry exists and given back with
the last one; calls from several threads and streams at once give the single-stream results; calls
can be captured into a CUDA graph and replayed."""
import gc
import threading

import torch

import pytest

from paper_2512_21180_gb300 import inputs as I
from paper_2512_21180_gb300 import ops
from paper_2512_21180_gb300 import projector as P

pytestmark = pytest.mark.gpu


def test_kept_memory_is_bounded_and_given_back():
    gc.collect()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    g = I.geometry("clinical")
    geom = P.Geometry(g)
    y = torch.rand((4,) + geom.proj_shape, device="cuda")   # 1.26 GB of weighted projections
    out = torch.empty((4,) + geom.vol_shape, device="cuda")
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    P.back_project(geom, y, out=out)
    torch.cuda.synchronize()
    kept = before - torch.cuda.mem_get_info()[0]
    assert kept <= (1 << 30) + (64 << 20)
    small = P.Geometry(I.geometry("tiny16"))
    geom.close()
    small.close()
    torch.cuda.synchronize()
    # (other tests' geometries may still be alive and keep theirs)
    assert before - torch.cuda.mem_get_info()[0] <= max(kept, 64 << 20)


def test_threads_and_streams():
    geom = P.Geometry(I.scaled(I.geometry("small64"), n=(40, 36, 30), nu=70, nv=41))
    xs = [torch.as_tensor(I.random_volume((1,) + geom.vol_shape, s), device="cuda") for s in range(4)]
    want = [(P.forward_project(geom, x), ops.fdk(geom, P.forward_project(geom, x))) for x in xs]
    want = [(f, r, P.back_project(geom, f)) for f, r in want]
    torch.cuda.synchronize()
    bad = []

    def work(i):
        with torch.cuda.stream(torch.cuda.Stream()):
            for _ in range(20):
                f = P.forward_project(geom, xs[i])
                r, b = ops.fdk(geom, f), P.back_project(geom, f)
                torch.cuda.current_stream().synchronize()
                if not (torch.equal(f, want[i][0]) and torch.equal(r, want[i][1]) and torch.equal(b, want[i][2])):
                    bad.append(i)

    ts = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    [t.start() for t in ts]
    [t.join() for t in ts]
    assert not bad


def test_calls_in_a_graph():
    geom = P.Geometry(I.geometry("small64"))
    x = torch.as_tensor(I.random_volume((1,) + geom.vol_shape, 1), device="cuda")
    f, b = torch.empty((1,) + geom.proj_shape, device="cuda"), torch.empty_like(x)
    P.forward_project(geom, x, out=f)
    P.back_project(geom, f, out=b)
    want = (f.clone(), b.clone())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        P.forward_project(geom, x, out=f)
        P.back_project(geom, f, out=b)
    f.zero_()
    b.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(f, want[0]) and torch.equal(b, want[1])


LAST_ONE = """
import torch
from paper_2512_21180_gb300 import inputs as I
from paper_2512_21180_gb300 import projector as P
a, b = P.Geometry(I.geometry("clinical")), P.Geometry(I.geometry("tiny16"))
y = torch.rand((2,) + a.proj_shape, device="cuda")      # 0.63 GB of weighted projections
out = torch.empty((2,) + a.vol_shape, device="cuda")
P.back_project(b, torch.zeros((1,) + b.proj_shape, device="cuda"))   # loads the kernels
torch.cuda.synchronize()
start = torch.cuda.mem_get_info()[0]
def held():
    torch.cuda.synchronize()
    return (start - torch.cuda.mem_get_info()[0]) >> 20
P.back_project(a, y, out=out)
print(held())
a.close()
print(held())
b.close()
print(held())
c = P.Geometry(I.geometry("clinical"))
P.back_project(c, y, out=out)
print(held())
c.close()
print(held())
"""


def test_the_last_geometry_gives_the_memory_back():
    """In a process of its own (no other geometries): MiB held after a call, after closing one of two
    geometries, after closing the last, and the same again with a new one."""
    import subprocess
    import sys
    r = subprocess.run([sys.executable, "-c", LAST_ONE], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    call, one_left, none_left, call2, none_left2 = (int(v) for v in r.stdout.split())
    assert 512 <= call <= 1024 + 64
    assert 512 <= one_left <= 1024 + 64
    assert none_left <= 64 and none_left2 <= 64
    assert 512 <= call2 <= 1024 + 64

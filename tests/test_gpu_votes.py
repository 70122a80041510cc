"""How a pipelined kernel leaves when one of its waits gives up: all threads of the CTA together,
with nothing written, whichever of them gave up; a lane of a warp-wide loop stays with its
warp to the end; and a tile that one thread finds odd is odd for
all of them while the loop goes on. The waits expire on a barrier in shared memory after a short
limit of the GPU's global timer (no fault, no hang)."""
import pytest
import torch

from paper_2512_21180_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    from paper_2512_21180_gb300 import build
    build.build()
    from paper_2512_21180_gb300 import _lib, projector
    return _lib, projector.Geometry(I.geometry("tiny16"))


def run(env, late, arrive, odd):
    L, geom = env
    assert geom.device_status(clear=True) == 0
    out = torch.full((288,), -7, dtype=torch.int32, device="cuda")
    L.check(L.load().cbct_vote_probe(geom.handle, 2_000_000, late, arrive, odd, out.data_ptr(),
                                     torch.cuda.current_stream().cuda_stream), "cbct_vote_probe")
    torch.cuda.synchronize()
    # every lane took part in all its warp's sums; a lane whose wait gave up did nothing else
    seen = [3 if arrive == 1 or (arrive == 2 and t >= late) else 0 for t in range(96)]
    assert out[192:].tolist() == [1100 * s + 96 for s in seen]
    return out[:192], geom.device_status(clear=True)


@pytest.mark.parametrize("late,arrive", [(96, 0), (0, 0), (40, 0), (1, 0), (95, 0), (40, 2), (64, 2), (95, 2)])
def test_a_wait_that_gives_up_ends_the_loop_for_all(env, late, arrive):
    out, status = run(env, late, arrive, -1)
    assert status == 1
    assert bool((out == -7).all())


@pytest.mark.parametrize("odd", [-1, 0, 31, 50, 95])
def test_odd_data_of_one_thread_is_odd_for_all(env, odd):
    out, status = run(env, 96, 1, odd)
    assert status == 0
    assert bool((out[:96] == (3 if odd < 0 else 2)).all())
    assert bool((out[96:] == (0 if odd < 0 else 1)).all())


def test_patient_threads_alone_go_on(env):
    out, status = run(env, 0, 2, -1)   # every thread waits ten times the limit: no one gives up
    assert status == 0
    assert bool((out[:96] == 3).all())

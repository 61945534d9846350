"""Making and dropping a run whose memory the caller owns waits for its own stream only, not for what
other streams of the device are doing -- for the process's only run too."""
import gc

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1909_09613_gb300 as pic  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1909_09613_gb300 import _build
    _build.build()


def _come_and_go(stream):
    run = pic.Run((64, 32, 1), (1.0, 1.0, 1.0), 0.3, 2, pic.PIC_SCHEME_WT, capacity=(64, 64),
                  stream=stream)
    run.step(1)
    run.field(0)
    run.close()


def test_runs_come_and_go_beside_a_busy_stream():
    gc.collect()  # no run of an earlier test is left
    own, other = torch.cuda.Stream(), torch.cuda.Stream()
    a = torch.randn(8192, 8192, device="cuda")
    _come_and_go(own)  # the kernels are loaded, the allocator's block and the page-locked memory there
    torch.cuda.synchronize()
    done = torch.cuda.Event()
    with torch.cuda.stream(other):
        for _ in range(40):
            a @ a
        done.record()
    _come_and_go(own)
    _come_and_go(own)
    waited = done.query()
    torch.cuda.synchronize()
    assert not waited

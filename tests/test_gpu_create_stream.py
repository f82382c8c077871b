"""A problem's tables are uploaded on its own stream, so that its kernels are ordered behind them: with a stream that the
default one does not synchronise with, creation waits for nothing on the default stream."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_tables_are_uploaded_on_the_problems_stream():
    from paper_2506_14792_gb300 import spadj
    def make(stream):
        return spadj.Problem(spadj.SPADJ_COUETTE3D, spadj.SPADJ_SBDF2, [8, 4, 8], [4 * np.pi, 2 * np.pi], [1000.0], 5e-3, stream=stream)
    side = torch.cuda.Stream()
    make(side).close()  # kernels loaded
    torch.cuda.synchronize()
    torch.cuda._sleep(4_000_000_000)  # about 2 s on the default stream
    busy = torch.cuda.Event()
    busy.record()
    p = make(side)
    assert not busy.query()
    torch.cuda.synchronize()
    p.close()

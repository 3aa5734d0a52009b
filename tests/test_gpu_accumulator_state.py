"""Whether a batch writes or adds to the accumulator is decided by what has run
on the device since the reset: a grouped accumulation that could not be launched
leaves its handles as they were, and captured launches count when they run."""
import ctypes

import numpy as np
import pytest

from paper_2105_00027_gb300 import inputs
from gpu_util import cuda, draw, ensure_built, run_lib

pytestmark = pytest.mark.gpu


def test_group_that_cannot_be_launched():
    """The shared stream is the legacy one, and another (blocking) stream is
    being captured: the group's graph launch is refused by the runtime.  Once the
    capture has ended the same call goes through, and gives the bits of a run
    without the refusal."""
    torch = cuda()
    g4 = ensure_built()
    assert torch.cuda.current_stream().cuda_stream == 0
    rt = ctypes.CDLL("libcudart.so.13")
    ps = [inputs.Problem(2, 2, 3, 2, 4, 8.0, 6, 4), inputs.Problem(3, 1, 4, 3, 2, 8.0, 6, 4)]
    data = [draw(p, seed=4, problem_index=i) for i, p in enumerate(ps)]
    Md = [d[0].cuda() for d in data]
    G0 = [torch.from_numpy(np.ascontiguousarray(d[1])).cuda() for d in data]
    hs = [g4.G4.for_problem(p, precision="mixed") for p in ps]

    def stage(lo, hi, f=1.0):
        for h, M, g0 in zip(hs, Md, G0):
            for r in range(lo, hi):
                h.compute_G((M[r] * f).contiguous(), g0, 1.0)

    def run(refused):
        stage(0, 4, 1e3)               # values that must not be seen again
        g4.accumulate_group(hs)
        for h in hs:
            h.reset()
        for lo, hi in ((0, 4), (4, 6)):
            stage(lo, hi)
            torch.cuda.synchronize()
            if refused:
                s, g = ctypes.c_void_p(), ctypes.c_void_p()
                assert rt.cudaStreamCreate(ctypes.byref(s)) == 0
                assert rt.cudaStreamBeginCapture(s, 2) == 0       # relaxed
                with pytest.raises(g4.G4Error) as e:
                    g4.accumulate_group(hs)
                assert e.value.status == g4.G4_ERR_CUDA
                rt.cudaStreamEndCapture(s, ctypes.byref(g))        # invalidated: an error, no graph
                rt.cudaGetLastError()
                assert rt.cudaStreamDestroy(s) == 0
            g4.accumulate_group(hs)
        out = [h.finalize()[0].cpu() for h in hs]
        for h in hs:
            h.reset()
        return out

    got = run(True)       # the first refusal comes before any graph of these handles is kept ...
    want = run(False)
    again = run(True)     # ... these refuse the relaunch of a kept one
    for h in hs:
        h.close()
    for a, b, c in zip(got, want, again):
        assert torch.equal(a, b) and torch.equal(c, b)


@pytest.mark.parametrize("channel,deferred", [("pp_updown", False), ("ph_transverse", False), ("pp_updown", True)])
@pytest.mark.parametrize("captured", ["fresh", "later"])
def test_captured_batch(channel, deferred, captured):
    """A batch captured in a CUDA graph, as a run's first or a later one, and
    launched twice after a reset: the sum of two batches."""
    torch = cuda()
    g4 = ensure_built()
    p = inputs.Problem(3, 2, 4, 3, 6, 8.0, 8, 8)
    M, G0, s = draw(p, seed=5)
    twice = torch.cat([M, M])
    want, _, h = run_lib(p, twice, G0, np.ones(16), "mixed", channel=channel, deferred=deferred)
    h.close()
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        Md, G0d = M.cuda(), torch.from_numpy(np.ascontiguousarray(G0)).cuda()
        h = g4.G4.for_problem(p, precision="mixed", channel=channel, deferred=deferred)
        for r in range(8):
            h.compute_G(Md[r] if deferred else (Md[r] * 1e3).contiguous(), G0d, 1.0)
        h.accumulate()
        if captured == "fresh":
            h.reset()
        stream.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            for r in range(8):
                h.compute_G(Md[r], G0d, 1.0)
            h.accumulate()
        h.reset()
        graph.replay()
        graph.replay()
        out, S = h.finalize(allow_zero_sign=True)   # the launches are not counted on the host
        assert S == 0.0
        got = out.cpu().numpy() / 16.0
        h.close()
    assert np.abs(got - want).max() <= 1e-13 * np.abs(want).max()

"""fr_rotate_noalloc as callers use it: captured into their own graph, with profiling on. Exact
arithmetic: word for word."""
import numpy as np
import pytest

from paper_2604_00546_gb300 import fr
from test_gpu_twiddle_classes import CHAINS, _residues

pytestmark = pytest.mark.gpu


def test_capture_under_profiling_records_no_region():
    """A profiled context times its own calls; a rotation captured into the caller's graph leaves no
    events of the library in it. Level 8: the ModDown's conversion is a launch of its own."""
    torch = pytest.importorskip("torch")
    s = torch.cuda.Stream()
    ctx = fr.Context(device=0, log_n=12, q_bits=[60] + [50] * 8, p_bits=[60] * 3, dnum=3, scale_bits=50, ell=64, n1=8,
                     cuda_stream=s.cuda_stream)
    ctx.load_keys(ctx.keygen([3], 5))
    a = _residues(ctx.primes()[:9], ctx.N, 9)
    ref = ctx.rotate(ctx.import_ct(a, 8).upload(), 3).export()
    d_in = torch.from_numpy(a.view(np.int64)).to("cuda:0")
    out = torch.zeros_like(d_in)
    torch.cuda.synchronize()
    ctx.rotate_noalloc(d_in.data_ptr(), 8, 3, out.data_ptr())
    ctx.sync()
    assert np.array_equal(out.cpu().numpy().view(np.uint64), ref)
    out.zero_()
    torch.cuda.synchronize()
    ctx.profile(True)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s, capture_error_mode="thread_local"):
        ctx.rotate_noalloc(d_in.data_ptr(), 8, 3, out.data_ptr())
    assert ctx.profile_read("moddown") == (0.0, 0, 0)
    ctx.profile(False)
    g.replay()
    torch.cuda.synchronize()
    assert np.array_equal(out.cpu().numpy().view(np.uint64), ref)

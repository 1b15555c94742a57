"""fr_rotate_noalloc as callers use it: captured into their own graph, on buffers at any word. Exact
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


@pytest.mark.parametrize("in_off,out_off", [(0, 0), (0, 1), (1, 0), (1, 1), (None, 0), (None, 1)])
@pytest.mark.parametrize("log_n", [10, 11, 12, 13, 14, 16])
def test_any_word_address(log_n, in_off, out_off):
    """Input and output at any word, or in place (in_off None): buffers off a 16-byte boundary leave
    the kernels that move 16 bytes, and c1 is copied before the conversion reads it. The words around
    the buffers keep their contents."""
    torch = pytest.importorskip("torch")
    ctx = fr.Context(device=0, log_n=log_n, dnum=2, ell=64, n1=8, **CHAINS["class1"])
    ctx.load_keys(ctx.keygen([3], 5))
    a = _residues(ctx.primes()[:3], ctx.N, 9)
    ref = ctx.rotate(ctx.import_ct(a, 2).upload(), 3).export()
    guard = np.int64(-7)

    def buffer(off, words=None):
        b = torch.full((a.size + 4,), int(guard), dtype=torch.int64, device="cuda:0")
        if words is not None:
            b[2 + off: 2 + off + a.size] = torch.from_numpy(words.view(np.int64).ravel()).to("cuda:0")
        return b

    d_out = buffer(out_off, a if in_off is None else None)
    d_in = d_out if in_off is None else buffer(in_off, a)
    torch.cuda.synchronize()
    ctx.rotate_noalloc(d_in.data_ptr() + 8 * (2 + (out_off if in_off is None else in_off)), 2, 3,
                       d_out.data_ptr() + 8 * (2 + out_off))
    ctx.sync()
    got = d_out.cpu().numpy()
    assert np.array_equal(got[2 + out_off: 2 + out_off + a.size].view(np.uint64).reshape(a.shape), ref)
    assert (got[: 2 + out_off] == guard).all() and (got[2 + out_off + a.size:] == guard).all()
    if in_off is not None:
        assert np.array_equal(d_in.cpu().numpy()[2 + in_off: 2 + in_off + a.size].view(np.uint64).reshape(a.shape), a)

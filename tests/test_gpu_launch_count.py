"""fr_launch_count counts kernels: a transform is one by the cluster kernel (rings up to 2^13 without
primes of class 2, and shape 4 at 2^14) and two by the two-pass kernels. Expected figures are the
calls' kernels, t a transform: upload and export t; rescale 2 t and the lift; rotation 4 t, two
conversions and the inner product; product the same and the tensor product; rotation on caller's
buffers 5 t, two conversions and the inner product."""
import numpy as np
import pytest

from paper_2604_00546_gb300 import fr
from test_gpu_twiddle_classes import CHAINS, _residues

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("log_n,chain,shape,t", [(10, "class1", None, 1), (12, "class0", None, 1), (13, "mixed", None, 2),
                                                 (12, "class2", None, 2), (14, "class1", 4, 1), (14, "class1", 0, 2),
                                                 (14, "class1", 5, 2), (15, "class0", 4, 2)])
def test_counts_of_the_calls(log_n, chain, shape, t):
    torch = pytest.importorskip("torch")
    ctx = fr.Context(device=0, log_n=log_n, dnum=2, ell=64, n1=8, **CHAINS[chain])
    n0 = ctx.launch_count()
    ctx.load_keys(ctx.keygen([3], 5))
    assert ctx.launch_count() - n0 == 2   # one conversion a key: the relinearisation's and one rotation's
    if shape is not None:
        ctx.ntt_set_shapes([shape] * 4)
    a = _residues(ctx.primes()[:3], ctx.N, 9)

    def count(f):
        n = ctx.launch_count()
        r = f()
        return ctx.launch_count() - n, r

    n, ct = count(lambda: ctx.import_ct(a, 2).upload())
    assert n == t
    assert count(ct.export)[0] == t
    assert count(lambda: ctx.rescale(ct))[0] == 2 * t + 1
    assert count(lambda: ctx.rotate(ct, 3))[0] == 4 * t + 3
    assert count(lambda: ctx.mul_relin(ct, ct))[0] == 4 * t + 4
    d = torch.from_numpy(a.view(np.int64)).to("cuda:0")
    torch.cuda.synchronize()
    assert count(lambda: ctx.rotate_noalloc(d.data_ptr(), 2, 3, d.data_ptr()))[0] == 5 * t + 3
    ctx.sync()

"""GPU parity of the single-launch cluster transform at N = 2^14, its largest ring (8 CTAs of 2048
elements, above the default shared-memory limit), which otherwise runs only where the tuner picks it:
rotation, rescale and product on chains of every twiddle class, and the threshold, whose transforms
end in the fused epilogues; and of the smallest rings where its primes rule it out. Exact arithmetic:
word for word."""
import numpy as np
import pytest

import oracle
from paper_2604_00546_gb300 import fr
from test_gpu_twiddle_classes import CHAINS, _residues

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chain", sorted(CHAINS))
def test_cluster_transform_at_its_largest_ring(chain):
    p = CHAINS[chain]
    ctx = fr.Context(device=0, log_n=14, dnum=2, ell=64, n1=8, **p)
    ctx.load_keys(ctx.keygen([3], 0x7D00))
    oc = oracle.Ctx(14, p["q_bits"], p["p_bits"], 2, p["scale_bits"])
    ok = oc.keygen(0x7D00)
    top = oc.top
    a, b = (_residues(ctx.primes()[: top + 1], ctx.N, 0x7D10 + s) for s in (1, 2))
    ctx.ntt_set_shapes([4] * 4)
    ca, cb = ctx.import_ct(a, top).upload(), ctx.import_ct(b, top).upload()
    assert np.array_equal(ctx.rotate(ca, 3).export(), ok.rotate(a, top, 3))
    assert np.array_equal(ctx.rescale(ca).export(), oc.rescale(a, top))
    assert np.array_equal(ctx.mul_relin(ca, cb).export(), ok.mul_relin(a, b, top))


@pytest.mark.parametrize("bits", [45, 52], ids=["class0", "class1"])
def test_threshold_by_cluster_transforms(bits):
    q_bits, p_bits = [bits + 2] + [bits] * 7, [bits + 2] * 3
    ctx = fr.Context(device=0, log_n=14, q_bits=q_bits, p_bits=p_bits, dnum=3, scale_bits=bits - 4, ell=64, n1=8,
                     cheb_degree=27, threshold=0.5)
    ctx.load_keys(ctx.keygen([], 92))
    oc = oracle.Ctx(14, q_bits, p_bits, 3, bits - 4)
    a = _residues(ctx.primes()[: oc.top + 1], ctx.N, 192)
    ctx.ntt_set_shapes([4] * 4)
    got = ctx.chebyshev(ctx.import_ct(a, oc.top).upload())
    assert np.array_equal(got.export(), oc.keygen(92).cheb_eval(a, oc.top, 27, 0.5))


@pytest.mark.parametrize("chain", ["class2", "mixed"])
@pytest.mark.parametrize("log_n", [10, 11])
def test_small_rings_without_the_cluster_kernel(chain, log_n):
    """Primes it does not take: the two-pass kernels at their smallest tiles."""
    p = CHAINS[chain]
    ctx = fr.Context(device=0, log_n=log_n, dnum=2, ell=64, n1=8, **p)
    ctx.load_keys(ctx.keygen([3], 0x7E00))
    oc = oracle.Ctx(log_n, p["q_bits"], p["p_bits"], 2, p["scale_bits"])
    ok = oc.keygen(0x7E00)
    top = oc.top
    a, b = (_residues(ctx.primes()[: top + 1], ctx.N, 0x7E10 + s) for s in (1, 2))
    ca, cb = ctx.import_ct(a, top).upload(), ctx.import_ct(b, top).upload()
    assert np.array_equal(ctx.rotate(ca, 3).export(), ok.rotate(a, top, 3))
    assert np.array_equal(ctx.rescale(ca).export(), oc.rescale(a, top))
    assert np.array_equal(ctx.mul_relin(ca, cb).export(), ok.mul_relin(a, b, top))

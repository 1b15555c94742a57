"""GPU parity of the NTT's twiddle classes: the butterfly's product and its ranges depend on the
prime (see mul_tw), so rotation, rescale and ct x ct product are checked bit for bit against the
oracle on chains of every class and on a mixed one, at the ring sizes with their own kernels,
with 8 and with 16 residues a thread where both exist. Exact arithmetic: no tolerance."""
import numpy as np
import pytest

import oracle
from paper_2604_00546_gb300 import fr

pytestmark = pytest.mark.gpu

CHAINS = {
    "class0": dict(q_bits=[51, 50, 45], p_bits=[51, 51], scale_bits=45),
    "class1": dict(q_bits=[60, 52, 55], p_bits=[58, 59], scale_bits=52),
    "class2": dict(q_bits=[36, 34, 34], p_bits=[36, 36], scale_bits=30),
    "mixed": dict(q_bits=[60, 50, 34], p_bits=[52, 60], scale_bits=34),
}


def _residues(primes, N, seed):
    """[2][limbs][N]: random residues with runs at both ends of the range."""
    rng = np.random.default_rng(seed)
    w = np.empty((2, len(primes), N), dtype=np.uint64)
    for i, q in enumerate(primes):
        w[:, i] = rng.integers(0, q, (2, N), dtype=np.uint64)
        w[:, i, : N // 8] = q - 1
        w[:, i, N // 8: N // 4] = 0
    return w


@pytest.mark.parametrize("log_n", [12, 13, 14, 15, 16])
@pytest.mark.parametrize("chain", sorted(CHAINS))
def test_transforms_of_every_class(chain, log_n):
    p = CHAINS[chain]
    ctx = fr.Context(device=0, log_n=log_n, dnum=2, ell=64, n1=8, **p)
    seed = 0x7C00 + log_n
    ctx.load_keys(ctx.keygen([3], seed))
    oc = oracle.Ctx(log_n, p["q_bits"], p["p_bits"], 2, p["scale_bits"])
    ok = oc.keygen(seed)
    top = oc.top
    a, b = (_residues(ctx.primes()[: top + 1], ctx.N, seed + s) for s in (1, 2))
    rot, rs, mul = ok.rotate(a, top, 3), oc.rescale(a, top), ok.mul_relin(a, b, top)
    for shape in ([0, 5] if log_n >= 14 else [0]):
        ctx.ntt_set_shapes([shape] * 4)
        ca, cb = ctx.import_ct(a, top).upload(), ctx.import_ct(b, top).upload()
        assert np.array_equal(ctx.rotate(ca, 3).export(), rot), shape
        assert np.array_equal(ctx.rescale(ca).export(), rs), shape
        assert np.array_equal(ctx.mul_relin(ca, cb).export(), mul), shape


@pytest.mark.parametrize("words_off", [0, 1])
def test_noalloc_rotation_on_any_word_address(words_off):
    """The caller's output buffer need not start on a 16-byte boundary."""
    torch = pytest.importorskip("torch")
    p = CHAINS["class1"]
    ctx = fr.Context(device=0, log_n=14, dnum=2, ell=64, n1=8, **p)
    ctx.load_keys(ctx.keygen([3], 5))
    ctx.ntt_set_shapes([5] * 4)
    a = _residues(ctx.primes()[:3], ctx.N, 9)
    ref = ctx.rotate(ctx.import_ct(a, 2).upload(), 3).export()
    d_in = torch.from_numpy(a.view(np.int64)).to("cuda:0")
    buf = torch.zeros(a.size + 2, dtype=torch.int64, device="cuda:0")
    torch.cuda.synchronize()
    ctx.rotate_noalloc(d_in.data_ptr(), 2, 3, buf.data_ptr() + 8 * words_off)
    ctx.sync()
    got = buf[words_off: words_off + a.size].cpu().numpy().view(np.uint64).reshape(a.shape)
    assert np.array_equal(got, ref)


@pytest.mark.parametrize("n_q,n_p", [(5, 5), (7, 6), (8, 8)])
@pytest.mark.parametrize("log_n", [11, 14])
def test_base_conversion_of_wide_digits(log_n, n_q, n_p):
    """One digit of up to 8 limbs, up to 8 special primes, 50- and 60-bit targets: the sums of
    every number of sources, without and with the rescale's lift (mul_relin, then rescale)."""
    p = dict(q_bits=[60] + [50, 60, 45] * 3, p_bits=[60, 60, 59, 60] * 2, scale_bits=45)
    p["q_bits"], p["p_bits"] = p["q_bits"][:n_q], p["p_bits"][:n_p]
    ctx = fr.Context(device=0, log_n=log_n, dnum=1, ell=64, n1=8, **p)
    ctx.load_keys(ctx.keygen([3], 77))
    oc = oracle.Ctx(log_n, p["q_bits"], p["p_bits"], 1, p["scale_bits"])
    ok = oc.keygen(77)
    top = oc.top
    a, b = (_residues(ctx.primes()[: top + 1], ctx.N, 177 + s) for s in (1, 2))
    ca, cb = ctx.import_ct(a, top).upload(), ctx.import_ct(b, top).upload()
    for l in (top, top - 1):
        x = np.ascontiguousarray(a[:, : l + 1])
        assert np.array_equal(ctx.rotate(ctx.import_ct(x, l).upload(), 3).export(), ok.rotate(x, l, 3)), l
    mul = ok.mul_relin(a, b, top)
    got = ctx.mul_relin(ca, cb)
    assert np.array_equal(got.export(), mul)
    assert np.array_equal(ctx.rescale(got).export(), oc.rescale(mul, top))


@pytest.mark.parametrize("log_n", [11, 13, 15])
@pytest.mark.parametrize("bits", [34, 45, 52], ids=["class2", "class0", "class1"])
def test_threshold_of_every_class(bits, log_n):
    """The whole threshold (products relinearised and rescaled through one transform, leaves, tree) on a
    chain of each class, at rings that run the cluster kernel, the two-pass kernels and, for class 2,
    the 8-residue fallback."""
    q_bits, p_bits = [bits + 2] + [bits] * 7, [bits + 2] * 3
    ctx = fr.Context(device=0, log_n=log_n, q_bits=q_bits, p_bits=p_bits, dnum=3, scale_bits=bits - 4, ell=64, n1=8,
                     cheb_degree=27, threshold=0.5)
    ctx.load_keys(ctx.keygen([], 91))
    oc = oracle.Ctx(log_n, q_bits, p_bits, 3, bits - 4)
    ok = oc.keygen(91)
    a = _residues(ctx.primes()[: oc.top + 1], ctx.N, 191)
    for shape in ([0, 5] if log_n >= 14 else [0]):
        ctx.ntt_set_shapes([shape] * 4)
        got = ctx.chebyshev(ctx.import_ct(a, oc.top).upload())
        assert np.array_equal(got.export(), ok.cheb_eval(a, oc.top, 27, 0.5)), shape

"""GPU parity on chains with 61-bit primes, the largest a context takes: their 30-bit halves reach 31
bits, so only four products, not eight, sum in 64 bits. The single-query and the batched MAC (splits of
the ring, of the pipeline, a ragged one and one with more than 64 baby steps), with the baby steps in
Q_l and in Q_l u P, and base conversions of up to eight 61-bit sources. Exact: word for word."""
import numpy as np
import pytest

import oracle
from paper_2604_00546_gb300 import fr
from paper_2604_00546_gb300 import workloads as W
from test_gpu_twiddle_classes import _residues

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ell,n1,pq", [(64, 8, 0), (128, 12, 0), (512, 32, 0), (512, 32, 1), (512, 80, 1)])
def test_diagonal_mac(ell, n1, pq):
    p = dict(log_n=11, q_bits=[61, 45, 61], p_bits=[61, 61], dnum=2, scale_bits=45)
    ctx = fr.Context(device=0, ell=ell, n1=n1, hoist_babies=pq, **p)
    keys = ctx.keygen(ctx.required_rotations(fr.FR_MODE_SCORES), 0x61)
    ctx.load_keys(keys)
    ok = oracle.Ctx(*p.values()).keygen(0x61)
    T = W.templates(ctx.n, ell, 21)
    db = ctx.load_db(T)
    qv = W.templates(3, ell, 22).astype(np.float64)
    cts = [ctx.encrypt(keys, q, 30 + b) for b, q in enumerate(qv)]
    oqs = [ok.encrypt(np.tile(q, ctx.n // ell), 30 + b) for b, q in enumerate(qv)]
    ref = [(ok.bsgs_scores_pq(o, T, ell, n1, pq=True) if pq else ok.bsgs_scores(o, T, ell, n1))[0] for o in oqs]
    assert np.array_equal(ctx.match(db, cts[0], fr.FR_MODE_SCORES)[0].export(), ref[0])
    for b, out in enumerate(ctx.match_batch(db, cts, fr.FR_MODE_SCORES)):
        assert np.array_equal(out[0].export(), ref[b]), b


@pytest.mark.parametrize("n", [5, 8])
@pytest.mark.parametrize("log_n", [11, 14])
def test_conversions_of_wide_digits(log_n, n):
    p = dict(log_n=log_n, q_bits=[61] * n, p_bits=[61] * n, dnum=1, scale_bits=45)
    ctx = fr.Context(device=0, ell=64, n1=8, **p)
    ctx.load_keys(ctx.keygen([3], 77))
    oc = oracle.Ctx(*p.values())
    ok = oc.keygen(77)
    a, b = (_residues(ctx.primes()[:n], ctx.N, 177 + s) for s in (1, 2))
    ca, cb = ctx.import_ct(a, n - 1).upload(), ctx.import_ct(b, n - 1).upload()
    assert np.array_equal(ctx.rotate(ca, 3).export(), ok.rotate(a, n - 1, 3))
    mul = ctx.mul_relin(ca, cb)
    ref = ok.mul_relin(a, b, n - 1)
    assert np.array_equal(mul.export(), ref)
    assert np.array_equal(ctx.rescale(mul).export(), oc.rescale(ref, n - 1))

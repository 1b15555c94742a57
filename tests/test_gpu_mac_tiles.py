"""GPU parity of the single-query MAC over the tiled diagonals: splits whose staged baby steps need
64, 32 and 16 points a CTA, ragged last giant steps, batches of eight that do not divide the split, a
single giant step, and the chunks in which diagonals are encoded (ell not a multiple of one).
Score ciphertexts are checked bit for bit against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2604_00546_gb300 import fr
from paper_2604_00546_gb300 import workloads as W

pytestmark = pytest.mark.gpu

QB, PB, DNUM, SB = [60, 45, 50], [60, 60], 3, 45


@pytest.mark.parametrize("log_n,ell,n1", [(10, 512, 129), (11, 512, 300), (11, 128, 128), (12, 128, 12), (12, 64, 8),
                                          (13, 256, 40)])
@pytest.mark.parametrize("tier", [1, 2, 3])
def test_scores_over_tiles(log_n, ell, n1, tier):
    ctx = fr.Context(device=0, log_n=log_n, q_bits=QB, p_bits=PB, dnum=DNUM, scale_bits=SB, ell=ell, n1=n1)
    seed = 0x3A00 + n1
    keys = ctx.keygen(ctx.required_rotations(fr.FR_MODE_SCORES), seed)
    ctx.load_keys(keys)
    ok = oracle.Ctx(log_n, QB, PB, DNUM, SB).keygen(seed)
    T = W.templates(ctx.n + 3, ell, seed)
    q = T[1].astype(np.float64)
    got = ctx.match(ctx.load_db(T, tier=tier), ctx.encrypt(keys, q, 4), fr.FR_MODE_SCORES)
    ref, lvl = ok.match(ok.encrypt(np.tile(q, ctx.n // ell), 4), T, ell, n1, fr.FR_MODE_SCORES)
    assert len(got) == len(ref) == 2
    for g in range(2):
        assert got[g].level == lvl
        assert np.array_equal(got[g].export(), ref[g]), g


@pytest.mark.parametrize("scale", [0.0, 1e-30, 1e-14, 3e3])
def test_encoder_rounding_of_extreme_templates(scale):
    """The encoder's rounding works on the mantissa bits: templates far below and above unit length
    (coefficients that round to 0 or +-1, and ones with more than 53 bits) match the oracle's words."""
    log_n, ell, n1 = 11, 64, 8
    ctx = fr.Context(device=0, log_n=log_n, q_bits=QB, p_bits=PB, dnum=DNUM, scale_bits=SB, ell=ell, n1=n1)
    keys = ctx.keygen(ctx.required_rotations(fr.FR_MODE_SCORES), 5)
    ctx.load_keys(keys)
    ok = oracle.Ctx(log_n, QB, PB, DNUM, SB).keygen(5)
    T = (W.templates(ctx.n, ell, 6) * scale).astype(np.float32)
    T[1] = 0.0
    T[2, ::3] *= -1.0
    q = W.templates(1, ell, 8)[0].astype(np.float64)
    ref, _ = ok.match(ok.encrypt(np.tile(q, ctx.n // ell), 4), T, ell, n1, fr.FR_MODE_SCORES)
    for tier in (1, 3):
        got = ctx.match(ctx.load_db(T, tier=tier), ctx.encrypt(keys, q, 4), fr.FR_MODE_SCORES)
        assert np.array_equal(got[0].export(), ref[0]), tier

"""The NTT tuner chooses between kernels, not between names of one: shapes 2 and 3 run the kernels of
0 and 1, so they report those times and are never chosen, whatever the timing noise."""
import pytest

from paper_2604_00546_gb300 import fr

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("log_n", [15, 16])
def test_aliases_are_not_chosen(log_n):
    for _ in range(3):
        ctx = fr.Context(device=0, log_n=log_n, q_bits=[60, 50, 50], p_bits=[60], dnum=1, scale_bits=50, ell=64, n1=8)
        t = ctx.ntt_tuning()
        for b in range(4):
            us = t["us"][b]
            assert us[2] == us[0] > 0 and us[3] == us[1] > 0
            assert t["shapes"][b] in (0, 1, 5)

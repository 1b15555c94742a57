"""A database load that fails part way (injected allocation failures, host side) gives back the
device memory it had taken, and the next load works."""
import numpy as np
import pytest

from paper_2604_00546_gb300 import fr
from paper_2604_00546_gb300 import workloads as W

pytestmark = pytest.mark.gpu

LOADS = ["plain diagonals", "integer coefficients", "encrypted, pre-rotated", "encrypted, rotated here"]


@pytest.mark.parametrize("kind", LOADS)
def test_failed_load_returns_its_memory(kind):
    torch = pytest.importorskip("torch")
    ell, n1 = 64, 8
    ctx = fr.Context(device=0, log_n=12, q_bits=[60, 45, 45], p_bits=[60, 60], dnum=2, scale_bits=45, ell=ell, n1=n1)
    neg = [-j for j in range(n1, ell, n1)]
    keys = ctx.keygen(sorted(set(ctx.required_rotations(fr.FR_MODE_SCORES)) | set(neg)), 3)
    ctx.load_keys(keys)
    T = W.templates(ctx.n, ell, 4)
    if kind in LOADS[:2]:
        load = lambda: ctx.load_db(T, tier=1 if kind == LOADS[0] else 3)
    else:
        pre = kind == LOADS[2]
        E = ctx.encrypt_db(keys, T, 2, 5, prerotate=pre)
        load = lambda: ctx.load_db_encrypted(E, len(T), prerotated=pre)
    q = ctx.encrypt(keys, W.templates(1, ell, 8)[0].astype(np.float64), 6)
    db = load()
    ref = ctx.match(db, q, fr.FR_MODE_SCORES)[0].export()
    size = db.info()["bytes"]
    del db
    ctx.sync()
    free = torch.cuda.mem_get_info()[0]
    for _ in range(6):
        for after in ((0,) if kind == LOADS[1] else (0, 1)):   # scratch the load allocates
            ctx.inject_alloc_failure(after)
            try:
                with pytest.raises(fr.FrError) as e:
                    load()
                assert e.value.status == fr.FR_ERR_HBM_BUDGET
            finally:
                ctx.inject_alloc_failure(-1)
    assert free - torch.cuda.mem_get_info()[0] < size   # the failed loads together keep less than one
    assert np.array_equal(ctx.match(load(), q, fr.FR_MODE_SCORES)[0].export(), ref)

"""GPU parity of the f32 pots' scorer (logits computed once, tiles of 16, 32 or 64 rows and keys) against the CPU checker,
at the edges of its tiles, channel stages, row batches and unit groups.  Eq. 2, Sec. 3.3.1."""
import numpy as np
import pytest

from paper_2410_01518_b200 import inputs, ipot
from parity import compare_cycle, gpu_cycle

pytestmark = pytest.mark.gpu

SHAPES = [
    # (rows used, cap_rows, Hq, Hkv, d, layers, batch): one row and one tile of keys, 15 to 17 and 63 to 65 rows and keys,
    # channel counts that end inside a stage of 32, more than 256 rows (two weight batches), several groups of units
    (17, 1, 1, 1, 32, 1, 1), (63, 5, 3, 1, 40, 1, 2), (65, 16, 4, 4, 64, 1, 1), (513, 17, 4, 2, 72, 2, 1), (1000, 65, 8, 2, 256, 1, 1),
    (4097, 64, 8, 8, 96, 4, 2), (2999, 63, 32, 4, 128, 6, 2),
]


@pytest.mark.parametrize("case", range(len(SHAPES)))
def test_f32_scorer_shapes(case):
    n, P, Hq, Hkv, d, L, B = SHAPES[case]
    cfg = inputs.small_config(cfg_id=950 + case, pot_size=n + 1, keep=n // 2, nuc_slots=n // 4, cap_rows=P, Hq=Hq, Hkv=Hkv, d=d,
                              dtype="f32", layers=L, batch=B)
    t = inputs.make_cycle(cfg)
    if case % 2:
        t["K_cap"] = inputs.make_kcap(cfg)
    units = None if cfg.units <= 16 else np.linspace(0, cfg.units - 1, 16).astype(np.int32)
    same, cnt = compare_cycle(cfg, t, gpu_cycle(cfg, t, ipot.IPOT_SCORER_AUTO, n=n), n=n, units=units)
    assert same >= cnt - 1


@pytest.mark.parametrize("d,dtype,P", [(64, "f32", 16), (128, "f32", 64), (96, "bf16", 16)])
def test_logits_below_the_range_of_fp32(d, dtype, P):
    """Finite inputs whose logits overflow to -inf for whole tiles of keys: those keys score 0 and the others as if they
    were not there."""
    cfg = inputs.small_config(cfg_id=960, pot_size=1300, keep=400, nuc_slots=100, cap_rows=P, Hq=8, Hkv=2, d=d, dtype=dtype, layers=2)
    t = inputs.make_cycle(cfg)
    Q, K = (inputs.widen(t[k], dtype).astype(np.float32) for k in ("Q", "K"))
    Q[..., 0], K[..., 0] = 1e10, 0
    K[..., 128:700, 0] = -1e30
    t["Q"], t["K"] = inputs.store(Q, dtype), inputs.store(K, dtype)
    gpu = gpu_cycle(cfg, t)
    same, cnt = compare_cycle(cfg, t, gpu)
    assert same >= cnt - 1 and (gpu[0][:, 128:700] == 0).all()

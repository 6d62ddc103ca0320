"""GPU parity of the in-place gather of the survivors (Appendix B "KV-cache compression") at the edges of its chunks of
about 16 KiB of whole rows, against the CPU checker: rows are moved, so every byte must match."""
import pytest

from paper_2410_01518_b200 import inputs, ipot
from parity import compare_cycle, gpu_cycle

pytestmark = pytest.mark.gpu

SHAPES = [
    # (d, dtype, rows used, keep, first row of a deferred chunk or None): rows per chunk 256, 204 (of 16320 bytes), 64, 16;
    # keep one below, at and above whole chunks, all but one slot kept (long waits for the chunk before), few kept of many
    # (sources of a chunk's slots in one early chunk), chunk rows on both sides of the pot's
    (32, "bf16", 700, 257, None), (40, "bf16", 500, 203, 100), (40, "bf16", 500, 205, None), (128, "bf16", 130, 129, None),
    (128, "bf16", 4096, 64, None), (128, "bf16", 2001, 1999, 1000), (128, "bf16", 1000, 191, 256), (256, "f32", 400, 17, None),
    (256, "f32", 300, 299, 16), (64, "f32", 5000, 4097, None), (128, "bf16", 9000, 8990, 0),
]


@pytest.mark.parametrize("rope", [False, True])
@pytest.mark.parametrize("case", range(len(SHAPES)))
def test_gather_chunk_edges(case, rope):
    d, dtype, n, keep, first = SHAPES[case]
    if rope and (d * (4 if dtype == "f32" else 2)) % 32:
        pytest.skip("the rotary mode takes rows of whole 32-byte pairs")
    cfg = inputs.small_config(cfg_id=860 + case, pot_size=n + 3, keep=keep, nuc_slots=keep // 3, cap_rows=4, Hq=6, Hkv=3, d=d,
                              dtype=dtype, batch=2)
    t = inputs.make_cycle(cfg)
    if rope:
        t["rope"] = (*inputs.make_rope_table(cfg.pot_size, d, dtype), case % 2 == 1)
    gpu = gpu_cycle(cfg, t, ipot.IPOT_SCORER_AUTO, n=n, deferred_from=first)
    same, cnt = compare_cycle(cfg, t, gpu, n=n)
    assert cnt == cfg.units and same >= cnt - 1


@pytest.mark.parametrize("rope", [False, True])
@pytest.mark.parametrize("in_place,first", [(0, None), (63, None), (64, None), (65, None), (192, 192), (192, 191), (192, 100), (192, 0), (256, None)])
def test_gather_rows_in_place(in_place, first, rope):
    """The most novel rows are the first ones, so they keep their slots: chunks of 64 rows that stay, that end in a row that
    moves, that reach into a deferred chunk (whose rows have to be copied all the same), and a gather that moves nothing."""
    n, keep = 600, 256
    cfg = inputs.small_config(cfg_id=880, pot_size=n, keep=keep, nuc_slots=keep, cap_rows=4, Hq=6, Hkv=3, d=128, dtype="bf16", batch=2)
    t = inputs.make_cycle(cfg)
    t["aux"][:, :in_place] += 2   # (the others are in [0, 1))
    t["aux"][:, in_place:in_place + 1] = -1
    if rope:
        t["rope"] = (*inputs.make_rope_table(cfg.pot_size, 128, "bf16"), False)
    gpu = gpu_cycle(cfg, t, ipot.IPOT_SCORER_AUTO, n=n, deferred_from=first)
    same, cnt = compare_cycle(cfg, t, gpu, n=n)
    assert same == cnt == cfg.units

"""GPU parity of the in-place gather of the survivors (Appendix B "KV-cache compression") at the edges of its chunks of
about 16 KiB of whole rows, against the CPU checker: rows are moved, so every byte must match."""
import numpy as np
import pytest
import torch

from paper_2410_01518_b200 import inputs, ipot
from parity import check_rotated, compare_cycle, from_dev_bits, gpu_cycle, make_pot, to_dev

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


def test_gather_wait_that_runs_out_leaves_rows_and_rotated_copy_together():
    """Chunk 0 of every tensor never reports that it has been read (a test hook): the chunk behind it cannot be overwritten, the
    launch ends by itself with IPOT_E_TIMEOUT, the rows it did not move still have their own rotated rows beside them, and
    after ipot_reset the same pot runs a correct cycle.  The scorers' limit does not apply to the gather: with it as short as
    it may be set, a cycle of a pot whose scorer has no waits ends without a status."""
    n, keep, d = 600, 500, 128
    cfg = inputs.small_config(cfg_id=890, pot_size=n, keep=keep, nuc_slots=0, cap_rows=4, Hq=3, Hkv=3, d=d, dtype="bf16")
    t = inputs.make_cycle(cfg)
    t["rope"] = (*inputs.make_rope_table(n, d, "bf16"), False)
    want = gpu_cycle(cfg, t, ipot.IPOT_SCORER_SIMT)
    Kd, Vd, Qd, cos, sin = (to_dev(x, "bf16") for x in (t["K"], t["V"], t["Q"], *t["rope"][:2]))
    h = make_pot(cfg)
    try:
        ipot.ipot_set_scorer(h, ipot.IPOT_SCORER_SIMT)
        ipot.ipot_enable_rope(h, cos, sin, ipot.IPOT_ROPE_HALF)
        ipot.ipot_set_tuning(h, ipot.IPOT_TUNE_WAIT_LIMIT_NS, 1000)
        for withheld in (-1, 0, -1):
            ipot.ipot_set_tuning(h, ipot.IPOT_TUNE_TEST_WITHHOLD_CHUNK, withheld)
            ipot.ipot_reset(h)
            ipot.ipot_append_chunk(h, Kd, Vd, n)
            if withheld < 0:
                ipot.ipot_score_and_compress(h, Qd, cfg.cap_rows, None)
                torch.cuda.synchronize()
                K = from_dev_bits(ipot.device_array(ipot.ipot_view(h)[0], (cfg.units, n, d), "bf16")[:, :keep], "bf16")
                rot = from_dev_bits(ipot.device_array(ipot.ipot_view_rope(h), (cfg.units, n, d), "bf16")[:, :keep], "bf16")
                assert (K == want[2]).all() and (rot == want[4]).all()
            else:
                assert ipot.ipot_sync_status(h) == 0   # (nothing before ran out)
                ipot.ipot_score_and_compress(h, Qd, cfg.cap_rows, None)
                assert ipot.ipot_sync_status(h) == ipot.IPOT_E_TIMEOUT
                K = from_dev_bits(ipot.device_array(ipot.ipot_view(h)[0], (cfg.units, n, d), "bf16")[:, :keep], "bf16")
                rot = from_dev_bits(ipot.device_array(ipot.ipot_view_rope(h), (cfg.units, n, d), "bf16")[:, :keep], "bf16")
                assert (K != want[2]).any()            # some chunk did give up
                for unit in range(cfg.units):
                    check_rotated(rot[unit], K[unit], np.arange(keep), t["rope"], "bf16")
    finally:
        ipot.ipot_destroy(h)

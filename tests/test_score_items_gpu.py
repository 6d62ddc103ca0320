"""GPU parity of the item-dealt two-sweep tensor-core scorer (IPOT_SCORER_TENSOR_ITEMS) against the CPU checker, through
the C ABI, under the tolerances of tests/parity.py.  Eq. 2, Sec. 3.3.1."""
import numpy as np
import pytest
import torch

import oracle
from paper_2410_01518_b200 import inputs, ipot
from parity import compare_cycle, gpu_cycle, make_pot, to_dev

pytestmark = pytest.mark.gpu
ITEMS = ipot.IPOT_SCORER_TENSOR_ITEMS

SHAPES = [
    # (pot_size, rows used, cap_rows, Hq, Hkv, d, layers, batch): one tile and one key, tiles of 127 to 129 keys, jobs of
    # 1 to 8 tiles with a shorter last one, 1 to 8 row blocks (whole and ragged), fewer and more items than SMs, and rows of
    # one to four 64-channel blocks (whole, half and a quarter filled)
    (64, 33, 1, 1, 1, 32, 1, 1), (128, 127, 16, 8, 2, 128, 1, 1), (300, 128, 32, 4, 1, 128, 2, 1), (300, 129, 32, 4, 1, 40, 1, 2),
    (1000, 999, 33, 8, 2, 96, 3, 1), (2048, 2047, 43, 12, 4, 128, 2, 2), (4096, 4096, 64, 8, 2, 64, 8, 1),
    (3000, 2999, 64, 8, 1, 192, 2, 1), (1500, 1281, 48, 16, 2, 256, 3, 1), (2000, 1999, 19, 3, 3, 256, 4, 2),
    (1100, 1025, 128, 8, 1, 128, 1, 2), (16384, 16257, 64, 8, 1, 128, 1, 2), (4096, 4095, 32, 32, 8, 128, 24, 1), (700, 600, 3, 2, 2, 72, 1, 1),
]


@pytest.mark.parametrize("case", range(len(SHAPES)))
def test_items_shapes(case):
    pot, n, P, Hq, Hkv, d, L, B = SHAPES[case]
    cfg = inputs.small_config(cfg_id=900 + case, pot_size=pot, keep=n // 2, nuc_slots=n // 4, cap_rows=P, Hq=Hq, Hkv=Hkv, d=d,
                              dtype="bf16", layers=L, batch=B)
    t = inputs.make_cycle(cfg)
    gpu = gpu_cycle(cfg, t, ITEMS, n=n)
    units = None if cfg.units <= 24 else np.linspace(0, cfg.units - 1, 24).astype(np.int32)
    same, cnt = compare_cycle(cfg, t, gpu, n=n, units=units)
    assert same >= cnt - 1
    first = (n // 2) // 128 * 128    # keys of a deferred chunk are read where they lie: the same products in the same order
    got = gpu_cycle(cfg, t, ITEMS, n=n, deferred_from=first)
    assert all((a == b).all() for a, b in zip(got, gpu))


def test_items_logits_outside_the_default_range():
    """Keys of very different size: a row's logits reach hundreds of exponent steps above and below the reference of 0,
    so the general path has to find one, tile by tile, without losing a term."""
    cfg = inputs.small_config(cfg_id=930, pot_size=1024, keep=400, nuc_slots=0, cap_rows=32, Hq=4, Hkv=1, d=128, dtype="bf16", layers=2)
    t = inputs.make_cycle(cfg)
    K = inputs.widen(t["K"], "bf16").astype(np.float32)
    K[:, :, :, :32] *= 0.01
    K[:, :, :, 300:340] *= 60.0
    K[1] = K[1, :, :, :1] * 40.0 + 0.01 * K[1]     # every key of the second layer nearly the same long one
    t["K"] = inputs.store(K, "bf16")
    compare_cycle(cfg, t, gpu_cycle(cfg, t, ITEMS))


def test_items_wait_that_runs_out_ends_the_launch_and_the_pot_recovers():
    """One job's statistics are never reported (a test hook: the others' wait for them cannot end) and the wait limit is 2 ms:
    the launch ends by itself with IPOT_E_TIMEOUT, and the same pot then scores correctly with the hook off."""
    cfg = inputs.small_config(cfg_id=931, pot_size=2048, keep=400, nuc_slots=0, cap_rows=16, Hq=8, Hkv=2, d=96, dtype="bf16", layers=2)
    t = inputs.make_cycle(cfg)
    want = gpu_cycle(cfg, t, ITEMS)[0]
    h = make_pot(cfg)
    try:
        ipot.ipot_set_scorer(h, ITEMS)
        ipot.ipot_set_tuning(h, ipot.IPOT_TUNE_WAIT_LIMIT_NS, 2_000_000)
        ipot.ipot_set_tuning(h, ipot.IPOT_TUNE_TEST_WITHHOLD_RANK, 1)
        Kd, Vd, Qd = to_dev(t["K"], "bf16"), to_dev(t["V"], "bf16"), to_dev(t["Q"], "bf16")
        ipot.ipot_append_chunk(h, Kd, Vd, cfg.pot_size)
        ipot.ipot_score_only(h, Qd, cfg.cap_rows)
        assert ipot.ipot_sync_status(h) == ipot.IPOT_E_TIMEOUT
        ipot.ipot_set_tuning(h, ipot.IPOT_TUNE_TEST_WITHHOLD_RANK, -1)
        ipot.ipot_set_tuning(h, ipot.IPOT_TUNE_WAIT_LIMIT_NS, 200_000_000)
        ipot.ipot_score_only(h, Qd, cfg.cap_rows)
        torch.cuda.synchronize()
        sp, nb = ipot.ipot_last_scores(h)
        assert (ipot.device_array(sp, (cfg.units, nb), "f32").cpu().numpy() == want).all()
    finally:
        ipot.ipot_destroy(h)


@pytest.mark.parametrize("d", [72, 256])
@pytest.mark.parametrize("M", [63, 64, 65])
def test_items_query_tile_heights(M, d):
    """Up to 64 query rows are fetched as half a tile and multiplied as 64 columns, more as whole ones; the CaP's own keys join
    the denominators of the rows there are."""
    cfg = inputs.small_config(cfg_id=940 + M - 63, pot_size=1300, keep=500, nuc_slots=100, cap_rows=M, Hq=4, Hkv=4, d=d, dtype="bf16", layers=5, batch=2)
    t = inputs.make_cycle(cfg)
    t["K_cap"] = inputs.make_kcap(cfg, 0)
    same, cnt = compare_cycle(cfg, t, gpu_cycle(cfg, t, ITEMS, n=1290), n=1290)
    assert same >= cnt - 1


@pytest.mark.parametrize("n", [1025, 1100, 4096 + 127])
def test_items_ragged_last_tile_beside_references(n):
    """The last tile's keys are summed against the reference there is, or, where the sum is out of range, against their own:
    with keys small everywhere, large everywhere but in the last tile, and large only in it."""
    cfg = inputs.small_config(cfg_id=950, pot_size=n, keep=300, nuc_slots=0, cap_rows=48, Hq=4, Hkv=1, d=128, dtype="bf16", layers=3)
    t = inputs.make_cycle(cfg)
    K = inputs.widen(t["K"], "bf16").astype(np.float32)
    last = (n - 1) // 128 * 128
    K[1, :, :, :last] *= 50.0
    K[2, :, :, last:] *= 50.0
    t["K"] = inputs.store(K, "bf16")
    compare_cycle(cfg, t, gpu_cycle(cfg, t, ITEMS))


@pytest.mark.parametrize("d,other", [(40, ipot.IPOT_SCORER_SIMT), (72, ipot.IPOT_SCORER_SIMT), (96, ipot.IPOT_SCORER_WARP_MMA),
                                     (192, ipot.IPOT_SCORER_WARP_MMA), (256, ipot.IPOT_SCORER_WARP_MMA), (128, ipot.IPOT_SCORER_TENSOR)])
def test_items_are_as_exact_as_the_kernels_they_stand_in_for(d, other):
    """Error against 64 bits, 2-norm and largest, beside that of the scorer such a pot would have otherwise.  Both sum 32-bit
    exponentials of 32-bit logits, so the two differ by the luck of their rounding: a factor of 2 is allowed, where a
    polynomial of degree 4 and denominators as one rounded logarithm made it 3 to 5."""
    cfg = inputs.small_config(cfg_id=970, pot_size=4000, keep=1000, nuc_slots=0, cap_rows=32, Hq=8, Hkv=4, d=d, dtype="bf16", layers=2)
    t = inputs.make_cycle(cfg)
    Q = inputs.widen(t["Q"], "bf16").astype(np.float32)
    t["Q"] = inputs.store(Q + 2.5 * Q[:, :, :, :1], "bf16")    # a query head's rows share a direction
    ref = oracle.cycle(t["Q"], t["K"], t["V"], t["aux"], cfg.keep, 0)["u"]
    err = []
    for scorer in (ITEMS, other):
        u = gpu_cycle(cfg, t, scorer)[0].astype(np.float64)
        err.append((np.linalg.norm(u - ref) / np.linalg.norm(ref), np.abs(u / ref - 1).max()))
    assert err[0][0] <= 2 * err[1][0] and err[0][1] <= 2 * err[1][1], err


@pytest.mark.parametrize("units,n,P,Hq_per_kv,d,want", [
    (64, 8192, 16, 4, 128, ipot.IPOT_SCORER_TENSOR), (64, 8193, 16, 4, 128, ITEMS), (40, 8192, 129, 4, 128, ITEMS), (35, 9216, 32, 4, 128, ipot.IPOT_SCORER_TENSOR),
    (35, 9216, 33, 4, 128, ITEMS), (32, 10240, 16, 1, 64, ITEMS), (64, 6143, 16, 1, 64, ipot.IPOT_SCORER_TENSOR), (64, 6144, 16, 1, 64, ITEMS),
    (16, 12288, 33, 4, 128, ipot.IPOT_SCORER_TENSOR), (2, 300, 16, 1, 96, ITEMS)])
def test_automatic_choice(units, n, P, Hq_per_kv, d, want):
    """Both sides of every line of the automatic choice; the scores agree with those of the kernel that was not chosen."""
    g = torch.Generator(device="cuda").manual_seed(n)
    K = torch.randn((units, 1, 1, n, d), generator=g, device="cuda").bfloat16()
    Q = torch.randn((units, 1, Hq_per_kv, P, d), generator=g, device="cuda").bfloat16()
    u = []
    for scorer in (ipot.IPOT_SCORER_AUTO, ipot.IPOT_SCORER_WARP_MMA):
        h = ipot.ipot_create_ex(n, n // 4, units, Hq_per_kv, 1, d, nuc_slots=0, max_cap_rows=P)
        try:
            ipot.ipot_set_scorer(h, scorer)
            ipot.ipot_set_profiling(h, True)
            ipot.ipot_append_chunk(h, K, K, n)
            ipot.ipot_score_and_compress(h, Q, P, None)
            assert ipot.ipot_sync_status(h) == 0
            assert ipot.ipot_kernel_ms(h)[2] == (want if scorer == ipot.IPOT_SCORER_AUTO else scorer)
            u.append(ipot.device_array(ipot.ipot_last_scores(h)[0], (units, n), "f32").clone())
        finally:
            ipot.ipot_destroy(h)
    assert ((u[0] - u[1]).norm() / u[1].norm()).item() < 2e-6   # (two kernels within 1e-6 of the exact scores each)

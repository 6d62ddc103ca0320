"""GPU parity of the one-sweep tensor-core scorer (IPOT_SCORER_TENSOR) at the edges of its tiles and statistics, against the CPU
checker, through the C ABI, under the tolerances of tests/parity.py.  Eq. 2, Sec. 3.3.1."""
import numpy as np
import pytest
import torch

from paper_2410_01518_b200 import inputs, ipot
from parity import compare_cycle, gpu_cycle, make_pot, to_dev

pytestmark = pytest.mark.gpu
TC = ipot.IPOT_SCORER_TENSOR

SHAPES = [
    # (rows used, cap_rows, Hq, Hkv, d, layers, batch): a part of one half slab, its end and the key behind it, a last slab of one half,
    # more statistics than one look takes (16 per half of the item), 1 to 128 rows in a block at the ends of the 32-row
    # quarters, a second block of one row
    (2, 1, 1, 1, 64, 1, 1), (100, 32, 1, 1, 128, 1, 1), (128, 33, 1, 1, 128, 1, 1), (129, 64, 2, 2, 128, 1, 2), (256, 13, 5, 1, 64, 1, 1),
    (257, 24, 4, 1, 128, 2, 1), (385, 97, 1, 1, 128, 1, 1), (2047, 32, 8, 2, 128, 3, 1), (2999, 19, 12, 4, 128, 5, 3), (4097, 43, 3, 1, 128, 1, 1),
    (4353, 25, 5, 1, 128, 2, 1), (8193, 50, 6, 1, 64, 1, 1), (4096, 32, 32, 8, 128, 21, 1),
]


@pytest.mark.parametrize("case", range(len(SHAPES)))
def test_one_sweep_edges(case):
    n, P, Hq, Hkv, d, L, B = SHAPES[case]
    cfg = inputs.small_config(cfg_id=960 + case, pot_size=n + 3, keep=max(1, n // 2), nuc_slots=n // 4, cap_rows=P, Hq=Hq, Hkv=Hkv, d=d,
                              dtype="bf16", layers=L, batch=B)
    t = inputs.make_cycle(cfg)
    units = None if cfg.units <= 24 else np.linspace(0, cfg.units - 1, 24).astype(np.int32)
    same, cnt = compare_cycle(cfg, t, gpu_cycle(cfg, t, TC, n=n), n=n, units=units)
    assert same >= cnt - 1


@pytest.mark.parametrize("cap_keys", [False, True])
@pytest.mark.parametrize("n", [1024, 999])
@pytest.mark.parametrize("big", [None, 3, 20, 40, 70, 100, 127, 200, 400])
def test_one_sweep_logits_outside_the_default_range(big, n, cap_keys):
    """Exponentials are summed against the reference 0 until a warp's sums leave the comfortable range; a key of enormous logits
    in each piece of a tile, with tiny keys in front of it, makes every way of leaving it happen.  None: every logit
    of a row lies hundreds of exponent steps below 0."""
    cfg = inputs.small_config(cfg_id=990, pot_size=1024, keep=400, nuc_slots=0, cap_rows=20, Hq=4, Hkv=1, d=128, dtype="bf16", layers=2)
    t = inputs.make_cycle(cfg)
    K, Q = (inputs.widen(t[x], "bf16").astype(np.float32) for x in "KQ")
    if big is None:
        axis = np.zeros(cfg.d, np.float32)
        axis[5] = 60.0
        Q, K = Q + axis, K - axis
    else:
        K[:, :, :, big] *= 60.0
        K[1, :, :, :16] *= 0.01
    t["K"], t["Q"] = inputs.store(K, "bf16"), inputs.store(Q, "bf16")
    if cap_keys:
        t["K_cap"] = inputs.make_kcap(cfg)
    compare_cycle(cfg, t, gpu_cycle(cfg, t, TC, n=n), n=n)


def test_one_sweep_calls_of_different_row_counts_share_one_pot():
    """The statistics of a launch are told from those of the launches before by their sign; calls with fewer rows in between must
    leave no row with a sign that a later call takes for its own."""
    cfg = inputs.small_config(cfg_id=991, pot_size=3000, keep=400, nuc_slots=0, cap_rows=32, Hq=8, Hkv=2, d=128, dtype="bf16", layers=4)
    t = inputs.make_cycle(cfg)
    Q = inputs.widen(t["Q"], "bf16").astype(np.float32)
    h = make_pot(cfg)

    class Scores:
        pass

    def score(P, scale):
        q = to_dev(inputs.store(np.ascontiguousarray(Q[..., :P, :] * scale), "bf16"), "bf16")
        ipot.ipot_score_only(h, q, P)
        ipot.ipot_sync_status(h)
        addr, n = ipot.ipot_last_scores(h)
        s = Scores()
        s.__cuda_array_interface__ = {"shape": (cfg.units, n), "typestr": "<f4", "data": (addr, False), "version": 2}
        return torch.as_tensor(s, device="cuda").clone()
    try:
        ipot.ipot_set_scorer(h, TC)
        K, V = to_dev(t["K"], "bf16"), to_dev(t["V"], "bf16")
        ipot.ipot_append_chunk(h, K, V, cfg.pot_size)
        want = {P: score(P, 1.0) for P in (32, 1, 9, 17)}
        for P in (32, 1, 32, 9, 9, 17, 1, 1, 32, 17, 32):
            score(P if P == 32 else 1, 0.5)      # other numbers in between
            assert torch.equal(score(P, 1.0), want[P])
        for P, got in want.items():              # each row's probabilities sum to 1
            assert torch.allclose(got.sum(1), torch.full((cfg.units,), float(P * cfg.Hq // cfg.Hkv), device="cuda"), rtol=1e-4)
    finally:
        ipot.ipot_destroy(h)


@pytest.mark.parametrize("n,P,Hq,Hkv,d,L,B", [
    # one to four 64-channel blocks, the last one whole, a quarter, half or an eighth filled; a query tile of 64 or 128 rows, so
    # that two or three half slabs of keys are in flight beside one or two query tiles; ragged ends as above
    (2047, 16, 8, 2, 96, 3, 1), (2300, 40, 4, 1, 40, 4, 2), (700, 3, 2, 2, 72, 8, 1), (999, 5, 6, 2, 136, 6, 1), (3000, 33, 8, 4, 192, 3, 1),
    (900, 16, 8, 2, 192, 5, 1), (1500, 48, 16, 2, 256, 3, 1), (1281, 19, 3, 3, 256, 4, 2), (4096, 32, 16, 8, 256, 21, 1)])
def test_one_sweep_rows_of_other_sizes(n, P, Hq, Hkv, d, L, B):
    """Head dimensions that reach the kernel through the automatic choice; keys of a deferred chunk are read where they lie from whole
    slabs on, the same products in the same order, and a chunk that starts between two slabs agrees within the tolerance."""
    cfg = inputs.small_config(cfg_id=980 + d, pot_size=n, keep=n // 2, nuc_slots=n // 4, cap_rows=P, Hq=Hq, Hkv=Hkv, d=d, dtype="bf16", layers=L, batch=B)
    t = inputs.make_cycle(cfg)
    units = None if cfg.units <= 24 else np.linspace(0, cfg.units - 1, 24).astype(np.int32)
    gpu = gpu_cycle(cfg, t)
    same, cnt = compare_cycle(cfg, t, gpu, units=units)
    assert same >= cnt - 1
    got = gpu_cycle(cfg, t, deferred_from=256)
    assert all((a == b).all() for a, b in zip(got, gpu))
    compare_cycle(cfg, t, gpu_cycle(cfg, t, deferred_from=384), units=units)


@pytest.mark.parametrize("d", [40, 72, 96, 136, 192, 256])
@pytest.mark.parametrize("P", [15, 17, 33, 50])   # times four query heads: both sides of 64 and 128 rows, two row blocks
def test_one_sweep_cap_keys_join_the_softmax_of_every_row_size(d, P):
    """Both CaP-inclusive calls on head dimensions that reach the kernel through the automatic choice.  The CaP keys take a share of
    every denominator, so that the scores add up to less than the number of rows."""
    cfg = inputs.small_config(cfg_id=1000 + d + P, pot_size=1100, keep=500, nuc_slots=100, cap_rows=P, Hq=16, Hkv=4, d=d, dtype="bf16", layers=2)
    t = inputs.make_cycle(cfg)
    t["K_cap"] = inputs.make_kcap(cfg)
    gpu = gpu_cycle(cfg, t)
    same, cnt = compare_cycle(cfg, t, gpu)
    assert same >= cnt - 1
    M = P * cfg.G
    assert (gpu[0].sum(1) < M * (1 - 1e-3)).all()
    h = make_pot(cfg)
    try:
        ipot.ipot_set_profiling(h, True)
        K, V, Q, Kc = (to_dev(t[x], "bf16") for x in ("K", "V", "Q", "K_cap"))
        ipot.ipot_append_chunk(h, K, V, cfg.pot_size)
        ipot.ipot_score_only_cap(h, Q, Kc, P)
        assert ipot.ipot_sync_status(h) == 0
        u = ipot.device_array(ipot.ipot_last_scores(h)[0], (cfg.units, cfg.pot_size), "f32").cpu().numpy()
        assert (u == gpu[0]).all()
        ipot.ipot_reset(h)
        ipot.ipot_append_chunk(h, K, V, cfg.pot_size)
        ipot.ipot_score_and_compress_cap(h, Q, Kc, P, torch.from_numpy(t["aux"]).cuda())
        assert ipot.ipot_sync_status(h) == 0
        assert ipot.ipot_kernel_ms(h)[2] == TC
    finally:
        ipot.ipot_destroy(h)


def _axis_cycle(cfg, rows, base, far, where, far_cap):
    """Logits along one axis: keys of `base` binary orders (drawn), one of `far` at slot where[layer] (None: among the CaP keys);
    rows: the factors of the query rows."""
    t = inputs.make_cycle(cfg)
    r = np.random.default_rng(7)
    to_key = np.log(2.0) * np.sqrt(cfg.d) / 8.0
    K = 0.01 * inputs.widen(t["K"], "bf16").astype(np.float32)
    K[..., 3] = r.uniform(*base, size=K.shape[:-1]) * to_key
    Kc = 0.01 * inputs.widen(inputs.make_kcap(cfg), "bf16").astype(np.float32)
    Kc[..., 3] = r.uniform(*base, size=Kc.shape[:-1]) * to_key
    for layer, slot in enumerate(where):
        if slot is None:
            Kc[layer, :, :, -1, 3] = far * to_key
        else:
            K[layer, :, :, slot, 3] = far * to_key
    Q = np.zeros_like(inputs.widen(t["Q"], "bf16"), dtype=np.float32)
    Q[..., 3] = 8.0 * np.asarray(rows)
    t["K"], t["Q"] = inputs.store(K, "bf16"), inputs.store(Q, "bf16")
    if far_cap:
        t["K_cap"] = inputs.store(Kc, "bf16")
    return t


@pytest.mark.parametrize("d", [64, 128, 96, 256])
@pytest.mark.parametrize("far", [30, 61, 99, 103, 117, 119, 126, 131, 150, 180, 226])
@pytest.mark.parametrize("rows", ["one", "equal", "mixed"])
def test_one_sweep_keeps_probabilities_beside_a_far_key(rows, far, d):
    """Keys of 20 to 45 binary orders and one far above them, in the first, a middle and the last piece of a half slab, in other slabs
    and halves, in the ragged end and among the CaP keys: every probability that fp32 holds has to come out, and the survivors
    beside the far key are chosen by it."""
    factors = {"one": [1.0], "equal": [1.0] * 16, "mixed": [1.0] + [0.1, -0.1, 0.02] * 5}[rows]
    where = [0, 5, 60, 127, 130, 255, 300, 690, None]
    cfg = inputs.small_config(cfg_id=1200 + d, pot_size=700, keep=128, nuc_slots=0, cap_rows=len(factors), Hq=1, Hkv=1, d=d, dtype="bf16",
                              layers=len(where))
    scorer = TC if d in (64, 128) else ipot.IPOT_SCORER_AUTO
    for cap in (False, True):
        t = _axis_cycle(cfg, factors, (20, 45), far, where, cap)
        compare_cycle(cfg, t, gpu_cycle(cfg, t, scorer))


@pytest.mark.parametrize("d", [64, 128, 96, 256])
@pytest.mark.parametrize("top", [-5, -20, -39, -60, -89, -95, -130, -300])
def test_one_sweep_keeps_probabilities_below_a_low_maximum(top, d):
    """Every logit of the rows far below 0: what is less than 2^126 below the largest counts."""
    where = [0, 5, 127, 130, 300, 690, None]
    cfg = inputs.small_config(cfg_id=1300 + d, pot_size=700, keep=400, nuc_slots=0, cap_rows=3, Hq=1, Hkv=1, d=d, dtype="bf16", layers=len(where))
    scorer = TC if d in (64, 128) else ipot.IPOT_SCORER_AUTO
    for cap in (False, True):
        t = _axis_cycle(cfg, [1.0, 0.9, 1.0], (top - 125, top - 5), top, where, cap)
        compare_cycle(cfg, t, gpu_cycle(cfg, t, scorer))


@pytest.mark.parametrize("n", [4100, 9000])
@pytest.mark.parametrize("d", [64, 128, 256])
def test_one_sweep_sums_of_many_slabs_far_apart(d, n):
    """Sums that are published as they are and as (reference, sum) in every mixture: each half of the item's slabs, more than one look's
    worth of them, and neighbours on both sides of 2^118 whose shares of the denominator differ by little."""
    far = [{}, {70: 126}, {70: 117.9, 300: 118.1, 2000: 119}, {n - 1: 127, 600: 118}, {9: 117, 2500: 128, n - 300: 128}, {5: 200, n - 2: 199},
           {k: 100 + k % 60 for k in range(3, n, 251)}, {k: -100 for k in range(n)}, {k: -89 - k // 400 for k in range(n)}]
    cfg = inputs.small_config(cfg_id=1400 + d, pot_size=n, keep=200, nuc_slots=0, cap_rows=40, Hq=1, Hkv=1, d=d, dtype="bf16", layers=len(far))
    factors = [1.0, 0.97] + [0.1, -0.1] * 19
    t = _axis_cycle(cfg, factors, (20, 45), 0, [], False)
    K = inputs.widen(t["K"], "bf16").astype(np.float32)
    for layer, at in enumerate(far):
        for slot, logit in at.items():
            K[layer, :, :, slot, 3] = logit * np.log(2.0) * np.sqrt(d) / 8.0
    t["K"] = inputs.store(K, "bf16")
    compare_cycle(cfg, t, gpu_cycle(cfg, t, TC if d < 256 else ipot.IPOT_SCORER_AUTO))


ITEMS = ipot.IPOT_SCORER_TENSOR_ITEMS


@pytest.mark.parametrize("units,n,P,G,d,first,want", [
    # beyond 40 slabs: number of keys for 64 channels; three row blocks; two; lengths beyond 64 and 96 slabs, with few and many units
    (31, 16384, 8, 1, 64, None, TC), (32, 16384, 8, 1, 64, None, ITEMS), (22, 12288, 65, 4, 128, None, TC), (22, 12289, 65, 4, 128, None, ITEMS),
    (63, 15360, 33, 4, 128, None, TC), (64, 15360, 33, 4, 128, None, ITEMS), (64, 15360, 32, 4, 128, None, TC), (31, 20480, 8, 4, 128, None, TC),
    (32, 20480, 8, 4, 128, None, ITEMS), (32, 16384, 8, 4, 128, None, TC), (11, 24576, 8, 4, 128, None, TC), (11, 24577, 8, 4, 128, None, ITEMS),
    (8, 24577, 8, 4, 128, None, TC), (33, 20480, 8, 1, 96, None, ITEMS), (33, 16384, 8, 1, 96, None, TC), (32, 20480, 8, 1, 256, None, TC),
    # 15 and 16 slabs of another head dimension; chunks that start on a slab, between two, and off every tile
    (3, 1280, 8, 1, 96, None, ITEMS), (4, 1024, 8, 1, 96, None, TC), (8, 1024, 8, 1, 96, 256, TC), (8, 1024, 8, 1, 96, 384, ITEMS), (8, 1024, 8, 1, 96, 300, TC),
    (33, 10752, 8, 4, 128, 256, TC), (33, 10752, 8, 4, 128, 384, ITEMS), (33, 10752, 8, 4, 128, 300, TC), (16, 16384, 8, 4, 128, 384, ITEMS),
    (8, 10752, 8, 4, 128, 384, TC), (40, 10752, 8, 1, 64, 384, ITEMS), (40, 10752, 8, 1, 64, 512, TC)])
def test_automatic_choice_beyond_40_slabs_and_of_other_rows(units, n, P, G, d, first, want):
    """Both sides of each line; the scores agree with those of a kernel that was not chosen."""
    g = torch.Generator(device="cuda").manual_seed(n)
    K = torch.randn((units, 1, 1, n, d), generator=g, device="cuda").bfloat16()
    Q = torch.randn((units, 1, G, P, d), generator=g, device="cuda").bfloat16()
    u = []
    for scorer in (ipot.IPOT_SCORER_AUTO, ipot.IPOT_SCORER_WARP_MMA):
        h = ipot.ipot_create_ex(n, n // 4, units, G, 1, d, nuc_slots=0, max_cap_rows=P)
        try:
            ipot.ipot_set_scorer(h, scorer)
            ipot.ipot_set_profiling(h, True)
            parts = [K] if first is None else [K[:, :, :, :first].contiguous(), K[:, :, :, first:].contiguous()]
            for i, part in enumerate(parts):
                ipot.ipot_set_deferred_append(h, i == 1)
                ipot.ipot_append_chunk(h, part, part, part.shape[3])
            ipot.ipot_score_and_compress(h, Q, P, None)
            assert ipot.ipot_sync_status(h) == 0
            assert ipot.ipot_kernel_ms(h)[2] == (want if scorer == ipot.IPOT_SCORER_AUTO else scorer)
            u.append(ipot.device_array(ipot.ipot_last_scores(h)[0], (units, n), "f32").clone())
        finally:
            ipot.ipot_destroy(h)
    assert ((u[0] - u[1]).norm() / u[1].norm()).item() < 2e-6   # (two kernels within 1e-6 of the exact scores each)

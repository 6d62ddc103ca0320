"""GPU parity: the CUDA path through the C ABI against the CPU checker, element by
element, on seeded inputs (see tests/parity.py for the tolerances)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2410_01518_b200 import inputs, ipot
from parity import compare_cycle, from_dev_bits, gpu_cycle, make_pot, read_results, to_dev

pytestmark = pytest.mark.gpu

SCORERS = [ipot.IPOT_SCORER_SIMT, ipot.IPOT_SCORER_TENSOR, ipot.IPOT_SCORER_WARP_MMA]


def tensor_scorer_applies(cfg, n=None):
    """The tcgen05 scorer takes bf16 with d = 128 or 64 (any pot size the library accepts)."""
    return cfg.dtype == "bf16" and cfg.d in (64, 128)


def scorer_applies(cfg, scorer):
    """fp32 FMAs: everything; tcgen05: see above; warp-level tensor cores: bf16 with d a multiple of 16."""
    if scorer == ipot.IPOT_SCORER_TENSOR:
        return tensor_scorer_applies(cfg)
    if scorer == ipot.IPOT_SCORER_WARP_MMA:
        return cfg.dtype == "bf16" and cfg.d % 16 == 0
    return True


def test_config1_tiny_f32_all_units():
    cfg = inputs.CONFIGS[1]
    t = inputs.make_cycle(cfg)
    gpu = gpu_cycle(cfg, t, ipot.IPOT_SCORER_SIMT)
    same, n = compare_cycle(cfg, t, gpu)
    assert n == cfg.units and same == n


@pytest.mark.parametrize("scorer", SCORERS)
def test_config2_mistral_layer_bf16_all_units(scorer):
    cfg = inputs.CONFIGS[2]
    t = inputs.make_cycle(cfg)
    gpu = gpu_cycle(cfg, t, scorer)
    same, n = compare_cycle(cfg, t, gpu)
    assert n == cfg.units and same >= n - 1  # at most one unit may sit on a tie


SMALL = [
    # several tiles and a ragged tail, odd sizes, degenerate selections
    dict(pot_size=96, keep=40, nuc_slots=20, cap_rows=5, Hq=4, Hkv=2, d=64, dtype="f32"),
    dict(pot_size=333, keep=100, nuc_slots=37, cap_rows=7, Hq=6, Hkv=2, d=64, dtype="bf16"),
    dict(pot_size=1000, keep=999, nuc_slots=1, cap_rows=3, Hq=2, Hkv=2, d=128, dtype="bf16"),
    dict(pot_size=200, keep=1, nuc_slots=0, cap_rows=1, Hq=2, Hkv=1, d=128, dtype="f32"),
    dict(pot_size=257, keep=64, nuc_slots=64, cap_rows=9, Hq=8, Hkv=2, d=64, dtype="bf16"),     # NuC only
    dict(pot_size=130, keep=65, nuc_slots=0, cap_rows=33, Hq=4, Hkv=4, d=40, dtype="bf16"),     # CaP only, G = 1
    dict(pot_size=2049, keep=1024, nuc_slots=512, cap_rows=16, Hq=8, Hkv=1, d=128, dtype="bf16", layers=2, batch=2),
    dict(pot_size=64, keep=63, nuc_slots=30, cap_rows=2, Hq=3, Hkv=3, d=256, dtype="f32", layers=3),
    dict(pot_size=1500, keep=700, nuc_slots=350, cap_rows=1, Hq=1, Hkv=1, d=128, dtype="bf16", batch=3),  # last-token rule
    dict(pot_size=777, keep=300, nuc_slots=150, cap_rows=24, Hq=8, Hkv=2, d=256, dtype="bf16", layers=2),   # 256 channels
    dict(pot_size=500, keep=250, nuc_slots=100, cap_rows=70, Hq=3, Hkv=1, d=96, dtype="bf16"),              # 96 channels, M = 210
]


@pytest.mark.parametrize("case", range(len(SMALL)))
@pytest.mark.parametrize("scorer", SCORERS)
def test_small_random_shapes(case, scorer):
    cfg = inputs.small_config(cfg_id=200 + case, **SMALL[case])
    if not scorer_applies(cfg, scorer):
        h = make_pot(cfg)
        try:  # a scorer that does not take the shape must refuse, not fall back
            t = inputs.make_cycle(cfg)
            ipot.ipot_set_scorer(h, scorer)
            ipot.ipot_append_chunk(h, to_dev(t["K"], cfg.dtype), to_dev(t["V"], cfg.dtype), cfg.pot_size)
            rc = ipot.lib().ipot_score_only(h, to_dev(t["Q"], cfg.dtype).data_ptr(), cfg.cap_rows, None)
            assert rc == ipot.IPOT_E_INVALID
        finally:
            ipot.ipot_destroy(h)
        return
    t = inputs.make_cycle(cfg)
    gpu = gpu_cycle(cfg, t, scorer)
    same, n = compare_cycle(cfg, t, gpu)
    assert n == cfg.units and same >= n - 1


def test_tensor_scorer_with_64_channel_heads():
    """d = 64 (one 64-channel half per tile): several slabs and row blocks, ragged tail, against the checker and
    against the fp32 scorer."""
    cfg = inputs.small_config(cfg_id=420, pot_size=3000, keep=1400, nuc_slots=700, cap_rows=40, Hq=8, Hkv=2, d=64,
                              dtype="bf16", layers=3, batch=2)
    t = inputs.make_cycle(cfg)
    gpu = gpu_cycle(cfg, t, ipot.IPOT_SCORER_TENSOR, n=2999)
    same, cnt = compare_cycle(cfg, t, gpu, n=2999)
    assert cnt == cfg.units and same >= cnt - 1
    simt = gpu_cycle(cfg, t, ipot.IPOT_SCORER_SIMT, n=2999)
    np.testing.assert_allclose(gpu[0], simt[0], rtol=2e-5, atol=1e-30)


TENSOR_SHAPES = [
    # (pot_size, rows used, cap_rows, Hq, Hkv, layers, batch): 1..64 slabs per item, ragged slabs, 1-4 row blocks,
    # fewer and more tasks than SMs
    (512, 512, 32, 4, 1, 1, 1), (640, 513, 16, 8, 2, 2, 1), (1536, 1500, 33, 8, 2, 1, 2), (2048, 2048, 64, 8, 2, 3, 1),
    (3000, 2999, 5, 6, 2, 1, 1), (4096, 3585, 64, 12, 2, 2, 1), (4096, 4096, 32, 32, 8, 5, 1), (300, 129, 1, 1, 1, 1, 1),
    (8192, 8192, 64, 8, 2, 1, 2), (16384, 16001, 64, 8, 1, 1, 2), (5000, 4097, 40, 4, 1, 20, 1),
]


@pytest.mark.parametrize("case", range(len(TENSOR_SHAPES)))
def test_tensor_scorer_shapes(case):
    pot, n, P, Hq, Hkv, L, B = TENSOR_SHAPES[case]
    cfg = inputs.small_config(cfg_id=400 + case, pot_size=pot, keep=n // 2, nuc_slots=n // 4, cap_rows=P, Hq=Hq,
                              Hkv=Hkv, d=128, dtype="bf16", layers=L, batch=B)
    t = inputs.make_cycle(cfg)
    gpu = gpu_cycle(cfg, t, ipot.IPOT_SCORER_TENSOR, n=n)
    same, cnt = compare_cycle(cfg, t, gpu, n=n)
    assert cnt == cfg.units and same >= cnt - 1
    simt = gpu_cycle(cfg, t, ipot.IPOT_SCORER_SIMT, n=n)
    np.testing.assert_allclose(gpu[0], simt[0], rtol=2e-5, atol=1e-30)  # the two GPU scorers agree far inside 1e-3


def test_config3_full_size_every_unit():
    """All 32 layers in one call (the launch the benchmark times); the checker follows every one of the 256 units."""
    cfg = inputs.CONFIGS[3]
    K0, V0 = inputs.make_kv(cfg, 2048, chunk=0)
    K1, V1 = inputs.make_kv(cfg, 2048, chunk=1)
    t = {"K": np.concatenate([K0, K1], axis=3), "V": np.concatenate([V0, V1], axis=3),
         "Q": inputs.make_q(cfg, 1), "aux": inputs.make_aux(cfg, 1)}
    gpu = gpu_cycle(cfg, t, ipot.IPOT_SCORER_AUTO)
    same, cnt = compare_cycle(cfg, t, gpu)
    # adjacent order statistics of 4096 scores lie ~3e-4 apart relatively and the decision is taken in fp32 on the
    # GPU, so a unit in a few hundred may resolve its last slot the other way (inside the tie band, checked per slot)
    assert cnt == cfg.units and same >= cnt - 3
    u, idx = gpu[0], gpu[1]
    assert np.abs(u.sum(axis=1) - cfg.G * cfg.cap_rows).max() < 2e-2      # holds at any size
    assert (np.diff(idx, axis=1) > 0).all() and idx.min() >= 0 and idx.max() < cfg.pot_size


@pytest.mark.parametrize("cfg_id,n_sample", [(4, 32), (5, 32)])
def test_configs_4_and_5_full_size_sampled_units(cfg_id, n_sample):
    """Llama-3-8B-shaped batch of 16 streams (pot 8192, 2 row blocks) and the 70B-shaped layer (pot 16384,
    4 row blocks, heavy-tailed keys, 5 % exactly duplicated tokens): the whole configuration runs on the
    GPU, the checker follows 32 units spread over all streams and heads; properties that hold at any size are
    checked on all units.  Every unit whose list differs from the checker's differs only in slots inside the
    tie band (asserted per slot by compare_cycle); at most one followed unit in eight may do so."""
    cfg = inputs.CONFIGS[cfg_id]
    t = inputs.make_cycle(cfg)
    gpu = gpu_cycle(cfg, t, ipot.IPOT_SCORER_AUTO)
    units = np.unique(np.concatenate([np.linspace(0, cfg.units - 1, n_sample - 2).astype(np.int32), [1, cfg.units - 2]]))
    same, cnt = compare_cycle(cfg, t, gpu, units=units)
    assert cnt >= n_sample - 2 and same >= cnt - cnt // 8
    u, idx, K, V = gpu
    M = cfg.G * cfg.cap_rows
    assert np.abs(u.sum(axis=1) - M).max() < 1e-4 * M
    assert (np.diff(idx, axis=1) > 0).all() and idx.min() >= 0 and idx.max() < cfg.pot_size
    Kin = t["K"].reshape(cfg.units, cfg.pot_size, cfg.d)
    for unit in range(0, cfg.units, 7):     # gathered bytes on more units than the checker follows
        assert (K[unit] == Kin[unit][idx[unit]]).all()
    for b in range(cfg.batch):              # the novelty slots are in every head of the stream
        nuc = set(oracle.nuc_top(t["aux"][b], cfg.nuc_slots).tolist())
        for g in range(cfg.Hkv):
            assert nuc <= set(idx[b * cfg.Hkv + g].tolist())


@pytest.mark.parametrize("deferred", [False, True])
def test_config3_full_size_stream_of_cycles(deferred):
    """The 32-layer stream at full size through three consecutive fill/distil rounds (Sec. 3.2), with the plain and
    with the deferred append.  The checker keeps its own pot for 40 units (the first and last eight and 24 spread
    over the layers); after every cycle scores, index lists and the pot's K, V bytes are compared, and the checker's
    pot is advanced with the validated GPU lists.  What a launch carries over to the next one (survivor rows, the
    deferred chunk, scorer state) is thereby followed at the shape the benchmark times."""
    cfg = inputs.CONFIGS[3]
    N, keep, d = cfg.pot_size, cfg.keep, cfg.d
    units = np.unique(np.concatenate([np.arange(8), np.arange(cfg.units - 8, cfg.units),
                                      np.linspace(8, cfg.units - 9, 24).astype(np.int64)])).astype(np.int32)
    shape5 = (cfg.layers, cfg.batch, cfg.Hkv)
    h = make_pot(cfg)
    alive = []
    try:
        if deferred:
            ipot.ipot_set_deferred_append(h, True)
        K0, V0 = inputs.make_kv(cfg, N - keep, chunk=0)
        alive.append((to_dev(K0, "bf16"), to_dev(V0, "bf16")))
        ipot.ipot_append_chunk(h, alive[-1][0], alive[-1][1], N - keep)
        refK = K0.reshape(cfg.units, N - keep, d)[units]       # the checker's pot, followed units only
        refV = V0.reshape(cfg.units, N - keep, d)[units]
        for cyc in range(1, 4):
            Kc, Vc = inputs.make_kv(cfg, N - refK.shape[1], chunk=cyc)
            alive.append((to_dev(Kc, "bf16"), to_dev(Vc, "bf16")))      # a deferred chunk is read where it lies
            ipot.ipot_append_chunk(h, alive[-1][0], alive[-1][1], Kc.shape[3])
            fullK = np.zeros((cfg.units, N, d), dtype=np.uint16)
            fullV = np.zeros((cfg.units, N, d), dtype=np.uint16)
            fullK[units] = np.concatenate([refK, Kc.reshape(cfg.units, -1, d)[units]], axis=1)
            fullV[units] = np.concatenate([refV, Vc.reshape(cfg.units, -1, d)[units]], axis=1)
            t = {"K": fullK.reshape(shape5 + (N, d)), "V": fullV.reshape(shape5 + (N, d)),
                 "Q": inputs.make_q(cfg, cyc), "aux": inputs.make_aux(cfg, cyc)}
            ipot.ipot_score_and_compress(h, to_dev(t["Q"], "bf16"), cfg.cap_rows, torch.from_numpy(t["aux"]).cuda())
            u, idx, K, V = read_results(h, cfg, N)
            same, cnt = compare_cycle(cfg, t, (u, idx, K, V), units=units)
            assert cnt == len(units) and same >= cnt - 2, (cyc, same)
            assert np.abs(u.sum(axis=1) - cfg.G * cfg.cap_rows).max() < 2e-2
            assert (np.diff(idx, axis=1) > 0).all() and idx.min() >= 0 and idx.max() < N
            refK = np.stack([oracle.gather(fullK[unit], idx[unit]) for unit in units])
            refV = np.stack([oracle.gather(fullV[unit], idx[unit]) for unit in units])
            assert (K[units] == refK).all() and (V[units] == refV).all()
            Kp, Vp, ln = ipot.ipot_view(h)
            assert ln == keep
            del alive[:-1]                                               # older chunks are in the pot by now
    finally:
        ipot.ipot_destroy(h)


def test_partially_filled_pot():
    cfg = inputs.small_config(cfg_id=220, pot_size=700, keep=300, nuc_slots=100, cap_rows=6, Hq=4, Hkv=2,
                              d=128, dtype="bf16", layers=2)
    t = inputs.make_cycle(cfg)
    gpu = gpu_cycle(cfg, t, n=555)
    same, n = compare_cycle(cfg, t, gpu, n=555)
    assert same >= n - 1


def test_exact_ties_resolve_to_lower_slots():
    # all keys identical -> every score equal; all aux equal -> first T slots reserved
    cfg = inputs.small_config(cfg_id=230, pot_size=300, keep=120, nuc_slots=50, cap_rows=4, d=64, dtype="f32")
    t = inputs.make_cycle(cfg)
    t["K"][:] = t["K"][:, :, :, :1, :]
    t["aux"][:] = 0.25
    u, idx, K, V = gpu_cycle(cfg, t)
    for unit in range(cfg.units):
        assert idx[unit].tolist() == list(range(120))
        assert np.unique(u[unit]).size == 1
    same, n = compare_cycle(cfg, t, (u, idx, K, V))
    assert same == n


@pytest.mark.parametrize("pattern", [0x7FFFFFFF, 0x7FC00000, 0x7F800001, 0xFFFFFFFF])
@pytest.mark.parametrize("n,count", [(1000, 400), (1000, 900), (200, 150)])   # more NaNs than reserved slots, and than slots kept; no ranking in the scorer's grid
def test_ranking_of_nan_novelty(pattern, n, count):
    """Novelty has to be finite; a NaN in it still takes one slot each and no more: exactly `keep` survivors, among them the
    lowest slots of the NaNs that rank above every number, or the numbers before the NaN that ranks below."""
    keep, T = n // 2, n // 4
    cfg = inputs.small_config(cfg_id=985, pot_size=n, keep=keep, nuc_slots=T, cap_rows=4, Hq=4, Hkv=2, d=64, dtype="bf16", batch=2)
    t = inputs.make_cycle(cfg)
    where = np.sort(np.random.default_rng(count).permutation(n)[:count])
    t["aux"].view(np.uint32)[:, where] = pattern
    _, idx, K, _ = gpu_cycle(cfg, t)   # (asserts the status)
    others = np.setdiff1d(np.arange(n), where)
    reserved = where[:T] if pattern < 0x80000000 else np.concatenate([others, where])[:T] if len(others) <= T else []
    for unit in range(cfg.units):
        assert len(set(idx[unit].tolist())) == keep and (np.diff(idx[unit]) > 0).all() and set(reserved) <= set(idx[unit].tolist())
        assert (K[unit] == t["K"].reshape(cfg.units, n, cfg.d)[unit][idx[unit]]).all()


@pytest.mark.parametrize("pot,keep,T", [(4096, 2048, 1024), (9000, 5001, 100), (16400, 5000, 0), (20000, 12288, 4096)])
def test_exact_ties_in_large_pots(pot, keep, T):
    """Every score equal and every novelty equal: the survivors are the first `keep` slots whatever the pot size.
    The sizes take the ranking kernels through each block shape (256, 512, 1024 threads; 16 and 32 slots a thread),
    pots that are not a multiple of 16 slots, index lists of more than one output round and of odd length."""
    cfg = inputs.small_config(cfg_id=231, pot_size=pot, keep=keep, nuc_slots=T, cap_rows=2, Hq=2, Hkv=2, d=32, dtype="f32")
    t = inputs.make_cycle(cfg)
    t["K"][:] = t["K"][:, :, :, :1, :]
    t["aux"][:] = 0.25
    u, idx, K, V = gpu_cycle(cfg, t)
    for unit in range(cfg.units):
        assert np.array_equal(idx[unit], np.arange(keep))
        assert np.unique(u[unit]).size == 1
    same, n = compare_cycle(cfg, t, (u, idx, K, V))
    assert same == n


def test_duplicated_tokens_and_heavy_tails():
    cfg = inputs.small_config(cfg_id=5, recipe="student_dup", dtype="bf16", pot_size=1200, keep=300,
                              nuc_slots=150, cap_rows=8, batch=2, Hq=8, Hkv=2, d=128)
    t = inputs.make_cycle(cfg)
    gpu = gpu_cycle(cfg, t)
    compare_cycle(cfg, t, gpu)  # duplicates may swap inside the tie band; bytes must still match


def test_outlier_channels_and_lognormal_norms():
    for recipe, cid in (("stream", 3), ("lognorm", 4)):
        cfg = inputs.small_config(cfg_id=cid, recipe=recipe, dtype="bf16", pot_size=900, keep=450,
                                  nuc_slots=225, cap_rows=8, batch=2, Hq=8, Hkv=2, d=128, chunk=900)
        t = inputs.make_cycle(cfg)
        same, n = compare_cycle(cfg, t, gpu_cycle(cfg, t))
        assert same >= n - 1


def test_nuc_only_keeps_identical_slots_in_every_head():
    cfg = inputs.small_config(cfg_id=240, pot_size=500, keep=200, nuc_slots=200, cap_rows=4, Hq=8, Hkv=4,
                              d=64, dtype="bf16", layers=2)
    t = inputs.make_cycle(cfg)
    u, idx, K, V = gpu_cycle(cfg, t)
    assert (idx == idx[0]).all()
    assert idx[0].tolist() == oracle.nuc_top(t["aux"][0], 200).tolist()


def test_stream_of_cycles_follows_the_checker():
    """Several fill/distil rounds (Sec. 3.2).  The checker keeps its own pot; after
    each cycle the GPU's index lists are validated against the checker's scores and
    the checker's pot is advanced with the validated lists, so a tie resolved the
    other way does not end the comparison."""
    cfg = inputs.small_config(cfg_id=3, recipe="stream", dtype="bf16", pot_size=512, keep=256, nuc_slots=128,
                              cap_rows=8, Hq=8, Hkv=2, d=128, layers=3, chunk=256)
    h = make_pot(cfg)
    try:
        K0, V0 = inputs.make_kv(cfg, 256, chunk=0)
        ipot.ipot_append_chunk(h, to_dev(K0, "bf16"), to_dev(V0, "bf16"), 256)
        refK, refV = K0, V0
        for cyc in range(1, 7):
            Kc, Vc = inputs.make_kv(cfg, 256, chunk=cyc)
            ipot.ipot_append_chunk(h, to_dev(Kc, "bf16"), to_dev(Vc, "bf16"), 256)
            refK, refV = np.concatenate([refK, Kc], axis=3), np.concatenate([refV, Vc], axis=3)
            t = {"K": refK, "V": refV, "Q": inputs.make_q(cfg, cyc), "aux": inputs.make_aux(cfg, cyc)}
            ipot.ipot_score_and_compress(h, to_dev(t["Q"], "bf16"), cfg.cap_rows, torch.from_numpy(t["aux"]).cuda())
            u, idx, K, V = read_results(h, cfg, 512)
            compare_cycle(cfg, t, (u, idx, K, V))
            # advance the checker's pot with the validated index lists
            flatK, flatV = refK.reshape(cfg.units, 512, cfg.d), refV.reshape(cfg.units, 512, cfg.d)
            refK = np.stack([oracle.gather(flatK[i], idx[i]) for i in range(cfg.units)]).reshape(
                cfg.layers, cfg.batch, cfg.Hkv, 256, cfg.d)
            refV = np.stack([oracle.gather(flatV[i], idx[i]) for i in range(cfg.units)]).reshape(
                cfg.layers, cfg.batch, cfg.Hkv, 256, cfg.d)
            assert (K.reshape(refK.shape) == refK).all() and (V.reshape(refV.shape) == refV).all()
    finally:
        ipot.ipot_destroy(h)


def test_host_buffer_calls_match_device_calls():
    cfg = inputs.small_config(cfg_id=250, pot_size=640, keep=320, nuc_slots=160, cap_rows=8, Hq=8, Hkv=2,
                              d=128, dtype="bf16", layers=2, batch=2)
    t = inputs.make_cycle(cfg)
    dev = gpu_cycle(cfg, t)
    h = make_pot(cfg)
    try:
        ipot.ipot_append_chunk_host(h, t["K"][:, :, :, :400].copy(), t["V"][:, :, :, :400].copy(), 400)
        ipot.ipot_append_chunk_host(h, t["K"][:, :, :, 400:].copy(), t["V"][:, :, :, 400:].copy(), 240)
        idx_host = np.full((cfg.units, cfg.keep), -1, dtype=np.int32)
        ipot.ipot_score_and_compress_host(h, t["Q"], cfg.cap_rows, t["aux"], idx_host)
        u, idx, K, V = read_results(h, cfg, 640)
        assert (idx_host == idx).all()
        assert (idx == dev[1]).all() and (K == dev[2]).all() and (V == dev[3]).all() and (u == dev[0]).all()
    finally:
        ipot.ipot_destroy(h)


def test_state_machine_and_argument_errors():
    cfg = inputs.small_config(cfg_id=260, pot_size=128, keep=64, nuc_slots=32, cap_rows=4, d=64, dtype="bf16")
    t = inputs.make_cycle(cfg)
    h = make_pot(cfg)
    L = ipot.lib()
    try:
        Kd, Vd, Qd = to_dev(t["K"], "bf16"), to_dev(t["V"], "bf16"), to_dev(t["Q"], "bf16")
        auxd = torch.from_numpy(t["aux"]).cuda()
        assert L.ipot_score_and_compress(h, Qd.data_ptr(), 4, auxd.data_ptr()) == ipot.IPOT_E_STATE  # empty
        ipot.ipot_append_chunk(h, Kd[:, :, :, :64].contiguous(), Vd[:, :, :, :64].contiguous(), 64)
        assert L.ipot_score_and_compress(h, Qd.data_ptr(), 4, auxd.data_ptr()) == ipot.IPOT_E_STATE  # len == keep
        assert L.ipot_append_chunk(h, Kd.data_ptr(), Vd.data_ptr(), 65) == ipot.IPOT_E_STATE          # overflow
        assert ipot.ipot_view(h)[2] == 64
        assert L.ipot_append_chunk(h, Kd.data_ptr() + 2, Vd.data_ptr(), 1) == ipot.IPOT_E_INVALID     # misaligned
        assert L.ipot_append_chunk(h, Kd.data_ptr(), Vd.data_ptr(), 0) == ipot.IPOT_E_INVALID
        ipot.ipot_append_chunk(h, Kd[:, :, :, 64:].contiguous(), Vd[:, :, :, 64:].contiguous(), 64)
        assert L.ipot_score_and_compress(h, Qd.data_ptr(), 5, auxd.data_ptr()) == ipot.IPOT_E_INVALID  # > max rows
        assert L.ipot_score_and_compress(h, Qd.data_ptr(), 4, None) == ipot.IPOT_E_INVALID             # T > 0, no aux
        assert L.ipot_set_nuc_slots(h, 65) == ipot.IPOT_E_INVALID
        assert L.ipot_set_scorer(h, 7) == ipot.IPOT_E_INVALID
        assert ipot.ipot_view(h)[2] == 128
        ipot.ipot_score_and_compress(h, Qd, 4, auxd)
        assert ipot.ipot_view(h)[2] == 64 and ipot.ipot_sync_status(h) == 0
        ipot.ipot_reset(h)
        assert ipot.ipot_view(h)[2] == 0
        assert ipot.ipot_launch_count(h) >= 6
    finally:
        ipot.ipot_destroy(h)


def test_set_nuc_slots_and_profiling_and_determinism():
    cfg = inputs.small_config(cfg_id=270, pot_size=777, keep=300, nuc_slots=0, cap_rows=8, Hq=8, Hkv=2, d=128,
                              dtype="bf16", layers=2)
    t = inputs.make_cycle(cfg)
    a = gpu_cycle(cfg, t)
    b = gpu_cycle(cfg, t)
    for x, y in zip(a, b):
        assert (x == y).all()  # same bytes twice
    h = make_pot(cfg, nuc_slots=10)
    try:
        ipot.ipot_set_nuc_slots(h, 0)
        ipot.ipot_set_profiling(h, 1)
        ipot.ipot_append_chunk(h, to_dev(t["K"], "bf16"), to_dev(t["V"], "bf16"), 777)
        ipot.ipot_score_and_compress(h, to_dev(t["Q"], "bf16"), 8, None)
        ms, cycles, scorer = ipot.ipot_kernel_ms(h)
        assert cycles == 1 and len(ms) == 4 and all(m >= 0 for m in ms) and ms[1] > 0 and scorer in (1, 2)
        c = read_results(h, cfg, 777)
        assert (c[1] == a[1]).all()
    finally:
        ipot.ipot_destroy(h)


def test_score_only_leaves_the_pot_alone():
    cfg = inputs.small_config(cfg_id=280, pot_size=400, keep=100, nuc_slots=50, cap_rows=8, Hq=8, Hkv=2, d=128,
                              dtype="bf16")
    t = inputs.make_cycle(cfg)
    h = make_pot(cfg)
    try:
        Kd, Vd = to_dev(t["K"], "bf16"), to_dev(t["V"], "bf16")
        ipot.ipot_append_chunk(h, Kd, Vd, 400)
        ipot.ipot_score_only(h, to_dev(t["Q"], "bf16"), 8)
        assert ipot.ipot_sync_status(h) == 0
        sp, nb = ipot.ipot_last_scores(h)
        u = ipot.device_array(sp, (cfg.units, nb), "f32").cpu().numpy()
        Kp, Vp, ln = ipot.ipot_view(h)
        assert ln == 400 and nb == 400
        assert (from_dev_bits(ipot.device_array(Kp, (cfg.units, 400, 128), "bf16"), "bf16")
                == t["K"].reshape(cfg.units, 400, 128)).all()
        ref = oracle.cycle(t["Q"], t["K"], t["V"], t["aux"], cfg.keep, cfg.nuc_slots, with_kv=False)
        np.testing.assert_allclose(u, ref["u"], rtol=1e-3, atol=1e-30)
        assert abs(u.sum(axis=1) - cfg.G * cfg.cap_rows).max() < 1e-2
    finally:
        ipot.ipot_destroy(h)


@pytest.mark.parametrize("scorer", SCORERS)
def test_largest_pot_the_library_accepts(scorer):
    """pot_size = 32768 (the create-time limit): 128 slabs per item on the tensor scorer, 512 key tiles on the
    fp32 scorer; one more slot is refused at create."""
    cfg = inputs.small_config(cfg_id=290, pot_size=32768, keep=8192, nuc_slots=4096, cap_rows=16, Hq=4, Hkv=1, d=128,
                              dtype="bf16")
    t = inputs.make_cycle(cfg)
    gpu = gpu_cycle(cfg, t, scorer)
    same, n = compare_cycle(cfg, t, gpu)
    assert n == cfg.units and same == n
    rc = ipot.lib().ipot_create(32769, 8192, 1, 4, 1, 128, __import__("ctypes").byref(__import__("ctypes").c_void_p()))
    assert rc == ipot.IPOT_E_INVALID


@pytest.mark.parametrize("seed", range(10))
def test_seeded_random_configurations(seed):
    """Shapes drawn from a seeded generator (pot fill, keep, NuC slots, CaP rows, heads, head dimension, dtype,
    layers, streams): whatever scorer the library picks must agree with the checker, and so must every scorer
    that accepts the shape."""
    g = np.random.default_rng(9000 + seed)
    dtype = "bf16" if g.random() < 0.7 else "f32"
    d = int(g.choice([32, 48, 64, 96, 128, 160, 256]))
    Hkv = int(g.choice([1, 2, 3]))
    G = int(g.choice([1, 2, 4, 5]))
    pot = int(g.integers(70, 1400))
    n = int(g.integers(max(2, pot // 2), pot + 1))
    keep = int(g.integers(1, n))
    T = int(g.integers(0, keep + 1))
    cfg = inputs.small_config(cfg_id=900 + seed, pot_size=pot, keep=keep, nuc_slots=T, cap_rows=int(g.integers(1, 40)),
                              Hq=Hkv * G, Hkv=Hkv, d=d, dtype=dtype, layers=int(g.integers(1, 3)), batch=int(g.integers(1, 3)))
    t = inputs.make_cycle(cfg)
    for scorer in [ipot.IPOT_SCORER_AUTO] + SCORERS:
        if scorer != ipot.IPOT_SCORER_AUTO and not scorer_applies(cfg, scorer):
            continue
        gpu = gpu_cycle(cfg, t, scorer, n=n)
        same, cnt = compare_cycle(cfg, t, gpu, n=n)
        assert cnt == cfg.units and same >= cnt - 1, (seed, scorer)


@pytest.mark.parametrize("seed", range(16))
def test_seeded_random_large_pots(seed):
    """As above with pots of up to 20000 slots (the ranking kernels change their block shape at 4096, 8192 and 16384
    slots), novelty scores quantised on a third of the cases so that ties straddle threads, and the chunk of a deferred
    append starting anywhere on half of them."""
    g = np.random.default_rng(77000 + seed)
    dtype = "bf16" if g.random() < 0.7 else "f32"
    d = int(g.choice([32, 64, 128]))
    Hkv = int(g.choice([1, 2]))
    G = int(g.choice([1, 2, 4]))
    pot = int(g.choice([g.integers(70, 1400), g.integers(4000, 4200), g.integers(4097, 9000), g.integers(9000, 20000)]))
    n = int(g.integers(max(2, pot // 2), pot + 1))
    keep = int(g.integers(1, n))
    T = int(g.integers(0, keep + 1))
    cfg = inputs.small_config(cfg_id=3000 + seed, pot_size=pot, keep=keep, nuc_slots=T, cap_rows=int(g.integers(1, 12)),
                              Hq=Hkv * G, Hkv=Hkv, d=d, dtype=dtype, layers=1, batch=int(g.integers(1, 3)))
    t = inputs.make_cycle(cfg)
    if g.random() < 0.3:
        t["aux"] = np.round(t["aux"] * 8) / 8
    deferred = int(g.integers(0, n)) if g.random() < 0.5 else None
    gpu = gpu_cycle(cfg, t, ipot.IPOT_SCORER_AUTO, n=n, deferred_from=deferred)
    same, cnt = compare_cycle(cfg, t, gpu, n=n)
    assert cnt == cfg.units and same >= cnt - 1, seed


@pytest.mark.parametrize("n", [2, 31, 511, 512, 513, 1024, 1025, 2047, 2048, 2049, 4095, 4096, 4097, 8191, 8192])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_selection_of_few_units_at_the_edges_of_its_block_shapes(n, dtype):
    """Pots of fewer units than SMs use blocks of other shapes (4 or 8 slots a thread), f32 pots of up to 2048 slots rank the novelty in
    the scorer's launch.  Against a sort of the scores that the same cycle reports: every third key is the same, so that whole runs
    of scores tie, and novelty has few values.  The survivors are whole numbers: no tolerance."""
    cfg = inputs.small_config(cfg_id=840, pot_size=n + 1, keep=max(1, n // 2 - 1), nuc_slots=n // 5, cap_rows=2, Hq=2, Hkv=2, d=64, dtype=dtype, layers=2)
    t = inputs.make_cycle(cfg)
    t["K"][:, :, :, ::3] = t["K"][:, :, :, :1]
    t["K"][1, :, :, :] = t["K"][1, :, :, :1]
    t["aux"] = np.round(t["aux"] * 16).astype(np.float32) / 16
    gpu = gpu_cycle(cfg, t, n=n)
    compare_cycle(cfg, t, gpu, n=n)
    slots = np.arange(n)
    novel = np.lexsort((slots, -t["aux"][0, :n]))[:cfg.nuc_slots]      # the last key is the first to sort by; ties: lower slot
    for u in range(cfg.units):
        reserved = np.zeros(n, bool)
        reserved[novel] = True
        order = np.lexsort((slots, -gpu[0][u], ~reserved))
        assert np.array_equal(gpu[1][u], np.sort(order[:cfg.keep])), (n, dtype, u)

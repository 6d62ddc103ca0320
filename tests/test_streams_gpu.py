"""A pot on a stream that does not wait for the default stream (every ``torch.cuda.Stream``): creation leaves its counters
ready, whatever the default stream is busy with."""
import numpy as np
import pytest
import torch

from paper_2410_01518_b200 import inputs, ipot
from parity import gpu_cycle, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("handed_over", [False, True])   # the pot is created on the stream, or on the default stream
@pytest.mark.parametrize("d,dtype", [(96, "bf16"), (128, "bf16"), (128, "f32")])   # item scorer, one-sweep scorer, f32 scorer
def test_pot_on_its_own_stream_while_the_default_stream_is_busy(d, dtype, handed_over):
    """The default stream is held up by a bounded spin, and the memory that the pot is likely to get held other bytes before:
    counters that were cleared behind the spin would not be zero when the pot's own kernels run."""
    cfg = inputs.small_config(cfg_id=960, pot_size=2000, keep=900, nuc_slots=300, cap_rows=16, Hq=8, Hkv=4, d=d, dtype=dtype, layers=2, batch=2)
    t = inputs.make_cycle(cfg)
    want = gpu_cycle(cfg, t)
    Kd, Vd, Qd, auxd = to_dev(t["K"], dtype), to_dev(t["V"], dtype), to_dev(t["Q"], dtype), torch.from_numpy(t["aux"]).cuda()
    K = torch.empty((cfg.units, cfg.keep, d), dtype=Kd.dtype, device="cuda")
    u, idx = torch.empty((cfg.units, cfg.pot_size), device="cuda"), torch.empty((cfg.units, cfg.keep), dtype=torch.int32, device="cuda")
    dirty = torch.full((64 << 20,), 0x5A, dtype=torch.uint8, device="cuda")
    s, held = torch.cuda.Stream(), torch.cuda.Event()
    torch.cuda.synchronize()
    del dirty
    torch.cuda.empty_cache()
    torch.cuda._sleep(1_000_000_000)   # about half a second
    held.record()
    h = ipot.ipot_create_ex(cfg.pot_size, cfg.keep, cfg.layers, cfg.Hq, cfg.Hkv, d, batch=cfg.batch,
                            dtype=ipot.IPOT_F32 if dtype == "f32" else ipot.IPOT_BF16, nuc_slots=cfg.nuc_slots, max_cap_rows=cfg.cap_rows,
                            stream=None if handed_over else s.cuda_stream)
    try:
        if handed_over:
            ipot.ipot_set_stream(h, s.cuda_stream)
        with torch.cuda.stream(s):
            for _ in range(2):
                ipot.ipot_reset(h)
                ipot.ipot_append_chunk(h, Kd, Vd, cfg.pot_size)
                ipot.ipot_score_and_compress(h, Qd, cfg.cap_rows, auxd)
            Kp = ipot.ipot_view(h)[0]
            K.copy_(ipot.device_array(Kp, (cfg.units, cfg.pot_size, d), dtype)[:, :cfg.keep])
            u.copy_(ipot.device_array(ipot.ipot_last_scores(h)[0], u.shape, "f32"))
            idx.copy_(ipot.device_array(ipot.ipot_last_indices(h), idx.shape, "i32"))
        s.synchronize()
        assert not held.query(), "the default stream was not busy any more: the test has shown nothing"
        assert ipot.ipot_sync_status(h) == 0
    finally:
        ipot.ipot_destroy(h)
    assert (u.cpu().numpy() == want[0]).all() and (idx.cpu().numpy() == want[1]).all()
    got = K.cpu().numpy() if dtype == "f32" else K.view(torch.int16).cpu().numpy().view(np.uint16)
    assert (got == want[2]).all()


@pytest.mark.parametrize("d,dtype,layers,n,rope", [(128, "bf16", 2, 1500, False), (128, "bf16", 32, 4096, False), (96, "bf16", 2, 1500, False),
                                                   (128, "bf16", 2, 1500, True), (64, "f32", 2, 1500, False)])
def test_captured_pass_replays_on_other_inputs(d, dtype, layers, n, rope):
    """A whole pass (reset, append, cycle, a generated token) captured into a CUDA graph: every replay is a pass over what the
    input buffers hold by then, also between and after passes that are not captured.  (The one-sweep scorer tells its own
    statistics from an earlier launch's by a sign; its replays all have the same one.)  The larger pot is ranked on the
    side stream, the others inside the scorer's grid or on the pot's own stream."""
    cfg = inputs.small_config(cfg_id=965, pot_size=n, keep=n // 3, nuc_slots=n // 6, cap_rows=8, Hq=16, Hkv=8, d=d, dtype=dtype, layers=layers)
    g = torch.Generator(device="cuda").manual_seed(5)
    dt = torch.float32 if dtype == "f32" else torch.bfloat16
    shapes = {"K": (layers, 1, cfg.Hkv, n, d), "V": (layers, 1, cfg.Hkv, n, d), "Q": (layers, 1, cfg.Hq, cfg.cap_rows, d), "q": (layers, 1, cfg.Hq, d)}
    data = [{k: torch.randn(s, generator=g, device="cuda", dtype=dt) for k, s in shapes.items()} | {"aux": torch.rand((1, n), generator=g, device="cuda")}
            for _ in range(2)]
    buf = {k: v.clone() for k, v in data[0].items()}
    out = torch.zeros(shapes["q"], device="cuda")
    if rope:
        cos, sin = (to_dev(x, dtype) for x in inputs.make_rope_table(n, d, dtype))
    s = torch.cuda.Stream()
    torch.cuda.synchronize()

    def new_pot():
        h = ipot.ipot_create_ex(n, cfg.keep, layers, cfg.Hq, cfg.Hkv, d, dtype=ipot.IPOT_F32 if dtype == "f32" else ipot.IPOT_BF16,
                                nuc_slots=cfg.nuc_slots, max_cap_rows=cfg.cap_rows, stream=s.cuda_stream)
        if rope:
            ipot.ipot_enable_rope(h, cos, sin, ipot.IPOT_ROPE_HALF)
        return h

    def one_pass(h):
        ipot.ipot_reset(h)
        ipot.ipot_append_chunk(h, buf["K"], buf["V"], n)
        ipot.ipot_score_and_compress(h, buf["Q"], cfg.cap_rows, buf["aux"])
        if d != 96:
            ipot.ipot_decode_attention(h, buf["q"], out)

    def results(h):
        s.synchronize()
        assert ipot.ipot_sync_status(h) == 0
        K = ipot.device_array(ipot.ipot_view(h)[0], (cfg.units, n, d), dtype)[:, :cfg.keep]
        return [x.clone() for x in (ipot.device_array(ipot.ipot_last_scores(h)[0], (cfg.units, n), "f32"),
                                    ipot.device_array(ipot.ipot_last_indices(h), (cfg.units, cfg.keep), "i32"), K, out)]

    def load(i):
        s.synchronize()
        for k in buf:
            buf[k].copy_(data[i][k])
        torch.cuda.synchronize()

    h, want, graph = new_pot(), [], torch.cuda.CUDAGraph()
    try:
        for i in range(2):
            load(i)
            h1 = new_pot()
            one_pass(h1)
            want.append(results(h1))
            ipot.ipot_destroy(h1)
        load(0)
        one_pass(h)
        results(h)
        with torch.cuda.graph(graph, stream=s):
            ipot.ipot_set_stream(h, s.cuda_stream)
            one_pass(h)
        for i, replay in ((1, True), (0, True), (1, True), (0, False), (1, False), (0, True), (1, True), (0, False)):
            load(i)
            with torch.cuda.stream(s):
                graph.replay() if replay else one_pass(h)
            assert all(torch.equal(a, b) for a, b in zip(results(h), want[i])), (i, replay)
    finally:
        torch.cuda.synchronize()
        del graph
        ipot.ipot_destroy(h)

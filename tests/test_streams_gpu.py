"""A pot on a stream that does not wait for the default stream (every ``torch.cuda.Stream``): creation leaves its counters
ready, whatever the default stream is busy with."""
import numpy as np
import pytest
import torch

from paper_2410_01518_b200 import inputs, ipot
from parity import gpu_cycle, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,dtype", [(96, "bf16"), (128, "bf16"), (128, "f32")])   # item scorer, one-sweep scorer, f32 scorer
def test_pot_on_its_own_stream_while_the_default_stream_is_busy(d, dtype):
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
                            stream=s.cuda_stream)
    try:
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

"""Creation near the device's memory limit: the scratch that only makes a scorer faster is left out where it does not fit."""
import pytest
import torch

from paper_2410_01518_b200 import ipot

pytestmark = pytest.mark.gpu


def test_pot_that_fits_only_without_the_item_scorers_scratch():
    L, Hq, Hkv, d, n, P = 32, 128, 8, 96, 4096, 64     # 1024 query rows a unit: the scratch is a good part of the pot
    g = torch.Generator(device="cuda").manual_seed(1)
    K = torch.randn((L, 1, Hkv, n, d), generator=g, device="cuda").bfloat16()
    Q = torch.randn((L, 1, Hq, P, d), generator=g, device="cuda").bfloat16()

    def scores(expect):
        h = ipot.ipot_create_ex(n, n // 2, L, Hq, Hkv, d, nuc_slots=0, max_cap_rows=P)
        try:
            used = torch.cuda.mem_get_info()[0]
            ipot.ipot_set_profiling(h, True)
            ipot.ipot_append_chunk(h, K, K, n)
            ipot.ipot_score_and_compress(h, Q, P, None)
            assert ipot.ipot_sync_status(h) == 0
            assert ipot.ipot_kernel_ms(h)[2] == expect
            return ipot.device_array(ipot.ipot_last_scores(h)[0], (L * Hkv, n), "f32").cpu(), used
        finally:
            ipot.ipot_destroy(h)

    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    want, _ = scores(ipot.IPOT_SCORER_TENSOR_ITEMS)    # (what the first launches load stays loaded)
    before = torch.cuda.mem_get_info()[0]
    want, during = scores(ipot.IPOT_SCORER_TENSOR_ITEMS)
    scratch = L * Hkv * 1024 * (n // 128) * 8
    filler = torch.empty(before - (before - during) + scratch // 2, dtype=torch.uint8, device="cuda")
    try:
        got, _ = scores(ipot.IPOT_SCORER_WARP_MMA)
    finally:
        del filler
        torch.cuda.empty_cache()
    assert ((got - want).norm() / want.norm()).item() < 2e-6

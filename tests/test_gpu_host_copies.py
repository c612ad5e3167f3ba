"""pyramidsd_verify_host below and above the size from which its copies overlap stage 1, with results in one block (one
copy back) and in four, against the device entry point on the same inputs."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,K_d,K_q,V,pinned", [(2, 6, 3, 4096, True), (3, 8, 4, 50257, True), (1, 5, 5, 128256, True), (3, 8, 4, 32000, False)])
def test_host_entry_point_matches_device(B, K_d, K_q, V, pinned):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_12966_b200 import binding as psd, workloads as wl
    psd.load_library()
    psd.set_stream()
    names = ("accept_len_q", "next_token_q", "accept_len", "next_token")
    for i in range(3):
        t = wl.make_pyramid_inputs(B, K_d, K_q, V, "bf16", seed=70 + i, sigma_q=0.4, sigma_d=0.9)
        want = psd.verify(*[x.cuda() for x in t], 0.2, 0.1, psd.FUZZY, 3, i)
        host = [x.pin_memory() if pinned else x for x in t]
        block = torch.full((4, B), -7, dtype=torch.int32)
        apart = [torch.full((B + 1,), -7, dtype=torch.int32)[:B] for _ in names]
        for out in (dict(zip(names, block)), dict(zip(names, apart))):
            psd.verify_host(*host, 0.2, 0.1, psd.FUZZY, 3, i, out=out)
            for k in names:
                assert torch.equal(out[k], want[k].cpu()), (k, i)


def test_results_in_neighbouring_buffers_pinned_one_by_one():
    """Four result arrays that happen to lie behind one another, each a page pinned on its own: no copy may span them."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_12966_b200 import binding as psd, workloads as wl
    psd.load_library()
    psd.set_stream()
    B = 1024                                               # 4096 bytes of int32 each
    names = ("accept_len_q", "next_token_q", "accept_len", "next_token")
    t = wl.make_pyramid_inputs(B, 1, 1, 2048, "bf16", seed=5, sigma_q=0.4, sigma_d=0.9)
    want = psd.verify(*[x.cuda() for x in t], 0.2, 0.1, psd.FUZZY, 3, 0)
    raw = torch.zeros(6 * 4096, dtype=torch.uint8)
    first = -raw.data_ptr() % 4096
    pages = [raw[first + 4096 * i:first + 4096 * (i + 1)].view(torch.int32) for i in range(4)]
    rt = torch.cuda.cudart()
    for p in pages:
        assert int(rt.cudaHostRegister(p.data_ptr(), 4096, 0)) == 0
    try:
        psd.verify_host(*[x.pin_memory() for x in t], 0.2, 0.1, psd.FUZZY, 3, 0, out=dict(zip(names, pages)))
        for p, k in zip(pages, names):
            assert torch.equal(p, want[k].cpu()), k
    finally:
        for p in pages:
            rt.cudaHostUnregister(p.data_ptr())


def test_schedule_of_a_large_call_is_the_threads():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_12966_b200 import binding as psd, workloads as wl
    psd.load_library()
    psd.set_stream()
    t = [x.pin_memory() for x in wl.make_pyramid_inputs(3, 8, 4, 50264, "bf16", seed=9, sigma_q=0.4, sigma_d=0.9)]
    outs, launches = [], []
    try:
        for policy in (psd.TWO_STAGE_FUSED, psd.TWO_STAGE_SEPARATE, psd.TWO_STAGE_FUSED_ROWS, psd.TWO_STAGE_AUTO):
            psd.set_two_stage_policy(policy)
            n0 = psd.launch_count()
            outs.append(psd.verify_host(*t, 0.2, 0.1, psd.FUZZY, 3, 1))
            launches.append(psd.launch_count() - n0)
    finally:
        psd.set_two_stage_policy(psd.TWO_STAGE_DEFAULT)
    assert launches == [2, 4, 2, 4]
    for o in outs[1:]:
        assert all(torch.equal(o[k], outs[0][k]) for k in o)

"""The LM-head form at the edges of its own cuts: 16, 17, 32 and 33 rows (the weight or the rows as the MMA's M), 128 and 129, tile
widths other than 256 or 128 (equal rounds of narrower tiles), one and several rounds, segments of 512 columns, rows that end a
256-row block or a group of blocks (with sequences that begin in one group and end in the next), against the oracle on the sequences sampled."""
import numpy as np
import pytest
import torch

from parity_utils import TOL

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,K,d,V", [(1, 1, 64, 100), (2, 3, 128, 511), (2, 3, 128, 513), (3, 5, 64, 16352), (4, 4, 192, 37889), (17, 1, 64, 5000),
                                     (16, 8, 448, 19001), (4, 8, 64, 5001), (11, 3, 128, 5001), (43, 3, 64, 2049), (32, 8, 64, 18945), (43, 6, 64, 2049), (130, 8, 64, 1000), (90, 7, 64, 56000), (150, 7, 64, 2049), (21, 31, 64, 44032)])
def test_divergences_and_tokens(oracle, B, K, d, V):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_12966_b200 import binding as psd, workloads as wl
    h, w_t, zs, tok = wl.make_fused_inputs(B, K, V, d, 40 + V, 0.7, device=torch.device("cuda"))
    for mode, tau in ((psd.FUZZY, 0.03), (psd.ASSISTED, 0.0)):
        out = psd.verify_fused_lmhead(h, w_t, zs, tok, tau, mode, 3, 1)
        assert psd.last_status() == 0
        # the same logits as a library GEMM in fp32 of the same bf16 operands gives
        z = (h.float() @ w_t.float().T).view(B, K, V)
        p, q = torch.softmax(z.double(), -1), torch.softmax(zs.double(), -1)
        m = 0.5 * (p + q)
        js = 0.5 * (torch.special.xlogy(p, p / m) + torch.special.xlogy(q, q / m)).nan_to_num(0.0).sum(-1)
        assert (out["div"].double() - js).abs().max() < 2e-5
        assert (out["resid_mass"].double() - (p - q).clamp(min=0).sum(-1)).abs().max() < 2e-5
        L, nxt = out["accept_len"].cpu(), out["next_token"].cpu()
        if mode == psd.FUZZY:
            acc = (js.cpu() <= tau).int().cumprod(-1).sum(-1)
            near = ((js.cpu() - tau).abs() < 1e-5).any(-1)
            assert torch.equal(L[~near], acc.to(torch.int32)[~near])
        ties = 0
        for b in range(B):
            k = int(L[b])
            if k == K:
                assert int(nxt[b]) == -1
                continue
            w = p[b, k] if mode == psd.ASSISTED else (p[b, k] - q[b, k]).clamp(min=0)
            c = torch.cumsum(w, 0).cpu()
            _, u2 = oracle.row_uniforms(3, 1, b * K + k)
            t = u2 * float(c[-1])
            x = int(nxt[b])
            lo = float(c[x - 1]) if x else 0.0
            slack = TOL["bf16"]["cdf"] * float(c[-1])   # the weights are fp32, the sums the library's
            assert lo - slack <= t <= float(c[x]) + slack and float(w[x]) > 0
            ties += not (lo <= t < float(c[x]))
        assert ties <= max(1, B // 8)


@pytest.mark.parametrize("B,K,d,V", [(4, 8, 64, 5001), (11, 3, 128, 511), (8, 32, 64, 2049), (32, 8, 64, 18945),
                                     (300, 1, 64, 56001), (32, 8, 64, 65537), (10, 32, 64, 53000), (43, 7, 64, 56000), (130, 8, 64, 16200)])
@pytest.mark.parametrize("tile_variant", [None, 1])
def test_kl_with_and_without_residual_masses(oracle, B, K, d, V, tile_variant):
    """KL(large || small) from the terms of the stored logits, and from 2^24 logits on out of the sweep's own sums: the same
    divergences, accept lengths and tokens whether the masses of all rows are formed or those of the rejected rows alone; any
    number of positions per sequence (the final kernel shares its warps out among them), tiles of 160 columns (V = 18945),
    several row blocks."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_12966_b200 import binding as psd, workloads as wl
    h, w_t, zs, tok = wl.make_fused_inputs(B, K, V, d, 40 + V, 0.7, device=torch.device("cuda"))
    z = (h.double() @ w_t.double().T).view(B, K, V)
    lp, lq = torch.log_softmax(z, -1), torch.log_softmax(zs.double(), -1)
    p, q = lp.exp(), lq.exp()
    kl, resid = (p * (lp - lq)).sum(-1), (p - q).clamp(min=0).sum(-1)
    large = B * K * V >= 1 << 24
    for mode, tau in ((psd.FUZZY, 0.06), (psd.FUZZY, float(kl.median())), (psd.STRICT, 0.0), (psd.ASSISTED, 0.0), (psd.FUZZY, 1e9)):
        n0 = psd.launch_count()
        a = psd.verify_fused_lmhead(h, w_t, zs, tok, tau, mode, 3, 1, div_kind=psd.DIV_KL, want_resid=True, tile_variant=tile_variant)
        n1 = psd.launch_count()
        c = psd.verify_fused_lmhead(h, w_t, zs, tok, tau, mode, 3, 1, div_kind=psd.DIV_KL, want_resid=False, tile_variant=tile_variant)
        n2 = psd.launch_count()
        assert psd.last_status() == 0
        assert n2 - n1 < n1 - n0 if large else n2 - n1 == n1 - n0   # no launch forms a large call's masses if nobody takes them
        assert (a["div"].double() - kl).abs().max() < 1e-5 and (a["resid_mass"].double() - resid).abs().max() < 1e-5
        assert torch.equal(a["div"], c["div"]) and torch.equal(a["accept_len"], c["accept_len"])
        L, nxt, other = a["accept_len"].cpu(), a["next_token"].cpu(), c["next_token"].cpu()
        assert ((nxt >= 0) == (L < K)).all()
        ties = 0
        for b in range(B):
            k = int(L[b])
            if k == K:
                assert int(nxt[b]) == int(other[b]) == -1
                continue
            w = p[b, k] if mode == psd.ASSISTED else (p[b, k] - q[b, k]).clamp(min=0)
            cum = torch.cumsum(w, 0).cpu()
            _, u2 = oracle.row_uniforms(3, 1, b * K + k)
            t, slack = u2 * float(cum[-1]), TOL["bf16"]["cdf"] * float(cum[-1])
            for x in {int(nxt[b]), int(other[b])}:
                lo = float(cum[x - 1]) if x else 0.0
                assert lo - slack <= t <= float(cum[x]) + slack and float(w[x]) > 0
                ties += not (lo <= t < float(cum[x]))
        assert ties <= max(1, B // 8)


@pytest.mark.parametrize("V,d", [(152064, 1024), (128256, 2048)])
def test_fewer_rows_take_no_longer(V, d):
    """The form for few rows ends where the pairs of CTAs take over: a call with half of a tile's 256 rows (or a quarter, or
    an eighth) is no slower than the full tile. Best of five; a tenth for what a shared GPU adds."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_12966_b200 import binding as psd, workloads as wl
    h, w_t, zs, tok = wl.make_fused_inputs(32, 8, V, d, 4, 0.7, device=torch.device("cuda"))

    def best(B):
        args = h[:B * 8], w_t, zs[:B], tok[:B], 0.05
        times = []
        for i in range(7):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            psd.verify_fused_lmhead(*args)
            e[1].record()
            torch.cuda.synchronize()
            times.append(e[0].elapsed_time(e[1]))
        return min(times[2:])

    full = best(32)
    for B in (16, 8, 4):
        assert best(B) < 1.1 * full, (B, full)


def test_scratch_is_one_block_of_logits():
    """A call of 1024 rows at V = 128256 keeps one block of 256 rows of logits, not 525 MB of them."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_12966_b200 import binding as psd, workloads as wl
    h, w_t, zs, tok = wl.make_fused_inputs(128, 8, 128256, 64, 4, 0.7, device=torch.device("cuda"))
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        out = torch.zeros(1 << 22, device="cuda")   # what torch itself takes on a new stream
        del out
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        psd.verify_fused_lmhead(h, w_t, zs, tok, 0.05)
        torch.cuda.synchronize()
        taken = before - torch.cuda.mem_get_info()[0]
    psd.release_stream(stream)
    assert taken < 200 << 20, taken


@pytest.mark.parametrize("M,K,V,d", [(1, 1, 3000, 64), (6, 2, 20001, 128), (16, 4, 19000, 64), (17, 1, 33000, 192), (32, 8, 40000, 64),
                                     (33, 3, 33001, 64), (48, 4, 50000, 128), (64, 8, 32000, 64)])
def test_few_rows_whose_first_columns_say_nothing_of_the_rest(M, K, V, d):
    """The epilogues of the form for few rows, either side of 4, 16, 32 and 64 rows: per row the first 128 columns' logits lie
    some 250 nats below the rest's, so that sums against their maximum overflow and are taken again; others above."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_12966_b200 import binding as psd
    g = torch.Generator(device="cuda").manual_seed(M + V)
    B = M // K
    h = torch.randn((M, d), generator=g, device="cuda").bfloat16()
    w = (torch.randn((V, d), generator=g, device="cuda") * 0.1).bfloat16()
    h[:, 0] = 1.0
    w[:, 0] = 0.0
    w[:128, 0] = -250.0
    h[::3, 0] = -0.03                                        # every third row: the first columns weigh more
    z = h.double() @ w.double().T
    zs = (z + torch.randn((M, V), generator=g, device="cuda") * 0.5).bfloat16().view(B, K, V)
    zs[0, 0, :100] = -float("inf")
    tok = torch.randint(0, V, (B, K), generator=g, device="cuda", dtype=torch.int32)
    out = psd.verify_fused_lmhead(h, w, zs, tok, 0.1, psd.FUZZY, 3, 1)
    torch.cuda.synchronize()
    assert psd.last_status() == 0
    p, q = torch.log_softmax(z, -1).view(B, K, V), torch.log_softmax(zs.double(), -1)
    m = torch.logaddexp(p, q) - 0.6931471805599453
    term = lambda a: torch.where(a > -1e300, a.exp() * (a - m), 0.0)
    js, resid = 0.5 * (term(p) + term(q)).sum(-1), (p.exp() - q.exp()).clamp_min(0).sum(-1)
    # the logits' own error: single-precision sums of up to d products of size |z| (250 here), 2^-24 |z| sqrt(d) in the exponent
    tol = 1e-5 + 250 * d ** 0.5 * 2.0 ** -24
    assert (out["div"].double() - js).abs().max() < tol and (out["resid_mass"].double() - resid).abs().max() < tol
    accept = (out["div"] <= 0.1).int().cumprod(1).sum(1)
    assert torch.equal(out["accept_len"], accept.int()) and bool(((out["next_token"] >= 0) == (accept < K)).all())

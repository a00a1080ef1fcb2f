"""Edges of the prompt pass: tile widths of the GEMM (32 .. 256 activation rows in steps of 32, one and more row tiles), whole tiles and
tiles cut along k, both head sizes of the fused epilogues, more than one block of prompt rows."""
import numpy as np
import pytest

import kg_inputs as ki
from oracle import kangaroo_oracle as ko

pytestmark = pytest.mark.gpu

HD64 = ki.KgShape("hd64", 3, 384, 6, 64, 640, 1024, 1, "bf16", logit_scale=10.0, max_seq=700, page_size=8, gamma_max=8,
                  gain_std=0.1, deep_resid_scale=0.1, adapter_resid_scale=0.1, n_gen=12, seed=11)
HD128 = HD64.with_(name="hd128", n_heads=3, head_dim=128)


@pytest.fixture(scope="module")
def binding():
    import __graft_entry__ as ge
    ge.build()
    from paper_2404_18911_b200 import binding as b
    b.load()
    return b


@pytest.mark.parametrize("shape,n", [(HD64, 17), (HD128, 16), (HD64, 32), (HD64, 65), (HD64, 129), (HD64, 257), (HD64, 600), (HD128, 63), (HD128, 64), (HD128, 193), (HD128, 321)])
def test_prompt_pass_against_the_oracle(binding, shape, n):
    """Logits of the last prompt row, then rounds that read every K / V row the pass wrote."""
    from parity_harness import lockstep
    g = binding.KangarooModel(shape, debug_logits=True, page_shuffle=True)
    o = ko.KangarooOracle(shape, ki.make_weights(shape), np.float64)
    prompt = ki.make_prompt(shape, n).tolist()
    x0 = o.prefill(prompt)
    z_ref = o.last_logits
    got = g.prefill(prompt)
    assert np.max(np.abs(g.debug_logits(1, 0).astype(np.float64) - z_ref)) < 2e-2
    assert got == x0 or ko.top2_gap(z_ref) < 2e-2
    g.reset()
    res = lockstep(g, o, prompt, shape.n_gen, shape.eta, 6, 0)
    assert len(res["flips"]) <= 2, res["flips"]
    assert res["max_logit_err"] < 2e-2 and res["max_conf_err"] < 1e-3


def test_two_blocks_of_prompt_rows(binding):
    """2100 rows are two blocks; the second attends to the first one's cache rows.  Against the 16-row chunked pass."""
    shape = HD128.with_(max_seq=2200)
    g = binding.KangarooModel(shape, debug_logits=True)
    prompt = ki.make_prompt(shape, 2100).tolist()
    z = []
    for mode in (0, 1):
        g.reset()
        g.set_prefill_mode(mode)
        g.prefill(prompt)
        z.append(g.debug_logits(1, 0))
    assert np.max(np.abs(z[0] - z[1])) < 2e-2


# N = 19200: 75 tiles of 256 weight rows, one more than the 74 CTA pairs; N = 384 ends in half a tile; K = 192: an odd number of k blocks
@pytest.mark.parametrize("N,K,M", [(128, 64, 64), (384, 192, 65), (19200, 192, 130), (19200, 512, 257), (2560, 4032, 511), (128, 8192, 256),
                                   (384, 192, 20), (2560, 512, 96), (19200, 192, 220)])
def test_gemm_tiles_against_fp64(binding, N, K, M):
    import torch
    from kg_inputs import synth
    W = synth.fill_f32(1, 50, N * K, 0.02, True).reshape(N, K)
    x = synth.fill_f32(2, 51, M * K, 1.0, False).reshape(M, K)
    resid = synth.fill_f32(4, 53, M * N, 1.0, False).reshape(M, N)
    Wd, xd, rd = torch.from_numpy(W).cuda().to(torch.bfloat16), torch.from_numpy(x).cuda(), torch.from_numpy(resid).cuda()
    ref = rd.double() + xd.double() @ Wd.double().T
    # every product keeps 2^-17 of x and fp32 sums: the bound of the decode path's linear operator
    assert (binding.op_gemm(Wd, xd, resid=rd).double() - ref).abs().max().item() < 2e-4 * np.sqrt(K) * 0.02

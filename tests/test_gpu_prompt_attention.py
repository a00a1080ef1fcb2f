"""The tensor-core attention of the prompt pass at the edges of its tiles (128 rows, 128 keys, boxes of a page) against the chunked pass."""
import numpy as np
import pytest

import kg_inputs as ki

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def binding():
    import __graft_entry__ as ge
    ge.build()
    from paper_2404_18911_b200 import binding as b
    b.load()
    return b


# heads of both sizes; pages smaller than, as large as and larger than a box; one more block of rows behind 2048
@pytest.mark.parametrize("H,hd,page,n", [(4, 128, 16, 129), (4, 128, 16, 255), (4, 128, 16, 256), (4, 128, 4, 257), (4, 128, 64, 300), (4, 128, 1, 131),
                                         (8, 64, 16, 129), (8, 64, 2, 200), (8, 64, 32, 385), (4, 128, 16, 2100), (8, 64, 8, 2049)])
def test_tile_edges(binding, H, hd, page, n):
    import torch
    shape = ki.KgShape("attn", 2, 512, H, hd, 1024, 1024, 1, "bf16", logit_scale=10.0, max_seq=n + 40, page_size=page, gamma_max=4, gain_std=0.1,
                       deep_resid_scale=1.0, adapter_resid_scale=1.0, seed=n)
    poison = torch.full((1 << 28,), float("nan"), device="cuda")      # what lies in the cache behind the last token must not matter
    del poison
    g = binding.KangarooModel(shape, debug_logits=True, page_shuffle=True)
    prompt = ki.make_prompt(shape, n).tolist()
    z = []
    for mode in (1, 0):                                               # chunked, tensor cores
        g.reset()
        g.set_prefill_mode(mode)
        g.prefill(prompt)
        z.append(g.debug_logits(1, 0).astype(np.float64))
    print(f"n={n} H={H} hd={hd} page={page}: deviation {np.abs(z[1] - z[0]).max():.2e} of {np.abs(z[0]).max():.2f}")
    assert np.isfinite(z[1]).all()
    assert np.abs(z[1] - z[0]).max() < 2e-2

"""The tensor-core attention of the prompt pass at the edges of its tiles (128 rows, 128 keys, boxes of a page): every output row against float64,
whole models against the chunked pass, and a wait that runs out."""
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


@pytest.mark.parametrize("H,hd,n", [(4, 128, 300), (8, 64, 2049)])
def test_fresh_caches_and_repeats(binding, H, hd, n):
    """The tensor-core pass first, on caches that hold only NaN (0xffff): a row that is read before this pass has written it shows.  Again and again it
    gives the same bits."""
    import torch
    shape = ki.KgShape("attn", 2, 512, H, hd, 1024, 1024, 1, "bf16", logit_scale=10.0, max_seq=n + 40, page_size=16, gamma_max=4, gain_std=0.1,
                       deep_resid_scale=1.0, adapter_resid_scale=1.0, seed=n)
    prompt = ki.make_prompt(shape, n).tolist()
    nbytes = binding.KangarooModel(shape, debug_logits=True).arena_bytes
    z = []
    for mode in (0, 1):
        arena = torch.full((nbytes,), 0xff, dtype=torch.uint8, device="cuda")
        g = binding.KangarooModel(shape, debug_logits=True, page_shuffle=True, arena=arena)
        g.set_prefill_mode(mode)
        g.prefill(prompt)
        z.append(g.debug_logits(1, 0))
        for _ in range(5 if mode == 0 else 0):
            g.reset()
            g.prefill(prompt)
            assert np.array_equal(g.debug_logits(1, 0), z[0])
    assert np.isfinite(z[0]).all()
    assert np.abs(z[1].astype(np.float64) - z[0]).max() < 2e-2


def _operands(H, hd, pos0, rows, page, seed):
    """Planes of q, a cache in shuffled pages with NaN behind the last key, and K and V by position."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(seed)
    T = pos0 + rows
    pages = (T + page - 1) // page + 2
    q = torch.empty(rows, H * hd, device="cuda").normal_(0.0, 2.0 / np.log(2.0) / np.sqrt(hd), generator=g)
    qh = q.bfloat16()
    ql = (q - qh.float()).bfloat16()
    k, v = (torch.empty(T, H, hd, device="cuda").normal_(generator=g).bfloat16() for _ in range(2))
    table = torch.randperm(pages, generator=g, device="cuda").to(torch.int32)
    kc, vc = (torch.full((pages, H, page, hd), float("nan"), device="cuda", dtype=torch.bfloat16) for _ in range(2))
    at = torch.arange(T, device="cuda")
    pg, slot = table[at // page].long(), at % page
    kc[pg, :, slot], vc[pg, :, slot] = k, v
    return qh, ql, k, v, kc, vc, table


def test_expired_wait_returns_and_leaves_the_gpu_usable(binding):
    """One softmax warp of one block leaves out an arrival (test hook).  The block's waits run out, it waits for its copies and MMAs and
    returns; the others' rows are complete, and the next call on the same buffers is as good as the one before."""
    import time
    import torch
    H, hd, rows, page = 2, 128, 700, 16
    qh, ql, _, _, kc, vc, table = _operands(H, hd, 0, rows, page, 1)
    want = binding.debug_prompt_attention(qh, ql, 0, H, kc, vc, table, page, kernel=2)
    assert want[2].item() == 0
    t0 = time.time()
    hi, lo, err = binding.debug_prompt_attention(qh, ql, 0, H, kc, vc, table, page, kernel=2, skip=0)
    torch.cuda.synchronize()
    assert err.item() != 0 and time.time() - t0 < 10
    keep = torch.ones_like(hi, dtype=torch.bool)
    keep[640:, :hd] = False                                           # block 0: the last rows of head 0
    assert torch.equal(hi[keep], want[0][keep]) and torch.equal(lo[keep], want[1][keep])
    again = binding.debug_prompt_attention(qh, ql, 0, H, kc, vc, table, page, kernel=2)
    assert again[2].item() == 0 and torch.equal(again[0], want[0]) and torch.equal(again[1], want[1])


# rows and keys around the tiles; a few rows behind many keys; pages below, at and above a box; a block of the largest size
@pytest.mark.parametrize("kernel", [1, 2])
@pytest.mark.parametrize("H,hd,pos0,rows,page", [(2, 128, 0, 1, 16), (2, 128, 0, 129, 16), (3, 128, 0, 300, 8), (2, 128, 127, 130, 1), (2, 128, 2048, 1, 16), (1, 128, 1000, 77, 64),
                                                 (1, 128, 2048, 2048, 16), (4, 64, 0, 127, 16), (3, 64, 0, 128, 4), (2, 64, 3, 257, 2), (2, 64, 640, 384, 32), (1, 64, 100, 2048, 16)])
def test_every_row(binding, H, hd, pos0, rows, page, kernel):
    """Every row of both kernels against float64.  K, V and the planes of q are exact in the reference; what is left is the split of P and of the output into
    two planes (2^-17 of a value at most, each) and fp32 scores of up to about 20 (2^-20 of a weight): 2e-5 at the very most.  Without one of the
    lo planes the error is 2^-9 of a value, 1e-3 of a row's norm."""
    import torch
    qh, ql, k, v, kc, vc, table = _operands(H, hd, pos0, rows, page, pos0 + rows)
    hi, lo, err = binding.debug_prompt_attention(qh, ql, pos0, H, kc, vc, table, page, kernel=kernel)
    assert err.item() == 0
    out = (hi.double() + lo.double()).view(rows, H, hd)
    q = (qh.double() + ql.double()).view(rows, H, hd)
    s = torch.einsum("rhd,thd->hrt", q, k.double())
    s.masked_fill_(torch.arange(pos0 + rows, device="cuda")[None, :] > pos0 + torch.arange(rows, device="cuda")[:, None], -float("inf"))
    ref = torch.einsum("hrt,thd->rhd", torch.softmax(s * np.log(2.0), -1), v.double())
    dev = (out - ref).norm(dim=-1) / ref.norm(dim=-1)
    print(f"kernel {kernel} hd {hd} pos0 {pos0} rows {rows}: mean {dev.mean().item():.2e}, largest {dev.max().item():.2e}")
    assert dev.max().item() < 2e-5
    for _ in range(5):                                                # fixed orders of every sum
        hi2, lo2, _ = binding.debug_prompt_attention(qh, ql, pos0, H, kc, vc, table, page, kernel=kernel)
        assert torch.equal(hi2, hi) and torch.equal(lo2, lo)

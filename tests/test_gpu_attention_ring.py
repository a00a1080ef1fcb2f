"""The attention that reads its keys from the weight ring, at the edges of its tiles, splits and pages, against float64."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    import __graft_entry__ as ge
    ge.build()
    from paper_2404_18911_b200 import binding as b
    b.load()
    return torch, b


# no old keys, one key, whole and partial tiles of 16, more than one ring slot, more than one wave of items; both row groups;
# pages smaller and larger than a tile
@pytest.mark.parametrize("H,hd", [(3, 128), (40, 128), (5, 64)])
@pytest.mark.parametrize("M,pos0,ps", [(1, 0, 16), (16, 0, 4), (3, 1, 1), (8, 15, 16), (9, 16, 32), (1, 17, 2), (7, 127, 8), (16, 1040, 16), (2, 3001, 64)])
def test_attention_ring(env, H, hd, M, pos0, ps):
    torch, b = env
    g = torch.Generator(device="cuda").manual_seed(pos0 * 17 + M)
    T, d = pos0 + M, H * hd
    pages = (T + ps - 1) // ps + 3
    # rows that no key lives in hold NaN: nothing of them may reach a result
    kc, vc = (torch.full((pages, H, ps, hd), float("nan"), device="cuda", dtype=torch.bfloat16) for _ in range(2))
    table = torch.randperm(pages, generator=g, device="cuda").to(torch.int32)
    pos = torch.arange(pos0, device="cuda")
    past = torch.empty(2, pos0, H, hd, device="cuda", dtype=torch.bfloat16).normal_(generator=g)
    kc[table[pos // ps].long(), :, pos % ps] = past[0]
    vc[table[pos // ps].long(), :, pos % ps] = past[1]
    qkv = torch.empty(M, 3 * d, device="cuda").normal_(generator=g)
    out = b.op_attention(qkv, pos0, H, hd, 10000.0, kc, vc, table, ps)
    out2 = b.op_attention(qkv, pos0, H, hd, 10000.0, kc, vc, table, ps)      # the appended rows are there already
    assert torch.equal(out, out2)
    new = torch.arange(pos0, T, device="cuda")
    at = table[torch.arange(T, device="cuda") // ps].long()
    K = kc[at, :, torch.arange(T, device="cuda") % ps].double()
    V = vc[at, :, torch.arange(T, device="cuda") % ps].double()
    inv = 10000.0 ** (-2 * torch.arange(hd // 2, device="cuda").double() / hd)
    cs, sn = torch.cos(new.double()[:, None] * inv)[:, None], torch.sin(new.double()[:, None] * inv)[:, None]
    rot = lambda x: torch.cat([x[..., :hd // 2] * cs - x[..., hd // 2:] * sn, x[..., hd // 2:] * cs + x[..., :hd // 2] * sn], -1)
    q, k, v = (qkv.double().reshape(M, 3, H, hd)[:, i] for i in range(3))
    # the rows written: bf16 of the rotated k (half a step of the element; the float32 rotation is good to 1e-5) and of v
    assert ((K[pos0:] - rot(k)).abs() <= 1.01 * 2.0 ** -8 * rot(k).abs() + 1e-5).all() and torch.equal(V[pos0:], v.to(torch.bfloat16).double())
    S = torch.einsum("mhd,thd->hmt", rot(q), K) / hd ** 0.5
    S = S.masked_fill(torch.arange(T, device="cuda")[None, None] > new[None, :, None], float("-inf"))
    ref = torch.einsum("hmt,thd->mhd", torch.softmax(S, -1), V).reshape(M, d)
    # q and p keep 17 bits, fp32 sums: about 5e-6 of the norm is seen, at most 7e-5 of the root mean square in one element
    e = out.double() - ref
    assert e.norm() / ref.norm() < 2e-5 and e.abs().max() < 3e-4 * ref.square().mean().sqrt().clamp_min(0.05)


# heads whose splits run on CTAs of two waves: calls on several streams share the SMs, and a CTA may start when others have ended
@pytest.mark.parametrize("H,hd,M,pos0", [(40, 128, 7, 3001), (12, 64, 16, 6000)])
def test_splits_of_calls_that_overlap(env, H, hd, M, pos0):
    torch, b = env
    g = torch.Generator(device="cuda").manual_seed(1)
    pages = (pos0 + M + 15) // 16
    kc, vc = (torch.empty(pages, H, 16, hd, device="cuda", dtype=torch.bfloat16).normal_(generator=g) for _ in range(2))
    table = torch.randperm(pages, generator=g, device="cuda").to(torch.int32)
    qkv = torch.empty(M, 3 * H * hd, device="cuda").normal_(generator=g)
    ref = b.op_attention(qkv, pos0, H, hd, 10000.0, kc, vc, table, 16)
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(3)]
    state = [(kc.clone(), vc.clone(), b.op_scratch(torch)) for _ in streams]
    torch.cuda.synchronize()
    outs = []
    for _ in range(8):
        for s, (k, v, scratch) in zip(streams, state):
            with torch.cuda.stream(s):
                outs.append(b.op_attention(qkv, pos0, H, hd, 10000.0, k, v, table, 16, scratch=scratch))
    torch.cuda.synchronize()
    assert all(torch.equal(o, ref) for o in outs)


# the attention without the ring: fp32 caches and heads of 32, with one and with many splits, every block of four rows
@pytest.mark.parametrize("bf,H,hd", [(False, 5, 128), (False, 40, 64), (False, 9, 32), (True, 12, 32)])
@pytest.mark.parametrize("M,pos0,ps", [(1, 0, 16), (4, 61, 4), (5, 300, 16), (16, 1500, 32), (1, 6001, 16)])
def test_attention_without_the_ring(env, bf, H, hd, M, pos0, ps):
    torch, b = env
    g = torch.Generator(device="cuda").manual_seed(pos0 + M)
    T, dt = pos0 + M, torch.bfloat16 if bf else torch.float32
    pages = (T + ps - 1) // ps + 1
    kc, vc = (torch.empty(pages, H, ps, hd, device="cuda", dtype=dt).normal_(generator=g) for _ in range(2))
    table = torch.randperm(pages, generator=g, device="cuda").to(torch.int32)
    qkv = torch.empty(M, 3 * H * hd, device="cuda").normal_(generator=g)
    out = b.op_attention(qkv, pos0, H, hd, 10000.0, kc, vc, table, ps)
    assert torch.equal(out, b.op_attention(qkv, pos0, H, hd, 10000.0, kc, vc, table, ps))
    pos = torch.arange(T, device="cuda")
    K, V = (c[table[pos // ps].long(), :, pos % ps].double() for c in (kc, vc))       # with the rows of this pass, as they were written
    new = pos[pos0:].double()
    inv = 10000.0 ** (-2 * torch.arange(hd // 2, device="cuda").double() / hd)
    cs, sn = torch.cos(new[:, None] * inv)[:, None], torch.sin(new[:, None] * inv)[:, None]
    rot = lambda x: torch.cat([x[..., :hd // 2] * cs - x[..., hd // 2:] * sn, x[..., hd // 2:] * cs + x[..., :hd // 2] * sn], -1)
    q, k, v = (qkv.double().reshape(M, 3, H, hd)[:, i] for i in range(3))
    half = 2.0 ** (-8 if bf else -23)                       # half a step of bf16, or a few roundings of fp32; cos and sin are good to 1e-6
    assert ((K[pos0:] - rot(k)).abs() <= 1.01 * half * rot(k).abs() + 1e-5).all() and torch.equal(V[pos0:], v.to(dt).double())
    S = torch.einsum("mhd,thd->hmt", rot(q), K) / hd ** 0.5
    S = S.masked_fill(pos[None, None] > pos[pos0:][None, :, None], float("-inf"))
    ref = torch.einsum("hmt,thd->mhd", torch.softmax(S, -1), V).reshape(M, -1)
    e = out.double() - ref                                  # fp32 sums of up to 6002 terms in blocks
    assert e.norm() / ref.norm() < 5e-6

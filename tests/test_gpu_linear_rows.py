"""The streamed linear operator at the edges of its row variants (4 | 8 | 12 | 16 rows) against float64."""
import numpy as np
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


def _norm(x, gain):
    x = x.double()
    return x * (x.square().mean(-1, keepdim=True) + 1e-6).rsqrt() * gain.double()


# K = 2064: one k16-step past a phase of 2048; N = 5 leaves CTAs without rows; N = 40000: more than one superchunk of 256 rows per CTA
@pytest.mark.parametrize("M", [4, 5, 8, 9, 11, 12, 13, 16])
@pytest.mark.parametrize("N,K", [(5, 16), (1000, 2064), (40000, 512), (4096, 6144)])
def test_rows(env, N, K, M):
    torch, b = env
    g = torch.Generator(device="cuda").manual_seed(N + M)
    W = torch.empty(N, K, device="cuda", dtype=torch.bfloat16).normal_(0, 0.02, generator=g)
    W2 = torch.empty(N, K, device="cuda", dtype=torch.bfloat16).normal_(0, 0.02, generator=g)
    x = torch.empty(M, K, device="cuda").normal_(generator=g)
    gain = 1 + torch.empty(K, device="cuda").normal_(0, 0.1, generator=g)
    resid = torch.empty(M, N, device="cuda").normal_(generator=g)
    n = _norm(x, gain)
    bound = 2e-4 * np.sqrt(K) * 0.02                     # x keeps 17 bits, fp32 sums
    assert (b.op_linear(W, x, gain=gain, resid=resid).double() - (resid + n @ W.double().T)).abs().max() < bound
    ga, up = n @ W.double().T, n @ W2.double().T
    ref = torch.nn.functional.silu(ga) * up
    assert (b.op_linear(W, x, gain=gain, W2=W2).double() - ref).abs().max() < bound * (1 + up.abs().max() + ga.abs().max())
    tok, p, z = b.op_lm_head(W, x, gain, 1e-6, 8.0)
    zr = 8.0 * ga
    assert (z.double() - zr).abs().max() < 8 * bound
    assert torch.equal(tok.long(), z.argmax(-1))
    assert (p.double() - torch.softmax(zr, -1).max(-1).values).abs().max() < 1e-3


# rows per CTA (of 148) at and behind the limits up to which a CTA keeps its warps' sums apart: 32 (M > 12), 48 (M > 8), 64; the pair of
# matrices has twice as many
@pytest.mark.parametrize("M", [1, 4, 8, 9, 12, 16])
@pytest.mark.parametrize("N", [2368, 4736, 4738, 7104, 7300, 9472, 9474])
def test_rows_per_cta(env, N, M):
    test_rows(env, N, 2064, M)


# row lengths around whole phases (2048 or 1024 elements) and those of the 33B and 7B shapes, whose phases are shorter
@pytest.mark.parametrize("M", [1, 7, 12, 16])
@pytest.mark.parametrize("K", [16, 1024, 1040, 2048, 2176, 4112, 6656, 11008])
def test_phases(env, K, M):
    test_rows(env, 300, K, M)


# 9 to 12 rows keep the sums apart from three phases on
@pytest.mark.parametrize("M", [9, 12])
@pytest.mark.parametrize("N", [4738, 7104, 7300])
def test_rows_per_cta_three_phases(env, N, M):
    test_rows(env, N, 4112, M)

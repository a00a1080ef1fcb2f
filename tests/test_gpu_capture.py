"""Calls that do not synchronise, captured into a CUDA graph: every replay is a run of its own, whatever was called in between."""
import pytest

import kg_inputs as ki
from test_gpu_parity import SMALL_BF

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    import __graft_entry__ as ge
    ge.build()
    from paper_2404_18911_b200 import binding as b
    b.load()
    return torch, b


# one decode launch in the graph (prompt pass on the tensor cores), two (the chunked pass is one of them), and seven
@pytest.mark.parametrize("case", ["small-40", "tiny-12", "small-rounds"])
def test_replayed_decode_gives_the_same_tokens(env, case):
    torch, b = env
    shape = ki.get_config("tiny") if case == "tiny-12" else SMALL_BF.with_(d_ffn=1408)      # widths that the tensor-core prompt pass takes
    n, new = (12, 24) if case == "tiny-12" else (40, 24)
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        g = b.KangarooModel(shape, stream=side)
        prompt = ki.make_prompt(shape, n)
        dev = torch.tensor(prompt.tolist(), dtype=torch.int32, device="cuda")

        def work():
            g.reset()
            g.prefill_device(dev)
            if case == "small-rounds":
                for _ in range(3):
                    g.draft(0.6, 4, sync=False)
                    g.verify(sync=False)
            g.decode(new, 0.6, 4, sync=False)

        work()
        ref = g.read_tokens()
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side):
            work()
        work()                                              # a capture alone changes nothing for the calls behind it
        assert g.read_tokens() == ref
        for i in range(4):
            graph.replay()
            assert g.read_tokens() == ref, i
            if i == 1:
                assert g.generate(prompt, new, 0.6, 4)[0] == ref[:new]
        assert len(ref) >= new

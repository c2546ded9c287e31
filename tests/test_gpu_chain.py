"""The unfused calls in a row on one stream, each launched while the one before it ends (programmatic launches), against
the same calls with the device idle between them: bit for bit."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _calls(x, between):
    import paper_2601_08670_gb300 as pced
    B, N = x["B"], x["N"]
    lp, lse = pced.lm_head_logprobs(x["h"], x["w"], logprobs=x["lp"], lse=x["lse"], ws=x["ws"])
    between()
    r = pced.relevance(x["ret"], pced.RET_DENSE, x["rer"])
    between()
    # the log-softmax pass rewrites lp in place right before each of its readers
    beta = pced.adacad_beta(lp, B, N, ws=x["ws"])
    between()
    first = pced.contrastive_select(lp, beta, r, 2.5, ws=x["ws"])
    between()
    pced.lm_head_logprobs(x["h2"], x["w"], logprobs=x["lp"], lse=x["lse"], ws=x["ws"])
    between()
    second = pced.contrastive_select(lp, beta, r, 2.5, ws=x["ws"])
    between()
    pced.lm_head_logprobs(x["h"], x["w"], logprobs=x["lp"], lse=x["lse"], ws=x["ws"])
    between()
    beta2 = pced.adacad_beta(lp, B, N, ws=x["ws"])
    return [lp, lse, r, beta, *first, *second, beta2]


def _clones(out):
    return [t.clone() for t in out]


@pytest.mark.parametrize("B,N,d,V", [(1, 8, 512, 128256), (1, 2, 64, 1000), (4, 16, 256, 30000), (12, 15, 128, 9000)])
def test_calls_in_a_row(cuda_ok, B, N, d, V):
    # 9 and 3 rows: the log-softmax in one pass; 68 rows: after a launch of its own; 192 rows: behind CTA pairs
    import paper_2601_08670_gb300 as pced
    g = torch.Generator(device="cuda").manual_seed(V)
    S = B * (N + 1)

    def normal(*shape, dtype=torch.float32, scale=1.0):
        return (torch.empty(shape, device="cuda").normal_(generator=g) * scale).to(dtype)

    nbytes = max(pced.lm_head_workspace_size(S, V), pced.contrastive_select_workspace_size(B, N, V),
                 int(pced.lib().pced_adacad_beta_workspace_size(B, N, V)))
    x = dict(B=B, N=N, w=normal(V, d, dtype=torch.bfloat16, scale=0.05), h=normal(S, d, dtype=torch.bfloat16),
             h2=normal(S, d, dtype=torch.bfloat16), ret=normal(B, N).clamp_(-1, 1), rer=normal(B, N),
             lp=torch.empty(S, V, device="cuda"), lse=torch.empty(S, device="cuda"), ws=pced.workspace(nbytes, "cuda"))
    for _ in range(20):
        x["h"].normal_(generator=g)
        x["h2"].normal_(generator=g)
        torch.cuda.synchronize()
        want = _clones(_calls(x, torch.cuda.synchronize))
        got = _clones(_calls(x, lambda: None))
        for a, b in zip(want, got):
            assert torch.equal(a, b)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = _calls(x, lambda: None)
    for _ in range(3):
        graph.replay()
        torch.cuda.synchronize()
        for a, b in zip(want, out):
            assert torch.equal(a, b)


def test_calls_joined_from_two_streams_in_a_graph(cuda_ok):
    # a programmatic launch whose stream has just waited for another one
    import paper_2601_08670_gb300 as pced
    B, N, V, d = 1, 8, 20000, 256
    S = B * (N + 1)
    g = torch.Generator(device="cuda").manual_seed(7)
    w = (torch.empty(V, d, device="cuda").normal_(generator=g) * 0.05).bfloat16()
    h = torch.empty(S, d, device="cuda").normal_(generator=g).bfloat16()
    ret, rer = torch.rand(B, N, device="cuda", generator=g), torch.rand(B, N, device="cuda", generator=g)
    side = torch.cuda.Stream()

    def work():
        main = torch.cuda.current_stream()
        side.wait_stream(main)
        with torch.cuda.stream(side):
            r = pced.relevance(ret, pced.RET_DENSE, rer)
        lp, _ = pced.lm_head_logprobs(h, w)
        beta = pced.adacad_beta(lp, B, N)
        main.wait_stream(side)
        return [r, beta, *pced.contrastive_select(lp, beta, r, 2.5)]

    want = _clones(work())
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = work()
    for _ in range(3):
        graph.replay()
        torch.cuda.synchronize()
        for a, b in zip(want, out):
            assert torch.equal(a, b)

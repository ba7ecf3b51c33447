"""Stacks whose arguments bound the layers that need the per-layer kernels (the
top-ratio rule, thresholds that nothing can miss) record those layers without
the device-driven loop, and other stacks take two layers per turn of it: the
results are those of the plain launches bit for bit, and nothing past a length
is written."""
import pytest
import torch

pytestmark = pytest.mark.gpu

RELATIVE, ABSOLUTE, TOP_RATIO = 0, 1, 2
CASES = [
    # layers, L, lens (None: no padding), rule, alphas
    (5, 700, None, TOP_RATIO, [0.9] * 5),                     # 700 ... 459, 414, then 372
    (5, 700, [700, 385, 384, 1], TOP_RATIO, [0.9] * 5),
    (4, 900, None, TOP_RATIO, [1.0, 0.4, 1.0, 1.0]),
    (1, 500, None, TOP_RATIO, [0.5]),
    (4, 500, None, RELATIVE, [0.0] * 4),
    (4, 500, [500, 400, 200, 37], RELATIVE, [0.0, -1.0, 0.0, 0.7]),   # the last alpha prunes
    (3, 640, [640, 1, 384, 385], ABSOLUTE, [-1.0, 0.0, 5.0]),
    (2, 700, None, RELATIVE, [0.0, 0.9]),
    # not bounded: the loop, left after an odd and an even number of layers
    (4, 700, None, RELATIVE, [0.3, 0.0, 0.0, 0.0]),
    (5, 700, [700, 500, 100, 650], RELATIVE, [0.1, 0.9, 0.9, 0.9, 0.9]),
    (6, 700, None, RELATIVE, [1e-3] * 6),                     # nothing pruned, 6 layers
    (7, 700, None, RELATIVE, [1e-3] * 7),
]


@pytest.mark.parametrize("host", [False, True])
@pytest.mark.parametrize("nl,L,lens,rule,alphas", CASES)
def test_graph_equals_plain_launches(nl, L, lens, rule, alphas, host):
    import paper_2310_07109_gb300 as sc
    B, H = 4, 4
    g = torch.Generator(device="cuda")
    g.manual_seed(L + nl)
    Q, K, V = (torch.randn((nl, B, L, H, 64), device="cuda", generator=g).bfloat16()
               for _ in range(3))
    mask = None
    if lens is not None:
        mask = (torch.arange(L)[None, :] < torch.tensor(lens)[:, None]).to(torch.uint8).cuda()
    if host:
        Q, K, V = (t.cpu().pin_memory() for t in (Q, K, V))
        mask = mask if mask is None else mask.cpu().pin_memory()

    def call(plain):
        if host:
            out = sc.new_host_outputs(nl, B, L, H)
            ws = sc.new_stack_host_workspace(nl, B, L, H)
        else:
            out = {"O": torch.empty((nl, B, L, H, 64), dtype=torch.bfloat16, device="cuda"),
                   "scores": torch.empty((nl, B, L), device="cuda"),
                   "pos": torch.empty((nl + 1, B, L), dtype=torch.int32, device="cuda"),
                   "len": torch.empty((nl + 1, B), dtype=torch.int32, device="cuda")}
            ws = sc.new_workspace(B, L, H)
        for t in out.values():
            t.fill_(7)
        fn = sc.stack_forward_host if host else sc.stack_forward
        fn(Q, K, V, mask, [0, 5, L // 2], 64, alphas, out=out, workspace=ws, keep_rule=rule,
           plain_launches=plain)
        torch.cuda.synchronize()
        assert sc.workspace_status(ws) == 0
        return {k: t.cpu() for k, t in out.items()}

    a, b = call(False), call(True)
    for k in a:
        x, y = (t[k].view(torch.int16) if k == "O" else t[k] for t in (a, b))
        if lens is None and rule != TOP_RATIO and not host and all(v <= 0 for v in alphas[:-1]):
            # every layer stays with the per-layer kernels in both (nothing gets short)
            assert int(a["len"][:-1].min()) == L
        assert torch.equal(x, y), k


def _graph_nodes(graph):
    import ctypes
    n = ctypes.c_size_t(0)
    rt = ctypes.CDLL("libcudart.so.13")   # the one that the library has loaded
    assert rt.cudaGraphGetNodes(ctypes.c_void_p(graph.raw_cuda_graph()), None, ctypes.byref(n)) == 0
    return n.value


@pytest.mark.parametrize("rule,alpha,groups", [(RELATIVE, 0.0, 1), (TOP_RATIO, 0.95, 2)])
def test_padded_stack_bounds_are_conditional(rule, alpha, groups):
    """With padding the bound comes from L and the true lengths may be short: the
    layers sit in conditional nodes beside the padding removal and the cluster
    kernel, so that a batch of short sequences launches none of them."""
    import paper_2310_07109_gb300 as sc
    nl, B, L, H = 12, 2, 2048, 2
    Q, K, V = (torch.zeros((nl, B, L, H, 64), device="cuda", dtype=torch.bfloat16)
               for _ in range(3))
    mask = torch.zeros((B, L), dtype=torch.uint8, device="cuda")
    mask[:, :300] = 1
    ws = sc.new_workspace(B, L, H)
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        out = sc.stack_forward(Q, K, V, mask, [0], 64, [alpha] * nl, workspace=ws, keep_rule=rule)
    assert _graph_nodes(graph) == 3 + groups   # with the counters' reset
    for n in (300, 1500, 2048):    # the same graph, other lengths
        mask.zero_()
        mask[:, :n] = 1
        graph.replay()
        torch.cuda.synchronize()
        assert sc.workspace_status(ws) == 0
        want = [n]
        for _ in range(nl):
            r = torch.tensor(alpha, dtype=torch.float32).double().item()
            want.append(want[-1] if rule == RELATIVE else -int(-r * want[-1] // 1))
        assert out["len"][:, 0].tolist() == want

"""Host-buffer stacks whose sequences first get short at the last layer: the final
lengths and positions reach the host buffers, as in the device call."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("alphas", [[0.7], [0.0, 0.7], [0.0, 5.0]])
def test_short_after_the_last_layer(alphas):
    import paper_2310_07109_gb300 as sc
    nl, B, L, H = len(alphas), 2, 520, 2
    g = torch.Generator().manual_seed(5)
    Q, K, V = (3 * torch.randn((nl, B, L, H, 64), generator=g).bfloat16() for _ in range(3))
    mask = torch.ones((B, L), dtype=torch.uint8)
    mask[1, 400:] = 0
    dev = {"O": torch.empty((nl, B, L, H, 64), dtype=torch.bfloat16, device="cuda"),
           "scores": torch.empty((nl, B, L), device="cuda"),
           "pos": torch.empty((nl + 1, B, L), dtype=torch.int32, device="cuda"),
           "len": torch.empty((nl + 1, B), dtype=torch.int32, device="cuda")}
    sc.stack_forward(Q.cuda(), K.cuda(), V.cuda(), mask.cuda(), [0, 9], 64, alphas, out=dev,
                     workspace=sc.new_workspace(B, L, H))
    host = sc.new_host_outputs(nl, B, L, H)
    for t in host.values():
        t.fill_(-9)
    sc.stack_forward_host(Q.pin_memory(), K.pin_memory(), V.pin_memory(), mask.pin_memory(),
                          [0, 9], 64, alphas, out=host,
                          workspace=sc.new_stack_host_workspace(nl, B, L, H))
    torch.cuda.synchronize()
    n = dev["len"].cpu()
    assert int(n[nl].max()) <= 384 < int(n[nl - 1].min())
    assert torch.equal(host["len"], n)
    for b in range(B):
        k = int(n[nl, b])
        assert torch.equal(host["pos"][nl, b, :k], dev["pos"][nl, b, :k].cpu())

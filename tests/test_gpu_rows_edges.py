"""The rows and scores kernels at the sizes where their splits can go wrong: the
64-key items and 128-row tiles at their edges, windows on both sides of an item,
a tile and the five- and nine-tile bands, groups of four global tokens, reloaded
key tiles, and logits that outgrow a row's first reference by far."""
import numpy as np
import pytest
import torch

from parity_utils import check_o, check_scores, layer_case, torch_bf16_to_f64, bits_to_torch

pytestmark = pytest.mark.gpu

CASES = [
    # L, lens, w, globals, scale of the keys
    (65, [65, 64, 63, 1], 63, [0], 2.0),
    (257, [257, 128, 129, 2], 64, [0, 1, 2, 64, 128], 2.0),
    (640, [640, 577], 127, [], 2.0),
    (641, [641, 575], 128, [0, 63, 127, 639], 2.0),
    (900, [900, 833], 255, list(range(0, 900, 57)), 2.0),      # 16 globals
    (1100, [1100], 257, [0, 500], 2.0),                        # nine-tile bands
    (1300, [1300], 511, [0, 640, 1299], 2.0),
    (700, [700, 130], 0, [0, 350], 2.0),
    (700, [700], 64, [0, 699], 40.0),                          # references raised by far
    (640, [640], 639, [5], 40.0),
    # scores: factors found by a thread per (head, global row), rows in batches of
    # four after the first, more key tiles than one batch of them
    (300, [300, 129], 64, list(range(0, 300, 19)), 2.0),       # 16 globals, two head blocks
    (1200, [1200, 1025], 100, [0, 3, 200, 600, 1024, 1199], 2.0),
]


@pytest.mark.parametrize("H", [1, 12, 17])
@pytest.mark.parametrize("L,lens,w,gl,scale", CASES)
def test_layer_edges(L, lens, w, gl, scale, H):
    import paper_2310_07109_gb300 as sc
    if H != 12 and L > 700:
        pytest.skip("head counts are covered by the shorter sequences")
    B = len(lens)
    case = layer_case(B, L, H, lens, w, gl, 0.8, seed=3 * L + w + H, scale_k=scale)
    Q, K, V = (bits_to_torch(case[k], "cuda") for k in ("Q", "K", "V"))
    length, pos = (torch.from_numpy(case[k]).cuda() for k in ("len", "pos"))
    ws = sc.new_workspace(B, L, H)
    # whatever the scratch of the partial results holds, no result may depend on it
    # (a layer reads the caller's rows: test_gpu_stale_rows.py covers compacted ones)
    ws.fill_(255)
    ws[:256] = 0       # (but for the status word)
    O, s, po, lo = sc.layer_forward(Q, K, V, length, pos, w, case["global_pos"], 0.8, workspace=ws)
    assert sc.workspace_status(ws) == 0
    O, s = torch_bf16_to_f64(O), s.cpu().numpy()
    for b, (Oe, se, kept) in enumerate(case["expected"]):
        n = lens[b]
        assert po[b, :int(lo[b])].cpu().tolist() == kept, b
        # the bars of the other parity tests: one bf16 rounding of P and of O
        check_o(O[b, :n], Oe, f"sequence {b}")
        check_scores(s[b, :n], se, f"sequence {b}")
        assert abs(float(s[b, :n].astype(np.float64).sum()) - 1.0) < 1e-4

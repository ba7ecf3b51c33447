"""Rows that hold no current token never reach a result: the operand tiles of the
matrix products take whole 16-, 64- or 128-row blocks, so they contain rows past a
sequence's length (the caller's padding, the next sequence's tokens, whatever the
workspace held before, tokens that a layer pruned).  Here those rows are NaN."""
import numpy as np
import pytest
import torch

import oracle
import workloads as wk
from parity_utils import (bits_to_torch, check_o, check_scores, check_stack, layer_case,
                          resample_stack, torch_bf16_to_f64)

pytestmark = pytest.mark.gpu

NAN = 0x7FC0   # bf16


def _dirty(ws):
    ws.fill_(255)      # NaN in bf16 and in fp32
    ws[:256] = 0       # (but for the status word)
    return ws


def _check_layer_past_length(sc, L, lens, w, gl, H):
    case = layer_case(len(lens), L, H, lens, w, gl, 0.8, seed=5 * L + w + H)
    for k in ("Q", "K", "V"):
        for b, n in enumerate(lens):
            case[k][b, n:] = NAN
    Q, K, V = (bits_to_torch(case[k], "cuda") for k in ("Q", "K", "V"))
    length, pos = (torch.from_numpy(case[k]).cuda() for k in ("len", "pos"))
    ws = _dirty(sc.new_workspace(len(lens), L, H))
    O, s, po, lo = sc.layer_forward(Q, K, V, length, pos, w, case["global_pos"], 0.8, workspace=ws)
    assert sc.workspace_status(ws) == 0
    O, s = torch_bf16_to_f64(O), s.cpu().numpy()
    for b, (Oe, se, kept) in enumerate(case["expected"]):
        n = lens[b]
        assert po[b, :int(lo[b])].cpu().tolist() == kept, b
        check_o(O[b, :n], Oe, f"sequence {b}")
        check_scores(s[b, :n], se, f"sequence {b}")


@pytest.mark.parametrize("gl", [[], [0, 1, 70]], ids=["band", "globals"])
@pytest.mark.parametrize("L,lens,w,H", [
    (640, [577, 0, 640], 64, 4),        # the next sequence's rows; an empty sequence
    (130, [130, 65, 1, 127], 256, 3),   # one to 127 rows past the end of a tile
    (700, [641, 575], 512, 2),          # nine-tile bands
])
def test_layer_rows_past_length(L, lens, w, gl, H):
    import paper_2310_07109_gb300 as sc
    _check_layer_past_length(sc, L, lens, w, gl, H)


@pytest.mark.parametrize("gl", [[], [0, 1, 70]], ids=["band", "globals"])
def test_single_pass_layer_rows_past_length(gl):
    import paper_2310_07109_gb300 as sc
    sc.select_rows_kernel(sc.SC_ROWS_SINGLE_PASS)
    try:
        _check_layer_past_length(sc, 640, [577, 0, 640, 513], 64, gl, 4)
    finally:
        sc.select_rows_kernel(sc.SC_ROWS_TWO_PASS)


STACKS = [
    wk.Workload("pruned_4x700", n_layers=4, B=2, L=700, H=4, w=64, n_extra_global=3,
                ragged=(600, 690), seed=41),
    wk.Workload("unpruned_2x520", n_layers=2, B=2, L=520, H=4, w=128, n_extra_global=2,
                alpha_first=0.0, alpha_last=0.0, ragged=(390, 510), seed=42),
]


@pytest.mark.parametrize("no_tail", [False, True], ids=["with_tail", "per_layer_only"])
@pytest.mark.parametrize("wl", STACKS, ids=[w.name for w in STACKS])
def test_stack_dirty_workspace_and_padding(wl, no_tail):
    import paper_2310_07109_gb300 as sc
    inp, res, _ = resample_stack(wl)
    for k in ("Q", "K", "V"):
        inp[k][:, inp["pad_mask"] == 0] = NAN
    Q, K, V = (bits_to_torch(inp[k], "cuda") for k in ("Q", "K", "V"))
    ws = _dirty(sc.new_workspace(wl.B, wl.L, wl.H))
    out = sc.stack_forward(Q, K, V, torch.from_numpy(inp["pad_mask"]).cuda(), inp["global_pos"],
                           wl.w, inp["alpha"], workspace=ws, no_tail=no_tail)
    assert sc.workspace_status(ws) == 0
    check_stack(wl, res, {"O": torch_bf16_to_f64(out["O"]), "scores": out["scores"].cpu().numpy(),
                          "pos": out["pos"].cpu().numpy(), "len": out["len"].cpu().numpy()})


@pytest.mark.parametrize("w", [64, 230])
@pytest.mark.parametrize("L,rho", [(200, 0.5), (380, 0.7)])
def test_cluster_kernel_rows_of_pruned_tokens(L, rho, w):
    """The first layer's V is NaN at the slots just past the second layer's length."""
    import paper_2310_07109_gb300 as sc
    wl = wk.Workload("stale", n_layers=2, B=2, L=L, H=4, w=w, n_extra_global=2, alpha_first=rho,
                     alpha_last=1.0, keep_rule=oracle.KEEP_TOP_RATIO, seed=43)
    inp, res, _ = resample_stack(wl)
    n1 = int(res["len"][1, 0])
    assert n1 % 16 != 0
    inp["V"][0, :, n1:n1 + 16] = NAN
    Q, K, V = (bits_to_torch(inp[k], "cuda") for k in ("Q", "K", "V"))
    out = sc.stack_forward(Q, K, V, None, inp["global_pos"], wl.w, inp["alpha"],
                           keep_rule=wl.keep_rule)
    np.testing.assert_array_equal(out["len"].cpu().numpy(), res["len"])
    pos, s, O = out["pos"].cpu().numpy(), out["scores"].cpu().numpy(), torch_bf16_to_f64(out["O"])
    for b in range(wl.B):
        np.testing.assert_array_equal(pos[1, b, :n1], res["pos"][1, b, :n1])
        for l in range(2):
            n = int(res["len"][l, b])
            check_scores(s[l, b, :n], res["scores"][l, b, :n], f"layer {l} seq {b}")
        check_o(O[1, b, :n1], res["O"][1, b, :n1], f"seq {b}")


def test_encoder_layer_dirty_workspace():
    """The projections' scratch rows past each length, as the workspace held them."""
    import paper_2310_07109_gb300 as sc
    from test_gpu_encoder import _check_layer, _weights
    L, lens, H = 500, np.array([430, 257], np.int32), 4
    rng = np.random.default_rng(44)
    X = wk.bf16_bits_to_f64(wk.f32_to_bf16_bits(
        rng.standard_normal((2, L, H * 64)).astype(np.float32)))
    w64, wdev = _weights(H * 64, seed=45)
    new = sc.new_encoder_workspace

    class Dirty:
        def __getattr__(self, name):
            return getattr(sc, name)

        @staticmethod
        def new_encoder_workspace(*a):
            return _dirty(new(*a))

    pos = np.tile(np.arange(L, dtype=np.int32), (2, 1))
    _check_layer(Dirty(), X, lens, pos, w64, wdev, L, H, 64, [0, 5], 0.7)

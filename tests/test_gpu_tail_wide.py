"""The cluster kernel's instance for wide windows, whose layers of more than 192
tokens take 64 columns at a time: the window and the token counts on both sides of
its limits, one and two key halves, and odd 64-column remainders, nothing pruned."""
import pytest

import oracle
import workloads as wk
from parity_utils import check_stack
from test_gpu_parity import _run_stack
from test_gpu_tail import sc  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("w", [191, 192, 230])
@pytest.mark.parametrize("L", [192, 193, 225, 256, 257, 321, 384])
def test_wide_windows(sc, L, w):  # noqa: F811
    wl = wk.Workload("wide", n_layers=2, B=2, L=L, w=w, H=4, n_extra_global=2, ragged=(L - 9, L),
                     alpha_first=0.0, alpha_last=0.0, seed=31)
    inp = wk.make_inputs(wl)
    mask = inp["pad_mask"].copy()
    mask[0] = 1   # one sequence of L tokens
    inp = dict(inp, pad_mask=mask)
    res = oracle.stack(inp["Q"], inp["K"], inp["V"], mask, inp["global_pos"], wl.w, inp["alpha"])
    check_stack(wl, res, _run_stack(sc, wl, inp))

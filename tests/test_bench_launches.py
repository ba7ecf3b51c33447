"""bench.py's count of the kernels that a stack call launches as a graph."""
import numpy as np
import pytest

import bench
import workloads as wk

TAIL = 384


def _lens(nl, *first):
    return np.array([list(first)] * (nl + 1))


def _ratio(nl, L, rho):
    return wk.Workload("top", n_layers=nl, B=1, L=L, alpha_first=rho, alpha_last=rho, keep_rule=2)


@pytest.mark.parametrize("wl,lens,padded,want", [
    # prep + cluster kernel
    (wk.Workload("a", n_layers=4, B=1, L=300), _lens(4, 300), True, 2),
    # top ratio without padding: 700, 630, 567, 511, 460, 414, then 373: six layers
    (_ratio(8, 700, 0.9), [[700], [630], [567], [511], [460], [414], [373], [336], [303]], False,
     1 + 3 * 6 - 1 + 1),
    # ... every layer: no cluster kernel
    (_ratio(3, 1000, 0.9), [[1000], [900], [810], [729]], False, 1 + 3 * 3 - 1),
    # ... with padding: layers 0 to 5 and 6 to 8 of the nine that L = 900 allows; the
    # second group only where layer 6 has a long sequence
    (_ratio(9, 900, 0.9), [[500], [450], [405], [365], [329], [297], [268], [242], [218], [197]],
     True, 2 + 1 + 3 * 6 + 1),
    (_ratio(9, 900, 0.9), [[900], [810], [729], [657], [592], [533], [480], [432], [389], [351]],
     True, 2 + 1 + 3 * 6 + 1 + 3 * 3 - 1),
    (_ratio(9, 900, 0.9), _lens(9, 384), True, 2),
    # nothing pruned
    (wk.Workload("u", n_layers=4, B=1, L=500, alpha_first=0., alpha_last=0.), _lens(4, 500), False,
     1 + 3 * 4 - 1),
    (wk.Workload("u", n_layers=4, B=2, L=500, alpha_first=0., alpha_last=0.), _lens(4, 500, 7),
     True, 2 + 1 + 3 * 4 - 1),
    (wk.Workload("u", n_layers=4, B=2, L=500, alpha_first=0., alpha_last=0.), _lens(4, 384, 7),
     True, 2),
    # the loop: layer 0, then two layers a turn
    (wk.Workload("l", n_layers=4, B=1, L=500), [[500], [385], [384], [100], [90]], False,
     1 + 4 + 2 * 4 + 1),
    (wk.Workload("l", n_layers=4, B=1, L=500), [[500], [400], [390], [385], [90]], True,
     2 + 4 + 4 * 4 + 1),
    (wk.Workload("l", n_layers=4, B=1, L=500), [[380], [300], [200], [100], [90]], True, 2 + 4 + 1),
])
def test_graph_launch_count(wl, lens, padded, want):
    assert bench.graph_launch_count(wl, np.asarray(lens), TAIL, padded) == want

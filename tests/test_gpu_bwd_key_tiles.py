"""The two-kernel backward's blocks against the oracle: a sink or gist key tile is walked by one block or shared by the two of
a cluster (an odd number of query tiles, a single one, so that the second block has none), raw key tiles are then dealt out
two to a cluster (an odd number of them, a single one), heads and batch indices share the block order; twice, bit for bit."""
import numpy as np
import pytest
import torch

import paper_2509_15763_b200 as ug
from paper_2509_15763_b200 import synth
from oracle import oracle

from gpu_util import TOL_GRAD, check_close, f64, run_attention

pytestmark = pytest.mark.gpu

CASES = [
    synth.Workload("one_tile_each", 1, 9, 3, 6, 1, 1, 64, seed=501),
    synth.Workload("sinks_only_tile", 1, 4, 4, 4, 2, 1, 64, num_sinks=3, seed=502),
    synth.Workload("odd_raw_tiles", 2, 3 * 128, 3, 60, 4, 2, 64, seed=503),
    synth.Workload("odd_raw_ragged", 3, 4 * 128 + 8, 8, 100, 3, 3, 64, num_sinks=1, seed=504),
    synth.Workload("two_gist_tiles", 1, 130 * 5, 5, 35, 8, 2, 64, num_sinks=130, seed=505),
    synth.Workload("two_gist_tiles_128", 1, 130 * 5, 5, 35, 4, 2, 128, num_sinks=130, seed=506),
    synth.Workload("odd_raw_128", 2, 3 * 128 + 7, 1, 50, 2, 1, 128, seed=507),
    synth.Workload("whole_odd_raw_128", 2, 3 * 128 + 7, 1, 50, 1, 1, 128, seed=508),
    # walks of more than 8 steps (query tiles times heads of a group): these, and some of the above, are shared
    synth.Workload("shared_one_tile_each", 1, 9, 3, 6, 12, 1, 64, seed=511),
    synth.Workload("shared_sinks_only_tile", 1, 4, 4, 4, 8, 1, 64, num_sinks=3, seed=512),
    synth.Workload("shared_odd_raw_tiles", 2, 3 * 128, 3, 60, 12, 2, 64, seed=513),
    synth.Workload("shared_odd_raw_ragged", 3, 4 * 128 + 8, 8, 100, 15, 3, 64, num_sinks=1, seed=514),
    synth.Workload("shared_two_gist_tiles_128", 1, 130 * 5, 5, 35, 8, 2, 128, num_sinks=130, seed=516),
    synth.Workload("shared_odd_raw_128", 2, 3 * 128 + 7, 1, 50, 8, 1, 128, seed=517),
]


@pytest.mark.parametrize("w", CASES, ids=lambda w: w.name)
def test_two_kernel_backward(w):
    flags = ug.FLAG_DETERMINISTIC_DQ if w.head_dim == 128 else 0
    out, again = run_attention(w, flags=flags), run_attention(w, flags=flags)
    k, scale, inp = oracle.window_units(w.window, w.ratio), w.head_dim ** -0.5, out["inputs"]
    want = oracle.attn_bwd(w.num_sinks, w.raw_len, w.ratio, k, scale, *(f64(inp[n]) for n in ("q", "k", "v", "dout")))
    for name, ref in zip(("dq", "dk", "dv"), want):
        assert torch.equal(out[name], again[name])
        check_close(name, f64(out[name]), np.asarray(ref), TOL_GRAD)

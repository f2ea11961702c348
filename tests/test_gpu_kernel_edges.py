"""GPU kernels at the sizes where they can go wrong (tile edges, remainders, the smallest
and largest of a range), against the fp64 oracle or a plain fp64 restatement of the op."""

import numpy as np
import pytest
import torch

from oracle import bag_oracle as O
from paper_2608_09231_gb300 import bag, configs, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gate_kind", ["mlp3", "flux6", "wan6"])
@pytest.mark.parametrize("grid", [(1, 1, 1), (1, 1, 127), (1, 8, 16), (1, 3, 43), (1, 33, 31), (1, 32, 32), (1, 25, 61)])
def test_gate_reduction_and_logit_at_thread_edges(grid, gate_kind, lib):
    """Row counts around the gate's 128 and, from 1024 rows, 512 threads (1, 127, 128, 129, 1023,
    1024, 1525): the logged drift and step change against the oracle's (fp32 sums of fp32 row sums: relative error under
    1e-5), the logit bit for bit on the logged inputs, the decisions from the logged bits."""
    cfg = configs.get_config("tiny", grid=grid, n_txt=5, gate_kind=gate_kind, n_single=1)
    T, B = 4, 2
    ctx = bag.create(cfg, T=T, B=B)
    inp = synth.make_inputs(cfg)
    x = torch.from_numpy(inp["x"].copy()).cuda()
    m, log, nfe = ctx.run(x, torch.from_numpy(inp["txt"]).cuda(), torch.from_numpy(inp["pooled"]).cuda())
    ctx.close()
    g = synth.make_gate_any(cfg["gate_seed"], gate_kind)
    ref = O.sample(cfg, synth.make_weights(cfg), g, inp, T=T, B=B, policy=[int(v) for v in m])
    assert nfe == B and list(m) == O.schedule_from_gate_bits([None] + [int(v) for v in log[1:, 4]], B, T)
    for t in range(1, T):
        drift, step = ref["log"][t]["drift"], ref["log"][t]["s_traj"][2]
        assert abs(float(log[t, 2]) - drift) <= 1e-5 * drift and abs(float(log[t, 13]) - step) <= 1e-5 * step
        cols = [0, 1, 2] if gate_kind == "mlp3" else [8, 9, 10, 7, 2, 13]
        f = [np.float32(v) for v in log[t, cols]]
        z = O.gate_logit(f, g) if gate_kind == "mlp3" else O.gate_logit6(f, g)
        assert z == np.float32(log[t, 3]) and bool(log[t, 4]) == bool(z > 0), t

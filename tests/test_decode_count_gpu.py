"""The decode step advances every row's position count by one, whatever 64-bit value it holds."""
import pytest
import torch

import oracle
from paper_2606_01294_gb300 import ccq
from paper_2606_01294_gb300 import inputs as gen
from tests.helpers import GDN, GLA, TOL, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("backbone", [GLA, GDN])
@pytest.mark.parametrize("H", [1, 2, 16, 64])
@pytest.mark.parametrize("t", [(1 << 52) - 1, 1 << 52, (3 << 52) + 17, (1 << 62) + 5, -7, -(1 << 40)])
def test_decode_counts_of_any_size(backbone, H, t):
    """Counts from 2^52 up and below zero (a caller's offset) are read whole by every head and advanced once a
    step; outputs against the oracle at the same counts."""
    B, d = 3, 64
    S = ccq.CCQState.zeros(B, H, d, d, torch.device("cuda"))
    start = [t, 5, t + 3]
    S.t.copy_(torch.tensor(start))
    tok = gen.make_decode_inputs(backbone, B, H, d, d, dtype=torch.float32, seed=53)["token"]
    T = {n: (None if x is None else x.cuda()) for n, x in tok.items()}
    zero = {"S": S.S.cpu().numpy(), "C": S.C.cpu().numpy(), "m": S.m.cpu().numpy(), "t": S.t.cpu().numpy()}
    for step in range(3):
        o = ccq.decode_step(backbone, T["q"], T["k"], T["v"], T["gate"], T["lam"], S, beta=T["beta"])
        if step == 0:
            ref = oracle.decode_step(backbone, tok["q"], tok["k"], tok["v"], tok["gate"], tok["lam"], zero["S"],
                                     zero["C"], zero["m"], zero["t"], beta=tok["beta"])
            assert rel_err(o, ref["o"]) <= TOL[torch.float32]
        assert S.t.tolist() == [x + step + 1 for x in start]
    ccq.device_status()

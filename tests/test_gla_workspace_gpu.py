"""The GLA forward on a workspace smaller than its finest split asks for: it takes the coarser one the workspace holds."""
import pytest
import torch

from paper_2606_01294_gb300 import ccq
from paper_2606_01294_gb300 import inputs as gen
from tests.helpers import GLA, TOL, compare, gpu_forward, oracle_forward, rel_err

pytestmark = pytest.mark.gpu

SEGMENT = (2 * 128 * 128 + 2 * 128) * 4  # bytes a segment of a sequence


@pytest.mark.parametrize("T,segments", [(576, 0), (700, 0), (1000, 2), (1792, 3)])
@pytest.mark.parametrize("algo", ["chunkwise", "wide"])
def test_forward_on_a_small_workspace(T, segments, algo):
    """Segments of eight chunks or more need 0, 2 or 3 slots a sequence at these lengths (the finest split 3 to 9);
    nothing past them is written, and a sequence that needs none takes any buffer."""
    H = 16
    assert ccq.gla_workspace(1, T, H, 128, 128, "cuda", algo=algo).numel() > segments * H * SEGMENT
    P = gen.make_inputs(GLA, 1, T, H, 128, 128, dtype=torch.bfloat16, seed=95, lam="trained", keys="structured")
    ref = oracle_forward(GLA, P)
    room = torch.zeros(segments * H * SEGMENT + 256, dtype=torch.uint8, device="cuda")
    fits = room[:segments * H * SEGMENT]
    tries = [fits] if segments else [fits, room[4:200]]
    for w in tries:
        o, S = gpu_forward(GLA, P, workspace=w, algo=algo)
        compare(o, S, ref, TOL[torch.bfloat16], f"T={T} {algo}")
        assert int(room[segments * H * SEGMENT:].sum()) == 0
    if segments:
        with pytest.raises(ccq.CCQError, match="workspace"):
            gpu_forward(GLA, P, workspace=room[:fits.numel() - 16], algo=algo)
    ccq.device_status()


def test_workspace_of_the_longest_length():
    """A workspace made for 30 chunks serves 28 and 9, whose finest splits have more segments."""
    w = ccq.gla_workspace(1, 30 * 64, 16, 128, 128, "cuda")
    for nc in (30, 28, 9):
        P = gen.make_inputs(GLA, 1, nc * 64, 16, 128, 128, dtype=torch.bfloat16, seed=96, lam="trained")
        o, S = gpu_forward(GLA, P, workspace=w)
        compare(o, S, oracle_forward(GLA, P), TOL[torch.bfloat16], f"{nc} chunks")


def test_pack_on_a_small_workspace():
    """Packed sequences that run one call each (the wide kernel) on the room of their coarser splits."""
    lens, H = [700, 64, 1000], 16
    cu = [0, 700, 764, 1764]
    P = gen.make_inputs(GLA, 1, cu[-1], H, 128, 128, dtype=torch.bfloat16, seed=97, lam="trained")
    D = {n: x[0].cuda().contiguous() for n, x in P.items() if x is not None}
    w = torch.empty(2 * H * SEGMENT, dtype=torch.uint8, device="cuda")
    o, S = ccq.fwd_varlen(GLA, D["q"], D["k"], D["v"], D["gate"], D["lam"], cu, algo="wide", workspace=w)
    torch.cuda.synchronize()
    for s in range(len(lens)):
        part = {n: (None if x is None else x[:, cu[s]:cu[s + 1]].contiguous()) for n, x in P.items()}
        ref = oracle_forward(GLA, part)
        assert rel_err(o[cu[s]:cu[s + 1]], ref["o"][0]) <= TOL[torch.bfloat16]
        assert rel_err(S.S[s], ref["S"][0]) <= TOL[torch.bfloat16]
    assert S.t.tolist() == lens
    ccq.device_status()

"""GPU parity of the size-dependent paths of the forwards, the decode step and the backward against the
fp64 oracle, at the sizes where their rules and their tiles end."""
import pytest
import torch

import oracle
from paper_2606_01294_gb300 import ccq
from paper_2606_01294_gb300 import inputs as gen
from tests.helpers import (GDN, GLA, TOL, compare, gpu_forward, oracle_forward, rel_err, slice_bh, state_f32,
                           state_to_dev)

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _status():
    yield
    ccq.device_status()


def _resumed(backbone, B, T, H, d, dtype, seed):
    P = gen.make_inputs(backbone, B, T, H, d, d, dtype=dtype, seed=seed, lam="trained", keys="structured")
    prev = gen.make_inputs(backbone, B, 40, H, d, d, dtype=dtype, seed=seed + 1, lam="trained")
    return P, state_f32(oracle_forward(backbone, prev))


@pytest.mark.parametrize("backbone", [GLA, GDN])
@pytest.mark.parametrize("dtype,d", [(torch.float32, 64), (torch.float32, 128), (torch.bfloat16, 64)])
@pytest.mark.parametrize("B,H,T", [(1, 1, 97), (1, 19, 33), (2, 10, 32), (2, 19, 31), (3, 13, 2), (4, 19, 1),
                                   (7, 11, 70)])
def test_recurrent_blocks(backbone, dtype, d, B, H, T):
    """The token-by-token forward in blocks of 32 tokens, on eight CTAs a sequence (up to 19 sequences on the
    152 SMs), four (up to 38), two (up to 76) and one; whole blocks and tails, resumed in place."""
    P, st = _resumed(backbone, B, T, H, d, dtype, 41)
    S = state_to_dev(st)
    o, _ = gpu_forward(backbone, P, S, algo="recurrent", final_state=S)
    compare(o, S, oracle_forward(backbone, P, st), TOL[dtype], f"B={B} H={H} T={T}")


@pytest.mark.parametrize("H,t", [(1, 0), (3, (1 << 33) + 5), (65, 7), (2048, 1), (2049, 2)])
def test_decode_position_count(H, t):
    """Every head of a row reads the row's count before the last one of them advances it (up to 2048 heads; a
    launch of its own above): three steps in place, rows of different counts."""
    B, d = 2, 64
    dev = torch.device("cuda")
    S = ccq.CCQState.zeros(B, H, d, d, dev)
    S.t.copy_(torch.tensor([t, t + 11]))
    tok = gen.make_decode_inputs(GDN, B, H, d, d, dtype=torch.float32, seed=51)["token"]
    T = {n: (None if x is None else x.cuda()) for n, x in tok.items()}
    zero = {"S": S.S.cpu().numpy(), "C": S.C.cpu().numpy(), "m": S.m.cpu().numpy(), "t": S.t.cpu().numpy()}
    for step in range(3):
        o = ccq.decode_step(GDN, T["q"], T["k"], T["v"], T["gate"], T["lam"], S, beta=T["beta"])
        if step == 0:
            ref = oracle.decode_step(GDN, tok["q"], tok["k"], tok["v"], tok["gate"], tok["lam"], zero["S"],
                                     zero["C"], zero["m"], zero["t"], beta=tok["beta"])
            assert rel_err(o, ref["o"]) <= TOL[torch.float32]
    assert S.t.tolist() == [t + 3, t + 14]


@pytest.mark.parametrize("T", [9 * 64 - 1, 9 * 64, 9 * 64 + 1, 1000, 15 * 64 + 1])
def test_gla_short_sequences_split(T):
    """B = 1, H = 16: from nine chunks on the forward is cut into segments of three chunks or more, the last one
    longer or ragged; resumed, the final state written over the initial one."""
    P, st = _resumed(GLA, 1, T, 16, 128, torch.bfloat16, 61)
    S = state_to_dev(st)
    o, _ = gpu_forward(GLA, P, S, final_state=S)
    compare(o, S, oracle_forward(GLA, P, st), TOL[torch.bfloat16], f"T={T}")


@pytest.mark.parametrize("backbone", [GLA, GDN])
@pytest.mark.parametrize("B,H,T", [(3, 17, 16 * 64), (4, 19, 16 * 64 + 1), (4, 16, 17 * 64)])
def test_two_segments_with_half_walks(backbone, B, H, T):
    """51 to 76 sequences of 16 chunks or more: two segments a sequence, the state pass over the first one in
    two halves; sampled heads, resumed."""
    P = gen.make_inputs(backbone, B, T, H, 128, 128, dtype=torch.bfloat16, seed=71, lam="trained", keys="structured")
    prev = gen.make_inputs(backbone, B, 40, H, 128, 128, dtype=torch.bfloat16, seed=72, lam="trained")
    _, S = gpu_forward(backbone, prev)
    st = {n: getattr(S, n).cpu().numpy() for n in ("S", "C", "m", "t")}
    o, fs = gpu_forward(backbone, P, S)
    for b, h in [(0, 0), (B - 1, H - 1)]:
        one = {n: (x[b:b + 1] if n == "t" else x[b:b + 1, h:h + 1]) for n, x in st.items()}
        sub = ccq.CCQState(fs.S[b:b + 1, h:h + 1], fs.C[b:b + 1, h:h + 1], fs.m[b:b + 1, h:h + 1], fs.t[b:b + 1])
        compare(o[b:b + 1, :, h:h + 1], sub, oracle_forward(backbone, slice_bh(P, b, h), one),
                TOL[torch.bfloat16], f"({b}, {h})")


@pytest.mark.parametrize("T", [1, 130])
def test_gdn_backward_workspace_at_sixteen_bytes(T):
    """A workspace that is 16-byte aligned and no more."""
    P = gen.make_inputs(GDN, 1, T, 3, 128, 128, dtype=torch.bfloat16, seed=81, lam="trained", keys="structured")
    G = gen.make_backward_inputs(1, T, 3, 128, 128, dtype=torch.bfloat16, seed=82, prefix=40, state_grads=False)
    D = {n: x.cuda().contiguous() for n, x in P.items()}
    room = ccq.gdn_bwd_workspace(1, T, 3, 128, 128, "cuda")
    w = torch.zeros(room.numel() + 128, dtype=torch.uint8, device="cuda")
    at = (16 - w.data_ptr()) % 128  # 16 bytes past a 128-byte boundary
    g = ccq.gdn_bwd(D["q"], D["k"], D["v"], D["gate"], D["beta"], D["lam"], G["dout"].cuda(),
                    state_to_dev(G["state"]), workspace=w[at:at + room.numel()])
    torch.cuda.synchronize()
    f32 = lambda x: None if x is None else x.float()
    s0 = G["state"]
    ref = oracle.gdn_backward(P["q"], P["k"], P["v"], P["gate"], P["beta"], P["lam"], G["dout"], S0=f32(s0["S"]),
                              C0=f32(s0["C"]), m0=f32(s0["m"]), t0=s0["t"])
    for n in ("dq", "dk", "dv", "dg", "dbeta", "dlambda", "dS0", "dC0", "dm0"):
        assert rel_err(g[n], ref["dlam" if n == "dlambda" else n]) <= TOL[torch.bfloat16], n
    assert int(w[at + room.numel():].sum()) == 0 and int(w[:at].sum()) == 0


@pytest.mark.parametrize("gates", [0.0, -1e-5, -1e-3])
@pytest.mark.parametrize("T", [700, 1000])
def test_gla_short_split_with_gates_near_zero(gates, T):
    """States that hardly forget keep what the segments' boundaries round off: outputs and final states of the split
    walk, the unsplit one and two segments, each against the oracle.  S is a sum of products of two bf16 operands, one of them
    of a bf16-rounded unit key (3 x 2^-9 of its norm); C and m of rounded unit keys (2 x 2^-9)."""
    P = gen.make_inputs(GLA, 1, T, 16, 128, 128, dtype=torch.bfloat16, seed=63, lam="trained", keys="structured",
                        gates=gates)
    ref = oracle_forward(GLA, P)
    for split in (0, 1, 2):
        o, S = gpu_forward(GLA, P, seq_split=split)
        compare(o, S, ref, TOL[torch.bfloat16], f"T={T} gates={gates} split={split}")
        for n, bound in (("S", 3 * 2.0 ** -9), ("C", 2 * 2.0 ** -9), ("m", 2 * 2.0 ** -9)):
            d = getattr(S, n).double().cpu() - torch.as_tensor(ref[n])
            assert float(d.norm()) <= bound * float(torch.as_tensor(ref[n]).norm()), (n, split)

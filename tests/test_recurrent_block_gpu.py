"""GPU checks of the fp32 forward in blocks of 32 tokens (ccq_recurrent_block.cu) where its blocks must not show:
values that are not finite reach no earlier token, and the rows past the sequence change no state."""
import pytest
import torch

from paper_2606_01294_gb300 import ccq
from paper_2606_01294_gb300 import inputs as gen
from tests.helpers import GDN, GLA, TOL, compare, gpu_forward, oracle_forward

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _status():
    yield
    ccq.device_status()


@pytest.mark.parametrize("backbone", [GLA, GDN])
@pytest.mark.parametrize("dtype,d", [(torch.float32, 64), (torch.float32, 128), (torch.bfloat16, 64)])
@pytest.mark.parametrize("B,H", [(1, 2), (2, 10), (2, 19), (7, 11)])  # eight, four, two CTAs a sequence and one
@pytest.mark.parametrize("name", ["q", "k", "v", "gate", "lam"])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_later_tokens_leave_earlier_outputs(backbone, dtype, d, B, H, name, bad):
    """A value at token 37 that is not finite (a right-padded batch whose padding was never written): the outputs
    of tokens 0 to 36, whole block and started block, are bit for bit those of the finite inputs."""
    T, at = 50, 37
    P = gen.make_inputs(backbone, B, T, H, d, d, dtype=dtype, seed=91, lam="trained", keys="structured")
    want, _ = gpu_forward(backbone, P, algo="recurrent")
    P[name] = P[name].clone()
    P[name][:, at:] = bad
    got, _ = gpu_forward(backbone, P, algo="recurrent")
    assert torch.equal(got[:, :at], want[:, :at])


@pytest.mark.parametrize("backbone", [GLA, GDN])
@pytest.mark.parametrize("dtype,d", [(torch.float32, 64), (torch.float32, 128), (torch.bfloat16, 64)])
@pytest.mark.parametrize("B,H", [(1, 2), (2, 10), (2, 19), (7, 11)])
@pytest.mark.parametrize("T", [1, 33, 46])
def test_rows_past_the_sequence_leave_an_infinite_state(backbone, dtype, d, B, H, T):
    """An infinite value in column 5 of the last token: the state's column is infinite after it (kbar v, whose every
    entry is non-zero), and the part of the block past the sequence keeps it so; the other columns are finite."""
    P = gen.make_inputs(backbone, B, T, H, d, d, dtype=dtype, seed=93, lam="trained")
    P["v"] = P["v"].clone()
    P["v"][:, -1, :, 5] = float("inf")
    _, S = gpu_forward(backbone, P, algo="recurrent")
    rest = [c for c in range(d) if c != 5]
    assert bool(torch.isinf(S.S[..., 5]).all()) and bool(torch.isfinite(S.S[..., rest]).all())
    want = torch.sign(P["k"][:, -1].float()).cuda()
    assert torch.equal(torch.sign(S.S[..., 5]), want)


@pytest.mark.parametrize("backbone", [GLA, GDN])
@pytest.mark.parametrize("dtype,d", [(torch.float32, 64), (torch.float32, 128), (torch.bfloat16, 64)])
@pytest.mark.parametrize("B,H", [(1, 15), (1, 16), (3, 12), (1, 37), (4, 19), (7, 11), (17, 9)])
def test_sequence_counts_where_the_cluster_size_changes(backbone, dtype, d, B, H):
    """15 and 16, 36 and 37, 76 and 77 sequences, where the clusters of eight, four and two CTAs stop fitting the
    device at once, and more sequences than SMs."""
    P = gen.make_inputs(backbone, B, 45, H, d, d, dtype=dtype, seed=94, lam="trained", keys="structured")
    o, S = gpu_forward(backbone, P, algo="recurrent")
    compare(o, S, oracle_forward(backbone, P), TOL[dtype], f"B={B} H={H}")


@pytest.mark.parametrize("backbone", [GLA, GDN])
@pytest.mark.parametrize("dtype,d", [(torch.float32, 64), (torch.float32, 128), (torch.bfloat16, 64)])
@pytest.mark.parametrize("B,H,lengths", [(1, 2, (0, 2, 3, 4, 5)), (2, 10, (4, 5, 6, 7)), (2, 19, (5, 6, 7, 8, 10, 11)),
                                         (7, 11, (8, 9, 10, 11, 12, 13, 14, 17, 18)), (10, 16, (17, 18, 22, 23, 33, 37, 38))])
def test_short_sequences_token_by_token_or_in_blocks(backbone, dtype, d, B, H, lengths):
    """Either side of the lengths where the token-by-token kernel hands over to the blocks, resumed in place; one
    kernel's state goes on in the other's."""
    prev = gen.make_inputs(backbone, B, 3, H, d, d, dtype=dtype, seed=98, lam="trained")
    _, S0 = gpu_forward(backbone, prev, algo="recurrent")
    st = {n: getattr(S0, n).cpu().numpy() for n in ("S", "C", "m", "t")}
    for T in lengths:
        P = gen.make_inputs(backbone, B, T, H, d, d, dtype=dtype, seed=99 + T, lam="trained", keys="structured")
        S = ccq.CCQState(S0.S.clone(), S0.C.clone(), S0.m.clone(), S0.t.clone())
        o, _ = gpu_forward(backbone, P, S, algo="recurrent", final_state=S)
        if T == 0:
            assert all(torch.equal(getattr(S, n), getattr(S0, n)) for n in ("S", "C", "m", "t"))
        else:
            compare(o, S, oracle_forward(backbone, P, st), TOL[dtype], f"B={B} H={H} T={T}")


@pytest.mark.parametrize("backbone", [GLA, GDN])
@pytest.mark.parametrize("dtype,d", [(torch.float32, 64), (torch.bfloat16, 128)])
def test_query_whose_square_overflows(backbone, dtype, d):
    """|q|^2 above fp32's range normalises to a zero query, and its output is zero, token by token as in blocks, also
    where m . q itself overflows."""
    for T in (3, 40):
        P = gen.make_inputs(backbone, 1, T, 2, d, d, dtype=dtype, seed=101, lam="trained")
        P["k"] = P["k"].abs()  # m . q: a sum of positive terms
        want, _ = gpu_forward(backbone, P, algo="recurrent")
        P["q"] = P["q"].clone()
        P["q"][:, -1] = 1e38
        got, _ = gpu_forward(backbone, P, algo="recurrent")
        assert torch.equal(got[:, :-1], want[:, :-1]) and not got[:, -1].any()

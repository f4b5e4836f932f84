"""Several samples a thread in the von Mises-Fisher draws: a draw depends on the
seed, its instance and its number alone, so a long list begins with the short
one's draws, whatever the number of samples a thread takes."""
import pytest
import torch

from paper_2602_20376_gb300 import lrq

pytestmark = pytest.mark.gpu


def _draw(O, S):
    C = torch.empty((O.shape[0], S, 4), dtype=torch.complex64, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    lrq.lrq_vmf_sample(O, S, 5, 77, C, st)
    assert int(st.item()) == 0
    return C


@pytest.mark.parametrize("B,S", [(1, 155649), (1, 400003), (3, 130001), (2, 1400000)])
def test_long_list_begins_with_the_short_one(B, S):
    g = torch.Generator(device="cuda").manual_seed(S)
    O = torch.randn((B, 160), device="cuda", generator=g)
    long, short = _draw(O, S), _draw(O, 1001)
    assert torch.equal(long[:, :1001], short)
    tail = long[:, -5:].abs().square().sum(2)  # the last draws are written: unit vectors
    assert (tail - 1).abs().max().item() < 1e-5

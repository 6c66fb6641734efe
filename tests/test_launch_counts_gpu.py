"""Kernels that a call launches, as the benchmark counts them: two where whole sequences are carried, a third for the summaries of
sequences cut into ranges, and a fourth, the scan, where more than four ranges share a sequence; one on the decode path."""
import pytest
import torch

from bench import kernel_launches
from paper_2511_21016_b200 import gka

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def inputs(shape, d):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(67)
    draw = lambda: torch.nn.functional.normalize(torch.randn(*shape, d, generator=gen, device=DEV), dim=-1).bfloat16()
    return draw(), draw(), draw(), torch.full(shape, 0.9, device=DEV), torch.ones(shape, device=DEV)


@pytest.mark.parametrize("heads,T,d,kernels", [(4, 4096, 128, 2), (1, 128 * 60, 128, 4), (40, 128 * 142, 128, 3), (16, 128 * 64, 128, 2),
                                               (4, 4096, 64, 2), (1, 128 * 60, 64, 4)])
def test_kernels_of_a_forward_call(heads, T, d, kernels):
    x = inputs((1, T, heads), d)
    ws = gka.alloc_workspace(1, T, heads, d, torch.device(DEV))
    out, st = gka.gka_fwd_chunked(*x, 1, workspace=ws)
    assert kernel_launches(gka, lambda: gka.gka_fwd_chunked(*x, 1, out=out, state_out=st, workspace=ws)) == kernels


def test_kernels_of_a_decode_step():
    x = inputs((2, 4), 128)
    state = torch.zeros(2, 4, 2 * 128 * 128, device=DEV)
    out = gka.gka_decode_step(state, *x, 1)
    assert kernel_launches(gka, lambda: gka.gka_decode_step(state, *x, 1, out=out)) == 1


@pytest.mark.parametrize("d", [128, 64])
@pytest.mark.parametrize("heads,tiles", [(1, 10), (1, 42), (1, 46), (10, 30), (10, 58), (10, 61), (16, 64), (40, 139), (40, 142),
                                         (155, 16), (155, 24)])
def test_work_items_are_those_of_a_call(heads, tiles, d):
    """Where the library answers with ranges that cut sequences a call has summaries, and where it answers with whole ones none."""
    T = 128 * tiles
    x = inputs((1, T, heads), d)
    ws = gka.alloc_workspace(1, T, heads, d, torch.device(DEV))
    out, st = gka.gka_fwd_chunked(*x, 0, workspace=ws)
    G = gka.gka_fwd_num_work_items(1, T, heads, d)
    cut = any(gka.gka_fwd_work_range(1, T, heads, d, G, i)[3] for i in range(G))
    kernels = kernel_launches(gka, lambda: gka.gka_fwd_chunked(*x, 0, out=out, state_out=st, workspace=ws))
    assert (kernels > 2) == cut

"""The rule that cuts dH's and dW's K loop over the CTAs of a cluster: host arithmetic, so no GPU is needed."""
import itertools

import pytest


@pytest.fixture(scope="module")
def choose():
    from paper_2606_29758_gb300 import _binding, _build
    _build.build()
    return _binding.ps_diag_choose_splitk


WHOLE = (76, 36, 16)   # clusters of 2, 4 and 8 CTAs on 152 SMs


def test_choices_on_the_whole_chip(choose):
    # dH at d = 3584, V = 152064 (2376 blocks of 64): few rows split the most, whole batches not at all
    assert choose(185, 3584, 2376, False, 152, WHOLE) == (8, 2)
    assert choose(100000, 3584, 2376, False, 152, WHOLE) == (1, 2)


@pytest.mark.parametrize("M,N,kb,narrow", [(185, 3584, 2376, False), (400, 3584, 2376, False), (3000, 3584, 2376, False),
                                           (400, 392, 32, False), (1, 8, 32, False), (1024, 128, 125, True)])
def test_cluster_sizes_that_do_not_fit_are_not_chosen(choose, M, N, kb, narrow):
    # a device, or a part of one, that holds no cluster of a size: another size, or no split
    for mask in itertools.product((0, 1), repeat=3):
        at_once = tuple(n * m for n, m in zip(WHOLE, mask))
        ranks, halves = choose(M, N, kb, narrow, 152, at_once)
        assert halves in (1, 2)
        assert ranks == 1 or at_once[{2: 0, 4: 1, 8: 2}[ranks]] > 0
    assert choose(M, N, kb, narrow, 152, (0, 0, 0))[0] == 1

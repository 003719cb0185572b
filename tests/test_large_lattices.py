"""Lattices whose word offsets and site counts need the top bits of 32: two
packings of the same run, which share no address arithmetic, have the same
energies and overlaps (the sites past the old limits lie in the last planes)."""
from __future__ import annotations

import numpy as np
import pytest

from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qisg():
    torch = need_gpu()
    if torch.cuda.mem_get_info()[0] < (100 << 30):
        pytest.skip("needs 100 GB of free device memory")
    from paper_2402_03920_gb300 import qisg as q
    return q


def _run(q, L_tau, slots, layout, word_bits, tile=None):
    lad = q.ladder_linear(0.25, 0.4, slots, 1.0)
    with q.Instance(q.Config(128, L_tau, lad, 2, 1, 7, word_bits=word_bits, layout=layout)) as inst:
        if tile is not None:
            inst.set_tiles((tile, 0), (0, 0))
        inst.sweep(2)
        return (*inst.energies(), inst.overlaps(), inst.permutation())


def _same(a, b):
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("word_bits,slots,tile", [(32, 2, 0), (32, 2, 2), (64, 1, 0)])
def test_samples_above_2_30_sites(qisg, word_bits, slots, tile):
    """17/16 of 2^30 sites: a thread per replica quad and per pair."""
    L_tau = (1 << 16) + (1 << 12)
    _same(_run(qisg, L_tau, slots, qisg.QISG_LAYOUT_SAMPLES, word_bits, tile),
          _run(qisg, L_tau, slots, qisg.QISG_LAYOUT_LANES, 32))


def test_lanes_at_2_31_sites(qisg):
    """The largest lattice, in two word groups of 32 bits and in one of 64."""
    a, b = (_run(qisg, 1 << 17, 17, qisg.QISG_LAYOUT_LANES, w) for w in (32, 64))
    _same(a, b)

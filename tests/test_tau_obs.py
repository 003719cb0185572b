"""Imaginary-time observables on the GPU (Appendix E.1) against the oracle,
in every packing, on configurations after sweeps with PT (so the slots hold
permuted walkers), for a sub-range of samples and with the antiperiodic
boundary."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from tests.gpu_util import make, need_gpu, oracle_state

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qisg():
    need_gpu()
    from paper_2402_03920_gb300 import qisg as q
    q.load()
    return q


@pytest.mark.parametrize("layout,W,L,Lt,n_a,ap", [("SAMPLES", 32, 6, 16, 40, 0), ("SAMPLES", 64, 8, 8, 70, 1),
                                                   ("LANES", 32, 4, 10, 3, 0), ("SITES", 32, 4, 64, 2, 0),
                                                   ("SAMPLES", 32, 24, 32, 33, 0)])
def test_tau_observables_match_oracle(qisg, layout, W, L, Lt, n_a, ap):
    lay = getattr(qisg, f"QISG_LAYOUT_{layout}")
    if layout == "SITES":
        ladder = qisg.ladder_equal(0.25, 0.45, 5)
        inst = qisg.Instance(qisg.Config(L, Lt, ladder, 3, n_a, 41, layout=lay))
        st = oracle.new_state(L, Lt, ladder[:, 0], ladder[:, 1], 3, 41, n_a=n_a, daemon=True)
    else:
        inst, ladder = make(qisg, L, Lt, 0.2, 0.5, 5, 1.0, 3, n_a, 41, layout=lay, word_bits=W, tau_antiperiodic=ap)
        st = oracle_state(ladder, L, Lt, 3, 41, 0, n_a, tau_ap=bool(ap))
    with inst:
        inst.sweep(9)
        oracle.run(st, 9)
        got = inst.tau_observables()
        want = oracle.tau_observables(L, Lt, st.S, st.walker_at)
        for name, g, w in zip(("S1", "S2", "S4"), got[:3], want[:3]):
            assert np.array_equal(g, w), name
        assert np.array_equal(got[3], want[3]) or np.allclose(got[3], want[3], rtol=1e-12, atol=0), "SF"
        lo, n = min(1, n_a - 1), min(2, n_a - 1)
        sub = inst.tau_observables(lo, n)
        for g, w in zip(sub, got):
            assert np.array_equal(g, w[lo:lo + n])


@pytest.mark.parametrize("L,Lt,n_slots,n_rep,pattern", [
    (2, 2, 1, 1, "chain"),       # one lag, 256 threads share it
    (2, 600, 1, 2, "chain"),     # more than 256 lags
    (10, 50, 2, 2, "chain"), (14, 34, 1, 2, "chain"),
    (18, 26, 1, 2, "chain"), (20, 1452, 1, 1, "chain"),   # the last: the largest L_tau shared memory takes at L = 20
    (32, 66, 1, 1, "chain"),
    (12, 20, 1, 2, "layers"), (20, 12, 1, 1, "layers"),   # uniform q~: SF is what its terms' rounding leaves
    (8, 12, 1, 2, "stripes"),                             # one wave at half the wave number only
])
def test_tau_observables_of_given_states(qisg, L, Lt, n_slots, n_rep, pattern):
    rng = np.random.default_rng(L * 1000 + Lt)
    shape = (1, n_rep, n_slots, Lt, L, L)
    if pattern == "chain":
        S = np.cumprod(np.where(rng.random(shape) < 0.2, -1, 1), axis=3)
    elif pattern == "layers":
        S = np.broadcast_to(rng.choice([-1, 1], size=(1, n_rep, n_slots, Lt, 1, 1)), shape)
    else:
        S = rng.choice([-1, 1], size=(1, n_rep, n_slots, Lt, 1, 1)) * np.where(np.arange(L) % 2, -1, 1)
        S = np.where(np.arange(Lt)[:, None, None] % 3 == 0, np.abs(S), np.broadcast_to(S, shape))
    S = np.ascontiguousarray(S.reshape(1, n_rep, n_slots, Lt * L * L), dtype=np.int8)
    wa = np.tile(np.arange(n_slots, dtype=np.int32), (1, n_rep, 1))
    inst, _ = make(qisg, L, Lt, 0.2, 0.5, n_slots, 1.0, n_rep, 1, 3, layout=qisg.QISG_LAYOUT_SAMPLES, word_bits=32)
    with inst:
        inst.set_state(S, wa, 0)
        got = inst.tau_observables()
    want = oracle.tau_observables(L, Lt, S, wa)
    for name, g, w in zip(("S1", "S2", "S4"), got[:3], want[:3]):
        assert np.array_equal(g, w), name
    # the integer sums leave a few roundings at most 16 times enlarged by
    # cancellation (below 1e-13); other lags are the oracle's sums themselves
    assert np.allclose(got[3], want[3], rtol=1e-12, atol=0), "SF"


@pytest.mark.parametrize("L,Lt", [(8, 2), (8, 6), (8, 70), (2, 600), (18, 34)])
def test_cancelling_lags(qisg, L, Lt):
    """Lags evaluated from the definition (a warp each, tau_1 over its lanes)
    beside lags of the integer form: uniform layers, but for one replica with a
    few layers of random spins."""
    rng = np.random.default_rng(L * 1000 + Lt)
    S = np.broadcast_to(rng.choice([-1, 1], size=(1, 3, 2, Lt, 1, 1)), (1, 3, 2, Lt, L, L)).copy()
    S[:, 1, :, :1] = rng.choice([-1, 1], size=(1, 2, 1, L, L))
    half = S[:, 2, :, :, :, : L // 2]   # q~ of period L / 2: no wave at the first wave number
    half[:] = rng.choice([-1, 1], size=(1, 2, Lt, L, L // 2))
    S[:, 2, :, :, :, L // 2:] = half
    S = np.ascontiguousarray(S.reshape(1, 3, 2, Lt * L * L), dtype=np.int8)
    wa = np.tile(np.arange(2, dtype=np.int32), (1, 3, 1))
    inst, _ = make(qisg, L, Lt, 0.2, 0.5, 2, 1.0, 3, 1, 3, layout=qisg.QISG_LAYOUT_SAMPLES, word_bits=32)
    with inst:
        inst.set_state(S, wa, 0)
        got = inst.tau_observables()
    want = oracle.tau_observables(L, Lt, S, wa)
    for name, g, w in zip(("S1", "S2", "S4"), got[:3], want[:3]):
        assert np.array_equal(g, w), name
    # sums of at most 600 terms that are not negative, in another order: below 1e-13
    assert np.allclose(got[3], want[3], rtol=1e-12, atol=0), "SF"


def test_two_threads(qisg):
    """Handles of one L and two L_tau, with different needs of shared memory, in two threads."""
    import threading
    insts = [make(qisg, 16, Lt, 0.2, 0.5, 2, 1.0, 1, 1, 3, layout=qisg.QISG_LAYOUT_LANES)[0] for Lt in (1024, 700)]
    want = [inst.tau_observables() for inst in insts]
    errors = []

    def calls(inst, w):
        try:
            for _ in range(200):
                got = inst.tau_observables()
                assert all(np.array_equal(x, y) for x, y in zip(got, w))
        except Exception as e:   # noqa: BLE001 - reported below
            errors.append(e)

    threads = [threading.Thread(target=calls, args=a) for a in zip(insts, want)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for inst in insts:
        inst.close()

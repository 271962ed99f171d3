"""CPU tests: the top-k similarity-table oracle against its pins, and planted
mistakes (in copies of the oracle, on the CPU) that the pins must catch."""
import numpy as np
import pytest

from oracle import topk_oracle as O
from tests import topk_pins as P


@pytest.mark.parametrize("pin", P.PINS, ids=lambda p: p.__name__)
def test_topk_pin(pin):
    P.run_pin(pin, O.topk_table)


def _order(C, k, tie_high=False, ascending=False):
    V = C.shape[1]
    idx = -np.arange(V) if tie_high else np.arange(V)
    key = C if ascending else -C
    return np.stack([np.lexsort((idx, key[r]))[:k] for r in range(C.shape[0])]).astype(np.int32)


def _no_normalisation(bits, k):
    x = (np.asarray(bits, dtype=np.uint16).astype(np.uint32) << 16).view(np.float32).astype(np.float64)
    return _order(x @ x.T, k)


def _ascending(bits, k):
    En = O.normalize_rows(bits)
    return _order(O.similarities(En), k, ascending=True)


def _ties_high_first(bits, k):
    En = O.normalize_rows(bits)
    return _order(O.similarities(En), k, tie_high=True)


def _normalise_columns(bits, k):
    x = (np.asarray(bits, dtype=np.uint16).astype(np.uint32) << 16).view(np.float32).astype(np.float64)
    n = np.linalg.norm(x, axis=0, keepdims=True)
    n[n == 0] = 1
    y = x / n
    return _order(y @ y.T, k)


def _k_off_by_one(bits, k):
    t = O.topk_table(bits, k)
    return np.concatenate([t[:, 1:], t[:, -1:]], axis=1)


MISTAKES = {"no_normalisation": _no_normalisation, "ascending": _ascending, "ties_high_first": _ties_high_first,
            "normalise_columns": _normalise_columns, "skips_first": _k_off_by_one}


@pytest.mark.parametrize("name", sorted(MISTAKES))
def test_topk_pins_catch_planted_mistake(name):
    failed = False
    for pin in P.PINS:
        try:
            P.run_pin(pin, MISTAKES[name])
        except AssertionError:
            failed = True
    assert failed, f"no pin caught the planted mistake {name}"


def test_division_shortcut_rounds_alike():
    """The normalisation's shortcut in fp32 arithmetic: x * (1 / n) rounds to the same bf16 as x / n wherever its low
    16 bits are more than 4 from the midpoint, for every bf16 mantissa x against random divisors."""
    rng = np.random.default_rng(5)
    x = (np.arange(128, 256, dtype=np.float32) / np.float32(128))[:, None]
    n = np.concatenate([rng.uniform(1, 2, 40000), 1 + 2.0 ** -rng.integers(1, 24, 2000)]).astype(np.float32)[None, :]
    q, p = (x / n).astype(np.float32), (x * (np.float32(1) / n)).astype(np.float32)
    qb, pb = q.view(np.uint32), p.view(np.uint32)
    assert np.abs(qb.astype(np.int64) - pb.astype(np.int64)).max() <= 3
    low = (pb & 0xFFFF).astype(np.int64)
    safe = np.abs(low - 0x8000) > 4

    def bf16(b):
        return (b + 0x7FFF + ((b >> 16) & 1)) >> 16

    assert safe.mean() > 0.999 and np.array_equal(bf16(qb)[safe], bf16(pb)[safe])


"""When the read of the next mini-batch's rows may start, on both sides of the size at which that changes (behind O's update, or
beside it where a mini-batch may hold more than 160 Mi lookups x floats): consecutive mini-batches share cold rows, and nothing
waits between them.  Integer data, bit for bit."""
import dataclasses

import pytest

import gen
from tests import harness

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lookahead", [1, 2])
@pytest.mark.parametrize("order", ["fig8", "eq5"])
@pytest.mark.parametrize("lookups", [(160 << 20) // 128, (160 << 20) // 128 + 1])
def test_read_behind_and_beside_the_popular_update(monkeypatch, lookups, order, lookahead):
    spec = dataclasses.replace(gen.CONFIGS["multi_hot"], batch=60, dim=128, rows=("fixed", 900),
                               hot_policy=("fraction", 40, 100), profile_batches=2)
    monkeypatch.setattr(harness, "max_nnz_of", lambda *a: lookups)
    stats = harness.run_pipelined_check(spec, steps=40, integer=True, native=True, order=order, lookahead=lookahead)
    assert stats["shared_cold_rows"] > 1000

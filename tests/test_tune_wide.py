"""The autotuner times the device-wide build where the batch would take it (host logic, no GPU), and only there."""
import numpy as np
import pytest

from paper_2601_05347_gb300 import tune


def fake_rule(off, **kw):
    return np.diff(off).max() > 100_000 and len(off) < 100


@pytest.mark.parametrize("off,batch_off,wide", [
    ([0, 500_000, 500_010], None, True),                                          # one large index
    ([0, 500_000, 500_010], [0, 500_000, 500_010, 900_000], True),
    ([0, 500_000], np.arange(0, 4097 * 500_000, 500_000), False),                 # the whole batch: blocks
    ([0, 1000, 2000], [0, 1000, 2000, 2_000_000], False),                         # the sample: blocks
    ([0, 1000, 2000], None, False),
])
def test_device_wide_form_is_a_trial_where_the_batch_takes_it(tmp_path, monkeypatch, off, batch_off, wide):
    monkeypatch.setattr(tune, "CACHE", str(tmp_path / "cache.json"))
    calls = []

    def time_config(*a, leaf_size, threads, radix_bits=8, **kw):
        calls.append((leaf_size, threads, radix_bits))
        return {(32, 0, 0): 1.0, (64, 256, 8): 2.0}.get(calls[-1], 9.0)

    monkeypatch.setattr(tune, "time_config", time_config)
    monkeypatch.setattr(tune.psi, "batch_device_wide", fake_rule)
    run = lambda: tune.autotune(off, None, None, None, None, 0, 10, dim=2, kind="spac_h", dist="walks",
                                sizes=np.diff(off), batch_off=batch_off)[:3]
    assert run() == ((32, 0, 0) if wide else (64, 256, 8))
    assert [c for c in calls if c[1] == 0] == ([(p, 0, 0) for p in tune.LEAF_SIZES] if wide else [])
    assert len(calls) == 15 + 3 * wide and run() and len(calls) == 15 + 3 * wide  # the second from the cache
    # a batch of the same mean size that is built by blocks has an entry of its own
    assert tune.cache_key("spac_h", 2, np.diff(off), "walks") + "/wide" * wide in tune._load()

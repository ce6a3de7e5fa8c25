"""The tuner's choice between the named variants and the default, with canned times."""
import pytest

torch = pytest.importorskip("torch")

from paper_2206_01784_gb300 import autotune  # noqa: E402
from paper_2206_01784_gb300 import onesweep as osw  # noqa: E402

pytestmark = pytest.mark.gpu
DEFAULT = osw.OS_TILE_CONFIG_DEFAULT


@pytest.mark.parametrize("default_ms,fastest,expected", [
    (0.5, None, (DEFAULT, 8)), (1.0, None, (DEFAULT, 8)),     # the default wins, or ties
    (1.0, (9, 8, 0.99), (DEFAULT, 8)), (1.0, (9, 8, 0.9), (9, 8)), (1.0, (4, 6, 0.5), (4, 6))])
def test_a_named_variant_has_to_beat_the_default(monkeypatch, default_ms, fastest, expected):
    asked = []

    def canned(*args):
        cfg, d = args[-2:]
        asked.append((cfg, d))
        if cfg == DEFAULT:
            return default_ms
        return fastest[2] if fastest and (cfg, d) == fastest[:2] else 1.0

    monkeypatch.setattr(autotune, "_time_sort", canned)
    saved = autotune.current()
    try:
        table = autotune.tune(key_bits=(32,), value_bytes=(0,), buckets=(1,), steps=1, warmup=0)
        rec = table[(32, 0, 1)]
        assert asked == autotune.candidates() + [(DEFAULT, 8)] and rec["default_ms"] == default_ms
        assert (rec["cfg"], rec["radix_bits"]) == expected
        assert osw.os_get_tile_config_bucket(32, 0, 1) == expected[0]
        assert osw.os_get_radix_bits_bucket(32, 0, 1) == expected[1]
    finally:
        autotune.apply(saved)


def test_small_sorts_are_left_to_the_default():
    # one launch against a memset, a histogram and four passes: no variant comes near
    saved = autotune.current()
    try:
        table = autotune.tune(key_bits=(32,), value_bytes=(4,), buckets=(0,), steps=20, warmup=3)
        assert table[(32, 4, 0)]["cfg"] == DEFAULT and table[(32, 4, 0)]["radix_bits"] == 8
    finally:
        autotune.apply(saved)

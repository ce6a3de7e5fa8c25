"""The process-wide tile variant as state that callers read, set and put back."""
import pytest

from paper_2206_01784_gb300 import autotune
from paper_2206_01784_gb300 import onesweep as osw

TYPES = [(osw.OS_KEY_U32, 32), (osw.OS_KEY_U64, 64)]
SIZES = [1_000, 500_000, 1_200_000, 1_900_000, 2_600_000, 3_000_000, 20_000_000]


def _tiles():
    return [osw.os_sort_workspace_layout(kt, n, vb, 0, kb).tile_keys for kt, kb in TYPES for vb in (0, 4) for n in SIZES]


@pytest.fixture
def unset():
    """Every bucket at the default; afterwards whatever was there before."""
    saved = autotune.current()
    for kb in (32, 64):
        for vb in (0, 4):
            assert osw.os_set_tile_config(kb, vb, osw.OS_TILE_CONFIG_DEFAULT) == osw.OS_OK
    yield
    autotune.apply(saved)


def test_default_takes_its_tile_by_size(unset):
    def tile(n):
        return osw.os_sort_workspace_layout(osw.OS_KEY_U32, n, 4, 0, 32).tile_keys

    assert [tile(n) for n in (1_900_000, 2_600_000, 3_000_000)] == [4096, 6144, 8192]
    assert osw.os_get_tile_config(32, 4) == osw.OS_TILE_CONFIG_DEFAULT
    assert osw.os_tile_config_keys(32, 4, osw.OS_TILE_CONFIG_DEFAULT) == osw.os_tile_config_keys(32, 4, 4)


def test_reading_and_writing_back_changes_nothing(unset):
    before = _tiles()
    for kb in (32, 64):
        for vb in (0, 4):
            assert osw.os_set_tile_config(kb, vb, osw.os_get_tile_config(kb, vb)) == osw.OS_OK
            for b in range(osw.os_num_size_buckets()):
                cfg = osw.os_get_tile_config_bucket(kb, vb, b)
                assert osw.os_set_tile_config_bucket(kb, vb, b, cfg) == osw.OS_OK
    autotune.apply(autotune.current())
    assert _tiles() == before


@pytest.mark.parametrize("cfg", range(12))
def test_a_set_variant_is_read_and_undone(unset, cfg, tmp_path):
    before, saved = _tiles(), autotune.current()
    for kb in (32, 64):
        for vb in (0, 4):
            assert osw.os_set_tile_config(kb, vb, cfg) == osw.OS_OK
            assert osw.os_get_tile_config(kb, vb) == cfg
            tile = osw.os_tile_config_keys(kb, vb, cfg)
            kt = osw.OS_KEY_U32 if kb == 32 else osw.OS_KEY_U64
            assert {osw.os_sort_workspace_layout(kt, n, vb, 0, kb).tile_keys for n in SIZES} == {tile}
    autotune.save(saved, str(tmp_path / "t.json"))
    autotune.apply(autotune.load(str(tmp_path / "t.json")))
    assert _tiles() == before


def test_values_that_name_no_variant_are_refused(unset):
    for bad in (-2, -1, osw.os_num_tile_configs(), 0x100, 0x105, 0x204):
        assert osw.os_set_tile_config(32, 4, bad) == osw.OS_ERR_INVALID_ARG
        assert osw.os_set_tile_config_bucket(32, 4, 1, bad) == osw.OS_ERR_INVALID_ARG
        assert osw.os_tile_config_keys(32, 4, bad) == 0
        if bad != -1:  # (of a call: the process-wide variant)
            assert osw.os_sort_keys_ex(osw.OS_KEY_U32, None, None, 0, 0, 32, None, 0, 0, tile_config=bad) == \
                osw.OS_ERR_INVALID_ARG
    for cfg in (osw.OS_TILE_CONFIG_DEFAULT, 4, -1):
        assert osw.os_sort_keys_ex(osw.OS_KEY_U32, None, None, 0, 0, 32, None, 0, 0, tile_config=cfg,
                                   radix_bits=6) == osw.OS_OK
    assert osw.os_sort_keys_ex(osw.OS_KEY_U32, None, None, 0, 0, 32, None, 0, 0, tile_config=3,
                               radix_bits=6) == osw.OS_ERR_INVALID_ARG

"""Rules of the library's internals, on the CPU."""
import ctypes as C

import pytest

import native_build


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    m = native_build.load("rules", tmp_path_factory.mktemp("native"))
    m.rule_slot_limit.restype = C.c_ulonglong
    m.rule_slot_cap.restype = C.c_uint32
    m.rule_slot_cap.argtypes = [C.c_int64]
    m.rule_chunk_first.restype = C.c_uint32
    m.rule_chunk_first.argtypes = [C.c_ulonglong, C.c_uint32]
    m.rule_rf_grown.restype = m.rule_round_limit.restype = C.c_int64
    m.rule_rf_grown.argtypes = [C.c_int64, C.c_ulonglong]
    return m


@pytest.mark.parametrize("chunk", [32, 64, 128, 256, 512])
def test_every_accepted_list_keeps_all_its_slots(rules, chunk):
    # totals are multiples of the chunk; below the limit a list is accepted
    limit = rules.rule_slot_limit()
    assert limit == 2**32 - 1
    total = (limit - 1) // chunk * chunk
    assert rules.rule_slot_cap(total + total // 8 + 1024) >= total  # (the buffer of a retry)
    for b in [0, chunk, 2**31, *(total - k * chunk for k in range(1, 5 * 512 // chunk))]:
        assert rules.rule_chunk_first(b, chunk) == b


@pytest.mark.parametrize("chunk", [32, 512])
def test_chunks_past_the_limit_do_not_wrap(rules, chunk):
    for b in (2**32 - chunk, 2**32, 2**33 + chunk, 2**63):
        assert rules.rule_chunk_first(b, chunk) + chunk < 2**32
    assert rules.rule_slot_cap(2**33) < 2**32


def test_launch_setup_is_made_once_per_device(rules):
    made = (C.c_int * 16)()
    assert rules.rule_per_device(16, 8, made) == 1
    assert list(made) == [1] * 16
    # (past the table: made on every use)
    made = (C.c_int * 65)()
    assert rules.rule_per_device(65, 1, made) == 1
    assert list(made) == [1] * 65


def test_a_round_that_fits_is_not_refused_for_its_retry(rules):
    limit = rules.rule_round_limit()
    assert limit == 2**30
    for cap in (1 << 16, 10**6, 2**29 + 1, limit - 1):
        for most in (cap + 1, 2 * cap, 2**29, limit - 1, limit):
            if cap < most <= limit:
                assert most <= rules.rule_rf_grown(cap, most) <= limit
        assert rules.rule_rf_grown(cap, limit + 1) > limit  # refused
    assert rules.rule_rf_grown(1 << 16, 100_000) == 200_000

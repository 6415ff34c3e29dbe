"""The bytes that bench.py's roofline rates a screen by, against counts made by
hand from the arrays of the present code."""
import bench


def test_bytes_of_the_24h_screen():
    m = {"boxes": 17392488, "refs": 17392488, "cells": 1, "records": 163639734,
         "open_runs": 28002408, "morton_bits": 12, "split_km": -1000.0, "T": 86400}
    b = bench.phase_bytes(m, 16848)
    N, runs, opens = m["boxes"], m["records"], m["open_runs"]
    # sorted box 32, link 16, node 14 a box; 8 a record
    assert b["traverse"] == N * 62 + (runs + opens) * 8 == 2611471392
    # six passes of 48-bit keys with values: key read twice, value once, both written
    assert b["sort"] == 6 * N * (8 + 8 + 4 + 8 + 4)
    # 15 + 15 + 17 bits: six digits, the last of seven bits left to the emission
    assert b["canon"] == 5 * 24 * (runs + opens) + runs * 32 + opens * 8
    assert b["boxes"] == 56 * 16848 + N * 48


def test_bytes_of_a_small_screen():
    m = {"boxes": 100000, "refs": 100000, "cells": 1, "records": 50000, "open_runs": 9000,
         "morton_bits": 12, "split_km": -1000.0, "T": 6000}
    b = bench.phase_bytes(m, 512)
    assert b["sort"] == 5 * 100000 * 24           # 40 of 48 bits, keys read once a pass
    assert b["canon"] == 3 * 16 * 59000 + 50000 * 32 + 9000 * 8  # 9 + 9 + 13 bits: 7 left


def test_bytes_of_a_decomposed_screen():
    m = {"boxes": 1000000, "refs": 1500000, "cells": 128, "records": 4000000,
         "open_runs": 500000, "morton_bits": 12, "split_km": -1000.0, "T": 86400}
    b = bench.phase_bytes(m, 4000)
    assert b["sort"] == 0
    # 48 + 1 + 7 bits: seven passes over the references
    assert b["build"] == 32000000 + 1500000 * (12 + 7 * 32 + 118)

"""How the decoding attention cuts the tokens' and heads' keys into runs, one per CTA, asked for caches of any length: the runs follow one
another, none is empty, and together they are all units of 16 keys (no GPU needed)."""
import ctypes

import pytest

import paper_2404_05567_b200 as dm

UNITS = [1, 2, 7, 19, 44, 148, 3000, 2 ** 20 + 1, 14_600_000, 2 ** 25 + 5]        # of one (token, head) pair: up to 2^29 keys, 64 GB at 64 wide


def _start(c, units, per, pairs, split):
    f = getattr(dm.lib(), "_ZN5dsmoe16decode_run_startEiiiib")
    f.restype, f.argtypes = ctypes.c_int, [ctypes.c_int] * 4 + [ctypes.c_bool]
    return f(c, units, per, pairs, split)


@pytest.mark.parametrize("units", UNITS)
@pytest.mark.parametrize("sms", [16, 148])
def test_runs_cover_every_unit_once(units, sms):
    for pairs in (1, 2, 3, 5, 16, 74, 147, 148, 149, 256, 1024):
        if pairs * (units + 1) > 2 ** 30:                        # the kernel's own limit
            continue
        split = pairs <= sms
        per = min(sms // pairs, units) if split else -(-pairs // sms)
        ctas = pairs * per if split else -(-pairs // per)
        starts = [_start(c, units, per, pairs, split) for c in range(ctas + 1)]
        assert starts[0] == 0 and starts[-1] == pairs * units
        assert all(a < b for a, b in zip(starts, starts[1:])), (pairs, per, [s for s in starts if s < 0][:3])

"""How the decoding attention cuts the tokens' and heads' keys into aligned runs, one per CTA, where all see equally many keys: asked for caches of
any length, the runs follow one another, none is empty, and together they are all units of 16 keys (no GPU needed)."""
import ctypes

import pytest

import paper_2404_05567_b200 as dm

UNITS = [1, 2, 7, 19, 44, 148, 3000, 2 ** 20 + 1, 2 ** 23 - 1, 2 ** 23, 14_600_000, 2 ** 25 + 5]      # of a (token, head) pair: up to 2^29 keys, 64 GB at 64 wide


def _f(name, result, *args):
    f = getattr(dm.lib(), name)
    f.restype, f.argtypes = result, [ctypes.c_bool if isinstance(a, bool) else ctypes.c_int for a in args]
    return f(*args)


@pytest.mark.parametrize("units", UNITS)
@pytest.mark.parametrize("sms", [16, 148, 255])
def test_runs_cover_every_unit_once(units, sms):
    aligned = 0
    for pairs in (1, 2, 3, 5, 16, 74, 147, 148, 149, 256, 1024):
        if pairs * (units + 1) > 2 ** 30:                        # the kernel's own limit
            continue
        split = pairs <= sms
        per = min(sms // pairs, units) if split else -(-pairs // sms)
        ctas = pairs * per if split else -(-pairs // per)
        longest = -(-units // per) if split else per * units
        if not _f("_ZN5dsmoe17decode_runs_alignEiii", ctypes.c_bool, units, longest, pairs * units):
            continue                                             # equal pieces of the whole list: nothing is multiplied
        aligned += 1
        starts = [_f("_ZN5dsmoe16decode_run_startEiiiib", ctypes.c_int, c, units, per, pairs, split) for c in range(ctas + 1)]
        assert starts[0] == 0 and starts[-1] == pairs * units
        assert all(a < b for a, b in zip(starts, starts[1:])), (pairs, per, [s for s in starts if s < 0][:3])
    assert aligned or units >= 2 ** 23 or sms < 100              # (so few CTAs: a run is more than a hundredth of the units)

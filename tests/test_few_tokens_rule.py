"""The rule that takes a call of one to seven tokens to few_tokens_kernel, asked for any number of SMs (a part of a GPU has fewer than
a layer has experts): the kernel cuts the selected experts' hidden units into equal runs, one per CTA, and reads a run from two
experts at most (no GPU needed)."""
import ctypes

import pytest

import paper_2404_05567_b200 as dm


def _fits(desc, ctas):
    f = getattr(dm.lib(), "_ZN5dsmoe8few_fitsERK16dsmoe_layer_desci")
    f.restype, f.argtypes = ctypes.c_bool, [ctypes.c_void_p, ctypes.c_int]
    return f(ctypes.addressof(desc), ctas)


def _experts_of_a_run(n_act, H, ctas):
    """The most experts that one CTA's run [total * i / ctas, total * (i + 1) / ctas) of hidden units touches."""
    total, most = n_act * H, 0
    for i in range(ctas):
        begin, end = total * i // ctas, total * (i + 1) // ctas
        if end > begin:
            most = max(most, (end - 1) // H - begin // H + 1)
    return most


@pytest.mark.parametrize("ctas", [7, 16, 18, 29, 36, 64, 74, 148])
def test_no_run_reaches_a_third_expert(ctas):
    for E in (1, 2, 8, 16, 29, 30, 32, 36, 37, 64):
        for H in (64, 192, 1408):
            desc = dm.make_desc(3, 512, H, E, dm.BF16, dm.SELECT_ALL)
            if _fits(desc, ctas):
                assert max(_experts_of_a_run(n, H, ctas) for n in range(1, E + 1)) <= 2, (E, H)


def test_a_whole_gpu_takes_every_number_of_experts():
    for E in (1, 32, 64):
        assert _fits(dm.make_desc(7, 6144, 768, E, dm.BF16, dm.SELECT_TOPK, K=1), 148)

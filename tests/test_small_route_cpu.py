"""Which kernels a mode's small spaces take, read from the launches of the library's host
code on the CPU (fake_runtime.py): forte_set_small_route, and a wait budget, which leaves
the choice alone unless it is shorter than the default one."""
import pytest

import fake_runtime as fr

DRIVER = r"""
C = np.zeros((20, 20))
S, G1, G2 = np.zeros_like(C), np.zeros((6,) * 2), np.zeros((6,) * 4)
DEFAULT = 4000000000

def kernels(mode, route, budget):
    ctx = problem(6, 3, 3, mode)
    fg.forte_set_small_route(ctx, route)
    fg.forte_set_wait_budget(ctx, budget)
    out = []
    for call in (lambda: lib.forte_sigma(ctx, C.ctypes.data, S.ctypes.data, 1),
                 lambda: lib.forte_rdms(ctx, C.ctypes.data, G1.ctypes.data, G2.ctypes.data)):
        log()
        assert call() == 0
        names = " ".join(log())
        out.append(next(k for k in ("k_ab_small", "k_ab_df", "k_ab_oz", "k_ab_mma", "k_uv_gram", "k_gram_oz") if k in names))
    lib.forte_destroy(ctx)
    return out

FP64 = ["k_ab_small", "k_uv_gram"]
OWN = {fg.FORTE_DF32: ["k_ab_df", "k_gram_oz"], fg.FORTE_OZ64: ["k_ab_oz", "k_gram_oz"],
       fg.FORTE_BF16X2: ["k_ab_mma", "k_gram_oz"], fg.FORTE_TF32: ["k_ab_mma", "k_gram_oz"]}

def test_routes():
    for mode, own in OWN.items():
        small = [own[0] if own[0] == "k_ab_mma" else FP64[0], FP64[1]]
        waits = [own[0] if own[0] != "k_ab_df" else FP64[0], own[1]]  # the tensor-core kernels
        for budget in (0, 4, DEFAULT - 1, DEFAULT, DEFAULT + 1, 10**12):
            assert kernels(mode, 0, budget) == own, (mode, budget)
            assert kernels(mode, 1, budget) == small, (mode, budget)
            want = waits if 0 < budget < DEFAULT else small
            assert kernels(mode, -1, budget) == want, (mode, budget)
    assert kernels(fg.FORTE_FP64, 0, 4) == FP64

def test_timed_choice_is_made_anew():
    # the restricted sigma's choice was timed against the kernels of the setting before
    a = ctypes.c_int * 3
    for change in (lambda c: fg.forte_set_wait_budget(c, 4), lambda c: fg.forte_set_wait_budget(c, 0),
                   lambda c: fg.forte_set_small_route(c, 0)):
        ctx = problem(6, 3, 3, fg.FORTE_OZ64)
        assert lib.forte_set_gas(ctx, 3, a(2, 2, 2), a(4, 0, 0), a(4, 4, 1), None) == 0
        assert lib.forte_sigma(ctx, C.ctypes.data, S.ctypes.data, 1) == 0
        assert fg.forte_get_gas_route(ctx)[0] >= 0
        change(ctx)
        assert fg.forte_get_gas_route(ctx)[0] == -1
        lib.forte_destroy(ctx)

globals()["test_" + sys.argv[1]]()
"""


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    return fr.compile_fake(tmp_path_factory.mktemp("fake"))


@pytest.mark.parametrize("what", ["routes", "timed_choice_is_made_anew"])
def test_small_route(fake, what):
    fr.run(fake, DRIVER, what)

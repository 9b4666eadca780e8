"""A failed device allocation, at every place where a call makes one: the call reports it,
the next call on the same context succeeds and launches the kernels of an undisturbed
context with no table missing, and nothing is left allocated after the context is gone.
Failed copies leave nothing allocated either.  Memory that only the faster of two routes
needs is not refused for: the other route serves the call.

Runs on the CPU: the library's host code in a process of its own on a runtime that records
launches and fails the allocation or copy it is told to (fake_cudart.cpp)."""
import os
import shutil
import subprocess

import pytest

import fake_runtime as fr

DRIVER = r"""
N, NA, NB = map(int, sys.argv[3:6])
h, eri = si.integrals(N, 2 * N, seed=1)
C = np.zeros((2, math.comb(N, NA), math.comb(N, NB)))
S = np.zeros_like(C)
G = [np.zeros((N,) * k) for k in (2, 4, 6)]

def create():
    return lib.forte_cas_create(N, NA, NB, h.ctypes.data, eri.ctypes.data)

def setup(mode):
    ctx = create()
    assert ctx
    fg.forte_set_precision(ctx, mode)
    fg.forte_set_small_route(ctx, 0)
    log()
    return ctx

def each_failure(make, call):
    # yields (context, codes of the disturbed and of the next call, launches of both)
    k = 0
    while True:
        k += 1
        ctx = make()
        log()
        fake.fake_fail_at(k)
        before = fake.fake_allocs()
        r1 = call(ctx)
        made = fake.fake_allocs() - before
        fake.fake_fail_at(-1)
        if made < k:
            assert r1 == 0
            lib.forte_destroy(ctx)
            assert k > 1, "the call allocates nothing: it tests nothing"
            return
        l1 = log()
        r2 = call(ctx)
        yield k, ctx, r1, r2, l1, log()

def check_call(make, call):
    ctx = make()
    log()
    first = (call(ctx), log())[1]
    steady = (call(ctx), log())[1]
    lib.forte_destroy(ctx)
    known = set(first) | set(steady)
    for k, ctx, r1, r2, l1, l2 in each_failure(make, call):
        what = f"allocation {k}: "
        assert r1 in (fg.FORTE_ERR_ALLOC, fg.FORTE_ERR_CUDA), what + f"code {r1}"
        assert r2 == 0, what + f"the next call returns {r2}: {fg.forte_last_error()}"
        assert set(l1) <= known and set(l2) <= known, what + f"launches {sorted((set(l1) | set(l2)) - known)}"
        it = iter(l2)
        assert all(x in it for x in steady), what + f"launches {l2}, undisturbed {steady}"
        r3, l3 = call(ctx), log()
        assert r3 == 0 and l3 == steady, what + f"third call {l3}"
        lib.forte_destroy(ctx)
        assert fake.fake_live() == 0, what + f"{fake.fake_live()} allocations left"

def sigma(ctx):
    return lib.forte_sigma(ctx, C.ctypes.data, S.ctypes.data, 2)

def test_create():
    for k in range(1, 1000):
        fake.fake_fail_at(k)
        ctx = create()
        if ctx:
            lib.forte_destroy(ctx)
            fake.fake_fail_at(-1)
            assert k > 10
            break
        assert fake.fake_live() == 0, f"allocation {k}: {fake.fake_live()} left"
        log()
    assert fake.fake_live() == 0

def test_sigma(mode):
    check_call(lambda: setup(mode), sigma)

def test_rdms(mode):
    check_call(lambda: setup(mode), lambda ctx: lib.forte_rdms(ctx, C.ctypes.data, G[0].ctypes.data, G[1].ctypes.data))

def test_rdm3(mode):
    check_call(lambda: setup(mode), lambda ctx: lib.forte_rdm3(ctx, C.ctypes.data, G[2].ctypes.data))

def gas(ctx):
    a = ctypes.c_int * 3
    return lib.forte_set_gas(ctx, 3, a(2, 2, 2), a(3, 0, 0), a(4, 4, 1), None)

def test_gas(mode):
    def kept_route():
        ctx = setup(mode)
        fg.forte_set_gas_route(ctx, 1)
        return ctx

    ctx = kept_route()
    assert gas(ctx) == 0
    log()
    kept = (sigma(ctx), log())[1]
    fg.forte_set_gas_route(ctx, 0)
    grid = (sigma(ctx), log())[1]
    lib.forte_destroy(ctx)
    assert any("k_gas_sigma" in x for x in kept) and not any("k_gas_sigma" in x for x in grid)
    served = 0
    for k, ctx, r1, r2, _, _ in each_failure(kept_route, gas):
        what = f"allocation {k}: "
        assert r2 == 0, what + f"the next call returns {r2}: {fg.forte_last_error()}"
        assert sigma(ctx) == 0 and log() == kept, what
        lib.forte_destroy(ctx)
        # the restriction that met the failure: refused, or served by the full grid
        ctx = kept_route()
        fake.fake_fail_at(k)
        assert gas(ctx) == r1
        if r1 == 0:
            log()
            assert sigma(ctx) == 0 and log() == grid, what
            served += 1
        else:
            assert r1 in (fg.FORTE_ERR_ALLOC, fg.FORTE_ERR_CUDA), what + f"code {r1}"
        lib.forte_destroy(ctx)
        assert fake.fake_live() == 0, what + f"{fake.fake_live()} allocations left"
    assert served == 10, f"served without {served} of the lists of the kept-determinant kernel"

def test_gas_copies(mode):
    k = 0
    while True:
        k += 1
        ctx = setup(mode)
        fake.fake_fail_copy_at(k)
        rc = gas(ctx)
        fake.fake_fail_copy_at(-1)
        lib.forte_destroy(ctx)
        assert fake.fake_live() == 0, f"copy {k}: {fake.fake_live()} allocations left"
        if rc == 0:
            break
        assert rc == fg.FORTE_ERR_CUDA
    assert k > 5

name, mode = sys.argv[1], int(sys.argv[2])
globals()["test_" + name](*([mode] if mode >= 0 else []))
"""

SMALL, TILED = (6, 3, 2), (11, 4, 5)  # orbitals, electrons: gathered and tiled FP64 sigma
CALLS = ([("create", -1, SMALL), ("sigma", 0, TILED), ("rdm3", 0, SMALL)] + [("sigma", m, SMALL) for m in range(1, 5)] +
         [("rdms", m, SMALL) for m in (0, 2)] + [("gas", 0, SMALL), ("gas_copies", 0, SMALL)])


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    return fr.compile_fake(tmp_path_factory.mktemp("fake"))


@pytest.mark.parametrize("call,mode,space", CALLS)
def test_failed_allocations_are_reported_and_recovered_from(fake, call, mode, space):
    fr.run(fake, DRIVER, call, mode, *space)


def test_rows_of_different_lengths_are_seen_before_they_are_read(tmp_path):
    """rows_alike guards the kernels that take as many entries from every row as the first has."""
    src = tmp_path / "rows.cpp"
    src.write_text('#include "forte_internal.h"\n#include <cstdio>\nint main() {\n'
                   '  for (const std::vector<int> &p : std::vector<std::vector<int>>{\n'
                   '           {0, 3}, {0, 3, 6, 9}, {0, 3, 6, 8}, {0, 2, 5, 8}, {0, 3, 7, 10}, {0, 0, 0}, {0, 0, 1}, {0}})\n'
                   '    printf("%d", (int)forte::rows_alike(p));\n}\n')
    exe = str(tmp_path / "rows")
    subprocess.run([shutil.which("g++"), "-std=c++17", "-I", fr.include_dir(), "-I", os.path.join(fr.ROOT, "paper_2405_10197_gb300", "csrc"),
                    str(src), "-o", exe], check=True)
    assert subprocess.run([exe], capture_output=True, text=True, check=True).stdout == "11000101"

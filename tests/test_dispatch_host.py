"""CPU check of the dispatch of steps (csrc/sakura_api.cu): its host code,
linked with a stand-in for the CUDA runtime and the launchers
(tests/dispatch_runtime.cpp, dispatch_host.cu) that records every launch and whether it reads
scratch that the library still holds."""
import ctypes
import os
import re

import numpy as np
import pytest

from paper_1402_3325_gb300 import build as sk_build
from paper_1402_3325_gb300 import sakura as sk

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def fake_library(tmp_path_factory):
    import subprocess
    d = tmp_path_factory.mktemp("dispatch")
    nvcc = sk_build._nvcc()
    home = os.path.dirname(os.path.dirname(os.path.realpath(nvcc)))
    objs = [str(d / f"{k}.o") for k in range(3)]
    for src, obj in ((os.path.join(sk_build.CSRC, "sakura_api.cu"), objs[0]),
                     (os.path.join(HERE, "dispatch_host.cu"), objs[1])):
        subprocess.run([nvcc, *sk_build.ARCH, "-O1", "-std=c++17", "-Xcompiler", "-fPIC", "-I",
                        sk_build.INCLUDE, "-I", sk_build.CSRC, "-c", src, "-o", obj], check=True)
    subprocess.run(["g++", "-O1", "-std=c++17", "-fPIC", "-I", os.path.join(home, "include"), "-c",
                    os.path.join(HERE, "dispatch_runtime.cpp"), "-o", objs[2]], check=True)
    out = str(d / "libdispatch.so")
    # -Bsymbolic: the stand-ins come before the runtime, which only registers
    # the object files
    lib64 = os.path.join(home, "lib64")
    subprocess.run(["g++", "-shared", "-Wl,-Bsymbolic", "-o", out, *objs, "-L", lib64,
                    "-Wl,-rpath," + lib64, "-lcudart"], check=True)
    lib = ctypes.CDLL(out)
    lib.dispatch_journal.restype = ctypes.c_char_p
    return lib


class Run:
    """A fresh context of the library with the given options."""

    def __init__(self, lib, **options):
        self.lib = lib
        c = sk.Config()
        lib.sakura_default_config(ctypes.byref(c))
        for k, v in options.items():
            setattr(c, k, v)
        assert lib.sakura_init(ctypes.byref(c)) == 0
        lib.dispatch_journal()

    def __enter__(self):
        return self

    def __exit__(self, *exc):
        self.lib.sakura_finalize()

    def evolve(self, n, dt, order, nsteps=1, host=False):
        x, m = np.zeros(6 * n), np.ones(n)
        p = [a.ctypes.data_as(ctypes.c_void_p) for a in (x, m)]
        fn = self.lib.sakura_evolve_host if host else self.lib.sakura_evolve
        assert fn(*p, ctypes.c_int64(n), ctypes.c_double(dt), order, nsteps) == 0
        return self.lib.dispatch_journal().decode().split()


FORMS = {"seeded": dict(guess=sk.GUESS_FP32), "standard": dict(guess=sk.GUESS_STANDARD),
         "df64": dict(guess=sk.GUESS_FP32, precision=sk.PREC_DF64),
         "literal": dict(guess=sk.GUESS_FP32, precision=sk.PREC_MIXED)}


@pytest.mark.parametrize("host", [False, True])
@pytest.mark.parametrize("n", [33, 700, 1000, 4100, 14000])
@pytest.mark.parametrize("form", FORMS)
def test_a_run_reads_only_scratch_that_it_holds(fake_library, form, n, host):
    # composed steps whose sub-steps lie on both sides of the range of the
    # short solve (1e-18 to 1e18), each in a fresh context
    for order, dts in ((4, (6.5e-19, 7.0e-19, 6.5e17, 2.0 ** -8)), (6, (5e-19, 7e17)),
                       (8, (5e-19, 8e17))):
        for dt in dts:
            with Run(fake_library, pair_mode=sk.PAIRS_SYMMETRIC, **FORMS[form]) as r:
                log = r.evolve(n, dt, order, 2, host)
            assert log and not [k for k in log if k.endswith("!")], (order, dt, log)
            pair = {k for k in log if re.fullmatch("(grp_|small_)?weak|sym|grp|df64|grp_df64", k)}
            assert len(pair) == 1, (order, dt, pair)


@pytest.mark.parametrize("n", [21, 129, 417, 928])
@pytest.mark.parametrize("form", FORMS)
def test_the_flags_choose_the_kernel_they_name(fake_library, form, n):
    for flag, kernel in ((0, "small_weak"), (sk.FLAG_TILES, "weak"), (sk.FLAG_GROUPS, "grp_weak")):
        if form == "df64" and flag == sk.FLAG_GROUPS:
            continue  # the flag is for the other two forms
        with Run(fake_library, pair_mode=sk.PAIRS_SYMMETRIC, flags=flag, **FORMS[form]) as r:
            log = r.evolve(n, 2.0 ** -8, 2)
        assert [k for k in log if k.endswith("weak") and not k.startswith("prep")] == [kernel], log


@pytest.mark.parametrize("n,order", [(1000, 2), (2999, 4), (4100, 2), (14000, 2)])
@pytest.mark.parametrize("form", FORMS)
def test_a_weak_step_launches_the_kernels_for_every_pair_too(fake_library, form, n, order):
    # the device chooses between the two; one launch of each per sub-step
    with Run(fake_library, pair_mode=sk.PAIRS_SYMMETRIC, **FORMS[form]) as r:
        log = r.evolve(n, 2.0 ** -8, order, 2)
    weak = [k for k in log if k in ("weak", "grp_weak")]
    every = [k for k in log if k.startswith("every_")]
    assert len(weak) == len(every) == 2 * (3 if order == 4 else 1)
    assert len(set(every)) == 1 and ("df64" in every[0]) == (form == "df64")

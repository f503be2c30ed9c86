"""A step that fails on the host between the wave-speed pass and the dt kernel must not leave its
maximum to the next one.  The failure is an error code: libdg's own launchers are replaced by ones
that return it when told to (a library loaded before libdg, whose calls between its files then
bind to the replacements)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

FAKE = """
#include <dlfcn.h>
#include <stdlib.h>
extern "C" int fail_dt = 0, fail_cfl = 0;  // fail the n-th call from now
static void *real(const char *name)
{
    static void *h = dlopen(getenv("DG_LIB"), RTLD_NOW | RTLD_NOLOAD);
    return dlsym(h, name);
}
#define STR2(x) #x
#define STR(x) STR2(x)
extern "C" int SYM_DT(const void *m, double cfl, double *dt, double *used, void *s)
{
    if (fail_dt > 0 && --fail_dt == 0) return 2;  // cudaErrorMemoryAllocation
    static auto f = (int (*)(const void *, double, double *, double *, void *))real(STR(SYM_DT));
    return f(m, cfl, dt, used, s);
}
extern "C" int SYM_CFL(int system, const void *a, long long n, void *s)
{
    if (fail_cfl > 0 && --fail_cfl == 0) return 2;
    static auto f = (int (*)(int, const void *, long long, void *))real(STR(SYM_CFL));
    return f(system, a, n, s);
}
"""

SCRIPT = """
import ctypes, sys
import numpy as np, torch
fake = ctypes.CDLL(sys.argv[1], mode=ctypes.RTLD_GLOBAL)
import paper_1609_00098_gb300 as dg
kind = sys.argv[2]

def state(m, speed):
    xyz = m.coords()
    prim = torch.zeros(5, xyz.shape[1], dtype=torch.float64, device="cuda")
    prim[0], prim[1], prim[4] = 1.0, speed, 0.1
    return m.from_prim(prim).contiguous()

def fails(call):
    try:
        call()
    except dg.abi.DGError as e:
        assert e.status == dg.abi.DG_ERR_CUDA
        return
    raise AssertionError("the call did not fail")

if kind == "ensemble":
    ms = [dg.Mesh(system=1, K=(3, 2, 2), n=n, flux=1, precision=1, gamma=4.0 / 3.0) for n in (3, 4)]
    U = [state(m, 0.9) for m in ms]
    ens = dg.abi.dg_ensemble_create([m.h for m in ms], U)
    ctypes.c_int.in_dll(fake, "fail_cfl").value = 2  # the second group's pass
    fails(lambda: dg.abi.dg_ensemble_step(ens, 0.2, int(sys.argv[3])))
    for m, V in zip(ms, U):
        V.copy_(state(m, 0.1))
    dg.abi.dg_ensemble_step(ens, 0.2, int(sys.argv[3]))
    got = torch.zeros(2, dtype=torch.float64, device="cuda")
    dg.abi.dg_ensemble_dt(ens, got)
    want = []
    for m in ms:
        f = dg.Mesh(system=1, K=(3, 2, 2), n=m.n, flux=1, precision=1, gamma=4.0 / 3.0)
        dt = torch.zeros(1, dtype=torch.float64, device="cuda")
        f.rk3_step(state(f, 0.1), cfl=0.2, dt_used=dt)
        want.append(dt.item())
    assert got.tolist() == want, (got.tolist(), want)
else:
    kw = dict(system=int(kind[0]), K=(3, 2, 2), n=4, flux=1, precision=int(kind[1]), gamma=4.0 / 3.0)
    m, f = dg.Mesh(**kw), dg.Mesh(**kw)
    dt = torch.zeros(2, dtype=torch.float64, device="cuda")
    ctypes.c_int.in_dll(fake, "fail_dt").value = 1
    if sys.argv[3] == "step":
        fails(lambda: m.rk3_step(state(m, 0.9), cfl=0.2))
    else:
        fails(lambda: dg.abi.dg_compute_dt(m.h, state(m, 0.9), 0.2, dt))
    m.rk3_step(state(m, 0.1), cfl=0.2, dt_used=dt[:1])
    f.rk3_step(state(f, 0.1), cfl=0.2, dt_used=dt[1:])
    assert dt[0].item() == dt[1].item() > 0.0, dt.tolist()
"""


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    from paper_1609_00098_gb300 import _binding
    from paper_1609_00098_gb300 import build as b
    lib = b.build()
    assert os.path.samefile(lib, _binding.LIB_PATH)
    names = subprocess.run(["nm", "-D", lib], check=True, capture_output=True, text=True).stdout.split()
    sym = {k: next(n for n in names if n.startswith(p)) for k, p in
           (("SYM_DT", "_ZN2dg9launch_dtE"), ("SYM_CFL", "_ZN2dg16launch_cfl_batchE"))}
    d = tmp_path_factory.mktemp("fake")
    src, so, script = str(d / "fake.cpp"), str(d / "libfake.so"), str(d / "run.py")
    for path, text in ((src, FAKE), (script, SCRIPT)):
        with open(path, "w") as f:
            f.write(text)
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", *[f"-D{k}={v}" for k, v in sym.items()], src, "-o", so, "-ldl"],
                   check=True)
    return script, so, lib


@pytest.mark.parametrize("args", [("00", "step"), ("10", "step"), ("01", "step"), ("11", "step"), ("00", "dt"),
                                  ("10", "dt"), ("ensemble", "0"), ("ensemble", "2")])
def test_a_failed_step_leaves_no_maximum(fake, args):
    script, so, lib = fake
    env = dict(os.environ, DG_LIB=lib, PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, script, so, *args], cwd=ROOT, env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout[-500:] + r.stderr[-2000:]

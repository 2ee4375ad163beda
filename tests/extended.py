"""The oracle's fit in the host's long double (64 bits of mantissa on x86, 113 on
Arm), to tell rounding errors of the FP64 fits apart: the oracle's source with
its type exchanged, compiled beside the test run."""
import ctypes
import os
import re
import subprocess

import numpy as np

import oracle


def build(folder):
    """Compile the exchanged source into `folder`; returns the library."""
    src = os.path.join(os.path.dirname(oracle.__file__), "kf_oracle")
    for ext, extra in ((".h", "typedef long double real;\n"), (".c", "#include <tgmath.h>\n")):
        with open(src + ext) as f:
            text = re.sub(r"\bdouble\b", "real", f.read())
        with open(os.path.join(folder, "kf_oracle" + ext), "w") as f:
            f.write(extra + text)
    lib = os.path.join(folder, "libextended.so")
    subprocess.check_call(["gcc", "-O2", "-std=c11", "-ffp-contract=off", "-fPIC", "-shared", "-o", lib,
                           os.path.join(folder, "kf_oracle.c"), "-lm", "-lpthread"])
    return ctypes.CDLL(lib)


def fit_batch(lib, ev, h_max=50.0, n_iter=3, mass=oracle.MUON_MASS, energy_loss=False):
    """oracle.fit_batch (RTS smoother, constant field) in long double."""
    T, S, M = int(ev["n_tracks"]), ev["center"].shape[1], ev["surface_id"].shape[0]
    keep = []

    def arr(a, dtype=np.longdouble):
        keep.append(np.ascontiguousarray(a, dtype=dtype))
        return keep[-1].ctypes.data_as(ctypes.c_void_p)

    ld, c_ld = np.longdouble, ctypes.c_longdouble

    class Material(ctypes.Structure):
        _fields_ = [(n, c_ld) for n, _ in oracle.Material._fields_]

    class Method(ctypes.Structure):
        _fields_ = [("smoother", ctypes.c_int), ("bf_scale", c_ld), ("energy_loss", ctypes.c_int), ("mat", Material),
                    ("map", ctypes.c_void_p)]

    mat = oracle.silicon()
    meth = Method(oracle.SMOOTHER_RTS, 1e4, int(energy_loss),
                  Material(*[getattr(mat, n) for n, _ in oracle.Material._fields_]), None)
    out = {"params": np.zeros((6, T), ld), "cov": np.zeros((21, T), ld), "chi2": np.zeros(T, ld),
           "ndf": np.zeros(T, np.int32), "status": np.zeros(T, np.uint8)}
    ptr = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
    rc = lib.kfo_fit_batch_ex(
        T, arr(ev["offsets"], np.int32), arr(ev["seed_params"]), arr(ev["seed_cov"]), S, arr(ev["center"].T),
        arr(ev["rot"].reshape(9, S).T), arr(ev["x_over_x0"]), ctypes.c_int64(M), arr(ev["surface_id"], np.int32),
        arr(ev["loc"]), arr(ev["cov"]), arr(ev["is_hole"], np.uint8), arr(ev["bfield"]), c_ld(mass), c_ld(h_max),
        n_iter, ctypes.byref(meth), ptr(out["params"]), ptr(out["cov"]), ptr(out["chi2"]), ptr(out["ndf"]),
        ptr(out["status"]), None, 0, T, min(16, os.cpu_count() or 1))
    assert rc == 0
    return out

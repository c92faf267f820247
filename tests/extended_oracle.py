"""The oracle's RHS in extended precision: its source compiled with ``long double`` for ``double``
(64-bit significands on x86, 113 on Arm), to measure the rounding error of FP64 evaluations."""
import ctypes as C
import os
import re
import subprocess
import tempfile

import numpy as np

from oracle import oracle as O

_WRAPPER = """
int ext_rhs(int p, int m, int surf, const double *prm, int nh, int np, int nt, int ny, int nv, const double *verts,
            const int *hv, const int *pv, const int *tv, const int *yv, const double *per, int threads, int ns,
            const double *U, double *hi, double *lo)
{
    long double *v = malloc(sizeof(*v) * 3 * nv), per_x[3];
    for (int i = 0; i < 3 * nv; i++) v[i] = verts[i];
    for (int i = 0; i < 3; i++) per_x[i] = per[i];
    int err = 0;
    void *h = or_create4(p, m, 5, surf, prm[0], prm[1], prm[2], prm[3], prm[4], prm[5], nh, np, nt, ny, nv, v, hv, pv,
                         tv, yv, per_x, &err);
    free(v);
    if (!h) return err ? err : -1;
    or_set_threads(h, threads);
    const long n = or_num_values(h);
    long double *u = malloc(sizeof(*u) * n), *r = malloc(sizeof(*r) * n);
    for (int k = 0; k < ns && err == 0; k++, U += n, hi += n, lo += n) {
        for (long i = 0; i < n; i++) u[i] = U[i];
        err = or_rhs(h, u, r);
        for (long i = 0; i < n; i++) { hi[i] = (double)r[i]; lo[i] = (double)(r[i] - hi[i]); }
    }
    free(u);
    free(r);
    or_destroy(h);
    return err;
}
"""
_lib = None


def _load():
    global _lib
    if _lib is None:
        with open(O.SRC) as f:
            src = f.read()
        src = re.sub(r"\bdouble\b", "long double", src).replace("<math.h>", "<tgmath.h>")
        d = tempfile.mkdtemp(prefix="extended_oracle")
        path, lib = os.path.join(d, "o.c"), os.path.join(d, "o.so")
        with open(path, "w") as f:
            f.write(src + _WRAPPER)
        subprocess.check_call(["gcc", "-O2", "-std=gnu99", "-ffp-contract=off", "-fopenmp", "-shared", "-fPIC", path,
                               "-o", lib, "-lm"])
        _lib = C.CDLL(lib)
    return _lib


def rhs(mesh, p, m, U, gamma=1.4, Pr=0.71, mu=1.0 / 1600, beta=0.5, tau=0.1, p_ref=0.0, surf=False, threads=4):
    """(hi, lo): the RHS of each FP64 state in U [states][values] in extended precision, hi + lo."""
    d = lambda x: np.ascontiguousarray(x, dtype=np.float64)  # noqa: E731
    conn = [np.ascontiguousarray(mesh.get(k, np.zeros((0, n))), dtype=np.int32)
            for k, n in (("hex_v", 8), ("pri_v", 6), ("tet_v", 4), ("pyr_v", 5))]
    verts, per, U, prm = d(mesh["verts"]), d(mesh["period"]), d(U), d([gamma, Pr, mu, beta, tau, p_ref])
    hi, lo = np.zeros_like(U), np.zeros_like(U)
    ptr = lambda a: C.c_void_p(a.ctypes.data)  # noqa: E731
    st = _load().ext_rhs(p, m, int(surf), ptr(prm), *[len(c) for c in conn], len(verts), ptr(verts),
                         *[ptr(c) for c in conn], ptr(per), threads, len(U), ptr(U), ptr(hi), ptr(lo))
    if st != 0:
        raise RuntimeError(f"extended oracle status {st}")
    return hi, lo

"""The oracle's operator and forces in numpy's extended precision (80 or 128 bits):
the same source with its complex type replaced, for errors of FP64 results."""
import os
import types

import numpy as np

LD, CLD = np.longdouble, np.clongdouble


def _module():
    path = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "oracle", "dirac.py")
    with open(path) as f:
        src = f.read()
    mod = types.ModuleType("oracle_dirac_extended")
    exec(compile(src.replace("complex128", "clongdouble"), path, "exec"), mod.__dict__)
    return mod


dirac = _module()


def rel(a, exact):
    """Relative 2-norm distance from the exact result."""
    a = np.asarray(a).reshape(-1).astype(CLD)
    e = np.asarray(exact).reshape(-1)
    return float(np.sqrt(np.sum(np.abs(a - e) ** 2) / np.sum(np.abs(e) ** 2)))

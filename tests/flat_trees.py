"""Matrices with flat elimination trees (nearly all supernodes on one level) and the shape of
their levels in the solves."""
import numpy as np

import paper_2202_09288_gb300 as P
from paper_2202_09288_gb300 import inputs

FLAT = ["diag60", "diag100", "diag152", "blocks100", "bordered100", "arrow140"]


def flat(name):
    """diagN: diagonal; blocksN: N dense 8 x 8 blocks; borderedN: N dense 30 x 30 blocks coupled to 60
    dense unknowns; arrowN: diagonal but for the last unknown's row and column."""
    kind = name.rstrip("0123456789")
    count = int(name[len(kind):])
    if kind == "diag":
        a = np.diag(1.0 + np.arange(float(count)))
    elif kind == "arrow":
        a = np.diag(2.0 + np.arange(float(count)))
        a[-1, :-1] = a[:-1, -1] = 0.5
        a[-1, -1] = 2.0 * count
    else:
        w, border = (8, 0) if kind == "blocks" else (30, 60)
        n = count * w + border
        a = np.zeros((n, n))
        for b in range(count):
            m = inputs.uniform(b + 1, 9, w * w).reshape(w, w)
            a[b * w:(b + 1) * w, b * w:(b + 1) * w] = m @ m.T + w * np.eye(w)
        if border:
            a[-border:, :-border] = 0.1 * inputs.uniform(1, 10, border * (n - border)).reshape(border, -1)
            a[:-border, -border:] = a[-border:, :-border].T
            m = inputs.uniform(2, 10, border * border).reshape(border, border)
            a[-border:, -border:] = m @ m.T + n * np.eye(border)
    A = inputs.from_dense(a, name)
    return A, np.arange(A.n, dtype=np.int32)


def level_tasks(sym):
    """[(tasks, supernodes) of every level], tasks of 128 rows below, at least one per
    supernode; and the ints of the backward solve's arrival counters."""
    ex = sym.export()
    start, level = ex["sn_start"], ex["sn_level"]
    rowptr, _ = P.chol_sym_rows(sym.handle)
    below = np.diff(rowptr) - np.diff(start)
    tasks = (np.maximum(below, 1) + 127) // 128
    nlev = int(level.max()) + 1
    return ([(int(tasks[level == l].sum()), int((level == l).sum())) for l in range(nlev)],
            3 * nlev + 8 + level.size)

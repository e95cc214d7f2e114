"""Writes softplus_nodes.inc: f(x) = ln(1 + exp(-x)) and s(x) = 1 / (1 + exp(x)) at the multiples of 1/32 up to 40.

All derivatives of f are polynomials in s (f' = -s, and s' = -s (1 - s)), so these two values give the Taylor series around a node,
and one 16-byte read replaces the twelve coefficients of a polynomial.  The nearest node is at most 1/64 away; what the series leaves
out after the sixth power is below (1/64)^7 / 5040 * max|f^(7)| = 2e-17.

Run:  python gen_softplus_nodes.py   (rewrites softplus_nodes.inc beside this file)
"""
import os

import numpy as np

STEP = 1 / 32
N_NODES = 40 * 32 + 1


def nodes():
    x = np.arange(N_NODES, dtype=np.longdouble) * np.longdouble(STEP)
    return np.stack([np.log1p(np.exp(-x)), 1 / (1 + np.exp(x))], axis=1).astype(np.float64)


def main():
    path = os.path.join(os.path.dirname(os.path.abspath(__file__)), "softplus_nodes.inc")
    with open(path, "w") as fh:
        fh.write("// Generated by gen_softplus_nodes.py -- do not edit.  Entry i: ln(1 + exp(-x)), 1 / (1 + exp(x)) at x = i / 32.\n")
        rows = ["{%s, %s}" % (float(f).hex(), float(s).hex()) for f, s in nodes()]
        for i in range(0, len(rows), 4):
            fh.write("  " + ", ".join(rows[i:i + 4]) + ",\n")
    print(f"wrote {path}: {N_NODES} nodes")


if __name__ == "__main__":
    main()

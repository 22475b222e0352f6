"""The tile program of levels 18 and 20 (contraction and gathered reverse
pass) against the interpreter's records, in FP64 on the host: energies, basis
values and dE/dM, and that no two records of a phase touch the same slot."""
import os
import re
import sys

import numpy as np
import pytest

PKG = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2510_00193_gb300")
sys.path.insert(0, PKG)
import basisgen  # noqa: E402


def run_records(lv, M, xi):
    """Forward and scattering reverse pass of the interpreter's records."""
    body, tables = basisgen.emit_contract_program(lv)
    prog = [int(v) for v in re.search(r"\{(.*)\}", tables[0]).group(1).split(",")]
    starts = [int(v) for v in re.search(r"\{(.*)\}", tables[1]).group(1).split(",")]
    nv, one, boff = (int(re.search(r"\b%s = (\d+)" % k, body[0]).group(1)) for k in ("NVALUES", "ONE", "BOFF"))
    V, A = np.zeros((nv, M.shape[1])), np.zeros((nv, M.shape[1]))
    V[lv.swept], V[one] = M, 1.0
    recs = []
    for s in starts:
        kind, dst, n = prog[s:s + 3]
        w = 3 if kind == 0 else 1
        recs.append((kind, dst, [prog[s + 3 + w * k:s + 3 + w * (k + 1)] for k in range(n)]))
    for kind, dst, t in recs:
        V[dst] = sum(w * V[a] * V[b] for a, b, w in t) if kind == 0 else np.prod([V[g] for g, in t], axis=0)
    B = V[boff:boff + lv.m]
    A[boff:boff + lv.m] = xi[:, None]
    for kind, dst, t in reversed(recs):
        for k, u in enumerate(t):
            if kind == 0:
                A[u[0]] += u[2] * A[dst] * V[u[1]]
                A[u[1]] += u[2] * A[dst] * V[u[0]]
            else:
                A[u[0]] += A[dst] * np.prod([V[g] for q, (g,) in enumerate(t) if q != k] + [np.ones(M.shape[1])], axis=0)
    return B, A[lv.swept]


def run_tile(lv, M, xi):
    """The encoded words, slab by slab, as the kernel reads them."""
    tp = basisgen.TileProgram(lv)
    words, slabs, off = tp.encode()
    S = np.full((tp.slots, M.shape[1]), np.nan)
    S[lv.swept], S[tp.one], S[tp.zero] = M, 1.0, 0.0
    B = None
    for p in range(len(off) - 1):
        if p == tp.n_forward:
            B = S[tp.basis].copy()
            S[[tp.aoff + b for b in tp.basis]] = xi[:, None]
        before, done = S.copy(), set()
        for first, meta in slabs[off[p]:off[p + 1]]:
            for lane in range(basisgen.TILE_LANES):
                col = []
                for q in range(meta >> 1):
                    at = 4 * (first + q * basisgen.TILE_LANES + lane)
                    col += words[at:at + 4]
                dst = col[0] & 0x1FFF
                if dst == basisgen.TILE_NONE:
                    continue
                assert dst not in done and dst < tp.slots
                done.add(dst)
                acc = before[dst].copy() if col[0] >> 13 & 1 else np.zeros(M.shape[1])
                for t in col[1:]:
                    x, y, w = t & 0x1FFF, t >> 13 & 0x1FFF, tp.weights[t >> 26]
                    assert w == 1 or not meta & 1
                    acc += w * before[x] * before[y]   # a slot written in this phase would differ from `before`
                S[dst] = acc
        for first, meta in slabs[off[p]:off[p + 1]]:    # nothing that the phase writes is read in it
            for k in range(16 * 4 * (meta >> 1)):
                t = words[4 * first + k]
                if k % 4 == 0 and k < 64:
                    continue
                assert not {t & 0x1FFF, t >> 13 & 0x1FFF} & done
    return B, S[[tp.aoff + c for c in lv.swept]]


@pytest.mark.parametrize("level", [18, 20])
def test_tile_program(level):
    lv = basisgen.Level(level)
    g = np.random.default_rng(level)
    # moments of random neighbourhoods: the components with a z-exponent of 2 and more follow from |u| = 1
    u = g.normal(size=(3, 7, 3))
    u /= np.linalg.norm(u, axis=-1, keepdims=True)
    f = g.normal(size=(3, 7, lv.nmu)) * 0.3
    M = np.array([(f[..., mu] * u[..., 0] ** K[0] * u[..., 1] ** K[1] * u[..., 2] ** K[2]).sum(1)
                  for mu, K in (lv.comps[c] for c in lv.swept)])
    xi = g.normal(size=lv.m)
    b0, d0 = run_records(lv, M, xi)
    b1, d1 = run_tile(lv, M, xi)
    # both are sums of at most a few thousand FP64 products of the same values
    assert np.abs(b1 - b0).max() <= 1e-11 * np.abs(b0).max()
    assert np.abs(d1 - d0).max() <= 1e-11 * np.abs(d0).max()

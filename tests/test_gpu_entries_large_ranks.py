"""Entries of a handle with a rank above 11600: the path of an index then needs
all of the shared memory for its two vectors.  The handle is loaded from a
checkpoint whose left half has rows of full rank (but for ten of its top node)
and whose other ranks are 1, so that entries can be formed on the host."""
import ctypes as C
import struct

import numpy as np
import pytest

from oracle.tree import halving_tree
from test_gpu_product import hss  # noqa: F401

pytestmark = pytest.mark.gpu


def test_rank_12000(hss, tmp_path):
    import torch

    import gpu_util as gu
    n, leaf, short = 24200, 100, 10
    rng = np.random.default_rng(1)
    nodes = halving_tree(n, leaf)
    kr, kc = [0] * len(nodes), [1] * len(nodes)
    mr, mc = [0] * len(nodes), [2] * len(nodes)
    kc[0] = mc[0] = 0
    for t in reversed(nodes[1:]):
        full = t.lo + t.size <= nodes[1].size
        mr[t.idx] = t.size if t.is_leaf else sum(kr[c] for c in t.children)
        kr[t.idx] = (mr[t.idx] if full else 1) - (short if t.idx == 1 else 0)
        if t.is_leaf:
            mc[t.idx] = t.size
    assert kr[1] > 11622
    path = tmp_path / "big.hss"
    with open(path, "wb") as f:
        def arr(a):
            f.write(struct.pack("q", -1 if a is None else a.size))
            if a is not None:
                f.write(np.ravel(a, order="F").tobytes())

        f.write(b"HSSGEN01" + struct.pack("8i", n, len(nodes), max(t.level for t in nodes), 1, 1, 4, 0, leaf))
        f.write(struct.pack("q", C.sizeof(hss.hss_stats)) + bytes(C.sizeof(hss.hss_stats)))
        for t in nodes:
            ch = t.children if t.children else [-1, -1]
            f.write(struct.pack("12i", t.lo, t.size, t.level, t.parent, *ch, int(t.is_leaf), 2,
                                mr[t.idx], kr[t.idx], mc[t.idx], kc[t.idx]))
            t.g = []
            for m, k in ((mr[t.idx], kr[t.idx]), (mc[t.idx], kc[t.idx])):
                piv, X = rng.permutation(m).astype(np.int32), rng.uniform(-1, 1, (k, m - k))
                t.g.append((k, np.argsort(piv), X))
                for a in (piv, X, np.full(k, t.lo, np.int32)):
                    arr(a if t.idx else None)
            arr(rng.standard_normal((t.size, t.size)) if t.is_leaf else None)
            for a, b in ((0, 1), (1, 0)):
                B = None if t.is_leaf else rng.standard_normal((kr[t.children[a]], kc[t.children[b]]))
                t.g.append(B)
                arr(B)

    def row(t, side, u):
        """u (a row of the node's sample as {position: value}) times the node's basis, dense."""
        k, inv, X = t.g[side]
        out = np.zeros(k)
        for q, v in u:
            pos = inv[q]
            if pos < k:
                out[pos] += v
            else:
                out += v * X[:, pos - k]
        return out

    def entry(i, j):
        t, (u, v) = nodes[0], (None, None)
        while not t.is_leaf:
            sides = [0 if x < nodes[t.children[1]].lo else 1 for x in (i, j)]
            if sides[0] != sides[1]:
                break
            t = nodes[t.children[sides[0]]]
        assert not t.is_leaf   # (the indices are in different leaves)
        vec = []
        for side, x, s in ((0, i, sides[0]), (1, j, sides[1])):
            path, c = [], nodes[t.children[s]]
            while True:
                path.append(c)
                if c.is_leaf:
                    break
                c = nodes[c.children[0 if x < nodes[c.children[1]].lo else 1]]
            w = row(path[-1], side, [(x - path[-1].lo, 1.0)])
            for p, a in zip(path[-2::-1], path[:0:-1]):
                off = 0 if p.children[0] == a.idx else (kr, kc)[side][p.children[0]]
                w = row(p, side, [(off + q, w[q]) for q in np.flatnonzero(w)])
            vec.append(w)
        return vec[0] @ t.g[2 if sides[0] == 0 else 3] @ vec[1]

    # rows of the left half (among them some beyond the top node's rank), and of the right
    k, inv, _ = nodes[1].g[0]
    I = np.concatenate([rng.integers(0, nodes[1].size, 40), rng.integers(nodes[2].lo, n, 3)]).astype(np.int32)
    J = np.concatenate([rng.integers(nodes[2].lo, n, 4), rng.integers(0, nodes[1].size, 4)]).astype(np.int32)
    H = hss.hss_load(str(path))
    out = torch.empty((J.size, I.size), dtype=torch.float64, device=gu.dev()).t()
    every = torch.arange(nodes[1].size, device=gu.dev(), dtype=torch.int32)
    col = torch.empty((1, every.numel()), dtype=torch.float64, device=gu.dev()).t()
    dI, dJ = (torch.from_numpy(x).to(gu.dev()) for x in (I, J))
    hss.hss_get_entries(H, dI, dJ, out)
    leaf_of = {}
    for t in nodes:
        if t.is_leaf:
            leaf_of.update({x: t.idx for x in range(t.lo, t.lo + t.size)})
    got = out.cpu().numpy()
    for a, i in enumerate(I):
        for b, j in enumerate(J):
            if leaf_of[i] != leaf_of[j]:
                e = entry(int(i), int(j))
                assert abs(got[a, b] - e) <= 1e-12 * max(1.0, abs(e)) * 120   # sums of up to 12000 terms below 1 times normals
    # one column of the left half against the right: the product's own
    hss.hss_get_entries(H, every, dJ[:1], col)
    X = torch.zeros((1, n), dtype=torch.float64, device=gu.dev()).t()
    X[int(J[0]), 0] = 1.0
    Y = torch.empty((1, n), dtype=torch.float64, device=gu.dev()).t()
    hss.hss_matvec(H, X, Y)
    assert (Y[:nodes[1].size, 0] - col[:, 0]).abs().max().item() <= 1e-10

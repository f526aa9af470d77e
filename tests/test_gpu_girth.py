"""The bound of the girth that a loaded graph gets (k_girth): the girth itself where a search stays within its
list, never more than it elsewhere; and the short neighbour
lists written beside it."""
import ctypes
import re
import subprocess

import numpy as np
import pytest

from paper_2508_21287_gb300 import inputs as I

pytestmark = pytest.mark.gpu
GIRTH_MAX = 32


@pytest.fixture(scope="module")
def launch():
    from paper_2508_21287_gb300 import build
    path = build.build()
    names = subprocess.run(["nm", "-D", "--defined-only", path], capture_output=True, text=True).stdout
    return getattr(ctypes.CDLL(path), re.search(r" T (_ZN3dmk\d+launch_girth\w*)", names).group(1))


def girth(g):
    best = GIRTH_MAX
    for v in range(g.n):
        dist, parent, queue = {v: 0}, {v: -1}, [v]
        for u in queue:
            if 2 * dist[u] + 1 >= best:
                break
            for w in map(int, g.col_idx[g.row_ptr[u]:g.row_ptr[u + 1]]):
                if w == parent[u]:
                    continue
                if w in dist:
                    best = min(best, dist[u] + dist[w] + 1)
                else:
                    dist[w], parent[w] = dist[u] + 1, u
                    queue.append(w)
    return best


def edges(n, e):
    return I.from_edges(n, sorted({tuple(sorted(x)) for x in e}))


GRAPHS = {
    "one": (I.from_edges(1, []), True), "edge": (I.path(2), True), "path": (I.path(300), True),
    "strip": (edges(40, [(i, i + 1) for i in range(39)] + [(i, i + 2) for i in range(38)]), True),
    "k33": (edges(6, [(i, 3 + j) for i in range(3) for j in range(3)]), True),
    "petersen": (edges(10, [(i, (i + 1) % 5) for i in range(5)] + [(5 + i, 5 + (i + 2) % 5) for i in range(5)] +
                       [(i, 5 + i) for i in range(5)]), True),
    "grid": (I.grid(9, 7), True), "heavyhex": (I.heavy_hex(5, 7), True), "heavyhex large": (I.heavy_hex(27, 28), True),
    "k40": (I.complete(40), True),  # levels of more than a warp
    "star and ring": (edges(220, [(0, i) for i in range(1, 90)] + [(i, i + 1) for i in range(100, 219)] + [(100, 219), (0, 100)]), False),
    "hub": (edges(200, [(0, i) for i in range(1, 200)]), False),  # more neighbours than the list holds
    "rr3": (I.random_regular3(64, 3), True), "rr3 large": (I.random_regular3(4096, 5), True),
    **{f"ring{n}": (I.cycle(n), True) for n in (3, 4, 5, 12, 13, 30, 31, 32, 33, 95, 200)},
}


@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_girth(launch, name):
    torch = pytest.importorskip("torch")
    g, exact = GRAPHS[name]
    rp = torch.tensor(np.asarray(g.row_ptr, dtype=np.int32), device="cuda")
    ci = torch.tensor(np.asarray(g.col_idx, dtype=np.int32), device="cuda") if len(g.col_idx) else torch.zeros(1, dtype=torch.int32, device="cuda")
    out = torch.full((1,), GIRTH_MAX, dtype=torch.int32, device="cuda")
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    deg = np.diff(g.row_ptr)
    adj4 = torch.zeros((g.n, 4), dtype=torch.int16, device="cuda") if deg.max(initial=0) <= 4 else None
    for lists in (adj4, None):
        assert launch(ctypes.c_void_p(rp.data_ptr()), ctypes.c_void_p(ci.data_ptr()), g.n, ctypes.c_void_p(out.data_ptr()),
                      ctypes.c_void_p(lists.data_ptr() if lists is not None else None), stream) == 0
        got = int(out.item())
        assert got == girth(g) if exact else got <= girth(g)
        out.fill_(GIRTH_MAX)
    if adj4 is not None:
        want = np.full((g.n, 4), -1, dtype=np.int16)
        for v in range(g.n):
            want[v, :deg[v]] = g.col_idx[g.row_ptr[v]:g.row_ptr[v + 1]]
        assert np.array_equal(adj4.cpu().numpy(), want)

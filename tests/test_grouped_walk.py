"""The grouped walk's stack, and what the bounds-checked build does with nodes that are out of
place.  On the CPU a model of the walk's rule shows that trees of the BVH's greatest depth
keep within the stack; on the GPU the checked walk itself stages every triangle of such a
tree once, and over a corrupt list of nodes records the fault, stays within its buffers
and ends."""
import ctypes as ct
import functools
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
THREADS = 128
DEPTH = 62                      # 30 bits of Morton code and the index's
SIZES = [(64, 512, 1), (128, 1024, 0)]     # triangles a pass, stack entries


def full(depth):
    return None if depth == 0 else (full(depth - 1), full(depth - 1))


def comb(depth, side, tail=None):
    t = tail
    for _ in range(depth):
        t = (None, t) if side else (t, None)
    return t


def ragged(rng, depth):
    """A tree whose leaves lie at any depth up to `depth`."""
    if depth == 0 or rng.random() < 0.25:
        return None
    if depth > 8:
        return (ragged(rng, depth - 1), None) if rng.random() < 0.5 else (None, ragged(rng, depth - 1))
    return (ragged(rng, depth - 1), ragged(rng, depth - 1))


def bushy(depth, bush, every=1):
    """`bush` levels of a full tree; one leaf in `every` is a comb down to `depth`, in turn on either side."""
    combs = [comb(depth - bush, 0), comb(depth - bush, 1)]
    level = [combs[i // every % 2] if i % every == 0 else None for i in range(1 << bush)]
    while len(level) > 1:
        level = [(level[i], level[i + 1]) for i in range(0, len(level), 2)]
    return level[0]


def nodes_of(tree):
    """The depth-first node list: float32 [n, 8], every box over the whole group."""
    esc, tri, todo, T = [], [], [(tree, None)], 0
    while todo:
        t, close = todo.pop()
        if close is not None:
            esc[close] = len(esc)
            continue
        i = len(esc)
        esc.append(-1)
        tri.append(-1 if t is not None else T)
        todo.append((None, i))
        if t is None:
            T += 1
            esc[i] = i + 1
            todo.pop()
        else:
            todo += [(t[1], None), (t[0], None)]
    n = len(esc)
    out = np.zeros((n, 8), np.float32)
    out[:, 0:2], out[:, 2], out[:, 4:6], out[:, 6] = -500.0, 0.0, 500.0, 10.0
    out[:, 3] = np.array(esc, np.int32).view(np.float32)
    out[:, 7] = np.array(tri, np.int32).view(np.float32)
    return out, T


@functools.lru_cache(maxsize=1)
def trees():
    rng = np.random.default_rng(5)
    t = {"full": full(12), "left comb": comb(DEPTH, 0), "right comb": comb(DEPTH, 1), "one leaf": None,
         "bush": bushy(DEPTH, 9), "wide bush": bushy(DEPTH, 15, 4), "late bush": comb(DEPTH - 10, 1, full(10))}
    for i in range(4):
        t[f"ragged {i}"] = (bushy(40, 6 + i % 3), ragged(rng, DEPTH - 1))
    return t


def model(nodes, chunk, stack):
    """(most entries on the stack, nodes visited, leaves staged) by the walk's rule."""
    esc, tri = nodes[:, 3].view(np.int32), nodes[:, 7].view(np.int32)
    st, leaves, staged, most, visits = [0], 0, 0, 1, 0
    while True:
        while st and leaves < chunk:
            take = min(THREADS, len(st), max(1, stack - 96 - len(st)))
            popped = [st.pop() for _ in range(take)]
            visits += take
            for i in popped:
                if tri[i] >= 0:
                    leaves += 1
                else:
                    st += [int(esc[i + 1]), i + 1]
            most = max(most, len(st))
        if not leaves:
            return most, visits, staged
        n = min(leaves, chunk)
        staged += n
        leaves -= n


@pytest.mark.parametrize("chunk,stack,small", SIZES)
def test_deepest_trees_keep_within_the_stack(chunk, stack, small):
    brought = 0
    for name, t in trees().items():
        nodes, T = nodes_of(t)
        most, visits, staged = model(nodes, chunk, stack)
        assert most <= stack and visits == len(nodes) and staged == T, name
        brought = max(brought, most)
    assert brought > stack - 96          # waves have ended, and a comb went on from there


def test_a_deeper_tree_would_not():
    """What the bound rests on: combs of 288 levels bring the same walk past 512 entries."""
    nodes, _ = nodes_of(bushy(300, 12, 4))
    assert model(nodes, 64, 512)[0] > 512


# ------------------------------------------------------------------------------- on the GPU
@pytest.fixture(scope="module")
def walk(cuda_lib, tmp_path_factory):
    from paper_1907_04435_gb300 import build as b
    so = str(tmp_path_factory.mktemp("walk") / "grouped_walk.so")
    cmd = [b.nvcc(), *b.ARCH, *b.NVCC_FLAGS, "-DSA_CHECKED", "-shared", "-o", so, os.path.join(HERE, "grouped_walk.cu")]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    L = ct.CDLL(so)
    P = ct.c_void_p
    L.run_walk.argtypes = [P, ct.c_int, ct.c_int, ct.c_int, P, P, P]

    def run(nodes, T, small):
        staged, visits, word = np.zeros(max(T, 1), np.uint32), np.zeros(1, np.uint64), np.zeros(3, np.uint64)
        nodes = np.ascontiguousarray(nodes)
        e = L.run_walk(nodes.ctypes.data, len(nodes), max(T, 1), small, staged.ctypes.data, visits.ctypes.data, word.ctypes.data)
        assert e == 0, e
        return staged, int(visits[0]), [int(x) for x in word.view(np.int64)]
    return run


@pytest.mark.gpu
@pytest.mark.parametrize("chunk,stack,small", SIZES)
def test_every_triangle_is_staged_once(walk, chunk, stack, small):
    for name, t in trees().items():
        nodes, T = nodes_of(t)
        staged, visits, word = walk(nodes, T, small)
        assert word[0] == 0 and visits == len(nodes) and (staged == 1).all(), (name, word, visits)


def corrupt(rng, nodes, T, how):
    """`nodes` with one link or triangle out of place."""
    out = nodes.copy()
    esc, tri = out[:, 3].view(np.int32).copy(), out[:, 7].view(np.int32).copy()
    n = len(out)
    inner = np.nonzero(tri < 0)[0]
    i = int(rng.choice(inner))
    if how == "beyond":                      # the right child lies past the list
        esc[i + 1] = n + int(rng.integers(0, 1000))
    elif how == "end":                       # ... at its end, where an escape link may point
        esc[i + 1] = n
    elif how == "back":                      # ... before its parent
        esc[i + 1] = int(rng.integers(-5, i + 2))
    elif how == "overlap":                   # every subtree overlaps its parent's neighbours
        esc[:] = np.minimum(np.arange(n) + 1 + (tri < 0), n)
    elif how == "last":                      # the list's last node has no children
        tri[n - 1] = -1
    else:                                    # a leaf's triangle
        tri[int(rng.choice(np.nonzero(tri >= 0)[0]))] = T + 7
    out[:, 3], out[:, 7] = esc.view(np.float32), tri.view(np.float32)
    return out


@pytest.mark.gpu
@pytest.mark.parametrize("how", ["beyond", "end", "back", "overlap", "last", "leaf"])
@pytest.mark.parametrize("chunk,stack,small", SIZES)
def test_nodes_out_of_place_are_reported(walk, how, chunk, stack, small):
    rng = np.random.default_rng(17)
    for name in ("full", "bush", "left comb"):
        nodes, T = nodes_of(trees()[name])
        staged, visits, word = walk(corrupt(rng, nodes, T, how), T, small)
        assert word[0] != 0 and visits <= len(nodes), (name, word, visits)


@pytest.mark.gpu
def test_a_tree_too_deep_for_the_stack_is_reported(walk):
    nodes, T = nodes_of(bushy(300, 12, 4))
    staged, visits, word = walk(nodes, T, 1)
    assert word[0] != 0 and word[2] == 512 and visits <= len(nodes) and staged.max() == 1, word

"""The fault guards of the pooled walks (pt_pool.cuh).  The scene builder refuses trees as deep as the traversal stack
and never makes a cycle, so these trees are built by hand and walked by a kernel of their own (pool_guards.cu): a comb
as deep as the stack holds, one deeper than that, and a node that is its own child.  The walk must keep to its stack
and must end, and must say so in the status word (1: traversal limit)."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
STACK, MISS, LEAF = 64, 0xFFFFFFFF, 0x80000000
BIG = 1e6


@pytest.fixture(scope="module")
def walk(tmp_path_factory):
    import torch

    from paper_2605_27323_gb300 import build as B
    assert torch.cuda.is_available()
    so = str(tmp_path_factory.mktemp("guards") / "pool_guards.so")
    subprocess.run([os.path.join(B._cuda_home(), "bin", "nvcc"), B.ARCH, "-O3", "-std=c++17", "-fmad=false", "-shared",
                    "-Xcompiler", "-fPIC", "-I" + B.INCLUDE, "-I" + B.CSRC, os.path.join(HERE, "pool_guards.cu"), "-o", so],
                   check=True)
    lib = C.CDLL(so)

    def run(nodes, tris, n, share=False, tlas=None, inst=None):
        t = np.zeros(2 * n, np.float32)
        tri = np.zeros(2 * n, np.uint32)
        st = C.c_uint32()
        p = lambda a: None if a is None else a.ctypes.data_as(C.c_void_p)
        e = lib.pool_guards_run(p(nodes), C.c_uint32(len(nodes)), p(tris), C.c_uint32(len(tris)), p(tlas),
                                C.c_uint32(0 if tlas is None else len(tlas)), p(inst),
                                C.c_uint32(0 if inst is None else len(inst)), C.c_uint32(n), int(share), p(t), p(tri),
                                C.byref(st))
        assert e == 0
        return t.reshape(n, 2), tri.reshape(n, 2), st.value

    return run


def _node(ref0, ref1, box0=(-BIG, BIG), box1=(-BIG, BIG)):
    f = np.zeros(16, np.float32)
    f[0:2], f[2:4] = box0[0], box0[1]
    f[4:6], f[6:8] = box1[0], box1[1]
    f[8], f[9], f[10], f[11] = box0[0], box0[1], box1[0], box1[1]
    f[12:14] = np.array([ref0, ref1], np.uint32).view(np.float32)
    return f


def _triangles(ts):
    """Triangles across the x axis at the distances ts, ids in order."""
    r = np.zeros((len(ts), 12), np.float32)
    for k, t in enumerate(ts):
        r[k, 0:3] = (t, -1, -1)
        r[k, 3] = np.array([k], np.uint32).view(np.float32)[0]
        r[k, 4:7] = (0, 4, 0)
        r[k, 8:11] = (0, 0, 4)
    return r


def _comb(depth):
    """Node i defers leaf i and goes on to node i + 1; the last one's other child is leaf `depth`.  The deferred leaves
    lie farther away the later they are deferred, the last leaf farthest."""
    nodes = [_node(i + 1 if i + 1 < depth else LEAF | depth << 3, LEAF | i << 3) for i in range(depth)]
    return np.stack(nodes), _triangles([1000.0 + 10 * i for i in range(depth + 1)])


def _right(t, tri):
    # the nearest leaf is the first one deferred; the any-hit rays are occluded
    return bool(np.all(t[:, 0] == 1000.0) and np.all(tri[:, 0] == 0) and np.all(t[:, 1] < 0))


@pytest.mark.parametrize("share", [False, True])
@pytest.mark.parametrize("n", [1, 3, 4, 16, 50])
@pytest.mark.parametrize("depth", [STACK - 1, STACK, STACK + 1, 2 * STACK, 2 * STACK + 1, 2 * STACK + 2, 500])
def test_a_tree_deeper_than_the_stack_is_reported(walk, depth, n, share):
    """One entry is deferred at each node.  Up to the stack's depth the walk must be right; beyond it, right or
    reported, and reported once it is deeper than the stack and the steps of two phases."""
    t, tri, st = walk(*_comb(depth), n, share)
    assert st in (0, 1)
    if depth <= STACK:
        assert st == 0
    if st == 0:
        assert _right(t, tri)
    if depth > 3 * STACK:
        assert st == 1


def test_two_levels_deeper_than_the_stack_are_reported(walk):
    """The walk of a two-level scene keeps both trees' entries on one stack of twice the size."""
    tlas = np.stack([_node(i + 1 if i + 1 < 40 else LEAF, LEAF) for i in range(40)])
    inst = np.zeros((1, 32), np.float32)
    inst[0, 0], inst[0, 5], inst[0, 10] = 1, 1, 1            # world to object: identity; mesh root 0, first id 0
    for depth, n in ((88, 1), (88, 16), (89, 16), (153, 16), (400, 1), (400, 16)):
        t, tri, st = walk(*_comb(depth), n, tlas=tlas, inst=inst)
        assert st in (0, 1)
        assert st == 1 if depth > 300 else (st == 0 or depth > 88)
        if st == 0:
            assert _right(t, tri)


@pytest.mark.parametrize("n,share", [(16, False), (1, False), (1, True)])
def test_a_cycle_ends_and_is_reported(walk, n, share):
    """Node 0 is its own child.  16 + 16 lanes repeat node steps, one lane turns, one lane in the shared end."""
    nodes = np.stack([_node(0, LEAF, box1=(-BIG, -BIG / 2))])
    t, tri, st = walk(nodes, _triangles([1000.0]), n, share)
    assert st == 1 and np.all(np.isinf(t[:, 0])) and np.all(tri[:, 0] == MISS) and np.all(t[:, 1] == 5000.0)

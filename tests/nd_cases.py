"""Test problems with a given size for every node of an ND tree (also none)."""
import numpy as np

from tests import helpers as H


def _tree(depth):
    """Per node of the postorder tree: its height and its first descendant."""
    height, first = [], []

    def walk(h):
        at = len(height)
        if h > 0:
            walk(h - 1)
            walk(h - 1)
        height.append(h)
        first.append(at)

    walk(depth)
    return height, first


def nd_problem(seed, sizes, density=0.5, chain=False, before=(), after=()):
    """One ND block with nodes of ``sizes`` rows (postorder), between BTF blocks of the
    sizes ``before`` and ``after``, each coupled to a later block.  A node's own block is
    random at ``density`` (leaves tridiagonal with ``chain``), and tied to every node
    below it (chains: at their first rows)."""
    rng = np.random.default_rng(seed)
    depth = (len(sizes) + 1).bit_length() - 2
    height, first = _tree(depth)
    blocks = list(before) + [int(np.sum(sizes))] + list(after)
    bptr = np.concatenate([[0], np.cumsum(blocks)]).astype(np.int32)
    n = int(bptr[-1])
    ptr = (bptr[len(before)] + np.concatenate([[0], np.cumsum(sizes)])).astype(np.int32)
    M = np.zeros((n, n))

    def fill(r0, r1, c0, c1, p):
        v = rng.uniform(-1, 1, (r1 - r0, c1 - c0)) * (rng.random((r1 - r0, c1 - c0)) < p)
        M[r0:r1, c0:c1] = v

    for t in range(len(sizes)):
        lo, hi = int(ptr[t]), int(ptr[t + 1])
        if chain and height[t] == 0:
            for k in range(lo, hi - 1):
                M[k, k + 1], M[k + 1, k] = rng.uniform(-1, 1, 2)
        else:
            fill(lo, hi, lo, hi, density)
        for s in range(first[t], t):
            a, z = int(ptr[s]), int(ptr[s + 1])
            if chain and height[s] == 0:
                z = min(z, a + 2)
            fill(lo, hi, a, z, max(density, 0.5))
            fill(a, z, lo, hi, max(density, 0.5))
    for d in range(len(blocks)):
        lo, hi = int(bptr[d]), int(bptr[d + 1])
        if d != len(before):
            fill(lo, hi, lo, hi, 1.0)
        if d + 1 < len(blocks):
            M[rng.integers(lo, hi), rng.integers(hi, n)] = rng.uniform(0.5, 1.0)
    M[np.arange(n), np.arange(n)] = rng.uniform(0.5, 1.0, n)
    return H.make_problem(M, block_ptr=bptr, nd_block=len(before), nd_leaves=1 << depth, nd_node_ptr=ptr,
                          scramble_seed=seed)


#: Node sizes with separators whose descendants are all empty.
EMPTY = {
    "first_pair": ([0, 0, 2, 1, 1, 1, 2], {}),                        # its first row is the block's
    "second_pair": ([3, 4, 2, 0, 0, 5, 6], {}),
    "half_tree": ([0, 0, 0, 0, 0, 0, 7, 9, 8, 3, 5, 0, 4, 6, 10], {}),
    "no_leaf": ([0, 0, 5, 0, 0, 40, 6], {}),
    "root_alone": ([0, 0, 0, 0, 0, 0, 30], {}),
    "beside_blocks": ([0, 0, 20, 17, 30, 9, 12], dict(before=[1, 2, 1], after=[2, 1, 30])),
    "dense": ([0, 0, 60, 50, 40, 30, 45], dict(density=1.0)),        # stored patterns first
}

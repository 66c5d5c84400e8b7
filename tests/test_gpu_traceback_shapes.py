"""mcm_traceback on split tables of chosen trees: combs, zigzags, balanced and
random ones, at the sizes where the kernel changes its way of following them."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _split(shape, r, i, j, depth):
    if shape == "left":       # (i, j-1) and one matrix: a left comb
        return j - 1
    if shape == "right":
        return i
    if shape == "zigzag":
        return i if depth % 2 else j - 1
    if shape == "balanced":
        return (i + j) // 2
    if shape == "steps":      # a right spine with 40-matrix subtrees hanging off it
        return min(j - 1, i + 39)
    return int(r.randint(i, j))


def _tree(shape, n, seed):
    r = np.random.RandomState(seed)
    s = np.full((n, n), -1, np.int16)
    order, stack = [], [(0, n - 1, 0)]
    while stack:  # root, right, left: the reverse of post-order
        i, j, d = stack.pop()
        if i < j:
            k = _split(shape, r, i, j, d)
            s[i, j] = k
            order.append((i, k, j))
            stack += [(i, k, d + 1), (k + 1, j, d + 1)]
    return s, np.array(order[::-1], np.int32).reshape(-1, 3)


@pytest.mark.parametrize("shape", ["left", "right", "zigzag", "balanced", "steps", "random"])
@pytest.mark.parametrize("n", [2, 31, 32, 33, 64, 257, 290, 1024, 1025, 2100, 4500])
def test_chosen_trees(shape, n):
    import torch
    import paper_2008_01938_gb300 as dp
    s, ref = _tree(shape, n, n)
    got = dp.mcm_traceback(torch.from_numpy(s).cuda())
    dp.sync_status()
    assert np.array_equal(got.cpu().numpy(), ref)


@pytest.mark.parametrize("n", [512, 513, 4500])
def test_captured_in_a_graph(n):
    """The second launch starts before the first has ended: replayed from a
    graph on other trees, back to back."""
    import torch
    import paper_2008_01938_gb300 as dp
    trees = [_tree(shape, n, n) for shape in ("balanced", "steps", "left", "random")]
    s = torch.from_numpy(trees[0][0]).cuda()
    steps = torch.empty((n - 1, 3), dtype=torch.int32, device="cuda")
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        dp.mcm_traceback(s, steps)  # kernels loaded before the capture
        stream.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            dp.mcm_traceback(s, steps)
        got = []
        for tree, _ in trees:
            s.copy_(torch.from_numpy(tree).cuda())
            steps.fill_(-1)
            g.replay()
            got.append(steps.clone())
        stream.synchronize()
    dp.sync_status()
    for x, (_, ref) in zip(got, trees):
        assert np.array_equal(x.cpu().numpy(), ref)


def _bad(where, i, j):
    return {"below": i - 1, "last": j, "above": j + 1}[where]


# the nodes by their number of matrices, from the root down: the first ones (a
# path begins after three lopsided ones), one in the middle, the smallest of
# more than 32 matrices, the largest of at most 32, the smallest of all
PLACES = ["root", 1, 2, 3, 4, 5, "middle", "last large", "first small", "leaf"]


@pytest.mark.parametrize("shape", ["left", "right", "zigzag", "balanced", "steps", "random"])
@pytest.mark.parametrize("n", [20, 600, 1300, 3000])
def test_a_split_outside_its_subtree_is_reported(shape, n):
    """One split of the tree set to i - 1, j or j + 1 at node (i, j): followed
    by a thread, a warp's and the block's path (at its start, inside it and at
    its end) and in a subtree expanded whole."""
    import torch
    import paper_2008_01938_gb300 as dp
    s, ref = _tree(shape, n, n)
    by_size = sorted(((int(j) - int(i) + 1, int(i), int(j)) for i, _, j in ref), reverse=True)
    large = [x for x in by_size if x[0] > 32]
    at = {"root": 0, "middle": len(large) // 2, "last large": len(large) - 1, "first small": len(large),
          "leaf": len(by_size) - 1}
    good = torch.from_numpy(s).cuda()
    for rank in sorted({min(max(at.get(p, p), 0), len(by_size) - 1) for p in PLACES}):
        _, i, j = by_size[rank]
        for where in ("below", "last", "above"):
            t = good.clone()
            t[i, j] = _bad(where, i, j)
            dp.mcm_traceback(t)
            with pytest.raises(dp.native.DpError) as e:
                dp.sync_status()
            assert e.value.code == dp.native.DP_EINVAL, (i, j, where)
    got = dp.mcm_traceback(good)
    dp.sync_status()
    assert np.array_equal(got.cpu().numpy(), ref)

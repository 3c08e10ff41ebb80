"""The batched window kernels on the float64 matrix instruction: edges of tiles, remainders of summation steps, slices beyond
shared memory, one and several tasks per slice, against the oracle at the float64 path's tolerances."""
import contextlib
import os
import sys

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
for p in (HERE, os.path.dirname(HERE)):
    if p not in sys.path:
        sys.path.insert(0, p)

from parity import check_workload, compare, run_gpu           # noqa: E402
from test_gpu_block import _workload                           # noqa: E402
from test_gpu_parity import family_forced                      # noqa: E402

pytestmark = pytest.mark.gpu


@contextlib.contextmanager
def workspace(what):
    """The library's testing aid BI_TEST_WORKSPACE, read when a handle is made."""
    os.environ["BI_TEST_WORKSPACE"] = what
    try:
        yield
    finally:
        del os.environ["BI_TEST_WORKSPACE"]

CASES = {   # n, dep, N, T
    "smallest": ([2, 2, 2], [[0, 1, 2]], 1024, 2),
    "odd_rank3": ([5, 3, 7], [[0, 1, 2], [1, 2]], 300, 7),                       # rows and columns of no whole tile
    "rank4": ([7, 5, 3, 6], [[0, 1, 2, 3], [0, 1, 3], [1, 3]], 260, 9),
    "exact_tiles": ([8, 16, 8], [[0, 1, 2], [1]], 130, 16),
    "several_chunks": ([9, 13, 11, 10], [[0, 1, 2, 3]], 64, 32),                 # more results than a warp accumulates at once
    "chunks_across_tiles": ([8, 9, 7, 10], [[0, 1, 2, 3], [1, 2, 3]], 90, 25),    # chunks that start within a tile, on either side
    "beyond_shared_memory": ([32, 31, 30], [[0, 1, 2]], 86, 24),                 # read through L1
    "wide_pairs": ([17, 32, 25], [[0, 1], [1, 2], [2]], 100, 21),
    "one_state": ([1, 6, 9], [[0, 1, 2], [0, 2]], 210, 10),
    "one_step": ([6, 5, 4], [[0, 1, 2], [1, 2], [0]], 2100, 1),                  # no transitions
    "long_tasks": ([3, 4, 6], [[0, 1, 2], [0, 1]], 2500, 20),                    # several trips of a task's warps
    "eight_warps_split": ([10, 10, 8, 6], [[0, 1], [0, 1, 2, 3]], 450, 20),      # up to 9472 units: V and W by different warps
    "eight_warps": ([10, 10, 8, 6], [[0, 1], [0, 1, 2, 3]], 620, 20),
    "many_planes": ([4, 5, 3], [[0, 1, 2], [0, 1], [1, 2], [0, 2]] * 3, 150, 14),
}


@pytest.mark.parametrize("algo", ["vmp", "mmp"])
@pytest.mark.parametrize("case", sorted(CASES))
def test_shapes(case, algo):
    n, dep, N, T = CASES[case]
    with family_forced("batch"):
        res = check_workload(_workload(300 + len(case), n, dep, N=N, T=T, K=5), algo, agents=range(0, N, max(1, N // 9)))
    assert res["family"] == f"batch_{algo}_f64", res


@pytest.mark.parametrize("bdep", [[[0, 1], [1], [2, 0]], [[1, 2, 0], [2], [0, 1]]])
def test_transitions(bdep):
    """One, two and three parents: edges on the pair kernel beside edges on the slice kernel, damped."""
    import oracle
    import torch
    import paper_2607_17855_b200 as bi
    w = _workload(330, [5, 6, 9], [[0, 1], [2]], N=190, T=11, K=6, bdep=bdep)
    with family_forced("batch"):
        md = bi.model_from_workload(w)
    md.set_damping(0.7)
    q = md.run("vmp", torch.from_numpy(w.obs).cuda(), torch.from_numpy(w.act).cuda(), w.K).cpu().numpy()
    assert md.last_family == "batch_vmp_f64" and md.status() == 0
    md.close()
    sel = list(range(0, w.N, 21))
    assert np.abs(q[sel] - oracle.run_workload(w.take_agents(sel), "vmp", damping=0.7)[0]).max() <= 1e-5


@pytest.mark.parametrize("n, bdep", [
    ([1, 5, 6], [[0, 1], [1, 0], [2]]),                     # a one-state factor as the slow column; as the only one
    ([6, 1, 9], [[0, 1, 2], [0, 1, 2], [2, 1]]),            # ... as the middle parent, as the child
    ([5, 1, 9], [[1, 2], [1], [1, 0]]),                     # ... as its own only parent
    ([1, 6, 9, 4], [[1, 2, 3], [2, 0, 3], [0, 2], [3]]),    # ... as the slow axis of either side of four
])
def test_one_state_factors_in_transitions(n, bdep):
    """Every message that the update reads is written: the workspace holds NaN before each call.  Also on a
    second call with fewer units, whose planes lie elsewhere."""
    import oracle
    import paper_2607_17855_b200 as bi
    dep = [[0, 1], list(range(len(n)))]
    w = _workload(350, n, dep, N=300, T=9, K=5, bdep=bdep)
    first = _workload(350, n, dep, N=270, T=13, K=5, bdep=bdep)
    with family_forced("batch"), workspace("nan"):
        md = bi.model_from_workload(w)
    for c in (first, w):
        *out, _ = run_gpu(c, "vmp", model=md)
        assert md.last_family == "batch_vmp_f64"
        compare(c, *out, *oracle.run_workload(c, "vmp"))
    md.close()


@pytest.mark.parametrize("damping", [1.0, 0.6])
@pytest.mark.parametrize("algo", ["vmp", "mmp"])
def test_call_forms(algo, damping):
    """Warm-started and continued calls, plain and damped, one after the other on one handle and of fewer and fewer units; every
    agent, with NaN in the workspace before each."""
    import oracle
    import torch
    import paper_2607_17855_b200 as bi
    n, T = [5, 1, 7, 4], 9
    w = _workload(380, n, [[0, 1, 2], [2, 3], [0, 2, 3], [0]], N=400, T=T, K=5)
    rng = np.random.default_rng(381)
    simplex = lambda *size: np.concatenate([rng.dirichlet(np.full(k, 1.5), size=size) for k in n], axis=-1).astype(np.float32)
    q_prev, q_init = simplex(w.N), simplex(w.N, T)
    act_prev = np.stack([rng.integers(0, int(u), size=w.N) for u in w.U], axis=1).astype(np.int32)
    cuda = lambda x: torch.from_numpy(x).cuda()
    with family_forced("batch"), workspace("nan"):
        md = bi.model_from_workload(w)
    md.set_damping(damping)
    warm = md.bi_vmp_warm if algo == "vmp" else md.bi_mmp_warm
    for N, call in ((400, "plain"), (350, "warm"), (300, "from"), (250, "from, warm")):
        obs, act, kw = cuda(w.obs[:N]), cuda(w.act[:N]), {}
        if "from" in call:
            kw = dict(q_prev=q_prev[:N].astype(np.float64), act_prev=act_prev[:N])
        if "warm" in call:
            kw["q_init"] = q_init[:N].astype(np.float64)
        if "from" in call:
            q = md.run_from(algo, obs, act, cuda(q_prev[:N]), cuda(act_prev[:N]), w.K, q_init=cuda(q_init[:N]) if "warm" in call else None)
        else:
            q = warm(obs, act, cuda(q_init[:N]), w.K) if call == "warm" else md.run(algo, obs, act, w.K)
        assert md.last_family == f"batch_{algo}_f64" and md.status() == 0
        ref = oracle.run(algo, w.n, w.m, w.dep, w.U, w.G, w.A, w.B, w.D, w.obs[:N], w.act[:N], w.K, damping=damping, **kw)[0]
        assert np.abs(q.cpu().numpy() - ref).max() <= 1e-5, call
    md.close()


FALLBACK = {   # n, dep, bdep, N, T, and who serves the call without a workspace
    "pairs": ([25, 27, 6, 28, 17], [[0, 3], [2], [4], [3], [0, 1]], None, 256, 10, "pair"),
    "blocks": ([14, 14, 2, 12], [[0, 1, 2, 3]], None, 300, 12, "block"),
    "several_parents": ([10, 10, 8], [[0, 1], [1, 2]], [[0, 1], [1, 2], [2, 0]], 200, 16, "block"),
    "few_units": ([28, 27, 26], [[0, 1, 2], [0]], None, 20, 16, "warp"),
}


@pytest.mark.parametrize("case", sorted(FALLBACK))
def test_without_a_workspace(case):
    """A call whose workspace cannot be had runs on the kernels that need none."""
    n, dep, bdep, N, T, family = FALLBACK[case]
    w = _workload(360, n, dep, N=N, T=T, K=3, bdep=bdep)
    few = range(0, N, max(1, N // 8))
    assert check_workload(w, "vmp", agents=few)["family"] == "batch_vmp_f64"
    with workspace("none"):
        assert check_workload(w, "vmp", agents=few)["family"] == f"{family}_vmp_f64"


def test_captured_calls():
    """A graph's calls keep their memory: the first call of a handle, captured, takes kernels without a workspace; one captured
    after a call of its size stays valid when a larger call obtains a larger workspace."""
    import torch
    import paper_2607_17855_b200 as bi
    n, dep, _, N, T, _ = FALLBACK["pairs"]
    w, large = (_workload(370, n, dep, N=k * N, T=T, K=3) for k in (1, 4))
    cuda = lambda x: torch.from_numpy(x).cuda()
    obs, act, big = cuda(w.obs), cuda(w.act), (cuda(large.obs), cuda(large.act), large.K)
    with workspace("none"):   # (and the pair kernel is loaded before the capture)
        plain = bi.model_from_workload(w)
    want = {"pair": plain.run("vmp", obs, act, w.K)}
    other = bi.model_from_workload(w)
    want["batch"] = other.run("vmp", obs, act, w.K)
    for family in ("pair", "batch"):
        md = bi.model_from_workload(w)
        o, q = obs.clone(), torch.zeros_like(want[family])
        if family == "batch":
            md.run("vmp", o, act, w.K, q_out=q)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            md.run("vmp", o, act, w.K, q_out=q)
        assert md.last_family == f"{family}_vmp_f64"
        g.replay()
        assert torch.equal(q, want[family])
        q_big = md.run("vmp", *big)
        assert md.last_family == "batch_vmp_f64"
        o.zero_()
        g.replay()
        assert torch.equal(q, (plain if family == "pair" else other).run("vmp", torch.zeros_like(obs), act, w.K))
        o.copy_(obs)
        g.replay()
        assert torch.equal(q, want[family]) and torch.equal(q_big, md.run("vmp", *big))
        assert md.status() == 0
        del g
        md.close()
    plain.close()
    other.close()


@pytest.mark.parametrize("N, family", [(32, "batch"), (31, "warp")])
def test_few_units_of_a_model_too_large_for_the_block_kernels(N, family):
    res = check_workload(_workload(340, [32, 31, 30], [[0, 1, 2], [0]], N=N, T=8, K=3), "vmp", agents=range(0, N, 5))
    assert res["family"] == f"{family}_vmp_f64", res

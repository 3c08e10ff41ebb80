"""The block kernels (a team of threads per agent and step, every thread a block of the summed slices in
registers) at the sizes where a plan can go wrong: one state more or less than a block, blocks left over for
shared memory, teams of one and of several warps, windows over one CTA and over a cluster, every kind of
prefix (groups of two to four factors), transitions with several parents."""
import numpy as np
import pytest

from biwl import Workload, make_model, sample_streams
from parity import check_workload

pytestmark = pytest.mark.gpu


def _workload(seed, n, dep, N, T, K, bdep=None, G=1):
    rng = np.random.default_rng(seed)
    m = [int(rng.integers(2, 7)) for _ in dep]
    U = [int(rng.integers(1, 4)) for _ in n]
    A, B, D = make_model(rng, n, m, dep, U, G, d_alpha=1.0, bdep=bdep)
    obs, act = sample_streams(rng, n, m, dep, U, G, A, B, D, N, T, bdep=bdep)
    return Workload(name="block", algo="filter", n=np.asarray(n, np.int32), m=np.asarray(m, np.int32), dep=dep,
                    U=np.asarray(U, np.int32), G=G, A=A, B=B, D=D, N=N, T=T, K=K, obs=obs, act=act, bdep=bdep)


FILTER = {
    "below_a_block": ([7, 3, 3], [[0, 1, 2]]),
    "one_block": ([8, 4, 2], [[0, 1, 2]]),
    "a_state_over": ([9, 5, 7], [[0, 1, 2], [1]]),
    "rank4_prefixes": ([2, 9, 3, 13], [[0, 1, 2, 3], [2, 0], [1]]),
    "several_groups": ([17, 8, 25, 6], [[0, 1], [1, 2, 3], [0, 2], [3, 0, 1], [2]]),
    "unobserved_factors": ([5, 1, 32, 7, 4], [[0, 2, 3], [1, 2]]),
    "shared_memory_blocks": ([32, 31, 30], [[0, 1, 2], [2]]),
}


@pytest.mark.parametrize("N", [1, 37])
@pytest.mark.parametrize("case", sorted(FILTER))
def test_filtering(case, N):
    n, dep = FILTER[case]
    res = check_workload(_workload(10 + N, n, dep, N=N, T=4, K=7), "filter")
    assert res["family"] == "block_filter_f64", res


def test_filtering_large_batches_share_a_cta():
    res = check_workload(_workload(3, [5, 4, 3], [[0, 1, 2], [1, 0, 2]], N=3701, T=2, K=3), "filter",
                         agents=range(0, 3701, 97))
    assert res["family"] == "block_filter_f64", res


WINDOW = {   # (n, dep, T): one CTA, idle steps in the last one of a cluster, the longest window, blocks in shared memory
    "one_step": ([9, 5, 7], [[0, 1, 2]], 1),
    "one_cta": ([3, 4, 2, 5], [[0, 1, 2], [1, 3]], 9),
    "ragged_cluster": ([9, 6, 12, 4], [[0, 1], [1, 2, 3], [0, 1, 2]], 13),
    "longest": ([4, 3, 5], [[0, 1, 2], [2, 1]], 64),
    "rank4": ([4, 6, 7, 5], [[0, 1, 2, 3]], 6),
    "shared_memory_blocks": ([18, 29, 11], [[0, 1, 2], [0, 2]], 10),
}


@pytest.mark.parametrize("algo", ["vmp", "mmp"])
@pytest.mark.parametrize("case", sorted(WINDOW))
def test_windows(case, algo):
    n, dep, T = WINDOW[case]
    res = check_workload(_workload(20, n, dep, N=5, T=T, K=6), algo)
    assert res["family"] == f"block_{algo}_f64", res


@pytest.mark.parametrize("algo", ["filter", "vmp", "mmp"])
def test_models_of_their_own(algo):
    res = check_workload(_workload(30, [6, 5, 9], [[0, 1, 2], [2, 1]], N=9, T=7, K=5, G=9), algo)
    assert res["family"] == f"block_{algo}_f64", res


@pytest.mark.parametrize("algo", ["filter", "vmp"])
@pytest.mark.parametrize("bdep", [[[0, 1], [1, 2], [2, 0]], [[2], [0, 1, 2], [1, 2]], [[1, 0, 2], [2, 1], [2]]])
def test_transitions_with_several_parents(bdep, algo):
    res = check_workload(_workload(40, [9, 4, 7], [[0, 1], [1, 2, 0]], N=7, T=6, K=5, bdep=bdep), algo)
    assert res["family"] == f"block_{algo}_f64", res


@pytest.mark.parametrize("n, dep, bdep, T", [
    ([9, 4, 7], [[0, 1], [1, 2, 0]], [[0, 1], [2], [2, 0, 1]], 7),           # any-shape slices, one to three parents
    ([10, 10, 8, 6], [[0, 1], [0, 2, 3]], [[0, 1], [1, 2], [2, 3], [3, 0]], 8),   # unrolled slices beside the transitions
    ([3, 2, 4, 2, 3], [[0], [3]], [[1, 0, 2, 3], [1], [4, 2], [3], [0]], 1),      # no slice to contract, one step
    ([3, 2, 4, 2, 3], [[0], [3]], [[1, 0, 2, 3], [1], [4, 2], [3], [0]], 9),      # four parents, a pure copy of another factor
])
def test_batched_transitions_with_several_parents(n, dep, bdep, T):
    from test_gpu_parity import family_forced
    N = 2100 if T == 1 else 2100 // T + 60
    with family_forced("batch"):
        res = check_workload(_workload(60 + T, n, dep, N=N, T=T, K=5, bdep=bdep), "vmp", agents=range(0, N, 23))
    assert res["family"] == "batch_vmp_f64", res


@pytest.mark.parametrize("algo", ["filter", "vmp", "mmp"])
def test_float32(algo):
    # (dense and few iterations: the tolerance of check_workload's strict=False form is not a numerical one)
    res = check_workload(_workload(50, [9, 5, 7, 6], [[0, 1, 2], [1, 3]], N=21, T=5, K=4), algo, arith="f32", strict=False)
    assert res["family"] == f"block_{algo}_f32", res
    assert res["q_max_err"] < 1e-3, res   # four undamped float32 iterations: 1e-6 of the logits' sums, amplified below 1e3


@pytest.mark.parametrize("bdep", [None, [[0, 1], [1], [2, 3], [3]]], ids=["one_parent", "several_parents"])
def test_filtering_in_blocks_of_steps_on_sparse_models(bdep):
    """bi_filter_continue promises the single call's beliefs bit for bit.  Zeros in A amplify the last bit of a
    belief to its first digit, so the kernel must not depend on how many steps a call has."""
    import torch
    import paper_2607_17855_b200 as bi
    from test_gpu_parity import _blockwise
    n, dep, U = [5, 7, 6, 4], [[0, 1, 2], [2, 3, 1], [3]], [2, 1, 3, 2]
    rng = np.random.default_rng(71)
    m = [9, 11, 5]
    A, B, D = make_model(rng, n, m, dep, U, 1, sparsity=0.7, d_alpha=1.0, bdep=bdep)
    obs, act = sample_streams(rng, n, m, dep, U, 1, A, B, D, 96, 10, bdep=bdep)
    w = Workload(name="sparse", algo="filter", n=np.asarray(n, np.int32), m=np.asarray(m, np.int32), dep=dep,
                 U=np.asarray(U, np.int32), G=1, A=A, B=B, D=D, N=96, T=10, K=16, obs=obs, act=act, bdep=bdep)
    md = bi.model_from_workload(w)
    whole = md.bi_filter(torch.from_numpy(w.obs).cuda(), torch.from_numpy(w.act).cuda(), w.K).cpu().numpy()
    for cuts in (list(range(11)), [0, 2, 4, 6, 8, 10], [0, 5, 6, 8, 10]):
        q, _ = _blockwise(md, w, cuts, w.K)
        assert np.array_equal(q, whole), (cuts, np.abs(q - whole).max())
    assert md.status() == 0
    md.close()


@pytest.mark.parametrize("case", ["tile", "rank5", "block", "pair"])
def test_the_model_is_packed_when_the_call_returns(case):
    """The caller may reuse A, B and D (on any stream) once bi_model_create has returned: whatever the kind of
    model, the packing is then done, also behind work that the stream had queued before."""
    import torch
    import paper_2607_17855_b200 as bi
    n, dep = {"tile": ([8, 8, 6], [[0, 1, 2]]), "rank5": ([3, 2, 4, 2, 3], [[0, 1, 2, 3, 4]]),
              "block": ([5, 4, 7], [[0, 1, 2]]), "pair": ([4, 3], [[0, 1]])}[case]
    w = _workload(80, n, dep, N=3, T=2, K=2)
    arrays = [[torch.from_numpy(x).cuda() for x in part] for part in (w.A, w.B, w.D)]
    x = torch.randn(4096, 4096, device="cuda")
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        for _ in range(40):   # some milliseconds each
            x = torch.mm(x, x).clamp_(-1, 1)
        md = bi.Model(w.n, w.m, w.dep, w.U, w.G, *arrays)
        assert s.query()
    md.close()


@pytest.mark.parametrize("K", [1, 2])
def test_improbable_states_under_many_future_messages(K):
    """A factor whose thirteen impossible outcomes put every state at the floor, ln 1e-16 each, and whose state is
    read by eight transitions that the uniform next beliefs contradict (K = 1: 15/16 of ln 1e-16 each): logits near
    -740, where exp underflows, so the softmax must be relative to the largest of them."""
    M, n, F = 14, [3] + [16] * 7, 8
    rng = np.random.default_rng(90)
    A = []
    for i in range(M):
        a = np.zeros((1, 4, 3), np.float32)   # (outcome 3 has probability zero in every state)
        a[0, :3] = rng.dirichlet(np.ones(3), 3).T
        if i == 0:
            a[0, 3], a[0, :3] = 0.25, 0.75 * a[0, :3]
        A.append(a)
    B, D = [], []
    for f, nf in enumerate(n):
        b = np.zeros((1, nf, 3, 2), np.float32)
        if f == 0:
            b[:] = 1.0 / 3.0
        else:
            b[:, 0] = 1.0
        B.append(b)
        D.append(np.full((1, nf), 1.0 / nf, np.float32))
    N, T = 4, 4
    w = Workload(name="improbable", algo="vmp", n=np.asarray(n, np.int32), m=np.full(M, 4, np.int32), dep=[[0]] * M,
                 U=np.full(F, 2, np.int32), G=1, A=A, B=B, D=D, N=N, T=T, K=K, obs=np.full((N, T, M), 3, np.int32),
                 act=np.zeros((N, T - 1, F), np.int32), bdep=[[0]] * F)
    res = check_workload(w, "vmp")
    assert res["family"] == "block_vmp_f64", res


@pytest.mark.parametrize("case", ["every_slice_unrolled", "too_large_for_blocks"])
def test_observation_vectors_form_every_slice_once(case):
    """Which kernels will read the slices is known before they are formed: one launch per group, one for the step
    indices, and the inference call's own (batched windows: the two at the start and two per iteration)."""
    import torch
    import oracle
    import paper_2607_17855_b200 as bi
    from test_gpu_parity import _soft_vectors
    if case == "every_slice_unrolled":
        n, dep, N, T, step = [10, 10, 8, 6], [[0, 1], [1, 2], [0, 2, 3]], 260, 16, 20
    else:
        n, dep, N, T, step = [32, 31, 30], [[0, 1, 2], [2]], 3, 4, 1
    w = _workload(100, n, dep, N=N, T=T, K=3)
    md = bi.model_from_workload(w)
    soft = _soft_vectors(w, 7)
    q = md.run_soft("vmp", torch.from_numpy(soft).cuda(), torch.from_numpy(w.act).cuda(), w.K).cpu().numpy()
    own = md.launch_count - (len(dep) + 1)
    sel = list(range(0, N, step))
    sub = w.take_agents(sel)
    ref = oracle.run("vmp", sub.n, sub.m, sub.dep, sub.U, sub.G, sub.A, sub.B, sub.D, None, sub.act, sub.K, obs_soft=soft[sel])[0]
    assert np.abs(q[sel] - ref).max() <= 1e-5
    kernel = md.last_kernel
    md.close()
    assert own in (1, 2 + 2 * w.K), (kernel, own)


def test_observation_vectors_reserve_one_layout():
    """The workspace of a call with observation vectors holds the slices in the layout that is read, not beside another
    one: [9,10,11] in blocks of 8 x 6 is 2 x 2 x 9 of them per step (the axes of ten and eleven states cut)."""
    import torch
    import paper_2607_17855_b200 as bi
    w = _workload(110, [9, 10, 11], [[0, 1, 2]], N=1000, T=20, K=2)
    md = bi.model_from_workload(w)
    soft = torch.rand((w.N, w.T, int(w.m.sum())), device="cuda")
    act, q = torch.from_numpy(w.act).cuda(), torch.empty((w.N, w.T, w.S), device="cuda")
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    md.run_soft("vmp", soft, act, w.K, q_out=q)
    torch.cuda.synchronize()
    used = before - torch.cuda.mem_get_info()[0]
    md.close()
    slices = w.N * w.T * 36 * 48 * 8
    assert used <= slices + (80 << 20), (used, slices)   # (the allocator takes whole chunks of 32 MB; kernels are loaded on first use)


def test_pair_models_keep_no_copy_that_no_call_reads():
    """The pair kernels take every call on a float64 model with one pair of factors of up to eight states."""
    import dataclasses
    import torch
    import paper_2607_17855_b200 as bi
    G = 120000
    w = _workload(120, [8, 7], [[0, 1]], N=1, T=2, K=2)
    rep = lambda x: np.broadcast_to(x, (G,) + x.shape[1:]).copy()
    w = dataclasses.replace(w, G=G, N=G, A=[rep(x) for x in w.A], B=[rep(x) for x in w.B], D=[rep(x) for x in w.D])
    arrays = [[torch.from_numpy(x).cuda() for x in part] for part in (w.A, w.B, w.D)]
    bi.Model(w.n, w.m, w.dep, w.U, w.G, *arrays).close()   # (the kernels of the packing are loaded)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    md = bi.Model(w.n, w.m, w.dep, w.U, w.G, *arrays)
    torch.cuda.synchronize()
    used = before - torch.cuda.mem_get_info()[0]
    md.close()
    slices = G * int(w.m[0]) * 8 * 8 * 8 * 2                          # rows and, for the filtering kernel, columns
    matrices = G * sum(6 * int(u) * int(k) * 8 * 8 for u, k in zip(w.U, w.n)) + G * 2 * 8 * 8
    assert used <= slices + matrices + (48 << 20), (used, slices, matrices)   # (sixteen allocations in whole 2 MB)


def test_a_model_that_fits_without_its_second_copy_is_made():
    """With room for the packed slices but not for the block-ordered ones beside them the handle is made without the
    latter, and the call runs on another kernel."""
    import torch
    import oracle
    import paper_2607_17855_b200 as bi
    G = 16000
    w = _workload(121, [9, 10, 11], [[0, 1, 2]], N=G, T=2, K=2)
    shared = [[torch.from_numpy(x).cuda() for x in part] for part in (w.A, w.B, w.D)]
    arrays = [[x.expand(G, *x.shape[1:]).contiguous() for x in part] for part in shared]
    bi.Model(w.n, w.m, w.dep, w.U, 1, *shared).close()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    packed = G * int(w.m[0]) * 9 * 10 * 12 * 8
    matrices = G * sum(6 * int(u) * int(k) * 12 * 8 for u, k in zip(w.U, w.n))   # (six forms of every action's, rows padded to 12)
    fill = torch.empty(torch.cuda.mem_get_info()[0] - (packed * 5 // 4 + matrices + (200 << 20)), dtype=torch.uint8, device="cuda")
    try:
        md = bi.Model(w.n, w.m, w.dep, w.U, G, *arrays)
    finally:
        del fill
        torch.cuda.empty_cache()
    q = md.bi_filter(torch.from_numpy(w.obs).cuda(), torch.from_numpy(w.act).cuda(), w.K).cpu().numpy()
    assert md.last_family == "cta_filter_f64" and md.status() == 0
    md.close()
    sel = list(range(0, G, 799))
    assert np.abs(q[sel] - oracle.run_workload(w.take_agents(sel), "filter")[0]).max() <= 1e-5


@pytest.mark.parametrize("where", [None, "first", "last", "middle"])
def test_a_single_zero_in_a_is_seen(where):
    """Filtering on a model with zeros in A stays on the CTA kernel; one zero anywhere is enough (the packing kernel's
    last warp is a partial one here)."""
    w = _workload(130, [5, 3, 7], [[0, 1, 2], [2]], N=3, T=2, K=3)
    for a in w.A:
        a[:] = np.maximum(a, 1e-6)
    if where:
        a = w.A[0] if where != "last" else w.A[1]
        a.reshape(-1)[{"first": 0, "last": -1, "middle": a.size // 2}[where]] = 0.0
    res = check_workload(w, "filter")
    assert res["family"] == ("cta_filter_f64" if where else "block_filter_f64"), res


@pytest.mark.parametrize("algo", ["filter", "vmp", "mmp"])
def test_actions_of_every_factor_are_checked(algo):
    """An action out of range raises the status flag whichever factor and step it is of, a factor of one state included."""
    import torch
    import paper_2607_17855_b200 as bi
    w = _workload(140, [3, 1, 4, 2], [[0, 2, 3], [0]], N=6, T=9, K=2)
    md = bi.model_from_workload(w)
    obs = torch.from_numpy(w.obs).cuda()
    for f in range(4):
        for step, bad in ((0, -1), (3, 9), (7, int(w.U[f]))):
            act = w.act.copy()
            act[2, step, f] = bad
            md.run(algo, obs, torch.from_numpy(act).cuda(), w.K)
            assert md.status() == 2, (f, step)
    md.run(algo, obs, torch.from_numpy(w.act).cuda(), w.K)
    assert md.status() == 0 and md.last_family == f"block_{algo}_f64"
    md.close()


@pytest.mark.parametrize("family", ["batch", "cta", "warp", "block"])
def test_threads_with_models_of_different_sizes(family):
    """Calls of several threads, each on a handle and stream of its own, on kernels that they share with different
    amounts of shared memory."""
    import threading
    import torch
    import paper_2607_17855_b200 as bi
    from test_gpu_parity import family_forced
    algo = "filter" if family == "cta" else "vmp"
    with family_forced(family):
        jobs = []
        for i, n in enumerate(([12, 12, 12], [3, 4, 5], [9, 7, 11], [6, 5, 3])):
            w = _workload(150 + i, n, [[0, 1, 2], [1, 2]], N=140, T=16, K=3)
            md = bi.model_from_workload(w)
            obs, act = torch.from_numpy(w.obs).cuda(), torch.from_numpy(w.act).cuda()
            jobs.append((md, obs, act, w.K, md.run(algo, obs, act, w.K)))
    torch.cuda.synchronize()
    failures, go = [], threading.Barrier(len(jobs))

    def work(md, obs, act, K, want):
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            q = torch.empty_like(want)
            go.wait()
            try:
                for _ in range(300):
                    md.run(algo, obs, act, K, q_out=q)
                s.synchronize()
                if not torch.equal(q, want):
                    failures.append("other beliefs")
            except Exception as e:
                failures.append(repr(e))

    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    for j in jobs:
        j[0].close()
    assert not failures, failures


@pytest.mark.parametrize("damping", [1.0, 0.5])
@pytest.mark.parametrize("case", ["warps_of_one_cta", "cluster", "shared_memory_blocks"])
def test_every_call_form(case, damping):
    """Continued, warm-started and damped calls and observation vectors, on teams of one and of several warps, windows over
    one CTA and over a cluster, blocks left over for shared memory; all by the name of the kernel that ran."""
    import torch
    import oracle
    import paper_2607_17855_b200 as bi
    from test_gpu_parity import _soft_vectors
    n, dep, T = {"warps_of_one_cta": ([3, 4, 2, 5], [[0, 1, 2], [1, 3]], 4), "cluster": ([9, 6, 12, 4], [[0, 1], [1, 2, 3], [0, 1, 2]], 13),
                 "shared_memory_blocks": ([18, 29, 11], [[0, 1, 2], [0, 2]], 7)}[case]
    N = 5
    w = _workload(160, n, dep, N=N, T=T, K=5)
    rng = np.random.default_rng(161)
    simplex = lambda *size: np.concatenate([rng.dirichlet(np.full(k, 1.5), size=size) for k in n], axis=-1).astype(np.float32)
    q_prev, q_init, soft = simplex(N), simplex(N, T), _soft_vectors(w, 162)
    act_prev = np.stack([rng.integers(0, int(u), size=N) for u in w.U], axis=1).astype(np.int32)
    cuda = lambda x: torch.from_numpy(x).cuda()
    obs, act = cuda(w.obs), cuda(w.act)
    md = bi.model_from_workload(w)
    md.set_damping(damping)
    for algo in ("filter", "vmp", "mmp"):
        prev = dict(q_prev=q_prev.astype(np.float64), act_prev=act_prev)
        start = dict(q_init=q_init.astype(np.float64))
        calls = [("from", lambda: md.run_from(algo, obs, act, cuda(q_prev), cuda(act_prev), w.K), prev),
                 ("soft", lambda: md.run_soft(algo, cuda(soft), act, w.K), dict(obs_soft=soft))]
        if algo != "filter":
            warm = md.bi_vmp_warm if algo == "vmp" else md.bi_mmp_warm
            calls += [("warm", lambda: warm(obs, act, cuda(q_init), w.K), start),
                      ("from, warm", lambda: md.run_from(algo, obs, act, cuda(q_prev), cuda(act_prev), w.K, q_init=cuda(q_init)),
                       {**prev, **start})]
        for name, call, kw in calls:
            q = call().cpu().numpy()
            assert md.last_family == f"block_{algo}_f64", (algo, name, md.last_family)
            ref = oracle.run(algo, w.n, w.m, w.dep, w.U, w.G, w.A, w.B, w.D, None if "obs_soft" in kw else w.obs, w.act, w.K,
                             damping=damping, **kw)[0]
            assert np.abs(q - ref).max() <= 1e-5, (algo, name, np.abs(q - ref).max())
    assert md.status() == 0
    md.close()


@pytest.mark.parametrize("algo", ["filter", "vmp", "mmp"])
def test_sixteen_modalities(algo):
    """More modalities than the softmax without a shift allows: log-beliefs and most probable states relative to the
    largest logit."""
    dep = [[0, 1, 2], [1, 2], [0, 2], [0]] * 4
    res = check_workload(_workload(170, [5, 4, 7], dep, N=6, T=5, K=4), algo)
    assert res["family"] == f"block_{algo}_f64", res


@pytest.mark.parametrize("case, family", [("large_tensors", "cta"), ("large_slices", "block")])
def test_filtering_with_several_parents_by_the_cost_of_a_step(case, family):
    """The prior of large transition tensors is cheaper on the CTA kernel, the iterations of large slices on the block
    kernels; which it is does not depend on the number of steps, so blocks of steps are the single call bit for bit."""
    import torch
    import paper_2607_17855_b200 as bi
    from test_gpu_parity import _blockwise
    n, dep, bdep, N, K = {"large_tensors": ([16, 7, 19], [[0, 1], [2]], [[2, 1, 0], [2, 1], [1, 0]], 4, 6),
                          "large_slices": ([4, 6, 2, 7], [[0, 1, 2, 3]], [[0, 3], [1, 2, 3], [1, 2], [0, 1, 3]], 300, 16)}[case]
    w = _workload(180, n, dep, N=N, T=7, K=K, bdep=bdep)
    res = check_workload(w, "filter", agents=range(0, N, max(1, N // 8)))
    assert res["family"] == f"{family}_filter_f64", res
    md = bi.model_from_workload(w)
    whole = md.bi_filter(torch.from_numpy(w.obs).cuda(), torch.from_numpy(w.act).cuda(), K).cpu().numpy()
    for cuts in (list(range(8)), [0, 2, 3, 7]):
        q, _ = _blockwise(md, w, cuts, K)
        assert np.array_equal(q, whole), cuts
    md.close()


@pytest.mark.parametrize("case, family", [("pairs_float32_many", "batch"), ("tiny_float32_many", "batch"),
                                          ("rank4_few", "block"), ("own_models_many", "block")])
def test_windows_by_the_estimate_of_both(case, family):
    n, dep, N, T, G, arith = {"pairs_float32_many": ([9, 32, 19], [[0, 2], [2]], 2975, 20, 1, "f32"),
                              "tiny_float32_many": ([5, 5, 2, 2, 4], [[3], [0, 1, 2], [0, 2, 3], [1, 2, 4], [0, 2, 3]], 2746, 20, 1, "f32"),
                              "rank4_few": ([14, 14, 2, 12], [[0, 1, 2, 3]], 206, 12, 1, "f64"),
                              "own_models_many": ([10, 10, 8, 6], [[0, 1], [1, 2], [0, 2, 3]], 260, 16, 260, "f64")}[case]
    res = check_workload(_workload(190, n, dep, N=N, T=T, K=6 if arith == "f32" else 16, G=G), "mmp", agents=range(0, N, N // 10), arith=arith, strict=arith == "f64")
    assert res["family"] == f"{family}_mmp_{arith}", res
    assert res["q_max_err"] < 1e-2, res   # (float32: six undamped iterations amplify 1e-6 of the logits by 1e3 at most)


@pytest.mark.parametrize("algo", ["filter", "vmp", "mmp"])
def test_float32_damped(algo):
    """The fast mode as it is used.  Logits are sums of some ten logarithms and messages, at most 60 in size: 60 x 6e-8 x 10
    roundings, 4e-5, and the damped iteration does not amplify; the bound is twice that."""
    import oracle
    import torch
    import paper_2607_17855_b200 as bi
    w = _workload(200, [9, 5, 7, 6], [[0, 1, 2], [1, 3]], N=21, T=5, K=12)
    md = bi.model_from_workload(w, arith="f32")
    md.set_damping(0.5)
    q = md.run(algo, torch.from_numpy(w.obs).cuda(), torch.from_numpy(w.act).cuda(), w.K).cpu().numpy()
    assert md.last_family == f"block_{algo}_f32"
    md.close()
    assert np.abs(q - oracle.run_workload(w, algo, damping=0.5)[0]).max() <= 8e-5


def test_long_trajectories_in_blocks_of_steps_on_the_cta_kernel():
    """The CTA filtering kernel keeps a trajectory's first observations in shared memory; a trajectory too long for that
    stays on it all the same, and equals its blocks bit for bit."""
    import torch
    import paper_2607_17855_b200 as bi
    from test_gpu_parity import _blockwise
    n, dep, T = [5, 4, 3], [[0, 1, 2]] + [[i % 3] for i in range(9)], 3000
    rng = np.random.default_rng(210)
    m, U = [9] + [3] * 9, [2, 1, 3]
    A, B, D = make_model(rng, n, m, dep, U, 1, sparsity=0.6, d_alpha=1.0)
    obs, act = sample_streams(rng, n, m, dep, U, 1, A, B, D, 3, T)
    w = Workload(name="long", algo="filter", n=np.asarray(n, np.int32), m=np.asarray(m, np.int32), dep=dep,
                 U=np.asarray(U, np.int32), G=1, A=A, B=B, D=D, N=3, T=T, K=16, obs=obs, act=act)
    md = bi.model_from_workload(w)
    whole = md.bi_filter(torch.from_numpy(obs).cuda(), torch.from_numpy(act).cuda(), w.K).cpu().numpy()
    assert md.last_family == "cta_filter_f64"
    for cuts in ([0, 1500, T], [0, 7, 900, T]):
        q, names = _blockwise(md, w, cuts, w.K)
        assert names == {"cta_filter_f64"} and np.array_equal(q, whole), cuts
    bad = obs.copy()
    bad[1, T - 1, 4] = 77   # (beyond the kept ones: clamped and flagged)
    q = md.bi_filter(torch.from_numpy(bad).cuda(), torch.from_numpy(act).cuda(), w.K).cpu().numpy()
    assert md.status() == 1 and np.array_equal(q[:, :T - 1], whole[:, :T - 1])
    bad[1, T - 1, 4] = 2
    assert np.array_equal(q, md.bi_filter(torch.from_numpy(bad).cuda(), torch.from_numpy(act).cuda(), w.K).cpu().numpy())
    md.close()

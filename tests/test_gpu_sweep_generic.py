"""Parity of the sweep and of the generic run evaluator against the CPU oracle (bit-exact)."""
import os

import numpy as np
import pytest
import torch

import oracle
from paper_2601_22996_b200 import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def par():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from tests import parity
    return parity


def _oracle_setting(inst, fam, M, tau, k):
    S = oracle.build_schedule(fam, inst.s, inst.o, M, tau=tau, k=k, s_bar=0)
    E = oracle.evaluate_events(S.run_start, S.run_len, S.run_s)
    return dict(peak=E.peak, flow=S.flow, n_completed=len(inst.o) - S.n_unfinished, horizon=S.horizon,
                job_steps=S.job_steps, feasible=int(E.peak <= M))


def _check_sweep(par, inst, fam, M, taus, ks, sample=None):
    out = par.scheduler().sweep(inst.to("cuda:0"), 0, fam, M, taus, ks)
    got = {f: t.cpu().numpy() for f, t in out.items()}
    cells = [(i, j) for i in range(len(taus)) for j in range(len(ks))] if sample is None else sample
    for i, j in cells:
        want = _oracle_setting(inst, fam, M, taus[i], ks[j])
        for f, v in want.items():
            assert int(got[f][i, j]) == v, f"{fam} tau={taus[i]} k={ks[j]} {f}: {int(got[f][i, j])} vs {v}"


@pytest.mark.parametrize("fam", ["SPS", "SIMS"])
def test_sweep_small_full_grid(par, fam):
    inst = workloads.config4(n=3000)
    taus = [1, 2, 3, 7, 16, 100, 257, 1024, 16384, 40000]
    ks = [1, 2, 3, 5, 16, 33, 100, 1000, 2999, 3000, 3001, 50000]
    _check_sweep(par, inst, fam, 1 << 20, taus, ks)


@pytest.mark.parametrize("fam", ["SPS", "SIMS"])
def test_sweep_on_any_instance_of_a_batch(par, fam):
    """The instance is a stretch of a larger batch (sizes are bounded by the batch's, not read): as a batch of its own."""
    sizes = [0, 1, 700, 3, 300]
    off = torch.tensor([0, 0, 1, 701, 704, 1004])
    c = torch.arange(1004)
    inst = workloads.Instances(off, workloads.uniform_int(83, c, 0, 90), workloads.pareto_int(84, c, 20.0, 1.1, 1, 900))
    for i, n in enumerate(sizes):
        a = int(off[i])
        own = workloads.Instances(torch.tensor([0, n]), inst.s[a:a + n].clone(), inst.o[a:a + n].clone())
        got, want = (par.scheduler().sweep(x.to("cuda:0"), k, fam, 5000, [1, 20, 400], [1, 7, 512]) for x, k in ((inst, i), (own, 0)))
        for f in want:
            assert torch.equal(got[f], want[f]), (i, f)


@pytest.mark.parametrize("fam", ["SPS", "SIMS"])
def test_sweep_ragged_and_tiny(par, fam):
    for n in (1, 2, 63, 64, 65, 8191, 8193):
        inst = workloads.config1(n=n)
        _check_sweep(par, inst, fam, 5000, [1, 5, 64, 1024, 2000], [1, 4, 64, 1000])


def test_sweep_paper_grid_sampled(par):
    """The 64 x 64 grid on a 200,000-job instance; a sample of cells against the oracle."""
    inst = workloads.config4(n=200_000)
    taus, ks = workloads.sweep_grids()
    rng = np.random.default_rng(4)
    cells = [(int(rng.integers(64)), int(rng.integers(64))) for _ in range(24)] + [(0, 0), (63, 63), (0, 63), (63, 0)]
    for fam in ("SPS", "SIMS"):
        _check_sweep(par, inst, fam, inst.meta["M"][0], taus, ks, sample=cells)


def test_sweep_agrees_with_fused_path(par):
    """Same (tau, k) through kvs_sweep and through kvs_evaluate_built (dense profile)."""
    from paper_2601_22996_b200 import binding
    inst = workloads.config2(n_inst=1, n=5000)
    taus, ks = [16, 90, 700], [2, 17, 300]
    for fam in ("SPS", "SIMS"):
        out = par.scheduler().sweep(inst.to("cuda:0"), 0, fam, 1 << 22, taus, ks)
        rows = [dict(instance=0, family=fam, M=1 << 22, tau=t, k=k) for t in taus for k in ks]
        res = par.scheduler().evaluate(inst.to("cuda:0"), binding.make_settings(rows), want_profile=True)
        assert torch.equal(res.peak.view(3, 3), out["peak"]) and torch.equal(res.flow.view(3, 3), out["flow"])
        assert torch.equal(res.horizon.view(3, 3), out["horizon"]) and torch.equal(res.job_steps.view(3, 3), out["job_steps"])


def _runs_to_gpu(batches, dev):
    off = np.zeros(len(batches) + 1, dtype=np.int64)
    off[1:] = np.cumsum([len(b[0]) for b in batches])
    cat = lambda i, dt: torch.tensor(np.concatenate([np.asarray(b[i], dtype=dt) for b in batches]) if batches else [], dtype=getattr(torch, np.dtype(dt).name)).to(dev)
    return torch.tensor(off).to(dev), cat(0, np.int64), cat(1, np.int32), cat(2, np.int32)


def test_generic_evaluator_random_runs(par):
    dev = torch.device("cuda:0")
    rng = np.random.default_rng(9)
    batches = []
    for e in range(40):
        R = int(rng.integers(0, 3000)) if e else 0
        batches.append((rng.integers(0, 20000, R), rng.integers(1, 900, R), rng.integers(0, 4000, R)))
    off, st, ln, ss = _runs_to_gpu(batches, dev)
    want = [oracle.evaluate_dense(*b) for b in batches]
    cap = torch.tensor([w.horizon for w in want], dtype=torch.int64, device=dev)
    M = torch.tensor([w.peak - (i % 2) for i, w in enumerate(want)], dtype=torch.int64, device=dev)
    res = par.scheduler().evaluate_runs(off, st, ln, ss, cap, M=M)
    prof, poff = res.profile.cpu().numpy(), res.profile_off.cpu().numpy()
    for e, w in enumerate(want):
        assert int(res.status[e]) == 0
        assert (int(res.peak[e]), int(res.horizon[e]), int(res.job_steps[e])) == (w.peak, w.horizon, w.job_steps)
        assert np.array_equal(prof[poff[e]:poff[e + 1]].astype(np.int64), w.profile)
        assert int(res.feasible[e]) == int(w.peak <= int(M[e]))


def test_generic_evaluator_paper_examples(par, golden_dir):
    """Example 1's two schedules as explicit runs, and the staggered schedule of the SimS lower bound."""
    dev = torch.device("cuda:0")
    batches, want = [], []
    for ln in open(os.path.join(golden_dir, "example1_memory.txt")):
        if ln.startswith("#") or not ln.strip():
            continue
        head, cells = ln.split(":")
        fam, k, tau, _ = head.split()
        k, tau = int(k), int(tau)
        starts = [(i * tau) // k if fam == "SPS" else (i // k) * tau for i in range(15)]
        batches.append((starts, [5] * 15, [0] * 15))
        want.append([int(x) for x in cells.split()])
    o, d, n = 60, 23, 12
    batches.append(([i * d for i in range(n)], [o] * n, [0] * n))
    off, st, ln_, ss = _runs_to_gpu(batches, dev)
    cap = torch.tensor([19, 25, (n - 1) * d + o], dtype=torch.int64, device=dev)
    res = par.scheduler().evaluate_runs(off, st, ln_, ss, cap)
    prof, poff = res.profile.cpu().numpy(), res.profile_off.cpu().numpy()
    assert list(prof[poff[0]:poff[1]]) == want[0] and list(prof[poff[1]:poff[2]]) == want[1]
    assert res.peak.cpu().tolist() == [15, 15, 3 * o - 3 * d]


def test_generic_evaluator_clips_at_capacity(par):
    dev = torch.device("cuda:0")
    off, st, ln, ss = _runs_to_gpu([([0, 4], [10, 3], [2, 1])], dev)
    res = par.scheduler().evaluate_runs(off, st, ln, ss, torch.tensor([6], dtype=torch.int64, device=dev))
    from paper_2601_22996_b200 import binding
    assert res.status.cpu().tolist() == [binding.EVAL_CAPACITY] and int(res.horizon[0]) == 10
    assert res.profile.cpu().tolist() == [3, 4, 5, 6, 7 + 2, 8 + 3]


@pytest.mark.parametrize("fam", ["SPS", "SIMS"])
@pytest.mark.parametrize("n,o_max", [(127, 3), (128, 300), (4096, 70_000), (4097, 1 << 24), (12_289, 40)])
def test_sweep_block_and_chunk_edges(par, fam, n, o_max):
    """Edges of the 64-rank blocks and 4,096-job chunks, one to four radix passes, more parallelism values than one batch of tables."""
    c = torch.arange(n)
    inst = workloads.Instances(torch.tensor([0, n]), workloads.pareto_int(77, c, 20.0, 0.8, 0, 9000), workloads.uniform_int(78, c, 1, o_max))
    taus = sorted({1, 2, o_max // 3 + 1, max(1, o_max - 1), o_max, 2 * o_max + 1})
    ks = [1, 2, 3, 63, 64, 65, n - 1, n, n + 1] + list(range(100, 340))
    cells = [(i, j) for i in range(len(taus)) for j in list(range(9)) + [9 + 118, 9 + 119, 9 + 130, len(ks) - 1]]
    _check_sweep(par, inst, fam, 1 << 26, taus, ks, sample=cells)


@pytest.mark.parametrize("case", ["tile edges", "many small", "one long", "wide sums", "odd offsets"])
def test_generic_evaluator_tiles(par, case):
    """Capacities around the tile sizes, runs that cross several tiles, runs outside the capacity, sums beyond 32 bits, and offsets that are not
    monotone (the 64-bit kernel takes the last two)."""
    from paper_2601_22996_b200 import binding
    dev = torch.device("cuda:0")
    rng = np.random.default_rng(5)
    sizes = {"tile edges": [1, 511, 1536, 1537, 11775, 11776, 11777, 40000], "many small": [7] * 300, "one long": [700_001],
             "wide sums": [3000, 20000], "odd offsets": [100, 100]}[case]
    batches = []
    for h in sizes:
        R = 5000 if case == "one long" else min(h, 400) + 1
        st = rng.integers(0, h, R)
        ln = np.minimum(rng.integers(1, max(2, h // 2), R), h - st)
        batches.append((st, np.maximum(ln, 1), rng.integers(0, (1 << 26) if case == "wide sums" else 4000, R)))
    off, st, ln, ss = _runs_to_gpu(batches, dev)
    want = [oracle.evaluate_dense(*b) for b in batches]
    cap = torch.tensor([w.horizon + (5 if i % 3 == 1 else 0) for i, w in enumerate(want)], dtype=torch.int64, device=dev)
    M = torch.tensor([w.peak for w in want], dtype=torch.int64, device=dev)
    if case == "odd offsets":
        poff = torch.tensor([0, 200, 100], dtype=torch.int64, device=dev)     # the second evaluation's capacity is negative
        ctx = par.scheduler().context(binding.workspace_bytes(0, 0, 0, 2, generic_capacity=200))
        ev = {**par.scheduler().scalars(2, dev), "profile_off": poff}
        ctx.evaluate_schedule(dict(run_off=off, run_start=st, run_len=ln, run_s=ss, M=M), ev, capacity_total=200)
        assert ev["status"].tolist() == [0, binding.EVAL_CAPACITY | binding.EVAL_BAD_INPUT]
        assert int(ev["peak"][0]) == want[0].peak and int(ev["peak"][1]) == -1
        return
    res = par.scheduler().evaluate_runs(off, st, ln, ss, cap, M=M)
    prof, poff = res.profile.cpu().numpy(), res.profile_off.cpu().numpy()
    for e, w in enumerate(want):
        over = w.peak > 0x7fffffff
        assert int(res.status[e]) == (binding.EVAL_RANGE if over else 0)
        assert (int(res.peak[e]), int(res.horizon[e]), int(res.job_steps[e])) == (w.peak, w.horizon, w.job_steps)
        got = prof[poff[e]:poff[e + 1]].astype(np.int64)
        assert np.array_equal(got[:w.horizon], np.minimum(w.profile, 0x7fffffff)) and (got[w.horizon:] == -7).all()
        assert int(res.feasible[e]) == 1

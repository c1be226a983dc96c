"""Variants inside the geometric classes on the GPU against the oracle: simultaneous batches as the
subroutine of every phase, the parallelism of a phase sized by the longest prompt among its participants,
and the sweep over tunable initial slices.  Bit-exact, every output."""
import os
import re

import numpy as np
import pytest
import torch

import oracle
from paper_2601_22996_b200 import binding, workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def par():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from tests import parity
    return parity


@pytest.mark.parametrize("sub,pc", [(1, 0), (0, 1), (1, 1)])
def test_tiny_instances_all_variants(par, sub, pc):
    inst = workloads.random_small(4100 + 10 * sub + pc, 60, 48, 30, 90)
    sizes = (inst.job_off[1:] - inst.job_off[:-1]).numpy()
    rows = []
    for i in range(inst.n_instances):
        if sizes[i] == 0:
            continue
        a, b = int(inst.job_off[i]), int(inst.job_off[i + 1])
        M = int(inst.s[a:b].max() + inst.o[a:b].max()) + 7 * i
        for fam in ("GBA", "GSA"):
            for alpha in ((2, 1), (3, 2)):
                rows.append(dict(instance=i, family=fam, M=M, alpha=alpha, subroutine=sub, per_class_s=pc))
            rows.append(dict(instance=i, family=fam, M=M, beta0=3, subroutine=sub, per_class_s=pc))
    par.check_batch(inst, binding.make_settings(rows), label=f"variants sub={sub} pc={pc}")


def test_variants_with_estimates_and_windows(par):
    inst = workloads.random_small(4200, 24, 64, 25, 80, with_est=True)
    # arrivals: nondecreasing per instance, a few windows each
    arr = torch.zeros_like(inst.o, dtype=torch.int64)
    for i in range(inst.n_instances):
        a, b = int(inst.job_off[i]), int(inst.job_off[i + 1])
        arr[a:b] = torch.arange(b - a, dtype=torch.int64) * 3
    inst.arrival = arr
    rows = []
    for i in range(inst.n_instances):
        a, b = int(inst.job_off[i]), int(inst.job_off[i + 1])
        if b == a:
            continue
        M = int(inst.s[a:b].max() + max(int(inst.o[a:b].max()), 1)) + 40
        for fam in ("GBA", "GSA"):
            for sub, pc in ((1, 0), (0, 1), (1, 1)):
                rows.append(dict(instance=i, family=fam, M=M, subroutine=sub, per_class_s=pc))
    par.check_batch(inst, binding.make_settings(rows), window=37, label="variants est+windows")


def test_config2_subset_variants(par):
    inst = workloads.config2(n_inst=4, n=10_000)
    st = np.concatenate([binding.settings_grid(range(4), ["GBA", "GSA"], [1 << 17, 1 << 21], subroutine=1),
                         binding.settings_grid(range(4), ["GBA", "GSA"], [1 << 18, 1 << 24], per_class_s=1),
                         binding.settings_grid(range(4), ["GBA", "GSA"], [1 << 19], subroutine=1, per_class_s=1)])
    par.check_batch(inst, st, want_runs=False, label="config 2 variants")


def test_uniform_experiment_both_subroutines(par):
    """The uniform experiment of the paper (n = 200, o = 16, s = 0, M = 256, alpha = 2): the batching algorithm
    gives 14083 with the staggered pipeline and, with simultaneous batches inside the same class, the
    simultaneous number 21632."""
    inst = workloads.Instances(torch.tensor([0, 200]), torch.zeros(200, dtype=torch.int32), torch.full((200,), 16, dtype=torch.int32))
    st = binding.make_settings([dict(instance=0, family="GBA", M=256), dict(instance=0, family="GBA", M=256, subroutine=1)])
    res = par.scheduler().evaluate(inst.to("cuda:0"), st, want_jobs=False)
    assert res.flow.tolist() == [14083, 21632] and res.status.tolist() == [0, 0]


def test_rejects_variants_on_other_families(par):
    inst = workloads.config1().to("cuda:0")
    with pytest.raises(binding.KvsError):
        par.scheduler().evaluate(inst, binding.make_settings([dict(instance=0, family="SPS", M=200_000, subroutine=1)]))


@pytest.mark.parametrize("fam", ["GBA", "GSA"])
def test_sweep_over_initial_slices(par, fam):
    inst = workloads.config2(n_inst=2, n=3000)
    one = inst.slice(1, 2)
    beta0 = [0, 1, 5, 64, 256, 5000]
    M = 1 << 18
    for sub in (0, 1):
        out = {f: t.cpu().numpy() for f, t in par.scheduler().sweep_beta0(inst.to("cuda:0"), 1, fam, M, beta0, subroutine=sub).items()}
        for i, b0 in enumerate(beta0):
            S = oracle.build_schedule(fam, one.s, one.o, M, beta0=b0, subroutine=sub)
            E = oracle.evaluate_dense(S.run_start, S.run_len, S.run_s, want_profile=False)
            got = tuple(int(out[f][i]) for f in ("peak", "flow", "horizon", "job_steps", "n_completed", "feasible"))
            assert got == (E.peak, S.flow, S.horizon, S.job_steps, 3000 - S.n_unfinished, int(E.peak <= M)), (fam, b0, sub)
    # an infeasible budget: nothing is scheduled and the cell says so
    out = par.scheduler().sweep_beta0(inst.to("cuda:0"), 1, fam, 100, [0, 64])
    assert out["feasible"].tolist() == [0, 0] and out["n_completed"].tolist() == [0, 0] and out["peak"].tolist() == [-1, -1]


@pytest.mark.parametrize("sub,pc", [(1, 0), (0, 1), (1, 1)])
def test_variants_peak_without_profile(par, sub, pc):
    """No profile stored: batches are summed per round in which one of their runs can end (short slices) or pair by pair (long
    ones); a call of a few evaluations shares them between CTAs."""
    inst = workloads.random_small(4300 + 10 * sub + pc, 80, 48, 30, 90)
    M = [int(inst.s[a:b].max() + inst.o[a:b].max()) + 7 * (i % 9) if b > a else 2 for i, (a, b) in enumerate(zip(inst.job_off[:-1].tolist(), inst.job_off[1:].tolist()))]
    rows = [dict(instance=i, family=f, M=m, alpha=al, beta0=b, subroutine=sub, per_class_s=pc)
            for i, m in enumerate(M) for f in ("GBA", "GSA") for al, b in (((2, 1), 0), ((3, 2), 0), ((2, 1), 3))]
    par.check_batch(inst, binding.make_settings(rows), want_runs=False, want_profile=False, label="peak of variants")
    inst.arrival = torch.cat([torch.arange(int(c), dtype=torch.int64) * 5 for c in (inst.job_off[1:] - inst.job_off[:-1])])
    par.check_batch(inst, binding.make_settings(rows), window=64, want_runs=False, want_profile=False, label="peak of variants, windows")
    c = torch.arange(7000)
    inst = workloads.Instances(torch.tensor([0, 1000, 7000]), workloads.uniform_int(97, c, 0, 700), workloads.pareto_int(98, c, 40.0, 1.1, 1, 9000))
    rows = [dict(instance=i, family=f, M=m, alpha=al, subroutine=sub, per_class_s=pc, **({} if s < 0 else dict(s_bar=s)))
            for i in (0, 1) for m in (12_000, 1 << 17, 1 << 21) for f in ("GBA", "GSA") for al in ((2, 1), (3, 2)) for s in (-1, 100)]
    for copies in (1, 4):
        par.check_batch(inst, binding.make_settings(rows * copies), want_runs=False, want_profile=False, label="peak of variants")


def test_sweep_over_the_only_instance_of_a_larger_array(par):
    """The instance is a part of the arrays: the same results as with arrays of its own."""
    c = torch.arange(900)
    s, o = workloads.uniform_int(81, c, 1, 60), workloads.uniform_int(82, c, 1, 300)
    part = workloads.Instances(torch.tensor([200, 700]), s, o).to("cuda:0")
    own = workloads.Instances(torch.tensor([0, 500]), s[200:700].clone(), o[200:700].clone()).to("cuda:0")
    for fam in ("GBA", "GSA"):
        a, b = (par.scheduler().sweep_beta0(inst, 0, fam, 4000, [0, 5, 64]) for inst in (part, own))
        for f in a:
            assert torch.equal(a[f], b[f]), (fam, f)


@pytest.mark.parametrize("copies", [1, 4])      # shared evaluations, a call that is split by family
def test_variants_with_and_without_profile_in_one_call(par, copies):
    """Some evaluations of a call store their profile, others have capacity 0: variants and plain schedules side by side."""
    inst = workloads.random_small(4400, 10, 60, 30, 90)
    M = [int(inst.s[a:b].max() + inst.o[a:b].max()) + 40 if b > a else 40 for a, b in zip(inst.job_off[:-1].tolist(), inst.job_off[1:].tolist())]
    rows = [dict(instance=i, family=f, M=m, subroutine=sub, per_class_s=pc) for i, m in enumerate(M) for f in ("GBA", "GSA") for sub, pc in ((0, 0), (1, 0), (0, 1))]
    st = binding.make_settings(rows * copies)
    P = st.shape[0]
    assert P > 148 if copies > 1 else P <= 148
    whole = par.scheduler().evaluate(inst.to("cuda:0"), st, want_profile=True)
    wanted = torch.arange(P) % 3 != 1
    cap = torch.where(wanted.to("cuda:0"), whole.horizon, 0)
    some = par.scheduler().evaluate(inst.to("cuda:0"), st, want_profile=True, profile_capacity=cap)
    for f in ("status", "flow", "peak", "horizon", "job_steps", "n_runs", "feasible", "job_start", "job_completion"):
        assert torch.equal(getattr(whole, f), getattr(some, f)), f
    for e in torch.nonzero(wanted).flatten().tolist():
        a, b = whole.profile_off[e:e + 2].tolist()
        c, d = some.profile_off[e:e + 2].tolist()
        assert torch.equal(whole.profile[a:b], some.profile[c:d]), e
    for e in range(0, P // copies, 7):
        row = st[e]
        a, b = inst.job_off[int(row["instance"]):int(row["instance"]) + 2].tolist()
        S = oracle.build_schedule(int(row["family"]), inst.s[a:b], inst.o[a:b], int(row["M"]), subroutine=int(row["subroutine"]), per_class_s=int(row["per_class_s"]))
        if S.status == 0:
            E = oracle.evaluate_dense(S.run_start, S.run_len, S.run_s, want_profile=False)
            assert (int(some.peak[e]), int(some.flow[e])) == (E.peak, S.flow), rows[e]


@pytest.mark.parametrize("want_profile", [True, False])
@pytest.mark.parametrize("kind", ["plain", "one variant", "estimates", "estimates and windows"])
def test_shared_evaluations_by_kernel(par, kind, want_profile):
    """Calls of few evaluations, each of which several CTAs share: without variants, with one among plain evaluations, on estimates."""
    est = kind.startswith("estimates")
    inst = workloads.random_small(4300, 5, 700, 60, 200, with_est=est)
    window = 0
    if kind == "estimates and windows":
        off = inst.job_off
        inst.arrival = torch.cat([torch.arange(int(off[i + 1] - off[i])) * 2 for i in range(inst.n_instances)])
        window = 151
    rows = []
    for i in range(inst.n_instances):
        for fam in ("GBA", "GSA", "SPS", "SIMS"):
            rows.append(dict(instance=i, family=fam, M=2_000 + 900 * i))
    if kind == "one variant":
        rows[5].update(subroutine=1, per_class_s=1)
    par.check_batch(inst, binding.make_settings(rows), window=window, want_runs=False, want_profile=want_profile, label=f"shared {kind}")


def _shared_phases(S, n, parts):
    """Slicing phases of a schedule that all CTAs of its evaluation look at: enough pairs of a run end and a run that may be active then,
    and cheaper so than round by round (the rule and its constants in kvs_fused.cu; tiles of 4,096 rounds, 512 threads)."""
    source = open(os.path.join(os.path.dirname(binding.__file__), "csrc", "kvs_fused.cu")).read()
    cycles = int(re.search(r"constexpr int PAIR_CYCLES = (\d+);", source)[1])
    least = 1 << int(re.search(r"constexpr u64 SHARED_PAIRS = 1u << (\d+);", source)[1])
    N, tau, k = (v.astype(np.int64).tolist() for v in (S.n_part, S.tau, S.k))
    first = next(q for q in range(len(N)) if q + 1 == len(N) or N[q + 1] != n)      # before it no job has left: prefix sums
    shared = []
    for q in range(first, len(N)):
        pairs, rounds = N[q] * min(N[q], k[q]), -(-((N[q] - 1) * tau[q] // k[q] + tau[q]) // 4096) * 6000
        if N[q] and pairs > least and rounds >= N[q] and pairs // 512 * cycles // parts < rounds:
            shared.append(q)
    return shared


@pytest.mark.parametrize("n, alpha", [(6_000, (2, 1)), (2_500, (3, 2)), (513, (2, 1)), (30_000, (2, 1))])
def test_few_long_phases_are_shared_between_ctas(par, n, alpha):
    """Evaluations without a profile whose long slices pair many run ends with many runs: every CTA of an evaluation takes some of the ends.
    Of 513 jobs no phase has enough pairs: there the phases are taken in turn.  (The batching rows are evaluated from their classes.)"""
    inst = workloads.config2(n_inst=1, n=n)
    rows = [dict(instance=0, family=fam, M=M, beta0=b, alpha=alpha) for fam in ("GBA", "GSA") for M in (1 << 20, 1 << 22) for b in (0, 40, 700, 3_000)]
    shared = [bool(_shared_phases(oracle.build_schedule("GSA", inst.s, inst.o, r["M"], alpha=alpha, beta0=r["beta0"]), n, 16)) for r in rows[8:]]
    assert any(shared) == (n > 513) and (n < 30_000 or shared[0])
    par.check_batch(inst, binding.make_settings(rows), want_runs=False, want_profile=False, label=f"long phases n={n}")
    par.check_batch(inst, binding.make_settings(rows[8:9]), want_runs=False, want_profile=False, label=f"long phases alone n={n}")

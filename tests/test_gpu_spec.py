"""Speculative runs on top of the slicing schedule (GSA-Spec) on the GPU against the oracle: every job's start and
completion, the per-round memory, peak, flow, horizon, executed runs and job-steps, bit for bit."""
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


def test_hand_worked_instance(par):
    """The instance of tests/golden/speculative_runs_hand_example.txt."""
    inst = workloads.Instances(torch.tensor([0, 3]), torch.zeros(3, dtype=torch.int32), torch.tensor([4, 4, 2], dtype=torch.int32))
    st = binding.make_settings([dict(instance=0, family="GSAS", M=6), dict(instance=0, family="GSA", M=6)])
    res = par.scheduler().evaluate(inst.to("cuda:0"), st, want_jobs=True, want_profile=True)
    assert res.job_start[:3].tolist() == [6, 8, 1] and res.job_completion[:3].tolist() == [10, 12, 3]
    assert res.job_completion[3:].tolist() == [10, 16, 5]
    assert res.flow.tolist() == [25, 31] and res.horizon.tolist() == [12, 16] and res.peak.tolist() == [6, 6]
    assert res.n_runs.tolist() == [11, 8] and res.job_steps.tolist() == [25, 19]
    a = int(res.profile_off[0])
    assert res.profile[a:a + 16].tolist() == [3, 3, 5, 5, 4, 3, 3, 5, 4, 6, 3, 4, 0, 0, 0, 0]


def test_tiny_instances(par):
    inst = workloads.random_small(6100, 80, 60, 30, 90)
    rows = []
    for i in range(inst.n_instances):
        a, b = int(inst.job_off[i]), int(inst.job_off[i + 1])
        if b == a:
            continue
        M = int(inst.s[a:b].max() + inst.o[a:b].max()) + 9 * i
        for alpha in ((2, 1), (3, 2), (4, 3)):
            rows.append(dict(instance=i, family="GSAS", M=M, alpha=alpha))
        rows.append(dict(instance=i, family="GSAS", M=M, beta0=4))
        rows.append(dict(instance=i, family="GSAS", M=4 * M))
        rows.append(dict(instance=i, family="GSA", M=M))          # other families beside it in one call
        rows.append(dict(instance=i, family="GBAD", M=M))
    par.check_batch(inst, binding.make_settings(rows), want_runs=False, label="spec tiny")


def test_single_prompt_length_and_edges(par):
    """Equal prompt lengths (the paper's model), one job, a budget that one job fills, an empty instance."""
    rng = np.random.default_rng(6200)
    offs, s, o = [0], [], []
    for n, sv in ((1, 3), (0, 0), (40, 0), (200, 7), (3, 7), (64, 1)):
        s += [sv] * n
        o += rng.integers(1, 50, n).tolist()
        offs.append(offs[-1] + n)
    inst = workloads.Instances(torch.tensor(offs), torch.tensor(s, dtype=torch.int32), torch.tensor(o, dtype=torch.int32))
    rows = []
    for i in range(inst.n_instances):
        for M in (57, 64, 300, 5000):
            rows.append(dict(instance=i, family="GSAS", M=M))
    par.check_batch(inst, binding.make_settings(rows), want_runs=False, label="spec edges")


def test_config2_subset(par):
    """Thousands of jobs, profiles of several tiles, speculative runs by the hundred at the larger budgets; the
    pipeline is kept, so no job completes later than in the slicing schedule."""
    inst = workloads.config2(n_inst=2, n=3_000)
    st = binding.settings_grid(range(2), ["GSAS"], [1 << 17, 1 << 19])
    par.check_batch(inst, st, want_runs=False, label="spec config 2")
    res_s = par.scheduler().evaluate(inst.to("cuda:0"), st, want_jobs=True, want_profile=True)
    st_b = st.copy()
    st_b["family"] = binding.GSA
    res_b = par.scheduler().evaluate(inst.to("cuda:0"), st_b, want_jobs=True, want_profile=True)
    assert bool((res_s.job_completion <= res_b.job_completion).all()) and bool((res_s.flow < res_b.flow).all())
    M = torch.from_numpy(np.ascontiguousarray(st["M"])).to(res_s.peak.device)
    assert bool((res_s.peak <= M).all()) and bool((res_s.feasible == 1).all())


def test_rejects_what_speculation_is_not_defined_on(par):
    est = workloads.random_small(6300, 3, 20, 10, 30, with_est=True).to("cuda:0")
    with pytest.raises(binding.KvsError):
        par.scheduler().evaluate(est, binding.make_settings([dict(instance=0, family="GSAS", M=500)]), want_profile=True)
    one = workloads.config1().to("cuda:0")
    with pytest.raises(binding.KvsError):      # no profile: no working storage
        par.scheduler().evaluate(one, binding.make_settings([dict(instance=0, family="GSAS", M=200_000)]), want_profile=False)
    with pytest.raises(binding.KvsError):
        par.scheduler().evaluate(one, binding.make_settings([dict(instance=0, family="GSAS", M=200_000, subroutine=1)]), want_profile=True)


def _spec_instance(n, seed, o_max, s_max):
    c = torch.arange(n)
    return workloads.uniform_int(seed, c, 0, s_max), workloads.pareto_int(seed + 1, c, 3.0, 1.1, 1, o_max)


@pytest.mark.parametrize("n", [9_000, 12_000, 20_500])
def test_evaluations_on_chip_by_size(par, n):
    """Three evaluations per CTA of the kernel in shared memory, three with the shortest ring of rounds, one."""
    s, o = _spec_instance(n, 63, 60, 20)
    inst = workloads.Instances(torch.tensor([0, n]), s, o)
    par.check_batch(inst, binding.settings_grid(range(1), ["GSAS"], [1 << 14, 1 << 16, 1 << 18]), want_runs=False, label=f"spec n={n}")


def test_evaluations_left_by_the_on_chip_kernel(par):
    """Response lengths of 65,535 and more, prompts of 65,536 and more, budgets of 2^30 and more do not fit its 16-bit and
    32-bit state; the instances beside them do."""
    sizes, s, o = [], [], []
    for k, (omax, smax) in enumerate(((65_534, 0), (65_535, 0), (70_000, 0), (40, 65_535), (40, 65_536), (40, 5))):
        a, b = _spec_instance(70, 64 + 2 * k, 40, 30)
        a[3], b[5] = max(smax, 1), omax
        sizes.append(70); s.append(a); o.append(b)
    inst = workloads.Instances(torch.tensor([0] + sizes).cumsum(0), torch.cat(s), torch.cat(o))
    rows = [dict(instance=i, family="GSAS", M=M) for i in range(len(sizes)) for M in (140_000, 200_000)]
    rows += [dict(instance=5, family="GSAS", M=M) for M in ((1 << 30) - 1, 1 << 30)]
    par.check_batch(inst, binding.make_settings(rows), want_runs=False, label="spec left")


@pytest.mark.parametrize("n", [31, 33, 127, 129, 4_095, 4_097])
def test_on_chip_maps_and_groups(par, n):
    """Edges of the words, the 128-job rows and the 4,096-job probes of the map of free jobs; five budgets make a CTA of
    three and one of two.  The small budgets' windows of 32 rounds are looked at as a whole, those of the large ones hold too many starts."""
    s, o = _spec_instance(n, 71, 60, 20)
    inst = workloads.Instances(torch.tensor([0, n]), s, o)
    st = binding.settings_grid(range(1), ["GSAS"], [1 << 8, 1 << 9, 1 << 11, 1 << 14, 1 << 17])
    par.check_batch(inst, st, want_runs=False, label=f"spec maps n={n}")
    st["alpha_num"], st["alpha_den"] = 3, 2               # slices that occur twice: phases that nobody leaves
    par.check_batch(inst, st[1:4], want_runs=False, label=f"spec maps 3/2 n={n}")


@pytest.mark.parametrize("n, lo, hi, M", [(900, 2_100, 4_000, 1 << 19), (900, 2_100, 4_000, 1 << 20), (500, 300, 1_300, 1 << 17), (60, 8_000, 40_000, 1 << 18)])
def test_long_runs_leave_the_plan(par, n, lo, hi, M):
    """Dropped runs that end within the ring of rounds, beyond it, and more of them at a time than the list of those holds."""
    c = torch.arange(n)
    inst = workloads.Instances(torch.tensor([0, n]), workloads.uniform_int(81, c, 0, 20), workloads.uniform_int(82, c, lo, hi))
    par.check_batch(inst, binding.settings_grid(range(1), ["GSAS"], [M]), want_runs=False, label=f"spec long {lo}..{hi} M={M}")


@pytest.mark.parametrize("n, instances, budgets", [(500, 2_400, 1), (300, 600, 5), (2_000, 800, 2), (5_000, 640, 1), (9_500, 320, 1)])
def test_groups_by_the_size_of_the_batch(par, n, instances, budgets):
    """More evaluations than the GPU holds, with one, two and five budgets per instance, against the same ones a few at a time: rings of other
    lengths, groups of other sizes.  Two instances against the oracle."""
    s, o = _spec_instance(n * instances, 91, 60, 20)
    inst = workloads.Instances(torch.arange(instances + 1) * n, s, o)
    st = binding.settings_grid(range(instances), ["GSAS"], np.array([[1 << (9 + (i + 2 * b) % 9) for b in range(budgets)] for i in range(instances)]))
    all_at_once = par.scheduler().evaluate(inst.to("cuda:0"), st, want_profile=True)
    assert not bool(all_at_once.status.any())
    step = 64
    for i in range(0, instances, step):
        j = min(instances, i + step)
        some = par.scheduler().evaluate(inst.slice(i, j).to("cuda:0"), binding.settings_grid(range(j - i), ["GSAS"], st["M"].reshape(instances, budgets)[i:j]), want_profile=True)
        for f in ("flow", "peak", "horizon", "job_steps", "n_runs", "n_unfinished", "feasible"):
            assert torch.equal(getattr(some, f), getattr(all_at_once, f)[i * budgets:j * budgets]), f
        for f, off in (("job_start", "job_out_off"), ("job_completion", "job_out_off"), ("profile", "profile_off")):
            ends = getattr(all_at_once, off)
            assert torch.equal(getattr(some, f), getattr(all_at_once, f)[int(ends[i * budgets]):int(ends[j * budgets])]), f
    par.check_batch(inst.slice(0, 2), binding.settings_grid(range(2), ["GSAS"], st["M"].reshape(instances, budgets)[:2]), want_runs=False, label="spec groups")

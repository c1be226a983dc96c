"""Parity of the CUDA path against the CPU oracle, through the C ABI.  Bit-exact: every
quantity is an int32/int64 token or round count."""
import numpy as np
import pytest
import torch

from paper_2601_22996_b200 import binding, workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def par():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from tests import parity
    return parity


def _all_settings(inst, M_of, families=("GBA", "GSA", "SPS", "SIMS"), alpha=(2, 1), **extra):
    rows = []
    for i in range(inst.n_instances):
        for fam in families:
            rows.append(dict(instance=i, family=fam, M=M_of(i), alpha=alpha, **extra))
    return binding.make_settings(rows)


def _tight_M(inst, slack):
    """Budget per instance: largest s + largest o + slack (so that every job fits alone)."""
    out = []
    for i in range(inst.n_instances):
        a, b = int(inst.job_off[i]), int(inst.job_off[i + 1])
        out.append((int(inst.s[a:b].max()) + int(inst.o[a:b].max()) if b > a else 2) + slack)
    return out


@pytest.mark.parametrize("alpha", [(2, 1), (3, 2), (4, 3), (7, 4)])
@pytest.mark.parametrize("seed", [1, 2])
def test_tiny_random_instances_all_families(par, alpha, seed):
    inst = workloads.random_small(seed * 100 + alpha[0], n_inst=150, n_max=64, s_max=40, o_max=90,
                                  equal_s=(seed == 2))
    M = _tight_M(inst, slack=17 * seed + 40)
    st = _all_settings(inst, lambda i: M[i], alpha=alpha)
    par.check_batch(inst, st, label=f"tiny a={alpha}")


def test_tiny_tight_budget_and_explicit_parameters(par):
    inst = workloads.random_small(7, n_inst=120, n_max=48, s_max=9, o_max=30)
    M = _tight_M(inst, slack=0)                       # k* = 1 in the last phases
    rows = []
    for i in range(inst.n_instances):
        rows += [dict(instance=i, family="GBA", M=M[i]), dict(instance=i, family="GSA", M=M[i]),
                 dict(instance=i, family="SPS", M=M[i] + 50, tau=1 + i % 7, k=1 + i % 5),       # unfinished jobs
                 dict(instance=i, family="SIMS", M=M[i] + 50, tau=3 + i % 11, k=1 + i % 4),
                 dict(instance=i, family="SPS", M=M[i] + 9, tau=35, k=200),                     # infeasible on purpose
                 dict(instance=i, family="GSA", M=M[i] + 100, s_bar=3),                         # s_bar below max s
                 dict(instance=i, family="GBA", M=M[i] + 300, beta0=4, alpha=(3, 2)),
                 dict(instance=i, family="GSA", M=M[i] + 300, beta0=64)]
    par.check_batch(inst, binding.make_settings(rows), label="explicit")


def test_estimates_and_windows(par):
    inst = workloads.random_small(11, n_inst=60, n_max=200, s_max=30, o_max=120, with_est=True)
    M = _tight_M(inst, slack=200)
    st = _all_settings(inst, lambda i: M[i], alpha=(2, 1))
    par.check_batch(inst, st, label="estimates")
    par.check_batch(inst, _all_settings(inst, lambda i: M[i], families=("GBA", "GSA"), alpha=(3, 2)), label="estimates 3/2")
    g = torch.Generator().manual_seed(5)               # arrivals: nondecreasing per instance
    arr = torch.zeros_like(inst.s, dtype=torch.int64)
    for i in range(inst.n_instances):
        a, b = int(inst.job_off[i]), int(inst.job_off[i + 1])
        arr[a:b] = torch.sort(torch.randint(0, 900, (b - a,), generator=g)).values
    inst.arrival = arr
    for W in (1, 37, 256, 5000):
        par.check_batch(inst, st, window=W, label=f"window {W}")
    inst.o_est = None
    par.check_batch(inst, st, window=64, label="window exact")


def test_config1_single_instance(par):
    inst = workloads.config1()
    for alpha in [(2, 1), (4, 3), (3, 2)]:
        st = _all_settings(inst, lambda i: 200_000, alpha=alpha)
        assert par.check_batch(inst, st, label="config1") > 0


def test_config2_subset_full_compare(par):
    inst = workloads.config2(n_inst=6)
    st = binding.settings_grid(range(6), ["GBA", "GSA"], inst.meta["M"])
    par.check_batch(inst, st, label="config2")


def test_config3_subset_online(par):
    inst = workloads.config3(n_inst=2, n=100_000)
    st = binding.settings_grid(range(2), ["GBA", "GSA"], inst.meta["M"])
    par.check_batch(inst, st, window=inst.meta["window"], label="config3")
    st = binding.settings_grid(range(2), ["SPS", "SIMS"], inst.meta["M"])
    par.check_batch(inst, st, window=inst.meta["window"], want_runs=False, label="config3 sps")


def test_config5_subset_mixed(par):
    inst = workloads.config5(n_inst=12)
    M = inst.meta["M_per_instance"].numpy()
    st = binding.settings_grid(range(12), ["GBA", "GSA"], M[:, None])
    par.check_batch(inst, st, want_runs=False, label="config5 geo")
    st = binding.settings_grid(range(12), ["SPS", "SIMS"], M[:, None])
    par.check_batch(inst, st, want_runs=False, want_profile=False, label="config5 sps")


def test_large_single_instance(par):
    inst = workloads.config4(n=300_000)
    st = binding.settings_grid([0], ["GBA", "GSA"], [1 << 22, 1 << 19])
    par.check_batch(inst, st, want_runs=False, label="big")


def test_many_runs_per_round_over_several_tiles(par):
    """Short prompts and a budget of some ten thousand tokens: the early phases of the geometric
    families start eight or more runs per round (k >= 8 tau) and, with 150,000 jobs, still last
    several tiles of rounds; with estimates both families carry killed jobs over."""
    g = torch.Generator().manual_seed(77)
    n = 150_000
    s = torch.randint(0, 4, (n,), generator=g, dtype=torch.int32)
    short = torch.randint(1, 41, (n,), generator=g, dtype=torch.int32)
    long_ = torch.randint(41, 401, (n,), generator=g, dtype=torch.int32)
    o = torch.where(torch.rand(n, generator=g) < 0.6, short, long_)
    inst = workloads.Instances(torch.tensor([0, n], dtype=torch.int64), s, o)
    st = binding.settings_grid([0], ["GBA", "GSA"], [35_003, 9_001, 300_007])
    par.check_batch(inst, st, want_runs=False, label="many runs per round")
    noise = torch.exp(0.5 * torch.randn(n, generator=g, dtype=torch.float64))
    inst.o_est = torch.clamp(torch.round(o.to(torch.float64) * noise), 1, 400).to(torch.int32)
    par.check_batch(inst, binding.settings_grid([0], ["GBA", "GSA"], [35_003]), want_runs=False, label="many runs per round, estimates")


def test_empty_and_degenerate(par):
    off = torch.tensor([0, 0, 1, 1, 4], dtype=torch.int64)
    inst = workloads.Instances(off, torch.tensor([5, 0, 0, 0], dtype=torch.int32), torch.tensor([3, 1, 1, 1], dtype=torch.int32))
    rows = [dict(instance=i, family=f, M=20) for i in range(4) for f in ("GBA", "GSA", "SPS", "SIMS")]
    rows += [dict(instance=3, family="GBA", M=1), dict(instance=1, family="GSA", M=8), dict(instance=1, family="GSA", M=7)]
    par.check_batch(inst, binding.make_settings(rows), label="degenerate")


def test_status_reports(par):
    dev = torch.device("cuda:0")
    off = torch.tensor([0, 3, 6, 9], dtype=torch.int64)
    s = torch.tensor([1, 2, 3, 1, 2, 3, 1, -2, 3], dtype=torch.int32)
    o = torch.tensor([4, 90, 6, 4, 0, 6, 4, 5, 6], dtype=torch.int32)
    inst = workloads.Instances(off, s, o).to(dev)
    st = binding.make_settings([dict(instance=0, family="GBA", M=50), dict(instance=1, family="GBA", M=50),
                                dict(instance=2, family="GSA", M=50), dict(instance=0, family="GBA", M=200)])
    res = par.scheduler().evaluate(inst, st, want_profile=True)
    status = res.status.cpu().tolist()
    assert status[0] == binding.EVAL_INFEASIBLE          # o = 90 > M - s_bar
    assert status[1] == binding.EVAL_BAD_INPUT           # o = 0
    assert status[2] == binding.EVAL_BAD_INPUT           # s < 0
    assert status[3] == 0 and res.feasible.cpu().tolist() == [0, 0, 0, 1]
    # capacity: a profile shorter than the horizon is clipped and flagged, scalars stay exact
    full = par.scheduler().evaluate(inst, st[3:], want_profile=True)
    cap = torch.tensor([5], dtype=torch.int64, device=dev)
    clip = par.scheduler().evaluate(inst, st[3:], want_profile=True, profile_capacity=cap)
    assert clip.status.cpu().tolist() == [binding.EVAL_CAPACITY]
    assert torch.equal(clip.profile, full.profile[:5]) and torch.equal(clip.peak, full.peak)
    # argument errors are found on the host, before any launch
    with pytest.raises(binding.KvsError):
        par.scheduler().evaluate(inst, binding.make_settings([dict(instance=5, family="GBA", M=50)]))
    with pytest.raises(binding.KvsError):
        par.scheduler().evaluate(inst, binding.make_settings([dict(instance=0, family="GBA", M=50, alpha=(2, 2))]))
    with pytest.raises(binding.KvsError):
        par.scheduler().evaluate(inst, binding.make_settings([dict(instance=0, family="GBA", M=1 << 24, alpha=(11, 10))]))
    with pytest.raises(binding.KvsError):
        par.scheduler().evaluate(inst, binding.make_settings([dict(instance=0, family=7, M=50)]))


def test_int64_times(par):
    """Horizon beyond 2^31: 32-bit outputs are flagged, 64-bit outputs are exact."""
    import oracle
    dev = torch.device("cuda:0")
    n = 3000
    inst = workloads.Instances(torch.tensor([0, n], dtype=torch.int64), torch.zeros(n, dtype=torch.int32),
                               torch.full((n,), 1_000_000, dtype=torch.int32))
    st = binding.make_settings([dict(instance=0, family="SPS", M=1_000_000)])      # k* = 1: horizon 3e9
    r32 = par.scheduler().evaluate(inst.to(dev), st)
    assert r32.status.cpu().tolist() == [binding.EVAL_RANGE]
    r64 = par.scheduler().evaluate(inst.to(dev), st, time64=True)
    S = oracle.build_schedule("SPS", inst.s, inst.o, 1_000_000)
    assert r64.status.cpu().tolist() == [0] and int(r64.horizon[0]) == S.horizon == 3_000_000_000
    assert np.array_equal(r64.job_completion.cpu().numpy(), S.job_completion) and int(r64.flow[0]) == S.flow
    assert int(r64.peak[0]) == oracle.evaluate_events(S.run_start, S.run_len, S.run_s).peak


def test_host_entry_point(par):
    """kvs_evaluate_built_host (host buffers in, scalars out, copies pipelined with the kernels over chunks of
    instances) against the oracle, with the evaluations in instance order and in a shuffled order."""
    import oracle
    from paper_2601_22996_b200.api import Scheduler
    cases = [(workloads.config2(n_inst=37, n=1500), 0, ("GBA", "GSA", "SPS", "SIMS")),
             (workloads.config3(n_inst=5, n=6000), None, ("GBA", "GSA"))]
    for inst, window, fams in cases:
        if window is None:
            window = inst.meta["window"]
        I = inst.n_instances
        st = binding.settings_grid(range(I), fams, [inst.meta["M"][len(inst.meta["M"]) // 2]])
        n = int((inst.job_off[1:] - inst.job_off[:-1]).max())
        sched = par.scheduler()
        for order in (np.arange(st.shape[0]), np.random.default_rng(7).permutation(st.shape[0])):
            s2 = np.ascontiguousarray(st[order])
            P = s2.shape[0]
            ctx = sched.context(binding.workspace_bytes(int(inst.s.numel()), I, n, P, host_staging=True))
            hev = {k: torch.full_like(v, -5, device="cpu").pin_memory() for k, v in Scheduler.scalars(P, "cpu").items()}
            hin = workloads.Instances(inst.job_off, inst.s.pin_memory(), inst.o.pin_memory(),
                                      None if inst.o_est is None else inst.o_est.pin_memory(),
                                      None if inst.arrival is None else inst.arrival.pin_memory())
            ctx.evaluate_built_host(hin, s2, hev, window=window, max_jobs=n)
            for e in range(0, P, max(1, P // 40)):
                S = par.oracle_eval(inst, s2[e], window)
                assert S.status == 0 and int(hev["status"][e]) == 0
                assert (int(hev["flow"][e]), int(hev["horizon"][e]), int(hev["job_steps"][e]), int(hev["n_unfinished"][e])) == \
                       (S.flow, S.horizon, S.job_steps, S.n_unfinished)
                E = oracle.evaluate_dense(S.run_start, S.run_len, S.run_s, want_profile=False)
                assert int(hev["peak"][e]) == E.peak and int(hev["feasible"][e]) == int(E.peak <= int(s2[e]["M"]))


@pytest.mark.parametrize("n", [1, 40, 700, 6000])
@pytest.mark.parametrize("beta0", [0, 1, 300, 9000])
def test_evaluations_shared_between_ctas(par, n, beta0):
    """Few evaluations per call: several CTAs share one, phases of hundreds of tiles are cut in their middle (slices below, at and above
    the tile size, carried and exact-key phases, simultaneous batches)."""
    c = torch.arange(3 * n)
    inst = workloads.Instances(torch.tensor([0, n, 2 * n, 3 * n]), workloads.uniform_int(91, c, 0, 700), workloads.pareto_int(92, c, 40.0, 1.1, 1, 9000))
    rows = [dict(instance=i, family=f, M=m, beta0=beta0) for i, m in enumerate((12_000, 20_000, 300_000)) for f in ("GBA", "GSA")]
    rows += [dict(instance=1, family=f, M=20_000, tau=t, k=k) for f in ("SPS", "SIMS") for t, k in ((9000, 2), (4096, 3), (70, 40))]
    par.check_batch(inst, binding.make_settings(rows), want_runs=False, label=f"shared n={n} beta0={beta0}")


def test_peak_without_profile_small(par):
    """No profile stored: peaks from bounds, run ends and prefix sums instead of walked rounds; offline, by windows and on
    estimates, budgets from one job at a time upwards."""
    inst = workloads.random_small(501, n_inst=120, n_max=64, s_max=30, o_max=90)
    for slack in (0, 60, 4000):
        M = _tight_M(inst, slack)
        par.check_batch(inst, _all_settings(inst, lambda i: M[i]), want_runs=False, want_profile=False, label=f"peak slack {slack}")
        par.check_batch(inst, _all_settings(inst, lambda i: M[i], families=("GBA", "GSA"), alpha=(3, 2)), want_runs=False, want_profile=False, label="peak 3/2")
    inst.arrival = torch.cat([torch.arange(int(c), dtype=torch.int64) * 5 for c in (inst.job_off[1:] - inst.job_off[:-1])])
    par.check_batch(inst, _all_settings(inst, lambda i: M[i]), window=64, want_runs=False, want_profile=False, label="peak windows")
    inst = workloads.random_small(502, n_inst=60, n_max=200, s_max=30, o_max=120, with_est=True)
    M = _tight_M(inst, 200)
    par.check_batch(inst, _all_settings(inst, lambda i: M[i]), want_runs=False, want_profile=False, label="peak estimates")


@pytest.mark.parametrize("copies", [1, 80])           # evaluations shared between CTAs, and one CTA each
@pytest.mark.parametrize("n,o_max", [(1, 5), (255, 300), (257, 4097), (6000, 9000)])
def test_peak_without_profile_sizes(par, copies, n, o_max):
    """Phases of one run to thousands, of fewer rounds than a tile to many tiles, with and without jobs that leave."""
    c = torch.arange(2 * n)
    inst = workloads.Instances(torch.tensor([0, n, 2 * n]), workloads.uniform_int(95, c, 0, 700), workloads.pareto_int(96, c, 40.0, 1.1, 1, o_max))
    rows = [dict(instance=i, family=f, M=m, beta0=b) for i, m in ((0, 11_000), (0, 1 << 20), (1, 1 << 17)) for f in ("GBA", "GSA") for b in (0, 300)]
    par.check_batch(inst, binding.make_settings((rows * copies)[:max(len(rows), 2 * copies)]), want_runs=False, want_profile=False, label=f"peak n={n}")


@pytest.mark.parametrize("n", [1 << 18, (1 << 18) + 1])       # the largest instance that CTAs share, the smallest that they do not
@pytest.mark.parametrize("families", [("GBA",), ("GSA",), ("SPS",), ("SIMS",), ("GBA", "GSA", "SIMS")])
def test_few_evaluations_of_large_instances(par, n, families):
    """Calls of one family, which go to that family's kernel where they are not shared, and of several."""
    inst = workloads.config4(n=n)
    st = binding.settings_grid(range(1), families, [1 << 22])
    st["tau"] = np.where(st["family"] >= binding.SPS, 512, 0)
    for profile in (True, False):
        par.check_batch(inst, st, want_runs=False, want_profile=profile, label=f"n={n} profile={int(profile)}")


@pytest.mark.parametrize("est", [False, True])
def test_host_entry_point_chunks(par, est):
    """Chunks of instances that take turns on the host entry point's pairs of streams: some with every family, some with one
    variant of the kernels only, some too small to be split by family, evaluations left to the general kernel; against the
    device entry point, with a second call behind the first."""
    from paper_2601_22996_b200.api import Scheduler
    inst = workloads.random_small(601, n_inst=900, n_max=90, s_max=30, o_max=200, with_est=est)
    M = _tight_M(inst, 500)
    rows = []
    for i in range(inst.n_instances):
        if i % 100 == 7:
            rows.append(dict(instance=i, family="SPS", M=1 << 30, tau=1 << 27, k=60))      # memory bound of 2^32 or more
        fams = ("GBA", "GSA", "SPS", "SIMS") if i < 400 else (("GSA", "GSA", "GSA") if i < 600 else (("GBA", "SPS", "SIMS") if i < 750 else ("GSA",) if i % 9 == 0 else ()))
        rows += [dict(instance=i, family=f, M=M[i] + 100 * k) for k, f in enumerate(fams)]
    for order in (np.arange(len(rows)), np.random.default_rng(8).permutation(len(rows))):
        st = np.ascontiguousarray(binding.make_settings(rows)[order])
        P, I, n = st.shape[0], inst.n_instances, int((inst.job_off[1:] - inst.job_off[:-1]).max())
        assert P >= 2048
        sched = par.scheduler()
        want = sched.evaluate(inst.to("cuda:0"), st, want_jobs=False)
        ctx = sched.context(binding.workspace_bytes(int(inst.s.numel()), I, n, P, host_staging=True))
        hin = workloads.Instances(inst.job_off, inst.s.pin_memory(), inst.o.pin_memory(), None if inst.o_est is None else inst.o_est.pin_memory())
        hev = [{k: torch.full_like(v, -5, device="cpu").pin_memory() for k, v in Scheduler.scalars(P, "cpu").items()} for _ in range(2)]
        for h in hev:
            ctx.evaluate_built_host(hin, st, h, window=0, max_jobs=n)
        for h in hev:
            for k, v in h.items():
                assert torch.equal(v, getattr(want, k).cpu()), k


@pytest.mark.parametrize("I,growing", [(1000, False), (900, False), (700, True)])
def test_host_entry_point_uneven_chunks(par, I, growing):
    """A chunk that has more evaluations of the light variant than the one before it on its lane, by its size or by its families:
    against the device entry point."""
    from paper_2601_22996_b200.api import Scheduler
    inst = workloads.random_small(602, n_inst=I, n_max=300, s_max=60, o_max=400)
    M = _tight_M(inst, 700)
    rows = []
    for i in range(I):
        fams = ("GSA",) + ("GBA", "SPS") * (1 + 3 * i // I) if growing else ("GBA", "GSA", "SPS", "SIMS")
        rows += [dict(instance=i, family=f, M=M[i] + 50 * k) for k, f in enumerate(fams)]
    st = binding.make_settings(rows)
    P, n = st.shape[0], int((inst.job_off[1:] - inst.job_off[:-1]).max())
    assert P >= 2048
    sched = par.scheduler()
    want = sched.evaluate(inst.to("cuda:0"), st, want_jobs=False)
    ctx = sched.context(binding.workspace_bytes(int(inst.s.numel()), I, n, P, host_staging=True))
    hin = workloads.Instances(inst.job_off, inst.s.pin_memory(), inst.o.pin_memory())
    for _ in range(3):
        hev = {k: torch.full_like(v, -5, device="cpu").pin_memory() for k, v in Scheduler.scalars(P, "cpu").items()}
        ctx.evaluate_built_host(hin, st, hev, window=0, max_jobs=n)
        for k, v in hev.items():
            assert torch.equal(v, getattr(want, k).cpu()), k


def test_capacities_written_by_the_library(par):
    """One horizon tensor, filled by the library's kernels for one batch after the other, as the profile capacity of each."""
    P = 8
    first = par.scheduler().scalars(P, torch.device("cuda:0"))
    for seed in (604, 605):
        inst = workloads.random_small(seed, n_inst=P, n_max=40 * (seed - 603), s_max=20, o_max=60 * (seed - 603)).to("cuda:0")
        st = binding.make_settings([dict(instance=i, family="GSA", M=400) for i in range(P)])
        n = int((inst.job_off[1:] - inst.job_off[:-1]).max())
        ctx = par.scheduler().context(binding.workspace_bytes(int(inst.s.numel()), P, n, P))
        ctx.build_schedule(inst, st, dict(n_runs=torch.zeros(P, dtype=torch.int64, device="cuda:0")), first, max_jobs=n)
        res = par.scheduler().evaluate(inst, st, want_profile=True, profile_capacity=first["horizon"])
        assert res.status.tolist() == [0] * P and torch.equal(res.horizon, first["horizon"])
        assert torch.equal(res.profile_off[1:] - res.profile_off[:-1], first["horizon"]) and int(res.profile.min()) >= 0
        runs = dict(run_off=torch.arange(P + 1, device="cuda:0"), run_start=torch.zeros(P, dtype=torch.int64, device="cuda:0"),
                    run_len=first["horizon"].to(torch.int32), run_s=torch.ones(P, dtype=torch.int32, device="cuda:0"))
        res = par.scheduler().evaluate_runs(**runs, capacity=first["horizon"])
        assert res.status.tolist() == [0] * P and torch.equal(res.peak, first["horizon"] + 1)


def test_capacities_of_the_wrong_shape_are_refused(par):
    inst = workloads.random_small(606, n_inst=2, n_max=20, s_max=9, o_max=20).to("cuda:0")
    st = binding.make_settings([dict(instance=i, family="GSA", M=400) for i in range(2)])
    one = torch.tensor([64], device="cuda:0")
    for want_jobs in (False, True):
        with pytest.raises(binding.KvsError):
            par.scheduler().evaluate(inst, st, want_jobs=want_jobs, want_profile=True, profile_capacity=one)
    i32 = dict(dtype=torch.int32, device="cuda:0")
    runs = dict(run_off=torch.arange(3, device="cuda:0"), run_start=torch.zeros(2, dtype=torch.int64, device="cuda:0"),
                run_len=torch.ones(2, **i32), run_s=torch.ones(2, **i32))
    with pytest.raises(binding.KvsError):
        par.scheduler().evaluate_runs(**runs, capacity=one)
    assert par.scheduler().evaluate_runs(**runs, capacity=torch.tensor([4, 4])).peak.tolist() == [2, 2]      # sizes may be host values


def test_calls_under_another_stream(par):
    """A scheduler made under one stream and called under another that is still busy making the inputs: results as on its own."""
    from paper_2601_22996_b200.api import Scheduler
    sched, other = Scheduler(), torch.cuda.Stream()
    inst = workloads.random_small(607, n_inst=12, n_max=200, s_max=30, o_max=200)
    st = _all_settings(inst, lambda i: 900)
    P = st.shape[0]

    def calls(inst, wait):
        wait()
        cap = torch.full((P,), 4096, dtype=torch.int64, device="cuda:0")
        yield vars(sched.evaluate(inst, st))
        wait()
        yield vars(sched.evaluate(inst, st, want_profile=True, profile_capacity=cap))
        wait()
        yield vars(sched.evaluate(inst, st, want_profile=True, want_runs=True))
        start = inst.o.to(torch.int64)
        wait()
        yield vars(sched.evaluate_runs(inst.job_off, start, inst.o, inst.s, cap[:inst.n_instances]))
        yield sched.bounds(inst, st[st["family"] == binding.GBA])
        yield sched.sweep_beta0(inst, 1, "GSA", 900, [0, 3, 16])
        yield sched.sweep(inst, 1, "SPS", 900, [2, 16], [1, 8])

    def flat(results):
        return [{k: v.cpu() for k, v in r.items() if isinstance(v, torch.Tensor)} for r in results]

    want = flat(calls(inst.to("cuda:0"), lambda: None))
    with torch.cuda.stream(other):
        got = flat(calls(inst.to("cuda:0"), lambda: torch.cuda._sleep(10_000_000)))
    for a, b in zip(want, got, strict=True):
        assert a.keys() == b.keys()
        for k in a:
            assert torch.equal(a[k], b[k]), k


@pytest.mark.parametrize("family", ["GBAD", "GSAS"])
def test_host_entry_point_refuses_before_it_launches(par, family):
    """A batch with one setting that the host entry point does not take is refused whole; the call right behind it is right."""
    from paper_2601_22996_b200.api import Scheduler
    inst = workloads.random_small(603, n_inst=520, n_max=60, s_max=30, o_max=90)
    M = _tight_M(inst, 300)
    st = _all_settings(inst, lambda i: M[i])
    bad = st.copy()
    bad["family"][-1] = binding.FAMILY[family]
    P, I, n = st.shape[0], inst.n_instances, int((inst.job_off[1:] - inst.job_off[:-1]).max())
    sched = par.scheduler()
    want = sched.evaluate(inst.to("cuda:0"), st, want_jobs=False)
    ctx = sched.context(binding.workspace_bytes(int(inst.s.numel()), I, n, P, host_staging=True))
    hin = workloads.Instances(inst.job_off, inst.s.pin_memory(), inst.o.pin_memory())
    hev = {k: torch.full_like(v, -5, device="cpu").pin_memory() for k, v in Scheduler.scalars(P, "cpu").items()}
    with pytest.raises(binding.KvsError, match="host entry point takes neither"):
        ctx.evaluate_built_host(hin, bad, hev, window=0, max_jobs=n)
    ctx.evaluate_built_host(hin, st, hev, window=0, max_jobs=n)
    for k, v in hev.items():
        assert torch.equal(v, getattr(want, k).cpu()), k


@pytest.mark.parametrize("copies,runs", [(1, False), (80, False), (1, True)])      # shared evaluations, one CTA each, general kernel
def test_outputs_of_evaluations_that_form_none(par, copies, runs):
    """Per-job results of an infeasible evaluation and rounds behind the end of a schedule take the values that the caller sets;
    a block of per-job results smaller than its instance is reported and left alone."""
    inst = workloads.Instances(torch.tensor([0, 3]), torch.tensor([2, 3, 4], dtype=torch.int32), torch.tensor([5, 6, 7], dtype=torch.int32)).to("cuda:0")
    st = binding.make_settings([dict(instance=0, family="GSA", M=10), dict(instance=0, family="GBA", M=50)] * copies)
    res = par.scheduler().evaluate(inst, st, want_jobs=True, want_profile=True, want_runs=runs)
    assert res.status[:2].tolist() == [binding.EVAL_INFEASIBLE, 0] and res.job_start[:3].tolist() == [-2, -2, -2] and int(res.job_start[3:6].min()) >= 0
    P = 2 * copies
    ctx = par.scheduler().context(binding.workspace_bytes(3, 1, 3, P))
    off = torch.arange(P + 1, dtype=torch.int64, device="cuda:0") * 3
    off[-1] -= 1
    out = dict(job_out_off=off, job_start=torch.full((3 * P,), 77, dtype=torch.int32, device="cuda:0"))
    if runs:
        out |= dict(run_off=torch.arange(P + 1, dtype=torch.int64, device="cuda:0") * 64, run_job=torch.zeros(64 * P, dtype=torch.int32, device="cuda:0"))
    ev = par.scheduler().scalars(P, torch.device("cuda:0"))
    ctx.evaluate_built(inst, st, out, ev, window=0, max_jobs=3)
    torch.cuda.synchronize()
    assert ev["status"].tolist()[-1] == (binding.EVAL_CAPACITY | binding.EVAL_BAD_INPUT) and out["job_start"][-3:].tolist() == [77, 77, 77]


@pytest.mark.parametrize("est", [False, True])
@pytest.mark.parametrize("W", [50, 700, 20_000])
def test_windows_of_shared_evaluations(par, est, W):
    """Few evaluations with windows: small windows go to one of the CTAs that share an evaluation, large ones to all of them, and
    idle rounds lie between some of them."""
    c = torch.arange(3000)
    o = workloads.pareto_int(99, c, 20.0, 1.1, 1, 900)
    arr = torch.sort(torch.cat([torch.randint(0, 9000, (1400,), generator=torch.Generator().manual_seed(W)), torch.full((1100,), 12_345), torch.arange(500) * 40 + 30_000])).values
    inst = workloads.Instances(torch.tensor([0, 3000]), workloads.uniform_int(98, c, 0, 90), o, torch.clamp((o * 5) // 4 - c.to(torch.int32) % 7, min=1) if est else None, arr)
    rows = [dict(instance=0, family=f, M=m) for f in ("GBA", "GSA", "SPS", "SIMS") for m in (1500, 40_000)]
    for prof in (True, False):
        par.check_batch(inst, binding.make_settings(rows), window=W, want_runs=False, want_profile=prof, label=f"shared windows {W}")


@pytest.mark.parametrize("n, o_max", [(31, 5), (33, 300), (2_047, 200), (2_049, 70_000), (4_096, 255), (4_097, 256), (65_536, 900), (65_537, 900)])
def test_order_at_the_edges_of_tiles(par, n, o_max):
    """One to three digits, rows and tiles that are full, one more and one less, 16-bit indices and beyond; two instances that
    do not start at a multiple of anything."""
    c = torch.arange(n)
    one = lambda k: (workloads.uniform_int(8100 + k, c, 0, 90), workloads.pareto_int(8200 + k, c, 2.0, 0.8, 1, o_max))
    (s0, o0), (s1, o1) = one(0), one(1)
    inst = workloads.Instances(torch.tensor([0, 7, 7 + n, 7 + 2 * n]), torch.cat([s0[:1].repeat(7), s0, s1]), torch.cat([o0[:1].repeat(7), o0, o1]))
    M = 4 * (90 + o_max)
    par.check_batch(inst, binding.settings_grid(range(3), ["GBA", "SPS", "SIMS"], [M, 1 << 21]), want_runs=False, want_profile=False, label=f"order n={n} o<={o_max}")


def test_sizes_read_by_the_library(par):
    """Sizes that the library reads itself (int64, on the device) against those that pass through the host: the same outputs, offsets and
    refusals, per-job results of 32 and 64 bits, with and without them, also under another stream and on a fresh workspace."""
    from paper_2601_22996_b200.api import Scheduler
    inst = workloads.random_small(8300, 40, 90, 30, 60).to("cuda:0")
    st = binding.settings_grid(range(40), ["GBA", "GSA", "SPS"], [400, 3_000])
    P = st.shape[0]
    cap = torch.full((P,), 1 << 14, dtype=torch.int64, device="cuda:0")
    cap[::5] = 0
    sch, by_host = Scheduler(), Scheduler()
    by_host._readable = lambda *tensors: False
    for jobs in (True, False):
        for wide in (False, True) if jobs else (False,):
            for c in (cap, None):
                kw = dict(want_jobs=jobs, time64=wide, want_profile=c is not None)
                a = sch.evaluate(inst, st, profile_capacity=c, **kw)
                b = by_host.evaluate(inst, st, profile_capacity=c, **kw)
                side = torch.cuda.Stream()
                with torch.cuda.stream(side):
                    d = sch.evaluate(inst, st, profile_capacity=c, **kw)
                side.synchronize()
                for x in (b, d):
                    for f, v in vars(a).items():
                        w = getattr(x, f)
                        assert (v is None) == (w is None), f
                        assert v is None or torch.equal(v, w), (f, kw)
    bad = st.copy()
    bad["instance"][7] = 40
    for c in (cap, None):
        with pytest.raises(binding.KvsError):
            sch.evaluate(inst, bad, want_profile=c is not None, profile_capacity=c)
    with pytest.raises(binding.KvsError):
        sch.evaluate(inst, st, want_profile=True, profile_capacity=cap[:-1])
    assert torch.equal(sch.evaluate(inst, st).flow, par.scheduler().evaluate(inst, st, want_jobs=False).flow)


def test_negative_sizes(par):
    """A negative capacity is refused before any launch, on both ways that sizes take; an instance whose offsets decrease is bad input with no
    job results, those behind it are as they are by themselves."""
    one = workloads.random_small(8400, 3, 50, 30, 60)
    inst, st = one.to("cuda:0"), binding.settings_grid(range(3), ["GBA", "GSA"], [3_000])
    for kind in (torch.int64, torch.int32):
        for at in (0, 5):
            cap = torch.full((6,), 1 << 12, dtype=kind, device="cuda:0")
            cap[at] = -1
            with pytest.raises(binding.KvsError):
                par.scheduler().evaluate(inst, st, want_profile=True, profile_capacity=cap)
    off = one.job_off
    falling = workloads.Instances(torch.stack([off[1], off[0], off[1], off[3]]).to("cuda:0"), inst.s, inst.o)
    apart = workloads.Instances(torch.stack([off[0], off[1], off[3]]).to("cuda:0"), inst.s, inst.o)
    want = par.scheduler().evaluate(apart, binding.settings_grid(range(2), ["GBA", "GSA"], [3_000]))
    for wide in (False, True):
        got = par.scheduler().evaluate(falling, st, time64=wide)
        assert got.status.tolist()[:2] == [binding.EVAL_BAD_INPUT] * 2 and got.job_out_off.tolist()[:3] == [0, 0, 0]
        assert torch.equal(got.job_start, want.job_start.to(got.job_start.dtype)) and torch.equal(got.job_completion, want.job_completion.to(got.job_start.dtype))
        assert torch.equal(got.flow[2:], want.flow)

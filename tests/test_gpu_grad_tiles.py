"""Tile shapes of the gradient product E X^T: which one runs, and how many bin splits it may have."""
import numpy as np
import pytest
import torch

from torch.profiler import ProfilerActivity, profile

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def glm():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1502_04993_gb300 as g
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    with profile(activities=[ProfilerActivity.CUDA]):  # a process's first profile may miss its kernels
        torch.zeros(3, device="cuda").sum().item()
    return g


def evaluate(c, Wd, bd):
    """An evaluation and the row tile of its gradient product: 1 (256 rows) or 2 (128)."""
    with profile(activities=[ProfilerActivity.CUDA]) as p:
        r = c.loglik_grad(Wd, bd)
        torch.cuda.synchronize()
    tiles = [e.key.split("tc_gemm_kernel<")[1][0] for e in p.key_averages() if "tc_gemm_kernel<" in e.key]
    tiles = [int(t) for t in tiles if t in "12"]
    assert len(tiles) == 1, [e.key for e in p.key_averages()]
    return r, tiles[0]


def workload(n, T, seed):
    w = synth.make_workload(None, n=n, n_exc=max(1, int(0.8 * n)), p=0.1, w_exc=0.3, w_inh=1.2, w_self=-3.0,
                            rate=8.0, tau=0.010, dt=0.001, n_bins=T, seed=seed)
    rng = np.random.default_rng(seed + 100)
    W = (w["W_true"] + rng.normal(0, 0.05, (n, n))).astype(np.float32)
    b = (w["b_true"] + rng.normal(0, 0.1, n)).astype(np.float32)
    return w, W, b


def splits(n, ksteps, units_per_sm):
    """Splits of 256-row tiles for that many units per SM, none of them empty; for 8 the most there are."""
    tiles = (-(-n // 256)) ** 2
    s = -(-units_per_sm * torch.cuda.get_device_properties(0).multi_processor_count // tiles)
    s = max(1, min(s, ksteps))
    return -(-ksteps // -(-ksteps // s))


def test_tuned_splits_stay_within_the_partials(glm):
    """The autotuner's choice for a stored recording is not taken for the same recording in chunks, whose shorter
    products have fewer splits at most, and so fewer planes of partial sums.  G of the two forms differs by the FP32
    accumulation of its partial sums only: at most 11 k-steps of 64 bins to a split, four instructions each, and 2^-23 of
    the sum lost by each, in both forms: 1.05e-5 of the terms."""
    n, T, chunk = 100, 100_000, 81_920
    w, W, b = workload(n, T, 1)
    Wd, bd = torch.from_numpy(W).cuda(), torch.from_numpy(b).cuda()
    with glm.GLM(0) as a, glm.GLM(0) as c, glm.GLM(0) as d:
        a.set_problem(w["offs"], w["bins"], T, w["dt"], w["tau"], prec="f16")
        assert a.autotune()["nsplit"] <= splits(n, -(-T // 64), 8)
        ra = a.loglik_grad(Wd, bd)
        C = a.spike_term()[0]
        for k, x in enumerate((c, d)):
            x.set_chunk_bins(chunk)
            x.set_problem(w["offs"], w["bins"], T, w["dt"], w["tau"], prec="f16")
            t = x.autotune()
            assert t["cached"] == k and t["nsplit"] <= splits(n, chunk // 64, 8)
            r = x.loglik_grad(Wd, bd)
            assert torch.all((r["G"] - ra["G"]).abs() <= 1.05e-5 * (C + (C - ra["G"])) + 1e-9)


@pytest.mark.parametrize("n,T", [(300, 70_000), (130, 12_000)])
def test_the_row_tile_asked_for_runs(glm, n, T):
    """Mode 1 runs 256-row tiles and mode 2 128-row tiles, set by hand or picked by the autotuner; by default, where 256
    rows would be wasteful, 128-row tiles form the sums of mode 1, bit for bit."""
    w, W, b = workload(n, T, n)
    Wd, bd = torch.from_numpy(W).cuda(), torch.from_numpy(b).cuda()
    with glm.GLM(0) as c:
        c.set_x_split(False)
        c.set_problem(w["offs"], w["bins"], T, w["dt"], w["tau"], prec="f16")
        default, tile = evaluate(c, Wd, bd)
        assert tile == 2
        for mode in (1, 2):
            for upm in (1, 2, 4, 8):
                c.set_grad_tile(mode, upm)
                r, tile = evaluate(c, Wd, bd)
                assert tile == mode
                if (mode, upm) == (1, 4):
                    assert torch.equal(r["G"], default["G"])
        t = c.autotune()
        assert t["cached"] == 0 and t["candidates"] == 8
        assert evaluate(c, Wd, bd)[1] == t["mode"]


def units_of_halves(n, T, units_per_sm):
    """Tiles that the last round of 256-row tiles deals out in row halves."""
    units = (-(-n // 256)) ** 2 * splits(n, -(-T // 64), units_per_sm)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return units % sms if units > sms and 2 * (units % sms) <= sms else 0


@pytest.mark.parametrize("form,n,T,upm", [("f16x1", 512, 6_400, 0), ("bf16", 400, 6_000, 0), ("f16x1", 203, 200_000, 0),
                                          ("bf16", 1000, 10_000, 0), ("f16x1", 600, 20_000, 1)])
def test_256_row_tiles_match_oracle(glm, form, n, T, upm):
    """Every element of the gradient formed by 256-row tiles, by default or set by hand (upm units per SM): whole rounds
    (512), and last rounds dealt out in row halves, the second half ragged (400, 203, 1000) or empty (600).  Worst-case
    rounding bounds: with u the half ulp of the 16-bit type and u_x that of X as U reads it, |dU_i| <= (u_x + 3e-5) K_i,
    K_i = max_t sum_j |W_ij| X_j[t], 3e-5 covering the FP32 accumulation (3 x 63 instructions at n = 1000, 2^-23 each);
    E and the X of the gradient are rounded once more each, and their partial sums lose 1e-5 at most."""
    u, ux = (2.0 ** -11, 2.0 ** -11) if form == "f16x1" else (2.0 ** -8, 2.0 ** -16)
    w, W, b = workload(n, T, n)
    ref = oracle.loglik_grad(w["offs"], w["bins"], T, w["dt"], w["tau"], W.astype(np.float64), b.astype(np.float64))
    X = oracle.filter(w["offs"], w["bins"], T, w["dt"], w["tau"])
    assert (units_of_halves(n, T, upm or 4) > 0) == (n != 512)
    with glm.GLM(0) as c:
        c.set_x_split(form != "f16x1")
        c.set_problem(w["offs"], w["bins"], T, w["dt"], w["tau"], prec="f16" if form == "f16x1" else form)
        if upm:
            c.set_grad_tile(1, upm)
        r, tile = evaluate(c, torch.from_numpy(W).cuda(), torch.from_numpy(b).cuda())
    assert tile == 1
    C = np.stack([X[:, w["bins"][w["offs"][i]:w["offs"][i + 1]]].sum(axis=1) for i in range(n)])
    dU = (ux + 3e-5) * (np.abs(W) @ X).max(axis=1)
    bound = (2 * u + dU + 1e-5)[:, None] * (C + (C - ref["G"])) + 1e-9
    assert np.all(np.abs(r["G"].cpu().numpy() - ref["G"]) <= bound)


@pytest.mark.parametrize("form,n,r0,r1,T", [("f16x1", 512, 31, 511, 6_000), ("bf16", 512, 33, 480, 6_000),
                                            ("f16x1", 1000, 5, 1000, 10_000)])
def test_row_range_off_the_blocks_with_256_row_tiles(glm, form, n, r0, r1, T):
    """A range that begins inside a 32-row block, so that a warp's rows lie in two of them, returns the full evaluation's
    rows, bit for bit (at n = 1000 some rates of this network are beyond FP16, and their rows of G are not finite)."""
    w, W, b = workload(n, T, n)
    Wd, bd = torch.from_numpy(W).cuda(), torch.from_numpy(b).cuda()
    with glm.GLM(0) as c:
        c.set_x_split(form != "f16x1")
        c.set_problem(w["offs"], w["bins"], T, w["dt"], w["tau"], prec="f16" if form == "f16x1" else form)
        full, tile = evaluate(c, Wd, bd)
        assert tile == 1
        c.set_row_range(r0, r1)
        part, tile = evaluate(c, Wd, bd)
        assert tile == 1
    for k in ("L_rows", "G", "gb"):
        want = torch.zeros_like(full[k])
        want[r0:r1] = full[k][r0:r1]
        assert torch.equal(part[k].view(torch.int64), want.view(torch.int64)), k


@pytest.mark.parametrize("n,T", [(70, 100_000), (50, 20_000), (203, 30_000)])
def test_a_cap_without_room_for_padded_partials(glm, n, T):
    """A cap that covers every buffer with n x n floats a split for the gradient's partials is enough, although those
    are stored with their columns padded to a multiple of four: there are fewer splits then.  dL/dtau, whose buffers come
    with the first request, has its room as well.  Fewer splits change G by the FP32 accumulation of its partial sums
    only: at most 8 k-steps of 64 bins to a split, four instructions each, and 2^-23 of the sum lost by each, in both
    contexts: 8e-6 of the terms."""
    w, W, b = workload(n, T, n)
    Wd, bd = torch.from_numpy(W).cuda(), torch.from_numpy(b).cuda()
    q, seg = int(w["offs"][-1]), -(-T // 256)
    ns, full = splits(n, -(-T // 64), 4), splits(n, -(-T // 64), 8)
    x = 2 * n * 256 * seg
    need = [8 * (n + 1), 4 * q, 8 * n * seg, 4 * n * seg, 8 * 257, 8 * n, 8 * n * n, x, x, 8 * n * seg,
            4 * n * n * full, 16, 8 * n, 64, 8 * n, 8 * n * seg, 4 * n * (-(-n // 64) * 64)]
    total = sum(-(-v // 256) * 256 for v in need)
    tau = sum(-(-v // 256) * 256 for v in (5 * 8 * n * seg, 8 * n))
    recording = (w["offs"], w["bins"], T, w["dt"], w["tau"], "f16")
    with glm.GLM(0) as a, glm.GLM(0, workspace_cap=total) as c, glm.GLM(0, workspace_cap=total + tau) as d:
        for g in (a, c, d):
            g.set_x_split(False)
            g.set_problem(*recording)
        C = a.spike_term()[0]
        wants = [a.loglik_grad(Wd, bd, tau_grad=t) for t in (False, True)]  # of another kernel each
        with pytest.raises(glm.GLMError) as e:
            c.loglik_grad(Wd, bd, tau_grad=True)
        assert e.value.code == -4
        for g, t in ((c, False), (d, True), (d, False)):
            got, want = g.loglik_grad(Wd, bd, tau_grad=t), wants[t]
            assert torch.equal(got["L_rows"], want["L_rows"]) and torch.equal(got["gb"], want["gb"])
            assert got["gtau"] == want["gtau"]
            if ns <= full * n // (-(-n // 4) * 4):
                assert torch.equal(got["G"], want["G"])
            assert torch.all((got["G"] - want["G"]).abs() <= 8e-6 * (C + (C - want["G"])) + 1e-9)


@pytest.mark.parametrize("n,T", [(2000, 30_000), (3000, 20_000)])
def test_a_row_range_reads_its_own_partials(glm, n, T):
    """The reduction of a range of a few rows reads those rows' partial sums and C only.  Of the bytes of all rows, 4 for
    each element and split and 8 each for C and G, that leaves the zeros of G: less than a third with four splits or
    more, so half the time at most."""
    rng = np.random.default_rng(n)
    rows = [np.flatnonzero(rng.random(T) < 0.008) for _ in range(n)]
    offs = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64)
    W, b = torch.zeros((n, n), device="cuda"), torch.full((n,), 2.0, device="cuda")
    with glm.GLM(0) as c:
        c.set_x_split(False)
        c.set_problem(offs, np.concatenate(rows).astype(np.int32), T, 0.001, 0.010, prec="f16")
        times = []
        for r0, r1 in ((0, 0), (n // 2, n // 2 + 40)):
            c.set_row_range(r0, r1)
            best = np.inf
            for _ in range(10):
                c.profile(True)
                c.loglik_grad(W, b)
                best = min(best, c.profile_read()["reduce"][1])
            times.append(best)
        print(f"n = {n}: reduction {1e3 * times[0]:.1f} us, of 40 rows {1e3 * times[1]:.1f} us")
        assert times[1] <= 0.5 * times[0]

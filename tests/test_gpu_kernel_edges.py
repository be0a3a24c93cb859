"""Sizes at the edges of the kernels' blocks and tiles, against the FP64 oracle.

Tolerances are worst-case rounding bounds, since short recordings do not average the rounding out.  With u the half
ulp of the 16-bit type (2^-11 FP16, 2^-8 BF16) and u_x that of X as U reads it (2^-11 for one FP16 X, 2^-16 for the
split BF16 X; W is split and adds no more than the latter), K_i = max_t sum_j |W_ij| X_j[t] bounds the argument:
|dU_i| <= (u_x + 1e-5) K_i, the 1e-5 covering FP32 accumulation over up to 257 sources.  Then
|dL_i| <= dU_i (q_i + dt sum e^U_i) and, as E and the X of the gradient product are rounded once more each,
|dG_ij| <= (2 u + dU_i) (C_ij + dt sum e^U_i X_j).  The FP32 form has its parity bounds (5e-8 and 1e-5)."""
import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu

U16 = {"f16x1": 2.0 ** -11, "bf16": 2.0 ** -8}   # one rounding to the 16-bit type
U_X = {"f16x1": 2.0 ** -11, "bf16": 2.0 ** -16}  # X as the U product reads it


@pytest.fixture(scope="module")
def glm():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1502_04993_gb300 as g
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    return g


def workload(n, T, seed):
    w = synth.make_workload(None, n=n, n_exc=max(1, int(0.8 * n)), p=0.1, w_exc=0.3, w_inh=1.2, w_self=-3.0,
                            rate=8.0, tau=0.010, dt=0.001, n_bins=T, seed=seed)
    rng = np.random.default_rng(seed + 100)
    W = (w["W_true"] + rng.normal(0, 0.05, (n, n))).astype(np.float32)
    b = (w["b_true"] + rng.normal(0, 0.1, n)).astype(np.float32)
    return w, W, b


def context(glm, w, form):
    c = glm.GLM(0)
    c.set_x_split(form != "f16x1")
    c.set_problem(w["offs"], w["bins"], w["n_bins"], w["dt"], w["tau"], prec="f16" if form == "f16x1" else form)
    return c


def reference(w, W, b):
    return oracle.loglik_grad(w["offs"], w["bins"], w["n_bins"], w["dt"], w["tau"], W.astype(np.float64),
                              b.astype(np.float64))


@pytest.mark.parametrize("form", ["f32", "f16x1", "bf16"])
@pytest.mark.parametrize("n,T", [(1, 300), (3, 257), (31, 4000), (32, 4000), (33, 20001), (65, 3000), (127, 2000),
                                 (129, 2000), (255, 1500), (257, 1500), (130, 70000), (65, 40000)])
def test_evaluation_at_block_edges(glm, form, n, T):
    """n around the 32-row blocks, 4-column groups and 128- and 256-row tiles; one split up to hundreds."""
    w, W, b = workload(n, T, n)
    ref = reference(w, W, b)
    with context(glm, w, form) as c:
        r = c.loglik_grad(torch.from_numpy(W).cuda(), torch.from_numpy(b).cuda())
    q = np.diff(w["offs"]).astype(np.float64)
    X = oracle.filter(w["offs"], w["bins"], T, w["dt"], w["tau"])
    Cx = np.stack([X[:, w["bins"][w["offs"][i]:w["offs"][i + 1]]].sum(axis=1) for i in range(n)])
    if form == "f32":
        row, grad = 5e-8 * (np.abs(ref["L"]) + q), np.full((n, 1), 1e-5)
    else:
        dU = (U_X[form] + 1e-5) * (np.abs(W) @ X).max(axis=1)
        row, grad = dU * (q + (q - ref["gb"])), (2 * U16[form] + dU)[:, None]
    assert np.all(np.abs(r["L_rows"].cpu().numpy() - ref["L"]) <= row + 1e-9)
    assert np.all(np.abs(r["gb"].cpu().numpy() - ref["gb"]) <= row + 1e-9)
    assert r["L_total"] == pytest.approx(float(r["L_rows"].sum()), rel=1e-13)
    assert np.all(np.abs(r["G"].cpu().numpy() - ref["G"]) <= grad * (Cx + (Cx - ref["G"])) + 1e-9)


@pytest.mark.parametrize("form", ["f16x1", "bf16"])
@pytest.mark.parametrize("T", [256, 257, 2687])
def test_spikes_per_tile(glm, form, T):
    """Rows with none, few (one to three register groups of the U epilogue) and more spikes in each 256-bin tile, at
    its edges too; the tolerances of test_evaluation_at_block_edges."""
    counts, rng, rows = [0, 1, 4, 5, 8, 9, 12, 13, 40, 256], np.random.default_rng(T), []
    for k in counts:
        first = np.array([0, 255, 128, 127, 31, 32])[:k]
        tile = np.concatenate([first, rng.permutation(np.setdiff1d(np.arange(256), first))[:max(0, k - 6)]])
        bins = np.sort((np.arange(0, T, 256)[:, None] + tile[None, :]).ravel())
        rows.append(bins[bins < T].astype(np.int32))
    n = len(counts)
    w = dict(offs=np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64), bins=np.concatenate(rows),
             n_bins=T, dt=0.001, tau=0.010)
    W, b = rng.normal(0, 0.05, (n, n)).astype(np.float32), rng.normal(2.0, 0.3, n).astype(np.float32)
    ref, X = reference(w, W, b), oracle.filter(w["offs"], w["bins"], T, w["dt"], w["tau"])
    with context(glm, w, form) as c:
        r = c.loglik_grad(torch.from_numpy(W).cuda(), torch.from_numpy(b).cuda())
    q = np.diff(w["offs"]).astype(np.float64)
    Cx = np.stack([X[:, w["bins"][w["offs"][i]:w["offs"][i + 1]]].sum(axis=1) for i in range(n)])
    dU = (U_X[form] + 1e-5) * (np.abs(W) @ X).max(axis=1)
    assert np.all(np.abs(r["L_rows"].cpu().numpy() - ref["L"]) <= dU * (q + (q - ref["gb"])) + 1e-9)
    assert np.all(np.abs(r["G"].cpu().numpy() - ref["G"]) <=
                  (2 * U16[form] + dU)[:, None] * (Cx + (Cx - ref["G"])) + 1e-9)


@pytest.mark.parametrize("form", ["f16x1", "bf16"])
@pytest.mark.parametrize("n,r0,r1", [(70, 5, 6), (300, 31, 289), (300, 250, 300)])
def test_row_range_off_the_blocks(glm, form, n, r0, r1):
    """A row range that starts and ends inside 32-row blocks returns the full evaluation's rows, bit for bit."""
    w, W, b = workload(n, 6000, n + r0)
    Wd, bd = torch.from_numpy(W).cuda(), torch.from_numpy(b).cuda()
    with context(glm, w, form) as c:
        full = c.loglik_grad(Wd, bd)
        c.set_row_range(r0, r1)
        part = c.loglik_grad(Wd, bd)
    for k in ("L_rows", "G", "gb"):
        want = torch.zeros_like(full[k])
        want[r0:r1] = full[k][r0:r1]
        assert torch.equal(part[k], want), k


@pytest.mark.parametrize("dtype,u", [("f32", 2.0 ** -24), ("bf16", 2.0 ** -8), ("f16", 2.0 ** -11)])
@pytest.mark.parametrize("t0,length", [(0, 1), (0, 20_000), (255, 2), (1_023, 4_098), (4_096, 256), (12_345, 7_655)])
def test_filter_ranges(glm, dtype, u, t0, length):
    """Any range into a buffer of odd stride, for silent, sparse, bursty (8 and 9 spikes per 256 bins are the two
    sides of the kernel's rule) and saturated trains.  X is rounded once from a double-float value, and once more to a
    16-bit type: half an ulp of the type (half the spacing of subnormal FP16) and 0.1 % for the first rounding's ties.
    Below 2^-100 (69 time constants after the last spike) the pair loses its low part: there X only has to be as
    small."""
    T, rng = 20_000, np.random.default_rng(5)
    seg = np.arange(0, T, 256)
    rows = [np.zeros(0, dtype=np.int64), np.flatnonzero(rng.random(T) < 0.008), np.flatnonzero(rng.random(T) < 0.2),
            np.arange(T), np.concatenate([s + np.arange(8) * 29 for s in seg]),
            np.concatenate([s + np.arange(9) * 28 for s in seg]), np.array([0, 7, 8, 255, 256, T - 1])]
    rows = [r[r < T] for r in rows]
    offs = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64)
    bins = np.concatenate(rows).astype(np.int32)
    Xo = oracle.filter(offs, bins, T, 0.001, 0.010)[:, t0:t0 + length]
    tdt = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}[dtype]
    wide = torch.full((len(rows), length + 3), -7.0, dtype=tdt, device="cuda")
    with glm.GLM(0) as c:
        c.set_problem(offs, bins, T, 0.001, 0.010, prec="f32")
        c.filter(t0, length, dtype, out=wide[:, 1:1 + length])
    got = wide.double().cpu().numpy()
    assert np.all(got[:, 0] == -7.0) and np.all(got[:, 1 + length:] == -7.0)
    x, sub = got[:, 1:1 + length], {"f32": 0.0, "bf16": 0.0, "f16": 2.0 ** -25}[dtype]
    assert np.all(np.where(Xo >= 2.0 ** -100, np.abs(x - Xo) <= 1.001 * np.maximum(u * Xo, sub), x < 2.0 ** -99))


@pytest.mark.parametrize("form", ["f32", "f16x1", "bf16"])
def test_windows_of_one_recording(glm, form):
    """Recordings of the same neurons and bins with other spikes, more and fewer of them and none, set one after the
    other on one context: the results of fresh contexts, bit for bit; a bad recording leaves the current one; and a fit
    may choose its L-BFGS memory for each."""
    n, T = 70, 6000
    w, W, b = workload(n, T, 9)
    Wd, bd = torch.from_numpy(W).cuda(), torch.from_numpy(b).cuda()
    rng, wins = np.random.default_rng(3), []
    for p in (0.008, 0.03, 0.002, 0.0, 0.03):
        rows = [np.flatnonzero(rng.random(T) < p) for _ in range(n)]
        wins.append((np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64),
                     np.concatenate(rows).astype(np.int32)))
    with context(glm, w, form) as c:
        prec = "f16" if form == "f16x1" else form
        for k, (offs, bins) in enumerate(wins):
            c.set_problem(offs, bins, T, 0.001, 0.010, prec=prec)
            got = c.loglik_grad(Wd, bd)
            with context(glm, dict(w, offs=offs, bins=bins), form) as f:
                want = f.loglik_grad(Wd, bd)
            assert got["L_total"] == want["L_total"]
            assert all(torch.equal(got[x], want[x]) for x in ("L_rows", "G", "gb"))
            if len(bins):
                bad = bins.copy()
                bad[len(bad) // 2] = T
                with pytest.raises(glm.GLMError) as e:
                    c.set_problem(np.append(offs[:-1], offs[-1] - 1), bad[:-1], T, 0.001, 0.010, prec=prec)
                assert e.value.code == -3
                assert torch.equal(c.loglik_grad(Wd, bd)["G"], want["G"])
                c.fit(max_iter=2, m=5 + k)


@pytest.mark.parametrize("form", ["f32", "f16x1"])
def test_row_ranges_over_many_windows(glm, form):
    """A row range set anew for each of many recordings that share a context's buffers, and many ranges on one of them:
    the context takes no more memory for each, and every evaluation returns the full one's rows, bit for bit."""
    n, T, rng = 40, 2000, np.random.default_rng(8)
    w, W, b = workload(n, T, 11)
    Wd, bd = torch.from_numpy(W).cuda(), torch.from_numpy(b).cuda()

    def check(full, part, r0, r1):
        for k in ("L_rows", "G", "gb"):
            want = torch.zeros_like(full[k])
            want[r0:r1] = full[k][r0:r1]
            assert torch.equal(part[k], want), k

    with context(glm, w, form) as c, context(glm, w, form) as f:
        prec = "f16" if form == "f16x1" else form
        for k in range(160):
            if k < 80:
                rows = [np.flatnonzero(rng.random(T) < 0.01) for _ in range(n)]
                rec = (np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64),
                       np.concatenate(rows).astype(np.int32), T, 0.001, 0.010, prec)
                c.set_problem(*rec)
                f.set_problem(*rec)
                full = f.loglik_grad(Wd, bd)
            r0 = k % (n - 1)
            r1 = min(n, r0 + 1 + k % 13)
            c.set_row_range(r0, r1)
            check(full, c.loglik_grad(Wd, bd), r0, r1)


@pytest.mark.parametrize("form", ["f32", "f16x1"])
def test_row_range_and_the_next_problem(glm, form):
    """A row range stays for a problem that has its rows; a problem with fewer neurons has all its rows evaluated and
    fitted."""
    prec = "f16" if form == "f16x1" else form
    with context(glm, workload(90, 2000, 1)[0], form) as c:
        c.set_row_range(50, 80)
        for n, r0, r1 in ((80, 50, 80), (120, 50, 80), (79, 0, 79), (120, 0, 120)):
            w, W, b = workload(n, 2000, n)
            Wd, bd = torch.from_numpy(W).cuda(), torch.from_numpy(b).cuda()
            c.set_problem(w["offs"], w["bins"], w["n_bins"], w["dt"], w["tau"], prec=prec)
            part = c.loglik_grad(Wd, bd)
            with context(glm, w, form) as f:
                full = f.loglik_grad(Wd, bd)
            for k in ("L_rows", "G", "gb"):
                want = torch.zeros_like(full[k])
                want[r0:r1] = full[k][r0:r1]
                assert torch.equal(part[k], want), k
            assert c.fit(max_iter=1)["report"]["excluded"] == n - (r1 - r0)


def test_another_recording_with_as_many_spikes(glm):
    """A recording of the same size with other spikes, but as many, is another problem all the same: a tile set by hand
    for the one before it is gone, and a fit may choose its L-BFGS memory (which stays refused within a problem)."""
    n, T = 70, 20_000
    w, W, b = workload(n, T, 9)
    Wd, bd = torch.from_numpy(W).cuda(), torch.from_numpy(b).cuda()
    offs, bins = w["offs"], (T - 1 - w["bins"]).astype(np.int32)
    for i in range(n):
        bins[offs[i]:offs[i + 1]].sort()
    v = dict(w, bins=bins)
    with context(glm, w, "f16x1") as c, context(glm, v, "f16x1") as f:
        c.set_grad_tile(2, 1)
        c.fit(max_iter=3, m=5)
        with pytest.raises(glm.GLMError) as e:
            c.fit(max_iter=3, m=6)
        assert e.value.code == -10
        c.set_problem(offs, bins, T, w["dt"], w["tau"], prec="f16")
        assert torch.equal(c.loglik_grad(Wd, bd)["G"], f.loglik_grad(Wd, bd)["G"])
        got, want = c.fit(max_iter=3, m=6), f.fit(max_iter=3, m=6)
        assert torch.equal(got["W"], want["W"]) and torch.equal(got["b"], want["b"])
        with pytest.raises(glm.GLMError) as e:
            c.fit(max_iter=3, m=5)
        assert e.value.code == -10

"""Kernels and dispatch rules at the sizes where they can go wrong: run lengths around the limits of the SpMM work lists, column
slices, row splits and tiles of the weight gradient, class counts of the losses.  References are computed in fp64; a sum of k fp32
terms t_i in any order is within k 2^-24 sum |t_i| of the exact one (u = 2^-24; one rounding per product and per addition), and the
TF32 contractions add at most 2^-20 of the same sum (two-term split, truncating accumulation)."""
import numpy as np
import pytest
import scipy.sparse as sp
import torch

from tests.gpu_util import dev, dev2d, empty2d

pytestmark = pytest.mark.gpu

U = 2.0 ** -24


@pytest.fixture(scope="module")
def B():
    import paper_2308_13466_b200.binding as binding
    return binding


def _graph(hubs, n):
    """Node i < len(hubs) is next to hubs[i] others (evenly spread); a ring keeps every node connected."""
    pairs = {(i, (i + 1) % n) for i in range(n)}
    for i, deg in enumerate(hubs):
        pairs |= {(i, int(j)) for j in np.linspace(0, n - 1, deg).astype(int) if j != i}
    a = np.array([(min(p), max(p)) for p in pairs if p[0] != p[1]])
    m = sp.coo_matrix((np.ones(len(a)), (a[:, 0], a[:, 1])), shape=(n, n))
    m = ((m + m.T) > 0).astype(np.float64).tocsr()
    m.sort_indices()
    return m


def _propagation(A):
    dinv = 1.0 / np.sqrt(np.asarray(A.sum(1)).ravel() + 1.0)
    return sp.diags(dinv) @ (A + sp.identity(A.shape[0])) @ sp.diags(dinv)


# degrees around the run lengths (32; 48 in a list with the longest of these rows) and far above: up to 61 runs, which the last one adds
HUBS = [29, 30, 31, 32, 33, 62, 64, 100, 500, 510, 520, 1000, 2900]


@pytest.mark.parametrize("d", [4, 5, 12, 31, 33, 64, 65, 100, 128, 129, 256, 260, 300, 512, 602])
def test_aggregation_and_its_transpose(B, d):
    n, M = 3000, 3
    A = _graph(HUBS, n)
    P = _propagation(A)
    rng = np.random.default_rng(d)
    X = rng.standard_normal((n, d)).astype(np.float32)
    part = rng.integers(0, M, n).astype(np.int32)
    ctx = B.sat_create(0, 0)
    try:
        B.sat_graph_load(ctx, A.indptr.astype(np.int64), A.indices.astype(np.int32))
        B.sat_partition(ctx, M, B.SAT_PART_GIVEN, part)
        perm = np.concatenate([np.flatnonzero(part == m) for m in range(M)])
        off = np.concatenate([[0], np.cumsum(np.bincount(part, minlength=M))])
        eye = dev(np.eye(d, 4, dtype=np.float32))            # four output columns on the CUDA cores: the aggregation itself, columns 0-3
        out = empty2d(n, 4)
        B.sat_layer_fwd(ctx, B.SAT_ALL_PARTS, 1, dev2d(X), None, eye, None, B.SAT_ACT_NONE | B.SAT_FWD_INPUT_GLOBAL, out)
        want, mag = P @ X.astype(np.float64), abs(P) @ np.abs(X.astype(np.float64))
        terms = np.diff(A.indptr).max() + 8
        err = np.abs(out.cpu().numpy() - want[perm][:, :4])
        assert (err <= terms * U * mag[perm][:, :4]).all()
        # every column through the weight gradient with one-hot gradients: G_W = AGG^T D picks rows of AGG
        rows = rng.choice(n, 3, replace=False)
        D = np.zeros((n, 3), np.float32)
        D[rows, np.arange(3)] = 1.0
        W3 = dev(np.zeros((d, 3), np.float32))
        B.sat_layer_fwd(ctx, B.SAT_ALL_PARTS, 1, dev2d(X), None, W3, None, B.SAT_ACT_NONE | B.SAT_FWD_INPUT_GLOBAL, empty2d(n, 3))
        gW, gb = torch.full((d, 3), float("nan"), device="cuda"), torch.full((3,), float("nan"), device="cuda")
        B.sat_layer_bwd(ctx, B.SAT_ALL_PARTS, 1, dev2d(D), W3, gW, gb, 0, None, None)
        assert (np.abs(gW.cpu().numpy().T - want[perm[rows]]) <= terms * U * mag[perm[rows]]).all()
        assert (gb.cpu().numpy() == 1.0).all()
        # G_in of a layer with W = first rows of the identity: P_in^T D; all partitions at once = one after the other
        k = min(d, 4)
        Wi = dev(np.eye(d, k, dtype=np.float32))
        G = rng.standard_normal((n, k)).astype(np.float32)
        h_in = dev2d(X[perm])
        n_halo = B.sat_part_sizes(ctx, B.SAT_ALL_PARTS)[1]
        halo = dev2d(np.zeros((n_halo, d), np.float32))
        B.sat_layer_fwd(ctx, B.SAT_ALL_PARTS, 2, h_in, halo, Wi, None, B.SAT_ACT_NONE, empty2d(n, k))
        gW2, g_in, g_halo = torch.empty((d, k), device="cuda"), empty2d(n, d), empty2d(n_halo, d)
        B.sat_layer_bwd(ctx, B.SAT_ALL_PARTS, 2, dev2d(G), Wi, gW2, None, 0, g_in, g_halo)
        same = sp.csr_matrix((P.tocoo().data * (part[P.tocoo().row] == part[P.tocoo().col]), (P.tocoo().row, P.tocoo().col)), shape=P.shape)
        Gn = np.zeros((n, k))
        Gn[perm] = G
        want_in, mag_in = same @ Gn, abs(same) @ np.abs(Gn)
        assert (np.abs(g_in.cpu().numpy()[:, :k] - want_in[perm]) <= terms * U * mag_in[perm]).all()
        one = empty2d(n, d)
        for m in range(M):
            r = slice(off[m], off[m + 1])
            B.sat_layer_bwd(ctx, m, 2, dev2d(G[r]), Wi, gW2, None, 0, one[r], None)
        assert torch.equal(one[:, :k], g_in[:, :k])
        lists = [B.sat_part_lists(ctx, m) for m in range(M)]
        gh, h0 = g_halo.cpu().numpy()[:, :k], 0
        for m in range(M):
            ids, inner = lists[m]["halo_gid"], perm[off[m]:off[m + 1]]
            sub = P.tocsr()[ids][:, inner]
            assert (np.abs(gh[h0:h0 + len(ids)] - sub @ Gn[inner]) <= terms * U * (abs(sub) @ np.abs(Gn[inner]))).all()
            h0 += len(ids)
        B.sat_sync_status(ctx)
    finally:
        B.sat_destroy(ctx)


@pytest.mark.parametrize("given", [False, True])
def test_historical_rows_read_from_the_ring(B, given):
    """SAT_FWD_HALO_CACHED against the pull through sat_predict: same bits once there is a snapshot, and zeros before."""
    n, M, d, d2 = 1500, 4, 40, 24
    A = _graph(HUBS[:9], n)
    rng = np.random.default_rng(2)
    part = rng.integers(0, M, n).astype(np.int32) if given else None
    ctx = B.sat_create(0, 0)
    try:
        B.sat_graph_load(ctx, A.indptr.astype(np.int64), A.indices.astype(np.int32))
        B.sat_partition(ctx, M, B.SAT_PART_GIVEN if given else B.SAT_PART_CONTIG_BLOCKS, part)
        B.sat_cache_init(ctx, [d], 2)
        sizes = [B.sat_part_sizes(ctx, m) for m in range(M)]
        H, W = dev2d(rng.standard_normal((n, d)).astype(np.float32)), dev(rng.standard_normal((d, d2)).astype(np.float32))
        for epoch in range(3):
            halo = empty2d(sum(s[1] for s in sizes), d)
            B.sat_predict(ctx, 1, B.SAT_ALL_PARTS, None, 0, halo)
            a, b, c = empty2d(n, d2), empty2d(n, d2), empty2d(n, d2)
            B.sat_layer_fwd(ctx, B.SAT_ALL_PARTS, 2, H, halo, W, None, B.SAT_ACT_NONE, a)
            B.sat_layer_fwd(ctx, B.SAT_ALL_PARTS, 2, H, None, W, None, B.SAT_ACT_NONE | B.SAT_FWD_HALO_CACHED, b)
            r0 = 0
            for m in range(M):
                r1 = r0 + sizes[m][0]
                B.sat_layer_fwd(ctx, m, 2, H[r0:r1], None, W, None, B.SAT_ACT_NONE | B.SAT_FWD_HALO_CACHED, c[r0:r1])
                r0 = r1
            assert torch.equal(b, c)
            assert torch.equal(a, b) if epoch else torch.allclose(a, b, rtol=0, atol=float(a.abs().max()) * 600 * U)
            B.sat_cache_update(ctx, B.SAT_ALL_PARTS, 1, dev2d(rng.standard_normal((n, d)).astype(np.float32)))
            B.sat_cache_commit(ctx)
        for bad in (B.SAT_FWD_HALO_GLOBAL, B.SAT_FWD_INPUT_GLOBAL):
            with pytest.raises(B.SatError) as ei:
                B.sat_layer_fwd(ctx, 0, 2, H, H, W, None, B.SAT_ACT_NONE | B.SAT_FWD_HALO_CACHED | bad, empty2d(n, d2))
            assert ei.value.status == B.SAT_EINVAL
        with pytest.raises(B.SatError):                       # layer 1 has no cached layer below it
            B.sat_layer_fwd(ctx, 0, 1, H, None, W, None, B.SAT_ACT_NONE | B.SAT_FWD_HALO_CACHED, empty2d(n, d2))
        B.sat_sync_status(ctx)
    finally:
        B.sat_destroy(ctx)


@pytest.mark.parametrize("rows", [3, 64, 255, 256, 257, 1000, 5000, 21000])
@pytest.mark.parametrize("m,n", [(4, 3), (16, 16), (20, 64), (130, 48), (128, 65), (100, 100), (256, 256), (300, 260), (65, 512)])
def test_weight_and_bias_gradient(B, rows, m, n):
    """G_W = AGG^T D and G_b = 1^T D of a layer on a ring graph (AGG from three rows each), one partition."""
    A = _graph([], rows)
    P = _propagation(A)
    rng = np.random.default_rng(rows + m + n)
    X, D = rng.standard_normal((rows, m)).astype(np.float32), rng.standard_normal((rows, n)).astype(np.float32)
    ctx = B.sat_create(0, 0)
    try:
        B.sat_graph_load(ctx, A.indptr.astype(np.int64), A.indices.astype(np.int32))
        B.sat_partition(ctx, 1, B.SAT_PART_CONTIG_BLOCKS)
        W = dev(np.zeros((m, n), np.float32))
        B.sat_layer_fwd(ctx, 0, 1, dev2d(X), None, W, None, B.SAT_ACT_NONE | B.SAT_FWD_INPUT_GLOBAL, empty2d(rows, n))
        gW, gb = torch.full((m, n), float("nan"), device="cuda"), torch.full((n,), float("nan"), device="cuda")
        B.sat_layer_bwd(ctx, 0, 1, dev2d(D), W, gW, gb, 0, None, None)
        X64, D64 = P @ X.astype(np.float64), D.astype(np.float64)
        mag = (abs(P) @ np.abs(X.astype(np.float64))).T @ np.abs(D64)       # AGG itself carries 8 roundings of its own terms
        assert (np.abs(gW.cpu().numpy() - X64.T @ D64) <= ((min(rows, 1500) + 8) * U + 2.0 ** -20) * mag).all()
        assert (np.abs(gb.cpu().numpy() - D64.sum(0)) <= min(rows, 1500) * U * np.abs(D64).sum(0)).all()
        B.sat_layer_bwd(ctx, 0, 1, dev2d(D), W, gW, gb, 1, None, None)      # accumulate
        assert (np.abs(gb.cpu().numpy() - 2 * D64.sum(0)) <= 2 * (min(rows, 1500) + 2) * U * np.abs(D64).sum(0)).all()
        assert (np.abs(gW.cpu().numpy() - 2 * (X64.T @ D64)) <= 2 * ((min(rows, 1500) + 10) * U + 2.0 ** -20) * mag).all()
        B.sat_sync_status(ctx)
    finally:
        B.sat_destroy(ctx)


@pytest.mark.parametrize("rows", [3, 31, 33, 1000, 30011])
@pytest.mark.parametrize("C", [1, 2, 8, 9, 16, 17, 32, 33, 64, 65, 100, 128, 129, 300])
@pytest.mark.parametrize("kind", ["ce", "bce"])
def test_losses(B, rows, C, kind):
    """Loss sum and gradient; expf / logf / log1pf are within 2 units in the last place, the sums of C terms as above."""
    rng = np.random.default_rng(C)
    A = _graph([], rows)
    z = (3 * rng.standard_normal((rows, C))).astype(np.float32)
    ctx = B.sat_create(0, 0)
    try:
        B.sat_graph_load(ctx, A.indptr.astype(np.int64), A.indices.astype(np.int32))
        B.sat_partition(ctx, 1, B.SAT_PART_CONTIG_BLOCKS)
        z64 = torch.from_numpy(z).double().requires_grad_()
        if kind == "ce":
            y = rng.integers(0, C, rows).astype(np.int32)
            per = torch.nn.functional.cross_entropy(z64, torch.from_numpy(y).long(), reduction="none")
        else:
            y = (rng.random((rows, C)) < 0.3).astype(np.uint8)
            per = torch.nn.functional.binary_cross_entropy_with_logits(z64, torch.from_numpy(y).double(), reduction="none").mean(1)
        want = per.sum() / rows
        want.backward()
        for view in (dev2d(z), torch.zeros((rows, C + 3), device="cuda")[:, :C]):      # rows of 16 bytes, and any rows
            view.copy_(torch.from_numpy(z))
            g, total = torch.full((rows, C + 1), float("nan"), device="cuda")[:, :C], torch.zeros(1, dtype=torch.float64, device="cuda")
            for _ in range(2):
                B.sat_loss_grad(ctx, 0, B.SAT_LOSS_SOFTMAX_CE if kind == "ce" else B.SAT_LOSS_SIGMOID_BCE, view, dev(y), total, g)
            # one term of a row: a few roundings of values up to |z| + log C, about 20
            assert abs(float(total) / 2 - float(want.detach())) <= (C + 16) * U * max(20.0, float(want.detach()))
            assert float((g.cpu().double() - z64.grad).abs().max()) <= (C + 16) * U / rows * (1.0 if kind == "ce" else 1.0 / C)
        B.sat_sync_status(ctx)
    finally:
        B.sat_destroy(ctx)


@pytest.mark.parametrize("d", [16, 17, 100, 256])
@pytest.mark.parametrize("h", [4, 8, 20, 60, 64, 68])       # 4 h gate columns: one tile up to h = 64, contractions and a cell kernel above
@pytest.mark.parametrize("steps", [1, 2, 5])
def test_gru_state(B, d, h, steps):
    """sat_predict_state against the cell in fp64.  With e the error of a pre-activation (bound of the module's docstring plus what the
    previous state brings through Uh) and sigma' <= 1/4, tanh' <= 1:  |ds| <= e_z / 2 + e_n + e_hn + |hn| e_r / 4 + |ds_prev| + 2^-20."""
    n, M = 700, 3
    A = _graph([300, 40], n)
    rng = np.random.default_rng(d + h)
    part = rng.integers(0, M, n).astype(np.int32)
    perm = np.concatenate([np.flatnonzero(part == m) for m in range(M)])
    W, Uh, b = rng.standard_normal((d, 3 * h)) / d ** 0.5, rng.standard_normal((h, 3 * h)) / h ** 0.5, rng.standard_normal(4 * h) / 4
    Wg, bg = np.zeros((h, d)), np.zeros(d)
    W, Uh, b, Wg, bg = (x.astype(np.float32) for x in (W, Uh, b, Wg, bg))
    ctx = B.sat_create(0, 0)
    try:
        B.sat_graph_load(ctx, A.indptr.astype(np.int64), A.indices.astype(np.int32))
        B.sat_partition(ctx, M, B.SAT_PART_GIVEN, part)
        B.sat_cache_init(ctx, [d], 5)
        n_halo = sum(B.sat_part_sizes(ctx, m)[1] for m in range(M))
        n_slots = B.sat_slot_map(ctx, n)[2]
        for _ in range(steps):
            B.sat_cache_update(ctx, B.SAT_ALL_PARTS, 1, dev2d(rng.standard_normal((n, d)).astype(np.float32)[perm]))
            B.sat_cache_commit(ctx)
        snaps = [B.sat_cache_read(ctx, 1, age, n_slots, d).astype(np.float64) for age in range(steps - 1, -1, -1)]
        params = B.make_pred_params(dev(W), dev(Uh), dev(b), dev(Wg), dev(bg), h, 0, B.SAT_CELL_GRU)
        B.sat_predict(ctx, 1, B.SAT_ALL_PARTS, params, 0, empty2d(n_halo, d))
        S = B.sat_predict_state(ctx, 1, n_slots, h)
        B.sat_sync_status(ctx)
    finally:
        B.sat_destroy(ctx)
    s, ds = np.zeros((n_slots, h)), np.zeros((n_slots, h))
    sig = lambda v: 1 / (1 + np.exp(-v))
    U64 = Uh.astype(np.float64)
    for x in snaps:
        ax, ah = x @ W + b[:3 * h], s @ U64
        e = ((d + h + 2) * U + 2.0 ** -20) * (np.abs(x) @ np.abs(W) + np.abs(s) @ np.abs(U64) + np.abs(b[:3 * h])) + ds @ np.abs(U64)
        hn = ah[:, 2 * h:] + b[3 * h:]
        r, z = sig(ax[:, :h] + ah[:, :h]), sig(ax[:, h:2 * h] + ah[:, h:2 * h])
        cand = np.tanh(ax[:, 2 * h:] + r * hn)
        ds = e[:, h:2 * h] / 2 + 2 * e[:, 2 * h:] + np.abs(hn) * e[:, :h] / 4 + ds + 2.0 ** -20
        s = (1 - z) * cand + z * s
    assert (np.abs(S - s) <= ds).all()


@pytest.mark.parametrize("n,k", [(16, 16), (40, 100), (72, 17), (128, 256), (256, 64), (257, 40), (300, 602)])
@pytest.mark.parametrize("rows", [-1, 0, 1, 128, 129, 256, 20000])      # relative to a wave of single CTAs (128 rows each): pairs above it
def test_contraction_by_single_ctas_and_by_pairs(B, n, k, rows):
    tiles_n = -(-n // 256)
    m = 128 * (torch.cuda.get_device_properties(0).multi_processor_count // tiles_n) + rows
    rng = np.random.default_rng(n + k)
    A, W, b = (rng.standard_normal(s).astype(np.float32) for s in ((m, k), (k, n), (n,)))
    ctx = B.sat_create(0, 0)
    try:
        out = empty2d(m, n)
        B.sat_dense_nn(ctx, dev2d(A), dev(W), dev(b), out)
        B.sat_sync_status(ctx)
    finally:
        B.sat_destroy(ctx)
    sel = np.unique(np.concatenate([np.arange(300), np.arange(m - 300, m), rng.integers(0, m, 300)]))
    a = A[sel].astype(np.float64)
    bound = ((k + 2) * U + 2.0 ** -20) * (np.abs(a) @ np.abs(W) + np.abs(b))
    assert (np.abs(out.cpu().numpy()[sel] - (a @ W + b)) <= bound).all()


@pytest.mark.parametrize("n,h,d,versions", [(700, h, d, v) for h in (16, 20, 32, 48, 60, 64) for d, v in ((16, [1]), (100, [1, 1]), (40, [1] * 6))] +
                         [(700, 64, 40, [1, 1, 2, 1, 1]), (700, 24, 40, [2, 1, 1, 1]), (45000, 64, 40, [1, 1, 1]), (45000, 20, 16, [1, 2, 1, 1])])
def test_lstm_state_over_cached_projections(B, n, h, d, versions):
    """State of the predictor after every epoch, its parameter version as given (steps over cached projections run as one launch, others on
    their own; more than 256 rows a CTA pair at the larger size) against the cell in fp64.  With e the error of a pre-activation (bound
    of the module's docstring, and what the previous state brings through Uh), eta = 2^-20 that of a gate, sigma' <= 1/4, tanh' <= 1:
    |dc| <= |c| (e_f / 4 + eta) + |dc_prev| + |g| (e_i / 4 + eta) + e_g + eta,  |ds| <= e_o / 4 + eta + |dc| + eta."""
    tau, M = 5, 3
    A = _graph([300, 40], n)
    rng = np.random.default_rng(d + h)
    part = rng.integers(0, M, n).astype(np.int32)
    perm = np.concatenate([np.flatnonzero(part == m) for m in range(M)])
    W, Uh, b = rng.standard_normal((d, 4 * h)) / d ** 0.5, rng.standard_normal((h, 4 * h)) / h ** 0.5, rng.standard_normal(4 * h) / 4
    W, Uh, b, Wg, bg = (x.astype(np.float32) for x in (W, Uh, b, np.zeros((h, d)), np.zeros(d)))
    ctx = B.sat_create(0, 0)
    try:
        B.sat_graph_load(ctx, A.indptr.astype(np.int64), A.indices.astype(np.int32))
        B.sat_partition(ctx, M, B.SAT_PART_GIVEN, part)
        B.sat_cache_init(ctx, [d], tau)
        out = empty2d(sum(B.sat_part_sizes(ctx, m)[1] for m in range(M)), d)
        n_slots = B.sat_slot_map(ctx, n)[2]
        weights = [dev(x) for x in (W, Uh, b, Wg, bg)]
        for version in versions:
            B.sat_cache_update(ctx, B.SAT_ALL_PARTS, 1, dev2d(rng.standard_normal((n, d)).astype(np.float32)[perm]))
            B.sat_cache_commit(ctx)
            B.sat_predict(ctx, 1, B.SAT_ALL_PARTS, B.make_pred_params(*weights, h, version, B.SAT_CELL_LSTM), 0, out)
        S = B.sat_predict_state(ctx, 1, n_slots, h)
        B.sat_sync_status(ctx)
        snaps = [B.sat_cache_read(ctx, 1, age, n_slots, d) for age in range(min(len(versions), tau) - 1, -1, -1)]
    finally:
        B.sat_destroy(ctx)
    sel = np.unique(np.concatenate([np.arange(300), np.arange(n_slots - 300, n_slots), rng.integers(0, n_slots, 400)]))
    s, c, ds, dc = (np.zeros((len(sel), h)) for _ in range(4))
    sig = lambda v: 1 / (1 + np.exp(-v))
    U64, eta = Uh.astype(np.float64), 2.0 ** -20
    for x in snaps:
        x = x[sel].astype(np.float64)
        z = x @ W + s @ U64 + b
        e = ((d + h + 2) * U + 2.0 ** -20) * (np.abs(x) @ np.abs(W) + np.abs(s) @ np.abs(U64) + np.abs(b)) + ds @ np.abs(U64)
        (zi, zf, zg, zo), (ei, ef, eg, eo) = (np.split(v, 4, axis=1) for v in (z, e))
        g = np.tanh(zg)
        dc = np.abs(c) * (ef / 4 + eta) + dc + np.abs(g) * (ei / 4 + eta) + eg + eta
        c = sig(zf) * c + sig(zi) * g
        s = sig(zo) * np.tanh(c)
        ds = eo / 4 + eta + dc + eta
    assert (np.abs(S[sel] - s) <= ds).all()


@pytest.mark.parametrize("tau,h", [(7, 20), (8, 32), (10, 24)])     # steps summed by one launch: up to eight, the rest by a second one
def test_predictor_gradient_over_long_windows(B, tau, h):
    from tests.test_gpu_pred_train import test_gradient_for_every_fill_level as check
    check(B, "medium", 16, {"tau": tau, "h": h})


@pytest.mark.parametrize("parts", [False, True])
@pytest.mark.parametrize("d_out", [40, 43, 256, 300])                 # one launch per slice of 256 columns; rows of many runs by their last run
def test_attention_layer_pushes_its_boundary_rows(B, d_out, parts):
    """SAT_FWD_PUSH of sat_gat_fwd against sat_cache_update: same bits in the ring and in h_out."""
    n, M, d = 3000, 3, 24
    A = _graph(HUBS, n)
    rng = np.random.default_rng(d_out)
    part = rng.integers(0, M, n).astype(np.int32)
    ctx = B.sat_create(0, 0)
    try:
        B.sat_graph_load(ctx, A.indptr.astype(np.int64), A.indices.astype(np.int32))
        B.sat_partition(ctx, M, B.SAT_PART_GIVEN, part)
        B.sat_cache_init(ctx, [d_out], 2)
        sizes = [B.sat_part_sizes(ctx, m) for m in range(M)]
        n_slots = B.sat_slot_map(ctx, n)[2]
        H, halo = dev2d(rng.standard_normal((n, d)).astype(np.float32)), dev2d(rng.standard_normal((sum(s[1] for s in sizes), d)).astype(np.float32))
        W, a1, a2, b = (dev(rng.standard_normal(s).astype(np.float32)) for s in ((d, d_out), (d_out,), (d_out,), (d_out,)))
        got = []
        for push in (0, B.SAT_FWD_PUSH):
            out = empty2d(n, d_out)
            r0 = u0 = 0
            for m in range(M) if parts else [B.SAT_ALL_PARTS]:
                r1, u1 = (r0 + sizes[m][0], u0 + sizes[m][1]) if parts else (n, len(halo))
                B.sat_gat_fwd(ctx, m, 1, H[r0:r1], halo[u0:u1], W, a1, a2, b, B.SAT_ACT_RELU | push, out[r0:r1])
                if not push:
                    B.sat_cache_update(ctx, m, 1, out[r0:r1])
                r0, u0 = r1, u1
            B.sat_cache_commit(ctx)
            got.append((out.cpu().numpy()[:, :d_out], B.sat_cache_read(ctx, 1, 0, n_slots, d_out)))
        assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1])
        with pytest.raises(B.SatError):                       # layer 2 is not cached
            B.sat_gat_fwd(ctx, B.SAT_ALL_PARTS, 2, H, halo, W, a1, a2, b, B.SAT_ACT_RELU | B.SAT_FWD_PUSH, empty2d(n, d_out))
        B.sat_sync_status(ctx)
    finally:
        B.sat_destroy(ctx)


@pytest.mark.parametrize("n", [2, 3, 4, 5, 31, 33, 100])          # four rows a warp
@pytest.mark.parametrize("d", [4, 7, 128, 130, 260])
def test_attention_scores(B, n, d):
    """Scores kept by sat_gat_fwd against a . (h W) in fp64 (two contractions one after the other)."""
    rng = np.random.default_rng(n + d)
    m = sp.coo_matrix((np.ones(n - 1), (np.arange(n - 1), np.arange(1, n))), shape=(n, n))
    A = (m + m.T).tocsr()
    A.sort_indices()
    k = 20
    H, W, a1, a2 = (rng.standard_normal(s).astype(np.float32) for s in ((n, k), (k, d), (d,), (d,)))
    ctx = B.sat_create(0, 0)
    try:
        B.sat_graph_load(ctx, A.indptr.astype(np.int64), A.indices.astype(np.int32))
        B.sat_partition(ctx, 1, B.SAT_PART_GIVEN, np.zeros(n, np.int32))
        out = empty2d(n, d)
        B.sat_gat_fwd(ctx, B.SAT_ALL_PARTS, 1, dev2d(H), None, dev(W), dev(a1), dev(a2), None, B.SAT_ACT_NONE, out)
        s_src, s_dst, _ = B.sat_gat_scores(ctx, 1, n, 0)
        B.sat_sync_status(ctx)
    finally:
        B.sat_destroy(ctx)
    z, terms = H.astype(np.float64) @ W, np.abs(H).astype(np.float64) @ np.abs(W)
    for got, a in ((s_src, a1), (s_dst, a2)):
        bound = ((k + 2) * U + 2.0 ** -20) * (terms @ np.abs(a)) + (d + 2) * U * (np.abs(z) @ np.abs(a)) * (1 + 2.0 ** -10)
        assert (np.abs(got - z @ a) <= bound + 1e-30).all()


@pytest.mark.parametrize("m,n", [(300, 256), (384, 512)])
def test_weight_gradient_error_with_an_odd_number_of_column_tiles(B, m, n):
    """Sums of positive terms: what is lost is the truncating accumulation, which grows with the rows that a split adds up.  At most two
    128-column tiles per SM decide that length; against 256 columns (two such tiles) the error may grow by the ratio of the lengths.
    (1.2: the loss per addition, relative to the sum, moves by the place of the sum between two powers of two.)"""
    rows, sms = 120000, torch.cuda.get_device_properties(0).multi_processor_count
    gen = torch.Generator(device="cuda")
    gen.manual_seed(m)
    A, D = (torch.empty((rows, w), device="cuda").normal_(generator=gen).abs_() for w in (m, n))
    lost, length = [], []
    ctx = B.sat_create(0, torch.cuda.current_stream().cuda_stream)
    try:
        for k in (256, m):
            C = torch.empty((k, n), device="cuda")
            B.sat_dense_tn(ctx, A[:, :k], D, C)
            B.sat_sync_status(ctx)
            want = A[:, :k].double().T @ D.double()
            lost.append(float((1 - C.double() / want).mean()))
            length.append(rows / -(-2 * sms // (-(-k // 128) * -(-n // 256))))
    finally:
        B.sat_destroy(ctx)
    assert 0 < lost[1] <= 1.2 * lost[0] * length[1] / length[0]


@pytest.mark.parametrize("m,n", [(16, 47), (256, 512)])               # the narrow kernel, and the converters of the tensor-core one
def test_bias_gradient_of_many_rows(B, m, n):
    """One large term and many of half its last place, which a plain running sum would lose (2^-25 each, 200 and more behind the large
    one); levels of at most 16 additions, 64 in all, lose at most 64 units of the sum."""
    rows = 400000
    ids = np.arange(rows)
    col = np.sort(np.stack([(ids - 1) % rows, (ids + 1) % rows], 1), 1).astype(np.int32).ravel()
    ctx = B.sat_create(0, torch.cuda.current_stream().cuda_stream)
    try:
        B.sat_graph_load(ctx, 2 * np.arange(rows + 1, dtype=np.int64), col)
        B.sat_partition(ctx, 1, B.SAT_PART_CONTIG_BLOCKS)
        X, D, W = torch.ones((rows, m), device="cuda"), empty2d(rows, n, fill=2.0 ** -25), torch.zeros((m, n), device="cuda")
        D[0] = 1.0
        B.sat_layer_fwd(ctx, 0, 1, X, None, W, None, B.SAT_ACT_NONE | B.SAT_FWD_INPUT_GLOBAL, empty2d(rows, n))
        gW, gb = torch.empty((m, n), device="cuda"), torch.empty(n, device="cuda")
        B.sat_layer_bwd(ctx, 0, 1, D, W, gW, gb, 0, None, None)
        B.sat_sync_status(ctx)
    finally:
        B.sat_destroy(ctx)
    want = 1.0 + (rows - 1) * 2.0 ** -25
    assert float((gb.double() - want).abs().max()) <= 64 * U * want


@pytest.mark.parametrize("n,k", [(256, 256), (512, 512), (100, 48), (40, 600)])
def test_pairs_give_the_bits_of_single_ctas_every_time(B, n, k):
    """Many tiles per CTA pair, again and again, against the same rows in launches of at most a wave of single CTAs: an order that the pair's
    barriers fail to keep would show as a tile that differs once in a while."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    step = 128 * (sms // -(-n // 256))
    m = 6 * step + 77
    gen = torch.Generator(device="cuda")
    gen.manual_seed(n)
    A, W, b = torch.randn((m, k), device="cuda", generator=gen), torch.randn((k, n), device="cuda", generator=gen), torch.randn(n, device="cuda", generator=gen)
    want, out = empty2d(m, n), empty2d(m, n)
    ctx = B.sat_create(0, torch.cuda.current_stream().cuda_stream)
    try:
        for r in range(0, m, step):
            B.sat_dense_nn(ctx, A[r:r + step], W, b, want[r:r + step])
        for _ in range(50):
            out.fill_(float("nan"))
            B.sat_dense_nn(ctx, A, W, b, out)
            assert torch.equal(out, want)
        B.sat_sync_status(ctx)
    finally:
        B.sat_destroy(ctx)


@pytest.mark.parametrize("h", [20, 64])
def test_lstm_steps_repeat_themselves(B, h):
    """The state after five steps over cached projections, more than one tile per slot of a CTA: the same bits in every run."""
    n, d, tau = 120000, 32, 5
    ids = np.arange(n)
    col = np.sort(np.stack([(ids - 1) % n, (ids + 1) % n], 1), 1).astype(np.int32).ravel()
    gen = torch.Generator(device="cuda")
    gen.manual_seed(h)
    rand = lambda *s: torch.randn(s, device="cuda", generator=gen)
    ctx = B.sat_create(0, torch.cuda.current_stream().cuda_stream)
    try:
        B.sat_graph_load(ctx, 2 * np.arange(n + 1, dtype=np.int64), col)
        B.sat_partition(ctx, 2, B.SAT_PART_GIVEN, (ids % 2).astype(np.int32))       # every node is a boundary node
        B.sat_cache_init(ctx, [d], tau)
        out, first = empty2d(n, d), None
        p = B.make_pred_params(rand(d, 4 * h) / d ** 0.5, rand(h, 4 * h) / h ** 0.5, rand(4 * h), rand(h, d) / h ** 0.5, rand(d), h, 1)
        for _ in range(tau):
            B.sat_cache_update(ctx, B.SAT_ALL_PARTS, 1, rand(n, d))
            B.sat_cache_commit(ctx)
            B.sat_predict(ctx, 1, B.SAT_ALL_PARTS, p, 0, out)
        first = out.clone()
        for _ in range(50):
            out.fill_(float("nan"))
            B.sat_predict(ctx, 1, B.SAT_ALL_PARTS, p, 0, out)
            assert torch.equal(out, first)
        B.sat_sync_status(ctx)
    finally:
        B.sat_destroy(ctx)


@pytest.mark.parametrize("h", [16, 28])
def test_lstm_cell_at_its_limits(B, h):
    """Pre-activations far beyond the gates' saturation, and infinite or undefined ones in single rows, over cached projections: the limits of the
    cell (to 2^-20, the error of a gate), a NaN stays a NaN, and every other row is as it is without them."""
    n, d, tau = 600, 16, 3
    ids = np.arange(n)
    col = np.sort(np.stack([(ids - 1) % n, (ids + 1) % n], 1), 1).astype(np.int32).ravel()
    rng = np.random.default_rng(h)
    x = rng.standard_normal((n, d)).astype(np.float32)
    x[:200] *= np.exp2(rng.integers(0, 40, (200, 1))).astype(np.float32)
    Wx, b = np.zeros((d, 4 * h), np.float32), rng.standard_normal(4 * h).astype(np.float32) / 4
    Wx[rng.integers(0, d, 4 * h), np.arange(4 * h)] = 2.0 ** rng.integers(-2, 3, 4 * h)      # one term each: the projections have no rounding but the bias's
    Uh, Wg, bg = np.zeros((h, 4 * h), np.float32), np.zeros((h, d), np.float32), np.zeros(d, np.float32)
    bad = {300: np.nan, 417: np.inf, 599: -np.inf}
    states = []
    for with_bad in (False, True):
        xs = x.copy()
        if with_bad:
            for r, v in bad.items():
                xs[r, :] = v
        ctx = B.sat_create(0, 0)
        try:
            B.sat_graph_load(ctx, 2 * np.arange(n + 1, dtype=np.int64), col)
            B.sat_partition(ctx, 2, B.SAT_PART_GIVEN, (ids % 2).astype(np.int32))
            B.sat_cache_init(ctx, [d], tau)
            perm = np.concatenate([np.flatnonzero(ids % 2 == m) for m in range(2)])
            out = empty2d(n, d)
            p = B.make_pred_params(*(dev(a) for a in (Wx, Uh, b, Wg, bg)), h, 1)
            for _ in range(tau):
                B.sat_cache_update(ctx, B.SAT_ALL_PARTS, 1, dev2d(xs[perm]))
                B.sat_cache_commit(ctx)
                B.sat_predict(ctx, 1, B.SAT_ALL_PARTS, p, 0, out)
            slot = np.asarray(B.sat_slot_map(ctx, n)[1])
            states.append(B.sat_predict_state(ctx, 1, n, h)[slot])
            B.sat_sync_status(ctx)
        finally:
            B.sat_destroy(ctx)
    rest = np.setdiff1d(ids, list(bad))
    assert np.array_equal(states[0][rest], states[1][rest])
    assert np.isnan(states[1][list(bad)]).all()
    z = x.astype(np.float64) @ Wx + b
    zi, zf, zg, zo = np.split(np.clip(z, -700, 700), 4, axis=1)
    sig = lambda v: 1 / (1 + np.exp(-v))
    c, e = 0.0, ((np.abs(x) @ np.abs(Wx) + np.abs(b)) * 2.0 ** -20).reshape(n, 4, h)
    e = np.minimum(e, 2.0) * np.stack([sig(v) * sig(-v) for v in (zi, zf, 2 * zg, zo)], 1) * 4 + 2.0 ** -20      # slope of the gates at z, four times it for tanh
    for _ in range(tau):
        c = sig(zf) * c + sig(zi) * np.tanh(zg)
    s = sig(zo) * np.tanh(c)
    assert (np.abs(states[0] - s) <= 3 * tau * e.sum(1)).all()


def _many_runs(kind):
    """"hub": one row of 9,000 entries in a small list, more runs than the last one adds (64 of at most 128 entries): the block reduction of
    k_spmm_fixup.  "large": above 2^20 entries, where k_spmm_fixup adds every row of more than one run: ordinary rows of one run of
    64, rows of 2 to 16 runs by a thread per column, longer ones by a block."""
    rng = np.random.default_rng(11)
    if kind == "hub":
        return _graph([9000, 40, 70], 12000)
    n = 30000
    pairs = rng.integers(0, n, (560000, 2))
    hubs = [np.stack([np.full(deg, i), rng.integers(0, n, deg)], 1) for i, deg in enumerate([20, 30, 90, 200, 500, 900, 1100, 1500, 4000, 25000])]
    ring = np.stack([np.arange(n), (np.arange(n) + 1) % n], 1)
    a = np.concatenate([pairs, ring] + hubs)
    a = a[a[:, 0] != a[:, 1]]
    m = sp.coo_matrix((np.ones(len(a)), (a[:, 0], a[:, 1])), shape=(n, n))
    m = ((m + m.T) > 0).astype(np.float64).tocsr()
    m.sort_indices()
    return m


@pytest.mark.parametrize("kind", ["hub", "large"])
@pytest.mark.parametrize("d", [40, 43, 260])
def test_rows_that_the_second_launch_finishes(B, kind, d):
    """GCN aggregation and the attention layer's forward, push and backward on rows of many runs, against fp64; all partitions at once and
    one after the other (same bits).  The second launch shows in the launch count: an equal call whose rows are all short has one less."""
    from tests.gpu_util import assert_close
    A, k, M = _many_runs(kind), 8, 2
    n = A.shape[0]
    if kind == "large":
        assert A.nnz + n > 2 ** 20
    rng = np.random.default_rng(d)
    part = rng.integers(0, M, n).astype(np.int32)
    perm = np.concatenate([np.flatnonzero(part == m) for m in range(M)])
    X, G = rng.standard_normal((n, k)).astype(np.float32), rng.standard_normal((n, d)).astype(np.float32)
    W, a1, a2, b = ((rng.standard_normal(s) * 0.4).astype(np.float32) for s in ((k, d), (d,), (d,), (d,)))
    Y = rng.standard_normal((n, d)).astype(np.float32)
    eye = np.eye(d, 4, dtype=np.float32)

    def calls(graph, rows):
        """Launches of the GCN forward and of the attention layer on the first `rows` nodes of the inputs, and their results."""
        pt = part[:rows]
        order = np.concatenate([np.flatnonzero(pt == m) for m in range(M)])
        ctx = B.sat_create(0, 0)
        try:
            B.sat_graph_load(ctx, graph.indptr.astype(np.int64), graph.indices.astype(np.int32))
            B.sat_partition(ctx, M, B.SAT_PART_GIVEN, pt)
            B.sat_cache_init(ctx, [d], 2)
            lists = [B.sat_part_lists(ctx, m) for m in range(M)]
            halo = np.concatenate([l["halo_gid"] for l in lists])
            n_in = [len(l["inner_gid"]) for l in lists]
            n_out = [len(l["halo_gid"]) for l in lists]
            n_slots = B.sat_slot_map(ctx, rows)[2]
            agg, h_in, h_halo, g = empty2d(rows, 4), dev2d(X[order]), dev2d(X[halo]), dev2d(G[order])
            Wd, a1d, a2d, bd = dev(W), dev(a1), dev(a2), dev(b)
            grads = [torch.empty_like(t) for t in (Wd, a1d, a2d, bd)]
            out, g_in, got, counts = empty2d(rows, d), empty2d(rows, k), [], []
            gcn = lambda: B.sat_layer_fwd(ctx, B.SAT_ALL_PARTS, 2, dev2d(Y[:rows]), None, dev(eye), None, B.SAT_ACT_NONE | B.SAT_FWD_INPUT_GLOBAL, agg)
            fwd = lambda: B.sat_gat_fwd(ctx, B.SAT_ALL_PARTS, 1, h_in, h_halo, Wd, a1d, a2d, bd, B.SAT_ACT_NONE | B.SAT_FWD_PUSH, out)
            bwd = lambda: B.sat_gat_bwd(ctx, B.SAT_ALL_PARTS, 1, g, None, h_in, h_halo, Wd, a1d, a2d, *grads, 0, g_in)
            for call in (gcn, fwd, bwd):
                call()                       # builds the lists
                at = B.sat_launch_count(ctx)
                call()
                counts.append(B.sat_launch_count(ctx) - at)
            ring = B.sat_cache_read(ctx, 1, -1, n_slots, d)
            scores = B.sat_gat_scores(ctx, 1, rows, len(halo))
            got = [t.cpu().numpy() for t in (agg, out, *grads, g_in)]
            out2, g_in2 = empty2d(rows, d), empty2d(rows, k)
            r0 = u0 = 0
            for m in range(M):
                r1, u1 = r0 + n_in[m], u0 + n_out[m]
                B.sat_gat_fwd(ctx, m, 1, h_in[r0:r1], h_halo[u0:u1], Wd, a1d, a2d, bd, B.SAT_ACT_NONE | B.SAT_FWD_PUSH, out2[r0:r1])
                B.sat_gat_bwd(ctx, m, 1, g[r0:r1], None, h_in[r0:r1], h_halo[u0:u1], Wd, a1d, a2d, *grads, 0, g_in2[r0:r1])
                r0, u0 = r1, u1
            B.sat_sync_status(ctx)
            assert np.array_equal(out2.cpu().numpy()[:, :d], got[1][:, :d]) and np.array_equal(g_in2.cpu().numpy()[:, :k], got[6][:, :k])
            assert np.array_equal(B.sat_cache_read(ctx, 1, -1, n_slots, d), ring)
            push = np.concatenate([np.stack([l["push_slot"], l["push_local"] + sum(n_in[:m])], 1) for m, l in enumerate(lists)])
            assert np.array_equal(ring[push[:, 0]], got[1][push[:, 1]][:, :d])
        finally:
            B.sat_destroy(ctx)
        return counts, got, scores, halo

    counts, (agg, out, gW, g1, g2, gb, g_in), (s_src, s_dst, s_halo), halo = calls(A, n)
    small, *_ = calls(_graph([], 1000), 1000)
    assert counts[0] == small[0] + 1 and counts[1] == small[1] + 1
    assert counts[2] >= small[2] + (2 if kind == "large" else 0)     # (the hub's row is half as long in either half of the backward pass)
    P = _propagation(A)
    want, mag = (P @ Y.astype(np.float64))[perm][:, :4], (abs(P) @ np.abs(Y.astype(np.float64)))[perm][:, :4]
    assert (np.abs(agg - want) <= (np.diff(A.indptr).max() + 8) * U * mag).all()
    # attention in fp64 on the edge list, slopes as the device decided them; a halo copy acts like the node it copies
    E = (A + sp.identity(n)).tocoo()
    c = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    v, u = c(E.row.astype(np.int64)), c(E.col.astype(np.int64))
    by_node = np.empty(n, np.float32), np.empty(n, np.float32)
    by_node[0][perm], by_node[1][perm] = s_src, s_dst
    pos = (c(by_node[1])[v] + c(by_node[0])[u]) > 0
    z, D = c(X).double() @ c(W).double(), c(G).double()
    pre = (z @ c(a2).double())[v] + (z @ c(a1).double())[u]
    slope = torch.where(pos, 1.0, float(np.float32(0.2))).double()
    e = slope * pre
    zero = lambda *s: torch.zeros(s, dtype=torch.float64, device="cuda")
    mx = torch.full((n,), -1e300, dtype=torch.float64, device="cuda").scatter_reduce(0, v, e, "amax")
    x = torch.exp(e - mx[v])
    al = x / zero(n).index_add(0, v, x)[v]
    chunks = torch.arange(len(v), device="cuda").split(1 << 18)
    o, dal, dz, dz_in = zero(n, d), zero(len(v)), zero(n, d), zero(n, d)
    inner = c(part)[v] == c(part)[u]
    for i in chunks:
        o.index_add_(0, v[i], al[i, None] * z[u[i]])
        dal[i] = (D[v[i]] * z[u[i]]).sum(1)
        dz.index_add_(0, u[i], al[i, None] * D[v[i]])
        dz_in.index_add_(0, u[i], (al[i] * inner[i])[:, None] * D[v[i]])
    t = zero(n).index_add(0, v, al * dal)
    dpre = al * (dal - t[v]) * slope
    ds, dd, ds_in = zero(n).index_add(0, u, dpre), zero(n).index_add(0, v, dpre), zero(n).index_add(0, u, dpre * inner)
    A1, A2 = c(a1).double(), c(a2).double()
    dz += ds[:, None] * A1 + dd[:, None] * A2
    dz_in += ds_in[:, None] * A1 + dd[:, None] * A2
    for what, got, ref in (("out", out[:, :d], (o + c(b).double())[c(perm)]), ("G_W", gW, c(X).double().T @ dz), ("G_a_src", g1, z.T @ ds),
                           ("G_a_dst", g2, z.T @ dd), ("G_b", gb, D.sum(0)), ("G_in", g_in[:, :k], (dz_in @ c(W).double().T)[c(perm)])):
        assert_close(got, ref.cpu().numpy(), what)


@pytest.mark.parametrize("hist", [False, True])
@pytest.mark.parametrize("d_in,d_out", [(16, 15), (33, 5), (40, 40), (72, 17), (256, 40), (260, 256), (300, 299), (24, 40)])
def test_input_gradient_in_both_orders(B, d_in, d_out, hist):
    """G_in = (P_in^T D + Q) W^T under the mask of the layer below (Q: stale rows of the boundary nodes, on request) at widths on both sides of the
    rule that picks the order, all partitions at once = one after the other."""
    n, M = 2000, 3
    A = _graph(HUBS[:11], n)
    Pm = _propagation(A).tocoo()
    rng = np.random.default_rng(d_in)
    part = rng.integers(0, M, n).astype(np.int32)
    perm = np.concatenate([np.flatnonzero(part == m) for m in range(M)])
    off = np.concatenate([[0], np.cumsum(np.bincount(part, minlength=M))])
    W1, W2 = (rng.standard_normal(s).astype(np.float32) for s in ((8, d_in), (d_in, d_out)))
    X, D = rng.standard_normal((n, 8)).astype(np.float32), rng.standard_normal((n, d_out)).astype(np.float32)
    ctx = B.sat_create(0, 0)
    try:
        B.sat_graph_load(ctx, A.indptr.astype(np.int64), A.indices.astype(np.int32))
        B.sat_partition(ctx, M, B.SAT_PART_GIVEN, part)
        B.sat_cache_init(ctx, [d_in], 2)
        _, slot, n_slots = B.sat_slot_map(ctx, n)
        n_halo = B.sat_part_sizes(ctx, B.SAT_ALL_PARTS)[1]
        H1, H2, g_in, one = empty2d(n, d_in), empty2d(n, d_out), empty2d(n, d_in), empty2d(n, d_in)
        B.sat_layer_fwd(ctx, B.SAT_ALL_PARTS, 1, dev2d(X), None, dev(W1), None, B.SAT_ACT_RELU | B.SAT_FWD_INPUT_GLOBAL, H1)
        B.sat_layer_fwd(ctx, B.SAT_ALL_PARTS, 2, H1, dev2d(np.zeros((n_halo, d_in), np.float32)), dev(W2), None, B.SAT_ACT_NONE, H2)
        Q = np.zeros((n_slots, d_out), np.float32)
        if hist:
            Q = rng.standard_normal((n_slots, d_out)).astype(np.float32)
            B.sat_grad_history_write(ctx, 2, d_out, Q)
        flags = B.SAT_BWD_MASK_G_IN | (B.SAT_BWD_GRAD_HISTORY if hist else 0)
        gW, gb = torch.empty((d_in, d_out), device="cuda"), torch.empty(d_out, device="cuda")
        Dd = dev2d(D[perm])
        B.sat_layer_bwd(ctx, B.SAT_ALL_PARTS, 2, Dd, dev(W2), gW, gb, flags, g_in, None)
        for m in range(M):
            r = slice(off[m], off[m + 1])
            B.sat_layer_bwd(ctx, m, 2, Dd[r], dev(W2), gW, gb, flags, one[r], None)
        B.sat_sync_status(ctx)
        got, keep = g_in.cpu().numpy(), H1.cpu().numpy() > 0
        assert torch.equal(g_in, one)
    finally:
        B.sat_destroy(ctx)
    same = sp.csr_matrix((Pm.data * (part[Pm.row] == part[Pm.col]), (Pm.row, Pm.col)), shape=Pm.shape)
    slot = np.asarray(slot)
    stale = np.where((slot >= 0)[:, None], Q[np.maximum(slot, 0)], 0.0)
    want, mag = (same @ D.astype(np.float64) + stale) @ W2.T, (abs(same) @ np.abs(D.astype(np.float64)) + np.abs(stale)) @ np.abs(W2.T)
    terms = np.diff(A.indptr).max() + d_out + 8
    assert (np.abs(got - want[perm] * keep) <= (terms * U + 2.0 ** -20) * mag[perm]).all()


# halves from 192 terms on in large graphs, from 384 on in all; B resident and not, one and two tiles of columns
@pytest.mark.parametrize("m,n,k", [(m, n, k) for m in (1, 130) for n, k in ((16, 384), (40, 401), (256, 400), (512, 512), (300, 602))] +
                         [(40000, 16, 192), (40000, 256, 256), (40000, 100, 320), (40000, 300, 602), (32767, 64, 383), (32768, 64, 192)])
def test_contraction_of_rows_of_any_size(B, m, n, k):
    """Long contractions split their operands into halves with a scale per row and per eight columns of W: rows and columns of very different sizes, rows of
    zeros, and rows that are not finite and stay by themselves.  |x s - hi - lo| <= 2^-22 |x s| + 2^-25 with the largest |x s| at 2^14 or more.
    In a graph without edges the product with P is the row itself."""
    rng = np.random.default_rng(n + k)
    A = (rng.standard_normal((m, k)) * np.exp2(rng.integers(-60, 60, (m, 1)))).astype(np.float32)
    A[::7] *= np.exp2(rng.integers(-12, 1, (len(A[::7]), k))).astype(np.float32)       # a spread inside the row, too
    A[5:6] = 0.0
    W = (rng.standard_normal((k, n)) * np.exp2(rng.integers(-6, 6, (1, n)))).astype(np.float32)
    out, bad = empty2d(m, n), empty2d(m, n)
    A2 = A.copy()
    not_finite = [r for r in (3, 64, 129) if r < m]
    for r, v in zip(not_finite, (np.nan, np.inf, -np.inf)):
        A2[r, rng.integers(0, k)] = v
    ctx = B.sat_create(0, 0)
    try:
        B.sat_graph_load(ctx, np.zeros(m + 1, np.int64), np.zeros(0, np.int32))
        B.sat_partition(ctx, 1, B.SAT_PART_CONTIG_BLOCKS)
        for x, y in ((A, out), (A2, bad)):
            B.sat_layer_fwd(ctx, B.SAT_ALL_PARTS, 2, dev2d(x), None, dev(W), None, B.SAT_ACT_NONE | B.SAT_FWD_INPUT_GLOBAL, y)
        B.sat_sync_status(ctx)
    finally:
        B.sat_destroy(ctx)
    out, bad = out.cpu().numpy(), bad.cpu().numpy()
    sel = np.unique(np.concatenate([np.arange(min(m, 130)), rng.integers(0, m, 500)]))
    a = A[sel].astype(np.float64)
    mag = np.abs(a) @ np.abs(W)
    floor = np.abs(a).max(1, keepdims=True) * 2.0 ** -39 * np.abs(W).sum(0)       # what a term loses below the smallest half
    assert (np.abs(out[sel] - a @ W) <= ((k + 2) * U + 2.0 ** -20) * mag + 2 * floor).all()
    assert (out[5:6] == 0).all()
    ok = np.ones(m, bool)
    ok[not_finite] = False
    assert np.array_equal(out[ok], bad[ok]) and not np.isfinite(bad[~ok]).any()


@pytest.mark.parametrize("kind", ["small", "hub", "large"])
@pytest.mark.parametrize("d,n_out", [(383, 16), (384, 16), (512, 64), (602, 300)])     # the last without and the first with halves, several slices of columns
def test_aggregated_rows_of_any_size(B, kind, d, n_out):
    """The transform takes the size of every aggregated row from the product that wrote it: rows of one run, rows added by their last run and rows of the
    second launch, one slice of columns and several.  A size that is too small would overflow a half, one that is too large lose the terms."""
    A = _graph(HUBS, 3000) if kind == "small" else _many_runs(kind)
    n, P = A.shape[0], _propagation(A)
    rng = np.random.default_rng(d)
    X = (rng.standard_normal((n, d)) * np.exp2(rng.integers(-30, 30, (n, 1)))).astype(np.float32)
    W = rng.standard_normal((d, n_out)).astype(np.float32)
    out = empty2d(n, n_out)
    ctx = B.sat_create(0, 0)
    try:
        B.sat_graph_load(ctx, A.indptr.astype(np.int64), A.indices.astype(np.int32))
        B.sat_partition(ctx, 2, B.SAT_PART_CONTIG_BLOCKS)
        B.sat_layer_fwd(ctx, B.SAT_ALL_PARTS, 2, dev2d(X), None, dev(W), None, B.SAT_ACT_NONE | B.SAT_FWD_INPUT_GLOBAL, out)
        B.sat_sync_status(ctx)
    finally:
        B.sat_destroy(ctx)
    agg, mag = P @ X.astype(np.float64), abs(P) @ np.abs(X.astype(np.float64))
    terms = np.diff(A.indptr).max() + d + 8
    floor = mag.max(1, keepdims=True) * 2.0 ** -39 * np.abs(W).sum(0)
    assert (np.abs(out.cpu().numpy() - agg @ W) <= (terms * U + 2.0 ** -20) * (mag @ np.abs(W)) + 2 * floor).all()


@pytest.mark.parametrize("d0,layer", [(24, 1), (400, 2)])      # pushed by either form of the contraction
def test_pushed_rows_and_imported_rows_predict_alike(B, d0, layer):
    """Snapshots that the layer pushed bring their rows' sizes along; imported ones have them looked for: the same prediction, bit for bit, also after a
    single partition has pushed over imported rows."""
    n, M, d, h = 1500, 3, 400, 32
    A = _graph(HUBS[:8], n)
    rng = np.random.default_rng(4)
    part = rng.integers(0, M, n).astype(np.int32)
    rand = lambda *s: dev(rng.standard_normal(s).astype(np.float32) / 8)
    ctx = B.sat_create(0, 0)
    try:
        B.sat_graph_load(ctx, A.indptr.astype(np.int64), A.indices.astype(np.int32))
        B.sat_partition(ctx, M, B.SAT_PART_GIVEN, part)
        B.sat_cache_init(ctx, [d] * layer, 2)
        n_halo, n_slots = B.sat_part_sizes(ctx, B.SAT_ALL_PARTS)[1], B.sat_slot_map(ctx, n)[2]
        off = np.concatenate([[0], np.cumsum(np.bincount(part, minlength=M))])
        W, out = rand(d0, d), empty2d(n, d)
        weights = [rand(d, 4 * h), rand(h, 4 * h), rand(4 * h), rand(h, d), rand(d)]
        push = B.SAT_ACT_RELU | B.SAT_FWD_PUSH | B.SAT_FWD_INPUT_GLOBAL
        for epoch in range(3):
            X = dev2d((rng.standard_normal((n, d0)) * np.exp2(rng.integers(-9, 9, (n, 1)))).astype(np.float32))
            B.sat_layer_fwd(ctx, B.SAT_ALL_PARTS, layer, X, None, W, None, push, out)
            B.sat_cache_commit(ctx)
        got = [empty2d(n_halo, d) for _ in range(4)]
        for i, version in ((0, 0), (1, 1)):
            p = B.make_pred_params(*weights, h, version, B.SAT_CELL_LSTM)
            B.sat_predict(ctx, layer, B.SAT_ALL_PARTS, p, 0, got[i])
        state = B.sat_cache_state(ctx)
        ring = B.sat_cache_export(ctx, layer, 2, n_slots, d)
        for i, version in ((2, 0), (3, 2)):
            B.sat_cache_import(ctx, layer, ring)
            B.sat_cache_set_state(ctx, *state)
            # the next snapshot: one partition's rows over imported ones
            B.sat_layer_fwd(ctx, 1, layer, X, None, W, None, push, out[off[1]:off[2]])
            p = B.make_pred_params(*weights, h, version, B.SAT_CELL_LSTM)
            B.sat_predict(ctx, layer, B.SAT_ALL_PARTS, p, 0, got[i])
        assert torch.equal(got[0], got[2]) and torch.equal(got[1], got[3])
        B.sat_cache_commit(ctx)                  # the mixed snapshot is the newest one
        B.sat_predict(ctx, layer, B.SAT_ALL_PARTS, B.make_pred_params(*weights, h, 0, B.SAT_CELL_LSTM), 0, got[0])
        state, ring = B.sat_cache_state(ctx), B.sat_cache_export(ctx, layer, 2, n_slots, d)
        B.sat_cache_import(ctx, layer, ring)
        B.sat_predict(ctx, layer, B.SAT_ALL_PARTS, B.make_pred_params(*weights, h, 0, B.SAT_CELL_LSTM), 0, got[2])
        assert torch.equal(got[0], got[2])
        B.sat_sync_status(ctx)
    finally:
        B.sat_destroy(ctx)


@pytest.mark.parametrize("h", [4, 20, 64])
@pytest.mark.parametrize("d", [384, 401])
def test_recurrent_cells_on_halves(B, d, h):
    """The cells' contractions over [x | s] and over projections where the input is wide enough for halves: the state's part has the scale of the input's
    rows or of one, whichever is larger."""
    test_gru_state(B, d, h, 3)
    for versions in ([0, 0, 0], [1, 2, 1, 1], [1, 1, 1]):
        test_lstm_state_over_cached_projections(B, 700, h, d, versions)


@pytest.mark.parametrize("dims", [(24, 20, 12, 5), (24, 400, 400, 24)])      # TF32 terms, half-precision pairs
def test_partitions_of_an_epoch_share_packed_weights(B, dims):
    """The passes of an epoch partition by partition take the weights that the first one packed; the next epoch packs its own, whatever happened to the
    parameters in between (here: a write to the same tensors).  Same bits as all partitions in one launch."""
    from paper_2308_13466_b200.epoch import SatEpoch
    n, M = 900, 3
    A = _graph([300, 40], n)
    rng = np.random.default_rng(dims[1])
    rand = lambda *s: dev(rng.standard_normal(s).astype(np.float32) / s[0] ** 0.5)
    X, labels = dev2d(rng.standard_normal((n, dims[0])).astype(np.float32)), dev(rng.integers(0, dims[-1], n).astype(np.int32))
    eps = [SatEpoch(A.indptr.astype(np.int64), A.indices.astype(np.int32), M, list(dims), 2, "ce") for _ in range(2)]
    try:
        W, b = [rand(x, y) for x, y in zip(dims, dims[1:])], [rand(y) for y in dims[1:]]
        for ep in eps:
            ep.set_inputs(X, labels)
        for epoch in range(3):
            eps[0].step_per_partition(W, b, None)
            eps[1].step(W, b, None)
            for l in range(1, len(dims)):
                assert torch.equal(eps[0].H[l], eps[1].H[l]), (epoch, l)
                assert torch.equal(eps[0].G[l], eps[1].G[l]), (epoch, l)
            for w in W + b:
                w.copy_(rand(*w.shape))
    finally:
        for ep in eps:
            ep.close()


@pytest.mark.parametrize("rows", [255, 256, 257, 21000])        # the general kernel below 256 rows
@pytest.mark.parametrize("m,n", [(16, 1), (17, 4), (64, 7), (65, 8), (130, 9), (300, 15)])
def test_weight_gradient_of_few_columns(B, rows, m, n):
    test_weight_and_bias_gradient(B, rows, m, n)


@pytest.mark.parametrize("parts", [False, True])
def test_prediction_from_rows_that_an_attention_layer_pushed(B, parts):
    """The ring's rows change under sat_gat_fwd as under sat_cache_update: the same prediction, from rows whose size a half does not hold without their own scale."""
    n, M, d, d_out, h = 1500, 3, 24, 400, 32
    A = _graph(HUBS[:8], n)
    rng = np.random.default_rng(7)
    part = rng.integers(0, M, n).astype(np.int32)
    rand = lambda *s: dev(rng.standard_normal(s).astype(np.float32) / 8)
    ctx = B.sat_create(0, 0)
    try:
        B.sat_graph_load(ctx, A.indptr.astype(np.int64), A.indices.astype(np.int32))
        B.sat_partition(ctx, M, B.SAT_PART_GIVEN, part)
        sizes = [B.sat_part_sizes(ctx, m) for m in range(M)]
        n_halo = sum(s[1] for s in sizes)
        H, halo = dev2d(1e6 * rng.standard_normal((n, d)).astype(np.float32)), dev2d(1e6 * rng.standard_normal((n_halo, d)).astype(np.float32))
        W, a1, a2, b = rand(d, d_out), 1e-6 * rand(d_out), 1e-6 * rand(d_out), rand(d_out)
        p = B.make_pred_params(1e-6 * rand(d_out, 4 * h), rand(h, 4 * h), rand(4 * h), rand(h, d_out), rand(d_out), h, 0, B.SAT_CELL_LSTM)
        got = []
        for push in (0, B.SAT_FWD_PUSH):
            B.sat_cache_init(ctx, [d_out], 2)
            out, pred = empty2d(n, d_out), empty2d(n_halo, d_out)
            r0 = u0 = 0
            for m in range(M) if parts else [B.SAT_ALL_PARTS]:
                r1, u1 = (r0 + sizes[m][0], u0 + sizes[m][1]) if parts else (n, n_halo)
                B.sat_gat_fwd(ctx, m, 1, H[r0:r1], halo[u0:u1], W, a1, a2, b, B.SAT_ACT_RELU | push, out[r0:r1])
                if not push:
                    B.sat_cache_update(ctx, m, 1, out[r0:r1])
                r0, u0 = r1, u1
            B.sat_cache_commit(ctx)
            B.sat_predict(ctx, 1, B.SAT_ALL_PARTS, p, 0, pred)
            got.append((out.clone(), pred.clone(), B.sat_predict_state(ctx, 1, B.sat_slot_map(ctx, n)[2], h)))
        assert float(got[0][0].abs().max()) > 65504 and np.isfinite(got[1][2]).all()
        assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1]) and np.array_equal(got[0][2], got[1][2])
        B.sat_sync_status(ctx)
    finally:
        B.sat_destroy(ctx)


def _rows_times(B, A, W, bias=None):
    """A W + bias by the transform of layer 2 of a graph without edges, where the product with P is the row itself."""
    m, n = len(A), W.shape[1]
    out = empty2d(m, n)
    ctx = B.sat_create(0, 0)
    try:
        B.sat_graph_load(ctx, np.zeros(m + 1, np.int64), np.zeros(0, np.int32))
        B.sat_partition(ctx, 1, B.SAT_PART_CONTIG_BLOCKS)
        B.sat_layer_fwd(ctx, B.SAT_ALL_PARTS, 2, dev2d(A), None, dev(W), None if bias is None else dev(bias), B.SAT_ACT_NONE | B.SAT_FWD_INPUT_GLOBAL, out)
        B.sat_sync_status(ctx)
    finally:
        B.sat_destroy(ctx)
    return out


# one column tile to three with B resident; one tile more than there are pairs of SMs, where it is not (18,944 columns are 74 tiles)
@pytest.mark.parametrize("m,n,k", [(33000, 300, 256), (33000, 700, 256), (33000, 770, 192), (33000, 18944, 192), (33000, 18945, 192), (257, 38000, 384)])
def test_contraction_with_many_column_tiles(B, m, n, k):
    rng = np.random.default_rng(n)
    A, W, bias = (rng.standard_normal(s).astype(np.float32) for s in ((m, k), (k, n), (n,)))
    out = _rows_times(B, A, W, bias)
    tiles = -(-n // 256)
    width = -(-(-(-n // tiles)) // 32) * 32
    cols = np.unique(np.concatenate([np.arange(0, n, width), np.arange(width - 1, n, width), rng.integers(0, n, 60), [n - 1]]))
    got = out[:, dev(cols.astype(np.int64))].cpu().numpy()
    a, w = A.astype(np.float64), W[:, cols].astype(np.float64)
    assert (np.abs(got - (a @ w + bias[cols])) <= ((k + 3) * U + 2.0 ** -20) * (np.abs(a) @ np.abs(w) + np.abs(bias[cols]))).all()


def _sizes_bound(a, w):
    """Of |result - a w| for operands split into halves, every row of a and every column of w with a scale of its own: |x s - hi - lo| <= 2^-22 |x s| + 2^-25 with
    the largest |x s| of the row (column) at 2^14 or more."""
    a, w = np.abs(a), np.abs(w)
    return ((a.shape[1] + 3) * U + 2.0 ** -20) * (a @ w) + 2.0 ** -38 * (a.max(1, keepdims=True) * w.sum(0) + a.sum(1, keepdims=True) * w.max(0))


# halves; TF32 terms; halves in a large graph; terms beyond those that the packing keeps in registers
@pytest.mark.parametrize("m,n,k", [(200, 61, 384), (200, 61, 383), (33000, 40, 200), (130, 256, 1030)])
def test_columns_of_very_different_sizes(B, m, n, k):
    """A column of W next to ones that are 2^60 times larger is as precise as by itself, and one that is not finite stays by itself."""
    rng = np.random.default_rng(k)
    A = rng.standard_normal((m, k)).astype(np.float32)
    W = (rng.standard_normal((k, n)) * np.exp2(rng.integers(-30, 31, (1, n)))).astype(np.float32)
    bad = W.copy()
    for j, x in ((2, np.inf), (11, -np.inf), (n - 1, np.nan)):
        bad[rng.integers(0, k), j] = x
    out, with_bad = _rows_times(B, A, W).cpu().numpy()[:, :n], _rows_times(B, A, bad).cpu().numpy()[:, :n]
    sel = np.unique(np.concatenate([np.arange(130), rng.integers(0, m, 200)]))
    a, w = A[sel].astype(np.float64), W.astype(np.float64)
    assert (np.abs(out[sel] - a @ w) <= _sizes_bound(a, w)).all()
    ok = np.setdiff1d(np.arange(n), [2, 11, n - 1])
    assert np.array_equal(out[:, ok], with_bad[:, ok]) and not np.isfinite(with_bad[:, [2, 11, n - 1]]).any()


@pytest.mark.parametrize("m,d_in,d_out", [(200, 400, 390), (300, 1030, 1030), (33000, 200, 200)])
def test_input_gradient_with_features_of_very_different_sizes(B, m, d_in, d_out):
    """The same for the rows of W, one of which makes a column of the input gradient.  In a graph without edges P is the identity."""
    rng = np.random.default_rng(d_out)
    X, D = rng.standard_normal((m, d_in)).astype(np.float32), rng.standard_normal((m, d_out)).astype(np.float32)
    W = (rng.standard_normal((d_in, d_out)) * np.exp2(rng.integers(-30, 31, (d_in, 1)))).astype(np.float32)
    out, g_in, gW, gb = empty2d(m, d_out), empty2d(m, d_in), torch.empty((d_in, d_out), device="cuda"), torch.empty(d_out, device="cuda")
    ctx = B.sat_create(0, 0)
    try:
        B.sat_graph_load(ctx, np.zeros(m + 1, np.int64), np.zeros(0, np.int32))
        B.sat_partition(ctx, 1, B.SAT_PART_CONTIG_BLOCKS)
        B.sat_layer_fwd(ctx, B.SAT_ALL_PARTS, 2, dev2d(X), None, dev(W), None, B.SAT_ACT_NONE | B.SAT_FWD_INPUT_GLOBAL, out)
        B.sat_layer_bwd(ctx, B.SAT_ALL_PARTS, 2, dev2d(D), dev(W), gW, gb, 0, g_in, None)
        B.sat_sync_status(ctx)
    finally:
        B.sat_destroy(ctx)
    sel = np.unique(np.concatenate([np.arange(130), rng.integers(0, m, 200)]))
    a, w = D[sel].astype(np.float64), W.T.astype(np.float64)
    assert (np.abs(g_in.cpu().numpy()[sel][:, :d_in] - a @ w) <= _sizes_bound(a, w)).all()


@pytest.mark.parametrize("h", [8, 64])
def test_lstm_gates_of_very_different_sizes(B, h):
    """Forget gates that saturate through a weight of 2^30 leave the other gates' columns of Uh as precise as they are by themselves (bound of
    test_lstm_state_over_cached_projections; a saturated gate has no error)."""
    n, d, tau = 600, 16, 3
    ids = np.arange(n)
    col = np.sort(np.stack([(ids - 1) % n, (ids + 1) % n], 1), 1).astype(np.int32).ravel()
    rng = np.random.default_rng(h)
    W, Uh, b = rng.standard_normal((d, 4, h)) / d ** 0.5, rng.standard_normal((h, 4, h)) / h ** 0.5, rng.standard_normal((4, h)) / 4
    W[:, :, 0], Uh[:, :, 0], b[:, 0] = 0, 0, 2           # unit 0: a positive state
    Uh[:, 1, :] = 0
    Uh[0, 1, :] = 2.0 ** 30
    W, Uh, b = (x.reshape(-1, 4 * h).astype(np.float32) for x in (W, Uh, b))
    snaps = rng.standard_normal((tau, n, d)).astype(np.float32)
    ctx = B.sat_create(0, 0)
    try:
        B.sat_graph_load(ctx, 2 * np.arange(n + 1, dtype=np.int64), col)
        B.sat_partition(ctx, 2, B.SAT_PART_GIVEN, (ids % 2).astype(np.int32))
        B.sat_cache_init(ctx, [d], tau)
        perm = np.concatenate([np.flatnonzero(ids % 2 == m) for m in range(2)])
        out = empty2d(n, d)
        p = B.make_pred_params(dev(W), dev(Uh), dev(b.ravel()), dev(np.zeros((h, d), np.float32)), dev(np.zeros(d, np.float32)), h, 1)
        for x in snaps:
            B.sat_cache_update(ctx, B.SAT_ALL_PARTS, 1, dev2d(x[perm]))
            B.sat_cache_commit(ctx)
            B.sat_predict(ctx, 1, B.SAT_ALL_PARTS, p, 0, out)
        got = B.sat_predict_state(ctx, 1, n, h)[np.asarray(B.sat_slot_map(ctx, n)[1])]
        B.sat_sync_status(ctx)
    finally:
        B.sat_destroy(ctx)
    s, c, ds, dc = (np.zeros((n, h)) for _ in range(4))
    U64, eta = Uh.astype(np.float64), 2.0 ** -20
    for x in snaps.astype(np.float64):
        z = x @ W + s @ U64 + b
        e = ((d + h + 2) * U + 2.0 ** -20) * (np.abs(x) @ np.abs(W) + np.abs(s) @ np.abs(U64) + np.abs(b)) + ds @ np.abs(U64)
        (zi, zf, zg, zo), (ei, ef, eg, eo) = (np.split(v, 4, axis=1) for v in (z, e))
        ef = np.where(zf > 2.0 ** 20, 0.0, ef)
        sig = lambda v: 1 / (1 + np.exp(-np.minimum(v, 700)))
        g = np.tanh(zg)
        dc = np.abs(c) * (ef / 4 + eta) + dc + np.abs(g) * (ei / 4 + eta) + eg + eta
        c = sig(zf) * c + sig(zi) * g
        s = sig(zo) * np.tanh(c)
        ds = eo / 4 + eta + dc + eta
    assert (np.abs(got - s) <= ds).all()


def test_scales_whose_product_is_no_float(B):
    """Large elements that meet zeros on either side: the sum is zero although the product of the two scales overflows."""
    A, W = np.zeros((130, 384), np.float32), np.zeros((384, 40), np.float32)
    A[:, 0], W[1] = 2.0 ** 100, 2.0 ** 80
    assert (_rows_times(B, A, W).cpu().numpy()[:, :40] == 0.0).all()


# halves in a large graph (one column tile, two; a narrow layer) and in a small one, TF32 terms
@pytest.mark.parametrize("n,k,m", [(33000, 200, 200), (33000, 256, 300), (33000, 383, 20), (600, 384, 64), (600, 200, 200)])
def test_the_push_does_not_change_the_layer(B, n, k, m):
    """sat_layer_fwd with SAT_FWD_PUSH = without, then sat_cache_update: output and ring, bit for bit, behind the first layer too."""
    ids = np.arange(n)
    col = np.sort(np.stack([(ids - 1) % n, (ids + 1) % n], 1), 1).astype(np.int32).ravel()
    rng = np.random.default_rng(k)
    X, W, b = dev2d(rng.standard_normal((n, k)).astype(np.float32)), dev(rng.standard_normal((k, m)).astype(np.float32)), dev(rng.standard_normal(m).astype(np.float32))
    act, rows = B.SAT_ACT_RELU | B.SAT_FWD_INPUT_GLOBAL, []
    ctx = B.sat_create(0, 0)
    try:
        B.sat_graph_load(ctx, 2 * np.arange(n + 1, dtype=np.int64), col)
        B.sat_partition(ctx, 2, B.SAT_PART_GIVEN, (ids % 2).astype(np.int32))       # every node is a boundary node
        B.sat_cache_init(ctx, [8, m], 1)
        outs = [empty2d(n, m) for _ in range(2)]
        for push, out in zip((0, B.SAT_FWD_PUSH), outs):
            B.sat_layer_fwd(ctx, B.SAT_ALL_PARTS, 2, X, None, W, b, act | push, out)
            if not push:
                B.sat_cache_update(ctx, B.SAT_ALL_PARTS, 2, out)
            rows.append(B.sat_cache_read(ctx, 2, -1, n, m))
            B.sat_cache_update(ctx, B.SAT_ALL_PARTS, 2, dev2d(np.zeros((n, m), np.float32)))
        B.sat_sync_status(ctx)
    finally:
        B.sat_destroy(ctx)
    assert torch.equal(outs[0], outs[1]) and np.array_equal(rows[0], rows[1]) and rows[0].any()


def _input_gradients(B, A, part, d_in, d_out, hist, seed):
    """G_in of layer 2 under the mask of layer 1 with (hist) and without stale rows: all partitions at once, one after the other, the value in fp64 and
    a bound of the error (that of test_input_gradient_in_both_orders, and what halves lose)."""
    n, M = A.shape[0], int(part.max()) + 1
    Pm = _propagation(A).tocoo()
    rng = np.random.default_rng(seed)
    perm = np.concatenate([np.flatnonzero(part == m) for m in range(M)])
    off = np.concatenate([[0], np.cumsum(np.bincount(part, minlength=M))])
    W1, W2 = (rng.standard_normal(s).astype(np.float32) for s in ((8, d_in), (d_in, d_out)))
    X, D = rng.standard_normal((n, 8)).astype(np.float32), rng.standard_normal((n, d_out)).astype(np.float32)
    ctx = B.sat_create(0, 0)
    try:
        B.sat_graph_load(ctx, A.indptr.astype(np.int64), A.indices.astype(np.int32))
        B.sat_partition(ctx, M, B.SAT_PART_GIVEN, part)
        B.sat_cache_init(ctx, [d_in], 2)
        _, slot, n_slots = B.sat_slot_map(ctx, n)
        n_halo = B.sat_part_sizes(ctx, B.SAT_ALL_PARTS)[1]
        H1, H2, g_in, one = empty2d(n, d_in), empty2d(n, d_out), empty2d(n, d_in), empty2d(n, d_in)
        B.sat_layer_fwd(ctx, B.SAT_ALL_PARTS, 1, dev2d(X), None, dev(W1), None, B.SAT_ACT_RELU | B.SAT_FWD_INPUT_GLOBAL, H1)
        B.sat_layer_fwd(ctx, B.SAT_ALL_PARTS, 2, H1, dev2d(np.zeros((n_halo, d_in), np.float32)), dev(W2), None, B.SAT_ACT_NONE, H2)
        Q = np.zeros((n_slots, d_out), np.float32)
        if hist:
            Q = (4 * rng.standard_normal((n_slots, d_out))).astype(np.float32)       # larger than the rows that they are added to
            B.sat_grad_history_write(ctx, 2, d_out, Q)
        flags = B.SAT_BWD_MASK_G_IN | (B.SAT_BWD_GRAD_HISTORY if hist else 0)
        gW, gb, Dd = torch.empty((d_in, d_out), device="cuda"), torch.empty(d_out, device="cuda"), dev2d(D[perm])
        B.sat_layer_bwd(ctx, B.SAT_ALL_PARTS, 2, Dd, dev(W2), gW, gb, flags, g_in, None)
        for m in range(M):
            r = slice(off[m], off[m + 1])
            B.sat_layer_bwd(ctx, m, 2, Dd[r], dev(W2), gW, gb, flags, one[r], None)
        B.sat_sync_status(ctx)
        keep = H1.cpu().numpy()[:, :d_in] > 0
    finally:
        B.sat_destroy(ctx)
    same = sp.csr_matrix((Pm.data * (part[Pm.row] == part[Pm.col]), (Pm.row, Pm.col)), shape=Pm.shape)
    slot = np.asarray(slot)
    stale = np.where((slot >= 0)[:, None], Q[np.maximum(slot, 0)], 0.0)
    rows, mag, w = (same @ D.astype(np.float64) + stale)[perm], (abs(same) @ np.abs(D.astype(np.float64)) + np.abs(stale))[perm], np.abs(W2.T).astype(np.float64)
    terms = np.diff(A.indptr).max() + d_out + 8
    bound = (terms * U + 2.0 ** -20) * (mag @ w) + 2.0 ** -38 * (mag.max(1, keepdims=True) * w.sum(0) + mag.sum(1, keepdims=True) * w.max(0))
    return g_in, one, (rows @ W2.T.astype(np.float64)) * keep, bound


@pytest.mark.parametrize("d_in,d_out", [(40, 40), (72, 17), (400, 384)])
def test_input_gradient_of_a_partition_without_cut_edges(B, d_in, d_out):
    """A partition that has no boundary rows, and so no stale ones, adds up as in the call on all partitions, where others have them."""
    n = 1500
    A = sp.block_diag([_graph(HUBS[:8], n), _graph([30, 200], 600)]).tocsr()
    part = np.concatenate([np.random.default_rng(3).integers(0, 2, n), np.full(600, 2)]).astype(np.int32)
    g_in, one, want, bound = _input_gradients(B, A, part, d_in, d_out, True, d_out)
    assert torch.equal(g_in, one)
    assert (np.abs(g_in.cpu().numpy()[:, :d_in] - want) <= bound).all()


# halves behind the product, whose rows' sizes come from one launch or two, one slice of columns or several, stale rows among them
@pytest.mark.parametrize("hist", [False, True])
@pytest.mark.parametrize("kind", ["hub", "large"])
@pytest.mark.parametrize("d_in,d_out", [(400, 384), (520, 512), (602, 401)])
def test_wide_input_gradient(B, kind, d_in, d_out, hist):
    A = _many_runs(kind)
    part = np.random.default_rng(5).integers(0, 2, A.shape[0]).astype(np.int32)
    g_in, one, want, bound = _input_gradients(B, A, part, d_in, d_out, hist, d_in)
    assert torch.equal(g_in, one)
    assert (np.abs(g_in.cpu().numpy()[:, :d_in] - want) <= bound).all()


# graphs of at least 32,768 nodes take the product first at any width below d_in: on CUDA cores (with the mask) below 16 columns, TF32 terms, halves
@pytest.mark.parametrize("d_in,d_out", [(200, 5), (33, 15), (200, 17), (200, 192), (192, 192)])
def test_input_gradient_in_a_large_graph(B, d_in, d_out):
    n = 33000
    rng = np.random.default_rng(d_out)
    A = _graph([9000, 300, 40], n)
    part = rng.integers(0, 3, n).astype(np.int32)
    g_in, one, want, bound = _input_gradients(B, A, part, d_in, d_out, False, d_out)
    assert torch.equal(g_in, one)
    assert (np.abs(g_in.cpu().numpy()[:, :d_in] - want) <= bound).all()


@pytest.mark.parametrize("parts", [False, True])
@pytest.mark.parametrize("route", ["layer", "update", "attention"])
@pytest.mark.parametrize("kind,d", [("hub", 400), ("hub", 1000), ("large", 400), ("ring", 200)])     # rows of one launch and of two, one to four slices of columns
def test_every_push_leaves_the_sizes_of_its_rows(B, kind, d, route, parts):
    """A prediction from pushed rows does not look for their sizes again (as many launches as the next one) and is the one from the same rows when they have
    been imported, whose sizes are looked for, bit for bit."""
    if kind == "ring":
        n = 33000
        ids = np.arange(n)
        col = np.sort(np.stack([(ids - 1) % n, (ids + 1) % n], 1), 1).astype(np.int32).ravel()
        A = sp.csr_matrix((np.ones(2 * n), col, 2 * np.arange(n + 1)), shape=(n, n))
    else:
        A = _many_runs(kind)
        n = A.shape[0]
    rng, M, h, k = np.random.default_rng(d), 2, 32, 8
    part = rng.integers(0, M, n).astype(np.int32)
    rand = lambda *s: dev(rng.standard_normal(s).astype(np.float32) / 8)
    ctx = B.sat_create(0, 0)
    try:
        B.sat_graph_load(ctx, A.indptr.astype(np.int64), A.indices.astype(np.int32))
        B.sat_partition(ctx, M, B.SAT_PART_GIVEN, part)
        B.sat_cache_init(ctx, [d], 1)
        sizes, n_slots = [B.sat_part_sizes(ctx, m) for m in range(M)], B.sat_slot_map(ctx, n)[2]
        n_halo = sum(s[1] for s in sizes)
        spread = np.exp2(rng.integers(-9, 9, (n, 1)))
        X, halo, Y = dev2d((rng.standard_normal((n, k)) * spread).astype(np.float32)), dev2d(rng.standard_normal((n_halo, k)).astype(np.float32)), empty2d(n, d)
        W, a1, a2, b = rand(k, d), 1e-3 * rand(d), 1e-3 * rand(d), rand(d)
        W1 = dev(rng.standard_normal((16, d)).astype(np.float32) * np.exp2(rng.integers(0, 9, (16, 1))).astype(np.float32))
        X1 = dev2d((rng.standard_normal((n, 16)) * spread).astype(np.float32))
        p = B.make_pred_params(rand(d, 4 * h) / 64, rand(h, 4 * h), rand(4 * h), rand(h, d), rand(d), h, 0, B.SAT_CELL_LSTM)
        out, counts = [empty2d(n_halo, d) for _ in range(4)], []

        def predict(i):
            at = B.sat_launch_count(ctx)
            B.sat_predict(ctx, 1, B.SAT_ALL_PARTS, p, 0, out[i])
            counts.append(B.sat_launch_count(ctx) - at)

        B.sat_cache_commit(ctx)          # a snapshot of zeros, and the lists that a first prediction makes
        B.sat_predict(ctx, 1, B.SAT_ALL_PARTS, p, 0, out[0])
        push = B.SAT_ACT_RELU | B.SAT_FWD_PUSH
        r0 = u0 = 0
        for m in range(M) if parts else [B.SAT_ALL_PARTS]:
            r1, u1 = (r0 + sizes[m][0], u0 + sizes[m][1]) if parts else (n, n_halo)
            if route == "layer":
                B.sat_layer_fwd(ctx, m, 1, X1, None, W1, b, push | B.SAT_FWD_INPUT_GLOBAL, Y[r0:r1])
            elif route == "attention":
                B.sat_gat_fwd(ctx, m, 1, X[r0:r1], halo[u0:u1], W, a1, a2, b, push, Y[r0:r1])
            else:
                Y[r0:r1] = dev((rng.standard_normal((r1 - r0, d)) * spread[:r1 - r0]).astype(np.float32))
                B.sat_cache_update(ctx, m, 1, Y[r0:r1])
            r0, u0 = r1, u1
        B.sat_cache_commit(ctx)
        predict(0)
        predict(1)
        state, ring = B.sat_cache_state(ctx), B.sat_cache_export(ctx, 1, 1, n_slots, d)
        B.sat_cache_import(ctx, 1, ring)
        B.sat_cache_set_state(ctx, *state)
        predict(2)
        predict(3)
        S = B.sat_predict_state(ctx, 1, n_slots, h)
        B.sat_sync_status(ctx)
    finally:
        B.sat_destroy(ctx)
    assert counts[0] == counts[1] == counts[3] == counts[2] - 1
    assert all(torch.equal(out[0], o) for o in out[1:]) and np.isfinite(S).all() and S.any()


@pytest.mark.parametrize("row,column", [(-60, 115), (60, -100), (60, 60), (-60, -58), (100, 0), (-110, 100), (110, -95)])
def test_rows_and_columns_far_from_one(B, row, column):
    """Rows of A near 2^row, columns of W near 2^column: the result is a float, and so is what the scales of either leave on the way."""
    rng = np.random.default_rng(7)
    A, W = (rng.uniform(0.25, 1, s) * rng.choice([-1, 1], s) for s in ((130, 384), (384, 40)))
    A, W = (A * 2.0 ** row).astype(np.float32), (W * 2.0 ** column).astype(np.float32)
    out = _rows_times(B, A, W).cpu().numpy()[:, :40]
    a, w = A.astype(np.float64), W.astype(np.float64)
    assert (np.abs(out - a @ w) <= _sizes_bound(a, w)).all()

"""Codebook training on the device (paper Section 3.6) against the oracle's trainer.

Given the same samples the two do the same arithmetic in the same order (exact assignment in double,
cells summed in sample order), so the mean-squared-distance trace, the number of updates and the
final f32 codebook must agree -- the trace to a summation-order tolerance (the oracle adds the
distances in a thread-parallel order), the codebook exactly.
"""
import numpy as np
import pytest
import torch

from conftest import load_golden_codebook

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2605_26339_b200 import binding as q

DEV = "cuda:0"


@pytest.mark.parametrize("K,n,iters", [(1, 4096, 3), (2, 5000, 20), (64, 1 << 14, 25), (256, 1 << 16, 12), (4096, 1 << 15, 4)])
def test_training_on_the_oracles_samples_reproduces_the_oracle(orc, K, n, iters):
    samples = orc.gauss_pairs(9, n)
    ref_cb, ref_mse, ref_iters, ref_trace = orc.train_codebook(K, n, 9, iters, 1e-7, want_trace=True)
    out = q.train_codebook_gpu(K, max_iters=iters, rel_tol=1e-7, samples=torch.from_numpy(samples).to(DEV))
    assert out["iters"] == ref_iters and len(out["trace"]) == len(ref_trace)
    np.testing.assert_allclose(out["trace"], ref_trace, rtol=1e-12)
    assert np.array_equal(out["codebook"], ref_cb)
    assert abs(out["mse"] - ref_mse) <= 1e-12 * ref_mse
    if K == 1:  # one cell: its codeword is the sample mean, the distortion the total variance
        assert np.allclose(out["codebook"][0], samples.mean(0), atol=1e-7)


def test_assignment_and_centroids_of_one_iteration(orc):
    """One update from a known codebook: the new codewords are the means of the oracle's cells."""
    n, K = 20000, 32
    samples = orc.gauss_pairs(3, n)
    out = q.train_codebook_gpu(K, max_iters=1, rel_tol=0.0, samples=torch.from_numpy(samples).to(DEV))
    cb0 = np.sqrt(2.0) * samples[:K]
    assign, mse0 = orc.lloyd_assign(samples, cb0)
    assert abs(out["trace"][0] - mse0) <= 1e-12 * mse0
    want = cb0.copy()
    for c in range(K):
        if (assign == c).any():
            want[c] = samples[assign == c].mean(0)
    order = np.lexsort((np.arctan2(want[:, 1], want[:, 0]), (want ** 2).sum(1)))
    assert np.allclose(out["codebook"], want[order].astype(np.float32), atol=1e-6)


def test_device_generated_samples_give_the_golden_codebook_quality(orc):
    """Without a sample array the device draws the counter-based Gaussian stream itself (its log / sin /
    cos may differ from the host's in the last bit, so codewords are compared to a tolerance) and the
    trained codebook has the distortion of the oracle-trained golden one."""
    K = 256
    hdr_mse = orc.codebook_mse(load_golden_codebook(K), 1 << 16, 1234)
    out = q.train_codebook_gpu(K, 1 << 20, 0, 100, 1e-6)
    assert abs(orc.codebook_mse(out["codebook"], 1 << 16, 1234) - hdr_mse) < 0.01 * hdr_mse
    host_cb, host_mse = q.train_codebook(K, 1 << 20, 0, 100, 1e-6)
    assert abs(out["mse"] - host_mse) < 1e-6 * host_mse
    assert np.abs(out["codebook"] - host_cb).max() < 1e-4
    print(f"LLOYD K={K}: device {out['seconds']:.3f} s, {out['iters']} updates")
    again = q.train_codebook_gpu(K, 1 << 20, 0, 100, 1e-6)
    assert np.array_equal(again["codebook"], out["codebook"])  # reproducible run to run


def test_codebook_fitted_to_a_matrix_beats_the_gaussian_one_on_it(orc):
    """Per-matrix codebook (Lloyd on the matrix's own rotated, scaled pairs): its quantisation error on
    those pairs is not above the Gaussian-trained codebook's, and the device trainer's result on the
    pairs equals the oracle trainer's."""
    from paper_2605_26339_b200.model_codec import fit_codebook
    g = torch.Generator().manual_seed(12)
    d_out, d_in, K = 512, 1024, 64
    # light-tailed rows (uniform entries): after a block-32 rotation the pairs are visibly non-Gaussian
    W = ((torch.rand((d_out, d_in), generator=g) - 0.5) * torch.exp(0.5 * torch.randn((d_out, 1), generator=g))).to(DEV)
    fit = fit_codebook(W, None, 0.0, 2, K, n_pairs=1 << 16, max_iters=40, rel_tol=1e-7)
    assert fit["codebook"].shape == (K, 2) and np.isfinite(fit["codebook"]).all()
    # the same pairs through the oracle: same codebook
    rows = (np.arange(fit["rows"]) * d_out) // fit["rows"]
    signs = q.make_signs(q.DEFAULT_SIGN_SEED, d_in)
    Wh = W.cpu().numpy()
    y = np.stack([orc.front_row(Wh[r], 2, None, signs)[0] for r in rows])
    z = (y.reshape(len(rows), d_in // 2, 2) / fit["sigma"].cpu().numpy()[None, :, None]).reshape(-1, 2)[: 1 << 16]
    ref_cb, ref_mse, _, _ = orc.train_codebook_on(z.astype(np.float64), K, 40, 1e-7)
    assert np.array_equal(fit["codebook"], ref_cb)
    gauss = load_golden_codebook(K)
    _, mse_gauss = orc.lloyd_assign(z.astype(np.float64), gauss.astype(np.float64))
    assert fit["mse"] < mse_gauss


@pytest.mark.parametrize("K,n", [(2, 1027), (32, 255), (64, 256), (128, 257), (32, 511), (512, 513), (16, 4095), (256, 4096),
                                 (1024, 4097), (2048, 9000)])
def test_tiles_and_chunks_that_do_not_fill(orc, K, n):
    """Sample counts around the edges of the spatial tiles (256) and sorting chunks (4096), every number of
    codewords per thread, samples with far outliers, exact duplicates and ties: same codebook as the oracle."""
    rng = np.random.default_rng(K + n)
    z = np.round(rng.standard_normal((n, 2)) * 8) / 8 + (rng.standard_normal((n, 2)) * 1e-3) * (rng.random((n, 1)) < 0.7)
    z[rng.integers(0, n, 5)] *= 1e4
    ref_cb, ref_mse, ref_iters, _ = orc.train_codebook_on(z, K, 9, 1e-9)
    out = q.train_codebook_gpu(K, max_iters=9, rel_tol=1e-9, samples=torch.from_numpy(z).to(DEV))
    assert out["iters"] == ref_iters and np.array_equal(out["codebook"], ref_cb)
    assert abs(out["mse"] - ref_mse) <= 1e-12 * ref_mse


@pytest.mark.parametrize("kind,K,n,iters", [
    ("plain", 64, 70000, 40),      # cells of more than one chunk of the merge
    ("plain", 64, 1152 * 64, 12),  # the largest cells that are updated incrementally,
    ("plain", 64, 1153 * 64, 12),  # and the smallest that are not
    ("plain", 2048, 60000, 60),    # tiles as wide as many codewords
    ("plain", 4096, 40000, 30),
    ("ties", 256, 20000, 40),      # a lattice: equal distances, equal samples, empty cells
    ("outliers", 512, 30001, 40),  # boxes that hold half of the codebook
    ("late", 128, 60000, 40),      # codewords that start in one place: cells still move when the incremental passes begin
    ("point", 64, 3000, 20),       # one sample many times
])
def test_incremental_updates(orc, kind, K, n, iters):
    """Training that goes on after the passes in full: the same codebook, updates and errors as the oracle.  (With a tolerance of zero
    the rule would compare errors that differ in the order of their sums only.)"""
    rng = np.random.default_rng(K + n)
    z = rng.standard_normal((n, 2))
    if kind == "ties":
        z = np.round(z * 6) / 6
    elif kind == "outliers":
        z[rng.integers(0, n, n // 50)] *= 30.0
    elif kind == "late":
        z[:K] = 4.0 + 1e-3 * z[:K]
    elif kind == "point":
        z[:] = z[0]
    ref_cb, ref_mse, ref_iters, ref_trace = orc.train_codebook_on(z, K, iters, 1e-12)
    out = q.train_codebook_gpu(K, max_iters=iters, rel_tol=1e-12, samples=torch.from_numpy(z).to(DEV))
    assert out["iters"] == ref_iters and np.array_equal(out["codebook"], ref_cb)
    assert abs(out["mse"] - ref_mse) <= 1e-12 * ref_mse
    again = q.train_codebook_gpu(K, max_iters=iters, rel_tol=1e-12, samples=torch.from_numpy(z).to(DEV))
    assert np.array_equal(again["codebook"], out["codebook"]) and np.array_equal(again["trace"], out["trace"])


def _repeated_passes(orc, z, K, iters, rel_tol):
    """Which incremental passes run out of room, by the oracle's assignments and the library's limits: (pass, limit that it meets,
    incremental updates before it in its batch)."""
    import os
    import re
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    src = open(os.path.join(root, "paper_2605_26339_b200", "csrc", "qamw_lloyd.cu")).read()
    first, again, batch, most = (int(re.search(rf"constexpr int {c} = (\d+);", src)[1])
                                 for c in ("kFullFirst", "kFullAgain", "kBatch", "kChanges"))
    n, cb, found = len(z), np.sqrt(2.0) * z[:K], []
    full, before, in_batch, changes_in_batch, updates, last = first, None, 0, 0, 0, None
    while True:
        cell, err = orc.lloyd_assign(z, cb)
        count = np.bincount(cell, minlength=K)
        if full == 0:
            moved = cell != before
            came, left = np.bincount(cell[moved], minlength=K), np.bincount(before[moved], minlength=K)
            what = "changes" if max(came.max(), left.max()) > most else "slots" if (size + came > slots)[came > 0].any() else None
            if what:
                found.append((updates, what, changes_in_batch))
                full, in_batch, changes_in_batch = again, 0, 0
                continue
            changes_in_batch += 1
        if last is not None and last - err <= rel_tol * last or updates >= iters:
            return found
        last, before, size = err, cell, count
        updates, in_batch = updates + 1, (in_batch + 1) % batch
        if in_batch == 0:
            changes_in_batch = 0
        total = np.zeros((K, 2))
        np.add.at(total, cell, z)
        cb = np.where(count[:, None] > 0, total / np.maximum(count, 1)[:, None], cb)
        if full and (full := full - 1) == 0:
            start = np.concatenate([[0], np.cumsum(count)])  # a quarter, and 64 and a quarter of the mean, to grow by
            slots = np.diff(start + start // 4 + (64 + n // K // 4) * np.arange(K + 1))


@pytest.mark.parametrize("K,n,iters,limits", [(128, 60000, 40, {"changes", "slots"}), (64, 20000, 40, {"changes", "slots"}),
                                              (128, 10000, 60, {"slots"}), (256, 60000, 60, {"changes", "slots"})])
def test_incremental_passes_that_run_out_of_room(orc, K, n, iters, limits):
    """Codewords that start in one place: passes in which more samples change cells than a pass may report, or cells outgrow
    their slots, are repeated in full, once and again: the same codebook, updates and errors as the oracle."""
    z = np.random.default_rng(K + n).standard_normal((n, 2))
    z[:K] = 4.0 + 1e-3 * z[:K]
    repeated = _repeated_passes(orc, z, K, iters, 1e-12)
    assert len(repeated) > 1 and {what for _, what, _ in repeated} == limits
    ref_cb, ref_mse, ref_iters, ref_trace = orc.train_codebook_on(z, K, iters, 1e-12)
    out = q.train_codebook_gpu(K, max_iters=iters, rel_tol=1e-12, samples=torch.from_numpy(z).to(DEV))
    assert out["iters"] == ref_iters and np.array_equal(out["codebook"], ref_cb)
    np.testing.assert_allclose(out["trace"], ref_trace, rtol=1e-12)
    assert abs(out["mse"] - ref_mse) <= 1e-12 * ref_mse


def test_samples_still_on_their_way_on_another_stream():
    """Samples that a stream of the caller's is still writing when the call is made: the call waits for them."""
    g = torch.Generator(device=DEV)
    g.manual_seed(5)
    z = torch.randn((20000, 2), generator=g, device=DEV, dtype=torch.float64)
    want = q.train_codebook_gpu(64, max_iters=5, rel_tol=0.0, samples=z)
    late = torch.zeros_like(z)
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.Stream()):
        torch.cuda._sleep(50_000_000)  # clocks: some 25 ms
        late.copy_(z)
        got = q.train_codebook_gpu(64, max_iters=5, rel_tol=0.0, samples=late)
    assert np.array_equal(got["codebook"], want["codebook"]) and np.array_equal(got["trace"], want["trace"])


def test_scratch_kept_between_calls_is_bounded_and_given_back():
    """Device memory that training with passes in full holds on to: at most 256 MB whatever a call needed, none after release_scratch, and
    the next call works as before."""
    q.train_codebook_gpu(16, 1 << 12, 0, 1)  # contexts, modules
    q.release_scratch()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    slack = 4 << 20
    first = q.train_codebook_gpu(256, 1 << 20, 0, 2)  # 60 MB of scratch
    kept = free - torch.cuda.mem_get_info()[0]
    assert (40 << 20) <= kept <= (256 << 20)
    q.train_codebook_gpu(256, 1 << 23, 0, 1)  # 480 MB
    assert free - torch.cuda.mem_get_info()[0] <= (256 << 20) + slack
    q.release_scratch()
    assert free - torch.cuda.mem_get_info()[0] <= slack
    q.release_scratch()
    assert np.array_equal(q.train_codebook_gpu(256, 1 << 20, 0, 2)["codebook"], first["codebook"])
    q.release_scratch()


def test_little_device_memory():
    """A call with memory for the passes in full but not for incremental updates: the same result, and the next one as before."""
    K, n = 2048, 1 << 22  # 190 MB, or 420
    g = torch.Generator(device=DEV)
    g.manual_seed(7)
    z = torch.randn((n, 2), generator=g, device=DEV, dtype=torch.float64)
    want = q.train_codebook_gpu(K, max_iters=12, rel_tol=0.0, samples=z)
    q.release_scratch()
    torch.cuda.empty_cache()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - (300 << 20), dtype=torch.uint8, device=DEV)
    try:
        got = q.train_codebook_gpu(K, max_iters=12, rel_tol=0.0, samples=z)
    finally:
        del hold
        torch.cuda.empty_cache()
    for out in (got, q.train_codebook_gpu(K, max_iters=12, rel_tol=0.0, samples=z)):
        assert np.array_equal(out["codebook"], want["codebook"]) and np.array_equal(out["trace"], want["trace"])
    q.release_scratch()


@pytest.mark.parametrize("iters,needed", [(7, 43), (8, 110)])
def test_scratch_of_a_call_without_incremental_updates(orc, iters, needed):
    """Eight passes in full come first: a call of up to seven updates (and the last assignment) takes memory for these alone,
    43 MB at 2^20 samples and K = 2048; one that goes on takes 110.  (A pool grows by 32 MB at a time.)"""
    K, n = 2048, 1 << 20
    z = torch.from_numpy(orc.gauss_pairs(4, n)).to(DEV)
    q.train_codebook_gpu(K, max_iters=9, rel_tol=0.0, samples=z[: 1 << 14])
    q.release_scratch()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    q.train_codebook_gpu(K, max_iters=iters, rel_tol=0.0, samples=z)
    kept = free - torch.cuda.mem_get_info()[0]
    q.release_scratch()
    assert needed <= kept >> 20 <= needed + 32


def test_scratch_of_incremental_updates_is_kept():
    """Calls of up to some 6 million samples find their scratch memory in the pool the next time; larger ones leave at most 640 MB
    there, and after release_scratch the limit of passes in full holds again."""
    K, n = 2048, 1 << 22  # 401 MB
    g = torch.Generator(device=DEV)
    g.manual_seed(7)
    z = torch.randn((9 << 20, 2), generator=g, device=DEV, dtype=torch.float64)  # 9 million: 880 MB
    q.train_codebook_gpu(K, max_iters=9, rel_tol=0.0, samples=z[: 1 << 14])
    q.release_scratch()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]

    def kept(K, n, iters):
        q.train_codebook_gpu(K, max_iters=iters, rel_tol=0.0, samples=z[:n])
        return (free - torch.cuda.mem_get_info()[0]) >> 20

    assert 401 <= kept(K, n, 9) <= 640 and 401 <= kept(K, n, 9) <= 640
    assert kept(K, 9 << 20, 9) <= 644
    q.release_scratch()
    assert kept(256, 8 << 20, 1) <= 260
    q.release_scratch()
    assert (free - torch.cuda.mem_get_info()[0]) >> 20 <= 4

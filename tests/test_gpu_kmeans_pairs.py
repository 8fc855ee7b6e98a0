"""K-means step with up to four clusters, which takes a warp's points two at a time: last pairs without a partner, every dimension, ties."""
import numpy as np
import pytest
import torch

from gpu_util import DEV

pytestmark = pytest.mark.gpu


# n around one and two points per warp (148 SMs x 8, 12 or 16 warps), k below the compiled bound
@pytest.mark.parametrize("n", [1, 2, 1775, 1777, 2369, 3553, 4736, 7105])
@pytest.mark.parametrize("dim,k", [(128, 4), (256, 3), (384, 4), (384, 1), (512, 2)])
def test_pairs_are_exact_on_small_integers(n, dim, k):
    """Components are integers of -2..2: every distance and sum is exact in fp32, so labels (ties to the lowest index), counts, centroids
    (one rounding of a double quotient) and inertia have to be equal.  Points of NaN and of infinity are nearest to nothing: label 0."""
    from paper_2505_08600_b200 import binding as sd
    rng = np.random.default_rng(n * 1000 + dim + k)
    x = rng.integers(-2, 3, (n, dim)).astype(np.float32)
    x[:, 8:] = 0                                      # few free components: many ties
    c = rng.integers(-2, 3, (k, dim)).astype(np.float32)
    d = ((x[:, None, :8].astype(np.float64) - c[None, :, :8]) ** 2).sum(2) + (c[:, 8:].astype(np.float64) ** 2).sum(1)
    want = d.argmin(1)
    counts = np.bincount(want, minlength=k)
    sums = np.stack([x[want == j].astype(np.float64).sum(0) for j in range(k)])
    centroids = np.where(counts[:, None] > 0, (sums / np.maximum(counts, 1)[:, None]).astype(np.float32), c)

    def run(points):
        labels = torch.full((n,), -1, dtype=torch.int32, device=DEV)
        out, cnt = torch.zeros((k, dim), device=DEV), torch.zeros(k, dtype=torch.int64, device=DEV)
        inertia = torch.zeros(1, dtype=torch.float64, device=DEV)
        sd.sd_kmeans_step(torch.from_numpy(points).to(DEV), torch.from_numpy(c).to(DEV), labels, out, cnt, inertia)
        torch.cuda.synchronize()
        return labels.cpu().numpy(), out.cpu().numpy(), cnt.cpu().numpy(), inertia.item()

    labels, out, cnt, inertia = run(x)
    assert np.array_equal(labels, want) and np.array_equal(cnt, counts) and np.array_equal(out, centroids)
    assert inertia == d.min(1).sum()
    x[n - 1] = np.nan                                 # the last point, beside a partner or alone
    x[n // 2, 0] = np.inf
    want[[n - 1, n // 2]] = 0
    labels, _, cnt, _ = run(x)
    assert np.array_equal(labels, want) and np.array_equal(cnt, np.bincount(want, minlength=k))


@pytest.mark.parametrize("dim,k,warps", [(384, 4, 1776), (512, 3, 1184)])
@pytest.mark.parametrize("per_warp,extra", [(128, 0), (128, 1), (129, 0), (130, -1), (256, 0), (257, 3)])
def test_runs_of_sums_hold_every_point_once(dim, k, warps, per_warp, extra):
    """A warp's sums are moved away every 128 points: numbers of points just at and beyond that, in all and in some warps; small integers,
    as above."""
    from paper_2505_08600_b200 import binding as sd
    n = per_warp * warps + extra
    g = torch.Generator(device=DEV)
    g.manual_seed(n + dim)
    x = torch.zeros((n, dim), device=DEV)
    x[:, :8] = torch.randint(-2, 3, (n, 8), generator=g, device=DEV).float()
    c = torch.zeros((k, dim), device=DEV)
    c[:, :8] = torch.randint(-2, 3, (k, 8), generator=g, device=DEV).float()
    labels = torch.full((n,), -1, dtype=torch.int32, device=DEV)
    out, cnt, inertia = torch.zeros((k, dim), device=DEV), torch.zeros(k, dtype=torch.int64, device=DEV), torch.zeros(1, dtype=torch.float64, device=DEV)
    sd.sd_kmeans_step(x, c, labels, out, cnt, inertia)
    d = ((x[:, None, :8].double() - c[None, :, :8].double()) ** 2).sum(2)
    near = d.min(1).values
    want = torch.stack([torch.where(d[:, j] == near, j, k) for j in range(k)], 1).min(1).values
    assert torch.equal(labels.long(), want) and torch.equal(cnt, torch.bincount(want, minlength=k)) and inertia.item() == near.sum().item()
    for j in range(k):
        assert torch.equal(out[j], (x[want == j].double().sum(0) / max(1, int(cnt[j]))).float() if cnt[j] else c[j])


@pytest.mark.parametrize("dim", [384, 512])
def test_sums_are_as_precise_as_those_of_two_blocks_per_sm(dim):
    """A million copies of one point: every addition of a warp's running fp32 sum rounds the same way, so that the centroid is off in
    proportion to the points in one sum.  No more than with 2,368 warps of n / 2368 points each, added by eights."""
    from paper_2505_08600_b200 import binding as sd
    n = 1_000_000
    v = np.random.default_rng(1).uniform(1, 2, dim).astype(np.float32)
    run = np.zeros_like(v)
    for _ in range(n // 2368):
        run += v
    block = np.zeros_like(v)
    for _ in range(8):
        block += run
    bound = np.linalg.norm(block.astype(np.float64) / (n // 2368 * 8) - v) / np.linalg.norm(v)
    x = torch.from_numpy(v).to(DEV).repeat(n, 1)
    labels, out = torch.empty(n, dtype=torch.int32, device=DEV), torch.zeros((4, dim), device=DEV)
    sd.sd_kmeans_step(x, torch.stack([x[0]] * 4), labels, out)
    assert np.linalg.norm(out[0].cpu().numpy().astype(np.float64) - v) / np.linalg.norm(v) <= 1.05 * bound      # (a few more points in some sums)

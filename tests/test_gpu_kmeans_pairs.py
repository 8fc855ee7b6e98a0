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

"""The screen's bound by the copies' own distance, on the CPU: for BF16 and e4m3 copies c of
seeded box coordinates u, |u_i - u_s| >= |c_i - c_s| - 2 E over all coordinates and over a prefix,
E the largest |u - c| of the node set, and what the device adds for float32 and tensor-core
rounding of |c_i|^2 + |c_s|^2 - 2 G (2^-9 |c_i||c_s|, 10 % slack) covers a float32 accumulation."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("kind", ["bf16", "e4m3"])
@pytest.mark.parametrize("r,R", [(65, 0.3), (300, 0.3), (1000, 0.3), (1000, 2.4)])
def test_distance_of_copies_bounds_distance(kind, r, R):
    rng = np.random.default_rng(r)
    n = 400
    u = (R * (2.0 * rng.random((n, r)) - 1.0)).astype(np.float32)
    u[1] = u[0] * np.float32(1.0 + 2.0 ** -9)          # near neighbours, where the margin is all there is
    s = 1.0 if kind == "bf16" else 2.0 ** np.floor(np.log2(448.0 / (8.0 * R)))
    t = torch.from_numpy(u * np.float32(s))
    c = t.to(torch.bfloat16 if kind == "bf16" else torch.float8_e4m3fn).to(torch.float64).numpy() / s
    E = np.sqrt(((u.astype(np.float64) - c) ** 2).sum(1)).max()
    for k in (64, 128, r):
        uu, cc = u[:, :k].astype(np.float64), c[:, :k]
        du = np.sqrt(((uu[:, None] - uu[None]) ** 2).sum(2))
        dc = np.sqrt(((cc[:, None] - cc[None]) ** 2).sum(2))
        assert np.all(du >= dc - 2.0 * E - 1e-12)
        q = (cc ** 2).sum(1)
        c32 = cc.astype(np.float32)
        g = np.zeros((n, n), dtype=np.float32)
        for d in range(k):                             # one float32 rounding per product added
            g += c32[:, d:d + 1] * c32[None, :, d]
        err = np.abs(q[:, None] + q[None] - 2.0 * g - dc ** 2)
        assert np.all(err <= 2.0 * 1.1 * 2.0 ** -9 * np.sqrt(q[:, None] * q[None]) + 2e-6 * (q[:, None] + q[None]))

"""The vector Ising half-sweep at the edges of its bit logic: thresholds at and
past their limits, draws of every shift, lattices from one chunk per row up,
strided draw layouts, several lattices in a launch."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1003_1898_gb300 as P  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1003_1898_gb300 import build
    build.build()
    P.lib()


def _half_sweep(s, draws, colour, shift, t4, t8):
    """The documented rule, site by site in whole numbers."""
    s = s.astype(np.int64)
    L = s.shape[0]
    y, x = np.indices((L, L))
    nb = np.roll(s, 1, 0) + np.roll(s, -1, 0) + np.roll(s, 1, 1) + np.roll(s, -1, 1)
    dE = 2 * s * nb
    r = (draws.astype(np.uint64) >> np.uint64(shift)).astype(np.int64)[(y * (L // 2) + x // 2)]
    accept = (dE <= 0) | ((dE == 4) & (r < t4)) | ((dE == 8) & (r < t8))
    return np.where(((x + y) % 2 == colour) & accept, -s, s).astype(np.int8)


@pytest.mark.parametrize("shift", [0, 7, 8])
@pytest.mark.parametrize("t4,t8", [(0, 0), (1, 0), (2883584, 495626), (2**24, 1), (2**24, 2**24),
                                   (2**24 - 1, 2**25 - 1), (2**32 - 1, 2**31), (1000, 2**24)])
def test_thresholds_and_shifts(shift, t4, t8):
    rng = np.random.default_rng(shift + t4)
    reqs, want, keep = [], [], []
    for i, L in enumerate((16, 48, 64, 112, 256)):
        s = rng.choice(np.array([-1, 1], np.int8), size=(L, L), p=[.5, .5] if i % 2 else [.1, .9])
        n = L * L // 2
        d = rng.integers(0, 2**32, size=n, dtype=np.uint64)
        near = rng.choice(np.array([t4, t8, 2**24], np.uint64), size=n) << np.uint64(shift)
        edge = (near + rng.integers(-2, 3, size=n).astype(np.uint64)) & np.uint64(2**32 - 1)
        d = np.where(rng.random(n) < .4, edge, d).astype(np.uint32)
        d[:4] = [0, 2**32 - 1, 2**24 - 1, 2**31]
        per, pitch = (0, 0) if i % 2 == 0 else (L * 2, L * 2 + 4 * i)       # 8-rank groups stay together
        ts = torch.from_numpy(s).cuda()
        if pitch:
            rows = np.zeros((n // per, pitch), np.uint32)
            rows[:, :per] = d.reshape(-1, per)
            td = torch.from_numpy(rows.view(np.int32)).cuda()
        else:
            td = torch.from_numpy(d.view(np.int32)).cuda()
        keep.append((ts, td))
        reqs.append({"d_spins": ts, "d_draws": td, "L": L, "colour": i & 1, "shift": shift, "t4": t4, "t8": t8,
                     "per": per, "pitch": pitch})
        want.append(_half_sweep(s, d, i & 1, shift, t4, t8))
    P.prng_ising_half_sweep(reqs)
    torch.cuda.synchronize()
    for (ts, _), w in zip(keep, want):
        np.testing.assert_array_equal(ts.cpu().numpy(), w)

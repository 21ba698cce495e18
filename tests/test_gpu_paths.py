"""GPU paths that are chosen by sizes, counts or the data itself, each at the
edges of its range, element by element against the CPU oracle or numpy.
Every value is an integer: the bar is equality."""
import numpy as np
import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def m():
    import paper_2409_03771_gb300 as msc
    from paper_2409_03771_gb300 import _build

    _build.build()
    msc.load()
    return msc


def cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def host(t):
    return t.cpu().numpy()


# ---------------------------------------------------------------------------
# cell ids: an extremum whose basin meets very many others


def hub_labels(n, hub_share, rng):
    """Labels that label themselves: a tenth of the vertices are extrema, and the last one holds `hub_share`."""
    roots = np.sort(rng.choice(n, n // 10, replace=False))
    lab = roots[np.clip(np.searchsorted(roots, np.arange(n)), 0, roots.size - 1)]  # the next root up
    lab[rng.random(n) < hub_share] = roots[-1]
    lab[roots] = roots
    return lab.astype(np.int32)


@pytest.mark.parametrize("side", ["minimum", "maximum", "both"])
@pytest.mark.parametrize("share", [0.0, 0.001, 0.3])
def test_ms_id_hub(m, side, share):
    n = (1 << 21) + 77  # a table too big for the cache
    rng = np.random.default_rng(11)
    asc = hub_labels(n, share if side != "maximum" else 0.0, rng)
    desc = hub_labels(n, share if side != "minimum" else 0.0, rng)
    keys, want = np.unique(asc.astype(np.int64) * n + desc, return_inverse=True)
    ms, k = m.ms_id(cuda(asc), cuda(desc))
    assert k == keys.size
    np.testing.assert_array_equal(host(ms), want)


def test_segment_valleys_in_a_noisy_plain(m, oracle_mod):
    dims = (150, 131, 129)
    f = workloads.smooth_field(dims, 8, (10.0, 30.0), seed=3, noise_amp=1e-3).numpy().ravel()
    want = oracle_mod.segment_grid(f, dims)
    got = m.segment(cuda(f), dims)
    for g, w in zip(got[:4], want[:4]):
        np.testing.assert_array_equal(host(g), w)
    assert got[4] == want[4]


@pytest.mark.parametrize("bad", [-1, 2 ** 31 - 1])
def test_ms_id_reports_labels_outside_a_large_table(m, bad):
    n = 1 << 21
    asc = np.arange(n, dtype=np.int32)
    asc[::7] = bad
    desc = np.arange(n, dtype=np.int32)
    with pytest.raises(m.MSCError) as e:
        m.ms_id(cuda(asc), cuda(desc))
    assert e.value.code == m.ERR_ARG

"""helm_batch_profile makes the launches that helm_batch_step makes: an engine of 63^2 solves is one
launch of their clusters, in bounded runs too, with the results of a step to completion; a caller
that has no place for that kind gets the same steps launch by launch."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _submit(B, f, g, ks):
    n = f.shape[0]
    batch = B.helm_batch_create(0)
    B.helm_batch_set_lanes(batch, 1)
    us = [torch.zeros_like(g) for _ in ks]
    ts = B.helm_batch_submit_many(batch, [(2, n, 1.0 / (n + 1), k, f, g, u) for k, u in zip(ks, us)],
                                  B.HELM_PREC_MIXED, 1e-8, 100)
    return batch, ts, us


@pytest.mark.parametrize("nkinds", [14, 13])
@pytest.mark.parametrize("chunk", [0, 5])
def test_profile_runs_the_steps_kernels(nkinds, chunk):
    from paper_2308_11469_gb300 import binding as B
    n, ks = 63, [1.0, 2.0, 3.0]
    rng = np.random.default_rng(1)
    f = torch.from_numpy(rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))).cuda()
    g = torch.from_numpy(rng.standard_normal((n + 2, n + 2)) + 0j).cuda()
    batch, ts, us = _submit(B, f, g, ks)
    while any(not r[0] for r in B.helm_batch_poll_many(batch, ts, release=False)):
        B.helm_batch_step(batch, 0)
    want = [B.helm_batch_poll(batch, t, 100) for t in ts]
    B.helm_batch_destroy(batch)
    batch, ts, vs = _submit(B, f, g, ks)
    la, ms, by = (C.c_uint64 * nkinds)(), (C.c_double * nkinds)(), (C.c_double * nkinds)()
    runs = 0
    while any(not r[0] for r in B.helm_batch_poll_many(batch, ts, release=False)):
        assert B.load().helm_batch_profile(batch.handle, chunk, la, ms, by, nkinds) == B.HELM_OK
        runs += 1
        if nkinds == 14:
            assert list(la) == [0] * 13 + [1] and ms[13] > 0.0 and by[13] > 0.0
        else:
            assert sum(la) > 1
        assert runs <= 30
    got = [B.helm_batch_poll(batch, t, 100) for t in ts]
    B.helm_batch_destroy(batch)
    most = max(r[1] for r in want)
    assert runs == (1 if chunk == 0 else -(-most // chunk))
    for a, b, u, v in zip(want, got, us, vs):
        assert a[:2] == b[:2] and np.array_equal(a[2], b[2]) and torch.equal(u, v)

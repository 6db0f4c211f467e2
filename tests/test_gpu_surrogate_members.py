"""Training and inference over many members: the members of an ensemble share grouped
launches (16 problems each) and one head pass, at member counts below, at and above the
sizes those are split by (1, 4, 5, 16 members)."""
import numpy as np
import pytest

import rve_inputs as ri  # noqa: F401  (puts the oracle on the path)
from oracle import surrogate as osg
from test_gpu_surrogate import emulate_member, unpack_member

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rve():
    import paper_1610_03484_gb300 as pkg
    from paper_1610_03484_gb300 import _build
    _build.build()
    pkg.load_library()
    return pkg


def data(n, seed):
    rng = np.random.default_rng(seed)
    feat = rng.normal(size=(n, 8)) * [10, 0.4, 1, 1e9, 4e9, 1e9, 5e8, 0.05] + [40, 0.75, 2, 3e9, 45e9, 12e9, 5e9, 0.2]
    A = rng.normal(size=(n, 6, 6))
    C = A @ np.swapaxes(A, 1, 2) + 6 * np.eye(6)
    B = rng.normal(size=(n, 3, 3))
    K = B @ np.swapaxes(B, 1, 2) + 3 * np.eye(3)
    return feat, C, K, 2 * K + np.eye(3)


@pytest.mark.parametrize("members,n", [(1, 64), (5, 128), (16, 192)])
def test_first_step_of_every_member(rve, members, n):
    """One Adam step of the ensemble is -lr g / (|g| + eps) with each member's own
    gradient.  The trainer sums the shuffled rows in another order (FP32, 1e-7 of the
    summed terms): where |g| > 1e-5 the step does not depend on that."""
    feat, C, K, D = data(n, members)
    lr = 1e-3
    with rve.Context() as ctx:
        s0 = rve.Surrogate(ctx, members=members, seed=5)
        buf0 = s0.get_params()
        s1 = rve.Surrogate(ctx, members=members, seed=5)
        s1.train(feat, C, K, D, epochs=1, batch=n, lr=lr, seed=1)
        buf1 = s1.get_params()
        ref = buf1[49:52].astype(np.float64)
        target = osg.factors_from_tensors(C / ref[0], K / ref[1], D / ref[2]).astype(np.float32)
        s0.set_params(np.concatenate([buf1[:52], buf0[52:]]).astype(np.float32))
        nparam = (len(buf0) - 52) // members
        for e in sorted({0, members // 2, members - 1}):
            g = s0.gradients(e, feat, target)[0].astype(np.float64)
            o = 52 + e * nparam
            w0, w1 = (b[o:o + nparam].astype(np.float64) for b in (buf0, buf1))
            big = np.abs(g) > 1e-5
            assert big.mean() > 0.3
            want = w0 - lr * g / (np.abs(g) + 1e-8)
            ulp = np.spacing(np.abs(w0).astype(np.float32)).astype(np.float64)
            assert (np.abs(w1 - want)[big] <= 4 * ulp[big] + 1e-5 * lr).all(), e
            assert (np.abs(w1 - w0) <= lr + 4 * ulp).all(), e
        s0.free()
        s1.free()


@pytest.mark.parametrize("members,n", [(1, 1), (4, 255), (5, 257), (16, 65)])
def test_ensemble_of_any_size_matches_oracle(rve, members, n):
    """Mean and spread of the member tensors against the oracle's head on emulated
    members; 2e-3 covers a BF16 activation rounded to its other neighbour."""
    feat, C, K, D = data(320, 40 + members)
    with rve.Context() as ctx:
        s = rve.Surrogate(ctx, members=members, seed=2)
        s.train(feat, C, K, D, epochs=2, batch=64, lr=1e-3, seed=1)
        f = feat[:n]
        s.set_fused(False)
        layers = s.predict(f)
        s.set_fused(True)
        fused = s.predict(f)
        buf = s.get_params()
        s.free()
    for x, y in zip(fused, layers):
        np.testing.assert_allclose(x, y, rtol=1e-6, atol=1e-12 * np.abs(y).max())
    nparam = (len(buf) - 52) // members
    ref = buf[49:52].astype(np.float64)
    Ts = []
    for e in range(members):
        z = emulate_member(unpack_member(buf, e, nparam), f, buf[:8], buf[8:16])
        Ts.append(osg.tensors_from_factors(osg.factor_entries(z)))
    spread = np.zeros(n)
    for b in range(3):
        mean = np.mean([T[b] for T in Ts], axis=0)
        den = np.linalg.norm(mean.reshape(n, -1), axis=1)
        err = np.linalg.norm((fused[b] / ref[b] - mean).reshape(n, -1), axis=1) / den
        assert err.max() < 2e-3, (b, err.max())
        for T in Ts:
            spread = np.maximum(spread, np.linalg.norm((T[b] - mean).reshape(n, -1), axis=1) / den)
    assert np.abs(fused[3] - spread).max() < 2e-3


@pytest.mark.parametrize("members,n,batch", [(4, 1024, 256), (1, 64, 64), (5, 1000, 192), (2, 8256, 8256)])
def test_loss_history_is_reproducible(rve, members, n, batch):
    """The same training twice returns the same history to the bit.  With one step an epoch
    the first loss is the mean of the members' losses at the initial parameters (FP32 sums of
    the same terms, the rows in another order: at most 1e-5 for 2e5 terms)."""
    feat, C, K, D = data(n, 7 * members)
    runs = []
    for _ in range(2):
        with rve.Context() as ctx:
            s = rve.Surrogate(ctx, members=members, seed=5)
            buf0 = s.get_params()
            hist = np.asarray(s.train(feat, C, K, D, epochs=3, batch=batch, lr=1e-3, seed=1))
            buf1 = s.get_params()
            if n == batch:
                ref = buf1[49:52].astype(np.float64)
                target = osg.factors_from_tensors(C / ref[0], K / ref[1], D / ref[2]).astype(np.float32)
                s.set_params(np.concatenate([buf1[:52], buf0[52:]]).astype(np.float32))
                want = np.mean([s.gradients(e, feat, target)[1] for e in range(members)])
                assert abs(hist[0] - want) < 1e-5 * want
            s.free()
        runs.append((hist, buf1))
    np.testing.assert_array_equal(runs[0][0], runs[1][0])
    np.testing.assert_array_equal(runs[0][1], runs[1][1])


def test_a_wait_that_gave_up_is_reported_by_every_call(rve):
    """The status word set on the host, as the kernels set it: training, gradients and both
    forms of the inference answer RVE_ERR_TIMEOUT, and work again once it is cleared."""
    import torch
    feat, C, K, D = data(128, 9)
    with rve.Context() as ctx:
        s = rve.Surrogate(ctx, members=2, seed=3)
        s.train(feat, C, K, D, epochs=1, batch=64, lr=1e-3, seed=1)
        f = torch.tensor(feat, device="cuda")
        out = [torch.zeros(len(feat), k, dtype=torch.float64, device="cuda") for k in (36, 9, 9, 1)]
        calls = [lambda: s.predict(feat),
                 lambda: s.predict_dev(len(feat), f.data_ptr(), *(v.data_ptr() for v in out)),
                 lambda: s.train(feat, C, K, D, epochs=1, batch=64, lr=1e-3, seed=1),
                 lambda: s.gradients(0, feat[:64], np.ones((64, 33), np.float32))]
        lib = rve.load_library()
        assert lib.rve_debug_gemm_timeout(1) == 0
        try:
            for call in calls:
                with pytest.raises(rve.RveError) as e:
                    call()
                assert e.value.code == -10
        finally:
            assert lib.rve_debug_gemm_timeout(0) == 1
        for call in calls:
            call()
        s.free()


@pytest.mark.parametrize("members,at_once", [(5, 3), (4, 1), (16, 8)])
def test_members_trained_in_groups(rve, members, at_once):
    """Too little room for all members' training buffers: they train in groups, with the
    parameters and the history of training together, to the bit."""
    feat, C, K, D = data(256, members)
    per_member = 64 * 13_320 + 4 * 230_464   # bytes for batches of 64 rows
    out = []
    for limit in (0, int(per_member * (at_once + 0.5))):
        with rve.Context() as ctx:
            s = rve.Surrogate(ctx, members=members, seed=5)
            assert ctx.lib.rve_debug_surrogate_work_limit(ctx.h, s.h, limit) == 0
            hist = s.train(feat, C, K, D, epochs=2, batch=64, lr=1e-3, seed=1)
            out.append((np.asarray(hist), s.get_params()))
            s.free()
    np.testing.assert_array_equal(out[0][0], out[1][0])
    np.testing.assert_array_equal(out[0][1], out[1][1])

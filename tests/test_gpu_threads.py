"""Contexts of different sizes side by side: the kernels' attributes belong to
the process, so no context may depend on the limits another one needs.

A problem with large tables (K_d = 32, q = 96: more than 48 KB of dynamic
shared memory in its window, trace and energy kernels) and one with small ones
are set up, assembled and stepped alternately and from two threads.
"""
import threading

import numpy as np
import pytest

from paper_1710_02401_gb300 import problems as P

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1710_02401_gb300 import build as B
    B.build()
    from paper_1710_02401_gb300 import swr as S_
    return S_


def _large(mode=P.TISE):
    if mode == P.TDSE:
        return P.small_tdse_2d(L=2, K_d=32, q_p=16, n_mid=4, n_steps=1)
    return P.small_tise_2d(L=2, K_d=32, q_p=16, n_mid=4).replace(ngf_tol=0.0, n_steps=2)


def _small(mode=P.TISE):
    if mode == P.TDSE:
        return P.small_tdse_2d(L=2, K_d=4, q_p=4, n_mid=1, n_steps=1)
    return P.small_tise_2d(L=2, K_d=4, q_p=4, n_mid=1).replace(ngf_tol=0.0, n_steps=2)


@pytest.mark.parametrize("precision,variant", [(0, 0), (0, 1), (1, 0), (1, 1), (1, 2), (1, 3), (1, 4), (2, 0)])
def test_a_small_context_leaves_the_large_ones_launches_alone(S, precision, variant):
    kw = dict(precision=precision, window_variant=variant, launch_mode=S.LAUNCH_DIRECT)
    big = S.SWR(_large(), **kw)
    small = S.SWR(_small(), **kw)
    big.assemble()
    small.assemble()
    for s in (big, small, big):
        s.step()
    assert np.all(np.isfinite(big.residual())) and np.all(np.isfinite(small.residual()))


@pytest.mark.parametrize("mode,precision", [(P.TISE, 0), (P.TISE, 1), (P.TDSE, 0), (P.TDSE, 2)])
def test_two_threads_with_problems_of_different_sizes(S, mode, precision):
    import torch
    errors = []
    start = threading.Barrier(2)

    def work(inst, assemblies, steps):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                s = S.SWR(inst, precision=precision, launch_mode=S.LAUNCH_DIRECT, contraction_path=S.CONTRACT_FP64)
                start.wait(60)
                for _ in range(assemblies):
                    s.assemble()
                    for _ in range(steps):
                        s.step()
                s.close()
        except Exception as e:  # noqa: BLE001  (reported by the test's thread)
            errors.append(e)
            start.abort()

    ts = [threading.Thread(target=work, args=(_large(mode), 12, 40)),
          threading.Thread(target=work, args=(_small(mode), 60, 40))]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not errors, errors


def test_two_threads_build_determinants_of_different_sizes(S):
    kw = dict(L=2, M=6, q_p=10, panel=0.4, nuclei=((-0.5, 1.0), (0.5, 1.0)))
    errors = []

    def work(kd, n):
        try:
            want = S.lsd_build(kd=kd, K=10, **kw)
            for _ in range(n):
                got = S.lsd_build(kd=kd, K=10, **kw)
                for key in want:
                    np.testing.assert_array_equal(got[key], want[key])
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    ts = [threading.Thread(target=work, args=(62, 40)), threading.Thread(target=work, args=(12, 150))]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not errors, errors

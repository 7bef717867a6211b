"""Arguments of a batched call, packed: the bytes that a ctypes structure per item would hold."""
import types

import numpy as np
import pytest

import workloads as wl
from paper_2404_02521_gb300 import _lib as L


def test_params_array_equals_the_structures():
    rng = np.random.default_rng(0)
    a, b = wl.random_params(rng, wl.BASKET), wl.paper_cash_or_nothing().params
    plain = types.SimpleNamespace(sigma1=np.float32(0.2), sigma2="0.3", rho=0, r=np.float64(0.05), T=1, strike=1,
                                  w1=0.5, w2=0.5, payoff=1.0)
    params = [a, a, plain, plain, b, a]
    want = (L.bs_params * 6)(*[L.to_params(p) for p in params])
    assert bytes(L._params_array(params, 6)) == bytes(want)
    # fewer sets than states: the rest is zero, as in a ctypes array; more are refused
    assert bytes(L._params_array(iter(params[:2]), 3)) == bytes((L.bs_params * 3)(*[L.to_params(a)] * 2))
    with pytest.raises(IndexError):
        L._params_array(params, 5)


def test_pointer_and_time_arrays():
    import torch
    t = torch.zeros(4)
    assert list(L._pointers([t, 16], 3)) == [t.data_ptr(), 16, None]
    assert list(L._doubles([np.float32(0.5), 1], 2)) == [0.5, 1.0]
    for f in (L._pointers, L._doubles):
        with pytest.raises(IndexError):
            f([1, 2], 1)

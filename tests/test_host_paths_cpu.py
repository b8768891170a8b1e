"""Host paths of the library against a CUDA runtime that runs no kernel
(tests/fake_cudart.cpp): what is set per device, where memory is taken, and what
a call does when it cannot be had."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2312_05647_gb300 import build as lib_build
from paper_2312_05647_gb300 import capi

HERE = os.path.dirname(os.path.abspath(__file__))
BD, TS, MP, AR = capi.BD1D, capi.TWOSTATE, capi.MRNA_PROT2D, capi.AUTOREG


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    lib_build.build()
    objs = [os.path.join(lib_build.OBJ_DIR, os.path.basename(s)[:-3] + ".o") for s in lib_build.sources()]
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(lib_build.nvcc()))), "include")
    so = str(tmp_path_factory.mktemp("fake") / "libmjp_fake.so")
    # -Bsymbolic: a real runtime in the process (torch's) does not take the fake's place.
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", inc, "-Wl,-Bsymbolic", "-Wl,-z,defs", "-o", so,
                    os.path.join(HERE, "fake_cudart.cpp"), *objs], check=True)
    L = ctypes.CDLL(so)
    for name, (res, args) in capi.SIGNATURES.items():
        f = getattr(L, name)
        f.restype, f.argtypes = res, args
    L.fake_memory.argtypes = [ctypes.c_longlong]
    for f in (L.fake_mallocs, L.fake_launches):
        f.restype = ctypes.c_long
    return L


@pytest.fixture
def L(lib):
    lib.fake_reset()
    return lib


def _p(a, t):
    return a.ctypes.data_as(t)


def _ok(L, rc):
    assert rc == 0, L.mjp_last_error()


def _net(L):
    h = ctypes.c_void_p()
    _ok(L, L.mjp_mlp_create(ctypes.byref(h), 1))
    return h


def _stencil(L, kind, dims, theta, prec):
    h = ctypes.c_void_p()
    d, t = np.asarray(dims, np.int64), np.asarray(theta, float)
    _ok(L, L.rate_model_create_stencil(ctypes.byref(h), kind, _p(d, capi._i64p), len(d), _p(t, capi._f64p), len(t), prec))
    return h


def _series(L, h, n, times, prec):
    t = np.asarray(times, float)
    rho = np.zeros(n, np.float32 if prec == 1 else np.float64)
    out = np.zeros((len(t), n), rho.dtype)
    return L.expv_series(h, rho.ctypes.data, _p(t, capi._f64p), len(t), out.ctypes.data, None, 0, 0.0, None)


@pytest.mark.parametrize("rows", [100, 2000, 9000])
def test_gradient_on_a_second_device(L, rows):
    psi, y = np.zeros((rows, 4)), np.zeros(rows)
    cfg = capi.TrainCfg(3, rows, 1e-3, 0.9, 0.999, 1e-8, 7, 0)
    for dev in (0, 1, 0):
        L.fake_device(dev)
        net = _net(L)
        _ok(L, L.mjp_mlp_loss_grad(net, psi.ctypes.data, y.ctypes.data, rows, None, None, capi.PTR_DEVICE, None))
        _ok(L, L.mjp_mlp_train(net, psi.ctypes.data, y.ctypes.data, rows, ctypes.byref(cfg), None, capi.PTR_DEVICE, None))
        L.mjp_mlp_destroy(net)


# Small-model chain with many windows, one CTA and a cluster of the register/tile chain.
@pytest.mark.parametrize("kind,dims,theta,nt", [(BD, [200], [7.0, 0.6], 20), (TS, [100], [9.0, 0.7, 2.0, 1.0], 20),
                                                (TS, [900], [9.0, 0.7, 2.0, 1.0], 9), (MP, [40, 30], [3.0, 0.5, 1.5, 0.2], 9),
                                                (MP, [120, 90], [3.0, 0.5, 1.5, 0.2], 9), (AR, [25, 30], [4.0, 0.5, 0.6, 0.1, 0.4, 0.05], 9)])
@pytest.mark.parametrize("prec", [1, 2])
def test_transient_distributions_on_a_second_device(L, kind, dims, theta, nt, prec):
    n = int(np.prod(dims)) * (2 if kind in (TS, AR) else 1)
    for dev in (0, 1, 70, 70, 0):
        L.fake_device(dev)
        h = _stencil(L, kind, dims, theta, prec)
        _ok(L, _series(L, h, n, np.linspace(0.1, 5.0, nt), prec))
        L.rate_model_destroy(h)


def _csr(L, n, prec):
    """A ring of n states."""
    h = ctypes.c_void_p()
    rp, col, rate = np.arange(n + 1, dtype=np.int64), ((np.arange(n) + 1) % n).astype(np.int32), np.ones(n)
    _ok(L, L.rate_model_create_csr(ctypes.byref(h), n, _p(rp, capi._i64p), _p(col, capi._i32p), _p(rate, capi._f64p), prec))
    return h


@pytest.mark.parametrize("prec", [1, 2])
def test_general_matrix_runs_on_two_vectors_where_nine_do_not_fit(L, prec):
    n, elt = 200000, 4 if prec == 1 else 8
    out = (2 * elt if prec == 1 else elt) * n  # one output and, in FP32, its compensation
    for spare, rc in ((9 * elt * n, 0), (3 * elt * n, 0), (elt * n, -3)):
        L.fake_memory(1 << 40)
        h = _csr(L, n, prec)
        L.fake_memory(out + spare + (1 << 16))
        assert _series(L, h, n, [0.5], prec) == rc
        if rc == 0:
            before = L.fake_mallocs()
            _ok(L, _series(L, h, n, [0.5], prec))
            assert L.fake_mallocs() == before  # nothing is tried again
        L.rate_model_destroy(h)


def test_general_matrix_gives_up_its_ring_for_more_outputs(L):
    n = 200000
    h = _csr(L, n, 2)
    L.fake_memory(8 * n * 10 + (1 << 16))
    _ok(L, _series(L, h, n, [0.5], 2))
    _ok(L, _series(L, h, n, [0.5, 1.0, 1.5, 2.0], 2))  # 4 + 9 vectors do not fit, 4 + 2 do
    L.rate_model_destroy(h)


def test_standardisation_of_device_data_takes_no_memory(L):
    """So that it can be captured in a graph on a new network."""
    n = 9000
    psi, y = np.zeros((n + 1, 4)), np.zeros(n)
    net = _net(L)
    base = psi.ctypes.data + (-psi.ctypes.data) % 16
    before = L.fake_mallocs()
    _ok(L, L.mjp_mlp_fit_norm(net, base, y.ctypes.data, n, capi.PTR_DEVICE, None))
    assert L.fake_mallocs() == before
    L.mjp_mlp_destroy(net)

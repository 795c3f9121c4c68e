"""CPU: the layer's entry points reject bad arguments on the host, before any CUDA
call (the addresses below are never dereferenced)."""
import pytest

from paper_2406_12580_gb300 import _lib
from paper_2406_12580_gb300 import build as blr_build

FAKE = 0x7f0000000000
OK, ARG, UNSUPPORTED = _lib.BLR_OK, _lib.BLR_ERR_INVALID_ARG, _lib.BLR_ERR_UNSUPPORTED


@pytest.fixture(scope="module")
def lib():
    if blr_build.stale():
        blr_build.build()
    return _lib.load()


def call(fn, names, sizes, **kw):
    args = dict.fromkeys(names, FAKE)
    args.update(kw)
    return fn(*sizes, *(args[n] for n in names), None)


def test_conv_silu(lib):
    fwd = ("hxz", "weight", "bias", "x", "z")
    bwd = ("dx", "dz", "hxz", "weight", "bias", "dhxz", "dweight", "dbias", "ws")
    run_f = lambda B=2, L=5, C=16, io=0, **kw: call(lib.blr_conv_silu_fwd, fwd, (B, L, C, io), **kw)  # noqa: E731
    run_b = lambda B=2, L=5, C=16, io=0, n=1 << 30, **kw: call(  # noqa: E731
        lib.blr_conv_silu_bwd, (*bwd, "n"), (B, L, C, io), n=n, **kw)
    need = lib.blr_conv_silu_workspace(2, 5, 16)
    assert need > 0 and lib.blr_conv_silu_workspace(2, 5, 12) == 0
    for run, names in ((run_f, fwd), (run_b, bwd)):
        assert run(C=12) == UNSUPPORTED and run(C=1032) == UNSUPPORTED
        assert run(B=-1) == ARG and run(L=-1) == ARG and run(io=2) == ARG
        assert run(B=0, **dict.fromkeys(names)) == OK
        for name in names:
            assert run(**{name: None}) == ARG, name
            assert run(**{name: FAKE + 2}) == ARG, name
    assert run_b(n=need - 1) == ARG


def test_linear(lib):
    fwd = ("x", "weight", "bias", "y")
    run_f = lambda T=5, N=8, K=12, **kw: call(lib.blr_linear_fwd, fwd, (T, N, K), **kw)  # noqa: E731

    def run_b(T=5, N=8, K=12, n=1 << 30, **kw):
        return call(lib.blr_linear_bwd, ("dy", "x", "weight", "dx", "add", "dweight", "dbias", "ws", "n"),
                    (T, N, K), add=0, n=n, **kw)

    need = lib.blr_linear_workspace(5, 8, 12)
    assert need > 0 and lib.blr_linear_workspace(5, 8, 10) == 0
    for run in (run_f, run_b):
        assert run(N=6) == UNSUPPORTED and run(K=10) == UNSUPPORTED and run(N=65540) == UNSUPPORTED
        assert run(T=-1) == ARG and run(T=0) == OK
    for name in fwd:
        assert run_f(**{name: FAKE + 8}) == ARG, name
        assert name == "bias" or run_f(**{name: None}) == ARG, name
    # nothing is launched for the input's gradient when the weight's cannot be computed
    for name in ("dy", "x", "weight", "dx", "dweight", "dbias", "ws"):
        assert run_b(**{name: FAKE + 2}) == ARG, name
        assert name in ("dx", "dweight") or run_b(**{name: None}) == ARG, name
    assert run_b(n=need - 1) == ARG

"""Argument checks of the validation entry points, before any device work."""
import ctypes

import pytest

import synth


@pytest.fixture(scope="module")
def env():
    from paper_2607_00756_gb300 import build
    build.build()
    from paper_2607_00756_gb300 import capi
    ctx = capi.bip_create(capi.make_config(synth.config1()))
    yield capi, ctx
    capi.bip_destroy(ctx)


@pytest.mark.parametrize("rows,cols,d_cols,dcol0", [(4, 20, 100, 2 ** 31 - 10), (4, 2 ** 31 - 1, 100, 2 ** 31 - 1),
                                                    (4, 20, 19, 0), (4, 20, 100, 81), (0, 20, 100, 0), (4, 20, 100, -1)])
def test_split_refuses_columns_outside_its_destination(env, rows, cols, d_cols, dcol0):
    """Sums past 31 bits included.  (The pointers are never followed.)"""
    capi, ctx = env
    p = ctypes.c_void_p(4096)
    status = capi.lib().bip_debug_split(ctx, rows, cols, p, 20, 1, d_cols, dcol0, 0, p, None)
    assert capi.STATUS[status] == "BIP_ERR_INVALID_ARG"

"""Params forms what every call needs of it once; copies, pickles, equality and replacement know
nothing of that."""
import copy
import ctypes
import dataclasses
import pickle

import pytest

from paper_1703_04594_gb300 import lbm
from tests.gpu_util import ensure_built


def test_params_keep_their_call_data_to_themselves():
    ensure_built()
    p = lbm.Params(40, 70, tau=0.7, gx=1e-4, precision=lbm.FP32_CONSERVED)
    q = lbm.Params(40, 70, tau=0.7, gx=1e-4, precision=lbm.FP32_CONSERVED)
    assert p._call is p._call and p._call.bytes == lbm.buffer_bytes(q) == 37 * 40 * 96 * 4
    assert p == q and hash(p) == hash(q) and repr(p) == repr(q)
    for c in (copy.copy(p), copy.deepcopy(p), pickle.loads(pickle.dumps(p))):
        assert c == p and "_call" not in c.__dict__ and c._call.bytes == p._call.bytes
    r = dataclasses.replace(p, precision=lbm.FP64, tau=0.9)
    struct = ctypes.cast(r._call.ref, ctypes.POINTER(lbm.CParams)).contents
    assert struct.tau == 0.9 and struct.precision == lbm.FP64 and r._call.bytes == 2 * p._call.bytes
    with pytest.raises(lbm.LbmError):
        lbm.Params(3, 70)._call


def test_params_hold_their_fields_alone():
    """What a program makes of a parameter set's attributes does not depend on calls made with it."""
    ensure_built()
    p = lbm.Params(40, 70, tau=0.7)
    before = dict(vars(p))
    assert p._call.bytes > 0
    assert dict(vars(p)) == before == dataclasses.asdict(p) and lbm.Params(**vars(p)) == p

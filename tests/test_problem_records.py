"""The records that Problem.params makes: the same bytes as a fresh Problem gives, whatever was set, copied or passed before."""
import copy
import dataclasses
import pickle

import torch

from paper_2409_12490_b200 import binding as cp

ARGS = (1, 8, 2, 300, 64, 64, 16, 8)


def test_fields_set_later_and_copies():
    p = cp.Problem(*ARGS)
    p.params()
    for name, value in (("alpha", 0.5), ("seq_len", 290), ("sm_scale", 0.25), ("dtype", torch.float16), ("n_sink", 2), ("flags", 1 << 40)):
        setattr(p, name, value)
        fresh = cp.Problem(*(getattr(p, f.name) for f in dataclasses.fields(p)))
        for q in (p, copy.copy(p), copy.deepcopy(p), pickle.loads(pickle.dumps(p)), dataclasses.replace(p)):
            assert bytes(q.params()) == bytes(fresh.params()) == bytes(q.params())
            assert q == fresh
    c = copy.copy(p)
    c.alpha = 0.125
    assert p.params().alpha == 0.5 and c.params().alpha == 0.125


def test_strides_and_records_are_the_callers_own():
    p = cp.Problem(*ARGS)
    plain = bytes(p.params())
    for pad in range(12):                                  # more strides than are kept
        K = torch.empty(1, 2, 300 + pad, 64)[:, :, :300]
        rec = p.params(K=K)
        assert tuple(rec.k_stride) == K.stride()[:3]
        rec.k_stride[1] = 7                                # a copy: the next call does not see it
        assert tuple(p.params(K=K).k_stride) == K.stride()[:3]
    assert bytes(p.params()) == plain


def test_nothing_but_the_fields():
    p = cp.Problem(*ARGS)
    p.params()
    assert set(vars(p)) == {f.name for f in dataclasses.fields(p)}
    assert cp.Problem(**vars(p)) == p
    vars(p).update(seq_len=290, alpha=0.5)                 # fields set behind the object's back
    assert bytes(p.params()) == bytes(cp.Problem(1, 8, 2, 290, 64, 64, 16, 8, alpha=0.5).params())
    # making an object and setting a field run no code of the class: a decoding step does both per token
    assert cp.Problem.__setattr__ is object.__setattr__

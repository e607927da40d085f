"""The batch tuner, on the CPU: what its cache tells apart, and the library's
own choice among the candidates."""
from dataclasses import replace

import pytest
import torch

from paper_2308_09348_gb300 import binding as B
from paper_2308_09348_gb300 import inputs as I
from paper_2308_09348_gb300 import tune


def _batch(lasers, bins=I.Bins(n_bins=64), sweep=False, precision="f32"):
    b = object.__new__(B.Batch)
    b.n_shots, b.bins, b.precision, b.max_phase = len(lasers), bins, precision, 64
    b.d_lasers = B._struct_array_to_device([B.make_laser(x) for x in lasers], B.qs_laser, "cpu")
    b.d_offsets = None if sweep else torch.zeros(len(lasers) + 1)
    return b


Q, L = I.Laser(model=I.MODEL_QFP), I.Laser(model=I.MODEL_LL)


def test_classes_are_told_apart():
    bins = I.Bins(n_bins=64)
    variants = [_batch([Q, Q]), _batch([L, L]), _batch([Q, L]), _batch([Q, replace(Q, variant=1)]),
                _batch([Q, replace(Q, variant=2)]), _batch([Q, Q], sweep=True),
                _batch([Q, Q], replace(bins, smooth_sigma_bins=2.0)),
                _batch([Q, Q], replace(bins, n_tx=8, n_ty=8, theta_max=1.0)),
                _batch([Q, Q], replace(bins, n_aeff=8, aeff_max=1.0)),
                _batch([Q, Q], replace(bins, log_spaced=1, lo=1.0)),
                _batch([Q, Q], precision="f64"), _batch([Q, Q, Q])]
    keys = [tune.batch_class(b, 1000) for b in variants]
    keys += [tune.batch_class(variants[0], 1000, weighted=True), tune.batch_class(variants[0], 4000)]
    assert len(set(keys)) == len(keys)
    # the order of the shots makes no other workload
    assert tune.batch_class(_batch([L, Q]), 1000) == tune.batch_class(_batch([Q, L]), 1000)


def test_the_open_schedule_is_a_candidate():
    assert (0, 0) in tune.BATCH_CANDIDATES
    assert any(t == 512 for _, t in tune.BATCH_CANDIDATES)


def test_other_kernels_are_tuned_again(monkeypatch, tmp_path):
    monkeypatch.setenv("QSCATTER_CACHE_DIR", str(tmp_path))
    monkeypatch.setattr(tune, "gpu_key", lambda: "gpu")
    runs = []
    monkeypatch.setattr(tune, "time_call", lambda fn, reps: fn())

    def tuned(times):
        return tune.tune("class", tuple(times), lambda c: lambda: runs.append(c) or times[c])[0]

    assert tuned({(0, 0): 2.0, (256, 512): 1.0}) == (256, 512) and len(runs) == 2
    assert tuned({(0, 0): 1.0, (256, 512): 2.0}) == (256, 512) and len(runs) == 2
    monkeypatch.setattr(tune, "sources_key", lambda: "other")
    assert tuned({(0, 0): 1.0, (256, 512): 2.0}) == (0, 0) and len(runs) == 4

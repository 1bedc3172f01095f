"""The run-time gate's part of the committed selector blobs (log-time head,
conversion-cost lines) against the committed timings of the kernels as they are,
on matrices it was not fitted to: a product's predicted time is within a quarter
of the measured one for half of the matrices and more, of R-MAT matrices too,
in the picked configuration and in default CSR, and each report says what is recomputed here."""
import gzip
import json
import math
import os

import numpy as np
import pytest

from paper_2302_05662_gb300 import selector as S
from paper_2302_05662_gb300 import sweep

BLOBS = {"f64": S.DEFAULT_BLOB, "f32": S.LOWP_BLOB, "bf16": S.BF16_BLOB}


@pytest.mark.parametrize("vt", list(BLOBS))
def test_heads_describe_the_kernels(vt):
    p = S.parse_blob(np.fromfile(BLOBS[vt], dtype=np.float32))
    labels = sweep.label_space(include_sell=True)
    recs = S.load_records([S.HEADS_DATA[vt]])
    X, T, D, ids, fams = S.dataset(recs, [sweep.config_key(c) for c in labels])
    held = ids >= 1800
    assert held.sum() == 200
    w = {k: p[k].astype(np.float64) for k in ("mu", "sigma", "W1", "b1", "W2", "b2")}
    lt = S.predict_logt(w, p["W3"], p["b3"], X[held])
    choice = np.argmax(np.where(np.isfinite(T[held]), S.predict(w, X[held]), -np.inf), axis=1)
    rows = np.arange(choice.size)
    e_sel = np.abs(lt[rows, choice] - np.log(T[held][rows, choice]))
    e_def = np.abs(lt[:, -1] - np.log(D[held]))
    for fam in sorted(set(fams)):
        of = np.array(fams)[held] == fam
        assert np.median(e_sel[of]) <= math.log(1.25) and np.median(e_def[of]) <= math.log(1.25), fam
    rep = json.load(open(BLOBS[vt][:-4] + "_report.json"))
    assert rep["time_head_heldout"]["median_abs_log_error_selected"] == pytest.approx(np.median(e_sel), abs=1e-3)
    assert rep["time_head_heldout"]["median_abs_log_error_default_csr"] == pytest.approx(np.median(e_def), abs=1e-3)
    assert rep["classifier_on_heads_data"]["heldout"] == S.evaluate(choice, T[held], D[held])
    with gzip.open(S.HEADS_CALIB, "rt") as fh:
        calib = [c for c in map(json.loads, fh) if c["dtype"] == vt and c["matrix"] >= 1800 and c["us"] is not None]
    pred = np.array([p["pack"][c["format"]].astype(np.float64) @ [1.0, c["nnz"], c["m"]] for c in calib])
    meas = np.array([c["us"] for c in calib])
    assert abs(np.log(pred.sum() / meas.sum())) <= math.log(1.25)
    assert rep["pack_model_heldout"]["n"] == len(calib)
    assert min(rep["gate_agreement_heldout"].values()) >= 0.75

"""The column-by-column panel kernels and the look-ahead, which run where the sub-block panel does not
fit (CQR_PANEL_BLK=0 asks for them): against the oracle and each other, and their waits between
CTAs running out (needs a GB300; the launches are correct, only the bound of a wait is short).
Each test looks at the kernels that ran.  Tolerance n u kappa, u = 8 times FP32's for 3xTF32."""
import re
import time

import numpy as np
import pytest

from oracle import oracle as O
from paper_2311_11943_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2311_11943_gb300 import binding as B  # noqa: E402

U32, U64 = np.finfo(np.float32).eps / 2, np.finfo(np.float64).eps / 2


def kernels(fn):
    """The names of the kernels that fn launches."""
    from torch.profiler import ProfilerActivity, profile
    with profile(activities=[ProfilerActivity.CUDA, ProfilerActivity.CPU]):
        torch.zeros(8, device="cuda").add_(1)  # the first profile of a process records nothing
        torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA, ProfilerActivity.CPU]) as p:
        fn()
        torch.cuda.synchronize()
    return " ".join(e.key for e in p.key_averages())


def device(A, dtype):
    Ad = B.colmajor_empty(*A.shape, torch.float64 if dtype == "f64" else torch.float32)
    Ad.copy_(torch.from_numpy(A))
    return Ad


def rel(X, Y):
    return np.linalg.norm(X - Y) / np.linalg.norm(Y)


# the register-resident panel of one cluster, the shared-memory panel of one cluster (its barriers are
# the hardware's: no wait to run out), the cooperative panel with a grid barrier (FP64, 10240 rows), the two-level exchange
# (FP32, 20480 x 256) and the flat grid in its place
CASES = {
    "register": ((1280, 1024, 8, 8, 2, 128, "f32", "3xtf32"), {}, r"k_panel_reg"),
    "cluster": ((1280, 1024, 8, 8, 2, 128, "f32", "3xtf32"), {"CQR_PANEL_REG": "0"},
                r"k_panel<float, \d+, true, true, false>"),
    "grid": ((8192, 256, 8, 4, 2, 64, "f64", "simt"), {}, r"k_panel<double, \d+, false, \w+, false>"),
    "two-level": ((16384, 768, 16, 8, 4, 256, "f32", "3xtf32"), {}, r"k_panel<float, \d+, false, true, true>"),
    "flat": ((16384, 768, 16, 8, 4, 256, "f32", "3xtf32"), {"CQR_PANEL_HIER": "0"},
             r"k_panel<float, \d+, false, \w+, false>"),
}


def run(shape, env, monkeypatch):
    m, n, p_r, p_c, f, b, dtype, mma = shape
    monkeypatch.setenv("CQR_PANEL_BLK", "0")
    for k, v in env.items():
        monkeypatch.setenv(k, v)
    A = synth.kappa_matrix(m, n, 1e2, seed=41)
    q = B.CodedQR(m, n, p_r, p_c, f, b, dtype=dtype, mma=mma, seed=6)
    Ad = device(A, dtype)
    q.encode(Ad)
    return q, Ad, A


@pytest.mark.parametrize("name", list(CASES))
def test_column_panels_match_the_oracle(name, monkeypatch):
    shape, env, kernel = CASES[name]
    m, n, p_r, p_c, f, b, dtype, mma = shape
    q, Ad, A = run(shape, env, monkeypatch)
    names = kernels(lambda: q.factor(0, -1))
    assert re.search(kernel, names) and "k_panel_blk" not in names, names
    assert q.sync_status() == 0
    Q, R = q.factors()
    Q, R = Q.double().cpu().numpy(), R.double().cpu().numpy()
    ref = O.run(A, p_r, p_c, f, b, seed=6)
    tol = n * (U64 if dtype == "f64" else U32 * (8 if mma == "3xtf32" else 1)) * 1e2
    assert rel(R, ref["R"]) < tol and rel(Q[: ref["geom"].M, :n], ref["Q"][:, :n]) < tol
    if name == "cluster":
        q.close()
        return
    # their waits run out
    q.encode(Ad)
    q.set_wait_limit(200)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    q.factor(0, -1)
    st = q.sync_status()
    assert st == B.CQR_ETIMEOUT, B.errstr(st)
    assert time.perf_counter() - t0 < 1.0
    q.set_wait_limit(0)
    q.encode(Ad)
    q.factor(0, -1)
    assert q.sync_status() == 0
    _, R2 = q.factors()
    assert np.array_equal(R2.double().cpu().numpy(), R)
    q.close()


@pytest.mark.parametrize("mma", ["3xtf32", "tf32", "bf16x3"])
def test_look_ahead_and_dependent_launch_change_rounding_only(mma, monkeypatch):
    m, n, p_r, p_c, f, b = 1280, 1024, 8, 8, 2, 128
    monkeypatch.setenv("CQR_PANEL_BLK", "0")
    A = synth.kappa_matrix(m, n, 10.0, seed=41)
    er = {3: synth.random_erasures(p_r + f, p_c + f, f, 2, seed=9)}
    ref = O.run(A, p_r, p_c, f, b, seed=6, erasures=er)
    tol = n * {"3xtf32": 8 * U32, "tf32": 2.0 ** -11, "bf16x3": 2.0 ** -16}[mma] * 10.0
    out = {}
    for name, env in {"look-ahead": {}, "one stream": {"CQR_LOOKAHEAD": "0"}, "no dependent launch": {"CQR_PDL": "0"}}.items():
        for k in ("CQR_LOOKAHEAD", "CQR_PDL"):
            monkeypatch.delenv(k, raising=False)
        for k, v in env.items():
            monkeypatch.setenv(k, v)
        q = B.CodedQR(m, n, p_r, p_c, f, b, dtype="f32", mma=mma, seed=6, reorth_block=True)
        q.profile(True)
        q.encode(device(A, "f32"))
        q.factor(0, 3)
        q.inject(er[3])
        q.recover()
        q.factor(3, -1)
        assert q.sync_status() == 0
        assert (q.profile_read()["tc_narrow_update"][0] > 0) == (name != "one stream")
        _, R = q.factors()
        out[name] = R.double().cpu().numpy()
        q.close()
        assert rel(out[name], ref["R"]) < tol, name
    assert np.array_equal(out["look-ahead"], out["no dependent launch"])

"""Child process of tests/test_gpu_debug_bounds_update.py: the kernels of large FP64 updates, of the
adjoints and of batches through the bounds-checked build, on odd shapes; prints one JSON line."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402
import torch  # noqa: E402

from oracle import oracle as O  # noqa: E402
from paper_2311_11943_gb300 import binding as B  # noqa: E402
from paper_2311_11943_gb300 import synth  # noqa: E402

assert B.LIB_PATH.endswith("libcoded_qr_debug.so"), B.LIB_PATH
out = {}


def take(name, **more):
    torch.cuda.synchronize()
    st, site = B.debug_bounds()
    out[name] = dict(bounds=int(st), site=int(site), **more)


def device(A, dtype):
    Ad = B.colmajor_empty(*A.shape, dtype)
    Ad.copy_(torch.from_numpy(np.asarray(A)))
    return Ad


# FP64 update by integer slices: ragged rows, a panel width that is no multiple of a stage, a
# ragged last panel
m, n = 2049, 260
A = synth.kappa_matrix(m, n, 10.0, seed=3)
q = B.CodedQR(m, n, 3, 4, 1, 120, dtype="f64", seed=3)
q.encode(device(A, torch.float64))
q.profile_read()
q.factor(0, -1)
ran = q.profile_read()["tc_update"][1]
_, R = q.factors()
R = R.cpu().numpy()
ref = O.run(A, 3, 4, 1, 120, seed=3)
take("f64 update", status=int(q.sync_status()), ran=int(ran), tol=float(n * 2.0 ** -53 * 10.0 * 16),
     err=float(np.abs(R - ref["R"]).max() / np.abs(ref["R"]).max()))
q.close()

# adjoints: tensor cores with inverted blocks (n > 128), CUDA cores, two right-hand sides
for name, dt, mma in (("adjoint f32", torch.float32, "3xtf32"), ("adjoint f64", torch.float64, "simt")):
    m, n, k = 1003, 276, 2
    A, y = device(synth.kappa_matrix(m, n, 4.0, seed=4), dt), device(synth.rhs(m, k, 4), dt)
    q = B.CodedQR(m, n, 8, 4, 1, 48, dtype="f32" if dt == torch.float32 else "f64", mma=mma, nrhs_max=k, seed=3)
    q.encode(A)
    q.factor(0, -1)
    mp = q.geo["m_pad"]
    Qo, x = B.colmajor_empty(mp, n, dt), B.colmajor_empty(n, k, dt)
    q.post_orth(Qo)
    q.solve(y, x)
    Qb, Rb, Ab = (B.colmajor_empty(r, c, dt) for r, c in ((mp, n), (n, n), (m, n)))
    yb, xb = B.colmajor_empty(m, k, dt), B.colmajor_empty(n, k, dt)
    for t in (Qb, Rb, xb):
        t.fill_(0.5)
    Ab.zero_()
    yb.zero_()
    q.adjoint_qr(Qo, Qb, torch.triu(Rb).t().contiguous().t(), Ab)
    q.adjoint_lstsq(A, y, x, xb, Ab, yb)
    take(name, status=int(q.sync_status()), finite=bool(torch.isfinite(Ab).all() and torch.isfinite(yb).all()))
    q.close()

# a batch: both codes in one pass, erasures, post-orthogonalisation
shapes = [(203, 24), (331, 36), (1001, 60), (64, 16)]
As = [device(synth.gaussian(m, n, m), torch.float32) for m, n in shapes]
bt = B.CodedQRBatch(shapes, 8, 4, 2, seed=5)
bt.run(As, [(i, 0, 1 + i, i) for i in range(len(shapes))], graph=False, post_orth=True)
st, _, _ = bt.sync_status()
take("batch", status=int(st))
bt.close()
print(json.dumps(out))

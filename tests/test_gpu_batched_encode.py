"""The batched encode in one pass (k_b_encode_both) and its two-pass form against the oracle: tile
columns at the edges of both register widths (4 | 5, 8 | 9), every checksum count up to the generic
one, ragged rows, tiles smaller than a block, leading dimensions above m, and R left unprotected.
The copy is exact; a checksum sums at most p_r p_c FP32 products of O(1) terms."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2311_11943_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2311_11943_gb300 import binding as B  # noqa: E402


@pytest.mark.parametrize("p_r,p_c,f,protect", [(8, 4, 2, True), (10, 5, 1, True), (7, 8, 3, True),
                                               (9, 8, 4, True), (4, 2, 1, True), (11, 9, 2, True),
                                               (12, 10, 5, True), (8, 4, 2, False)])
def test_batched_encode_matches_the_oracle(p_r, p_c, f, protect):
    As = [synth.gaussian(m, n * p_c, m) for m, n in ((p_r * 40 + 3, 1), (p_r * 33, 9), (500, 17))]
    As = [np.asfortranarray(a.astype(np.float32).astype(np.float64)) for a in As]
    bt = B.CodedQRBatch([a.shape for a in As], p_r, p_c, f, b=4, protect_r=protect, seed=11)
    dev = []
    for k, a in enumerate(As):
        d = torch.full((a.shape[1], a.shape[0] + 5 * k), float("nan"), device="cuda")
        d[:, : a.shape[0]] = torch.from_numpy(np.ascontiguousarray(a.T))
        dev.append(d.t()[: a.shape[0]])
    bt.encode(dev)
    torch.cuda.synchronize()
    for i, a in enumerate(As):
        g = O.geom(a.shape[0], a.shape[1], p_r, p_c, f, protect_r=protect)
        Gt, Gh = O.generator(f, p_r, p_c, 11)
        ref = O.encode(g, Gt, Gh, a)
        M, N = bt.geo[i]["M"], bt.geo[i]["N"]
        Q = bt.factors(i)[0].double().cpu().numpy()[:M, :N]
        assert ref.shape == Q.shape and np.array_equal(Q[: a.shape[0], : a.shape[1]], a)
        assert np.abs(Q - ref).max() / np.abs(ref).max() < 4 * (p_r + p_c) * 2.0 ** -24
    bt.close()

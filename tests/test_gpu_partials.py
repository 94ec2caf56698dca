"""What the header states about the partial of a slot: where its reference m lies, and what repeats between calls."""
from __future__ import annotations

import numpy as np
import pytest

import workloads
from helpers import gpu_quantize
from test_gpu_parity import iq, torch  # noqa: F401 (fixtures)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("heads", [(8, 2), (8, 1)])
@pytest.mark.parametrize("levels", ["int8", "fp16"])
@pytest.mark.parametrize("d,S", [(128, 1), (128, 7), (256, 3)])
def test_reference_of_a_slot(iq, torch, d, S, levels, heads):  # noqa: F811
    """Fewer slots than the balanced mode takes: a slot's rows are the same in every call, so the run with the argmax output says
    what the exact maximum of each slot is."""
    H_q, H_kv = heads
    lens = [1, 129, 3000, 2222]
    w = workloads.tiny(1300 + S, 4, H_q, H_kv, d, 3000, lens=lens)
    w.k *= np.linspace(0.1, 3, 3000, dtype=np.float16)[None, :, None, None]  # scores grow along the rows: the reference lags behind and is raised
    cb = iq.iq_lloyd_max_codebook(d, 3, levels)
    shape, rot, cache, status = gpu_quantize(iq, torch, w, cb, n_new=lens)
    q = torch.from_numpy(w.q).cuda()
    lens_dev = torch.tensor(lens, dtype=torch.int32, device="cuda")

    def partials(want_argmax):
        ws = iq.DecodeWorkspace(shape, S, want_argmax=want_argmax)
        iq.iq_decode_attention(shape, rot, cb, q, cache, lens_dev, S, ws.part_acc, ws.part_ml, ws.part_argmax, ws.status)
        used = ws.part_ml[..., 1] > 0
        acc = torch.where(used[..., None], ws.part_acc, 0.0)
        return ws.part_ml.cpu().numpy().astype(np.float64), acc.cpu().numpy(), ws.part_argmax.cpu().numpy() if want_argmax else None

    exact, _, row = partials(True)
    ml, acc, _ = partials(False)
    used = exact[..., 1] > 0
    assert np.array_equal(used, ml[..., 1] > 0) and used.any() and (S == 1 or not used.all())
    above = ml[..., 0][used] - exact[..., 0][used]
    tol = 8 * 2.0 ** -24 * np.abs(exact[..., 0][used]).max()  # roundings of a score, of the reference and of its change of units
    assert above.max() <= 3 * np.log(2) + tol and above.min() >= -4 * np.log(2) - tol
    assert above.max() > 0                                   # (a slot of one block: its maximum and the margin of a raise)
    again, acc_again, _ = partials(False)
    assert np.array_equal(ml, again) and np.array_equal(acc, acc_again)
    exact_again, _, row_again = partials(True)
    assert np.array_equal(exact, exact_again) and np.array_equal(row, row_again)

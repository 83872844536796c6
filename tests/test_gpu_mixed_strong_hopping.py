"""C(t) of truncated chains on the mixed path at strong hopping per step (V dt up to 1).  There
the columns that hold only contraction noise, and with them the last bits of every QR and Krylov
step, move C(t) by up to 3e-4; the values are pinned to those of the FP64-FMA gauge QR."""
import json
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

GOLDEN = json.load(open(os.path.join(os.path.dirname(__file__), "golden",
                                     "mixed_strong_hopping.json")))
# complex64 contractions: the tolerance of a float32 result
TOL = 2e-5


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2003_13245_gb300.build import build_library
    build_library()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def model(c, **kw):
    from paper_2003_13245_gb300 import PREC_C64_3XTF32, Model
    m = Model(c["N"], [1.0], [1.0], [c["nmax"]], c["V"], precision=PREC_C64_3XTF32, **kw)
    m.thermal_prepare(2 * c["dt"], c["dt"], c["M"])
    return m


def close(C, c):
    ref = np.array(c["C"]) @ np.array([1.0, 1.0j])
    assert np.linalg.norm(C - ref) <= TOL * np.linalg.norm(ref)


@pytest.mark.parametrize("c", GOLDEN["single"], ids=lambda c: "V%.1f-dt%g-N%d" % (c["V"], c["dt"], c["N"]))
def test_single_chain(c):
    m = model(c)
    close(m.correlation(np.arange(2) * c["dt"], c["dt"]), c)
    m.close()


@pytest.mark.parametrize("batch", GOLDEN["batch"], ids=lambda b: "dt%g" % b[0]["dt"])
def test_batch(batch):
    from paper_2003_13245_gb300 import binding
    dt = batch[0]["dt"]
    models = [model(c, krylov=(1e-7, 32, 8)) for c in batch]
    for m in models:
        m.realtime_init()
    C = binding.Batch(models).correlation(np.arange(2) * dt, dt)
    for row, c in zip(np.asarray(C), batch):
        close(row, c)

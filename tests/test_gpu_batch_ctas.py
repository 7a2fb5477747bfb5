"""A limit on the batch's persistent CTAs holds for both of its kernels and changes no value: one CTA, a few, and more
than the force-field kernel launches by itself."""
import numpy as np
import pytest

from paper_2401_14564_gb300 import batch
from test_gpu_batch import cases

pytestmark = pytest.mark.gpu


def test_few_ctas_write_the_same_molecules():
    cs = cases(3, 5000)
    want = None
    for ctas in (0, 1, 5, 1000):
        b = batch.Batch(cs, ctas=ctas)
        b.ff.fill_(float("nan"))
        b.run()
        assert b.status() == (0, 0)
        got = [b.molecule(n)[k].cpu().numpy() for n in range(len(cs)) for k in ("ff", "fz", "df", "iters")]
        want = want or got
        assert all(np.array_equal(x, y) for x, y in zip(got, want)), ctas

"""Heterogeneous batches at the row widths the check pass is compiled for (8, 16 and 24 slots: one below,
at and above each), J from 1 to 4 and odd circulants, bit for bit against the per-code decoder."""
import pytest

from test_gpu_batch import batch_vs_single, pkg  # noqa: F401  (the module's fixture)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("opts_kw", [dict(max_iter=9, early_stop=1, msg=0), dict(max_iter=9, early_stop=1, msg=1),
                                     dict(max_iter=9, early_stop=0, msg=1), dict(max_iter=9, early_stop=1, algo=1, msg=2)])
def test_row_widths(pkg, opts_kw):
    specs = [(1, 2, 9, 40, 1), (2, 7, 31, 33, 2), (3, 8, 17, 65, 3), (4, 9, 23, 1, 4), (3, 15, 12, 64, 5),
             (4, 16, 29, 66, 6), (2, 17, 25, 31, 7), (3, 23, 27, 90, 8), (4, 24, 13, 129, 9)]
    batch_vs_single(pkg, specs, opts_kw, seeds=[3], ebn0=1.0)

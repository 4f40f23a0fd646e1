"""The Python binding's own argument handling (no GPU)."""
import pytest
import torch

from paper_2503_22695_gb300 import ibfe
from paper_2503_22695_gb300 import inputs as I

MODELS = [I.HO, I.NEO_HOOKEAN]


def test_material_table_rows():
    for cols in (9, 10):
        t = torch.arange(3.0 * cols, dtype=torch.float64).reshape(3, cols)
        mats = ibfe._mats_from(MODELS, t)            # a row more than models: unused
        for i, (m, a) in enumerate(zip(MODELS, mats)):
            assert a.model == m
            assert list(a.params) == t[i, :ibfe.N_PARAMS[m]].tolist()
            assert a.Ta == (float(t[i, 9]) if cols == 10 else 0.0)


@pytest.mark.parametrize("shape", [(1, 10), (1, 9), (0, 10), (10,), (20,)])
def test_material_table_without_a_row_for_every_model_is_refused(shape):
    with pytest.raises(IndexError):
        ibfe._mats_from(MODELS, torch.zeros(shape, dtype=torch.float64))

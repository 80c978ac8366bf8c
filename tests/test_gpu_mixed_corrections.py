"""A batch may mix the edge corrections.  A group of one order takes the operator
tables of its first member: on Gauss points, which batches need, the lifting
operators of the nodal DG schemes are the derivatives of the Radau polynomials,
so the tables of all three corrections are the same to rounding.

Tolerances: those of batches against single contexts (FP64 1e-12, FP32 2e-6)."""
import pytest

from paper_1709_01619_gb300 import _native as nat
from test_gpu_batch import TOL, initial, rel, singles

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("per_instance", [False, True])
@pytest.mark.parametrize("dtype", [nat.F64, nat.F32])
def test_mixed_corrections_in_one_group(dtype, per_instance):
    cs = [nat.Config(eqn=nat.EULER, nx=13, ny=9 + k, p=p, x1=6.5, y1=5.0, corr=corr, dtype=dtype)
          for p in (1, 2, 3, 4) for k, corr in enumerate((nat.CORR_NDG, nat.CORR_GDG, nat.CORR_NDG_LUMPED))]
    q0s = [initial(c, 3.0) for c in cs]
    ref, _ = singles(cs, q0s, 5, 0.004)
    with nat.Batch(cs) as b:
        b.set_form(per_instance)
        qs = [q.clone() for q in q0s]
        b.step(qs, 5, 0.004)
    for i, (q, r) in enumerate(zip(qs, ref)):
        assert rel(q, r) <= TOL[dtype], i

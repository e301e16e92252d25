"""The work counts of the traced kernels stand beside the peak of the unit that does the work.

No kernel of a step can run above the hardware's rate: a fraction above one (5 % for the clock that
the FP64 peak assumes) means operations counted against another unit's peak.  (H2O)8, mixed precision:
the solves of the fit and of the gradient, the digit-plane products and the integrals all have a count.
"""
import pytest

import bench
from paper_2407_19614_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_fractions_of_the_peaks(precision):
    from paper_2407_19614_gb300 import rihf as R
    mol = W.water8(0)
    ctx = R.Context(mol, precision=R.PRECISION_MIXED if precision == "mixed" else R.PRECISION_FP64, conv_e=1e-6,
                    conv_diis=1e-4, cuda_graphs=0)
    ctx.trace(True)
    ctx.update_geometry(mol.xyz)
    ctx.scf(guess=0, outputs=False)
    ctx.gradient()
    pk, src = bench.peaks()
    entries = {s["name"]: bench.roofline_entry(s, pk, src) for s in ctx.trace_stats() if s["work"] > 0}
    ctx.close()
    assert len(entries) >= 8
    assert {n: e["frac"] for n, e in entries.items() if e["frac"] > 1.05} == {}
    if precision == "mixed":
        assert [e["bound"] for n, e in entries.items() if n.startswith("fit trsm")] == ["tensor"]

"""An expired device wait is reported by the call it belongs to, whatever follows it in the call.

The status word of the bounded waits is set from the host (rihf_inject_timeout); no kernel waits or
fails.  After the error the context works again.
"""
import pytest

from paper_2407_19614_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("point", ["FIT", "GUESS", "ITERATION", "HISTORY", "GRADIENT"])
def test_expired_wait_is_reported(point, precision):
    from paper_2407_19614_gb300 import rihf as R
    mol = W.water_monomer(1)
    ctx = R.Context(mol, precision=R.PRECISION_MIXED if precision == "mixed" else R.PRECISION_FP64)
    guess = 3 if point == "HISTORY" else 0

    def step():
        ctx.update_geometry(mol.xyz)
        e = ctx.scf(guess=guess, outputs=False)["energy"]
        return e, ctx.gradient()

    ref, g = step()
    ctx.inject_timeout(point)
    with pytest.raises(R.RihfError) as err:
        step()
    assert err.value.code == -5
    if point in ("GUESS", "ITERATION"):
        with pytest.raises(R.RihfError) as err:   # no converged SCF to differentiate
            ctx.gradient()
        assert err.value.code == -7
    e, g2 = step()
    assert abs(e - ref) <= 1e-9 and abs(g2 - g).max() <= 1e-8
    ctx.close()


def test_a_point_that_is_not_reached_raises_nothing():
    from paper_2407_19614_gb300 import rihf as R
    mol = W.water_monomer(1)
    ctx = R.Context(mol)
    ctx.inject_timeout("HISTORY")   # guess 0 keeps no Loewdin history
    ctx.scf(guess=0, outputs=False)
    ctx.gradient()
    ctx.close()


def test_batch_reports_the_member():
    from paper_2407_19614_gb300 import rihf as R
    mols = [W.water_n(n, n) for n in (1, 2)]
    ctx = [R.Context(m) for m in mols]
    ref, _, _ = R.batch_step(ctx, [m.xyz for m in mols], guess=0)
    for point in ("FIT", "GUESS", "GRADIENT"):
        ctx[1].inject_timeout(point)
        with pytest.raises(R.RihfError, match="molecule 1") as err:
            R.batch_step(ctx, [m.xyz for m in mols], guess=0)
        assert err.value.code == -5
        E, _, _ = R.batch_step(ctx, [m.xyz for m in mols], guess=0)
        assert abs(E - ref).max() <= 1e-9
    for c in ctx:
        c.close()

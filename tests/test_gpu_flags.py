"""Device error flags become the same status on every path that reads them: a step, a group
step and a truncation (the flags are set on the host)."""
import pytest

from paper_2605_27515_gb300 import inputs, systems
from paper_2605_27515_gb300 import qlb as Q

pytestmark = pytest.mark.gpu

STATUS = {1: Q.ENOTCONV, 2: Q.ENONFINITE, 4: Q.ETIMEOUT, 5: Q.ETIMEOUT, 6: Q.ETIMEOUT}


@pytest.fixture(scope="module")
def built():
    cfg = inputs.config("cat_r5")
    cfg.update(R=[3], alpha2=1.0, dt=1e-2)
    ctx = Q.Ctx(device=0)
    b = systems.build(ctx, cfg)
    yield ctx, b, cfg
    ctx.close()


@pytest.mark.parametrize("path", ["step", "group", "truncate"])
@pytest.mark.parametrize("flags", sorted(STATUS))
def test_flags_become_a_status(built, path, flags):
    ctx, b, cfg = built
    st = b.sys.state(b.init)
    group = Q.Group(ctx, [st]) if path == "group" else None
    call = {"step": lambda: st.step(cfg["dt"], 1), "group": lambda: group.step(cfg["dt"], 1),
            "truncate": lambda: st.truncate(tol=1e-12)}[path]
    call()
    st.inject_flags(flags)
    with pytest.raises(Q.QlbError) as e:
        call()
    assert e.value.status == STATUS[flags]
    if flags & 4:
        assert "bounded wait" in str(e.value) and "truncation solve" in str(e.value)
    call()  # the flags are cleared
    if group:
        group.close()
    st.close()

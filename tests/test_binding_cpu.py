"""What the binding marshals follows the engine's buffers, shape and settings as they are at the call (no GPU needed)."""
import pytest
import torch

from paper_2605_11354_b200 import binding as lt
from paper_2605_11354_b200 import build as lb


@pytest.fixture(scope="module", autouse=True)
def built_library():
    lb.build()


def moved(t):
    """Other storage of the same size for a tensor object that stays the same."""
    return torch.empty(t.shape, dtype=t.dtype)


def test_structs_of_buffers_given_other_storage():
    shape = lt.Shape(1, 2, 300, 64, 64)
    x, plan = lt.alloc_fp8(shape, "cpu"), lt.alloc_plan(shape, 0.25, 0.25, "cpu")
    x.c_struct(), plan.c_struct()
    for obj, name in ((x, "codes"), (x, "scales"), (x, "colsum"), (plan, "cls"), (plan, "crit_idx"), (plan, "marg_idx")):
        t = getattr(obj, name)
        for give in (t.set_, lambda new: setattr(t, "data", new), lambda new: setattr(obj, name, new)):
            new = moved(t)
            give(new)
            assert getattr(obj.c_struct(), name) == new.data_ptr(), name


def test_counts_that_the_library_writes_are_not_kept(monkeypatch):
    """lite3r_sla_plan writes the counts of its fractions into the struct it is given; a plan made for others stays as it is."""
    shape = lt.Shape(1, 2, 300, 64, 64)
    x, plan = lt.alloc_fp8(shape, "cpu"), lt.alloc_plan(shape, 0.25, 0.25, "cpu")

    class Lib:
        @staticmethod
        def lite3r_sla_plan(q, k, s, crit, neg, p, stream):
            p.k_crit += 1
            return 0

    monkeypatch.setattr(lt, "_lib", Lib)
    monkeypatch.setattr(lt, "_stream_ptr", lambda stream: 0)
    with pytest.raises(AssertionError):
        lt.lite3r_sla_plan(x, x, shape, 0.5, 0.25, plan)
    assert plan.c_struct().k_crit == plan.k_crit


CHANGES = {
    "shape": lambda e: setattr(e.shape, "heads", 1), "crit": lambda e: setattr(e, "crit", 0.5),
    "neg": lambda e: setattr(e, "neg", 0.1), "phi": lambda e: setattr(e, "phi", lt.PHI_ELU1),
    "plan_inside": lambda e: setattr(e, "plan_inside", True), "counts": lambda e: setattr(e.plan, "k_crit", 2),
    "no column sums": lambda e: setattr(e.q8, "colsum", None), "smaller workspace": lambda e: e.workspace.set_(e.workspace[:512]),
    "status": lambda e: setattr(e, "status", torch.zeros(1, dtype=torch.int32)),
    **{f"{where} {how}": (lambda e, w=where, h=how: change(e, w, h))
       for where in ("q8.codes", "k8.scales", "k8.colsum", "v8.codes", "plan.cls", "plan.crit_idx", "plan.marg_idx", "workspace")
       for how in ("set_", "data", "assigned")},
}


def change(engine, where, how):
    *path, name = where.split(".")
    obj = engine
    for p in path:
        obj = getattr(obj, p)
    t = getattr(obj, name)
    new = moved(t)
    if how == "set_":
        t.set_(new)
    elif how == "data":
        t.data = new
    else:
        setattr(obj, name, new)


@pytest.mark.parametrize("what", CHANGES)
def test_a_step_is_marshalled_again_after_a_change(what, monkeypatch):
    """run() keeps its arguments between calls; whatever they hold that has changed makes it marshal them again."""
    marshalled = []

    class Lib:
        @staticmethod
        def lite3r_sla_step(step, stream):
            return 0

    def marshal(self, key, *tensors):
        marshalled.append(key)
        return key, None, None

    monkeypatch.setattr(lt, "_lib", Lib)
    monkeypatch.setattr(lt, "_stream_ptr", lambda stream: 0)
    monkeypatch.setattr(lt.SlaForward, "_marshal_step", marshal)
    with monkeypatch.context() as m:
        m.setattr(lt, "_lib", None)  # sizes come from the real library
        eng = lt.SlaForward(1, 2, 300, 64, 0.25, 0.25, device="cpu")
    held = [getattr(eng, n) for n in ("q8", "k8", "v8", "plan", "workspace", "status")]
    args = [torch.empty(1, 2, 300, 64) for _ in range(3)] + [torch.empty(2, 64, 64)]
    eng.run(*args)
    eng.run(*args)
    assert len(marshalled) == 1
    CHANGES[what](eng)
    eng.run(*args)
    assert len(marshalled) == 2 and held

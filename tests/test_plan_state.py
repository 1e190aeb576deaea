"""A plan is marked usable only once all of its device arrays exist, and every entry that launches from
a plan asks for that mark: an update whose last allocation fails leaves a model that is refused, not one
that renders from a null table.  Read off the source (the failure itself would fault a GPU)."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2008_05858_gb300", "csrc", "api.cu")


def _function(src, head):
    """The text of the function whose definition starts with `head`."""
    a = src.index(head)
    depth, i = 0, src.index("{", a)
    for j in range(i, len(src)):
        depth += {"{": 1, "}": -1}.get(src[j], 0)
        if depth == 0:
            return src[a:j + 1]
    raise AssertionError(head)


def test_the_mark_is_set_last():
    src = open(SRC).read()
    plan = _function(src, "int plan_model(Model* m) {")
    marks = [m.start() for m in re.finditer(r"P\.ok = true", src)]
    assert len(marks) == 1
    mark = plan.index("P.ok = true")
    assert not re.search(r"upload\(|cudaMalloc|launch_|plan_bands_and_tiles\(", plan[mark:])
    assert plan[mark:].count("return") == 1  # E2E_OK
    assert "upload(&P.d_egroups" in plan[:mark]


def test_every_user_of_a_plan_asks_for_the_mark():
    src = open(SRC).read()
    for head in ("int render_impl(", "int render_host_banded(", "int e2e_render_static(", "int e2e_render_adjoint("):
        body = _function(src, head)
        assert "if (!P.ok) return fail(" in body, head
        assert body.index("if (!P.ok)") < body.index("P.groups"), head

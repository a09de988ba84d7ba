"""The autotuner beside the choice by rule: the rule's own choice is one of those timed
and stays by rule when it wins; another variant holds for the batch that it was timed
with; lines of an earlier generation of kernels are not used.  Which variant ran is
read from the result's bits, which differ between the forms compared here."""
import json

import pytest

pytestmark = pytest.mark.gpu
DT, DX = 0.004, 12.5
NT, NX, V, MAXB = 700, 40, [1500.0, 2200.0, 2900.0, 3600.0], 6


def _pair(plan, batch):
    import torch
    gen = torch.Generator(device="cuda").manual_seed(11)
    m = torch.randn((batch,) + plan.model_shape, device="cuda", generator=gen)
    d = torch.randn((batch,) + plan.data_shape, device="cuda", generator=gen)
    od, om = torch.empty_like(d), torch.empty_like(m)
    plan.forward(m, od, batch=batch)
    plan.adjoint(d, om, batch=batch)
    return od, om


def _same(a, b):
    import torch
    return all(torch.equal(x, y) for x, y in zip(a, b))


def _plan():
    from paper_1711_10214_gb300 import ashrt
    return ashrt.Plan(NT, NX, DT, DX, V, max_batch=MAXB)


def _tuned_line(tmp_path):
    cache = str(tmp_path / "tune.jsonl")
    plan = _plan()
    mb, cols = plan.autotune(batch=4, cache_path=cache)
    line = json.loads(open(cache).read())
    assert line["rows_minb"] == mb and line["xfft_cols"] == cols and line["rule"] in (0, 1)
    plan.close()
    return line


def _from_line(tmp_path, line, name):
    path = tmp_path / name
    path.write_text(json.dumps(line) + "\n")
    plan = _plan()
    got = plan.autotune(batch=4, cache_path=str(path))
    return plan, got


def test_rule_is_kept_as_a_rule(lib, tmp_path):
    line = dict(_tuned_line(tmp_path), rule=1, xfft_cols=16)
    tuned, got = _from_line(tmp_path, line, "rule.jsonl")
    assert got[0] in range(1, 10)
    free = _plan()
    for batch in (1, 2, 4, 6):
        assert _same(_pair(tuned, batch), _pair(free, batch))
    tuned.close()
    free.close()


def test_variant_holds_for_its_batch(lib, tmp_path):
    line = dict(_tuned_line(tmp_path), rule=0, rows_minb=3, xfft_cols=16)
    tuned, got = _from_line(tmp_path, line, "three.jsonl")
    assert got == (3, 16)
    free, fixed = _plan(), _plan()
    fixed.set_variant(3, 16)
    assert _same(_pair(tuned, 4), _pair(fixed, 4))
    assert not _same(_pair(free, 4), _pair(fixed, 4))
    for batch in (1, 2, 6):
        assert _same(_pair(tuned, batch), _pair(free, batch))
        assert not _same(_pair(free, batch), _pair(fixed, batch))
    tuned.set_variant(3, 16)                       # set: for every batch
    assert _same(_pair(tuned, 2), _pair(fixed, 2))
    for p in (tuned, free, fixed):
        p.close()


def test_old_lines_are_not_used(lib, tmp_path):
    line = dict(_tuned_line(tmp_path), rows_minb=1)
    assert "|rows=2|" in line["key"]
    old = dict(line, key=line["key"].replace("|rows=2|", "|variants=9|"), pair_ms=0.0)
    old.pop("rule")
    plan, _ = _from_line(tmp_path, old, "old.jsonl")
    lines = [json.loads(x) for x in open(tmp_path / "old.jsonl")]
    assert len(lines) == 2 and "|rows=2|" in lines[1]["key"]       # timed again
    plan.close()

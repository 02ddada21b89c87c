"""The benchmark's result line: one short JSON line on stdout, the long sections as JSON
lines on stderr."""
import json


def test_the_line_is_short_and_the_sections_follow_on_stderr(capsys):
    import bench
    line = {"metric": "m", "value": 1.5, "unit": "u", "learned": None,
            "roofline": {"bound": "alu"}, "serving": {"table": ["x" * 100] * 200},
            "variants": {"runs": list(range(3000))}}
    bench.print_line(line)
    out, err = capsys.readouterr()
    assert out.count("\n") == 1 and len(out) < 2000
    got = json.loads(out)
    assert got["value"] == 1.5 and got["roofline"] == {"bound": "alu"}
    assert got["sections_on_stderr"] == ["serving", "variants"]
    sections = [json.loads(s) for s in err.splitlines()]
    assert [s["section"] for s in sections] == got["sections_on_stderr"]
    assert sections[1]["variants"] == line["variants"]

"""The result line of bench.py stays short enough to be kept whole where output is cut at 3000 characters; its tables go beside it."""
import json

import bench


def test_result_line_is_short_and_tables_go_beside_it():
    line = {"metric": "m", "value": 1.0, "config": {"text": "x" * 700}, "roofline": {"text": "x" * 900}, "e2e": {"text": "x" * 200}, "clocks": {"text": "x" * 70},
            "cpu_baseline": {"value": 2.0, "sample": "x" * 330, "single_thread": {"one_thread": "x" * 150}}}
    tables = {k: [{"row": i, "text": "x" * 150} for i in range(40)] for k in bench.DETAILS}
    short, details = bench.split_details({**line, **tables})
    assert len(json.dumps(short)) < 2600 and short["value"] == 1.0 and short["cpu_baseline"]["value"] == 2.0
    assert {k: details[k] for k in bench.DETAILS} == tables and details["cpu_baseline"] == line["cpu_baseline"]

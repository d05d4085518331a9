"""Host rule for the lanes that share a row of the pair sweep (no GPU):
compiled from its header.  Sizes at which four lanes were measured to be the
slower choice (one lane takes less time there, and no more than a build
without shared rows) get one, those at which they were measured to be the
faster one get four."""
from test_persistent_host import compiled

# natom, atoms in 3-D replicas, FP64, persistent launch -> lanes
MEASURED = [
    (6736, 0, 0, 1, 4), (9683, 0, 1, 1, 4), (15156, 0, 1, 0, 1), (15156, 0, 0, 1, 1), (25260, 0, 1, 1, 1), (38732, 0, 1, 0, 1),
    (38732, 0, 0, 0, 1), (9915, 9915, 1, 0, 4), (14272, 14272, 1, 1, 4), (15864, 15864, 1, 0, 1), (15864, 15864, 0, 0, 4),
    (19830, 19830, 1, 0, 4), (19830, 19830, 1, 1, 4), (23796, 23796, 1, 0, 4), (23796, 23796, 1, 1, 1), (28544, 28544, 1, 1, 1), (28544, 28544, 1, 0, 4),
    (37677, 37677, 1, 0, 1), (37677, 37677, 1, 1, 1), (37677, 37677, 0, 1, 4), (39660, 39660, 0, 0, 1), (57088, 57088, 1, 0, 1)]


def test_lanes_at_the_measured_sizes(tmp_path):
    calls = ", ".join("row_lanes(%d, %d, %d, %d)" % m[:4] for m in MEASURED)
    out = compiled(tmp_path, 'const int v[] = {%s}; for (int x : v) printf("%%d\\n", x);' % calls)
    assert [int(v) for v in out] == [m[4] for m in MEASURED]


def test_lanes_are_one_or_four(tmp_path):
    out = compiled(tmp_path, "int bad = 0, far = 0; for (long long n = 1; n <= 200000; n += 7) for (int k = 0; k < 12; ++k) {"
                             " const int v = row_lanes(n, n * (k >> 2) / 2, k & 1, (k >> 1) & 1); bad += v != 1 && v != 4;"
                             ' far += v != 1 && n >= 38912; } printf("%d %d\\n", bad, far);')
    assert out == ["0", "0"]

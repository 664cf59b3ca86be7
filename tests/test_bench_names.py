"""bench.py names the kernels that ran, on the CPU: a mixed context launches the
line kernels or the x-y tiles, by its box."""

import bench


def test_mixed_form_is_named_by_its_launches():
    lines, tiles = bench.df64_kernel_names((9, 9, 9)), bench.df64_kernel_names((9, 0, 9))
    assert lines == ("k_df_line_x", "k_df_tline_y", "k_df_tline_z")
    assert "k_df_line_x" not in tiles and tiles[1] == "-" and tiles[2] == lines[2]
    for k in lines + tiles:
        assert k == "-" or k in bench.KERNEL_VALUES_PER_NODE

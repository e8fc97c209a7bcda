/*
 * lbp_test_hooks.h -- entry points of liblbp that exist for the test suite
 * only.  They are not part of the library's interface (include/lbp.h) and an
 * application has no use for them.
 */
#ifndef LBP_TEST_HOOKS_H_
#define LBP_TEST_HOOKS_H_

#include <stddef.h>
#include <stdint.h>

#ifdef __cplusplus
extern "C" {
#endif

/* Failure injection for the bounded waits of the persistent products kernel
 * (bf16 low-rank path of lbp_backward).  While switched on (per calling
 * thread), the TMA producer of every products launch issues no load at all.
 * Nothing is then in flight, the tensor-core issuer and the epilogue warps run
 * into their wait limits (about a second), the kernel reports LBP_ERR_TIMEOUT
 * in the status block of the call's workspace, releases its tensor memory and
 * returns; the outputs of that call are undefined and the context stays
 * usable.  The paper has no counterpart; this is how the exit path behind
 * lbp_poll_status is exercised without faulting or hanging a device.
 * `on`: bit 0 stalls the products kernels as described; bit 1 does the same to
 * the TMA producers of the tcgen05 projection kernel (orders 8 and 16, bf16, r <= 48:
 * lbp_project and the first kernel of lbp_backward); bit 2 to the loads of the fp32
 * products on the tensor cores; 0 switches all off.
 * Returns LBP_OK. */
int lbp_test_stall_products(int on);

/* Host-side tile plan of the persistent products kernel for a layer of Cin x
 * Cout channels whose low-rank rows fill G groups of 128 rows (bpt blocks per
 * group, order k), on `units` CTAs (pair = 0) or CTA pairs (pair = 1).
 * out6 = {BNw, BNx, K slices of g_W, k-blocks per slice, listed, tiles listed};
 * first: 161 entries, ids: 1536 entries: unit u works, in this order, on the
 * tiles ids[first[u]] .. ids[first[u+1]-1]; ids below (row tiles of g_W) *
 * (column tiles) * slices are GW tiles, the others GX tiles.  No device needed. */
int lbp_test_tile_plan(int Cin, int Cout, int G, int bpt, int k, int units, int pair,
                       int max_splits, int epi_kind, int32_t* out6, uint16_t* first, uint16_t* ids);

/* The plan that a call with this bf16 layer, basis list and number of tokens outside the
 * grid runs on `units` CTAs (pair = 0) or CTA pairs (1); set = NULL: exact backpropagation
 * of the whole grid.  out8 = {BNw, BNx, blocks of a GX tile, K slices of g_W, k-blocks of a
 * slice, listed, k-blocks of g_W, K slices there is room for}; first and ids as above (where
 * listed).  No device needed. */
int lbp_test_products_plan(const lbp_layer* layer, const lbp_basis* set, int r, int n_extra, int units, int pair,
                           int32_t* out8, uint16_t* first, uint16_t* ids);

/* The plan of the two fp32 products over `rows` rows of a layer of Cin x Cout channels with
 * `room` bytes for planes (gemm_fp32.cu).  out6 = {form, bytes of planes,
 * k-blocks of an item of g_x and items of K per tile of it, the same of g_W}.  No device
 * needed. */
int lbp_test_float_plan(int Cin, int Cout, long long rows, size_t room, int64_t* out6);

/* The library reads its tuning switches (LBP_FUSED, LBP_PAIR, LBP_FUSED_TILES,
 * LBP_FUSED_VERBOSE) from the environment once, at first use.  This reads them
 * again, so that one test process can run the same layer through the paths
 * the switches select.  Returns LBP_OK. */
int lbp_test_reload_env(void);

/* Calls inside(arg) in the section in which lbp_backward_batch uses the stream and the
 * events that the library keeps for `device` (0..63), and returns its result.  No
 * device needed. */
int lbp_test_side_section(int device, int (*inside)(void*), void* arg);

/* What the library does once on each device (the opt-in of a kernel to more shared
 * memory): done[i] = 1 where a run over devices[0..n-1] would have done it at i. */
int lbp_test_per_device(const int* devices, int n, uint8_t* done);

/* sizeof of the structs of include/lbp.h as the library was compiled (which: 0
 * lbp_layer, 1 lbp_extras, 2 lbp_view, 3 lbp_basis; anything else: 0), so that a
 * binding in another language can check its own declarations against them. */
size_t lbp_test_struct_size(int which);

#ifdef __cplusplus
}
#endif
#endif /* LBP_TEST_HOOKS_H_ */

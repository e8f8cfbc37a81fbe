// Exchange skeleton of the whole-block persistent kernel with all workers in one cluster (no arithmetic of the method).
#define PK_BODY_FILE "persistent_body.inc"
#define PK_KERNEL_NAME persistent_local_wide_floor_kernel
#define PK_LOOKUP_NAME pk_lookup_local_wide_floor
#define PK_PLUS 0
#define PK_EF 0
#define PK_FLOOR 1
#define PK_LOCAL 1
#define PK_ONE_CHUNK
#include "persistent_method.inc"

// Persistent kernel, all workers in one cluster: instantiations and their lookup.
#define PK_BODY_FILE "persistent_roles.inc"
#define PK_KERNEL_NAME persistent_local_ef_kernel
#define PK_LOOKUP_NAME pk_lookup_local_ef
#define PK_PLUS 0
#define PK_EF 1
#define PK_FLOOR 0
#define PK_LOCAL 1
#include "persistent_method.inc"
